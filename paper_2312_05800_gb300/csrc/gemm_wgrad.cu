// gemm_wgrad.cu -- weight and bias gradients of the network's layers in one
// launch: dW_l = dZ_l^T H_{l-1} and db_l = column sums of dZ_l (Sec. 3.2, backward pass).
//
// Both factors lie in memory with the contracted dimension (the batch) as rows, so
// both go to the tensor cores M- and N-major as TMA loads them (boxes of 64 columns
// x 64 rows, 128-byte swizzle); no transposed copies are made. A CTA computes one
// 128 x 128 tile of one layer over the whole batch; the layers' tiles form one grid,
// longest layers first, since one layer alone leaves most SMs idle (29 x 400 outputs are
// four tiles). The bias gradient is one more product of the same A operand
// with a tile of ones (16 columns of TMEM) in the CTAs of a layer's first tile
// column.
//
// What bounds it: the loads, 32 KB of operands per 64 rows and CTA from L2. It replaces per layer two
// transposes, a product on 2 to 70 CTAs and a column-sum kernel: 248 us of the 4096-row step of the
// 32-1600-800-400-29 network before, 35 us in this kernel.
//
// Roles (192 threads): warp 0 TMA producer, warp 1 TMEM allocation and MMA, warps
// 2..5 epilogue (one per TMEM lane quadrant). Every wait is bounded as in gemm.cuh.
#include "gemm_launch.cuh"

namespace chemgb {
namespace {

constexpr int kWgStages = 6;
constexpr int kWgThreads = 192;
constexpr int kWgMaxLayers = 4;
constexpr uint32_t kWgOperand = 128 * kBK * 2;      // 128 columns x 64 rows of BF16 (two boxes)
constexpr uint32_t kWgOnes = 16 * 128;              // 16 rows x 64 columns of ones
constexpr uint32_t kWgSmem = 1024 + kWgStages * 2 * kWgOperand + kWgOnes + (2 * kWgStages + 2) * 8 + 16;

struct WgradProblem {
    CUtensorMap dz, h;
    int out, in, n_tiles, first;                    // first: index of the layer's first tile in the grid
    float *gW, *gb;
    int64_t ldg;
};
struct WgradArgs {
    WgradProblem p[kWgMaxLayers];
    int count, B;
    uint32_t spin;
};

__global__ void __launch_bounds__(kWgThreads, 1) gemm_wgrad_kernel(const __grid_constant__ WgradArgs a, int *err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sA = smem, *sB = smem + kWgStages * kWgOperand, *ones = smem + 2 * kWgStages * kWgOperand;
    uint64_t *full = reinterpret_cast<uint64_t *>(ones + kWgOnes);
    uint64_t *empty = full + kWgStages, *done = empty + kWgStages;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int l = 0;
    while (l + 1 < a.count && (int)blockIdx.x >= a.p[l + 1].first) ++l;
    const WgradProblem &p = a.p[l];
    const int t = (int)blockIdx.x - p.first, m_blk = t / p.n_tiles, n_blk = t % p.n_tiles;
    const int kblocks = (a.B + kBK - 1) / kBK;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kWgStages; ++s) { tc::mbar_init(&full[s], 1); tc::mbar_init(&empty[s], 1); }
        tc::mbar_init(done, 1);
        tc::fence_barrier_init();
    }
    for (int i = threadIdx.x; i < (int)kWgOnes / 4; i += kWgThreads)
        reinterpret_cast<uint32_t *>(ones)[i] = 0x3F803F80u;
    tc::fence_proxy_async_smem();
    if (warp == 1) {
        tc::tmem_alloc(tmem_slot, 256);
        tc::tmem_relinquish();
    }
    tc::grid_wait();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (warp == 0) {
        if (lane == 0) {
            tc::tma_prefetch_desc(&p.dz);
            tc::tma_prefetch_desc(&p.h);
            int it = 0;
            for (; it < kblocks; ++it) {
                const int s = it % kWgStages;
                if (!tc::mbar_wait(&empty[s], (uint32_t)((it / kWgStages) & 1) ^ 1u, a.spin)) {
                    atomicExch(err, tc::kErrTimeoutEmpty);
                    break;
                }
                tc::mbar_arrive_expect_tx(&full[s], 2 * kWgOperand);
                for (int j = 0; j < 2; ++j) {
                    tc::tma_load_2d(sA + s * kWgOperand + j * 8192, &p.dz, &full[s], m_blk * 128 + j * 64, it * kBK);
                    tc::tma_load_2d(sB + s * kWgOperand + j * 8192, &p.h, &full[s], n_blk * 128 + j * 64, it * kBK);
                }
            }
            // every issued load lands before the CTA may exit (full limit)
            for (int j = (it > kWgStages ? it - kWgStages : 0); j < it; ++j)
                if (!tc::mbar_wait(&full[j % kWgStages], (uint32_t)(j / kWgStages) & 1u)) {
                    atomicExch(err, tc::kErrTimeoutDrain);
                    break;
                }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t id_w = tc::idesc_bf16_f32(128, 128) | tc::kIdescAMNMajor | tc::kIdescBMNMajor;
            constexpr uint32_t id_b = tc::idesc_bf16_f32(128, 16) | tc::kIdescAMNMajor;
            const uint32_t one = tc::smem_u32(ones);
            bool ok = true;
            for (int it = 0; it < kblocks; ++it) {
                const int s = it % kWgStages;
                if (!tc::mbar_wait(&full[s], (uint32_t)(it / kWgStages) & 1u, a.spin)) {
                    atomicExch(err, tc::kErrTimeoutFull);
                    ok = false;
                    break;
                }
                tc::tc_fence_after();
                const uint32_t a0 = tc::smem_u32(sA + s * kWgOperand), b0 = tc::smem_u32(sB + s * kWgOperand);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint64_t ad = tc::sdesc_mnmajor_sw128(a0 + kk * 2048, 8192);
                    const uint32_t acc = (it > 0 || kk > 0) ? 1u : 0u;
                    tc::umma_f16(tmem, ad, tc::sdesc_mnmajor_sw128(b0 + kk * 2048, 8192), id_w, acc);
                    if (n_blk == 0) tc::umma_f16(tmem + 128, ad, tc::sdesc_kmajor_sw128(one + kk * 32), id_b, acc);
                }
                tc::umma_commit(&empty[s]);
            }
            // all issued MMAs complete (the epilogue reads, TMEM is released); full limit
            tc::umma_commit(done);
            if (!tc::mbar_wait(done, 0)) { atomicExch(err, tc::kErrTimeoutDrain); ok = false; }
            tmem_slot[1] = ok ? 1u : 0u;
        }
    }
    __syncthreads();
    tc::tc_fence_after();
    if (warp >= 2 && tmem_slot[1]) {
        const int quad = warp & 3;
        const int row = m_blk * 128 + quad * 32 + lane;
        const uint32_t base = tmem + ((uint32_t)(quad * 32) << 16);
        for (int c = 0; c < 8; ++c) {
            const int col0 = n_blk * 128 + c * 16;
            if (col0 >= p.in) break;                // warp-uniform
            float v[16];
            tc::tmem_ld16(base + (uint32_t)(c * 16), v);
            if (row < p.out) {
                float *o = p.gW + (int64_t)row * p.ldg + col0;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (col0 + 4 * i < p.in)        // in and ldg are multiples of 4
                        reinterpret_cast<float4 *>(o)[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
            __syncwarp();
        }
        if (n_blk == 0) {
            float v[16];
            tc::tmem_ld16(base + 128u, v);
            if (row < p.out) p.gb[row] = v[0];
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, 256);
    }
}

}  // namespace

int gemm_wgrad(const WgradLayer *layers, int count, int B, int *err, cudaStream_t st) {
    if (count < 1 || count > kWgMaxLayers || B < 1) return set_error(CHEM_EINVAL, "weight gradients: bad sizes");
    static DeviceOnce configured;
    if (int rc = dynamic_smem_limit(configured, gemm_wgrad_kernel, kWgSmem, "weight gradient smem attribute")) return rc;
    WgradArgs a;
    std::memset(&a, 0, sizeof(a));
    a.count = count;
    a.B = B;
    a.spin = gemm_wait_limit();
    int tiles = 0;
    for (int l = 0; l < count; ++l) {
        const WgradLayer &L = layers[l];
        if ((L.in & 3) != 0 || (L.ldg & 3) != 0 || !aligned16(L.gW))
            return set_error(CHEM_EINVAL, "weight gradients: rows must be multiples of 16 bytes");
        WgradProblem &p = a.p[l];
        int rc = make_tmap_operand(&p.dz, L.dz, B, L.out, L.ldz, kBK, 2);
        if (!rc) rc = make_tmap_operand(&p.h, L.h, B, L.in, L.ldh, kBK, 2);
        if (rc) return rc;
        p.out = L.out;
        p.in = L.in;
        p.n_tiles = (L.in + 127) / 128;
        p.first = tiles;
        p.gW = L.gW;
        p.gb = L.gb;
        p.ldg = L.ldg;
        tiles += (L.out + 127) / 128 * p.n_tiles;
    }
    void *pb = prof_begin(st);
    launch_dependent(gemm_wgrad_kernel, tiles, tiles, kWgThreads, kWgSmem, st, a, err);
    if (pb) {
        double fl = 0.0, by = 0.0;
        for (int l = 0; l < count; ++l) {
            fl += 2.0 * B * layers[l].out * layers[l].in;
            by += 2.0 * B * (layers[l].out + layers[l].in) + 4.0 * layers[l].out * layers[l].in;
        }
        prof_end(pb, st, "gemm_wgrad_kernel", fl, by);
    }
    return check_cuda(cudaGetLastError(), "weight gradient launch");
}

}  // namespace chemgb
