// gemm_launch.cuh -- host-side launch of gemm_tn_kernel: TMA descriptors,
// tile-width dispatch and the persistent grid. Included by the translation
// units that instantiate the kernel for their epilogue.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

#include <cstring>
#include <mutex>
#include <string>

#include "gemm.cuh"
#include "internal.cuh"
#include "tile_width.h"

namespace chemgb {

// cuTensorMapEncodeTiled resolved through the runtime (no link-time libcuda dependency).
inline PFN_cuTensorMapEncodeTiled_v12000 encode_tiled_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        else
            cudaGetLastError();
    });
    return fn;
}

// 2-D operand tensor map over a row-major [rows][cols] matrix of BF16 (esize 2)
// or E4M3 (esize 1) with row stride ld (elements): box = box_rows x 128 bytes,
// 128-byte swizzle, zero fill outside.
inline int make_tmap_operand(CUtensorMap *map, const void *ptr, int64_t rows, int64_t cols, int64_t ld, int box_rows,
                             int esize) {
    if (!aligned16(ptr) || (ld * esize) % 16 != 0)
        return set_error(CHEM_EINVAL, "GEMM operand: base must be 16-byte aligned and rows a multiple of 16 bytes");
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)(ld * esize)};
    cuuint32_t box[2] = {(cuuint32_t)(128 / esize), (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_tiled_fn();
    if (!enc) return set_error(CHEM_EUNSUPPORTED, "cuTensorMapEncodeTiled is not available from the driver");
    CUresult r = enc(map, esize == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 2,
                     const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(CHEM_ECUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
    return CHEM_OK;
}

// A GEMM operand: row-major rows of K elements with row stride ld; for a grouped launch its
// map kind and the elements between consecutive groups (rows x ld for stacked rows, the column
// offset for side-by-side columns).
struct GemmOperand {
    const void *ptr;
    int64_t ld;
    int kind;
    int64_t gstride;
};

// 3-D operand map of one of the grouped kinds: box = box_rows x 128 bytes of one group.
// Stacked rows: dims (K, rows, G), strides (ld, gstride); side-by-side columns: dims
// (K, G, rows), strides (gstride, ld). Zero fill outside, so K and rows clip per group.
inline int make_tmap_operand_grouped(CUtensorMap *map, const GemmOperand &op, int64_t rows, int64_t cols, int G,
                                     int box_rows, int esize) {
    if (!aligned16(op.ptr) || (op.ld * esize) % 16 != 0 || (op.gstride * esize) % 16 != 0 || op.gstride <= 0)
        return set_error(CHEM_EINVAL, "grouped GEMM operand: base, row and group strides must be 16-byte multiples");
    const bool rowg = op.kind == kMapRowGrp;
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)(rowg ? rows : G), (cuuint64_t)(rowg ? G : rows)};
    cuuint64_t strides[2] = {(cuuint64_t)((rowg ? op.ld : op.gstride) * esize),
                             (cuuint64_t)((rowg ? op.gstride : op.ld) * esize)};
    cuuint32_t box[3] = {(cuuint32_t)(128 / esize), (cuuint32_t)(rowg ? box_rows : 1), (cuuint32_t)(rowg ? 1 : box_rows)};
    cuuint32_t estr[3] = {1, 1, 1};
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_tiled_fn();
    if (!enc) return set_error(CHEM_EUNSUPPORTED, "cuTensorMapEncodeTiled is not available from the driver");
    CUresult r = enc(map, esize == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 3,
                     const_cast<void *>(op.ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        return set_error(CHEM_ECUDA, "cuTensorMapEncodeTiled (grouped) failed (" + std::to_string((int)r) + ")");
    return CHEM_OK;
}

inline int make_operand_map(CUtensorMap *map, const GemmOperand &op, int64_t rows, int64_t cols, int G, int box_rows,
                            int esize) {
    if (op.kind == kMap2D) return make_tmap_operand(map, op.ptr, rows, cols, op.ld, box_rows, esize);
    return make_tmap_operand_grouped(map, op, rows, cols, G, box_rows, esize);
}

// Tries of each pipeline wait of the GEMMs launched by this host thread (tc::kSpinLimit unless a
// network handle with a smaller limit is launching; see WaitLimitScope).
inline uint32_t &gemm_wait_limit() {
    static thread_local uint32_t limit = tc::kSpinLimit;
    return limit;
}
// Sets this thread's GEMM wait limit for the lifetime of the object, then restores it.
struct WaitLimitScope {
    uint32_t saved;
    explicit WaitLimitScope(uint32_t limit) : saved(gemm_wait_limit()) { gemm_wait_limit() = limit; }
    ~WaitLimitScope() { gemm_wait_limit() = saved; }
    WaitLimitScope(const WaitLimitScope &) = delete;
    WaitLimitScope &operator=(const WaitLimitScope &) = delete;
};

inline int num_sms() {
    static DeviceInt sms;
    int dev = 0;
    cudaGetDevice(&dev);
    return sms.value(dev, [dev] {
        int v = 0;
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v;
    });
}

// Output tensor map for the TMA-store epilogue: [rows][cols] of BF16 (esize 2)
// or E4M3 (esize 1), box 32 rows x box_cols columns, no swizzle.
inline int make_tmap_out(CUtensorMap *map, const void *ptr, int64_t rows, int64_t cols, int64_t ld, int esize,
                         int box_cols) {
    if (!aligned16(ptr) || (ld * esize) % 16 != 0)
        return set_error(CHEM_EINVAL, "GEMM output: base must be 16-byte aligned and rows a multiple of 16 bytes");
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)(ld * esize)};
    cuuint32_t box[2] = {(cuuint32_t)box_cols, 32};
    cuuint32_t estr[2] = {1, 1};
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_tiled_fn();
    if (!enc) return set_error(CHEM_EUNSUPPORTED, "cuTensorMapEncodeTiled is not available from the driver");
    CUresult r = enc(map, esize == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 2,
                     const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(CHEM_ECUDA, "cuTensorMapEncodeTiled (output) failed (" + std::to_string((int)r) + ")");
    return CHEM_OK;
}

// Output map of a grouped TMA-store epilogue: box 32 rows x box_cols columns of one group.
inline int make_tmap_out_grouped(CUtensorMap *map, const void *ptr, int kind, int64_t rows, int64_t cols, int G,
                                 int64_t ld, int64_t gstride, int esize, int box_cols) {
    if (kind == kMap2D) return make_tmap_out(map, ptr, rows, cols, ld, esize, box_cols);
    if (!aligned16(ptr) || (ld * esize) % 16 != 0 || (gstride * esize) % 16 != 0 || gstride <= 0)
        return set_error(CHEM_EINVAL, "grouped GEMM output: base, row and group strides must be 16-byte multiples");
    const bool rowg = kind == kMapRowGrp;
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)(rowg ? rows : G), (cuuint64_t)(rowg ? G : rows)};
    cuuint64_t strides[2] = {(cuuint64_t)((rowg ? ld : gstride) * esize), (cuuint64_t)((rowg ? gstride : ld) * esize)};
    cuuint32_t box[3] = {(cuuint32_t)box_cols, (cuuint32_t)(rowg ? 32 : 1), (cuuint32_t)(rowg ? 1 : 32)};
    cuuint32_t estr[3] = {1, 1, 1};
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_tiled_fn();
    if (!enc) return set_error(CHEM_EUNSUPPORTED, "cuTensorMapEncodeTiled is not available from the driver");
    CUresult r = enc(map, esize == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 3,
                     const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        return set_error(CHEM_ECUDA, "cuTensorMapEncodeTiled (grouped output) failed (" + std::to_string((int)r) + ")");
    return CHEM_OK;
}

// Launches a GEMM kernel so that it may start while the kernel before it in the stream still runs (programmatic
// dependent launch): it sets up its barriers and TMEM and then waits, in the kernel, for that kernel's end
// (tc::grid_wait) before it reads or writes anything in global memory. For short launches only, at most two
// tiles per SM: the training step of 4,096 rows, eight such products in a row, takes 173 us instead of 191, the learned
// step of 2,500 cells 85 instead of 93, but a long product gains nothing and the dense layer of 262,144 rows
// took 563 us instead of 549.
template <class... P, class... A>
inline void launch_dependent(void (*kernel)(P...), int64_t tiles, int grid, int threads, size_t smem, cudaStream_t st,
                             A &&...args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = tiles <= 2 * (int64_t)num_sms() ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, P(args)...);       // an error stays for the caller's cudaGetLastError
}

// G products of M x N x K in one persistent launch; out_kind / out_gstride describe the
// TMA-store output (used when the epilogue stores by TMA; element stores use the functor's
// own group offsets, which must agree).
template <int BN, int STAGES, class Epi>
int launch_gemm_grouped_bn(const GemmOperand &A, const GemmOperand &B, int G, int out_kind, int64_t out_gstride, int M,
                           int N, int K, const Epi &epi, int *err, cudaStream_t st, int max_ctas) {
    using L = GemmSmem<BN, STAGES>;
    static DeviceOnce configured;
    int rc = dynamic_smem_limit(configured, gemm_tn_kernel<BN, STAGES, Epi>, L::kTotal, "GEMM smem attribute");
    if (rc) return rc;
    const int esize = Epi::kF8 ? 1 : 2;
    CUtensorMap ta, tb, tc, tc1;
    rc = make_operand_map(&ta, A, M, K, G, kBM, esize);
    if (rc) return rc;
    // N-major B: [K][N], boxes of 64 columns x 64 rows
    rc = Epi::kBNMajor ? make_operand_map(&tb, B, K, N, G, kBK, esize) : make_operand_map(&tb, B, N, K, G, BN, esize);
    if (rc) return rc;
    std::memset(&tc, 0, sizeof(tc));
    std::memset(&tc1, 0, sizeof(tc1));
    if (const void *op = epi.tma_ptr()) {                    // 32-byte row pieces; one E4M3 chunk by itself
        const int os = Epi::kOutBytes / 16;
        rc = make_tmap_out_grouped(&tc, op, out_kind, M, N, G, epi.ldo, out_gstride, os, 32 / os);
        if (!rc && os == 1) rc = make_tmap_out_grouped(&tc1, op, out_kind, M, N, G, epi.ldo, out_gstride, os, 16);
        if (rc) return rc;
    }
    const int64_t tiles64 = (int64_t)((M + kBM - 1) / kBM) * ((N + BN - 1) / BN) * G;
    if (tiles64 > 0x7fffffff) return set_error(CHEM_EINVAL, "GEMM: too many tiles for one launch");
    const int tiles = (int)tiles64;
    int grid = num_sms();
    if (max_ctas > 0 && max_ctas < grid) grid = max_ctas;
    if (tiles < grid) grid = tiles;
    const GemmGroups grp{G, A.kind, B.kind, out_kind, gemm_wait_limit()};
    void *pb = prof_begin(st);
    launch_dependent(gemm_tn_kernel<BN, STAGES, Epi>, tiles, grid, kGemmThreads, L::kTotal, st, ta, tb, tc, tc1, M, N, K, grp,
                     epi, err);
    if (pb)
        prof_end(pb, st, "gemm_tn_kernel<" + std::to_string(BN) + (Epi::kF8 ? ",e4m3> " : "> ") +
                             (G > 1 ? std::to_string(G) + "x" : std::string()) + std::to_string(N) + "x" +
                             std::to_string(K),
                 2.0 * M * N * K * G, (double)esize * ((double)M * K + (double)N * K) * G);
    return check_cuda(cudaGetLastError(), "GEMM launch");
}

// G products in one launch (single-CTA tiles only).
template <class Epi>
int launch_gemm_grouped(int bn, const GemmOperand &A, const GemmOperand &B, int G, int out_kind, int64_t out_gstride,
                        int M, int N, int K, const Epi &epi, int *err, cudaStream_t st, int max_ctas = 0) {
    if (M <= 0 || N <= 0 || K <= 0 || G <= 0) return CHEM_OK;
    switch (bn) {
#define CHEMGB_GROUPED_CASE(W_, S_)                                                                                 \
    case W_:                                                                                                        \
        return launch_gemm_grouped_bn<W_, S_>(A, B, G, out_kind, out_gstride, M, N, K, epi, err, st, max_ctas);
        CHEMGB_GROUPED_CASE(32, 8)
        CHEMGB_GROUPED_CASE(64, 8)
        CHEMGB_GROUPED_CASE(128, 6)
        CHEMGB_GROUPED_CASE(160, 5)
        CHEMGB_GROUPED_CASE(208, 4)
        CHEMGB_GROUPED_CASE(256, 4)
#undef CHEMGB_GROUPED_CASE
        default: return set_error(CHEM_EINVAL, "GEMM: unsupported tile width " + std::to_string(bn));
    }
}

template <class Epi>
int launch_gemm(int bn, const void *X, int64_t ldx, const void *W, int64_t ldw, int M, int N, int K,
                const Epi &epi, int *err, cudaStream_t st, int max_ctas = 0) {
    if (M <= 0 || N <= 0 || K <= 0) return CHEM_OK;
    return launch_gemm_grouped(bn, GemmOperand{X, ldx, kMap2D, 0}, GemmOperand{W, ldw, kMap2D, 0}, 1, kMap2D, 0, M, N,
                               K, epi, err, st, max_ctas);
}

// Forward declarations of the per-epilogue launchers (one translation unit each).
int gemm_gelu(int bn, const void *X, int64_t ldx, const void *W, int64_t ldw, int M, int N, int K, const float *bias,
              void *out, int64_t ldo, float *pre, int64_t ldp, int *err, cudaStream_t st, int max_ctas = 0);
int gemm_linear(int bn, const void *X, int64_t ldx, const void *W, int64_t ldw, int M, int N, int K,
                const float *bias, float *out, int64_t ldo, int *err, cudaStream_t st, int max_ctas = 0);
// X W with W the layer's own weights [K][N] (row-major, N-major operand), times GELU'(z)
int gemm_gelu_grad(const void *X, int64_t ldx, const void *W, int64_t ldw, int M, int N, int K, const float *z,
                   int64_t ldz, void *out, int64_t ldo, int *err, cudaStream_t st);
// Grouped forms: G products of M x N x K in one launch (the per-species networks). Output
// groups sit side by side in each row (group g's columns start at g x g_out), except for
// gemm_linear_grouped, whose g_out is any element offset (stacked weight gradients: rows x ldo).
int gemm_gelu_grouped(int bn, const GemmOperand &X, const GemmOperand &W, int G, int M, int N, int K,
                      const float *bias, int64_t g_bias, void *out, int64_t ldo, int64_t g_out, float *pre,
                      int64_t ldp, int64_t g_pre, int *err, cudaStream_t st, int max_ctas = 0);
int gemm_linear_grouped(int bn, const GemmOperand &X, const GemmOperand &W, int G, int M, int N, int K,
                        const float *bias, int64_t g_bias, float *out, int64_t ldo, int64_t g_out, int *err,
                        cudaStream_t st, int max_ctas = 0);
int gemm_gelu_grad_grouped(const GemmOperand &X, const GemmOperand &W, int G, int M, int N, int K, const float *z,
                           int64_t ldz, int64_t g_z, void *out, int64_t ldo, int64_t g_out, int *err, cudaStream_t st);
// Weight and bias gradients of several layers in one launch (gemm_wgrad.cu): gW[o][i] = sum_b dz[b][o] h[b][i]
// for o < out, i < in (FP32, rows of ldg floats), gb[o] = sum_b dz[b][o]. dz [B][ldz] and h [B][ldh] BF16.
struct WgradLayer {
    const void *dz, *h;
    int64_t ldz, ldh;
    int out, in;
    float *gW;
    int64_t ldg;
    float *gb;
};
int gemm_wgrad(const WgradLayer *layers, int count, int B, int *err, cudaStream_t st);
// The last hidden layer and the output layer in one launch, h3 kept on chip (gemm_fused34.cuh):
// u = bf16(GELU(X W3^T + b3)) W4^T + b4 in FP32, bitwise gemm_gelu (layer 3) then gemm_linear
// (layer 4). X [M][ldx] BF16 with K3 columns, W3 [N3][ldw3], W4 [N4][ldw4] (K = N3), u [M][ldu].
bool fused34_supported(int K3, int N3, int N4);
int gemm_fused34(const void *X, int64_t ldx, int K3, const void *W3, int64_t ldw3, const void *W4, int64_t ldw4, int M,
                 int N3, int N4, const float *b3, const float *b4, float *u, int64_t ldu, int *err, cudaStream_t st);
// Reduced-precision hidden layer (EpiGeluQ): f8in selects E4M3 operands (X, W) with the per-column
// scale cs, f8out an E4M3 output scaled by inv_so; otherwise BF16.
int gemm_gelu_q(bool f8in, bool f8out, int bn, const void *X, int64_t ldx, const void *W, int64_t ldw, int M, int N,
                int K, const float *bias, const float *cs, void *out, int64_t ldo, float inv_so, int *err,
                cudaStream_t st, int max_ctas = 0);

}  // namespace chemgb
