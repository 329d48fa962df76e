// props.cu -- props_eval: NASA-7 mixture thermo and mixture-averaged
// transport for every cell (Sec. 2: thermal and transport properties on the
// GPU; Sec. 3.1: Hirschfelder-Curtiss mixture-averaged model).
//
// Three kernels: thermo_kernel (cp and h alone), props_tc_kernel (the full pass
// in FP32, species-pair sums on the tensor cores), and the pair loop below for
// FP64 and for what the tensor-core pass does not take (more than 56 species, or tables
// that FP16 pairs do not hold: 524,288 cells of 9 / 30 species 69 / 389 us in FP32 with the
// instances for 16 and 32 species, 188 / 664 us with the one for 64).
//
// The pair loop: one thread per cell, persistent grid-stride loop. Cell data are SoA, so a
// warp's loads of T, p and each Y_k row are 128-byte coalesced. The per-pair
// tables (Wilke weights, binary-resistance fits) are read with uniform
// addresses (one broadcast per warp) through the read-only cache. The
// per-cell vectors X_j and 1 / r_j (r = sqrt(mu)) live in registers: the inner
// species loop is unrolled to a compile-time bound NMAX.
//
// Wilke: sum_j X_j Phi_kj with Phi_kj = c_kj (1 + w_jk r_k / r_j)^2 is
// evaluated per pair as T0 + t (T1 + t T2), t = r_k / r_j, with constant tables
// T0 = c, T1 = 2 c w, T2 = c w^2 (expanded once at load time): one multiply
// more per pair than three separate sums, for a third fewer registers (which
// bound the kernel's occupancy).
#include <cuda_fp16.h>

#include <cmath>

#include "internal.cuh"
#include "tc.cuh"

namespace chemgb {
namespace {

template <typename real>
__device__ __forceinline__ void load4(const real *p, real &a, real &b, real &c, real &d) {
    if constexpr (sizeof(real) == 4) {
        float4 v = __ldg(reinterpret_cast<const float4 *>(p));
        a = v.x; b = v.y; c = v.z; d = v.w;
    } else {
        double2 v0 = __ldg(reinterpret_cast<const double2 *>(p));
        double2 v1 = __ldg(reinterpret_cast<const double2 *>(p) + 1);
        a = v0.x; b = v0.y; c = v1.x; d = v1.y;
    }
}

// FP32 tables always fit (8 N Np floats <= 131 KB for N <= 64); FP64 tables stay in global memory.
constexpr size_t kPropsSmemMax = (8 * 64 * 64 + 28 * 64) * 4;
template <typename real>
__host__ __device__ constexpr bool tables_in_smem() { return sizeof(real) == 4; }

// Copies the per-pair tables (3 Wilke + 5 resistance rows per species) into
// shared memory when they fit; the inner loops then read them with broadcast
// LDS.128 instead of uniform global loads.
template <typename real>
__device__ __forceinline__ void stage_pair_tables(const PropTables<real> &tb, int N, int Np, real *sh) {
    const int nw = 3 * N * Np, nd = 5 * N * Np;
    for (int e = threadIdx.x; e < nw; e += blockDim.x) sh[e] = tb.wilke[e];
    for (int e = threadIdx.x; e < nd; e += blockDim.x) sh[nw + e] = tb.diff[e];
    __syncthreads();
}

// Per-species coefficient rows (NASA cp and h of both ranges, the ln(mu) fit, 1/W) in
// the global tables' own layout, copied to shared memory after the pair tables so
// that the species loops read them as broadcasts.
constexpr int kSpeciesFloats = 2 * 5 + 2 * 6 + 5 + 1;   // floats per species
template <typename real>
__device__ __forceinline__ void stage_species_tables(const PropTables<real> &tb, int N, real *sh) {
    for (int e = threadIdx.x; e < 10 * N; e += blockDim.x) sh[e] = tb.nasa_cp[e];
    for (int e = threadIdx.x; e < 12 * N; e += blockDim.x) sh[10 * N + e] = tb.nasa_h[e];
    for (int e = threadIdx.x; e < 5 * N; e += blockDim.x) sh[22 * N + e] = tb.visc[e];
    for (int e = threadIdx.x; e < N; e += blockDim.x) sh[27 * N + e] = tb.invW[e];
    __syncthreads();
}

template <typename real>
__device__ __forceinline__ void load4s(const real *p, real &a, real &b, real &c, real &d) {
    if constexpr (sizeof(real) == 4) {
        const float4 v = *reinterpret_cast<const float4 *>(p);
        a = v.x; b = v.y; c = v.z; d = v.w;
    } else {
        const double2 v0 = reinterpret_cast<const double2 *>(p)[0];
        const double2 v1 = reinterpret_cast<const double2 *>(p)[1];
        a = v0.x; b = v0.y; c = v1.x; d = v1.y;
    }
}

// state value -> working precision; FP64 -> FP32 on the integer pipe (truncation, < 2^-23 relative)
template <typename real, typename in_t>
__device__ __forceinline__ real to_real(in_t x) {
    if constexpr (sizeof(real) == 4 && sizeof(in_t) == 8) return f64_to_f32_trunc(x);
    else return real(x);
}

// Species k is all there is (1 - X_k < 1e-12): D_k is then the mean binary value. FP32 holds an X_k
// within 3e-8 of 1 as 1, so there the traces' own sum ds (mean resistance gs / (N - 1)) decides, unless
// 1 - Y_k is lost as well.
template <typename real>
__device__ __forceinline__ bool pure_species(real Xk, real y, real ds, real gs, int N) {
    if (!(real(1) - Xk < real(1e-12))) return false;
    return sizeof(real) == 8 || y >= real(1) || ds * real(N - 1) <= real(1e-12) * gs;
}

template <typename real, typename in_t, int NMAX>
__global__ void __launch_bounds__(128, sizeof(real) == 4 && NMAX <= 32 ? 4 : 1) props_kernel(int N, int Np, real T_mid, PropTables<real> tb, int64_t ncells,
                                                    int64_t ld, const in_t *__restrict__ Tg,
                                                    const in_t *__restrict__ pg, const in_t *__restrict__ Yg,
                                                    real *__restrict__ cpg, real *__restrict__ hg,
                                                    real *__restrict__ mug, real *__restrict__ lamg,
                                                    real *__restrict__ Dkg) {
    const real R = real(kR);
    const bool transport = (mug != nullptr) || (lamg != nullptr) || (Dkg != nullptr);
    extern __shared__ __align__(16) unsigned char props_smem[];
    real *shtab = reinterpret_cast<real *>(props_smem);
    constexpr bool in_smem = tables_in_smem<real>();
    if (in_smem && transport) stage_pair_tables(tb, N, Np, shtab);
    real *sp = shtab + (transport ? 8 * N * Np : 0);
    if (in_smem) stage_species_tables(tb, N, sp);
    const real *wil = in_smem ? shtab : tb.wilke;
    const real *dif = in_smem ? shtab + 3 * N * Np : tb.diff;
    const real *t_cp = in_smem ? sp : tb.nasa_cp;
    const real *t_h = in_smem ? sp + 10 * N : tb.nasa_h;
    const real *t_visc = in_smem ? sp + 22 * N : tb.visc;
    const real *t_iw = in_smem ? sp + 27 * N : tb.invW;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ncells; i += stride) {
        const real T = to_real<real>(Tg[i]);
        const real p = to_real<real>(pg[i]);
        const int rng = (T >= T_mid) ? 1 : 0;
        const real iT = real(1) / T;
        const real x = log(T) - real(6.907755278982137);   // ln(T / 1000)
        real S = 0, cpm = 0, hm = 0;
        real X[NMAX], ir[NMAX];
        // pass 1: thermo sums; keep Y_k / W_k
#pragma unroll
        for (int k = 0; k < NMAX; ++k) {
            if (k < N) {
                const real y = to_real<real>(Yg[(int64_t)k * ld + i]);
                const real iw = t_iw[k];
                const real *a = t_cp + (rng * N + k) * 5;
                const real *b = t_h + (rng * N + k) * 6;
                real cpR = a[4];
                cpR = fma(cpR, T, a[3]);
                cpR = fma(cpR, T, a[2]);
                cpR = fma(cpR, T, a[1]);
                cpR = fma(cpR, T, a[0]);
                real hR = b[4];
                hR = fma(hR, T, b[3]);
                hR = fma(hR, T, b[2]);
                hR = fma(hR, T, b[1]);
                hR = fma(hR, T, b[0]);
                hR = fma(b[5], iT, hR);                          // H_k / (R T)
                const real yw = y * iw;
                S += yw;
                cpm = fma(yw, cpR, cpm);
                hm = fma(yw, hR, hm);
                X[k] = yw;
            } else {
                X[k] = 0;
            }
        }
        if (cpg) cpg[i] = cpm * R;
        if (hg) hg[i] = hm * R * T;
        if (!transport) continue;
        const real Wbar = real(1) / S;
#pragma unroll
        for (int k = 0; k < NMAX; ++k) {
            if (k < N) {
                const real *c = t_visc + k * 5;
                real lm = c[4];
                lm = fma(lm, x, c[3]);
                lm = fma(lm, x, c[2]);
                lm = fma(lm, x, c[1]);
                lm = fma(lm, x, c[0]);
                ir[k] = exp(real(-0.5) * lm);                      // 1 / sqrt(mu_k)
                X[k] = X[k] * Wbar;
            } else {
                ir[k] = 0;
            }
        }
        const real T15 = T * sqrt(T);
        real mu = 0, lam = 0;
        real y_next = to_real<real>(Yg[i]);
        for (int k = 0; k < N; ++k) {
            // per-species values, recomputed from the tables (no dynamic register indexing);
            // the next species' mass fraction is loaded one iteration ahead
            const real y = y_next;
            if (k + 1 < N) y_next = to_real<real>(Yg[(int64_t)(k + 1) * ld + i]);
            const real iw = t_iw[k];
            const real Xk = y * iw * Wbar;
            const real *c = t_visc + k * 5;
            real lm = c[4];
            lm = fma(lm, x, c[3]);
            lm = fma(lm, x, c[2]);
            lm = fma(lm, x, c[1]);
            lm = fma(lm, x, c[0]);
            const real muk = exp(lm);
            const real rk = sqrt(muk);
            const real *a = t_cp + (rng * N + k) * 5;
            real cpR = a[4];
            cpR = fma(cpR, T, a[3]);
            cpR = fma(cpR, T, a[2]);
            cpR = fma(cpR, T, a[1]);
            cpR = fma(cpR, T, a[0]);
            const real lamk = muk * (cpR + real(1.25)) * R * iw;   // Eucken
            const real *t0 = wil + (0 * N + k) * Np;
            const real *t1 = wil + (1 * N + k) * Np;
            const real *t2 = wil + (2 * N + k) * Np;
            const real *d0 = dif + (0 * N + k) * Np;
            const real *d1 = dif + (1 * N + k) * Np;
            const real *d2 = dif + (2 * N + k) * Np;
            const real *d3 = dif + (3 * N + k) * Np;
            const real *d4 = dif + (4 * N + k) * Np;
            real a0 = 0, ds = 0, gs = 0;
            [[maybe_unused]] uint64_t a02 = 0, ds2 = 0, gs2 = 0;       // FP32: (even j, odd j) sums
            [[maybe_unused]] const uint64_t rk2 = sizeof(real) == 4 ? pk2(float(rk), float(rk)) : 0;
            [[maybe_unused]] const uint64_t x2 = sizeof(real) == 4 ? pk2(float(x), float(x)) : 0;
#pragma unroll
            for (int j4 = 0; j4 < NMAX; j4 += 4) {
                if (j4 < N) {
                    real w0[4], w1[4], w2[4], g0[4], g1[4], g2[4], g3[4], g4[4];
                    if constexpr (in_smem) {
                        load4s(t0 + j4, w0[0], w0[1], w0[2], w0[3]);
                        load4s(t1 + j4, w1[0], w1[1], w1[2], w1[3]);
                        load4s(t2 + j4, w2[0], w2[1], w2[2], w2[3]);
                        load4s(d0 + j4, g0[0], g0[1], g0[2], g0[3]);
                        load4s(d1 + j4, g1[0], g1[1], g1[2], g1[3]);
                        load4s(d2 + j4, g2[0], g2[1], g2[2], g2[3]);
                        load4s(d3 + j4, g3[0], g3[1], g3[2], g3[3]);
                        load4s(d4 + j4, g4[0], g4[1], g4[2], g4[3]);
                    } else {
                        load4(t0 + j4, w0[0], w0[1], w0[2], w0[3]);
                        load4(t1 + j4, w1[0], w1[1], w1[2], w1[3]);
                        load4(t2 + j4, w2[0], w2[1], w2[2], w2[3]);
                        load4(d0 + j4, g0[0], g0[1], g0[2], g0[3]);
                        load4(d1 + j4, g1[0], g1[1], g1[2], g1[3]);
                        load4(d2 + j4, g2[0], g2[1], g2[2], g2[3]);
                        load4(d3 + j4, g3[0], g3[1], g3[2], g3[3]);
                        load4(d4 + j4, g4[0], g4[1], g4[2], g4[3]);
                    }
                    if constexpr (sizeof(real) == 4) {
                        // two species j at a time on the packed FP32x2 pipe (even and odd j summed
                        // apart, joined after the loop)
#pragma unroll
                        for (int u = 0; u < 4; u += 2) {
                            const int j = j4 + u;   // padded columns have zero weights
                            // Phi_kj = T0 + t (T1 + t T2) with t = r_k / r_j
                            const uint64_t t = mul2(pk2(ir[j], ir[j + 1]), rk2);
                            const uint64_t phi =
                                fma2(t, fma2(t, pk2(w2[u], w2[u + 1]), pk2(w1[u], w1[u + 1])), pk2(w0[u], w0[u + 1]));
                            const uint64_t Xj = pk2(X[j], X[j + 1]);
                            a02 = fma2(phi, Xj, a02);
                            uint64_t g = fma2(pk2(g4[u], g4[u + 1]), x2, pk2(g3[u], g3[u + 1]));
                            g = fma2(g, x2, pk2(g2[u], g2[u + 1]));
                            g = fma2(g, x2, pk2(g1[u], g1[u + 1]));
                            g = fma2(g, x2, pk2(g0[u], g0[u + 1]));
                            ds2 = fma2(g, Xj, ds2);
                            gs2 = add2(gs2, g);
                        }
                    } else {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int j = j4 + u;   // padded columns have zero weights
                            // Phi_kj = T0 + t (T1 + t T2) with t = r_k / r_j
                            const real t = ir[j] * rk;
                            a0 = fma(fma(t, fma(t, w2[u], w1[u]), w0[u]), X[j], a0);
                            real g = fma(fma(fma(fma(g4[u], x, g3[u]), x, g2[u]), x, g1[u]), x, g0[u]);
                            ds = fma(g, X[j], ds);
                            gs += g;
                        }
                    }
                }
            }
            if constexpr (sizeof(real) == 4) {
                float e, o;
                upk2(a02, e, o);
                a0 = e + o;
                upk2(ds2, e, o);
                ds = e + o;
                upk2(gs2, e, o);
                gs = e + o;
            }
            const real den = a0;
            mu = fma(Xk, muk / den, mu);
            lam = fma(Xk, lamk / den, lam);
            if (Dkg) {
                real D;
                if (pure_species(Xk, y, ds, gs, N)) D = T15 / (p * gs / real(N - 1));
                else D = (real(1) - y) * T15 / (p * ds);
                Dkg[(int64_t)k * ld + i] = D;
            }
        }
        if (mug) mug[i] = mu;
        if (lamg) lamg[i] = lam;
    }
}

// The same in FP64 with G threads per cell (G lanes of a warp, species k = lane, lane + G, ...), for calls
// whose cells do not fill the chip with a thread each: FP64 issues one warp instruction per 64 clocks and
// SM sub-partition, so 4,096 cells of 9 species on 32 of the SMs took 80 us, a serial chain of about 1,800
// such instructions, and take 33 us spread over all of them. Per species one exponential (r = sqrt(mu), mu =
// r^2) and two divisions; X_j enters the sums as Y_j / W_j and 1 / Wbar cancels in mu and lambda. Beyond
// kSplitWarps warps per SM the loop above does less work per cell (its scalars serve 32 cells a
// warp).
constexpr int kSplitWarps = 4;
template <int G>
__global__ void __launch_bounds__(128)
    props_split_kernel(int N, int Np, double T_mid, PropTables<double> tb, int64_t ncells, int64_t ld,
                       const double *__restrict__ Tg, const double *__restrict__ pg, const double *__restrict__ Yg,
                       double *__restrict__ cpg, double *__restrict__ hg, double *__restrict__ mug,
                       double *__restrict__ lamg, double *__restrict__ Dkg) {
    extern __shared__ double split_smem[];                    // [128 / G][3][N]: Y / W, r, 1 / r
    const int l = threadIdx.x & (G - 1), slot = threadIdx.x / G;
    const int64_t cell = (int64_t)blockIdx.x * (128 / G) + slot;
    const bool valid = cell < ncells;
    const int64_t i = valid ? cell : ncells - 1;
    const bool transport = (mug != nullptr) || (lamg != nullptr) || (Dkg != nullptr);
    double *xs = split_smem + (size_t)slot * 3 * N, *rs = xs + N, *is = rs + N;
    auto group_sum = [](double v) {
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
    const double T = Tg[i], p = pg[i];
    const int rng = (T >= T_mid) ? 1 : 0;
    const double iT = 1.0 / T;
    const double x = log(T) - 6.907755278982137;              // ln(T / 1000)
    double S = 0.0, cpm = 0.0, hm = 0.0;
    for (int k = l; k < N; k += G) {
        const double *a = tb.nasa_cp + (rng * N + k) * 5, *b = tb.nasa_h + (rng * N + k) * 6, *c = tb.visc + k * 5;
        const double yw = Yg[(int64_t)k * ld + i] * __ldg(tb.invW + k);
        const double cpR = fma(fma(fma(fma(__ldg(a + 4), T, __ldg(a + 3)), T, __ldg(a + 2)), T, __ldg(a + 1)), T, __ldg(a));
        double hR = fma(fma(fma(fma(__ldg(b + 4), T, __ldg(b + 3)), T, __ldg(b + 2)), T, __ldg(b + 1)), T, __ldg(b));
        hR = fma(__ldg(b + 5), iT, hR);                       // H_k / (R T)
        S += yw;
        cpm = fma(yw, cpR, cpm);
        hm = fma(yw, hR, hm);
        if (transport) {
            const double lm = fma(fma(fma(fma(__ldg(c + 4), x, __ldg(c + 3)), x, __ldg(c + 2)), x, __ldg(c + 1)), x, __ldg(c));
            const double r = exp(0.5 * lm);
            xs[k] = yw;
            rs[k] = r;
            is[k] = 1.0 / r;
        }
    }
    S = group_sum(S);
    cpm = group_sum(cpm);
    hm = group_sum(hm);
    if (l == 0 && valid) {
        if (cpg) cpg[i] = cpm * kR;
        if (hg) hg[i] = hm * kR * T;
    }
    if (!transport) return;
    __syncwarp();                                             // a cell's threads are one warp's
    const double Wbar = 1.0 / S;
    const double T15 = T * sqrt(T);
    double mu = 0.0, lam = 0.0;
    for (int k = l; k < N; k += G) {
        const double rk = rs[k];
        const double2 *t0 = reinterpret_cast<const double2 *>(tb.wilke + (size_t)k * Np);
        const double2 *d0 = reinterpret_cast<const double2 *>(tb.diff + (size_t)k * Np);
        const size_t s2 = (size_t)N * Np / 2;
        double den = 0.0, ds = 0.0, gs = 0.0;
        for (int j = 0; j < N; j += 2) {                      // tables are padded with zeros to Np
            const double2 w0 = __ldg(t0 + j / 2), w1 = __ldg(t0 + s2 + j / 2), w2 = __ldg(t0 + 2 * s2 + j / 2);
            const double2 g0 = __ldg(d0 + j / 2), g1 = __ldg(d0 + s2 + j / 2), g2 = __ldg(d0 + 2 * s2 + j / 2),
                          g3 = __ldg(d0 + 3 * s2 + j / 2), g4 = __ldg(d0 + 4 * s2 + j / 2);
            const double xa = xs[j], ta = rk * is[j];
            den = fma(fma(ta, fma(ta, w2.x, w1.x), w0.x), xa, den);
            const double ga = fma(fma(fma(fma(g4.x, x, g3.x), x, g2.x), x, g1.x), x, g0.x);
            ds = fma(ga, xa, ds);
            gs += ga;
            if (j + 1 < N) {
                const double xb = xs[j + 1], tb2 = rk * is[j + 1];
                den = fma(fma(tb2, fma(tb2, w2.y, w1.y), w0.y), xb, den);
                const double gb = fma(fma(fma(fma(g4.y, x, g3.y), x, g2.y), x, g1.y), x, g0.y);
                ds = fma(gb, xb, ds);
                gs += gb;
            }
        }
        const double *a = tb.nasa_cp + (rng * N + k) * 5;
        const double cpR = fma(fma(fma(fma(__ldg(a + 4), T, __ldg(a + 3)), T, __ldg(a + 2)), T, __ldg(a + 1)), T, __ldg(a));
        const double wk = xs[k] / den * (rk * rk);            // X_k mu_k / sum_j X_j Phi_kj
        mu += wk;
        lam = fma(wk, (cpR + 1.25) * kR * __ldg(tb.invW + k), lam);   // Eucken
        if (Dkg && valid) {
            const double y = Yg[(int64_t)k * ld + i], Xk = xs[k] * Wbar;
            ds *= Wbar;
            Dkg[(int64_t)k * ld + i] = pure_species(Xk, y, ds, gs, N) ? T15 / (p * gs / double(N - 1)) : (1.0 - y) * T15 / (p * ds);
        }
    }
    mu = group_sum(mu);
    lam = group_sum(lam);
    if (l == 0 && valid) {
        if (mug) mug[i] = mu;
        if (lamg) lamg[i] = lam;
    }
}

template <int G>
int launch_props_split(const chem_mech *m, int64_t ncells, int64_t ld, const void *T, const void *p, const void *Y,
                       void *cp, void *h, void *mu, void *lam, void *Dk, cudaStream_t st) {
    const int per = 128 / G;
    void *pb = prof_begin(st);
    props_split_kernel<G><<<(unsigned)((ncells + per - 1) / per), 128, (size_t)per * 3 * m->N * sizeof(double), st>>>(
        m->N, m->dev.Np, m->T_mid, m->dev.f64, ncells, ld, static_cast<const double *>(T), static_cast<const double *>(p),
        static_cast<const double *>(Y), static_cast<double *>(cp), static_cast<double *>(h), static_cast<double *>(mu),
        static_cast<double *>(lam), static_cast<double *>(Dk));
    prof_end(pb, st, "props_kernel<f64>", (double)ncells * (16.0 * m->N * m->N + 30.0 * m->N),
             (double)ncells * ((m->N + 2) * 8 + (4 + m->N) * 8));
    return check_cuda(cudaGetLastError(), "props_eval launch");
}

// Thermo only (cp and h; the memory-bound part of props_eval), FP32 arithmetic,
// with the state staged through shared memory by bulk copies.
//
// A CTA (one per SM) takes tiles of kThTile consecutive cells. The tile's state
// rows (T, then Y_0 .. Y_{N-1}) arrive in groups of kThRows rows, one 1-D bulk
// copy (cp.async.bulk) per row segment, into a ring of stages: a producer warp
// keeps up to kStages groups in flight (about 190 KB per SM for FP64 state, far
// more bytes than the HBM latency needs), while kThTile consumer threads, one
// per cell, read their column of each landed group, accumulate cp and h and
// release the stage. Row segments are read once and in whole 16-byte units: a
// tile's last segment is rounded up to 4 cells, which stays inside ld (a
// multiple of 4). The NASA-7 rows of both ranges and 1/W sit in shared memory (3
// float4 per species and range). The arithmetic and the species order per cell
// are those of props_kernel's first pass, so cp and h are bitwise the full
// pass's. A copy wait that runs out (bounded, spin tries) records
// kPropsErrCounter and writes NaN to cp and h of the tile and of every tile the CTA had
// still to do; the CTA ends after its issued copies have landed.
constexpr int kThTile = 512;                  // cells per tile = consumer threads
constexpr int kThRows = 8;                    // state rows per stage
constexpr int kThThreads = kThTile + 32;      // + the producer warp

template <typename in_t>
struct ThLayout {
    static constexpr int kStages = sizeof(in_t) == 8 ? 6 : 8;
    static constexpr uint32_t kRowBytes = kThTile * sizeof(in_t);
    static constexpr uint32_t kStage = kThRows * kRowBytes;
    static constexpr uint32_t kStageTotal = kStages * kStage;
    static size_t bytes(int N) { return kStageTotal + (size_t)6 * N * sizeof(float4) + 2 * kStages * 8; }
};

template <typename in_t>
__global__ void __launch_bounds__(kThThreads, 1)
    thermo_kernel(int N, float T_mid, PropTables<float> tb, int64_t ncells, int64_t ld,
                  const in_t *__restrict__ Tg, const in_t *__restrict__ Yg, float *__restrict__ cpg,
                  float *__restrict__ hg, unsigned int *err, uint32_t spin) {
    using L = ThLayout<in_t>;
    constexpr int S = L::kStages;
    extern __shared__ __align__(128) uint8_t th_smem[];
    uint8_t *stages = th_smem;
    float4 *tab = reinterpret_cast<float4 *>(th_smem + L::kStageTotal);
    uint64_t *full = reinterpret_cast<uint64_t *>(tab + 6 * N);
    uint64_t *empty = full + S;
    for (int e = threadIdx.x; e < 2 * N; e += blockDim.x) {
        const int rg = e / N, k = e % N;
        const float *a = tb.nasa_cp + (rg * N + k) * 5;
        const float *b = tb.nasa_h + (rg * N + k) * 6;
        tab[e * 3 + 0] = make_float4(a[0], a[1], a[2], a[3]);
        tab[e * 3 + 1] = make_float4(a[4], b[0], b[1], b[2]);
        tab[e * 3 + 2] = make_float4(b[3], b[4], b[5], tb.invW[k]);
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], kThTile / 32);
        }
        tc::fence_barrier_init();
    }
    __syncthreads();
    const int64_t ntiles = (ncells + kThTile - 1) / kThTile;
    const int groups = (N + 1 + kThRows - 1) / kThRows;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == kThTile / 32) {
        if (lane == 0) {
            int u = 0;
            bool ok = true;
            for (int64_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                const int64_t c0 = t * kThTile;
                const int64_t cells = ncells - c0 < kThTile ? ncells - c0 : kThTile;
                const uint32_t bytes = (uint32_t)(((cells + 3) & ~int64_t(3)) * sizeof(in_t));
                for (int g = 0; g < groups; ++g, ++u) {
                    const int s = u % S;
                    if (!tc::mbar_wait(&empty[s], (uint32_t)((u / S) & 1) ^ 1u, spin)) {
                        atomicExch(err, 1u);
                        ok = false;
                        break;
                    }
                    const int r0 = g * kThRows, rows = (N + 1 - r0) < kThRows ? N + 1 - r0 : kThRows;
                    tc::mbar_arrive_expect_tx(&full[s], rows * bytes);
                    for (int r = 0; r < rows; ++r) {
                        const int q = r0 + r;          // state row: 0 = T, q = Y_{q-1}
                        const in_t *src = (q == 0 ? Tg : Yg + (int64_t)(q - 1) * ld) + c0;
                        tc::bulk_load_1d(stages + s * L::kStage + r * L::kRowBytes, src, bytes, &full[s]);
                    }
                }
            }
            // the last fill of each stage lands before the CTA may exit (full limit); u counts the
            // groups whose copies were issued
            for (int j = (u > S ? u - S : 0); j < u; ++j)
                if (!tc::mbar_wait(&full[j % S], (uint32_t)(j / S) & 1u)) {
                    atomicExch(err, 1u);
                    break;
                }
        }
        return;
    }
    const float R = float(kR);
    int u = 0;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t i = t * kThTile + threadIdx.x;
        float T = 300.0f, iT = 1.0f / 300.0f, cpm = 0.0f, hm = 0.0f;
        const float4 *tr = tab;
        bool ok = true;
        for (int g = 0; g < groups; ++g, ++u) {
            const int s = u % S;
            if (!__all_sync(0xffffffffu, tc::mbar_wait(&full[s], (uint32_t)(u / S) & 1u, spin))) {
                ok = false;
                break;
            }
            const in_t *col = reinterpret_cast<const in_t *>(stages + s * L::kStage) + threadIdx.x;
            const int r0 = g * kThRows;
#pragma unroll
            for (int r = 0; r < kThRows; ++r) {
                const int q = r0 + r;
                if (q > N) break;
                const float v = to_real<float>(col[r * kThTile]);
                if (q == 0) {
                    T = v;
                    iT = 1.0f / T;
                    tr = tab + ((T >= T_mid) ? 3 * N : 0);
                    continue;
                }
                const int k = q - 1;
                const float4 q0 = tr[3 * k], q1 = tr[3 * k + 1], q2 = tr[3 * k + 2];
                float cpR = q1.x;
                cpR = fmaf(cpR, T, q0.w);
                cpR = fmaf(cpR, T, q0.z);
                cpR = fmaf(cpR, T, q0.y);
                cpR = fmaf(cpR, T, q0.x);
                float hR = q2.y;
                hR = fmaf(hR, T, q2.x);
                hR = fmaf(hR, T, q1.w);
                hR = fmaf(hR, T, q1.z);
                hR = fmaf(hR, T, q1.y);
                hR = fmaf(q2.z, iT, hR);
                const float yw = v * q2.w;
                cpm = fmaf(yw, cpR, cpm);
                hm = fmaf(yw, hR, hm);
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&empty[s]);
        }
        if (!ok) {
            if (lane == 0) atomicExch(err, 1u);
            for (int64_t q = i; q < ncells; q += (int64_t)gridDim.x * kThTile) {
                if (cpg) cpg[q] = __int_as_float(0x7fc00000);
                if (hg) hg[q] = __int_as_float(0x7fc00000);
            }
            break;
        }
        if (i < ncells) {
            if (cpg) __stcs(cpg + i, cpm * R);
            if (hg) __stcs(hg + i, hm * R * T);
        }
    }
}

template <typename in_t>
int launch_thermo(const chem_mech *m, int64_t ncells, int64_t ld, const void *T, const void *Y, void *cp, void *h,
                  cudaStream_t st) {
    using L = ThLayout<in_t>;
    if (!aligned16(T) || !aligned16(Y) || (ld & 3) != 0)
        return set_error(CHEM_EINVAL, "props_eval: the state arrays must be 16-byte aligned and ld a multiple of 4");
    const size_t smem = L::bytes(m->N);
    static DeviceOnce configured;
    if (int rc = dynamic_smem_limit(configured, thermo_kernel<in_t>, L::bytes(kMaxSpecies),
                                    "props_eval (thermo) smem attribute"))
        return rc;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t ntiles = (ncells + kThTile - 1) / kThTile;
    const int blocks = (int)(ntiles < sms ? ntiles : sms);
    void *pb = prof_begin(st);
    thermo_kernel<in_t><<<blocks, kThThreads, smem, st>>>(m->N, float(m->T_mid), m->dev.f32, ncells, ld,
                                                          static_cast<const in_t *>(T), static_cast<const in_t *>(Y),
                                                          static_cast<float *>(cp), static_cast<float *>(h),
                                                          m->dev.counters + kPropsErrCounter, m->wait_limit);
    prof_end(pb, st, "thermo_kernel", (double)ncells * 24.0 * m->N,
             (double)ncells * ((m->N + 1) * sizeof(in_t) + 2 * sizeof(float)));
    return check_cuda(cudaGetLastError(), "props_eval (thermo) launch");
}

// ---- the full pass in FP32, with the species-pair sums on the tensor cores ------------------
//
// Per cell and species k the transport needs sum_j X_j Phi_kj and sum_j X_j g_kj. With
// Phi_kj = T0_kj + t (T1_kj + t T2_kj), t = r_k / r_j, and g_kj = sum_n d_n,kj x^n these are
//   T0 X + r_k (T1 (X / r) + r_k T2 (X / r^2))      and      sum_n x^n (D_n X):
// eight products of constant N x N tables with three per-cell vectors, a contraction. A tile of
// 128 cells is the M of tcgen05.mma (kind::f16), the tables' rows are its N (2 NR + 6 NP columns of
// TMEM: 256 for 30 species, 464 for 53) and the species j its K.
//
// Precision: both factors are pairs of FP16 terms, hi = fp16(v) and lo = fp16(v - hi), 22 bits, and
// three products hi hi + lo hi + hi lo are accumulated in FP32. To stay clear of FP16's small range
// 1/r is divided by the power of two at the cell's largest 1/r (r_k is multiplied by it), every
// vector entry is then at most 1 in magnitude and scaled by 2^14, and the tables' rows by powers of
// two (PropTcTables). What is left of absolute error, 2^-39 of a mole fraction, only shows in D_k of
// a species that is nearly alone (its sum runs over traces): for X_k > 0.999 that sum is taken in FP32
// from the FP32 tables (near_pure_D), and a cell with |X_k| >= 4 (mass fractions of both signs), past FP16's
// range, is redone in FP32 as a whole (wide_cell). The tensor core cuts its accumulator instead of rounding it:
// a sum loses 0.4e-7 of itself (0.6e-7 as mu and lambda show it) in the instruction that takes a species in and
// 1.8 to 2.4e-7 in each K step after that, so how much depends on where in the species' order a cell has its
// moles. The mean is given back per cell (`cut`), with the mole fraction of each K step as its share of every sum.
// Mean signed errors of mu / D without it, with one constant per step count, and so (60,000 cells, FP32 state):
//   30 species, premixed profiles              2.8e-7 / 2.7e-7    0.1e-7 /  0.0e-7    0.1e-7 /  0.0e-7
//   53 species, premixed profiles              5.8e-7 / 5.6e-7    0.4e-7 /  0.0e-7   -0.2e-7 /  0.0e-7
//   53 species, X spread by a Dirichlet law    2.8e-7 / 2.5e-7   -2.6e-7 / -3.1e-7   -1.7e-7 / -1.7e-7
//   53 species, three quarters of Y the last   1.3e-7 / 1.1e-7   -4.0e-7 / -4.5e-7   -0.6e-7 / -0.6e-7
//   40 species (3 steps), same of the first    3.7e-7 / 3.3e-7   -0.5e-7 / -0.9e-7   -0.5e-7 / -0.7e-7
//   9 species, Dirichlet law                   0.8e-7 / 0.5e-7   -0.1e-7 /  0.1e-7   -0.1e-7 /  0.1e-7
// (The resistance polynomials' sums have both signs, and lose the same within 0.5e-7.) r_k = 2^(polynomial) is formed with
// the whole part of its exponent taken out at load time. Relative errors against 64 bits (2-norm, 100,003
// cells, FP32 state; the former pair loop -> this kernel): 30 species mu 3.6e-7 -> 1.2e-7, lambda 3.2e-7 ->
// 1.1e-7, D 2.0e-7 -> 1.6e-7; 53 species 3.2e-7 -> 1.3e-7, 3.1e-7 -> 1.2e-7, 2.4e-7 -> 1.8e-7; 9 species
// 2.4e-7 -> 0.9e-7, 2.7e-7 -> 1.0e-7, 1.1e-7 -> 1.1e-7.
//
// What bounds it: instruction issue (51 % of the slots) and its latencies for the per-species FP32
// work that is left; the tensor cores are busy a few per cent of the time, HBM 10 %. The pair loop (10
// instructions a pair, tables from shared memory) took 1,580 us on 2,097,152 cells of 30 species from
// FP64 state and 799 us on 300,001 of 53 from FP32; this kernel takes 629 and 188 us.
//
// Layout: a thread per cell and chunk of eight species (2, 4 or 8 threads a cell for up to 16, 32 or
// 56 species: 256 to 1,024 threads, 64 registers; two threads a cell with twice the species each
// and 128 registers left half the warps and took 792 us). Each thread turns its species into operand
// entries (no-swizzle K-major core matrices, [chunk][row][16 bytes]: a warp's 16-byte stores are
// consecutive) and later finishes the same species from TMEM. cp and h are summed over all species in
// ascending order by one thread each while the tensor cores work, with thermo_kernel's operations, so
// they are bitwise its results.
struct TcArgs {
    int N;
    float T_mid;
    PropTables<float> tb;
    PropTcTables tc;
    int64_t ncells, ld;
    float *cp, *h, *mu, *lam, *Dk;
    unsigned int *err;
    uint32_t spin;
};

template <int NMAX>
struct TcLayout {
    static constexpr int kChunks = NMAX / 8;                    // chunks of 8 species
    static constexpr int kTPR = kChunks;                        // threads per cell, a chunk each
    static constexpr int kThreads = 128 * kTPR;
    static constexpr int kCtas = NMAX <= 16 ? 4 : (NMAX <= 32 ? 2 : 1);   // resident per SM
    static constexpr bool kStageY = NMAX <= 32;                 // mass fractions in FP32 kept in shared memory
    static constexpr uint32_t kABytes = 6 * kChunks * 2048;     // 3 vectors x 2 terms x [chunk][128][16 B]
    static constexpr uint32_t kYBytes = kStageY ? NMAX * 128 * 4 : 0;
    static constexpr int kPad = NMAX < kTcMaxSpecies ? NMAX : kTcMaxSpecies;   // species of the padded tables
    static constexpr int kRedRows = NMAX <= 32 ? 4 : 2;         // sums between a cell's threads (two pairs, or one reused)
    static constexpr int kShares = kPad / 8;                    // threads of a cell that hold species
    static constexpr uint32_t kRed = kRedRows * kShares * 128 * 4;
    static constexpr bool kEuk = NMAX <= 32;                    // conductivity rows of their own
    static constexpr uint32_t kTab = (kPad * (6 + 2 + (kEuk ? 4 : 0)) + 2) * 16;   // species tables (float4 each)
    static size_t bytes(int rows) { return (size_t)kABytes + 2 * kChunks * rows * 16 + kYBytes + kTab + kRed + 32; }
};

// 2 columns of each of 8 TMEM addresses, 32 lanes; one wait. v[2 a + u] = column u of address a.
__device__ __forceinline__ void tmem_ld8x2(const uint32_t (&a)[8], float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%16];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%2, %3}, [%17];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%4, %5}, [%18];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%6, %7}, [%19];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%8, %9}, [%20];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%10, %11}, [%21];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%12, %13}, [%22];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%14, %15}, [%23];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7])
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// D_k of a species that is nearly alone (X_k > 0.999), the sums over the traces in FP32
template <typename in_t>
__device__ __noinline__ float near_pure_D(const PropTables<float> &tb, int N, int Np, int k, int64_t ld, int64_t i,
                                          const in_t *__restrict__ Yg, float Wbar, float x, float y, float Xk,
                                          float T15, float p) {
    float ds = 0.0f, gs = 0.0f;
    for (int j = 0; j < N; ++j) {
        const float Xj = to_real<float>(Yg[(int64_t)j * ld + i]) * __ldg(tb.invW + j) * Wbar;
        float g = 0.0f;
        for (int n = 4; n >= 0; --n) g = fmaf(g, x, __ldg(tb.diff + ((size_t)n * N + k) * Np + j));
        ds = fmaf(g, Xj, ds);
        gs += g;
    }
    if (pure_species(Xk, y, ds, gs, N)) return T15 / (p * gs / float(N - 1));
    return (1.0f - y) * T15 / (p * ds);
}

// Transport of cell i where the tensor-core sums are not finite although the state is: mole fractions that FP16 does
// not hold (|X_k| >= 4, from mass fractions of both signs). The pair loop's sums in FP32, by one thread.
template <typename in_t>
__device__ __forceinline__ void wide_cell(const TcArgs &g, const in_t *__restrict__ Tg, const in_t *__restrict__ pg,
                                       const in_t *__restrict__ Yg, int64_t i) {
    const PropTables<float> &tb = g.tb;
    const int N = g.N, Np = (N + 3) & ~3;
    const int64_t ld = g.ld;
    const float out = g.mu ? g.mu[i] : (g.lam ? g.lam[i] : g.Dk[i]);
    if (fabsf(out) < INFINITY) return;
    const float T = to_real<float>(Tg[i]), p = to_real<float>(pg[i]), x = logf(T * 1e-3f);
    float S = 0.0f;
    for (int k = 0; k < N; ++k) S = fmaf(to_real<float>(Yg[(int64_t)k * ld + i]), __ldg(tb.invW + k), S);
    if (!(fabsf(S) < INFINITY && fabsf(x) < INFINITY)) return;
    const float Wbar = 1.0f / S;
    const int rng = (T >= g.T_mid) ? 1 : 0;
    float *mug = g.mu, *lamg = g.lam, *Dkg = g.Dk;
    const float T15 = T * sqrtf(T), R = float(kR);
    auto log_mu = [&](int k) {
        const float *c = tb.visc + k * 5;
        return fmaf(fmaf(fmaf(fmaf(__ldg(c + 4), x, __ldg(c + 3)), x, __ldg(c + 2)), x, __ldg(c + 1)), x, __ldg(c));
    };
    float mu = 0.0f, lam = 0.0f;
    for (int k = 0; k < N; ++k) {
        const float y = to_real<float>(Yg[(int64_t)k * ld + i]), iw = __ldg(tb.invW + k), Xk = y * iw * Wbar;
        const float muk = expf(log_mu(k)), rk = sqrtf(muk);
        const float *a = tb.nasa_cp + (rng * N + k) * 5;
        const float cpR = fmaf(fmaf(fmaf(fmaf(__ldg(a + 4), T, __ldg(a + 3)), T, __ldg(a + 2)), T, __ldg(a + 1)), T, __ldg(a));
        float den = 0.0f, ds = 0.0f, gs = 0.0f;
        for (int j = 0; j < N; ++j) {
            const float Xj = to_real<float>(Yg[(int64_t)j * ld + i]) * __ldg(tb.invW + j) * Wbar;
            const float t = expf(-0.5f * log_mu(j)) * rk;
            const float *w = tb.wilke + (size_t)k * Np + j, *d = tb.diff + (size_t)k * Np + j;
            const size_t st = (size_t)N * Np;
            den = fmaf(fmaf(t, fmaf(t, __ldg(w + 2 * st), __ldg(w + st)), __ldg(w)), Xj, den);
            float g = 0.0f;
            for (int n = 4; n >= 0; --n) g = fmaf(g, x, __ldg(d + n * st));
            ds = fmaf(g, Xj, ds);
            gs += g;
        }
        mu = fmaf(Xk, muk / den, mu);
        lam = fmaf(Xk, muk * (cpR + 1.25f) * R * iw / den, lam);      // Eucken
        if (Dkg)
            Dkg[(int64_t)k * ld + i] = pure_species(Xk, y, ds, gs, N) ? T15 / (p * gs / float(N - 1)) : (1.0f - y) * T15 / (p * ds);
    }
    if (mug) mug[i] = mu;
    if (lamg) lamg[i] = lam;
}
template <typename in_t>
__device__ __noinline__ void wide_cells(const TcArgs *g, const in_t *Tg, const in_t *pg, const in_t *Yg) {
    if (threadIdx.x >= 128) return;
    for (int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x; i < g->ncells; i += (int64_t)gridDim.x * 128)
        wide_cell(*g, Tg, pg, Yg, i);
}

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// eight values as FP16 pairs: the hi and lo terms, 16 bytes each
__device__ __forceinline__ void split8(const float (&v)[8], uint4 &hi, uint4 &lo) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const __half2 a = __floats2half2_rn(v[2 * u], v[2 * u + 1]);
        const float2 f = __half22float2(a);
        const __half2 b = __floats2half2_rn(v[2 * u] - f.x, v[2 * u + 1] - f.y);
        h[u] = *reinterpret_cast<const uint32_t *>(&a);
        l[u] = *reinterpret_cast<const uint32_t *>(&b);
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// Descriptor of a no-swizzle K-major operand: core matrices of 8 rows x 16 bytes, consecutive
// along the rows (128 bytes apart), `lbo` bytes from one 16-byte chunk of K to the next.
__device__ __forceinline__ uint64_t sdesc_kmajor_plain(uint32_t saddr, uint32_t lbo) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(128u >> 4) << 32) |
           ((uint64_t)1 << 46);
}

template <typename in_t, int NMAX>
__global__ void __launch_bounds__(TcLayout<NMAX>::kThreads, TcLayout<NMAX>::kCtas)
    props_tc_kernel(const __grid_constant__ TcArgs g, const in_t *__restrict__ Tg, const in_t *__restrict__ pg, const in_t *__restrict__ Yg) {
    using L = TcLayout<NMAX>;
    constexpr int TPR = L::kTPR, SH = L::kShares;
    extern __shared__ __align__(128) uint8_t tc_smem[];
    const int N = g.N, rows = g.tc.rows, NP = g.tc.NP, NR = g.tc.NR;
    uint8_t *sA = tc_smem;
    uint8_t *sB = sA + L::kABytes;
    const uint32_t b_lbo = (uint32_t)rows * 16, b_term = L::kChunks * b_lbo;
    float *sY = reinterpret_cast<float *>(sB + 2 * b_term);            // [NMAX][128] (kStageY)
    // per species, padded to PAD: thermo_kernel's NASA rows of both ranges (3 float4 each), log2 r
    // (2 float4: c0 .. c3 | c4, 1/W, 1/dscale, 2^n), R (cp/R + 5/4) / W of both ranges (2 float4 each)
    float4 *tab = reinterpret_cast<float4 *>(reinterpret_cast<uint8_t *>(sY) + L::kYBytes);
    constexpr int PAD = L::kPad;
    constexpr int TAB2 = 3 * PAD + 1, EUK2 = 2 * PAD + 1;              // the high range, in other banks than the low
    float4 *vis = tab + 2 * TAB2 - 1;
    float4 *euk = vis + 2 * PAD;
    float *red = reinterpret_cast<float *>(euk + (L::kEuk ? 4 * PAD + 1 : 1));   // [kRedRows][SH][128]
    constexpr int RED2 = (L::kRedRows - 2) * SH;                       // first row of mu and lambda
    uint64_t *bars = reinterpret_cast<uint64_t *>(red + L::kRedRows * SH * 128);
    uint64_t *bar_b = bars, *bar_m = bars + 1;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2);
    volatile uint32_t *wide = tmem_slot + 1;                           // 1: some cell's sums are not finite; 2: a wait ran out
    const int warp = threadIdx.x >> 5;
    const int grp = warp >> 2;                                         // which share of the species
    const int row = threadIdx.x & 127;                                 // cell of the tile = TMEM lane
    const uint32_t ncols = rows <= 128 ? 128u : (rows <= 256 ? 256u : 512u);

    if (threadIdx.x == 0) {
        tc::mbar_init(bar_b, 1);
        tc::mbar_init(bar_m, 1);
        tc::fence_barrier_init();
        *wide = 0;
        tc::mbar_arrive_expect_tx(bar_b, 2 * b_term);
        for (uint32_t o = 0; o < 2 * b_term; o += 16384) {
            const uint32_t n = 2 * b_term - o < 16384 ? 2 * b_term - o : 16384;
            tc::bulk_load_1d(sB + o, static_cast<const uint8_t *>(g.tc.B) + o, n, bar_b);
        }
    }
    if (warp == 0) {
        tc::tmem_alloc(tmem_slot, ncols);
        tc::tmem_relinquish();
    }
    const float R = float(kR);
    const int ks16 = (N + 15) / 16;                                    // K steps: 16 species each
    // the accumulator's cuts (above): of a K step after a species', for 2, 3 and 4 steps; `later` counts up to NMAX / 16
    const float per_step = NMAX <= 32 ? 2.37e-7f : (ks16 == 3 ? 2.0e-7f : 1.76e-7f);
    const float first = NMAX <= 32 ? 4e-8f : (ks16 == 3 ? 4e-8f - 2.0e-7f : 4e-8f);
    for (int e = threadIdx.x; e < 2 * PAD; e += blockDim.x) {
        const int rg = e / PAD, k = e % PAD;
        float a[5] = {0, 0, 0, 0, 0}, b[6] = {0, 0, 0, 0, 0, 0}, iw = 0.0f;
        if (k < N) {
            for (int q = 0; q < 5; ++q) a[q] = g.tb.nasa_cp[(rg * N + k) * 5 + q];
            for (int q = 0; q < 6; ++q) b[q] = g.tb.nasa_h[(rg * N + k) * 6 + q];
            iw = g.tb.invW[k];
        }
        float4 *o = tab + rg * TAB2 + 3 * k;
        o[0] = make_float4(a[0], a[1], a[2], a[3]);
        o[1] = make_float4(a[4], b[0], b[1], b[2]);
        o[2] = make_float4(b[3], b[4], b[5], iw);
        if (L::kEuk) {
            const float f = R * iw;
            euk[rg * EUK2 + 2 * k] = make_float4((a[0] + 1.25f) * f, a[1] * f, a[2] * f, a[3] * f);
            euk[rg * EUK2 + 2 * k + 1] = make_float4(a[4] * f, 0.0f, 0.0f, 0.0f);
        }
    }
    for (int k = threadIdx.x; k < PAD; k += blockDim.x) {
        const float *q = g.tc.species + 8 * k;
        vis[2 * k] = k < N ? make_float4(q[0], q[1], q[2], q[3]) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        vis[2 * k + 1] = k < N ? make_float4(q[4], g.tb.invW[k], q[5], q[6]) : make_float4(0.0f, 0.0f, 0.0f, 1.0f);
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const int64_t ntiles = (g.ncells + 127) / 128;
    uint32_t phase = 0;
    bool b_ready = false;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x, phase ^= 1u) {
        const int64_t cell = tile * 128 + row;
        const bool valid = cell < g.ncells;
        const int64_t i = valid ? cell : g.ncells - 1;
        const in_t *Yi = Yg + i;
        const float T = to_real<float>(Tg[i]);
        const float p = to_real<float>(pg[i]);
        // own species: mass fraction, r = sqrt(mu), and their share of 1 / Wbar and of the smallest r
        const int k0 = grp * 8;
        float y[8], rk[8];
        {
            const in_t *q = Yi + (int64_t)k0 * g.ld;
#pragma unroll
            for (int u = 0; u < 8; ++u) y[u] = k0 + u < N ? to_real<float>(q[u * g.ld]) : 0.0f;
        }
        const float x = logf(T * 1e-3f);                               // ln(T / 1000)
        float S = 0.0f, rmin = 3.0e38f;
        if (PAD == NMAX || k0 < PAD) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float4 v0 = vis[2 * (k0 + u)], v1 = vis[2 * (k0 + u) + 1];
                float lr = v1.x;
                lr = fmaf(lr, x, v0.w);
                lr = fmaf(lr, x, v0.z);
                lr = fmaf(lr, x, v0.y);
                lr = fmaf(lr, x, v0.x);
                rk[u] = ex2_approx(lr) * v1.w;
                S = fmaf(y[u], v1.y, S);
                rmin = fminf(rmin, rk[u]);
                if (L::kStageY) sY[(k0 + u) * 128 + row] = y[u];
            }
        } else {                                                       // a chunk of zeros (warp-uniform)
#pragma unroll
            for (int u = 0; u < 8; ++u) rk[u] = 1.0f;
        }
        if (SH == TPR || grp < SH) {
            red[grp * 128 + row] = S;
            red[(SH + grp) * 128 + row] = rmin;
        }
        // the next tile's rows on their way to L2
        if (const int64_t next = tile + gridDim.x; threadIdx.x >= 32 && threadIdx.x < 64 && (next + 1) * 128 <= g.ncells)
            for (int q = threadIdx.x - 32; q < N + 2; q += 32) {
                const in_t *src = (q == 0 ? Tg : q == 1 ? pg : Yg + (int64_t)(q - 2) * g.ld) + next * 128;
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"((uint32_t)(128 * sizeof(in_t)))
                             : "memory");
            }
        __syncthreads();
        S = 0.0f;
        rmin = 3.0e38f;
        float later = 0.0f;                                            // shares of S times the K steps that may follow theirs
#pragma unroll
        for (int q = 0; q < SH; ++q) {
            const float Sq = red[q * 128 + row];
            S += Sq;
            if (NMAX / 16 - 1 - q / 2 > 0) later = fmaf(Sq, (float)(NMAX / 16 - 1 - q / 2), later);
            rmin = fminf(rmin, red[(SH + q) * 128 + row]);
        }
        const float Wbar = 1.0f / S;
        const float cut = NMAX <= 16 ? 4e-8f : fmaf(per_step * later, Wbar, first);
        // r is scaled by a power of two that brings the smallest one to 1 .. 2, and 1/r by its reciprocal
        int e = 127 - (int)(__float_as_uint(rmin) >> 23);
        e = e < -100 ? -100 : (e > 100 ? 100 : e);
        const float up = __int_as_float((127 + e) << 23), down = __int_as_float((127 - e) << 23);
        const float xs = Wbar * kTcXScale;
        {
            float v[8], ir[8];
            uint8_t *dst = sA + grp * 2048 + row * 16;
            uint4 hi, lo;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                ir[u] = rcp_approx(rk[u]) * down;
                v[u] = PAD < NMAX && k0 >= PAD ? 0.0f : y[u] * vis[2 * (k0 + u) + 1].y * xs;
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) {                              // X, X / r, X / r^2
                split8(v, hi, lo);
                *reinterpret_cast<uint4 *>(dst + (2 * q) * L::kChunks * 2048) = hi;
                *reinterpret_cast<uint4 *>(dst + (2 * q + 1) * L::kChunks * 2048) = lo;
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] *= ir[u];
            }
        }
        tc::fence_proxy_async_smem();
        tc::tc_fence_before();
        __syncthreads();
        bool ok = true;
        if (threadIdx.x == 0) {
            if (!b_ready) {
                ok = tc::mbar_wait(bar_b, 0, g.spin);
                b_ready = ok;
            }
            if (ok) {
                tc::tc_fence_after();
                // the three column groups: vector 1 on T1, vector 0 on T0 and the resistances (two parts
                // where it is wider than one instruction), vector 2 on T2
                const int nx = 6 * NP, ksteps = (N + 15) / 16;
                const int part_v[4] = {1, 0, 0, 2};
                const int part_r[4] = {0, NR, NR + (nx < 256 ? nx : 256), NR + nx};
                const int part_n[4] = {NR, nx < 256 ? nx : 256, nx < 256 ? 0 : nx - 256, NR};
                const uint32_t a0 = tc::smem_u32(sA), b0 = tc::smem_u32(sB);
                for (int q = 0; q < 4; ++q) {
                    if (part_n[q] == 0) continue;
                    const uint32_t idesc = tc::idesc_e4m3_f32(128, part_n[q]);   // format code 0 is F16 for kind::f16
                    uint32_t acc = 0;
                    // hi lo, lo hi, hi hi: the accumulator is cut, not rounded, after every instruction, so
                    // the small products come first and only the last K / 16 cuts are of full size
                    for (int t = 0; t < 3; ++t) {
                        const uint32_t at = a0 + (uint32_t)(2 * part_v[q] + (t == 1)) * (L::kChunks * 2048);
                        const uint32_t bt = b0 + (t == 0 ? b_term : 0u) + (uint32_t)part_r[q] * 16;
                        for (int ks = 0; ks < ksteps; ++ks) {
                            tc::umma_f16(tmem + part_r[q], sdesc_kmajor_plain(at + ks * 4096, 2048),
                                         sdesc_kmajor_plain(bt + ks * 2 * b_lbo, b_lbo), idesc, acc);
                            acc = 1;
                        }
                    }
                }
                tc::umma_commit(bar_m);
            }
        }
        __syncwarp();
        const int hot = (T >= g.T_mid) ? 1 : 0;
        // beside the products: cp and h over all species, ascending, one thread each (of the last chunks,
        // which have the fewest species)
        if (grp >= TPR - 2) {
            const float4 *tr = tab + hot * TAB2;
            auto mass = [&](int k) {
                if constexpr (L::kStageY) return sY[k * 128 + row];
                else return to_real<float>(Yi[(int64_t)k * g.ld]);
            };
            if (grp == TPR - 1 && g.cp) {
                float cpm = 0.0f;
#pragma unroll 4
                for (int k = 0; k < N; ++k) {
                    const float yk = mass(k);
                    const float4 q0 = tr[3 * k];
                    float cpR = tr[3 * k + 1].x;
                    cpR = fmaf(cpR, T, q0.w);
                    cpR = fmaf(cpR, T, q0.z);
                    cpR = fmaf(cpR, T, q0.y);
                    cpR = fmaf(cpR, T, q0.x);
                    const float yw = yk * tr[3 * k + 2].w;
                    cpm = fmaf(yw, cpR, cpm);
                }
                if (valid) g.cp[i] = cpm * R;
            }
            if (grp == TPR - 2 && g.h) {
                const float iT = 1.0f / T;
                float hm = 0.0f;
#pragma unroll 4
                for (int k = 0; k < N; ++k) {
                    const float yk = mass(k);
                    const float4 q1 = tr[3 * k + 1], q2 = tr[3 * k + 2];
                    float hR = q2.y;
                    hR = fmaf(hR, T, q2.x);
                    hR = fmaf(hR, T, q1.w);
                    hR = fmaf(hR, T, q1.z);
                    hR = fmaf(hR, T, q1.y);
                    hR = fmaf(q2.z, iT, hR);
                    const float yw = yk * q2.w;
                    hm = fmaf(yw, hR, hm);
                }
                if (valid) g.h[i] = hm * R * T;
            }
        }
        ok = ok && tc::mbar_wait(bar_m, phase, g.spin);
        tc::tc_fence_after();
        const float T15 = T * sqrtf(T), T15p = T15 / p;
        constexpr int ES = L::kEuk ? 2 : 3;
        const float4 *er = L::kEuk ? euk + hot * EUK2 : tab + hot * TAB2;
        const float pure = 0.999f * S;
        float mu = 0.0f, lam = 0.0f;
        bool alone = false;
        float *Dp = g.Dk + (int64_t)k0 * g.ld + i;
#pragma unroll
        for (int u0 = 0; u0 < 8; u0 += 2) {
            if (k0 + u0 >= N) break;                                   // warp-uniform
            float v[16];
            uint32_t ad[8];
            ad[0] = tlane + k0 + u0;                                   // T1
#pragma unroll
            for (int q = 0; q < 6; ++q) ad[1 + q] = tlane + NR + q * NP + k0 + u0;   // T0, resistances
            ad[7] = tlane + NR + 6 * NP + k0 + u0;                     // T2
            __syncwarp();                                              // converged for the TMEM loads
            tmem_ld8x2(ad, v);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int k = k0 + u0 + u;
                const float yk = y[u0 + u], r = rk[u0 + u], rn = r * up;
                const float4 e0 = er[ES * k], v1 = vis[2 * k + 1];
                float lk = er[ES * k + 1].x;                           // lambda_k / mu_k (Eucken)
                lk = fmaf(lk, T, e0.w);
                lk = fmaf(lk, T, e0.z);
                lk = fmaf(lk, T, e0.y);
                lk = fmaf(lk, T, e0.x);
                if (!L::kEuk) lk = (lk + 1.25f) * (R * v1.y);
                const float yw = yk * v1.y;
                const float den = fmaf(rn, fmaf(rn, v[14 + u], v[u]), v[2 + u]);
                const float wk = (r * r) * (yw * rcp_approx(den));     // X_k mu_k / sum, up to a factor of the cell
                if (k < N) {                                           // (columns past N hold zeros: 0 / 0)
                    mu += wk;
                    lam = fmaf(wk, lk, lam);
                }
                if (g.Dk) {
                    float ds = v[12 + u];
                    ds = fmaf(ds, x, v[10 + u]);
                    ds = fmaf(ds, x, v[8 + u]);
                    ds = fmaf(ds, x, v[6 + u]);
                    ds = fmaf(ds, x, v[4 + u]);
                    float ri = rcp_approx(ds);
                    ri = fmaf(ri, fmaf(-ds, ri, 1.0f) - cut, ri);
                    alone |= yw > pure;
                    if (valid && ok && k < N) *Dp = (1.0f - yk) * T15p * (ri * v1.z);
                    Dp += g.ld;
                }
            }
        }
        if (g.Dk && alone && valid && ok) {                            // rare: redone in FP32
            for (int k = k0; k < k0 + 8 && k < N; ++k) {
                const float yk = to_real<float>(Yi[(int64_t)k * g.ld]);
                const float yw = yk * vis[2 * k + 1].y;
                if (yw > pure)
                    g.Dk[(int64_t)k * g.ld + i] = near_pure_D(g.tb, N, (N + 3) & ~3, k, g.ld, i, Yg, Wbar, x, yk,
                                                              yw * Wbar, T15, p);
            }
        }
        const float unit = Wbar * (kTcXScale * kTcWilkeScale) * (1.0f - (cut + 2e-8f));
        if (SH == TPR || grp < SH) {
            red[(RED2 + grp) * 128 + row] = mu * unit;
            red[(RED2 + SH + grp) * 128 + row] = lam * unit;
        }
        tc::tc_fence_before();                                         // TMEM reads before the next tile's products
        const bool fin = __syncthreads_and(ok && fabsf(mu) < INFINITY);
        const bool all_ok = fin || __syncthreads_and(ok);
        if (!fin && threadIdx.x == 0) *wide = 1;
        if (grp == 0) {
            mu = 0.0f;
            lam = 0.0f;
#pragma unroll
            for (int q = 0; q < SH; ++q) {
                mu += red[(RED2 + q) * 128 + row];
                lam += red[(RED2 + SH + q) * 128 + row];
            }
            if (!all_ok) mu = lam = __int_as_float(0x7fc00000);
            if (valid && g.mu) g.mu[i] = mu;
            if (valid && g.lam) g.lam[i] = lam;
        }
        if (!all_ok) {
            // a wait ran out: NaN for the tile's transport and for every output of the tiles the CTA had
            // still to do, and the CTA ends once what it issued has finished
            const float nan = __int_as_float(0x7fc00000);
            if (threadIdx.x == 0) {
                atomicExch(g.err, 1u);
                *wide = 2;
            }
            for (int64_t c = cell; c < g.ncells; c += (int64_t)gridDim.x * 128) {
                if (g.Dk)
                    for (int k = grp; k < N; k += TPR) g.Dk[(int64_t)k * g.ld + c] = nan;
                if (grp == 0 && c != cell) {
                    if (g.cp) g.cp[c] = nan;
                    if (g.h) g.h[c] = nan;
                    if (g.mu) g.mu[c] = nan;
                    if (g.lam) g.lam[c] = nan;
                }
            }
            break;
        }
        if (RED2 == 0) __syncthreads();                                // the sums' rows are written again
    }
    // An entry past FP16's range (|X_k| >= 4) has made every sum of its cell NaN: such cells, found by their own
    // output, are redone here, out of the loop above, whose registers a call would spill. (A state that is itself
    // not finite stays as it is.)
    __syncthreads();
    if (*wide == 1) wide_cells(&g, Tg, pg, Yg);
    if (threadIdx.x == 0) {
        // nothing in flight when the CTA ends (full limit): the table copy, then the products
        if (!b_ready && !tc::mbar_wait(bar_b, 0)) atomicExch(g.err, 1u);
        uint64_t *bar_d = bars + 3;
        tc::mbar_init(bar_d, 1);
        tc::fence_barrier_init();
        tc::umma_commit(bar_d);
        if (!tc::mbar_wait(bar_d, 0)) atomicExch(g.err, 1u);
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, ncols);
    }
}

template <typename in_t, int NMAX>
int launch_props_tc(const chem_mech *m, int64_t ncells, int64_t ld, const void *T, const void *p, const void *Y,
                    void *cp, void *h, void *mu, void *lam, void *Dk, cudaStream_t st) {
    using L = TcLayout<NMAX>;
    const size_t smem = L::bytes(m->dev.tc.rows);
    static DeviceOnce configured;
    if (int rc = dynamic_smem_limit(configured, props_tc_kernel<in_t, NMAX>, NMAX <= 32 ? 113 * 1024 : 227 * 1024,
                                    "props_eval smem attribute"))
        return rc;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t ntiles = (ncells + 127) / 128;
    const int64_t most = (int64_t)sms * L::kCtas;                      // the resident CTAs
    const TcArgs a{m->N, float(m->T_mid), m->dev.f32, m->dev.tc, ncells, ld, static_cast<float *>(cp),
                   static_cast<float *>(h), static_cast<float *>(mu), static_cast<float *>(lam),
                   static_cast<float *>(Dk), m->dev.counters + kPropsErrCounter, m->wait_limit};
    void *pb = prof_begin(st);
    props_tc_kernel<in_t, NMAX><<<(unsigned)(ntiles < most ? ntiles : most), L::kThreads, smem, st>>>(
        a, static_cast<const in_t *>(T), static_cast<const in_t *>(p), static_cast<const in_t *>(Y));
    prof_end(pb, st, "props_kernel<f32>", (double)ncells * (16.0 * m->N * m->N + 30.0 * m->N),
             (double)ncells * ((m->N + 2) * sizeof(in_t) + (4 + m->N) * sizeof(float)));
    return check_cuda(cudaGetLastError(), "props_eval launch");
}

template <typename real, typename in_t, int NMAX>
int launch_props(const chem_mech *m, int64_t ncells, int64_t ld, const void *T, const void *p, const void *Y,
                 void *cp, void *h, void *mu, void *lam, void *Dk, cudaStream_t st) {
    const bool transport = mu || lam || Dk;
    const size_t smem = tables_in_smem<real>() ? ((transport ? (size_t)8 * m->N * m->dev.Np : 0) +
                                                  (size_t)kSpeciesFloats * m->N) * sizeof(real)
                                               : 0;
    static DeviceOnce configured;
    if (smem > 0)
        if (int rc = dynamic_smem_limit(configured, props_kernel<real, in_t, NMAX>, kPropsSmemMax,
                                        "props_eval smem attribute"))
            return rc;
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, props_kernel<real, in_t, NMAX>, 128, smem);
    const int max_blocks = sms * (per_sm > 0 ? per_sm : 1);
    int64_t need = (ncells + 127) / 128;
    int blocks = (int)(need < max_blocks ? need : max_blocks);
    const PropTables<real> &tb = (sizeof(real) == 4) ? *reinterpret_cast<const PropTables<real> *>(&m->dev.f32)
                                                      : *reinterpret_cast<const PropTables<real> *>(&m->dev.f64);
    void *pb = prof_begin(st);
    props_kernel<real, in_t, NMAX><<<blocks, 128, smem, st>>>(
        m->N, m->dev.Np, real(m->T_mid), tb, ncells, ld, static_cast<const in_t *>(T), static_cast<const in_t *>(p),
        static_cast<const in_t *>(Y), static_cast<real *>(cp), static_cast<real *>(h), static_cast<real *>(mu),
        static_cast<real *>(lam), static_cast<real *>(Dk));
    prof_end(pb, st, std::string("props_kernel<") + (sizeof(real) == 4 ? "f32" : "f64") + ">",
             (double)ncells * (16.0 * m->N * m->N + 30.0 * m->N),
             (double)ncells * ((m->N + 2) * sizeof(in_t) + (4 + m->N) * sizeof(real)));
    return check_cuda(cudaGetLastError(), "props_eval launch");
}

template <typename real, typename in_t>
int dispatch_props(const chem_mech *m, int64_t ncells, int64_t ld, const void *T, const void *p, const void *Y,
                   void *cp, void *h, void *mu, void *lam, void *Dk, cudaStream_t st) {
    if constexpr (sizeof(real) == 4) {
        if (!mu && !lam && !Dk) return launch_thermo<in_t>(m, ncells, ld, T, Y, cp, h, st);
        // the tensor-core pass wherever its operands fit (up to 56 species with coefficients that FP16
        // pairs hold); the pair loop for the rest
        if (m->dev.tc.B) {
            if (m->N <= 16) return launch_props_tc<in_t, 16>(m, ncells, ld, T, p, Y, cp, h, mu, lam, Dk, st);
            if (m->N <= 32) return launch_props_tc<in_t, 32>(m, ncells, ld, T, p, Y, cp, h, mu, lam, Dk, st);
            return launch_props_tc<in_t, 64>(m, ncells, ld, T, p, Y, cp, h, mu, lam, Dk, st);
        }
    } else {
        // the fewest threads per cell that give every SM kSplitWarps warps, at most one per species
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const int64_t want = (int64_t)sms * kSplitWarps * 32;
        if (ncells < want && m->N >= 4) {
            if (ncells * 4 >= want || m->N < 8)
                return launch_props_split<4>(m, ncells, ld, T, p, Y, cp, h, mu, lam, Dk, st);
            if (ncells * 8 >= want || m->N < 16)
                return launch_props_split<8>(m, ncells, ld, T, p, Y, cp, h, mu, lam, Dk, st);
            if (ncells * 16 >= want || m->N < 24)
                return launch_props_split<16>(m, ncells, ld, T, p, Y, cp, h, mu, lam, Dk, st);
            return launch_props_split<32>(m, ncells, ld, T, p, Y, cp, h, mu, lam, Dk, st);
        }
    }
    if (m->N <= 16) return launch_props<real, in_t, 16>(m, ncells, ld, T, p, Y, cp, h, mu, lam, Dk, st);
    if (m->N <= 32) return launch_props<real, in_t, 32>(m, ncells, ld, T, p, Y, cp, h, mu, lam, Dk, st);
    return launch_props<real, in_t, 64>(m, ncells, ld, T, p, Y, cp, h, mu, lam, Dk, st);
}

}  // namespace

// Properties (FP32 outputs from the FP64 state) of cells [0, ncells) for the learned step's
// fused entry point; the same kernels as props_eval(CHEM_F64_IN_F32).
int props_f64_in_f32(const chem_mech *m, int64_t ncells, int64_t ld, const double *T, const double *p,
                     const double *Y, float *cp, float *h, float *mu, float *lam, float *Dk, cudaStream_t st) {
    if (ncells <= 0) return CHEM_OK;
    return dispatch_props<float, double>(m, ncells, ld, T, p, Y, cp, h, mu, lam, Dk, st);
}

}  // namespace chemgb

using namespace chemgb;

extern "C" int props_eval(const chem_mech *m, int64_t ncells, int64_t ld, int dtype, const void *T, const void *p,
                          const void *Y, void *cp, void *h, void *mu, void *lambda, void *Dk,
                          chem_stream_t stream) {
    if (!m) return set_error(CHEM_EINVAL, "props_eval: null mechanism");
    if (ncells < 0 || ld < ncells || (ld & 3) != 0)
        return set_error(CHEM_EINVAL, "props_eval: need 0 <= ncells <= ld and ld a multiple of 4");
    if (dtype != CHEM_F32 && dtype != CHEM_F64 && dtype != CHEM_F64_IN_F32)
        return set_error(CHEM_EINVAL, "props_eval: bad dtype");
    if (ncells == 0) return CHEM_OK;
    if (!T || !p || !Y) return set_error(CHEM_EINVAL, "props_eval: null input array");
    const void *ptrs[] = {T, p, Y, cp, h, mu, lambda, Dk};
    for (const void *q : ptrs)
        if (q && !aligned16(q)) return set_error(CHEM_EINVAL, "props_eval: arrays must be 16-byte aligned");
    std::string why;
    if (!device_ok(&why)) return set_error(CHEM_EUNSUPPORTED, "props_eval: " + why);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (dtype == CHEM_F32) return dispatch_props<float, float>(m, ncells, ld, T, p, Y, cp, h, mu, lambda, Dk, st);
    if (dtype == CHEM_F64_IN_F32)
        return dispatch_props<float, double>(m, ncells, ld, T, p, Y, cp, h, mu, lambda, Dk, st);
    return dispatch_props<double, double>(m, ncells, ld, T, p, Y, cp, h, mu, lambda, Dk, st);
}
