// stiff.cu -- chem_step_stiff: FP64 constant-pressure reactor integration over
// dt for every cell (Sec. 3.1: the compositions are integrated over dt = 1 us;
// Sec. 4.2: direct integration, "CPU-DI", is the plain method the network
// replaces).
//
// Design for sm_103a:
//  - One warp per cell, or two (many cells of up to 15 species). Cells are popped from a device work queue (one atomic
//    per cell), so cells with very different step counts balance across the
//    persistent grid.
//  - The state vector y = (T, Y_1..Y_N) is distributed over the lanes:
//    component c lives in lane c % 32, register slot c / 32 (n = N + 1 <= 64;
//    one slot up to n = 32).
//  - Species work runs lane-per-species, reaction work lane-per-reaction.
//    Up to n = 32 the LU factors live in registers, lane i holding row i: the
//    pivot search is a warp reduction, rows are not moved (each lane tracks its
//    row's position), the pivot row is broadcast by shuffles, and the triangular
//    solves are one shuffle and one multiply-add per column. Above, the matrix
//    is factored in the warp's shared-memory slice, columns over lanes.
//  - What bounds it: FP64 issues one warp instruction per 16 clocks and SM (64
//    per sub-partition), so the reaction and species passes count FP64
//    instructions: no integer-to-FP64 conversions (stoichiometric coefficients are
//    kept as the high half of their FP64 pattern), d q / d C_l from the mass-action
//    factors directly, several warp sums in one butterfly, T-dependent data in
//    tables that a warp reads coalesced. The Jacobian's sparse part is summed entry
//    by entry from lists sorted by length (ELLPACK). The former kernel (row-owner
//    sums over each species' reactions, the factors in shared memory, 23 KB per warp and
//    8 warps per SM) took 54,000 warp instructions and 1,600 FP64 ones a step of the
//    30-species mixed mode, with the FP64 pipe 44 % busy; this one 30,000 and 1,350 at 16
//    warps per SM (12 KB each), 60 %. 65,536 cells at rtol 1e-2: 148 -> 87 ms; 4,096
//    cells of the 9-species mechanism in FP64 at rtol 1e-6: 111 -> 76 ms, with two per warp 57 ms; the 2 % fallback
//    of 262,144 learned cells: 14.5 -> 9.1 ms.
//  - Few cells (at most one per SM, e.g. the learned step's out-of-distribution
//    cells): a team of kWarps warps integrates each cell, one per SM
//    sub-partition. The reaction pass, the Jacobian's lists and the species' sums
//    are split over the team, the rest runs redundantly in every warp on identical
//    data, and one warp writes the shared results. Every value is computed by the
//    same operations in the same order as by a lone warp, so the results are
//    bitwise those of one warp per cell.
//  - Integrator: Rodas3 (Sandu et al. 1997), an embedded L-stable Rosenbrock
//    method of order 3(2), in the transformed form
//      (I/(h g) - J) K_i = f(y + sum_j a_ij K_j) + sum_j (c_ij / h) K_j,
//    y_new = y + sum_i m_i K_i, error estimate sum_i e_i K_i, with the
//    step-size controller of chem_ode_opts. The FP64 mode is FP64 throughout; the mixed mode takes
//    the rate constants' exponentials, the fall-off blending and the linear algebra in FP32.
#include <math_constants.h>

#include <cmath>
#include <mutex>
#include <type_traits>

#include "internal.cuh"
#include "stiff_lu.cuh"

namespace chemgb {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kWarps = 4;
constexpr size_t kSmemHeader = 16;   // the team's queue ticket, ahead of the warp slices
constexpr double kMixedMinRtol = 1e-5;   // tightest rtol the mixed mode integrates (below it: FP64)

// Rodas3 coefficients (g = 1/2 on the diagonal)
constexpr double kGam = 0.5;
// a31 = a41 = 2, a43 = 1, the others 0; m = (2, 0, 1, 1), e = (0, 0, 0, 1)
constexpr double kC21 = 4.0, kC31 = 1.0, kC32 = -1.0, kC41 = 1.0, kC42 = -1.0, kC43 = -8.0 / 3.0;

// Lanes per cell, LPC: 32, or 16 with two cells in the halves of a warp (n <= 16). Every shuffle is a whole
// warp's; sums over 16 lanes have the bits of sums over 32 whose upper lanes hold zeros.
template <int LPC>
__device__ __forceinline__ double warp_sum(double v) {
    // butterfly: every lane ends with the same bits (addition is commutative)
#pragma unroll
    for (int o = LPC / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}
// Two (four) sums in one butterfly: the halves (quarters) of the warp carry one sum each, so the FP64
// pipe sees 5 (6) additions instead of 10 (20). Every lane ends with all of them.
template <int LPC>
__device__ __forceinline__ void warp_sum2(double &a, double &b, int lane) {
    const bool up = lane & (LPC / 2);
    double v = (up ? b : a) + __shfl_xor_sync(kFull, up ? a : b, LPC / 2);
#pragma unroll
    for (int o = LPC / 4; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    a = __shfl_sync(kFull, v, 0, LPC);
    b = __shfl_sync(kFull, v, LPC / 2, LPC);
}
template <int LPC>
__device__ __forceinline__ void warp_sum3(double &a, double &b, double &c, int lane) {
    const bool up = lane & (LPC / 2), mid = lane & (LPC / 4);
    const double ab = (up ? b : a) + __shfl_xor_sync(kFull, up ? a : b, LPC / 2);
    const double cc = c + __shfl_xor_sync(kFull, c, LPC / 2);
    double v = (mid ? cc : ab) + __shfl_xor_sync(kFull, mid ? ab : cc, LPC / 4);
#pragma unroll
    for (int o = LPC / 8; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    a = __shfl_sync(kFull, v, 0, LPC);
    b = __shfl_sync(kFull, v, LPC / 2, LPC);
    c = __shfl_sync(kFull, v, LPC / 4, LPC);
}

// The warps integrating one cell: W = 1 (a lone warp) or W = kWarps (the block).
template <int W>
struct Team {
    static constexpr int kWarps = W;
    int wt;                    // rank of this warp in the team
    __device__ __forceinline__ void sync() const {
        if (W == 1) __syncwarp();
        else asm volatile("bar.sync 1, %0;" ::"n"(W * 32) : "memory");
    }
    __device__ __forceinline__ bool lead() const { return W == 1 || wt == 0; }
};

// One warp's shared-memory slice. mreal is the type of the matrix and of what only the matrix reads:
// FP32 in the mixed mode (values cut from FP64 once, when they are stored). BIG (n > 32): the LU
// factors live in shared memory too. Absent species have index N: C = 1, g = H = 0; the absent reaction
// has index R: rq = rdqT = 0.
template <bool MX>
struct Slice {
    using mreal = typename std::conditional<MX, float, double>::type;
    double *C, *g, *H;             // [N+1] concentration, S/R - H/RT, H/RT
    double *rq, *rdqT;             // [R+1] rate of progress, its derivative to T
    double *xs;                    // [n] this warp's own vector buffer
    mreal *G;                      // [n][n] I/(h g) - J
    mreal *F, *invd;               // [n][n], [n] LU factors, reciprocal pivots (BIG)
    mreal *cpR, *wdot, *wT, *JCC, *U, *V, *HR;   // [N] (wT [n])
    mreal *rc3, *rdq;              // [n_tb] third-body coefficient, [R][nslot] d q / d C of its species
    float *Cf;                     // [N] concentrations in FP32 (mixed mode)
    int *piv;                      // [n] (BIG)
};

// Lays the slice out from `base` (null: only counts) and returns its bytes. Overlaps: in FP64 up to n = 32
// the matrix (dead once its rows are in registers) shares its space with rq and rdqT (dead when it
// is built); BIG mixed factors share theirs with rdq (dead when the matrix is built), and BIG pivots and
// reciprocal pivots with wT and rc3 (likewise), without which a mechanism of third-body reactions with six species
// each took more than the layout before.
template <bool MX, bool BIG>
__host__ __device__ inline size_t make_slice(char *base, int N, int R, int n_tb, int nslot, Slice<MX> *s) {
    using mreal = typename Slice<MX>::mreal;
    const int n = N + 1;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        char *p = base + o;
        o += (bytes + 7) & ~size_t(7);
        return p;
    };
    Slice<MX> t;
    t.C = reinterpret_cast<double *>(take((size_t)(N + 1) * 8));
    t.g = reinterpret_cast<double *>(take((size_t)(N + 1) * 8));
    t.H = reinterpret_cast<double *>(take((size_t)(N + 1) * 8));
    t.xs = reinterpret_cast<double *>(take((size_t)n * 8));
    const size_t g_bytes = (size_t)n * n * sizeof(mreal), q_bytes = (size_t)(R + 1) * 8;
    if (!MX && !BIG) {
        char *p = take(g_bytes > 2 * q_bytes ? g_bytes : 2 * q_bytes);
        t.G = reinterpret_cast<mreal *>(p);
        t.rq = reinterpret_cast<double *>(p);
        t.rdqT = t.rq + R + 1;
    } else {
        t.rq = reinterpret_cast<double *>(take(q_bytes));
        t.rdqT = reinterpret_cast<double *>(take(q_bytes));
        t.G = reinterpret_cast<mreal *>(take(g_bytes));
    }
    const size_t d_bytes = (size_t)R * nslot * sizeof(mreal);
    if (MX && BIG) {
        char *p = take(g_bytes > d_bytes ? g_bytes : d_bytes);
        t.F = t.rdq = reinterpret_cast<mreal *>(p);
    } else {
        t.rdq = reinterpret_cast<mreal *>(take(d_bytes));
        t.F = t.G;
    }
    mreal **small[] = {&t.cpR, &t.wdot, &t.wT, &t.JCC, &t.U, &t.V, &t.HR};
    for (mreal **q : small) *q = reinterpret_cast<mreal *>(take((size_t)(q == &t.wT ? n : N) * sizeof(mreal)));
    t.rc3 = reinterpret_cast<mreal *>(take((size_t)(BIG && n > n_tb ? n : n_tb) * sizeof(mreal)));
    t.invd = BIG ? t.rc3 : nullptr;
    t.Cf = MX ? reinterpret_cast<float *>(take((size_t)N * 4)) : nullptr;
    t.piv = BIG ? reinterpret_cast<int *>(t.wT) : nullptr;
    if (s) *s = t;
    return (o + 15) & ~size_t(15);
}

// values of the last right-hand-side evaluation needed by the Jacobian
struct EvalInfo {
    double T, invT, rho, cp, dcpdT, Wbar, Q;
};

// the FP64 (FP32) value whose high 16 bits a code word carries
template <typename real>
__device__ __forceinline__ real code_value(unsigned w) {
    if constexpr (sizeof(real) == 4) return __uint_as_float(w & 0xFFFF0000u);
    else return __hiloint2double((int)(w & 0xFFFF0000u), 0);
}
// an FP64 value in the matrix type (FP32: cut on the integer pipe)
template <typename real>
__device__ __forceinline__ real rd(double x) {
    if constexpr (sizeof(real) == 4) return f64_to_f32_trunc(x);
    else return x;
}

// Troe blending function F(T, Pr) (Gilbert, Luther and Troe 1983), with
// glg = d log10 F / d log10 Pr and dF/dT at fixed Pr. tp = (a, 1/T***, 1/T*, T**).
__device__ void troe_F(const double *tp, double T, double invT, double Prd, double &F, double &glg,
                       double &dFdT_atPr) {
    const double a = __ldg(tp), r3 = __ldg(tp + 1), r1 = __ldg(tp + 2), T2 = __ldg(tp + 3);
    const double e3 = exp(-T * r3), e1 = exp(-T * r1), e2 = exp(-T2 * invT);
    const double Fc = (1.0 - a) * e3 + a * e1 + e2;
    const double dFc = -(1.0 - a) * r3 * e3 - a * r1 * e1 + T2 * invT * invT * e2;
    const double phi = log10(Fc);
    const double c = -0.4 - 0.67 * phi, nn = 0.75 - 1.27 * phi, d = 0.14;
    const double L = log10(Prd) + c;
    const double rden = 1.0 / (nn - d * L);
    const double f1 = L * rden;
    const double rq = 1.0 / (1.0 + f1 * f1);
    F = exp10(phi * rq);
    const double df1_dL = nn * rden * rden;
    glg = -phi * 2.0 * f1 * rq * rq * df1_dL;
    const double df1_dphi = (-0.67 * (nn - d * L) - L * (-1.27 + d * 0.67)) * rden * rden;
    const double dlgF_dphi = rq - phi * 2.0 * f1 * rq * rq * df1_dphi;
    const double dphi_dT = dFc / (Fc * 2.302585092994046);
    dFdT_atPr = F * 2.302585092994046 * dlgF_dphi * dphi_dT;
}

// The same blending in FP32 (the mixed mode): F, glg and dF/dT at fixed Pr to FP32 accuracy.
__device__ void troe_F_f32(const double *tp, float T, float invT, float Prd, float &F, float &glg, float &dFdT_atPr) {
    const float a = f64_to_f32_trunc(__ldg(tp)), r3 = f64_to_f32_trunc(__ldg(tp + 1));
    const float r1 = f64_to_f32_trunc(__ldg(tp + 2)), T2 = f64_to_f32_trunc(__ldg(tp + 3));
    const float e3 = expf(-T * r3), e1 = expf(-T * r1), e2 = expf(-T2 * invT);
    const float Fc = (1.0f - a) * e3 + a * e1 + e2;
    const float dFc = -(1.0f - a) * r3 * e3 - a * r1 * e1 + T2 * invT * invT * e2;
    const float phi = log10f(Fc);
    const float c = -0.4f - 0.67f * phi, nn = 0.75f - 1.27f * phi, d = 0.14f;
    const float L = log10f(Prd) + c;
    const float rden = 1.0f / (nn - d * L);
    const float f1 = L * rden;
    const float rq = 1.0f / (1.0f + f1 * f1);
    F = exp10f(phi * rq);
    const float df1_dL = nn * rden * rden;
    glg = -phi * 2.0f * f1 * rq * rq * df1_dL;
    const float df1_dphi = (-0.67f * (nn - d * L) - L * (-1.27f + d * 0.67f)) * rden * rden;
    const float dlgF_dphi = rq - phi * 2.0f * f1 * rq * rq * df1_dphi;
    const float dphi_dT = dFc / (Fc * 2.30258509f);
    dFdT_atPr = F * 2.30258509f * dlgF_dphi * dphi_dT;
}

// exp(x) for the mixed mode: the argument and the result cross between FP64 and FP32 on the
// integer pipe (truncation: relative error below 2^-23 of the argument), exp in FP32
__device__ __forceinline__ double exp_mx(double x) { return f32_to_f64_int(expf(f64_to_f32_trunc(x))); }

// f = f(y) for the warp's cell. JAC: also what build_matrix needs. MX (the mixed mode): the rate
// constants' exponentials and the fall-off blending in FP32, the rest FP64.
template <int W, int NS, bool MX, bool JAC, int LPC = 32>
__device__ __forceinline__ EvalInfo eval_rhs(const DevMech &m, const Slice<MX> &sh, Team<W> tm, int lane, double p,
                                             double Rinvp, const double (&y)[NS], double (&f)[NS]) {
    using mreal = typename Slice<MX>::mreal;
    const int N = m.N, R = m.R, n = N + 1;
    EvalInfo info;
    const double T = __shfl_sync(kFull, y[0], 0, LPC);
    const double invT = 1.0 / T;
    const double lnT = log(T);
    info.T = T;
    info.invT = invT;
    const double *tab = m.nasa_t + (T >= m.T_mid ? 17 * 64 : 0);
    tm.sync();                 // every warp of the team is done reading the previous evaluation
    // species pass: thermo and mixture sums (lane per species; in a team every warp
    // computes them and the first writes the shared copies)
    const bool wr = tm.lead();
    double S = 0.0, cp = 0.0, dcp = 0.0;
    double yw_s[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const int c = lane + 32 * s;
        f[s] = 0.0;
        yw_s[s] = 0.0;
        if (c >= 1 && c < n) {
            const int k = c - 1;
            const double *q = tab + k;
            const double a0 = __ldg(q), a1 = __ldg(q + 64), a2 = __ldg(q + 128), a3 = __ldg(q + 192),
                         a4 = __ldg(q + 256);
            const double cpR = a0 + T * (a1 + T * (a2 + T * (a3 + T * a4)));
            q += 5 * 64;
            const double HRT = __ldg(q) + T * (__ldg(q + 64) + T * (__ldg(q + 128) + T * (__ldg(q + 192) + T * __ldg(q + 256))))
                               + __ldg(q + 320) * invT;
            q += 6 * 64;
            const double SR = __ldg(q) * lnT + T * (__ldg(q + 64) + T * (__ldg(q + 128) + T * (__ldg(q + 192) + T * __ldg(q + 256))))
                              + __ldg(q + 320);
            const double yw = y[s] * __ldg(m.f64.invW + k);
            yw_s[s] = yw;
            S += yw;
            cp += yw * cpR;
            if (wr) {
                sh.H[k] = HRT;
                sh.g[k] = SR - HRT;
                if (JAC) sh.cpR[k] = rd<mreal>(cpR);
            }
            if (JAC) dcp += yw * (a1 + T * (2.0 * a2 + T * (3.0 * a3 + T * 4.0 * a4)));
        }
    }
    if (JAC) warp_sum3<LPC>(S, cp, dcp, lane);
    else warp_sum2<LPC>(S, cp, lane);
    cp *= kR;
    const double Wbar = 1.0 / S;
    const double rho = p * invT * Wbar * (1.0 / kR);
    // FP64 mode: 1 / rho without another division. The mixed mode keeps every FP64 rounding as it is
    // (see stage_add)
    const double invrho = MX ? 1.0 / rho : Rinvp * (T * S);
    info.rho = rho;
    info.cp = cp;
    info.dcpdT = JAC ? dcp * kR : 0.0;
    info.Wbar = Wbar;
    if (wr) {
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int c = lane + 32 * s;
            if (c >= 1 && c < n) {
                const double C = rho * yw_s[s];
                sh.C[c - 1] = C;
                if (MX) sh.Cf[c - 1] = f64_to_f32_trunc(C);
            }
        }
        if (lane == 0) {                             // the absent species, the absent reaction
            sh.C[N] = 1.0;
            sh.g[N] = 0.0;
            sh.H[N] = 0.0;
            sh.rq[R] = 0.0;
            if (JAC) sh.rdqT[R] = 0.0;
        }
    }
    tm.sync();
    // reaction pass (thread per reaction over the team's lanes)
    const double lnPRT = m.lnPR - lnT;
    for (int j = tm.wt * 32 + lane; j < R; j += LPC * W) {
        const uint2 sp = __ldg(m.rspec + j);
        const int r0 = sp.x & 255, r1 = (sp.x >> 8) & 255, p0 = sp.y & 255, p1 = (sp.y >> 8) & 255;
        const double beta = __ldg(m.beta + j), EaR = __ldg(m.EaR + j);
        const double lnkf = __ldg(m.lnA + j) + beta * lnT - EaR * invT;
        const double kf = MX ? exp_mx(lnkf) : exp(lnkf);
        double lnKp = sh.g[p0] - sh.g[r0];
        lnKp += sh.g[p1];
        lnKp -= sh.g[r1];
        double C0 = sh.C[r0], C1 = sh.C[r1], D0 = sh.C[p0], D1 = sh.C[p1];
        double Pf = C0 * C1, Pr = D0 * D1, C2 = 1.0, D2 = 1.0;
        const int r2 = (sp.x >> 16) & 255, p2 = (sp.y >> 16) & 255;
        if (m.three) {
            C2 = sh.C[r2];
            D2 = sh.C[p2];
            lnKp += sh.g[p2];
            lnKp -= sh.g[r2];
            Pf *= C2;
            Pr *= D2;
        }
        const double dnu = __ldg(m.dnu_d + j);
        // k_r = k_f / K_c, ln K_c = ln K_p + dnu ln(P_std / RT)
        const double kr = MX ? exp_mx(lnkf - lnKp - dnu * lnPRT) : exp(lnkf - lnKp - dnu * lnPRT);
        const int type = __ldg(m.rtype + j);
        const double dlnkf = (beta + EaR * invT) * invT;
        double F = 1.0, dFdC = 0.0, dFdT = 0.0;
        if (type != 0) {
            double M = 0.0;
            if (MX) {
                const float *e = m.eff_f + (size_t)j * N;
                float Mf = 0.0f;
#pragma unroll 8
                for (int k = 0; k < N; ++k) Mf = fmaf(__ldg(e + k), sh.Cf[k], Mf);
                M = f32_to_f64_int(Mf);
            } else {
                const double *e = m.eff + (size_t)j * N;
#pragma unroll 8
                for (int k = 0; k < N; ++k) M += __ldg(e + k) * sh.C[k];
            }
            if (type == 1) {
                F = M;
                dFdC = 1.0;
            } else {
                const double beta0 = __ldg(m.beta0 + j), Ea0R = __ldg(m.Ea0R + j);
                const double lr = __ldg(m.lnA0 + j) + beta0 * lnT - Ea0R * invT - lnkf;
                const double ratio = MX ? exp_mx(lr) : exp(lr);   // k0 / k_inf
                double Prd = M * ratio;
                if (Prd < 1e-300) Prd = 1e-300;
                double Ft, glg, dFtdT;
                if (MX) {
                    float Ff, gf, df;
                    troe_F_f32(m.troe_r + 4 * j, f64_to_f32_trunc(T), f64_to_f32_trunc(invT),
                               fmaxf(f64_to_f32_trunc(Prd), 1e-37f), Ff, gf, df);
                    Ft = f32_to_f64_int(Ff);
                    glg = f32_to_f64_int(gf);
                    dFtdT = f32_to_f64_int(df);
                } else {
                    troe_F(m.troe_r + 4 * j, T, invT, Prd, Ft, glg, dFtdT);
                }
                const double ip = 1.0 / (1.0 + Prd);
                const double blend = Prd * ip;
                F = blend * Ft;
                if (JAC) {
                    const double dF_dPrd = Ft * ip * (ip + glg);
                    dFdC = dF_dPrd * ratio;
                    const double dlnk0 = (beta0 + Ea0R * invT) * invT;
                    dFdT = dF_dPrd * Prd * (dlnk0 - dlnkf) + blend * dFtdT;
                }
            }
        }
        const double rop = fma(kf, Pf, -__dmul_rn(kr, Pr));
        double q = rop;
        if (type != 0) q = F * rop;
        sh.rq[j] = q;
        if (JAC) {
            double dH = sh.H[p0] - sh.H[r0];
            dH += sh.H[p1];
            dH -= sh.H[r1];
            if (m.three) {
                dH += sh.H[p2];
                dH -= sh.H[r2];
            }
            const double dlnKc = (dH - dnu) * invT;
            const double dkfdT = kf * dlnkf, dkrdT = kr * (dlnkf - dlnKc);
            double dq = dkfdT * Pf - dkrdT * Pr;
            if (type != 0) {
                dq = F * dq + rop * dFdT;
                sh.rc3[j] = rd<mreal>(rop * dFdC);
            }
            sh.rdqT[j] = dq;
            // d q / d C_l through the mass-action products, for the distinct species l
            mreal *o = sh.rdq + (size_t)j * m.nslot;
            auto put = [&](int u, double d) { o[u] = rd<mreal>(type != 0 ? F * d : d); };
            if (sp.x >> 24) {                        // every species once, in slot order
                put(0, kf * (m.three ? C1 * C2 : C1));
                int u = 1;
                if (r1 < N) put(u++, kf * (m.three ? C0 * C2 : C0));
                if (m.three && r2 < N) put(u++, kf * (C0 * C1));
                if (p0 < N) put(u++, -(kr * (m.three ? D1 * D2 : D1)));
                if (p1 < N) put(u++, -(kr * (m.three ? D0 * D2 : D0)));
                if (m.three && p2 < N) put(u++, -(kr * (D0 * D1)));
            } else {
                for (int u = 0; u < 6; ++u) {
                    const int l = __ldg(m.rsp + 6 * j + u);
                    if (l < 0) break;
                    double dPf = 0.0, dPr = 0.0;
                    if (r0 == l) dPf += C1 * C2;
                    if (r1 == l) dPf += C0 * C2;
                    if (r2 == l) dPf += C0 * C1;
                    if (p0 == l) dPr += D1 * D2;
                    if (p1 == l) dPr += D0 * D2;
                    if (p2 == l) dPr += D0 * D1;
                    put(u, kf * dPf - kr * dPr);
                }
            }
        }
    }
    tm.sync();
    // species gather: wdot_k = sum_j nu_kj q_j (reactions ascending). Lists are padded with the absent reaction: a rate
    // that is not finite reaches its own species only
    double w[NS], wt[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const unsigned *lst = m.gath + lane + 32 * s - 1;    // species c - 1
        const bool on = lane + 32 * s >= 1 && lane + 32 * s < n;
        w[s] = 0.0;
        wt[s] = 0.0;
        if (on)
            for (int t = 0; t < m.gath_len; t += 4) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const unsigned e = __ldg(lst + (t + u) * 64);
                    const double nu = code_value<double>(e);
                    w[s] += nu * sh.rq[e & 0xFFFFu];
                    if (JAC) wt[s] += nu * sh.rdqT[e & 0xFFFFu];
                }
            }
    }
    double Q = 0.0;
    const double RT = kR * T;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const int c = lane + 32 * s;
        if (c >= 1 && c < n) {
            const int k = c - 1;
            const double Wk = __ldg(m.W + k);
            const double H = sh.H[k];
            if (JAC && wr) {
                sh.wdot[k] = rd<mreal>(w[s]);
                sh.wT[k] = rd<mreal>(wt[s]);
                sh.U[k] = rd<mreal>(Wk * invrho);
                sh.V[k] = rd<mreal>(Wk * w[s] * Wbar * invrho);
                sh.HR[k] = rd<mreal>(H) * ((mreal)kR * rd<mreal>(T));
            }
            f[s] = Wk * w[s] * invrho;
            Q += H * RT * w[s];
        }
    }
    Q = warp_sum<LPC>(Q);
    info.Q = Q;
    if (lane == 0) f[0] = MX ? -Q / (rho * cp) : -(Q * invrho) / cp;
    return info;
}

// a b + c d and a b - c d with the first product rounded; FP32 written out, so that the mixed mode's
// results do not depend on how the compiler contracts sums of two products (a last-bit change of the
// matrix moves T by up to 1e-8 relative in a step)
__device__ __forceinline__ float mul_add(float a, float b, float c, float d) { return fmaf(c, d, __fmul_rn(a, b)); }
__device__ __forceinline__ double mul_add(double a, double b, double c, double d) { return a * b + c * d; }
__device__ __forceinline__ float mul_sub(float a, float b, float c, float d) { return fmaf(-c, d, __fmul_rn(a, b)); }
__device__ __forceinline__ double mul_sub(double a, double b, double c, double d) { return a * b - c * d; }

// G = I/(h g) - J from the data of eval_rhs<JAC> (the FP64 matrix, or in the mixed mode an FP32 one:
// the Jacobian then carries FP32 rounding, about 1e-7 relative, which the mixed mode's loose
// tolerances absorb). In a team the entry lists and the third-body rows are split over the warps and
// the first warp does the rest.
template <int W, int NS, bool MX, int LPC = 32>
__device__ void build_matrix(const DevMech &m, const Slice<MX> &sh, Team<W> tm, int lane, const EvalInfo &in, double ih) {
    using real = typename Slice<MX>::mreal;
    const int N = m.N, n = N + 1;
    real *G = sh.G;
    if (!MX) tm.sync();                      // FP64: the matrix may share its space with the rates read above
    for (int r = 1 + tm.wt; r < n; r += W) { // zero the species block
#pragma unroll
        for (int s = 0; s < NS; ++s)
            if (lane + 32 * s < n) G[r * n + lane + 32 * s] = 0;
    }
    tm.sync();
    // sparse part of JC = d wdot / d C: an entry per lane, its reactions ascending
    const unsigned *ell = MX ? m.ell_f : m.ell_d;
    for (int q = tm.wt; q < m.ell_groups; q += W) {
        const int len = __ldg(m.ell_len + q);
#pragma unroll
        for (int half = 0; half < 32; half += LPC) {
            const int pos = __ldg(m.ell_pos + 32 * q + half + lane);
            const unsigned *p = ell + __ldg(m.ell_off + q) + half + lane;
            real acc = 0;
            for (int t = 0; t < len; ++t) {
                const unsigned e = __ldg(p + 32 * t);
                if (e >> 16) acc += code_value<real>(e) * sh.rdq[e & 0xFFFFu];
            }
            if (pos >= 0) G[pos] = acc;
        }
    }
    tm.sync();
    // dense third-body part: row k takes nu_kj (rop dF/dM)_j eff_j of its reactions j, columns over lanes
    if (m.n_tb > 0) {
        const unsigned *tbc = MX ? m.tbrow_f : m.tbrow_d;
        for (int k = tm.wt; k < N; k += W) {
            const int b = __ldg(m.tbrow_ptr + k), e = __ldg(m.tbrow_ptr + k + 1);
            if (b == e) continue;
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int c = lane + 32 * s;
                if (c >= 1 && c < n) {
                    real acc = G[(1 + k) * n + c];
                    for (int t = b; t < e; ++t) {
                        const unsigned w = __ldg(tbc + t);
                        const int j = w & 0xFFFFu;
                        real ef;
                        if constexpr (MX) ef = __ldg(m.eff_f + (size_t)j * N + c - 1);
                        else ef = __ldg(m.eff + (size_t)j * N + c - 1);
                        acc += code_value<real>(w) * (sh.rc3[j] * ef);
                    }
                    G[(1 + k) * n + c] = acc;
                }
            }
        }
        tm.sync();
    }
    if (tm.lead()) {
        // JCC[k] = sum_l JC[k][l] C_l (row owners)
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int c = lane + 32 * s;
            if (c >= 1 && c < n) {
                real acc = 0;
                for (int l = 0; l < N; ++l) {
                    real C;
                    if constexpr (MX) C = sh.Cf[l];
                    else C = sh.C[l];
                    acc += G[c * n + 1 + l] * C;
                }
                sh.JCC[c - 1] = acc;
            }
        }
        __syncwarp();
        // chain rule through C(T, Y) and rho(T, Y); then G = I/(h g) - J
        const real invT = rd<real>(in.invT), cp = rd<real>(in.cp), Wbar = rd<real>(in.Wbar);
        const real Q = rd<real>(in.Q), rho = rd<real>(in.rho), dcpdT = rd<real>(in.dcpdT);
        const real invrcp = (real)1 / (rho * cp);
        const real qq = Q * invrcp / cp;              // Q / (rho cp^2)
        const real Rr = (real)kR;
        const real ghinv = rd<real>(ih * (1.0 / kGam));         // 1 / (h g), g a power of two
        real sT = 0;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int c = lane + 32 * s;
            if (c < 1 || c >= n) continue;
            // species column c (column owner)
            const int mm = c - 1;
            const real iWm = rd<real>(__ldg(m.f64.invW + mm));
            const real a = rho * iWm, b = Wbar * iWm;
            real sTr = 0;
            for (int k = 0; k < N; ++k) {
                real *g = G + (size_t)(1 + k) * n + c;
                const real dw = mul_add(-b, sh.JCC[k], *g, a);
                sTr += sh.HR[k] * dw;
                const real J = mul_add(sh.U[k], dw, sh.V[k], iWm);
                *g = (1 + k == c) ? ghinv - J : -J;
            }
            G[c] = mul_add(qq * mul_sub(cp, Wbar, sh.cpR[mm], Rr), iWm, sTr, invrcp);   // -J[0][c]
            // temperature column entry of row c (row owner)
            const real dwdT = sh.wT[mm] - sh.JCC[mm] * invT;
            const real Um = sh.U[mm], wm = sh.wdot[mm];
            G[(size_t)c * n] = -mul_add(Um * wm, invT, Um, dwdT);
            sT += mul_add(sh.cpR[mm] * Rr, wm, sh.HR[mm], dwdT);
        }
#pragma unroll
        for (int o = LPC / 2; o > 0; o >>= 1) sT += __shfl_xor_sync(kFull, sT, o);
        if (lane == 0) G[0] = ghinv + sT * invrcp + qq * (cp * invT - dcpdT);
    }
    tm.sync();
}

// The largest of the lanes' non-negative values (FP32 or FP64 patterns compare as integers) among those
// with `valid`, the smallest `pos` among equals: the lane that holds it, or -1 when it is zero, not
// finite or none is valid.
__device__ __forceinline__ int pivot_lane(float v, bool valid, int pos, int lane) {
    const unsigned key = valid && v == v ? __float_as_uint(v) : 0u;
    const unsigned top = __reduce_max_sync(kFull, key);
    if (top == 0u || top >= 0x7F800000u) return -1;
    const bool cand = valid && key == top;
    const unsigned first = __reduce_min_sync(kFull, cand ? (unsigned)pos : 64u);
    return __ffs(__ballot_sync(kFull, cand && (unsigned)pos == first)) - 1;
}
__device__ __forceinline__ int pivot_lane(double v, bool valid, int pos, int lane) {
    valid = valid && v == v;
    const unsigned hi = valid ? (unsigned)__double2hiint(v) : 0u, lo = (unsigned)__double2loint(v);
    const unsigned top = __reduce_max_sync(kFull, hi);
    if (top >= 0x7FF00000u) return -1;
    const unsigned low = __reduce_max_sync(kFull, valid && hi == top ? lo : 0u);
    if ((top | low) == 0u) return -1;
    const bool cand = valid && hi == top && lo == low;
    const unsigned first = __reduce_min_sync(kFull, cand ? (unsigned)pos : 64u);
    return __ffs(__ballot_sync(kFull, cand && (unsigned)pos == first)) - 1;
}

// The same over 16 lanes (both halves of the warp at once): values as 64-bit keys, four shuffle steps.
__device__ __forceinline__ int pivot_lane16(unsigned long long key, int pos, int lane) {
    unsigned long long best = key;
    int first = key ? pos : 64;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
        const unsigned long long ob = __shfl_xor_sync(kFull, best, o);
        const int of = __shfl_xor_sync(kFull, first, o);
        if (ob > best || (ob == best && of < first)) {
            best = ob;
            first = of;
        }
    }
    const unsigned who = __ballot_sync(kFull, key == best && pos == first && key != 0);
    return (best == 0 || first == 64) ? -1 : __ffs((who >> (threadIdx.x & 16)) & 0xFFFFu) - 1;
}
__device__ __forceinline__ int pivot_lane16(double v, bool valid, int pos, int lane) {
    const unsigned long long k = (unsigned long long)__double_as_longlong(v);
    const int p = pivot_lane16(valid && k <= 0x7FF0000000000000ull ? k : 0ull, pos, lane);   // NaN: no candidate
    const double top = __shfl_sync(kFull, v, p < 0 ? 0 : p, 16);
    return p < 0 || __double2hiint(top) >= 0x7FF00000 ? -1 : p;
}
__device__ __forceinline__ int pivot_lane16(float v, bool valid, int pos, int lane) {
    const unsigned k = __float_as_uint(v);
    const int p = pivot_lane16(valid && k <= 0x7F800000u ? (unsigned long long)k : 0ull, pos, lane);
    const float top = __shfl_sync(kFull, v, p < 0 ? 0 : p, 16);
    return p < 0 || __float_as_uint(top) >= 0x7F800000u ? -1 : p;
}

// LU with partial pivoting of an n x n matrix, n <= NC <= 32, in registers: lane i holds row i of the
// matrix, then (moved once, after the factorisation) the factors' row of its pivoted place i.
template <typename real, int NC, int LPC = 32>
struct RowLU {
    real row[NC];
    real rinv;                 // reciprocal pivot of this lane's row
    int mine;                  // the row of the matrix that this lane's factors come from

    __device__ __forceinline__ bool factor(const real *G, int lane, int n) {
#pragma unroll
        for (int c = 0; c < NC; ++c) row[c] = (lane < n && c < n) ? G[lane * n + c] : (real)0;
        int pos = lane;            // place of this lane's row
        mine = lane;
        rinv = 0;
        bool ok = true;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            if (k < n && (LPC == 16 || ok)) {
                int p;
                if constexpr (LPC == 16) {
                    p = pivot_lane16((real)fabs(row[k]), pos >= k && lane < n, pos, lane);
                    if (p < 0) { ok = false; p = 0; }     // the other half goes on: this one's result is not used
                } else {
                    p = pivot_lane((real)fabs(row[k]), pos >= k && lane < n, pos, lane);
                }
                if (p < 0) {
                    ok = false;
                } else {
                    const int was = __shfl_sync(kFull, pos, p, LPC);
                    if (pos == k) pos = was;          // the row that stood there takes the pivot's place
                    if (lane == p) pos = k;
                    if (lane == k) mine = p;
                    const real rp = (real)1 / __shfl_sync(kFull, row[k], p, LPC);
                    if (lane == p) rinv = rp;
                    const bool below = pos > k;
                    if (below) row[k] *= rp;
#pragma unroll
                    for (int cb = (k + 1) & ~3; cb < NC; cb += 4) {
                        if (cb < n) {
#pragma unroll
                            for (int c = cb; c < cb + 4; ++c)
                                if (c > k) {
                                    const real akc = __shfl_sync(kFull, row[c], p, LPC);
                                    if (below) row[c] -= row[k] * akc;
                                }
                        }
                    }
                }
            }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (c < n) row[c] = __shfl_sync(kFull, row[c], mine, LPC);
        rinv = __shfl_sync(kFull, rinv, mine, LPC);
        if constexpr (sizeof(real) == 8) {
            // FP64: the rows of U divided by their pivots once, instead of each unknown in every solve
#pragma unroll
            for (int k = 1; k < NC; ++k)
                if (lane < k) row[k] *= rinv;
        }
        return ok;
    }

    // x = A^-1 b, component c in lane c
    __device__ __forceinline__ real solve(real b, int lane, int n) const {
        b = __shfl_sync(kFull, b, mine, LPC);
#pragma unroll
        for (int k = 0; k < NC - 1; ++k) {
            if (k < n - 1) {
                const real bk = __shfl_sync(kFull, b, k, LPC);
                if (lane > k) b -= row[k] * bk;
            }
        }
        if constexpr (sizeof(real) == 8) b *= rinv;
#pragma unroll
        for (int k = NC - 1; k >= 0; --k) {
            if (k < n) {
                if constexpr (sizeof(real) == 4) {
                    if (lane == k) b *= rinv;
                }
                const real bk = __shfl_sync(kFull, b, k, LPC);
                if (lane < k) b -= row[k] * bk;
            }
        }
        return b;
    }
};

// b <- G^-1 b with the factors G, invd in shared memory (n > 32); b is lane-distributed, bsw this
// warp's own buffer.
template <typename real>
__device__ void tri_solve(const int *piv, const real *G, const real *invd, real *bsw, int lane, int n, real (&b)[2]) {
    for (int s = 0; s < 2; ++s) {
        const int c = lane + 32 * s;
        if (c < n) bsw[c] = b[s];
    }
    __syncwarp();
    if (lane == 0) {
        for (int k = 0; k < n; ++k) {
            const int p = piv[k];
            if (p != k) { const real t = bsw[k]; bsw[k] = bsw[p]; bsw[p] = t; }
        }
    }
    __syncwarp();
    for (int s = 0; s < 2; ++s) {
        const int c = lane + 32 * s;
        b[s] = (c < n) ? bsw[c] : (real)0;
    }
    for (int k = 0; k < n - 1; ++k) {
        const real bk = __shfl_sync(kFull, k >> 5 ? b[1] : b[0], k & 31);
        for (int s = 0; s < 2; ++s) {
            const int i = lane + 32 * s;
            if (i > k && i < n) b[s] -= G[i * n + k] * bk;
        }
    }
    for (int k = n - 1; k >= 0; --k) {
        if ((k & 31) == lane) {
            if (k >> 5) b[1] *= invd[k];
            else b[0] *= invd[k];
        }
        const real bk = __shfl_sync(kFull, k >> 5 ? b[1] : b[0], k & 31);
        for (int s = 0; s < 2; ++s) {
            const int i = lane + 32 * s;
            if (i < k) b[s] -= G[i * n + k] * bk;
        }
    }
    __syncwarp();
}

// The factored system of one step: NC <= 32 in registers, NC = 64 in shared memory.
template <int W, int NC, bool MX, int LPC = 32>
struct Factors {
    using real = typename Slice<MX>::mreal;
    static constexpr bool kBig = NC > 32;
    typename std::conditional<kBig, int, RowLU<real, kBig ? 4 : NC, LPC>>::type lu;

    __device__ __forceinline__ bool factor(const Slice<MX> &sh, Team<W> tm, int lane, int n) {
        if constexpr (kBig) {
            if (MX) {                        // the matrix is kept for the refinement; its factors take rdq's space
                for (int r = tm.wt; r < n; r += W)
                    for (int c = lane; c < n; c += 32) sh.F[r * n + c] = sh.G[r * n + c];
                tm.sync();
            }
            return lu_factor<Team<W>, real>(sh.piv, sh.F, sh.invd, tm, lane, n);
        } else {
            return lu.factor(sh.G, lane, n);
        }
    }
    template <int NS>
    __device__ __forceinline__ void tri(const Slice<MX> &sh, real *buf, int lane, int n, real (&v)[NS]) const {
        if constexpr (kBig) tri_solve<real>(sh.piv, sh.F, sh.invd, buf, lane, n, v);
        else v[0] = lu.solve(v[0], lane, n);
    }
    // b <- A^-1 b. The mixed mode: x = Gf^-1 b with the FP32 factors, then one step of iterative
    // refinement, r = b - G x in FP64 arithmetic and x += Gf^-1 r. The correction solves the residual to
    // FP32's relative accuracy, so the refined x carries about cond(G) 2^-24 times that error. The
    // conversions between FP64 and FP32 run on the integer pipe (truncation; magnitudes below 2^-126
    // become 0). A matrix with an infinity or a NaN has no finite pivot or solution, whatever the
    // conversion of finite values makes of it.
    template <int NS>
    __device__ __forceinline__ void solve(const Slice<MX> &sh, double *xs, int lane, int n, double (&b)[NS]) const {
        if constexpr (!MX) {
            tri(sh, xs, lane, n, b);
        } else {
            double x[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) x[s] = 0.0;
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {
                float v[NS];
#pragma unroll
                for (int s = 0; s < NS; ++s) v[s] = f64_to_f32_trunc(b[s]);
                tri(sh, reinterpret_cast<float *>(xs), lane, n, v);
                if (pass == 1) {
#pragma unroll
                    for (int s = 0; s < NS; ++s) b[s] = x[s] + f32_to_f64_int(v[s]);
                    break;
                }
                __syncwarp();
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    const int c = lane + 32 * s;
                    x[s] = f32_to_f64_int(v[s]);
                    if (c < n) xs[c] = x[s];
                }
                __syncwarp();
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    const int c = lane + 32 * s;
                    if (c < n) {
                        const float *row = sh.G + (size_t)c * n;
                        double acc = b[s];
#pragma unroll 4
                        for (int j = 0; j < n; ++j) acc = fma(-f32_to_f64_finite(row[j]), xs[j], acc);
                        b[s] = acc;
                    } else {
                        b[s] = 0.0;
                    }
                }
                __syncwarp();
            }
        }
    }
};

// v + c k, a term of the right-hand sides of stages 3 and 4. In the mixed mode the product is rounded before it
// is added (the FP64 mode fuses it): the mode's exponentials cut their FP64 arguments to FP32, so where a
// last-bit change moves an argument across a cut, a rate jumps by 2e-6 and T by up to 6e-8. Fused here, one
// step of h0 = 1e-9 differs by 1e-16 of T, but 20,000 integrations at rtol 1e-2 by up to 2e-7 of T and 4e-7 of a
// species' maximum. Every rounding of that mode is therefore written out.
template <bool MX>
__device__ __forceinline__ double stage_add(double v, double c, double k) {
    if constexpr (MX) return __dadd_rn(v, __dmul_rn(c, k));
    else return v + c * k;
}

// Integrates cells popped from the work queue until it is exhausted; W warps per cell. MX: the
// mixed mode (FP32 rate exponentials and fall-off blending; FP32 LU with one FP64 refinement).
template <int W, int NC, bool MX>
__device__ __forceinline__ void integrate_cells(const DevMech &m, char *smem, int *blk_pos, int64_t limit, int64_t ld,
                                                double dt, const chem_ode_opts &o, double *__restrict__ Tg,
                                                const double *__restrict__ pg, double *__restrict__ Yg,
                                                int32_t *__restrict__ status, int32_t *__restrict__ nsteps_out,
                                                unsigned int *__restrict__ queue, const int32_t *__restrict__ list,
                                                int ok_status) {
    constexpr int NS = NC > 32 ? 2 : 1;
    constexpr bool BIG = NC > 32;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int N = m.N, n = N + 1;
    const size_t sb = make_slice<MX, BIG>(nullptr, N, m.R, m.n_tb, m.nslot, nullptr);
    Team<W> tm{W == 1 ? 0 : warp};
    // the team's shared data live in its first warp's slice; every warp keeps its own vector buffer
    Slice<MX> sh, own;
    make_slice<MX, BIG>(smem + (size_t)(W == 1 ? warp : 0) * sb, N, m.R, m.n_tb, m.nslot, &sh);
    make_slice<MX, BIG>(smem + (size_t)warp * sb, N, m.R, m.n_tb, m.nslot, &own);
    double *xs = own.xs;
    const double rn = 1.0 / (double)n;
    for (;;) {
        unsigned int pos = 0;
        if (W == 1) {
            if (lane == 0) pos = atomicAdd(queue, 1u);
            pos = __shfl_sync(kFull, pos, 0);
        } else {
            if (tm.lead() && lane == 0) *blk_pos = (int)atomicAdd(queue, 1u);
            tm.sync();
            pos = (unsigned int)*blk_pos;
            tm.sync();                       // every warp has its ticket before the next one is drawn
        }
        if ((int64_t)pos >= limit) break;
        const int64_t cell = list ? (int64_t)list[pos] : (int64_t)pos;
        double y[NS], f0[NS], K1[NS], K2[NS], K3[NS], K4[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int c = lane + 32 * s;
            y[s] = (c == 0) ? Tg[cell] : (c < n ? Yg[(int64_t)(c - 1) * ld + cell] : 0.0);
        }
        const double p = pg[cell], Rinvp = kR / p;
        double t = 0.0, h = (o.h0 < dt) ? o.h0 : dt;
        int nst = 0, rejected_last = 0, stat = CHEM_CELL_OK;
        while (t < dt) {
            if (nst >= o.max_steps) { stat = CHEM_CELL_MAXSTEPS; break; }
            if (h < 1e-20 * dt) { stat = CHEM_CELL_UNDERFLOW; break; }
            const double rem = dt - t;
            bool last = false;
            if (h >= rem) { h = rem; last = true; }
            const EvalInfo info = eval_rhs<W, NS, MX, true>(m, sh, tm, lane, p, Rinvp, y, f0);
            bool bad = false;
#pragma unroll
            for (int s = 0; s < NS; ++s)
                if (lane + 32 * s < n && !isfinite(f0[s])) bad = true;
            if (__any_sync(kFull, bad)) { stat = CHEM_CELL_NONFINITE; break; }
            const double ih = 1.0 / h;
            build_matrix<W, NS, MX>(m, sh, tm, lane, info, ih);
            ++nst;
            Factors<W, NC, MX> A;
            if (!A.factor(sh, tm, lane, n)) { h *= 0.2; rejected_last = 1; continue; }
#pragma unroll
            for (int s = 0; s < NS; ++s) K1[s] = K2[s] = K3[s] = K4[s] = 0.0;
            // stages 1 .. 4 in one body: the stage points are y, y, y + 2 K1, y + 2 K1 + K3
#pragma unroll 1
            for (int st = 0; st < 4; ++st) {
                double v[NS];
#pragma unroll
                for (int s = 0; s < NS; ++s) v[s] = f0[s];
                if (st >= 2) {
                    double ys[NS];
#pragma unroll
                    for (int s = 0; s < NS; ++s) ys[s] = y[s] + 2.0 * K1[s] + K3[s];
                    eval_rhs<W, NS, MX, false>(m, sh, tm, lane, p, Rinvp, ys, v);
                }
                if (st == 1) {
#pragma unroll
                    for (int s = 0; s < NS; ++s) v[s] = fma(kC21 * ih, K1[s], v[s]);
                }
                if (st >= 2) {
                    const double c1 = (st == 2 ? kC31 : kC41) * ih, c2 = (st == 2 ? kC32 : kC42) * ih;
                    const double c3 = (st == 3 ? kC43 : 0.0) * ih;
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        v[s] = stage_add<MX>(stage_add<MX>(v[s], c1, K1[s]), c2, K2[s]);
                        v[s] = fma(c3, K3[s], v[s]);
                    }
                }
                A.solve(sh, xs, lane, n, v);
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    if (st == 0) K1[s] = v[s];
                    else if (st == 1) K2[s] = v[s];
                    else if (st == 2) K3[s] = v[s];
                    else K4[s] = v[s];
                }
            }
            // y_new = y + 2 K1 + K3 + K4, error = K4
            double acc = 0.0, yn[NS];
            bool nonfinite = false;
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int c = lane + 32 * s;
                yn[s] = 0.0;
                if (c < n) {
                    double v = y[s];
                    v += 2.0 * K1[s];
                    v += K3[s];
                    v += K4[s];
                    yn[s] = v;
                    const double e = K4[s];
                    const double ay = fabs(y[s]), ayn = fabs(v);
                    const double sc = ((c == 0) ? o.atol_T : o.atol_Y) + o.rtol * (ay > ayn ? ay : ayn);
                    const double r = e / sc;
                    acc += r * r;
                    if (!isfinite(v) || !isfinite(e)) nonfinite = true;
                }
            }
            acc = warp_sum<32>(acc);
            nonfinite = __any_sync(kFull, nonfinite);
            // reformulated in the FP64 mode only (see stage_add)
            double err = sqrt(MX ? acc / (double)n : acc * rn);
            double fac;
            if (nonfinite || !isfinite(err)) {
                fac = 0.2;
                err = 2.0;
            } else {
                fac = (err > 0.0) ? 0.9 * (MX ? pow(err, -1.0 / 3.0) : rcbrt(err)) : 5.0;
                fac = fmin(5.0, fmax(0.2, fac));
            }
            if (err <= 1.0) {
                t = last ? dt : t + h;
#pragma unroll
                for (int s = 0; s < NS; ++s) y[s] = yn[s];
                if (rejected_last && fac > 1.0) fac = 1.0;
                h *= fac;
                rejected_last = 0;
            } else {
                h *= fac;
                rejected_last = 1;
            }
        }
        if (tm.lead()) {
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int c = lane + 32 * s;
                if (c == 0) Tg[cell] = y[s];
                else if (c < n) Yg[(int64_t)(c - 1) * ld + cell] = y[s];
            }
            if (lane == 0) {
                status[cell] = (stat == CHEM_CELL_OK) ? ok_status : stat;
                if (nsteps_out) nsteps_out[cell] = nst;
            }
        }
    }
}

// The same for n <= 16 with two cells per warp, one in each half (16 lanes): the FP64 pipe, which counts warp
// instructions, then serves two cells with each. The halves run their steps in lock step; one that
// has finished its cell (or finds its step rejected) goes on with its own next cell or step, so neither
// waits for the other's step count. Operations and orders per cell are those of integrate_cells.
template <int NC, bool MX>
__device__ __forceinline__ void integrate_halves(const DevMech &m, char *smem, int64_t limit, int64_t ld, double dt,
                                                 const chem_ode_opts &o, double *__restrict__ Tg,
                                                 const double *__restrict__ pg, double *__restrict__ Yg,
                                                 int32_t *__restrict__ status, int32_t *__restrict__ nsteps_out,
                                                 unsigned int *__restrict__ queue, const int32_t *__restrict__ list,
                                                 int ok_status) {
    static_assert(NC <= 16, "a cell's components in 16 lanes");
    const int lane = threadIdx.x & 15, slot = threadIdx.x >> 4;
    const unsigned half = 0xFFFFu << (threadIdx.x & 16);
    const int N = m.N, n = N + 1;
    const Team<1> tm{0};
    Slice<MX> sh;
    make_slice<MX, false>(smem + (size_t)slot * make_slice<MX, false>(nullptr, N, m.R, m.n_tb, m.nslot, nullptr), N, m.R,
                          m.n_tb, m.nslot, &sh);
    const double rn = 1.0 / (double)n;
    bool have = false, done = false;
    int64_t cell = 0;
    double y[1] = {lane == 0 ? 1000.0 : rn}, p = 101325.0, t = 0.0, h = dt;     // a state for an idle half to run on
    int nst = 0, rejected_last = 0, stat = CHEM_CELL_OK;
    for (;;) {
        if (!have && !done) {
            unsigned int pos = 0;
            if (lane == 0) pos = atomicAdd(queue, 1u);
            pos = __shfl_sync(half, pos, 0, 16);
            if ((int64_t)pos < limit) {
                cell = list ? (int64_t)list[pos] : (int64_t)pos;
                y[0] = (lane == 0) ? Tg[cell] : (lane < n ? Yg[(int64_t)(lane - 1) * ld + cell] : 0.0);
                p = pg[cell];
                t = 0.0;
                h = (o.h0 < dt) ? o.h0 : dt;
                nst = 0;
                rejected_last = 0;
                stat = CHEM_CELL_OK;
                have = true;
            } else {
                done = true;
            }
        }
        __syncwarp();
        if (__all_sync(kFull, done)) break;
        bool fin = false;
        if (have) {
            if (nst >= o.max_steps) { stat = CHEM_CELL_MAXSTEPS; fin = true; }
            else if (h < 1e-20 * dt) { stat = CHEM_CELL_UNDERFLOW; fin = true; }
        }
        if (!__any_sync(kFull, fin)) {
            const double rem = dt - t;
            bool last = false;
            if (h >= rem) { h = rem; last = true; }
            const double Rinvp = kR / p;
            double f0[1];
            const EvalInfo info = eval_rhs<1, 1, MX, true, 16>(m, sh, tm, lane, p, Rinvp, y, f0);
            const bool bad = (__ballot_sync(kFull, lane < n && !isfinite(f0[0])) & half) != 0;
            const double ih = 1.0 / h;
            build_matrix<1, 1, MX, 16>(m, sh, tm, lane, info, ih);
            Factors<1, NC, MX, 16> A;
            const bool ok = A.factor(sh, tm, lane, n);
            double K1 = 0.0, K2 = 0.0, K3 = 0.0, K4 = 0.0;
#pragma unroll 1
            for (int st = 0; st < 4; ++st) {
                double v[1] = {f0[0]};
                if (st >= 2) {
                    const double ys[1] = {y[0] + 2.0 * K1 + K3};
                    eval_rhs<1, 1, MX, false, 16>(m, sh, tm, lane, p, Rinvp, ys, v);
                }
                if (st == 1) v[0] = fma(kC21 * ih, K1, v[0]);
                if (st >= 2) {
                    const double c1 = (st == 2 ? kC31 : kC41) * ih, c2 = (st == 2 ? kC32 : kC42) * ih;
                    v[0] = stage_add<MX>(stage_add<MX>(v[0], c1, K1), c2, K2);
                    v[0] = fma((st == 3 ? kC43 : 0.0) * ih, K3, v[0]);
                }
                A.solve(sh, sh.xs, lane, n, v);
                if (st == 0) K1 = v[0];
                else if (st == 1) K2 = v[0];
                else if (st == 2) K3 = v[0];
                else K4 = v[0];
            }
            // y_new = y + 2 K1 + K3 + K4, error = K4
            double acc = 0.0, yn = 0.0;
            bool nonfinite = false;
            if (lane < n) {
                double v = y[0];
                v += 2.0 * K1;
                v += K3;
                v += K4;
                yn = v;
                const double ay = fabs(y[0]), ayn = fabs(v);
                const double sc = ((lane == 0) ? o.atol_T : o.atol_Y) + o.rtol * (ay > ayn ? ay : ayn);
                const double r = K4 / sc;
                acc = r * r;
                nonfinite = !isfinite(v) || !isfinite(K4);
            }
            acc = warp_sum<16>(acc);
            nonfinite = (__ballot_sync(kFull, nonfinite) & half) != 0;
            double err = sqrt(MX ? acc / (double)n : acc * rn);
            double fac;
            if (nonfinite || !isfinite(err)) {
                fac = 0.2;
                err = 2.0;
            } else {
                fac = (err > 0.0) ? 0.9 * (MX ? pow(err, -1.0 / 3.0) : rcbrt(err)) : 5.0;
                fac = fmin(5.0, fmax(0.2, fac));
            }
            if (have) {
                if (bad) {
                    stat = CHEM_CELL_NONFINITE;
                    fin = true;
                } else {
                    ++nst;
                    if (!ok) {
                        h *= 0.2;
                        rejected_last = 1;
                    } else if (err <= 1.0) {
                        t = last ? dt : t + h;
                        y[0] = yn;
                        if (rejected_last && fac > 1.0) fac = 1.0;
                        h *= fac;
                        rejected_last = 0;
                        fin = !(t < dt);
                    } else {
                        h *= fac;
                        rejected_last = 1;
                    }
                }
            }                                // an idle half's state stays as it is
        }
        if (fin) {
            if (lane == 0) {
                Tg[cell] = y[0];
                status[cell] = (stat == CHEM_CELL_OK) ? ok_status : stat;
                if (nsteps_out) nsteps_out[cell] = nst;
            } else if (lane < n) {
                Yg[(int64_t)(lane - 1) * ld + cell] = y[0];
            }
            have = false;
            t = 0.0;
            h = dt;
        }
        __syncwarp();
    }
}

// Blocks that take a cell each in team mode: one per SM (the first blocks of a
// grid are spread over the SMs), at most the grid.
inline int team_blocks(int sms, int blocks) { return sms < blocks ? sms : blocks; }

// Resident blocks the registers are budgeted for: the mixed mode (32 FP32 row registers) runs 16 warps
// per SM, the FP64 mode (64 row registers) 12; above 31 species shared memory decides (5 to 8 warps).
constexpr int stiff_min_blocks(int NC, bool MX) { return NC > 32 ? 1 : (MX ? 4 : 3); }
constexpr int kBigWarps = 8;         // most warps of a block above 31 species

// Cells 0..ncells-1, or (list != null) the *list_count cells list[0..) of a
// device-built queue; status of a successful cell = ok_status. When the cells
// number at most team_blocks, the first team_blocks blocks integrate them with
// kWarps warps per cell and the other blocks return at once; otherwise
// every warp takes cells of its own, from halves_from cells on one in each half.
template <int NC, bool MX>
__global__ void __launch_bounds__(NC > 32 ? 32 * kBigWarps : 32 * kWarps, stiff_min_blocks(NC, MX))
    stiff_kernel(const __grid_constant__ DevMech m, int64_t ncells, int64_t ld, double dt, chem_ode_opts o,
                 double *__restrict__ Tg, const double *__restrict__ pg, double *__restrict__ Yg,
                 int32_t *__restrict__ status, int32_t *__restrict__ nsteps_out, unsigned int *__restrict__ queue,
                 const int32_t *__restrict__ list, const unsigned int *__restrict__ list_count, int ok_status,
                 int team_blocks, int64_t halves_from) {
    extern __shared__ __align__(16) char smem_raw[];
    int *blk_pos = reinterpret_cast<int *>(smem_raw);
    char *smem = smem_raw + kSmemHeader;
    const int64_t limit = list ? (int64_t)(*list_count < (unsigned int)ncells ? *list_count : (unsigned int)ncells)
                               : ncells;
    if (limit <= (int64_t)team_blocks) {
        if ((int)blockIdx.x >= team_blocks || threadIdx.x >= 32 * kWarps) return;
        integrate_cells<kWarps, NC, MX>(m, smem, blk_pos, limit, ld, dt, o, Tg, pg, Yg, status, nsteps_out, queue,
                                        list, ok_status);
        return;
    }
    if constexpr (NC <= 16) {
        if (limit >= halves_from) {
            integrate_halves<NC, MX>(m, smem, limit, ld, dt, o, Tg, pg, Yg, status, nsteps_out, queue, list,
                                     ok_status);
            return;
        }
    }
    integrate_cells<1, NC, MX>(m, smem, blk_pos, limit, ld, dt, o, Tg, pg, Yg, status, nsteps_out, queue, list,
                               ok_status);
}

// The launch of one kernel variant: warps per block and resident blocks for this mechanism.
template <int NC, bool MX>
int launch_stiff_nc(const chem_mech *m, int64_t capacity, int64_t ld, double dt, const chem_ode_opts &o, double *T,
                    const double *p, double *Y, int32_t *status, int32_t *nsteps, unsigned int *queue,
                    const int32_t *list, const unsigned int *count, int ok_status, cudaStream_t st, const char *who) {
    constexpr size_t kSmemMax = 227 * 1024;
    const size_t slice = make_slice<MX, (NC > 32)>(nullptr, m->N, m->R, m->dev.n_tb, m->dev.nslot, nullptr);
    int warps = kWarps;
    // above 31 species one block of up to kBigWarps warps where two blocks of kWarps do not fit
    if (NC > 32 && 2 * (kSmemHeader + kWarps * slice) > kSmemMax)
        while (warps < kBigWarps && kSmemHeader + (warps + 1) * slice <= kSmemMax) ++warps;
    // two slices per warp, where they cost no resident block
    const bool halves = NC <= 16 && stiff_min_blocks(NC, MX) * (kSmemHeader + 2 * kWarps * slice) <= kSmemMax;
    const size_t smem = kSmemHeader + slice * (halves ? 2 * warps : warps);
    if (smem > kSmemMax)
        return set_error(CHEM_EUNSUPPORTED, std::string(who) + ": mechanism too large for shared memory");
    auto kernel = stiff_kernel<NC, MX>;
    // the largest size, once: launches of other mechanisms from other threads find it large enough
    static DeviceOnce configured;
    int rc = dynamic_smem_limit(configured, kernel, kSmemMax, who);
    if (rc) return rc;
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, warps * 32, smem);
    if (per_sm < 1) per_sm = 1;
    const int64_t need = (capacity + warps - 1) / warps;
    int blocks = (int)((int64_t)sms * per_sm < need ? (int64_t)sms * per_sm : need);
    if (!list && capacity <= sms) blocks = (int)capacity;      // one block (a team of warps) per cell
    if (blocks < 1) blocks = 1;
    rc = check_cuda(cudaMemsetAsync(queue, 0, sizeof(unsigned int), st), who);
    if (rc) return rc;
    // Two cells per warp from 5/4 cells per resident warp on. Below, a warp of its own ends each cell sooner
    // than the pipe, shared by fewer warps, gains. 9 species, one / two cells per warp: FP64 mode (1,824
    // warps) rtol 1e-6 1,824 cells 38.0 / 39.3 ms, 2,600 54.3 / 47.4, 16,384 261 / 169; mixed mode (2,432
    // warps) 2,600 cells 1.66 / 1.73 ms, 4,096 2.36 / 1.81, 16,384 8.2 / 5.1.
    const int64_t from = halves ? (int64_t)sms * per_sm * warps * 5 / 4 : INT64_MAX;
    kernel<<<blocks, warps * 32, smem, st>>>(m->dev, capacity, ld, dt, o, T, p, Y, status, nsteps, queue, list, count,
                                             ok_status, team_blocks(sms, blocks), from);
    return check_cuda(cudaGetLastError(), who);
}

// Stiff integration of cells 0..capacity-1 (list null) or of a device-built list; queue: a work-queue
// counter that this call clears on its stream. The mixed mode takes tolerances no tighter than
// kMixedMinRtol (its FP32 rates carry about 1e-6 relative noise).
int launch_stiff(const chem_mech *m, int64_t capacity, int64_t ld, double dt, const chem_ode_opts &o, double *T,
                 const double *p, double *Y, int32_t *status, int32_t *nsteps, unsigned int *queue,
                 const int32_t *list, const unsigned int *count, int ok_status, cudaStream_t st, const char *who) {
    const bool mx = o.mode == CHEM_ODE_MIXED && o.rtol >= kMixedMinRtol;
    const int n = m->N + 1;
#define CHEMGB_STIFF(NC_, MX_)                                                                                      \
    return launch_stiff_nc<NC_, MX_>(m, capacity, ld, dt, o, T, p, Y, status, nsteps, queue, list, count, ok_status, \
                                     st, who)
    if (n <= 16) {
        if (mx) CHEMGB_STIFF(16, true);
        CHEMGB_STIFF(16, false);
    }
    if (n <= 32) {
        if (mx) CHEMGB_STIFF(32, true);
        CHEMGB_STIFF(32, false);
    }
    if (mx) CHEMGB_STIFF(64, true);
    CHEMGB_STIFF(64, false);
#undef CHEMGB_STIFF
}

// PaSR scaling (Sec. 4.1), one warp per cell. The species times Y_k / |dY_k/dt| come from the
// reactor right-hand side at the state before the step (the same FP64 evaluation as the
// integrator's); tau_c is the largest over the species with Y_k >= y_min and a non-zero rate
// (the slowest formation rate), +inf when none qualifies; tau_mix = sqrt(tau_T tau_K);
// kappa = tau_c / (tau_c + tau_mix), 1 for an infinite tau_c. With T, Y given (the chemistry
// step's result), they become T0 + kappa (T - T0), Y0 + kappa (Y - Y0).
__host__ __device__ inline size_t pasr_slice_bytes(int N, int R) { return (size_t)(3 * (N + 1) + R + 1) * 8; }
template <int NS>
__global__ void __launch_bounds__(kWarps * 32) pasr_kernel(const __grid_constant__ DevMech m, int64_t ncells,
                                                            int64_t ld, double y_min, const double *__restrict__ T0,
                                                            const double *__restrict__ pg,
                                                            const double *__restrict__ Y0,
                                                            const double *__restrict__ tau_t,
                                                            const double *__restrict__ tau_k, double *__restrict__ T,
                                                            double *__restrict__ Y, double *__restrict__ tau_c_out,
                                                            double *__restrict__ kappa_out) {
    extern __shared__ __align__(16) char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int N = m.N, n = N + 1;
    Slice<false> sh{};
    sh.C = reinterpret_cast<double *>(smem_raw + (size_t)warp * pasr_slice_bytes(N, m.R));
    sh.g = sh.C + N + 1;
    sh.H = sh.g + N + 1;
    sh.rq = sh.H + N + 1;
    const Team<1> tm{0};
    for (int64_t cell = (int64_t)blockIdx.x * kWarps + warp; cell < ncells; cell += (int64_t)gridDim.x * kWarps) {
        double y[NS], f[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int c = lane + 32 * s;
            y[s] = (c == 0) ? T0[cell] : (c < n ? Y0[(int64_t)(c - 1) * ld + cell] : 0.0);
        }
        eval_rhs<1, NS, false, false>(m, sh, tm, lane, pg[cell], kR / pg[cell], y, f);
        double tmax = -1.0;                       // species times are >= 0: -1 marks none
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const int c = lane + 32 * s;
            if (c >= 1 && c < n) {
                const double r = fabs(f[s]);
                if (y[s] >= y_min && r > 0.0) tmax = fmax(tmax, y[s] / r);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tmax = fmax(tmax, __shfl_xor_sync(kFull, tmax, o));
        const double tau_c = (tmax >= 0.0) ? tmax : CUDART_INF;
        const double tau_mix = sqrt(tau_t[cell] * tau_k[cell]);
        const double kap = (tmax >= 0.0) ? tau_c / (tau_c + tau_mix) : 1.0;
        if (lane == 0) {
            if (tau_c_out) tau_c_out[cell] = tau_c;
            if (kappa_out) kappa_out[cell] = kap;
        }
        if (T && Y)
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const int c = lane + 32 * s;
                if (c == 0) T[cell] = y[s] + kap * (T[cell] - y[s]);
                else if (c < n) {
                    const int64_t q = (int64_t)(c - 1) * ld + cell;
                    Y[q] = y[s] + kap * (Y[q] - y[s]);
                }
            }
    }
}

}  // namespace
}  // namespace chemgb

using namespace chemgb;

extern "C" int chem_pasr(const chem_mech *m, int64_t ncells, int64_t ld, double y_min, const double *T0,
                         const double *p, const double *Y0, const double *tau_taylor, const double *tau_kolmogorov,
                         double *T, double *Y, double *tau_c, double *kappa, chem_stream_t stream) {
    if (!m) return set_error(CHEM_EINVAL, "chem_pasr: null mechanism");
    if (ncells < 0 || ld < ncells || (ld & 3) != 0 || ncells > (int64_t)0x7fffffff)
        return set_error(CHEM_EINVAL, "chem_pasr: need 0 <= ncells <= ld < 2^31, ld a multiple of 4");
    if (!(y_min > 0.0)) return set_error(CHEM_EINVAL, "chem_pasr: y_min must be positive");
    if (m->N > 63) return set_error(CHEM_EUNSUPPORTED, "chem_pasr: at most 63 species");
    if (ncells == 0) return CHEM_OK;
    if (!T0 || !p || !Y0 || !tau_taylor || !tau_kolmogorov) return set_error(CHEM_EINVAL, "chem_pasr: null input");
    if ((T == nullptr) != (Y == nullptr)) return set_error(CHEM_EINVAL, "chem_pasr: give both T and Y or neither");
    const void *ptrs[] = {T0, p, Y0, tau_taylor, tau_kolmogorov, T, Y, tau_c, kappa};
    for (const void *q : ptrs)
        if (q && !aligned16(q)) return set_error(CHEM_EINVAL, "chem_pasr: arrays must be 16-byte aligned");
    std::string why;
    if (!device_ok(&why)) return set_error(CHEM_EUNSUPPORTED, "chem_pasr: " + why);
    const size_t smem = pasr_slice_bytes(m->N, m->R) * kWarps;
    if (smem > 227 * 1024) return set_error(CHEM_EUNSUPPORTED, "chem_pasr: mechanism too large for shared memory");
    auto kernel = m->N <= 31 ? pasr_kernel<1> : pasr_kernel<2>;
    static DeviceOnce configured[2];
    int rc = dynamic_smem_limit(configured[m->N > 31], kernel, 227 * 1024, "chem_pasr: smem attribute");
    if (rc) return rc;
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kWarps * 32, smem);
    if (per_sm < 1) per_sm = 1;
    const int64_t need = (ncells + kWarps - 1) / kWarps;
    const int blocks = (int)((int64_t)sms * per_sm < need ? (int64_t)sms * per_sm : need);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    void *pb = prof_begin(st);
    kernel<<<blocks, kWarps * 32, smem, st>>>(m->dev, ncells, ld, y_min, T0, p, Y0, tau_taylor, tau_kolmogorov, T, Y,
                                              tau_c, kappa);
    prof_end(pb, st, "pasr_kernel", 0.0, (double)ncells * ((m->N + 2) * 8 + 2 * 8 + (T ? 2 * (m->N + 1) * 8 : 0)));
    return check_cuda(cudaGetLastError(), "chem_pasr launch");
}

extern "C" int chem_step_stiff(const chem_mech *m, int64_t ncells, int64_t ld, double dt, const chem_ode_opts *opts,
                               double *T, const double *p, double *Y, int32_t *status, int32_t *nsteps,
                               chem_stream_t stream) {
    if (!m) return set_error(CHEM_EINVAL, "chem_step_stiff: null mechanism");
    if (ncells < 0 || ld < ncells || (ld & 3) != 0 || ncells > (int64_t)0x7fffffff)
        return set_error(CHEM_EINVAL, "chem_step_stiff: need 0 <= ncells <= ld < 2^31, ld a multiple of 4");
    if (!(dt > 0.0)) return set_error(CHEM_EINVAL, "chem_step_stiff: dt must be positive");
    if (m->N > 63) return set_error(CHEM_EUNSUPPORTED, "chem_step_stiff: at most 63 species");
    if (ncells == 0) return CHEM_OK;
    if (!T || !p || !Y || !status) return set_error(CHEM_EINVAL, "chem_step_stiff: null array");
    const void *ptrs[] = {T, p, Y, status, nsteps};
    for (const void *q : ptrs)
        if (q && !aligned16(q)) return set_error(CHEM_EINVAL, "chem_step_stiff: arrays must be 16-byte aligned");
    chem_ode_opts o;
    chem_ode_opts_default(&o);
    if (opts) o = *opts;
    if (!(o.rtol > 0.0) || !(o.atol_Y > 0.0) || !(o.atol_T > 0.0) || !(o.h0 > 0.0) || o.max_steps < 1)
        return set_error(CHEM_EINVAL, "chem_step_stiff: tolerances, h0 and max_steps must be positive");
    if (o.mode != CHEM_ODE_FP64 && o.mode != CHEM_ODE_MIXED)
        return set_error(CHEM_EINVAL, "chem_step_stiff: mode must be CHEM_ODE_FP64 or CHEM_ODE_MIXED");
    std::string why;
    if (!device_ok(&why)) return set_error(CHEM_EUNSUPPORTED, "chem_step_stiff: " + why);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    void *pb = prof_begin(st);
    const int rc = launch_stiff(m, ncells, ld, dt, o, T, p, Y, status, nsteps, m->dev.counters, nullptr, nullptr,
                                CHEM_CELL_OK, st, "chem_step_stiff");
    prof_end(pb, st, "stiff_kernel", 0.0, 0.0);
    return rc;
}

namespace chemgb {
// Stiff integration of the cells a device queue lists (the fallback of the
// learned step): list[0..*count) with count <= capacity, status ok_status on
// success. Uses the mechanism's second work-queue counter.
int launch_stiff_list(const chem_mech *m, int64_t capacity, int64_t ld, double dt, const chem_ode_opts &o, double *T,
                      const double *p, double *Y, int32_t *status, const int32_t *list, const unsigned int *count,
                      int ok_status, cudaStream_t st) {
    if (m->N > 63) return set_error(CHEM_EUNSUPPORTED, "fallback: at most 63 species");
    return launch_stiff(m, capacity, ld, dt, o, T, p, Y, status, nullptr, m->dev.counters + 1, list, count, ok_status,
                        st, "fallback");
}
}  // namespace chemgb

// ---------------------------------------------------------------------------
// Allocation-free variant of chem_step_stiff.
//
// The regular entry point keeps its only global scratch (the work-queue
// counter) inside the mechanism handle. This variant keeps it in the
// file-scope array below instead, so a call neither allocates device memory
// nor writes into the handle. The array is 256 bytes (64 32-bit words) and
// every GPU that loads the library holds it until the process exits. A call
// uses word 0 as its queue counter and clears it first on its stream; calls
// that overlap on the GPU share that word and race.
// ---------------------------------------------------------------------------
namespace chemgb {
namespace {

constexpr int kNoAllocWords = 64;
// Largest ncells one call accepts: every resident warp takes one ticket past
// the last cell, so the 32-bit counter needs headroom below 2^32.
constexpr int64_t kNoAllocMaxCells = (int64_t)1 << 30;

static __device__ __align__(256) unsigned int g_noalloc_scratch[kNoAllocWords];

// Device address of g_noalloc_scratch for the current device, looked up once
// per device (with that device current). In host code the array's name is only
// a host-side stand-in, so kernels must be given this address.
int noalloc_scratch(unsigned int **out) {
    static std::mutex mu;
    static unsigned int *addr[64] = {nullptr};
    int dev = -1;
    int rc = check_cuda(cudaGetDevice(&dev), "chem_step_stiff_noalloc: cudaGetDevice");
    if (rc) return rc;
    if (dev < 0 || dev >= 64) return set_error(CHEM_EUNSUPPORTED, "chem_step_stiff_noalloc: device index above 63");
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void *p = nullptr;
        rc = check_cuda(cudaGetSymbolAddress(&p, g_noalloc_scratch), "chem_step_stiff_noalloc: cudaGetSymbolAddress");
        if (rc) return rc;
        addr[dev] = static_cast<unsigned int *>(p);
    }
    *out = addr[dev];
    return CHEM_OK;
}

}  // namespace
}  // namespace chemgb

extern "C" int chem_step_stiff_noalloc(const chem_mech *m, int64_t ncells, int64_t ld, double dt,
                                       const chem_ode_opts *opts, double *T, const double *p, double *Y,
                                       int32_t *status, int32_t *nsteps, chem_stream_t stream) {
    if (!m) return set_error(CHEM_EINVAL, "chem_step_stiff_noalloc: null mechanism");
    if (ncells < 0 || ld < ncells || (ld & 3) != 0)
        return set_error(CHEM_EINVAL, "chem_step_stiff_noalloc: need 0 <= ncells <= ld, ld a multiple of 4");
    if (ncells > kNoAllocMaxCells)
        return set_error(CHEM_EINVAL, "chem_step_stiff_noalloc: ncells exceeds the 2^30-cell limit of its static "
                                      "work-queue scratch");
    if (!(dt > 0.0)) return set_error(CHEM_EINVAL, "chem_step_stiff_noalloc: dt must be positive");
    if (m->N > 63) return set_error(CHEM_EUNSUPPORTED, "chem_step_stiff_noalloc: at most 63 species");
    if (ncells == 0) return CHEM_OK;
    if (!T || !p || !Y || !status) return set_error(CHEM_EINVAL, "chem_step_stiff_noalloc: null array");
    const void *ptrs[] = {T, p, Y, status, nsteps};
    for (const void *q : ptrs)
        if (q && !aligned16(q))
            return set_error(CHEM_EINVAL, "chem_step_stiff_noalloc: arrays must be 16-byte aligned");
    chem_ode_opts o;
    chem_ode_opts_default(&o);
    if (opts) o = *opts;
    if (!(o.rtol > 0.0) || !(o.atol_Y > 0.0) || !(o.atol_T > 0.0) || !(o.h0 > 0.0) || o.max_steps < 1)
        return set_error(CHEM_EINVAL, "chem_step_stiff_noalloc: tolerances, h0 and max_steps must be positive");
    std::string why;
    if (!device_ok(&why)) return set_error(CHEM_EUNSUPPORTED, "chem_step_stiff_noalloc: " + why);
    unsigned int *queue = nullptr;
    int rc = noalloc_scratch(&queue);
    if (rc) return rc;
    return launch_stiff(m, ncells, ld, dt, o, T, p, Y, status, nsteps, queue, nullptr, nullptr, CHEM_CELL_OK,
                        reinterpret_cast<cudaStream_t>(stream), "chem_step_stiff_noalloc");
}
