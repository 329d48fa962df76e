// internal.cuh -- device-side mechanism layout and helpers shared by the
// library's translation units (not part of the public ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "chemgb.h"
#include "device_once.h"

#define CHEMGB_STR2(x) #x
#define CHEMGB_STR(x) CHEMGB_STR2(x)

namespace chemgb {

constexpr double kR = 8.314462618;        // J/mol/K
constexpr int kMaxSpecies = 64;
constexpr int kMaxReactions = 4096;

// Device tables of one mechanism. Every pointer is device memory owned by the
// chem_mech handle. Square per-pair tables are stored row k, column j with a
// padded row length Np (a multiple of 4) so that rows start on 16 bytes.
template <typename real>
struct PropTables {
    const real *invW;      // [N] 1 / W_k
    const real *nasa_cp;   // [2][N][5] cp/R Horner coefficients, range 0 = low, 1 = high
    const real *nasa_h;    // [2][N][6] H/RT: a1, a2/2, a3/3, a4/4, a5/5, a6
    const real *visc;      // [N][5] ln mu_k polynomial in x = ln(T/1000)
    const real *wilke;     // [3][N][Np] T0 = c_kj, T1 = 2 c_kj w_jk, T2 = c_kj w_jk^2
    const real *diff;      // [N][Np][5]... stored as [5][N][Np]: coefficient n of g_jk at (k, j)
};

// Tables of the tensor-core properties pass (props.cu): the Wilke and binary-resistance coefficients
// as two FP16 terms (hi = fp16(v), lo = fp16(v - hi)) in the shared-memory layout of its B operand,
// [term 2][chunk of 8 species j][row][8], rows = NR rows of T1, then NP of T0 and of each of the five
// resistance coefficients, then NR of T2 (row r of a block = species k; NP = N to 8, NR = N to 16).
struct PropTcTables {
    const void *B;         // 2 x (K / 8) x rows x 16 bytes; null: coefficients that FP16 pairs cannot hold
    // [N][8]: c0 .. c4 of log2 r_k (r = sqrt(mu)) as a polynomial in x, its leading term less the
    // whole n; the reciprocal of the scaling of species k's resistance rows and of X; 2^n; 0
    const float *species;
    int rows, NP, NR;
};
constexpr int kTcMaxSpecies = 56;         // 2 NR + 6 NP columns fit TMEM and the operands shared memory
constexpr float kTcXScale = 16384.0f;     // X, X / r, X / r^2 (each at most 1 in magnitude) before rounding
constexpr float kTcWilkeScale = 1024.0f;  // Wilke tables (at most a few units)
inline int tc_k(int N) { return N <= 16 ? 16 : (N <= 32 ? 32 : 64); }   // padded contraction length

struct DevMech {
    int N, R, Np, n_tb;
    PropTcTables tc;
    double P_std, T_mid;
    PropTables<float> f32;
    PropTables<double> f64;
    // FP64 kinetics
    const double *W;        // [N]
    const int *rtype;       // [R] in device order: Troe fall-off, three-body, elementary, so a reaction with
                            // a third body is its own row of eff
    const double *lnA;      // [R]
    const double *beta;     // [R]
    const double *EaR;      // [R] Ea / R (K)
    const double *lnA0;     // [R]
    const double *beta0;    // [R]
    const double *Ea0R;     // [R]
    const double *troe;     // [R][4]
    const double *eff;      // [n_tb][N]
    // derived tables of the stiff integrator. "code" words hold a small integer as the high half of its
    // floating-point pattern (FP32 or the high word of FP64) in bits 16..31, an index in bits 0..15.
    const double *nasa_t;   // [2][17][64] per species (coalesced over lanes): cp/R 5, H/RT 6, S/R 6
    const double *dnu_d;    // [R] dnu as FP64
    const uint2 *rspec;     // [R] reactant species (bytes, N where absent), flags | product species, flags:
                            // byte 3 of x is 1 when every species of the reaction occurs once
    int nslot;              // distinct species of a reaction, at most (row length of d q / d C)
    int three;              // some reaction has a third reactant or product
    int gath_len;           // longest species incidence list, rounded up to 4
    const unsigned *gath;   // [gath_len][64] code: nu (FP64), reaction; pads: 0, R
    int ell_groups;         // groups of 32 entries of the sparse part of d wdot / d C, longest first
    const int *ell_off, *ell_len, *ell_pos;   // [groups] first word, iterations; [groups][32] matrix offset or -1
    const unsigned *ell_f, *ell_d;            // code: nu (FP32 / FP64), index in d q / d C [R][nslot]; 0 pads
    const int *tbrow_ptr;   // [N+1] third-body reactions of each species (net nu != 0), ascending
    const unsigned *tbrow_f, *tbrow_d;        // code: nu, third-body reaction
    const float *eff_f;     // [n_tb][N] eff cut to FP32
    const double *troe_r;   // [R][4] a, 1/T***, 1/T*, T**
    const int *rsp;         // [R][6] distinct species of reaction j (first-occurrence order), -1 pad
    double lnPR;            // ln(P_std / R)
    unsigned int *counters; // [kNumCounters] work-queue counters (scratch) and error words
};

constexpr int kNumCounters = 8;
constexpr int kPropsErrCounter = 7;       // props_eval: a pipeline wait ran out (its cells' outputs are NaN)

}  // namespace chemgb

struct chem_mech {
    int N, R, E, bath;
    double P_std, T_lo, T_mid, T_hi;
    chemgb::DevMech dev;
    void *blob;            // single device allocation holding every table
    size_t blob_bytes;
    int device;
    uint32_t wait_limit;   // tries of each pipeline wait of props_eval (chem_mech_set_wait_limit)
};

namespace chemgb {
int set_error(int code, const std::string &msg);
int check_cuda(cudaError_t e, const char *what);
// Opts a kernel into `bytes` of dynamic shared memory on the current device, once per device.
template <class Kernel>
inline int dynamic_smem_limit(DeviceOnce &once, Kernel *kernel, size_t bytes, const char *what) {
    int dev = -1;
    cudaGetDevice(&dev);
    return once.run(dev, [&] {
        return check_cuda(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes), what);
    });
}
// opt-in per-kernel timing (chem_prof_enable): events around tagged launches
bool prof_on();
void *prof_begin(cudaStream_t st);
void prof_end(void *begin, cudaStream_t st, const std::string &tag, double flops, double bytes);
bool device_ok(std::string *why);
inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Precision conversions by integer operations. On this part the FP64 pipe (which
// also converts between FP32 and FP64) runs at 1/64 of the FP32 rate, so the
// per-species conversions of the cell kernels are done on the integer pipe.
// FP64 -> FP32 by truncating the mantissa (relative error < 2^-23); magnitudes
// below 2^-126 become signed zero, at or above 2^128 infinity; NaN stays NaN.
// For |x| in range the FP32 bits are the double's high word with the exponent
// rebased (- (1023 - 127) << 20) and the 20 + 3 leading mantissa bits shifted
// into place, one funnel shift of the two words.
__device__ __forceinline__ float f64_to_f32_trunc(double x) {
    const unsigned int hi = static_cast<unsigned int>(__double2hiint(x));
    const unsigned int lo = static_cast<unsigned int>(__double2loint(x));
    const unsigned int a = hi & 0x7FFFFFFFu;
    unsigned int r = __funnelshift_l(lo, a - 0x38000000u, 3);      // exponent - 896, mantissa 23 bits
    r = (a < 0x38100000u) ? 0u : r;                                  // below 2^-126
    if (a >= 0x47F00000u)                                            // 2^128 and above, infinity, NaN
        r = (a > 0x7FF00000u || (a == 0x7FF00000u && lo != 0u)) ? 0x7FC00000u : 0x7F800000u;
    return __uint_as_float(r | (hi & 0x80000000u));
}
// FP32 -> FP64, exact for normal numbers and zero; FP32 subnormals (below 2^-126)
// become signed zero; infinities and NaN are kept.
__device__ __forceinline__ double f32_to_f64_int(float x) {
    const unsigned int b = __float_as_uint(x);
    const unsigned long long sign = static_cast<unsigned long long>(b & 0x80000000u) << 32;
    const unsigned int e = (b >> 23) & 0xFFu;
    if (e == 0) return __longlong_as_double(static_cast<long long>(sign));
    const unsigned long long ed = (e == 0xFFu) ? 0x7FFull : static_cast<unsigned long long>(e) + 896ull;
    const unsigned long long mant = static_cast<unsigned long long>(b & 0x7FFFFFu) << 29;
    return __longlong_as_double(static_cast<long long>(sign | (ed << 52) | mant));
}
// The same for a finite value.
__device__ __forceinline__ double f32_to_f64_finite(float x) {
    const unsigned b = __float_as_uint(x);
    const bool zero = (b & 0x7F800000u) == 0u;
    const unsigned hi = ((b & 0x7FFFFFFFu) >> 3) + 0x38000000u;
    return __hiloint2double((int)((zero ? 0u : hi) | (b & 0x80000000u)), (int)(zero ? 0u : b << 29));
}
}  // namespace chemgb
