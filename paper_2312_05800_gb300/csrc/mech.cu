// mech.cu -- mechanism loading (host parse, derived tables, one device blob),
// error reporting and option defaults of the C ABI.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <sstream>
#include <string>
#include <vector>

#include "internal.cuh"
#include "tc.cuh"

namespace chemgb {

static thread_local std::string g_last_error;

int set_error(int code, const std::string &msg) {
    g_last_error = msg;
    return code;
}

int check_cuda(cudaError_t e, const char *what) {
    if (e == cudaSuccess) return CHEM_OK;
    return set_error(CHEM_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

bool device_ok(std::string *why) {
    // cached per device: 1 = sm_103, 2 = other architecture
    static int state[64] = {0};
    static int cc[64] = {0};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) {
        cudaGetLastError();
        if (why) *why = "no CUDA device";
        return false;
    }
    if (dev < 64 && state[dev] == 0) {
        int major = 0, minor = 0;
        if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess) {
            cudaGetLastError();
            if (why) *why = "cannot query the device";
            return false;
        }
        cc[dev] = major * 10 + minor;
        state[dev] = (major == 10 && minor == 3) ? 1 : 2;
    }
    if (dev >= 64 || state[dev] != 1) {
        if (why) *why = "device is sm_" + std::to_string(dev < 64 ? cc[dev] : 0) +
                        "; this library is built for sm_103a only";
        return false;
    }
    return true;
}

namespace {

struct Reader {
    const uint8_t *p, *end;
    bool ok = true;
    template <typename T>
    void read(T *dst, size_t n) {
        size_t b = sizeof(T) * n;
        if (!ok || (size_t)(end - p) < b) { ok = false; return; }
        std::memcpy(dst, p, b);
        p += b;
    }
};

// Appends a typed array to the host image of the device blob (256-byte aligned).
struct BlobBuilder {
    std::vector<uint8_t> bytes;
    template <typename T>
    size_t add(const std::vector<T> &v) {
        size_t off = (bytes.size() + 255) & ~size_t(255);
        bytes.resize(off + sizeof(T) * v.size());
        if (!v.empty()) std::memcpy(bytes.data() + off, v.data(), sizeof(T) * v.size());
        return off;
    }
};

template <typename real>
struct PropOffsets { size_t invW, nasa_cp, nasa_h, visc, wilke, diff; };

template <typename real>
PropOffsets<real> add_prop_tables(BlobBuilder &bb, int N, int Np, const std::vector<double> &W,
                                  const std::vector<double> &lo, const std::vector<double> &hi,
                                  const std::vector<double> &visc, const std::vector<double> &diff) {
    std::vector<real> invW(N), cp(2 * N * 5), h(2 * N * 6), vis(N * 5);
    std::vector<real> wil((size_t)3 * N * Np, real(0)), dif((size_t)5 * N * Np, real(0));
    for (int k = 0; k < N; ++k) {
        invW[k] = real(1.0 / W[k]);
        for (int r = 0; r < 2; ++r) {
            const double *a = (r == 0 ? lo.data() : hi.data()) + 7 * k;
            for (int i = 0; i < 5; ++i) cp[(r * N + k) * 5 + i] = real(a[i]);
            h[(r * N + k) * 6 + 0] = real(a[0]);
            h[(r * N + k) * 6 + 1] = real(a[1] / 2.0);
            h[(r * N + k) * 6 + 2] = real(a[2] / 3.0);
            h[(r * N + k) * 6 + 3] = real(a[3] / 4.0);
            h[(r * N + k) * 6 + 4] = real(a[4] / 5.0);
            h[(r * N + k) * 6 + 5] = real(a[5]);
        }
        for (int i = 0; i < 5; ++i) vis[k * 5 + i] = real(visc[k * 5 + i]);
        for (int j = 0; j < N; ++j) {
            // Wilke weights: Phi_kj = c_kj (1 + w_jk r_k / r_j)^2, r = sqrt(mu)
            double c = 1.0 / std::sqrt(8.0 * (1.0 + W[k] / W[j]));
            double w = std::pow(W[j] / W[k], 0.25);
            wil[(0 * (size_t)N + k) * Np + j] = real(c);
            wil[(1 * (size_t)N + k) * Np + j] = real(2.0 * c * w);
            wil[(2 * (size_t)N + k) * Np + j] = real(c * w * w);
            for (int n = 0; n < 5; ++n)
                dif[((size_t)n * N + k) * Np + j] = (j == k) ? real(0) : real(diff[((size_t)j * N + k) * 5 + n]);
        }
    }
    PropOffsets<real> o;
    o.invW = bb.add(invW);
    o.nasa_cp = bb.add(cp);
    o.nasa_h = bb.add(h);
    o.visc = bb.add(vis);
    o.wilke = bb.add(wil);
    o.diff = bb.add(dif);
    return o;
}

// The B operand of the tensor-core properties pass (PropTcTables) from the FP64 coefficients. Row k of
// the resistance blocks is scaled by a power of two that brings its largest coefficient to 2^14 .. 2^15.
// Returns false when a value does not fit an FP16 pair (then the pass is not used for the mechanism).
bool add_tc_tables(BlobBuilder &bb, int N, const std::vector<double> &W, const std::vector<double> &visc,
                   const std::vector<double> &diff, PropTcTables &t, size_t &off_B, size_t &off_species) {
    t = PropTcTables{};
    if (N > kTcMaxSpecies) return false;
    const int K = tc_k(N);
    t.NP = (N + 7) & ~7;
    t.NR = (N + 15) & ~15;
    t.rows = 2 * t.NR + 6 * t.NP;
    std::vector<double> v((size_t)t.rows * K, 0.0);
    std::vector<float> species((size_t)8 * N, 0.0f);
    auto at = [&](int row, int j) -> double & { return v[(size_t)row * K + j]; };
    for (int k = 0; k < N; ++k) {
        double top = 0.0;
        for (int j = 0; j < N; ++j)
            for (int n = 0; n < 5; ++n)
                if (j != k) top = std::fmax(top, std::fabs(diff[((size_t)j * N + k) * 5 + n]));
        if (!std::isfinite(top)) return false;
        const int e = top > 0.0 ? 14 - std::ilogb(top) : 0;
        if (e < -80 || e > 80) return false;
        if (!(std::fabs(visc[5 * k]) < 100.0)) return false;
        const double half_log2e = 0.5 / std::log(2.0);            // log2 r = ln mu / (2 ln 2)
        const int n = (int)std::lround(visc[5 * k] * half_log2e);
        float *q = species.data() + (size_t)8 * k;
        q[0] = (float)(visc[5 * k] * half_log2e - n);
        for (int i = 1; i < 5; ++i) q[i] = (float)(visc[5 * k + i] * half_log2e);
        q[5] = (float)std::ldexp((double)kTcXScale, e);
        q[6] = (float)std::ldexp(1.0, n);
        for (int j = 0; j < N; ++j) {
            const double c = 1.0 / std::sqrt(8.0 * (1.0 + W[k] / W[j])), w = std::pow(W[j] / W[k], 0.25);
            at(k, j) = 2.0 * c * w * kTcWilkeScale;                                   // T1
            at(t.NR + k, j) = c * kTcWilkeScale;                                      // T0
            at(t.NR + 6 * t.NP + k, j) = c * w * w * kTcWilkeScale;                   // T2
            for (int n = 0; n < 5; ++n)
                at(t.NR + (1 + n) * t.NP + k, j) = j == k ? 0.0 : std::ldexp(diff[((size_t)j * N + k) * 5 + n], e);
        }
    }
    std::vector<__half> B((size_t)2 * t.rows * K);
    for (int r = 0; r < t.rows; ++r)
        for (int j = 0; j < K; ++j) {
            const double x = v[(size_t)r * K + j];
            if (!(std::fabs(x) < 65504.0)) return false;
            const __half hi = __double2half(x);
            const __half lo = __double2half(x - (double)__half2float(hi));
            const size_t q = ((size_t)(j / 8) * t.rows + r) * 8 + j % 8;
            B[q] = hi;
            B[(size_t)t.rows * K + q] = lo;
        }
    off_B = bb.add(B);
    off_species = bb.add(species);
    return true;
}

template <typename real>
PropTables<real> resolve(const PropOffsets<real> &o, uint8_t *base) {
    PropTables<real> t;
    t.invW = reinterpret_cast<const real *>(base + o.invW);
    t.nasa_cp = reinterpret_cast<const real *>(base + o.nasa_cp);
    t.nasa_h = reinterpret_cast<const real *>(base + o.nasa_h);
    t.visc = reinterpret_cast<const real *>(base + o.visc);
    t.wilke = reinterpret_cast<const real *>(base + o.wilke);
    t.diff = reinterpret_cast<const real *>(base + o.diff);
    return t;
}

}  // namespace
}  // namespace chemgb

using namespace chemgb;

extern "C" int chem_mech_load_bytes(const void *data, size_t nbytes, chem_mech **out) {
    if (!data || !out) return set_error(CHEM_EINVAL, "chem_mech_load_bytes: null argument");
    *out = nullptr;
    Reader rd{static_cast<const uint8_t *>(data), static_cast<const uint8_t *>(data) + nbytes};
    char magic[8];
    rd.read(magic, 8);
    if (!rd.ok || std::memcmp(magic, "CHMECH01", 8) != 0) return set_error(CHEM_EIO, "mechanism: bad magic");
    int32_t hdr[4];
    double th[4];
    rd.read(hdr, 4);
    rd.read(th, 4);
    int N = hdr[0], R = hdr[1], E = hdr[2], bath = hdr[3];
    if (!rd.ok) return set_error(CHEM_EIO, "mechanism: truncated header");
    if (N < 1 || N > kMaxSpecies || R < 1 || R > kMaxReactions || E < 1 || E > 16 || bath < 0 || bath >= N)
        return set_error(CHEM_EINVAL, "mechanism: sizes out of range (1 <= N <= 64, 1 <= R <= 4096)");
    std::vector<double> W(N), lo(7 * N), hi(7 * N), sigma(N), eps(N), visc(5 * N), diff((size_t)5 * N * N);
    std::vector<int32_t> elem(N * E), rtype(R), reac(3 * R), prod(3 * R);
    std::vector<double> A(R), beta(R), Ea(R), A0(R), beta0(R), Ea0(R), troe(4 * R), eff((size_t)R * N);
    rd.read(W.data(), N); rd.read(lo.data(), 7 * N); rd.read(hi.data(), 7 * N); rd.read(elem.data(), N * E);
    rd.read(sigma.data(), N); rd.read(eps.data(), N); rd.read(visc.data(), 5 * N); rd.read(diff.data(), diff.size());
    rd.read(rtype.data(), R); rd.read(reac.data(), 3 * R); rd.read(prod.data(), 3 * R);
    rd.read(A.data(), R); rd.read(beta.data(), R); rd.read(Ea.data(), R);
    rd.read(A0.data(), R); rd.read(beta0.data(), R); rd.read(Ea0.data(), R);
    rd.read(troe.data(), 4 * R); rd.read(eff.data(), eff.size());
    if (!rd.ok) return set_error(CHEM_EIO, "mechanism: truncated body");
    for (int k = 0; k < N; ++k)
        if (!(W[k] > 0.0)) return set_error(CHEM_EIO, "mechanism: non-positive molar mass");
    for (int j = 0; j < R; ++j) {
        if (rtype[j] < 0 || rtype[j] > 2) return set_error(CHEM_EIO, "mechanism: bad reaction type");
        for (int i = 0; i < 3; ++i)
            if (reac[3 * j + i] < -1 || reac[3 * j + i] >= N || prod[3 * j + i] < -1 || prod[3 * j + i] >= N)
                return set_error(CHEM_EIO, "mechanism: species index out of range");
        if (reac[3 * j] < 0 || prod[3 * j] < 0) return set_error(CHEM_EIO, "mechanism: empty reaction side");
        if (!(A[j] > 0.0) || (rtype[j] == 2 && !(A0[j] > 0.0)))
            return set_error(CHEM_EIO, "mechanism: non-positive pre-exponential factor");
    }
    int Np = (N + 3) & ~3;

    // Device order of the reactions: Troe fall-off first, then three-body, then
    // elementary (stable within each type). Lanes of a warp take consecutive
    // reactions, so the long fall-off and third-body code paths then occupy
    // few warp iterations; sums over reactions only change their order.
    {
        std::vector<int> order;
        for (int t : {2, 1, 0})
            for (int j = 0; j < R; ++j)
                if (rtype[j] == t) order.push_back(j);
        auto perm_d = [&](std::vector<double> &v, int w) {
            std::vector<double> o(v.size());
            for (int j = 0; j < R; ++j)
                for (int i = 0; i < w; ++i) o[(size_t)j * w + i] = v[(size_t)order[j] * w + i];
            v.swap(o);
        };
        auto perm_i = [&](std::vector<int32_t> &v, int w) {
            std::vector<int32_t> o(v.size());
            for (int j = 0; j < R; ++j)
                for (int i = 0; i < w; ++i) o[(size_t)j * w + i] = v[(size_t)order[j] * w + i];
            v.swap(o);
        };
        perm_i(rtype, 1); perm_i(reac, 3); perm_i(prod, 3);
        perm_d(A, 1); perm_d(beta, 1); perm_d(Ea, 1); perm_d(A0, 1); perm_d(beta0, 1); perm_d(Ea0, 1);
        perm_d(troe, 4); perm_d(eff, N);
    }

    BlobBuilder bb;
    auto o32 = add_prop_tables<float>(bb, N, Np, W, lo, hi, visc, diff);
    auto o64 = add_prop_tables<double>(bb, N, Np, W, lo, hi, visc, diff);
    PropTcTables tct;
    size_t off_tcB = 0, off_tcs = 0;
    const bool tc_ok = add_tc_tables(bb, N, W, visc, diff, tct, off_tcB, off_tcs);
    std::vector<double> lnA(R), EaR(R), lnA0(R), Ea0R(R);
    std::vector<double> dnu(R, 0.0);
    std::vector<double> effc;
    int n_tb = 0;
    for (int j = 0; j < R; ++j) {
        lnA[j] = std::log(A[j]);
        EaR[j] = Ea[j] / kR;
        lnA0[j] = (A0[j] > 0.0) ? std::log(A0[j]) : 0.0;
        Ea0R[j] = Ea0[j] / kR;
        for (int i = 0; i < 3; ++i) dnu[j] += (prod[3 * j + i] >= 0) - (reac[3 * j + i] >= 0);
        if (rtype[j] != 0) {
            ++n_tb;                             // these reactions come first: row j of eff is reaction j's
            for (int k = 0; k < N; ++k) effc.push_back(eff[(size_t)j * N + k]);
        }
    }
    if (effc.empty()) effc.push_back(0.0);
    std::vector<uint32_t> counters(kNumCounters, 0u);
    std::vector<double> nasa_t((size_t)2 * 17 * 64, 0.0), troe_r(4 * R);
    for (int r = 0; r < 2; ++r)
        for (int k = 0; k < N; ++k) {
            const double *a = (r == 0 ? lo.data() : hi.data()) + 7 * k;
            const double v[17] = {a[0], a[1], a[2], a[3], a[4],
                                  a[0], a[1] / 2.0, a[2] / 3.0, a[3] / 4.0, a[4] / 5.0, a[5],
                                  a[0], a[1], a[2] / 2.0, a[3] / 3.0, a[4] / 4.0, a[6]};
            for (int i = 0; i < 17; ++i) nasa_t[((size_t)r * 17 + i) * 64 + k] = v[i];
        }
    for (int j = 0; j < R; ++j) {
        troe_r[4 * j + 0] = troe[4 * j + 0];
        troe_r[4 * j + 1] = (troe[4 * j + 1] != 0.0) ? 1.0 / troe[4 * j + 1] : 0.0;
        troe_r[4 * j + 2] = (troe[4 * j + 2] != 0.0) ? 1.0 / troe[4 * j + 2] : 0.0;
        troe_r[4 * j + 3] = troe[4 * j + 3];
    }
    // distinct species of each reaction (first occurrence) with their net coefficients
    std::vector<int32_t> rsp(6 * R, -1), rnu(6 * R, 0);
    std::vector<uint2> rspec(R);
    int nslot = 1, three = 0;
    for (int j = 0; j < R; ++j) {
        int cnt = 0, present = 0;
        for (int slot = 0; slot < 6; ++slot) {
            int sp = slot < 3 ? reac[3 * j + slot] : prod[3 * j + slot - 3];
            if (sp < 0) continue;
            ++present;
            if (slot % 3 == 2) three = 1;
            bool seen = false;
            for (int u = 0; u < cnt; ++u) seen |= (rsp[6 * j + u] == sp);
            if (seen) continue;
            int nu = 0;
            for (int i = 0; i < 3; ++i) nu += (prod[3 * j + i] == sp) - (reac[3 * j + i] == sp);
            rsp[6 * j + cnt] = sp;
            rnu[6 * j + cnt] = nu;
            ++cnt;
        }
        nslot = cnt > nslot ? cnt : nslot;
        unsigned w[2] = {0u, 0u};
        for (int i = 0; i < 3; ++i) {
            w[0] |= (unsigned)(reac[3 * j + i] >= 0 ? reac[3 * j + i] : N) << (8 * i);
            w[1] |= (unsigned)(prod[3 * j + i] >= 0 ? prod[3 * j + i] : N) << (8 * i);
        }
        if (present == cnt) w[0] |= 1u << 24;
        rspec[j] = make_uint2(w[0], w[1]);
    }
    // code words of the integrator's index lists
    auto code_d = [](int nu, int idx) {
        const double x = (double)nu;
        uint64_t b;
        std::memcpy(&b, &x, 8);
        return (unsigned)((b >> 48) << 16) | (unsigned)idx;
    };
    auto code_f = [](int nu, int idx) {
        const float x = (float)nu;
        uint32_t b;
        std::memcpy(&b, &x, 4);
        return (b & 0xFFFF0000u) | (unsigned)idx;
    };
    // species -> (reaction, nu) incidence, reactions ascending, one column of `gath` per species
    std::vector<std::vector<unsigned>> inc(N);
    std::vector<int32_t> tbrow_ptr(N + 1, 0);
    std::vector<unsigned> tbrow_f, tbrow_d;
    size_t longest = 1;
    for (int k = 0; k < N; ++k) {
        tbrow_ptr[k] = (int)tbrow_f.size();
        for (int j = 0; j < R; ++j)
            for (int u = 0; u < 6 && rsp[6 * j + u] >= 0; ++u)
                if (rsp[6 * j + u] == k && rnu[6 * j + u] != 0) {
                    inc[k].push_back(code_d(rnu[6 * j + u], j));
                    if (rtype[j] != 0) {
                        tbrow_f.push_back(code_f(rnu[6 * j + u], j));
                        tbrow_d.push_back(code_d(rnu[6 * j + u], j));
                    }
                }
        longest = inc[k].size() > longest ? inc[k].size() : longest;
    }
    tbrow_ptr[N] = (int)tbrow_f.size();
    if (tbrow_f.empty()) { tbrow_f.push_back(0u); tbrow_d.push_back(0u); }
    const int gath_len = (int)((longest + 3) & ~size_t(3));
    std::vector<unsigned> gath((size_t)gath_len * 64, (unsigned)R);      // pads: the absent reaction, rate 0
    for (int k = 0; k < N; ++k)
        for (size_t t = 0; t < inc[k].size(); ++t) gath[t * 64 + k] = inc[k][t];
    // entries (row, column) of the sparse part of d wdot / d C: their reactions ascending, entries
    // sorted by length into groups of 32 (one per lane) so that a group's lanes finish together
    struct Entry { int pos; std::vector<unsigned> f, d; };
    std::vector<Entry> ent;
    {
        std::vector<int> at((size_t)N * N, -1);
        for (int j = 0; j < R; ++j)
            for (int u = 0; u < 6 && rsp[6 * j + u] >= 0; ++u) {
                if (rnu[6 * j + u] == 0) continue;
                for (int q = 0; q < 6 && rsp[6 * j + q] >= 0; ++q) {
                    int &e = at[(size_t)rsp[6 * j + u] * N + rsp[6 * j + q]];
                    if (e < 0) {
                        e = (int)ent.size();
                        ent.push_back({(1 + rsp[6 * j + u]) * (N + 1) + 1 + rsp[6 * j + q], {}, {}});
                    }
                    ent[e].f.push_back(code_f(rnu[6 * j + u], j * nslot + q));
                    ent[e].d.push_back(code_d(rnu[6 * j + u], j * nslot + q));
                }
            }
        std::stable_sort(ent.begin(), ent.end(),
                         [](const Entry &a, const Entry &b) { return a.f.size() > b.f.size(); });
    }
    const int ell_groups = (int)((ent.size() + 31) / 32);
    std::vector<int32_t> ell_off(ell_groups + 1, 0), ell_len(ell_groups + 1, 0), ell_pos((size_t)32 * ell_groups + 1, -1);
    std::vector<unsigned> ell_f, ell_d;
    for (int q = 0; q < ell_groups; ++q) {
        const int len = (int)ent[(size_t)32 * q].f.size();
        ell_off[q] = (int)ell_f.size();
        ell_len[q] = len;
        ell_f.resize(ell_f.size() + (size_t)32 * len, 0u);
        ell_d.resize(ell_d.size() + (size_t)32 * len, 0u);
        for (int l = 0; l < 32; ++l) {
            const size_t e = (size_t)32 * q + l;
            if (e >= ent.size()) break;
            ell_pos[e] = ent[e].pos;
            for (size_t t = 0; t < ent[e].f.size(); ++t) {
                ell_f[ell_off[q] + 32 * t + l] = ent[e].f[t];
                ell_d[ell_off[q] + 32 * t + l] = ent[e].d[t];
            }
        }
    }
    if (ell_f.empty()) { ell_f.push_back(0u); ell_d.push_back(0u); }
    std::vector<float> eff_f(effc.size());
    for (size_t i = 0; i < effc.size(); ++i) {                // toward zero, as f64_to_f32_trunc
        float v = (float)effc[i];
        if (std::fabs((double)v) > std::fabs(effc[i])) v = std::nextafterf(v, 0.0f);
        eff_f[i] = v;
    }

    size_t off_W = bb.add(W), off_rtype = bb.add(rtype), off_lnA = bb.add(lnA), off_beta = bb.add(beta),
           off_EaR = bb.add(EaR), off_lnA0 = bb.add(lnA0), off_beta0 = bb.add(beta0), off_Ea0R = bb.add(Ea0R),
           off_troe = bb.add(troe), off_eff = bb.add(effc), off_cnt = bb.add(counters), off_troe_r = bb.add(troe_r),
           off_rsp = bb.add(rsp), off_nasa_t = bb.add(nasa_t), off_dnu = bb.add(dnu), off_rspec = bb.add(rspec),
           off_gath = bb.add(gath), off_eo = bb.add(ell_off), off_el = bb.add(ell_len), off_ep = bb.add(ell_pos),
           off_ef = bb.add(ell_f), off_ed = bb.add(ell_d), off_tp = bb.add(tbrow_ptr), off_tf = bb.add(tbrow_f),
           off_td = bb.add(tbrow_d), off_eff_f = bb.add(eff_f);

    std::string why;
    if (!device_ok(&why)) return set_error(CHEM_EUNSUPPORTED, "chem_mech_load: " + why);
    void *blob = nullptr;
    int rc = check_cuda(cudaMalloc(&blob, bb.bytes.size()), "chem_mech_load: cudaMalloc");
    if (rc) return rc;
    rc = check_cuda(cudaMemcpy(blob, bb.bytes.data(), bb.bytes.size(), cudaMemcpyHostToDevice),
                    "chem_mech_load: cudaMemcpy");
    if (rc) { cudaFree(blob); return rc; }

    chem_mech *m = new chem_mech();
    m->N = N; m->R = R; m->E = E; m->bath = bath;
    m->P_std = th[0]; m->T_lo = th[1]; m->T_mid = th[2]; m->T_hi = th[3];
    m->blob = blob;
    m->blob_bytes = bb.bytes.size();
    cudaGetDevice(&m->device);
    m->wait_limit = tc::kSpinLimit;
    uint8_t *base = static_cast<uint8_t *>(blob);
    DevMech &d = m->dev;
    d.N = N; d.R = R; d.Np = Np; d.n_tb = n_tb; d.P_std = th[0]; d.T_mid = th[2];
    d.f32 = resolve(o32, base);
    d.f64 = resolve(o64, base);
    d.tc = tct;
    d.tc.B = tc_ok ? base + off_tcB : nullptr;
    d.tc.species = tc_ok ? reinterpret_cast<const float *>(base + off_tcs) : nullptr;
    d.W = reinterpret_cast<const double *>(base + off_W);
    d.rtype = reinterpret_cast<const int *>(base + off_rtype);
    d.lnA = reinterpret_cast<const double *>(base + off_lnA);
    d.beta = reinterpret_cast<const double *>(base + off_beta);
    d.EaR = reinterpret_cast<const double *>(base + off_EaR);
    d.lnA0 = reinterpret_cast<const double *>(base + off_lnA0);
    d.beta0 = reinterpret_cast<const double *>(base + off_beta0);
    d.Ea0R = reinterpret_cast<const double *>(base + off_Ea0R);
    d.troe = reinterpret_cast<const double *>(base + off_troe);
    d.eff = reinterpret_cast<const double *>(base + off_eff);
    d.counters = reinterpret_cast<unsigned int *>(base + off_cnt);
    d.troe_r = reinterpret_cast<const double *>(base + off_troe_r);
    d.rsp = reinterpret_cast<const int *>(base + off_rsp);
    d.nasa_t = reinterpret_cast<const double *>(base + off_nasa_t);
    d.dnu_d = reinterpret_cast<const double *>(base + off_dnu);
    d.rspec = reinterpret_cast<const uint2 *>(base + off_rspec);
    d.nslot = nslot;
    d.three = three;
    d.gath_len = gath_len;
    d.gath = reinterpret_cast<const unsigned *>(base + off_gath);
    d.ell_groups = ell_groups;
    d.ell_off = reinterpret_cast<const int *>(base + off_eo);
    d.ell_len = reinterpret_cast<const int *>(base + off_el);
    d.ell_pos = reinterpret_cast<const int *>(base + off_ep);
    d.ell_f = reinterpret_cast<const unsigned *>(base + off_ef);
    d.ell_d = reinterpret_cast<const unsigned *>(base + off_ed);
    d.tbrow_ptr = reinterpret_cast<const int *>(base + off_tp);
    d.tbrow_f = reinterpret_cast<const unsigned *>(base + off_tf);
    d.tbrow_d = reinterpret_cast<const unsigned *>(base + off_td);
    d.eff_f = reinterpret_cast<const float *>(base + off_eff_f);
    d.lnPR = std::log(th[0] / kR);
    *out = m;
    return CHEM_OK;
}

extern "C" int chem_mech_load(const char *path, chem_mech **out) {
    if (!path || !out) return set_error(CHEM_EINVAL, "chem_mech_load: null argument");
    std::ifstream f(path, std::ios::binary);
    if (!f) return set_error(CHEM_EIO, std::string("chem_mech_load: cannot open ") + path);
    std::stringstream ss;
    ss << f.rdbuf();
    std::string s = ss.str();
    return chem_mech_load_bytes(s.data(), s.size(), out);
}

extern "C" int chem_mech_free(chem_mech *m) {
    if (!m) return set_error(CHEM_EINVAL, "chem_mech_free: null handle");
    int prev = -1;
    cudaGetDevice(&prev);
    cudaSetDevice(m->device);
    cudaDeviceSynchronize();
    cudaFree(m->blob);
    if (prev >= 0) cudaSetDevice(prev);
    delete m;
    return CHEM_OK;
}

extern "C" int chem_mech_nspecies(const chem_mech *m) { return m ? m->N : -1; }
extern "C" int chem_mech_nreactions(const chem_mech *m) { return m ? m->R : -1; }

extern "C" int chem_mech_set_wait_limit(chem_mech *m, int32_t tries) {
    if (!m) return set_error(CHEM_EINVAL, "chem_mech_set_wait_limit: null handle");
    m->wait_limit = tries == 0 ? tc::kSpinLimit : (tries < 0 ? 0u : (uint32_t)tries);
    return CHEM_OK;
}

extern "C" void chem_ode_opts_default(chem_ode_opts *o) {
    if (!o) return;
    o->rtol = 1e-6;
    o->atol_Y = 1e-12;
    o->atol_T = 1e-6;
    o->h0 = 1e-9;
    o->max_steps = 10000;
    o->mode = CHEM_ODE_FP64;
}

extern "C" const char *chem_last_error(void) { return chemgb::g_last_error.c_str(); }

extern "C" const char *chem_version(void) {
    return "chemgb 0.1 (CUDA " CHEMGB_STR(__CUDACC_VER_MAJOR__) "." CHEMGB_STR(__CUDACC_VER_MINOR__) ", sm_103a)";
}
