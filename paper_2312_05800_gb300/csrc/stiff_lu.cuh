// stiff_lu.cuh -- the stiff integrator's dense LU in shared memory, for systems of more than 32
// unknowns. Team: the warps that factor one matrix (kWarps of them, wt the rank of this one, sync() their
// barrier, lead() true in the first). Only warp shuffles and the team's barrier are used, so that
// a host build with these can check the accesses.
#pragma once

namespace chemgb {

// In-place LU with partial pivoting in shared memory (n > 32), the reciprocal pivots in invd and the
// pivot rows in piv; false for a zero or non-finite pivot column. In a team every warp searches the
// pivot, the first warp swaps and scales, and the trailing update splits the rows over the warps. No warp
// may still search when the first one swaps: it could miss the pivot, and then return alone
// while the others wait for it.
template <class Team, typename real>
__device__ bool lu_factor(int *piv, real *G, real *invd, Team tm, int lane, int n) {
    for (int k = 0; k < n; ++k) {
        real best = -1;
        int bi = n;
        for (int s = 0; s < 2; ++s) {
            const int i = lane + 32 * s;
            if (i >= k && i < n) {
                const real v = fabs(G[i * n + k]);
                if (v > best || (v == best && i < bi)) { best = v; bi = i; }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const real ob = __shfl_xor_sync(0xFFFFFFFFu, best, o);
            const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
            if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
        }
        if (!(best > 0) || !(best < (real)INFINITY) || bi >= n) return false;     // the same in every warp
        tm.sync();
        if (tm.lead()) {
            if (lane == 0) piv[k] = bi;
            if (bi != k) {
                for (int s = 0; s < 2; ++s) {
                    const int c = lane + 32 * s;
                    if (c < n) {
                        const real t = G[k * n + c];
                        G[k * n + c] = G[bi * n + c];
                        G[bi * n + c] = t;
                    }
                }
            }
        }
        tm.sync();
        const real rp = (real)1 / G[k * n + k];
        if (tm.lead()) {
            if (lane == 0) invd[k] = rp;
            for (int s = 0; s < 2; ++s) {
                const int i = lane + 32 * s;
                if (i > k && i < n) G[i * n + k] *= rp;
            }
        }
        tm.sync();
        for (int s = 0; s < 2; ++s) {
            const int c = lane + 32 * s;
            if (c > k && c < n) {
                const real akc = G[k * n + c];
                for (int i = k + 1 + tm.wt; i < n; i += Team::kWarps) G[i * n + c] -= G[i * n + k] * akc;
            }
        }
        tm.sync();
    }
    return true;
}

}  // namespace chemgb
