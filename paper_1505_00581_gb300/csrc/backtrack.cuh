// backtrack.cuh -- the backtracking walk of Eq. 12 for one unit, shared by the backtrack kernel and the
// fused recursion+backtrack variant of the recursion kernel.
#pragma once

#include "hgm_internal.cuh"

namespace hgm {

// From the initial pair (z_1, z_2) of Eq. 13 follow z_i = beta_i(z_{i-1}, z_{i-2}) through the unit's byte
// tables ub ([(M-2) x K x K], row (i-2)*K + slot(z_{i-1}), column slot(z_{i-2})); slots map to sorted scene
// indices through the candidate lists cidx ([M x K]) and then to the caller's indices, written in the
// caller's model order. Infeasible units (z1 < 0) get a row of -1; energy is written as given.
// A whole warp calls it: every lane walks the chain (the same addresses, one load per step), lane l keeps the slot of
// point i0 + l of each run of 32, and the lanes then look up and write their points together. The walk is a chain
// of one dependent load per step; with the look-ups inside it, three.
__device__ __forceinline__ void backtrack_unit(const Unit &un, const ModelRec &md, const SceneRec &sc, int K,
                                               const int32_t *cidx, const uint8_t *ub, float value, int z1, int z2,
                                               float *energy, int32_t *assign, int lane)
{
    const int M = md.M;
    if (energy && lane == 0) energy[un.out_e] = value;
    if (!assign) return;
    int32_t *out = assign + un.out_a;
    int s2 = z1, s1 = z2;   // slots of z_{i-2}, z_{i-1}
    bool ok = z1 >= 0;
    for (int i0 = 0; i0 < M; i0 += 32) {
        int mine = kNoSlot;
        const int end = min(M, i0 + 32);
        for (int i = i0; i < end && ok; ++i) {
            int s0 = i == 0 ? z1 : z2;
            if (i >= 2) {
                s0 = ub[((int64_t)(i - 2) * K + s1) * K + s2];
                ok = s0 != kNoSlot;
                s2 = s1;
                s1 = s0;
            }
            if (i - i0 == lane) mine = s0;
        }
        const int i = i0 + lane;
        if (i < M) out[md.perm[i]] = mine == kNoSlot ? -1 : sc.perm[cidx[(int64_t)i * K + mine]];
    }
}

}  // namespace hgm
