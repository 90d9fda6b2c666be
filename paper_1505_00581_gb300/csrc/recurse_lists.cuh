// recurse_lists.cuh -- candidate lists in shared memory, shared by the recursion kernels with and without the dummy
// assignment.
#pragma once

#include "recurse_common.cuh"

namespace hgm {

constexpr float kInf = __builtin_huge_valf();
constexpr float kGeoMax = 4.45f;   // > pi*sqrt(2) = 4.4429, bound of the FP32 D^g

template <int KM>
struct alignas(16) List {   // 16-byte aligned arrays: tiles read four consecutive entries at once
    float2 xy[KM];
    int32_t t[KM];
    float u[KM];
    int32_t idx[KM];
    int32_t n;
};

template <int KM>
__device__ void load_list(List<KM> &L, const SceneRec &sc, const int32_t *cidx, const float *cu, int n,
                          int tid, int nt)
{
    for (int k = tid; k < KM; k += nt) {
        if (k < n) {
            int j = cidx[k];
            L.idx[k] = j;
            L.xy[k] = sc.xy[j];
            L.t[k] = sc.t[j];
            L.u[k] = cu[k];
        } else {
            L.idx[k] = -1;
            L.xy[k] = make_float2(0.f, 0.f);
            L.t[k] = 0x3fffffff;
            L.u[k] = kInf;
        }
    }
    if (tid == 0) L.n = n;
}

// (value, slot) minimum with ties to the lower slot
__device__ __forceinline__ void argmin_merge(float &v, int &k, float ov, int ok)
{
    if (ov < v || (ov == v && ok < k)) { v = ov; k = ok; }
}

}  // namespace hgm
