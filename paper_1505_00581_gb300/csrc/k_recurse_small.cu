// k_recurse_small.cu -- kernel (b) for short candidate lists (the pruned form: K' <= 16).
//
// Same recursion as k_recurse.cu (Eqs. 10-13, readings R1-R6) for lists of at
// most KS candidates. With K' = 8 a step has 64 cells of 8 candidates each, so
// a whole CTA of the large-list kernel per unit would idle: here a group of warps (one for KS = 8, two or four for
// 16) owns a unit, threads own cells (b, c) and minimise over a in slot order. Per step the per-(a, b) terms (base,
// p1, p2) and the theta(a->c) table are computed once by the group; then a thread owns CT consecutive cells of one b.
// A cell's result is written as the next step's base (as in k_recurse.cu), and the next step's list is fetched while
// the tables are built. Every value is computed with the same FP32 operations in the same order as in the
// large-list kernel (fast_atan2 directions, wrap, the two circular folds, sqrt.approx, fma; the model constants from
// the same per-model table), so both kernels give the same bits.
//
// A unit is a chain of M - 2 steps, so a batch cannot end before its longest unit, and more warps per unit shorten
// the steps. Lists of up to 16, time of one, two and four warps per unit: 46 units of 40 points 274, 176 and 119 us,
// 3,840 of up to 256 points 2,140, 1,826 and 1,905 us (2,691 us with one warp, lists loaded at the start of their step
// and base recomputed from alpha), 15,360 units 6.7, 6.5 and 7.4 ms, 45,680 of up to 64 points 5.23, 5.18 and 6.00 ms.
// So two warps, and four for up to kFewPerSm units per SM.
#include "recurse_common.cuh"

namespace hgm {
namespace {

constexpr float kInf = __builtin_huge_valf();
constexpr int kThreads = 128;
constexpr int kFewPerSm = 8;   // CTAs of four warps that fit an SM beside each other, about

template <int KS>
struct GroupSmem {
    float2 xy[3][KS];
    int32_t t[3][KS];
    float u[3][KS];
    int32_t idx[3][KS];
    int32_t n[3];
    float alpha[KS * (KS + 1)];                 // base(a,b) of the coming step at b*(KS+1)+a (alpha at the end)
    alignas(16) float4 fb[KS * KS];             // per (b, a) at b*KS+a: (base(a,b) or +inf, p1, p2, -)
    alignas(16) float thac[KS * (KS + 4)];      // theta(a->c) or +inf at a*(KS+4)+c (rows of whole 16-byte groups)
};

// Threads own CT consecutive cells (b, c0 .. c0+CT-1) of one b: the per-(a, b) terms are read once per a for
// CT cells, and the cells go through the packed FP32x2 arithmetic in pairs. G threads per unit: one warp (four units
// share a CTA) or a whole CTA of G threads.
template <int KS, int G>
__global__ void __launch_bounds__(G == 32 ? kThreads : G) recurse_small_kernel(
    const Unit *__restrict__ units, int64_t n_units, const ModelRec *__restrict__ models,
    const SceneRec *__restrict__ scenes, Params p, const int32_t *__restrict__ cand_idx,
    const float *__restrict__ cand_u, const int32_t *__restrict__ cand_cnt, uint8_t *__restrict__ beta,
    UnitResult *__restrict__ res)
{
    constexpr int kGroups = G == 32 ? kThreads / 32 : 1;
    __shared__ GroupSmem<KS> all[kGroups];
    const int tid = threadIdx.x % G, lane = threadIdx.x & 31;
    GroupSmem<KS> &sm = all[threadIdx.x / G];
    constexpr int AS = KS + 1;
    constexpr int RS = KS + 4;
    constexpr int CT = KS * KS / G;         // cells per thread: 8, 4 or 2
    static_assert(CT % 2 == 0 && KS % CT == 0, "cells per thread");
    auto sync = [] {
        if constexpr (G == 32) __syncwarp();
        else __syncthreads();
    };
    const int K = p.K, T = p.T;
    const float lam2 = p.lambda2, lam23 = p.lambda2 * p.lambda3;
    const int my_b = tid / (KS / CT), my_c0 = (tid % (KS / CT)) * CT;

    for (int64_t u = (int64_t)blockIdx.x * kGroups + threadIdx.x / G; u < n_units; u += (int64_t)gridDim.x * kGroups) {
        const Unit un = units[u];
        const ModelRec md = models[un.model];
        const SceneRec sc = scenes[un.scene];
        const int M = md.M;
        const int32_t *cidx = cand_idx + un.cand;
        const float *cu = cand_u + un.cand;
        const int32_t *ccnt = cand_cnt + un.cand / K;
        uint8_t *ubeta = beta + un.beta;
        auto store = [&](int slot, int k, int n, int j, float2 xy, int t, float uc) {
            const bool ok = k < n;
            sm.idx[slot][k] = ok ? j : -1;
            sm.xy[slot][k] = ok ? xy : make_float2(0.f, 0.f);
            sm.t[slot][k] = ok ? t : 0x3fffffff;
            sm.u[slot][k] = ok ? uc : kInf;
            if (k == 0) sm.n[slot] = n;
        };
        // the lists of the first step
        for (int q = 1; q <= 3; ++q) {
            const int i = M - q, n = ccnt[i];
            for (int k = tid; k < KS; k += G) {
                const int j = k < n ? cidx[(int64_t)i * K + k] : 0;
                const bool ok = k < n;
                store(i % 3, k, n, j, ok ? sc.xy[j] : make_float2(0.f, 0.f), ok ? sc.t[j] : 0,
                      ok ? cu[(int64_t)i * K + k] : 0.0f);
            }
        }
        float4 g = md.geo[M - 1];
        sync();
        {   // its base: alpha_{M+1} = 0
            const int sa = (M - 1) % 3, sb = (M - 2) % 3;
            for (int e = tid; e < KS * KS; e += G) {
                const int a = e % KS, b = e / KS;
                sm.alpha[b * AS + a] = base_cost(sm.u[sa][a], lam2, __float_as_int(g.z), sm.t[sa][a], sm.t[sb][b], 0.0f);
            }
        }
        sync();
        for (int i = M - 1; i >= 2; --i) {
            const int sa = i % 3, sb = (i - 1) % 3, scc = (i - 2) % 3;
            // list i - 3 and the model's constants of the next step are fetched meanwhile
            const bool pf = i >= 3 && tid < KS;
            int pf_n = 0, pf_j = 0, pf_t = 0;
            float pf_u = 0.0f;
            float2 pf_xy = make_float2(0.f, 0.f);
            if (pf) {
                pf_n = ccnt[i - 3];
                if (tid < K) {   // entries past the count hold nothing that is used
                    pf_j = cidx[(int64_t)(i - 3) * K + tid];
                    pf_u = cu[(int64_t)(i - 3) * K + tid];
                }
            }
            const float4 gn = md.geo[i - 1];
            const int na = sm.n[sa], nb = sm.n[sb], nc = sm.n[scc];
            const float A1 = g.x, k2 = g.y;
            const float k2c = wrap_pi(__fsub_rn(k2, kPi));   // a and b at the same position (reading R1)
            const int dt_bc = __float_as_int(g.w);
            // per (a, b): base, p1 = A1 + theta(b->a), p2 = p1 + k2; per (a, c): theta(a->c), +inf where (a, c)
            // breaks closeness or distinctness
            for (int e = tid; e < KS * KS; e += G) {
                const int a = e % KS, x = e / KS;
                const int ta = sm.t[sa][a], ia = sm.idx[sa][a];
                const float2 pa = sm.xy[sa][a];
                float4 f = make_float4(kInf, 0.f, 0.f, 0.f);
                if (a < na && x < nb && ta >= sm.t[sb][x] && ia != sm.idx[sb][x]) {
                    const float2 pb = sm.xy[sb][x];
                    f.x = sm.alpha[x * AS + a];
                    f.y = wrap_pi(__fadd_rn(A1, direction(pb, pa)));
                    f.z = __fadd_rn(f.y, pa.x == pb.x && pa.y == pb.y ? k2c : k2);
                }
                sm.fb[x * KS + a] = f;
                float tr = kInf;
                if (a < na && x < nc && !(T > 0 && ta - sm.t[scc][x] >= T) && ia != sm.idx[scc][x])
                    tr = direction(pa, sm.xy[scc][x]);
                sm.thac[a * RS + x] = tr;
            }
            if (pf && tid < pf_n) {
                pf_xy = sc.xy[pf_j];
                pf_t = sc.t[pf_j];
            }
            sync();   // the tables are complete; the base values and list A are not read any more
            if (pf) store(sa, tid, pf_n, pf_j, pf_xy, pf_t, pf_u);
            uint8_t *bstep = ubeta + (int64_t)(i - 2) * K * K;
            const int b = my_b;
            if (b < nb) {
                const int tb = sm.t[sb][b], ib = sm.idx[sb][b];
                const float2 pb = sm.xy[sb][b];
                const float ub = sm.u[sb][b];
                float best[CT];
                int arg[CT];
                unsigned long long q1p[CT / 2];
#pragma unroll
                for (int q = 0; q < CT; q += 2) {
                    float q1[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int c = my_c0 + q + h;
                        q1[h] = c < nc && sm.t[scc][c] <= tb && sm.idx[scc][c] != ib ? direction(pb, sm.xy[scc][c])
                                                                                      : kInf;   // theta(b->c)
                        best[q + h] = kInf;
                        arg[q + h] = kNoSlot;
                    }
                    q1p[q / 2] = pk2(q1[0], q1[1]);
                }
                const unsigned long long lamp = pk2(lam23, lam23);
                for (int a = 0; a < na; ++a) {
                    const float4 f = sm.fb[b * KS + a];
                    if (!(f.x < kInf)) continue;      // a breaks causality or distinctness with b
                    const unsigned long long bp = pk2(f.x, f.x), p1p = pk2(f.y, f.y), p2p = pk2(f.z, f.z);
#pragma unroll
                    for (int q = 0; q < CT; q += 2) {
                        const float2 r2 = *reinterpret_cast<const float2 *>(&sm.thac[a * RS + my_c0 + q]);
                        float v0, v1;
                        triple_cost2(bp, p1p, p2p, q1p[q / 2], pk2(r2.x, r2.y), lamp, v0, v1);
                        if (v0 < best[q]) { best[q] = v0; arg[q] = a; }
                        if (v1 < best[q + 1]) { best[q + 1] = v1; arg[q + 1] = a; }
                    }
                }
#pragma unroll
                for (int q = 0; q < CT; ++q) {
                    const int c = my_c0 + q;
                    if (c < nc) {
                        // alpha_i(b, c), and before the last step the next step's base; best = +inf stays +inf
                        const float al = cell_alpha(best[q], lam2, dt_bc, tb, sm.t[scc][c]);
                        sm.alpha[c * AS + b] = i > 2 ? base_cost(ub, lam2, dt_bc, tb, sm.t[scc][c], al) : al;
                        bstep[b * K + c] = (uint8_t)arg[q];
                    }
                }
            }
            g = gn;
            sync();
        }
        // Eq. 13 over alpha_3(z_2, z_1); ties -> lowest (z_1, z_2); the unit's first warp
        if (tid < 32) {
            const int n0 = sm.n[0], n1 = sm.n[1];
            float bv = kInf;
            int bk = 0x7fffffff;
            for (int e = lane; e < KS * KS; e += 32) {
                const int c = e / KS, b = e % KS;
                if (c < n0 && b < n1) {
                    const float v = sm.u[0][c] + sm.u[1][b] + sm.alpha[c * AS + b];
                    if (v < bv || (v == bv && e < bk)) { bv = v; bk = e; }
                }
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                const float ov = __shfl_xor_sync(0xffffffffu, bv, off);
                const int ok = __shfl_xor_sync(0xffffffffu, bk, off);
                if (ov < bv || (ov == bv && ok < bk)) { bv = ov; bk = ok; }
            }
            if (lane == 0) {
                const bool ok = bv < kInf;
                res[u] = UnitResult{ok ? bv : kInf, ok ? bk / KS : -1, ok ? bk % KS : -1, 0};
            }
        }
        sync();
    }
}

template <int KS, int G>
cudaError_t launch_small(const Unit *units, int64_t n_units, const ModelRec *models, const SceneRec *scenes, Params p,
                         const int32_t *cand_idx, const float *cand_u, const int32_t *cand_cnt, uint8_t *beta,
                         UnitResult *res, cudaStream_t st)
{
    constexpr int kGroups = G == 32 ? kThreads / 32 : 1;
    // a CTA per group of units: the longest come first, and a CTA that ends makes room for the next
    const int64_t grid = std::min<int64_t>((n_units + kGroups - 1) / kGroups, (int64_t)1 << 30);
    prof_begin(kProfRecurse, st);
    recurse_small_kernel<KS, G><<<(unsigned)grid, G == 32 ? kThreads : G, 0, st>>>(units, n_units, models, scenes, p, cand_idx,
                                                                                  cand_u, cand_cnt, beta, res);
    prof_end(kProfRecurse, st);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_recurse_small(const Unit *units, int64_t n_units, const ModelRec *models, const SceneRec *scenes,
                                 Params p, const int32_t *cand_idx, const float *cand_u, const int32_t *cand_cnt,
                                 uint8_t *beta, UnitResult *res, cudaStream_t st)
{
    if (n_units <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (p.K <= 8)
        return launch_small<8, 32>(units, n_units, models, scenes, p, cand_idx, cand_u, cand_cnt, beta, res, st);
    if (n_units <= (int64_t)sms * kFewPerSm)
        return launch_small<16, 128>(units, n_units, models, scenes, p, cand_idx, cand_u, cand_cnt, beta, res, st);
    return launch_small<16, 64>(units, n_units, models, scenes, p, cand_idx, cand_u, cand_cnt, beta, res, st);
}

cudaError_t preload_recurse_small()
{
    cudaFuncAttributes a;
    const void *kerns[] = {(const void *)recurse_small_kernel<8, 32>, (const void *)recurse_small_kernel<16, 64>,
                           (const void *)recurse_small_kernel<16, 128>};
    for (const void *k : kerns) {
        cudaError_t e = cudaFuncGetAttributes(&a, k);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace hgm
