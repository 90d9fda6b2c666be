// k_recurse.cu -- kernel (b): the exact second-order min-sum recursion.
//
// For one unit (model, scene, offset), with lists A = C_i, B = C_{i-1},
// C = C_{i-2} (0-based chain index i = M-1 .. 2, the paper's i+1), Eq. 10:
//   alpha_i(b,c) = min_{a in A feasible} [ U(a) + D(a,b,c) + alpha_{i+1}(a,b) ]
// with alpha_{M+1} = 0 (Eq. 11), the argmin kept in beta_i(b,c) (Eq. 12),
// and finally the initial pair search of Eq. 13 over alpha_3.
//
// GB300 design (differs from the paper's one-launch-per-i OpenCL kernel with
// the CPU as global barrier, Sec. 3.1): one CTA owns a whole unit for its
// lifetime and steps i with CTA barriers; CTAs are persistent and take units
// from a global counter in decreasing-size order. Everything a step touches
// lives in shared memory (Sec. 3.5's local-memory rows, extended to the whole
// alpha table and the geometry). Writing theta(p->q) = atan2(q-p) and A1, A2
// for the model's angles at i-1 and at i, the angle differences of Eq. 6 are
//   d1 = wrap(A1 + theta(b->a) - theta(b->c)),  d2 = wrap(A2 + theta(a->b) - theta(a->c))
// so that, with every pair-only term hoisted (Sec. 3.3's look-up idea applied
// to the geometry), a triple costs two subtractions, two circular folds, a
// squared norm, a square root and an FMA:
//   base(a,b) = U(a) + lambda2 Delta(i,i-1) + alpha_{i+1}(a,b),  p1(a,b) = wrap(A1 + theta(b->a))
//   v(a,b,c)  = base(a,b) + lambda2 lambda3 sqrt(d1^2 + d2^2)   [+ lambda2 Delta(i-1,i-2), after the min]
// Infeasible pairs are +inf (causality t'(c)<=t'(b)<=t'(a), closeness
// t'(a)-t'(c) < T, distinct points; Eqs. 7-8, Sec. 3.2's validity mask).
//
// Exact branch and bound: the geometric term is bounded, 0 <= D^g <= pi*sqrt(2),
// so v(a,b,c) >= base(a,b), and an a with base(a,b) > m(b,c) + lambda2 lambda3
// pi sqrt(2) (plus rounding slack), m(b,c) the smallest base among the a
// feasible with the cell, can never beat the cell's best. Any threshold at or
// above max_c m(b,c) + that bound is therefore exact. Per b the witness w is the
// a of smallest base, m(b,c) = base(w) wherever w is feasible with c; for the
// cells where it is not, m(b,c) is at most the runner-up's base when the
// runner-up is feasible with c; where neither the witness nor the runner-up is
// feasible with some c, no threshold is taken and every a of b is kept. (Which
// c rule them out is read off C by bisection: C is sorted by scene index, hence
// by time, so "too far in time" is a prefix and "same point" a lookup.) Only
// the kept a (about a third of the feasible ones on the batched workload) enter the
// triple loop, in increasing slot order with a strict '<', so the lowest slot
// still wins exact ties -- the result is bit-identical to the full minimisation.
//
// Work split per step (three CTA barriers): phase 1, NT / KM threads per b, each with a run of row b's base in
// registers, find the row's two smallest, its threshold and its kept list with shuffles among neighbours only (the
// bisections of list C go to different lanes); the same threads then fill the theta(a->c) table; then every thread
// takes part in ordering the b by decreasing kept count and laying out the tile table; phase 3, tiles of one b and
// CT consecutive c with t'(c) <= t'(b) are flattened across the CTA's threads in that order (similar loop lengths
// within a warp), each thread looping over the kept a of its b. A cell's alpha_i(b,c) is written as the next step's
// base: with a = b and b = c it is U(b) + lambda2 Delta(b,c) + alpha_i(b,c), the same Delta as in alpha itself.
// The per-step model constants come from a table built at model creation, and the list C of the next step is
// fetched from global memory during phase 1 and stored in the buffer of the list A, which phase 3 no longer reads,
// so no step waits on a global load. Argmin bytes are written for the tiled cells only, a tile's four at once: the
// cells past b's time prefix are never on a chain, so the backtrack never reads them.
#include <algorithm>
#include <climits>

#include <cooperative_groups.h>

#include "backtrack.cuh"
#include "recurse_lists.cuh"

namespace hgm {
namespace {

template <int KM, int NT, int CL>
struct Smem {
    // row strides: rows of different b read at the same place fall into different banks (FS, SS); rows of r and
    // alpha are whole 16-byte groups whose starts are 4 banks apart, and their four words past the KM columns hold
    // the step's tile table
    static constexpr int FS = KM + 1, SS = KM + 4, RS = KM + 4, AS = KM + 4;
    float2 fb[KM * FS];                   // per b: kept (base, p1) in increasing a
    float r[KM * RS];                     // theta(a->c) or +inf, at a*RS + c | 16 bytes of tile_b per row
    // base(a,b) of the coming step at b*AS + a | rank key, tile info of b; a cluster's CTAs write one another's rows
    // of the next step while this one's are still read (step i: half i & 1)
    float alpha[(CL > 1 ? 2 : 1) * KM * AS];
    uint8_t fs[KM * SS];                  // slot a of each kept entry, | 0x80 when a lies at b's position
    List<KM> list[3];
    float4 geo[2];                        // model constants of step i at geo[i & 1]
    float red_v[CL * NT / 32];
    int32_t red_k[CL * NT / 32];
    int32_t ntile;                        // tiles of the step
    int32_t unit;
    int32_t coin[2];                      // step i: some kept a lies at its b's position (coin[i & 1])

    // b of tile t (tiles of >= 4 cells); per b: (sort key << 5) | tile count, key 0 for b without tiles; first tile
    // << 12 | kept count << 5 | tile count
    __device__ uint8_t &tile_b(int t) { return reinterpret_cast<uint8_t *>(&r[(t >> 4) * RS + KM])[t & 15]; }
    __device__ int32_t &key(int b) { return reinterpret_cast<int32_t *>(alpha)[b * AS + KM]; }
    __device__ int32_t &info(int b) { return reinterpret_cast<int32_t *>(alpha)[b * AS + KM + 1]; }
};

// A warp's searches of a list's first n (<= KM) entries: how many of an ascending array lie below x, and the slot
// that holds x (KM: none).
template <int KM>
__device__ __forceinline__ int entries_below(const int32_t *arr, int n, int x, int lane)
{
    int c = 0;
#pragma unroll
    for (int k = 0; k < KM; k += 32) c += __popc(__ballot_sync(0xffffffffu, k + lane < n && arr[k + lane] < x));
    return c;
}

template <int KM>
__device__ __forceinline__ int entry_at(const int32_t *arr, int n, int x, int lane)
{
    int f = KM;
#pragma unroll
    for (int k = KM - 32; k >= 0; k -= 32) {
        const unsigned m = __ballot_sync(0xffffffffu, k + lane < n && arr[k + lane] == x);
        if (m) f = k + __ffs((int)m) - 1;
    }
    return f;
}

// The smallest of a warp's values (order-preserving keys; a NaN counts as +inf, as fminf takes it).
__device__ __forceinline__ float warp_min(float x)
{
    const uint32_t u = __float_as_uint(fminf(x, kInf));
    const uint32_t k = __reduce_min_sync(0xffffffffu, (u >> 31) ? ~u : (u | 0x80000000u));
    return __uint_as_float((k >> 31) ? (k & 0x7fffffffu) : ~k);
}

// kCount = true builds the accounting variant: identical work, plus a count of
// the (a, b, c) evaluations the triple loop performs (kept a x CT per tile).
// kFused = true builds the self-contained variant used for the exact fallback
// of the pruned form: the number of units is read from n_dev (written by an
// earlier kernel, so nothing waits on the host), the argmin tables of a unit
// live in a per-CTA scratch block (beta + blockIdx.x * beta_cta, reused unit
// after unit), and the CTA backtracks its own unit and writes the energy and
// the assignment itself.
// CL > 1 builds the variant in which a cluster of CL CTAs shares a unit: CTA r owns the rows b with b % CL == r, their
// kept lists and their tiles, holds the theta(a->c) table whole, and writes a cell's base into the next step's row c
// in the shared memory of that row's owner; one cluster barrier per step takes the place of the last CTA barrier.
template <int KM, int NT, int MB, int CT, int UR, bool kCount, bool kFused, int CL>
__global__ void __launch_bounds__(NT, MB)
recurse_kernel(const Unit *__restrict__ units, int64_t n_units, const ModelRec *__restrict__ models,
               const SceneRec *__restrict__ scenes, Params p, const int32_t *__restrict__ cand_idx,
               const float *__restrict__ cand_u, const int32_t *__restrict__ cand_cnt, uint8_t *__restrict__ beta,
               UnitResult *__restrict__ res, int *__restrict__ work_counter, unsigned long long *__restrict__ evaluated,
               const int *__restrict__ n_dev, int n_from, int n_to, int64_t beta_cta, float *__restrict__ energy_out,
               int32_t *__restrict__ assign_out)
{
    if constexpr (kFused) {
        const int64_t nd = *n_dev;
        if (nd <= n_from || nd > n_to) return;   // the launch for the other range of counts takes it
        n_units = nd < n_units ? nd : n_units;
    }
    unsigned long long n_eval = 0;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using SM = Smem<KM, NT, CL>;
    SM &sm = *reinterpret_cast<SM *>(smem_raw);
    constexpr int RS = SM::RS, AS = SM::AS, FS = SM::FS, SS = SM::SS;
    constexpr int NW = NT / 32;
    constexpr int TPC = NT / KM;           // threads per c: neighbouring lanes
    constexpr int TPB = TPC * CL;          // threads per b of the CTA's rows
    constexpr int AH = KM / TPB;           // slots a per thread: a = AH h + 0 .. AH - 1
    static_assert(CL == 1 ? TPB == 4 || TPB == 8 : TPB == 32, "threads per b");
    constexpr bool kWarpRow = TPB == 32;   // a warp per b: ballots in place of searches and exchanges
    constexpr int kHalf = CL > 1 ? KM * AS : 0;
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = p.K;
    const int T = p.T;
    const float lam2 = p.lambda2;
    const float lam23 = p.lambda2 * p.lambda3;
    const float gmax = lam23 * kGeoMax;
    unsigned rank = 0;
    int64_t u_next = 0;                    // CL > 1: units go to the clusters in turn
    if constexpr (CL > 1) {
        rank = cooperative_groups::this_cluster().block_rank();
        u_next = blockIdx.x / CL;
        cooperative_groups::this_cluster().sync();   // every CTA runs before its memory is written
    }
    const int h = tid % TPB, row = tid / TPB * CL + (int)rank;
    const int hc = tid % TPC, rowc = tid / TPC;
    // a thread reads its run of slots from a start of its own, so that a warp's reads hit every bank once
    const int rot = TPB == 4 ? h : TPB == 8 ? (h & 1) + ((h >> 2) << 1) : 0;

    for (;;) {
        int64_t u;
        if constexpr (CL > 1) {
            u = u_next;
            u_next += gridDim.x / CL;
        } else {
            if (tid == 0) sm.unit = atomicAdd(work_counter, 1);
            __syncthreads();
            u = sm.unit;
        }
        if (u >= n_units) {
            if constexpr (kCount) atomicAdd(evaluated, n_eval);
            break;
        }
        const Unit un = units[u];
        const ModelRec md = models[un.model];
        const SceneRec sc = scenes[un.scene];
        const int M = md.M;
        const int32_t *cidx = cand_idx + un.cand;
        const float *cu = cand_u + un.cand;
        const int32_t *ccnt = cand_cnt + un.cand / K;
        uint8_t *ubeta = kFused ? beta + (int64_t)(blockIdx.x / CL) * beta_cta : beta + un.beta;

        // the three lists and the constants of the first step
        for (int q = 1; q <= 3 && q <= M; ++q)
            load_list<KM>(sm.list[(M - q) % 3], sc, cidx + (int64_t)(M - q) * K, cu + (int64_t)(M - q) * K,
                          ccnt[M - q], tid, NT);
        if (tid == 0 && M >= 3) {
            sm.geo[(M - 1) & 1] = md.geo[M - 1];
            sm.coin[0] = sm.coin[1] = 0;
        }
        __syncthreads();
        {   // the first step's base: alpha_{M+1} == 0 (Eq. 11)
            const List<KM> &LA = sm.list[(M - 1) % 3], &LB = sm.list[(M - 2) % 3];
            const int dt_ab = __float_as_int(sm.geo[(M - 1) & 1].z);
            float *first = sm.alpha + ((M - 1) & 1) * kHalf;
            for (int e = tid; e < KM * KM / CL; e += NT) {
                const int b = e / KM * CL + (int)rank, a = e % KM;
                // slots past a list hold t = 0x3fffffff, idx = -1, u = inf
                const bool ok = a < LA.n && b < LB.n && LA.t[a] >= LB.t[b] && LA.idx[a] != LB.idx[b];
                first[b * AS + a] = ok ? base_cost(LA.u[a], lam2, dt_ab, LA.t[a], LB.t[b], 0.0f) : kInf;
            }
            if constexpr (CL > 1)   // the other CTAs' rows have no tiles here
                for (int b = tid; b < KM; b += NT) sm.key(b) = 0;
        }
        __syncthreads();

        for (int i = M - 1; i >= 2; --i) {
            List<KM> &LA = sm.list[i % 3];
            List<KM> &LB = sm.list[(i - 1) % 3];
            List<KM> &LC = sm.list[(i - 2) % 3];
            const float4 g = sm.geo[i & 1];
            const float A1 = g.x, k2 = g.y;
            // p2 = p1 + k2 uses theta(a->b) = theta(b->a) + pi, which fails for a and b at the same position
            // (both directions are atan2(0, 0) = 0, reading R1): such entries (flagged in fs) take k2c
            const float k2c = wrap_pi(__fsub_rn(k2, kPi));
            const int dt_bc = __float_as_int(g.w);
            const int na = LA.n, nb = LB.n, nc = LC.n;

            // list C of the next step (chain index i-3) is fetched by the first threads
            const bool pf = i >= 3 && tid < K;
            int pf_n = 0, pf_j = -1;
            float pf_u = kInf;
            float2 pf_xy = make_float2(0.f, 0.f);
            int pf_t = 0x3fffffff;
            if (pf) {
                pf_n = ccnt[i - 3];
                pf_j = cidx[(int64_t)(i - 3) * K + tid];
                pf_u = cu[(int64_t)(i - 3) * K + tid];
            }
            if (tid == NT - 1 && i >= 3) sm.geo[(i - 1) & 1] = md.geo[i - 1];

            // ---- phase 1: the kept a list of b = row
            {
                const int b = row;
                const bool inb = b < nb;
                float2 pb = make_float2(0.f, 0.f);
                int tb = 0, ib = -1;
                if (inb) { pb = LB.xy[b]; tb = LB.t[b]; ib = LB.idx[b]; }
                const float *arow = sm.alpha + (i & 1) * kHalf + b * AS + AH * h;
                // the a with t'(a) >= t'(b) form a suffix of list A (time order): the slots before it are never
                // feasible with b, and the row holds nothing of this step there
                int lo = 0;
                if constexpr (kWarpRow) {
                    if (inb) lo = entries_below<KM>(LA.t, na, tb, lane);
                } else {
                    for (int hi = inb ? na : 0; lo < hi;) {
                        const int mid = (lo + hi) >> 1;
                        if (LA.t[mid] < tb) lo = mid + 1;
                        else hi = mid;
                    }
                }
                const int j0 = lo - AH * h, j1 = (inb ? na : 0) - AH * h;
                // smallest and second smallest base over all feasible a
                float v[AH], m1 = kInf, m2 = kInf;
#pragma unroll
                for (int k = 0; k < AH; ++k) {
                    const int j = (k + rot) & (AH - 1);
                    const float x = arow[j];
                    v[k] = j >= j0 && j < j1 ? x : kInf;
                    m2 = fminf(m2, fmaxf(m1, v[k]));
                    m1 = fminf(m1, v[k]);
                }
                // lowest slot of a value among the row's (1 << 20: none)
                auto slot_of_value = [&](float x, int skip) {
                    int s = 1 << 20;
                    if constexpr (kWarpRow) {
                        unsigned has = 0, at[AH];
#pragma unroll
                        for (int k = 0; k < AH; ++k) {
                            at[k] = __ballot_sync(full, v[k] == x && AH * h + k != skip);
                            has |= at[k];
                        }
                        const int f = __ffs((int)has) - 1;
#pragma unroll
                        for (int k = AH - 1; k >= 0; --k)
                            if (has && (at[k] >> f) & 1u) s = AH * f + k;
                        return s;
                    }
#pragma unroll
                    for (int k = 0; k < AH; ++k) {
                        const int a = AH * h + ((k + rot) & (AH - 1));
                        if (v[k] == x && a != skip) s = min(s, a);
                    }
#pragma unroll
                    for (int off = 1; off < TPB; off <<= 1) s = min(s, __shfl_xor_sync(full, s, off));
                    return s;
                };
                int s1;
                if constexpr (kWarpRow) {
                    const float own1 = m1, own2 = m2;
                    m1 = warp_min(own1);
                    s1 = slot_of_value(m1, -1);
                    m2 = warp_min(s1 / AH == h ? own2 : own1);
                } else {
#pragma unroll
                    for (int off = 1; off < TPB; off <<= 1) {
                        const float o1 = __shfl_xor_sync(full, m1, off), o2 = __shfl_xor_sync(full, m2, off);
                        m2 = fminf(fmaxf(m1, o1), fminf(m2, o2));
                        m1 = fminf(m1, o1);
                    }
                    s1 = slot_of_value(m1, -1);   // every lane takes part in the exchanges
                }
                const bool any = m1 < kInf;
                if (!any) s1 = 0;
                const int tw = LA.t[s1], iw = any ? LA.idx[s1] : -2;
                // C is in increasing scene index, hence in increasing time: the c with t'(c) <= x form a prefix, and
                // a point's slot is found by bisection. Four lanes take one search each: c not after b, c too far
                // from the witness, b's point, the witness's point.
                auto lower_bound = [&](const int32_t *arr, int x) {
                    int l = 0, r = nc;
                    while (l < r) {
                        const int mid = (l + r) >> 1;
                        if (arr[mid] < x) l = mid + 1;
                        else r = mid;
                    }
                    return l;
                };
                const int base_lane = lane & ~(TPB - 1);
                int ccount, nT, pbs, pw;
                if constexpr (kWarpRow) {
                    ccount = inb ? entries_below<KM>(LC.t, nc, tb + 1, lane) : 0;
                    nT = min(entries_below<KM>(LC.t, nc, T > 0 ? tw - T + 1 : INT32_MIN, lane), ccount);
                    pbs = entry_at<KM>(LC.idx, nc, ib, lane);
                    pw = entry_at<KM>(LC.idx, nc, iw, lane);
                } else {
                    const int q = h & 3;
                    const int32_t *arr = q < 2 ? LC.t : LC.idx;
                    const int x = q == 0 ? tb + 1 : q == 1 ? (T > 0 ? tw - T + 1 : INT32_MIN) : q == 2 ? ib : iw;
                    int f = lower_bound(arr, x);
                    if (q >= 2 && !(f < nc && arr[f] == x)) f = KM;
                    ccount = __shfl_sync(full, f, base_lane);
                    if (!inb) ccount = 0;
                    nT = min(__shfl_sync(full, f, base_lane + 1), ccount);
                    pbs = __shfl_sync(full, f, base_lane + 2);
                    pw = __shfl_sync(full, f, base_lane + 3);
                }
                const bool live = any && ccount > 0;
                // cells (b,c) where the witness s1 is infeasible (the cells of b's own point never count; witness and
                // runner-up are feasible with b, so their points differ from b's): their best base is the second
                // smallest over the a feasible with c -- exactly m2 when the runner-up s2 is feasible with c;
                // otherwise (rare) every a is kept
                const bool anybad = live && (nT - (pbs < nT ? 1 : 0) > 0 || pw < ccount);
                bool loose = false;
                if (__any_sync(full, anybad)) {
                    const bool has2 = m2 < kInf;
                    const int s2 = slot_of_value(m2, s1);
                    const int t2 = has2 ? LA.t[s2] : 0, i2 = has2 ? LA.idx[s2] : -2;
                    int nT2, p2;
                    if constexpr (kWarpRow) {
                        nT2 = min(entries_below<KM>(LC.t, nc, T > 0 ? min(tw, t2) - T + 1 : INT32_MIN, lane), ccount);
                        p2 = entry_at<KM>(LC.idx, nc, i2, lane);
                    } else {
                        const int q = h & 1;
                        const int32_t *arr = q == 0 ? LC.t : LC.idx;
                        const int x = q == 0 ? (T > 0 ? min(tw, t2) - T + 1 : INT32_MIN) : i2;
                        int f = lower_bound(arr, x);
                        if (q == 1 && !(f < nc && arr[f] == x)) f = KM;
                        nT2 = min(__shfl_sync(full, f, base_lane), ccount);
                        p2 = __shfl_sync(full, f, base_lane + 1);
                    }
                    // a c that rules out both: too far from both, or at one's point and too far from the other
                    loose = !has2 || nT2 - (pbs < nT2 ? 1 : 0) > 0 || p2 < nT || (pw < ccount && T > 0 && t2 - tw >= T);
                }
                float thr = m1 + gmax + 1e-6f * m1;
                if (anybad) thr = loose ? kInf : fmaxf(thr, m2 + gmax + 1e-6f * m2);
                thr = live ? fminf(thr, 3.402823466e38f) : -kInf;   // no infeasible a, and none for a b without cells
                // keep base <= thr, in increasing a: positions from the kept counts of the row's threads
                unsigned mk = 0;
#pragma unroll
                for (int k = 0; k < AH; ++k)
                    if (v[k] <= thr) mk |= 1u << k;
                mk = ((mk << rot) | (mk >> (AH - rot))) & ((1u << AH) - 1);
                int pos = 0, kept = __popc(mk);
                if constexpr (kWarpRow) {
                    kept = 0;
#pragma unroll
                    for (int k = 0; k < AH; ++k) {
                        const unsigned m = __ballot_sync(full, (mk >> k) & 1u);
                        kept += __popc(m);
                        pos += __popc(m & ((1u << lane) - 1));
                    }
                } else {
#pragma unroll
                    for (int off = 1; off < TPB; off <<= 1) {
                        const int o = __shfl_xor_sync(full, kept, off);
                        if (h & off) pos += o;
                        kept += o;
                    }
                }
                for (unsigned m = mk; m; m &= m - 1, ++pos) {
                    const int j = __ffs((int)m) - 1, a = AH * h + j;
                    const float2 pa = LA.xy[a];
                    const bool same = pa.x == pb.x && pa.y == pb.y;
                    if (same) sm.coin[i & 1] = 1;
                    // p1 = A1 + theta(b->a)
                    sm.fb[b * FS + pos] = make_float2(arow[j], wrap_pi(__fadd_rn(A1, direction(pb, pa))));
                    sm.fs[b * SS + pos] = (uint8_t)(a | (same ? 0x80 : 0));
                }
                // tiles in decreasing kept count, then increasing b (the lanes of a warp then loop over
                // similar numbers of a): b's first tile = sum of the tile counts of the b ranked before it
                if (h == 0) {
                    const int nt_b = (ccount + CT - 1) / CT;
                    const int key = nt_b > 0 ? ((kept + 1) << 8) | (255 - b) : 0;
                    sm.key(b) = (key << 5) | nt_b;
                }
            }
            if (pf && tid < pf_n) {
                pf_xy = sc.xy[pf_j];
                pf_t = sc.t[pf_j];
            }
            // ---- phase 2: theta(a->c) for every a and the c = row with t'(c) <= t'(a). A kept a of a cell (b, c) has
            // t'(a) >= t'(b) >= t'(c), so only the rows from the first a with t'(a) >= t'(c) are read; entries of c
            // past the list belong to cells whose theta(b->c) is +inf, so their value is never used either
            if (rowc < nc) {
                const int c = rowc;
                const int tc = LC.t[c], ic = LC.idx[c];
                const float2 pc = LC.xy[c];
                int lo = 0;
                for (int hi = na; lo < hi;) {
                    const int mid = (lo + hi) >> 1;
                    if (LA.t[mid] < tc) lo = mid + 1;
                    else hi = mid;
                }
#pragma unroll 2
                for (int a = lo + hc; a < na; a += TPC) {
                    const int ta = LA.t[a];
                    float r = direction(LA.xy[a], pc);   // theta(a->c)
                    if ((T > 0 && ta - tc >= T) || LA.idx[a] == ic) r = kInf;
                    sm.r[a * RS + c] = r;
                }
            }
            __syncthreads();

            // tile layout, by every thread (NT / KM per b): b's first tile = the tile count of the b ranked
            // before it (decreasing kept count, then increasing b)
            {
                const int b = rowc, wb = sm.key(b), key = wb >> 5, nt_b = wb & 31;
                int before = 0, total = 0;
                for (int b2 = hc; b2 < KM; b2 += TPC) {
                    const int w = sm.key(b2);
                    total += w & 31;
                    if ((w >> 5) > key) before += w & 31;
                }
#pragma unroll
                for (int off = 1; off < TPC; off <<= 1) {
                    before += __shfl_xor_sync(full, before, off);
                    total += __shfl_xor_sync(full, total, off);
                }
                if (hc == 0) sm.info(b) = before << 12 | max((key >> 8) - 1, 0) << 5 | nt_b;
                for (int t = hc; t < nt_b; t += TPC) sm.tile_b(before + t) = (uint8_t)b;
                if (tid == 0) {
                    sm.ntile = total;
                    sm.coin[(i - 1) & 1] = 0;
                }
            }

            // list A is not read from here on: its buffer receives list C of the next step
            if (i >= 3 && tid < KM) {
                const bool ok = tid < pf_n;
                LA.idx[tid] = ok ? pf_j : -1;
                LA.xy[tid] = pf_xy;
                LA.t[tid] = pf_t;
                LA.u[tid] = ok ? pf_u : kInf;
                if (tid == 0) LA.n = pf_n;
            }

            __syncthreads();   // the tile layout is complete

            // ---- phase 3: tiles (b, CT consecutive c)
            const int ntile = sm.ntile;
            const bool coin = sm.coin[i & 1] != 0;
            // where the next step's base of row c goes: the half of the CTA that owns the row
            float *anext = sm.alpha + ((i - 1) & 1) * kHalf;
            auto put = [&](int c, int b, float x) {
                if constexpr (CL > 1)
                    *cooperative_groups::this_cluster().map_shared_rank(anext + c * AS + b, (unsigned)c % CL) = x;
                else
                    sm.alpha[c * AS + b] = x;
            };
            uint8_t *bstep = ubeta + (int64_t)(i - 2) * K * K;
            // tiles in decreasing kept count, dealt to the threads back and forth (round r: thread t takes
            // tile r NT + t for even r, r NT + NT - 1 - t for odd r) so that per-thread sums even out
            for (int r0 = 0; r0 < ntile; r0 += NT) {
                const int tile = r0 + (((r0 / NT) & 1) ? NT - 1 - tid : tid);
                if (tile >= ntile) continue;
                const int b = sm.tile_b(tile);
                const int info = sm.info(b);
                const int c0 = (tile - (info >> 12)) * CT;
                const float2 pb = LB.xy[b];
                const int tb = LB.t[b], ib = LB.idx[b];
                const float ub = LB.u[b];
                float q1[CT], best[CT];
                int arg[CT], tcq[CT];
#pragma unroll
                for (int q4 = 0; q4 < CT; q4 += 4) {   // the tile's cells of list C, four at a time
                    const int4 t4 = *reinterpret_cast<const int4 *>(&LC.t[c0 + q4]);
                    const int4 i4 = *reinterpret_cast<const int4 *>(&LC.idx[c0 + q4]);
                    const float4 xa = *reinterpret_cast<const float4 *>(&LC.xy[c0 + q4]);
                    const float4 xb = *reinterpret_cast<const float4 *>(&LC.xy[c0 + q4 + 2]);
                    const int tv[4] = {t4.x, t4.y, t4.z, t4.w}, iv[4] = {i4.x, i4.y, i4.z, i4.w};
                    const float2 xv[4] = {make_float2(xa.x, xa.y), make_float2(xa.z, xa.w), make_float2(xb.x, xb.y),
                                          make_float2(xb.z, xb.w)};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int c = c0 + q4 + k;
                        const bool ok = c < nc && tv[k] <= tb && iv[k] != ib;
                        const float d = direction(pb, xv[k]);            // theta(b->c)
                        q1[q4 + k] = ok ? d : kInf;
                        tcq[q4 + k] = tv[k];
                        best[q4 + k] = kInf;
                        arg[q4 + k] = kNoSlot;
                    }
                }
                const int nf = (info >> 5) & 127;
                // cells in pairs: packed FP32x2 arithmetic, same roundings as triple_cost
                static_assert(CT % 4 == 0, "tiles of a multiple of 4 cells");
                unsigned long long q1p[CT / 2];
#pragma unroll
                for (int q = 0; q < CT / 2; ++q) q1p[q] = pk2(q1[2 * q], q1[2 * q + 1]);
                const unsigned long long lamp = pk2(lam23, lam23);
                const float2 *fb = sm.fb + b * FS;
                const uint8_t *fs = sm.fs + b * SS;
                const float *rc = sm.r + c0;
                if constexpr (kCount) n_eval += CT * nf;
                auto triples = [&](const float2 e, int a, float p2) {
                    const unsigned long long bp = pk2(e.x, e.x), p1p = pk2(e.y, e.y), p2p = pk2(p2, p2);
#pragma unroll
                    for (int q4 = 0; q4 < CT; q4 += 4) {
                        const float4 r4 = *reinterpret_cast<const float4 *>(rc + a * RS + q4);
                        float v[4];
                        triple_cost2(bp, p1p, p2p, q1p[q4 / 2], pk2(r4.x, r4.y), lamp, v[0], v[1]);
                        triple_cost2(bp, p1p, p2p, q1p[q4 / 2 + 1], pk2(r4.z, r4.w), lamp, v[2], v[3]);
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (v[q] < best[q4 + q]) { best[q4 + q] = v[q]; arg[q4 + q] = a; }
                    }
                };
                if (!coin) {
#pragma unroll UR
                    for (int k = 0; k < nf; ++k) triples(fb[k], fs[k], __fadd_rn(fb[k].y, k2));
                } else {
#pragma unroll 1
                    for (int k = 0; k < nf; ++k)
                        triples(fb[k], fs[k] & 0x7f, __fadd_rn(fb[k].y, (fs[k] & 0x80) ? k2c : k2));
                }
                // argmin bytes of the tile's cells, four at a time (c0 is a multiple of 4, and K, the row
                // stride, is a multiple of 4 whenever a tile reaches past c0 + 3: the packed store is used
                // only then); a cell without a feasible a keeps best = +inf and arg = kNoSlot
                uint32_t packed[CT / 4];
#pragma unroll
                for (int q4 = 0; q4 < CT / 4; ++q4) packed[q4] = 0;
#pragma unroll
                for (int q = 0; q < CT; ++q) {
                    const int c = c0 + q;
                    // alpha_i(b,c), and before the last step the next step's base: U(b) and the same Delta with it
                    const float al = cell_alpha(best[q], lam2, dt_bc, tb, tcq[q]);
                    const float out = i > 2 ? base_cost(ub, lam2, dt_bc, tb, tcq[q], al) : al;
                    if (c < nc) put(c, b, out);
                    packed[q / 4] |= (uint32_t)arg[q] << (8 * (q % 4));
                }
                const bool aligned = (K & 3) == 0;
#pragma unroll
                for (int q4 = 0; q4 < CT / 4; ++q4) {
                    const int c = c0 + 4 * q4;
                    if (aligned && c + 3 < K) {
                        *reinterpret_cast<uint32_t *>(bstep + b * K + c) = packed[q4];
                    } else {
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (c + q < nc) bstep[b * K + c + q] = (uint8_t)(packed[q4] >> (8 * q));
                    }
                }
            }
            // cells (b, c) beyond the tiled prefix are infeasible: the backtrack never reads their argmin (a
            // chain's cells are feasible) and the next step never reads their alpha (the pair (b, c) is
            // infeasible there); only the initial pair search of Eq. 13 reads every cell of the last step
            if (i == 2) {
                for (int b = warp * CL + (int)rank; b < nb; b += NW * CL) {
                    const int covered = (sm.info(b) & 31) * CT;
                    for (int c = covered + lane; c < nc; c += 32) put(c, b, kInf);
                }
            }
            if constexpr (CL > 1) cooperative_groups::this_cluster().sync();
            else __syncthreads();
        }

        // Eq. 13: (z_1, z_2) = argmin U(z_1) + U(z_2) + alpha_3(z_2, z_1); ties -> lowest (z_1, z_2)
        {
            const List<KM> &L0 = sm.list[0];
            const List<KM> &L1 = sm.list[1];
            const int n0 = L0.n, n1 = L1.n;
            float bv = kInf;
            int bk = 0x7fffffff;
            const float *last = sm.alpha + kHalf;   // step 2 wrote the half of step 1
            for (int e = tid; e < KM * KM / CL; e += NT) {
                const int c = e / KM * CL + (int)rank, b = e % KM;    // z1 * KM + z2: lexicographic order
                if (c < n0 && b < n1) argmin_merge(bv, bk, L0.u[c] + L1.u[b] + last[c * AS + b], CL > 1 ? c * KM + b : e);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1)
                argmin_merge(bv, bk, __shfl_xor_sync(0xffffffffu, bv, off), __shfl_xor_sync(0xffffffffu, bk, off));
            if constexpr (CL > 1) {   // to CTA 0; the other CTAs' argmin bytes are visible to it after the barrier
                if (lane == 0) {
                    auto cl = cooperative_groups::this_cluster();
                    *cl.map_shared_rank(&sm.red_v[rank * NW + warp], 0) = bv;
                    *cl.map_shared_rank(&sm.red_k[rank * NW + warp], 0) = bk;
                }
                cooperative_groups::this_cluster().sync();
            } else {
                if (lane == 0) { sm.red_v[warp] = bv; sm.red_k[warp] = bk; }
                __syncthreads();
            }
            if (warp == 0 && rank == 0) {
                // every lane merges the warps' results: the same values
                bv = sm.red_v[0];
                bk = sm.red_k[0];
                for (int w = 1; w < NW * CL; ++w) argmin_merge(bv, bk, sm.red_v[w], sm.red_k[w]);
                const bool ok = bv < kInf;
                const int z1 = ok ? bk / KM : -1, z2 = ok ? bk % KM : -1;
                if constexpr (kFused)
                    backtrack_unit(un, md, sc, K, cidx, ubeta, ok ? bv : kInf, z1, z2, energy_out, assign_out, lane);
                else if (lane == 0) res[u] = UnitResult{ok ? bv : kInf, z1, z2, 0};
            }
            __syncthreads();
        }
    }
}

constexpr int kURW = 4;      // unroll of the triple loop in the forms of one unit per SM or cluster
constexpr int kFusedPerSm = 3;   // CTAs per SM of the fused variant (its argmin scratch is per CTA)

struct FusedArgs {
    const int *n_dev = nullptr;
    int n_from = -1, n_to = INT32_MAX;   // counts this launch solves: n_from < n <= n_to
    int64_t beta_cta = 0;
    float *energy = nullptr;
    int32_t *assign = nullptr;
};

template <int KM, int NT, int MB, int CT, int UR, bool kCount, bool kFused, int CL = 1>
cudaError_t launch_recurse_t(const Unit *units, int64_t n_units, const ModelRec *models, const SceneRec *scenes,
                             Params p, const int32_t *cand_idx, const float *cand_u, const int32_t *cand_cnt,
                             uint8_t *beta, UnitResult *res, int *work_counter, unsigned long long *evaluated,
                             const FusedArgs &fa, cudaStream_t st)
{
    // three CTAs of 256 threads per SM: 3 x (shared memory + 1 KB reserved) <= 228 KB
    static_assert(MB * (sizeof(Smem<KM, NT, CL>) + 1024) <= 228 * 1024, "recursion shared memory exceeds the CTAs' budget");
    auto kern = recurse_kernel<KM, NT, MB, CT, UR, kCount, kFused, CL>;
    const size_t smem = sizeof(Smem<KM, NT, CL>);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if constexpr (CL > 1) {   // a cluster per unit
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(n_units * CL));
        cfg.blockDim = dim3(NT);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = CL;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        prof_begin(kProfRecurse, st);
        e = cudaLaunchKernelEx(&cfg, kern, units, n_units, models, scenes, p, cand_idx, cand_u, cand_cnt, beta, res,
                               work_counter, evaluated, fa.n_dev, fa.n_from, fa.n_to, fa.beta_cta, fa.energy, fa.assign);
        prof_end(kProfRecurse, st);
        return e;
    }
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem)) != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    int64_t grid = (int64_t)sms * per_sm;
    if (grid > n_units) grid = n_units;
    if ((e = cudaMemsetAsync(work_counter, 0, sizeof(int), st)) != cudaSuccess) return e;
    prof_begin(kProfRecurse, st);
    if (kFused)   // the per-CTA scratch was sized for sms * kFusedPerSm CTAs
        grid = std::min<int64_t>(std::min<int64_t>(grid, (int64_t)sms * kFusedPerSm), n_units);
    kern<<<(unsigned)grid, NT, smem, st>>>(units, n_units, models, scenes, p, cand_idx, cand_u, cand_cnt, beta, res,
                                           work_counter, evaluated, fa.n_dev, fa.n_from, fa.n_to, fa.beta_cta, fa.energy,
                                           fa.assign);
    prof_end(kProfRecurse, st);
    return cudaGetLastError();
}

template <bool kCount, bool kFused>
cudaError_t dispatch(int variant, const Unit *units, int64_t n_units, const ModelRec *models, const SceneRec *scenes,
                     Params p, const int32_t *cand_idx, const float *cand_u, const int32_t *cand_cnt, uint8_t *beta,
                     UnitResult *res, int *work_counter, unsigned long long *evaluated, const FusedArgs &fa,
                     cudaStream_t st)
{
#define HGM_RECURSE(KM_, NT_, MB_, CT_, UR_)                                                                      \
    return launch_recurse_t<KM_, NT_, MB_, CT_, UR_, kCount, kFused>(units, n_units, models, scenes, p, cand_idx,  \
                                                                     cand_u, cand_cnt, beta, res, work_counter,   \
                                                                     evaluated, fa, st)
    if (p.K <= 32) {
        if (variant == 1) HGM_RECURSE(32, 128, 4, 8, 2);
        if (variant == 2) HGM_RECURSE(32, 128, 4, 4, 4);
        HGM_RECURSE(32, 128, 4, 4, 2);
    }
    if (variant == 1) HGM_RECURSE(64, 256, 3, 8, 2);
    if (variant == 2) HGM_RECURSE(64, 256, 3, 4, 4);
    HGM_RECURSE(64, 256, 3, 4, 2);
#undef HGM_RECURSE
}

int g_variant = 0;   // recursion variant: 0 = 4 c per tile, 1 = 8 c per tile, 2 = 4 c per tile, triple loop unrolled by 4

// At most one unit per SM: twice the threads per unit. A step's phases are chains of dependent operations that
// more threads per row and per tile round shorten (model of 30 points, 150 units against 153: K = 64 268 and 415 us,
// K = 32 160 and 201 us); with two units on an SM the second one's warps already fill the gaps (271 units of K = 64:
// 439 us with 512 threads each, 444 with 256).
template <bool kFused>
cudaError_t launch_wide(const Unit *units, int64_t n_units, const ModelRec *models, const SceneRec *scenes, Params p,
                        const int32_t *cand_idx, const float *cand_u, const int32_t *cand_cnt, uint8_t *beta,
                        UnitResult *res, int *work_counter, const FusedArgs &fa, cudaStream_t st)
{
    if (p.K <= 32)
        return launch_recurse_t<32, 256, 1, 4, kURW, false, kFused>(units, n_units, models, scenes, p, cand_idx, cand_u,
                                                                 cand_cnt, beta, res, work_counter, nullptr, fa, st);
    return launch_recurse_t<64, 512, 1, 4, kURW, false, kFused>(units, n_units, models, scenes, p, cand_idx, cand_u,
                                                             cand_cnt, beta, res, work_counter, nullptr, fa, st);
}

// Few units: a cluster of four CTAs per unit, a warp per row in each, while the clusters of all units surely find
// their SMs at once (five sixths of the SMs: clusters keep to one GPC). A step is then bound by its chain of
// dependent operations: about 1,200 cycles (K = 32) and 2,200 (K = 64) of row lists, 1,400 and 2,300 of theta(a->c),
// 2,000 and 4,000 of tiles, 1,000 of the cluster barrier. Two CTAs or half the threads per CTA were slower; theta(a->c)
// computed by quarters and written to all four CTAs was too (its barrier costs more than the directions), and two or
// four threads per tile changed nothing. 31 units of 16 points (K = 32): 67 -> 55 us; one to three fallback units of
// 256 points (K = 64): 1,970 -> 1,430 us, both against one CTA per unit.
constexpr int kCL = 4, kNT32 = 256, kNT64 = 512;

template <bool kFused>
cudaError_t launch_shared(const Unit *units, int64_t n_units, const ModelRec *models, const SceneRec *scenes, Params p,
                          const int32_t *cand_idx, const float *cand_u, const int32_t *cand_cnt, uint8_t *beta,
                          UnitResult *res, int *work_counter, const FusedArgs &fa, cudaStream_t st)
{
    if (p.K <= 32)
        return launch_recurse_t<32, kNT32, 1, 4, kURW, false, kFused, kCL>(units, n_units, models, scenes, p, cand_idx, cand_u,
                                                                       cand_cnt, beta, res, work_counter, nullptr, fa, st);
    return launch_recurse_t<64, kNT64, 1, 4, kURW, false, kFused, kCL>(units, n_units, models, scenes, p, cand_idx, cand_u,
                                                                   cand_cnt, beta, res, work_counter, nullptr, fa, st);
}

int64_t shared_units(int64_t sms) { return sms * 5 / (6 * kCL); }

int64_t wide_units()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return sms;
}

}  // namespace

namespace {
__global__ void model_geo_kernel(const float2 *__restrict__ xy, const int32_t *__restrict__ t, int M,
                                 float4 *__restrict__ geo)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M; i += gridDim.x * blockDim.x) {
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i >= 2) {
            const float2 mi = xy[i], mj = xy[i - 1], mk = xy[i - 2];
            const float A1 = signed_angle(mj, mi, mk);   // at i-1, from ->i to ->i-2
            const float A2 = signed_angle(mi, mj, mk);   // at i, from ->i-1 to ->i-2
            g = make_float4(A1, wrap_pi(__fadd_rn(__fsub_rn(A2, A1), kPi)), __int_as_float(t[i] - t[i - 1]),
                            __int_as_float(t[i - 1] - t[i - 2]));
        }
        geo[i] = g;
    }
}
}  // namespace

cudaError_t launch_model_geo(const float2 *xy, const int32_t *t, int M, float4 *geo, cudaStream_t st)
{
    if (M <= 0) return cudaSuccess;
    model_geo_kernel<<<(M + 127) / 128, 128, 0, st>>>(xy, t, M, geo);
    return cudaGetLastError();
}

cudaError_t preload_recurse()
{
    cudaFuncAttributes a;
    const void *kerns[] = {(const void *)recurse_kernel<32, 128, 4, 8, 2, false, false, 1>,
                           (const void *)recurse_kernel<32, 128, 4, 4, 4, false, false, 1>,
                           (const void *)recurse_kernel<32, 128, 4, 4, 2, false, false, 1>,
                           (const void *)recurse_kernel<64, 256, 3, 8, 2, false, false, 1>,
                           (const void *)recurse_kernel<64, 256, 3, 4, 4, false, false, 1>,
                           (const void *)recurse_kernel<64, 256, 3, 4, 2, false, false, 1>,
                           (const void *)recurse_kernel<32, 256, 1, 4, kURW, false, false, 1>,
                           (const void *)recurse_kernel<64, 512, 1, 4, kURW, false, false, 1>,
                           (const void *)recurse_kernel<32, kNT32, 1, 4, kURW, false, false, kCL>,
                           (const void *)recurse_kernel<64, kNT64, 1, 4, kURW, false, false, kCL>};
    for (const void *k : kerns) {
        cudaError_t e = cudaFuncGetAttributes(&a, k);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

int recurse_variant_count() { return 3; }
void set_recurse_variant(int v) { g_variant = (v >= 0 && v < 3) ? v : 0; }
int get_recurse_variant() { return g_variant; }

cudaError_t launch_recurse(const Unit *units, int64_t n_units, const ModelRec *models, const SceneRec *scenes,
                           Params p, const int32_t *cand_idx, const float *cand_u, const int32_t *cand_cnt,
                           uint8_t *beta, UnitResult *res, int *work_counter, cudaStream_t st)
{
    if (n_units <= 0) return cudaSuccess;
    if (p.K <= kShortK)   // short lists (pruned form)
        return launch_recurse_small(units, n_units, models, scenes, p, cand_idx, cand_u, cand_cnt, beta, res, st);
    const int64_t wide = wide_units();
    if (n_units <= shared_units(wide))
        return launch_shared<false>(units, n_units, models, scenes, p, cand_idx, cand_u, cand_cnt, beta, res,
                                    work_counter, FusedArgs{}, st);
    if (n_units <= wide)
        return launch_wide<false>(units, n_units, models, scenes, p, cand_idx, cand_u, cand_cnt, beta, res, work_counter,
                                  FusedArgs{}, st);
    return launch_recurse_variant(units, n_units, models, scenes, p, cand_idx, cand_u, cand_cnt, beta, res, work_counter, st);
}

cudaError_t launch_recurse_variant(const Unit *units, int64_t n_units, const ModelRec *models, const SceneRec *scenes,
                                   Params p, const int32_t *cand_idx, const float *cand_u, const int32_t *cand_cnt,
                                   uint8_t *beta, UnitResult *res, int *work_counter, cudaStream_t st)
{
    if (n_units <= 0) return cudaSuccess;
    return dispatch<false, false>(g_variant, units, n_units, models, scenes, p, cand_idx, cand_u, cand_cnt, beta,
                                  res, work_counter, nullptr, FusedArgs{}, st);
}

int64_t recurse_fused_scratch(int K, int max_M)
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess)
        return -1;
    const int64_t per = ((int64_t)std::max(max_M - 2, 1) * K * K + 255) / 256 * 256;
    return (int64_t)sms * kFusedPerSm * per;
}

cudaError_t launch_recurse_fused(const Unit *units, int64_t n_max, const int *n_dev, const ModelRec *models,
                                 const SceneRec *scenes, Params p, const int32_t *cand_idx, const float *cand_u,
                                 const int32_t *cand_cnt, uint8_t *scratch, int max_M, float *energy,
                                 int32_t *assign, int *work_counter, cudaStream_t st)
{
    if (n_max <= 0) return cudaSuccess;
    FusedArgs fa;
    fa.n_dev = n_dev;
    fa.beta_cta = ((int64_t)std::max(max_M - 2, 1) * p.K * p.K + 255) / 256 * 256;
    fa.energy = energy;
    fa.assign = assign;
    // the count is known on the device only: a launch for every range of counts (an idle one costs 2-3 us)
    const int64_t few = wide_units(), least = shared_units(few);
    fa.n_to = (int)least;
    cudaError_t e = launch_shared<true>(units, std::min(n_max, least), models, scenes, p, cand_idx, cand_u, cand_cnt,
                                        scratch, nullptr, work_counter, fa, st);
    if (e != cudaSuccess || n_max <= least) return e;
    fa.n_from = (int)least;
    fa.n_to = (int)few;
    e = launch_wide<true>(units, std::min(n_max, few), models, scenes, p, cand_idx, cand_u, cand_cnt, scratch, nullptr,
                          work_counter, fa, st);
    if (e != cudaSuccess || n_max <= few) return e;
    fa.n_from = (int)few;
    fa.n_to = INT32_MAX;
    return dispatch<false, true>(0, units, n_max, models, scenes, p, cand_idx, cand_u, cand_cnt, scratch, nullptr,
                                 work_counter, nullptr, fa, st);
}

cudaError_t launch_recurse_count(const Unit *units, int64_t n_units, const ModelRec *models, const SceneRec *scenes,
                                 Params p, const int32_t *cand_idx, const float *cand_u, const int32_t *cand_cnt,
                                 uint8_t *beta, UnitResult *res, int *work_counter, unsigned long long *evaluated,
                                 cudaStream_t st)
{
    if (n_units <= 0) return cudaSuccess;
    return dispatch<true, false>(g_variant, units, n_units, models, scenes, p, cand_idx, cand_u, cand_cnt, beta,
                                 res, work_counter, evaluated, FusedArgs{}, st);
}

}  // namespace hgm
