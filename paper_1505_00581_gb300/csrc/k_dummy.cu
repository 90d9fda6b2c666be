// k_dummy.cu -- the recursion with the dummy assignment of Eq. 2 (reading R5).
//
// Every candidate list C_i(o) gets one more slot, eps, after its real candidates, with U(eps) = lambda1 W^d. A term
// that involves eps vanishes (Delta(i,j) if z_i or z_j is eps; D^g if any point of the triangle is), and a triple
// holding eps is feasible iff its real points, in chain order, are distinct, time-ordered and less than T frames
// apart. So the all-eps chain is always feasible and every offset has a finite optimum.
//
// The real cells (b, c) run as in k_recurse.cu (its comments hold here: row lists from registers, tiles of four c of
// one b in decreasing kept count, the next step's base written with alpha), with three differences:
//  * a cell starts from the triple (eps, b, c), which is feasible and costs base(eps, b) alone, so no a above it is
//    kept; the row's smallest base a1 lowers that bound to base(a1, b) + max D^g when a1 is feasible with every open
//    c and with (b, eps). With W^d small most rows keep nothing, and their cells need no direction at all;
//  * theta(a->c) is computed only for the a that some row keeps, once the kept lists are there;
//  * the cells that hold eps are minima without a geometric term: (b, eps) over the a within T of b, by the row's
//    threads; (eps, c) over base(a, eps), by the threads of c; (eps, eps) by one warp. Their base values are three
//    small arrays, kept for the coming and the current step.
// Ties prefer the lower slot, eps last: a cell's walk starts from the next float above base(eps, b), at most +inf, so a
// real a of equal cost replaces it. The argmin slots go to a per-CTA global scratch, and the CTA backtracks its own unit (Eq.
// 12); eps is reported as -2 in the assignment.
//
// Bound by issue and the latency of the step's phases. Measured with the earlier kernel (a warp per row ranking the
// kept a by counting, base, row and list passes between five barriers, two CTAs per SM) and with this one, three CTAs
// per SM: 2,710 units of up to 64 points at W^d = 8 (K = 64) 5,707 -> 2,208 us.
#include <algorithm>
#include <climits>

#include "hgm_internal.cuh"
#include "recurse_lists.cuh"

namespace hgm {
namespace {

template <int KM, int NT>
struct DummySmem {
    static constexpr int FS = KM + 1, SS = KM + 4, RS = KM + 4, AS = KM + 4;   // as in k_recurse.cu
    float2 fb[KM * FS];                   // per b: kept (base, p1) in increasing a
    float r[KM * RS];                     // theta(a->c) or +inf at a*RS + c | 16 bytes of tile_b per row
    float alpha[KM * AS];                 // base(a,b) of the coming step at b*AS + a | key, be, ea
    uint8_t fs[KM * SS];                  // slot of each kept entry, | 0x80 when a lies at b's position | tile info
    List<KM> list[3];
    float ea1[KM];
    float4 geo[2];
    float ee[2];                          // base(eps, eps) of step i at ee[i & 1]
    float red_v[NT / 32];
    int32_t red_k[NT / 32];
    int32_t ntile, unit;
    int32_t coin[2];
    unsigned akept[2];                    // a kept by some row (bits of slots 0-31, 32-63)

    __device__ uint8_t &tile_b(int t) { return reinterpret_cast<uint8_t *>(&r[(t >> 4) * RS + KM])[t & 15]; }
    __device__ int32_t &key(int b) { return reinterpret_cast<int32_t *>(alpha)[b * AS + KM]; }
    __device__ int32_t &info(int b) { return *reinterpret_cast<int32_t *>(fs + b * SS + KM); }
    // step i: base(eps, b) and base(a, eps), of parity i & 1
    __device__ float &be(int par, int b) { return alpha[b * AS + KM + 1 + par]; }
    __device__ float &ea(int par, int a) { return par ? ea1[a] : alpha[a * AS + KM + 3]; }
};

// kCount = true builds the accounting variant: identical work, plus a count of the (a, open cell) triples the walks
// evaluate, added to *evaluated (work accounting; not used on the timed path).
template <int KM, int NT, int MB, bool kCount>
__global__ void __launch_bounds__(NT, MB) dummy_recurse_kernel(
    const Unit *__restrict__ units, int64_t n_units, const ModelRec *__restrict__ models,
    const SceneRec *__restrict__ scenes, Params p, float wd, const int32_t *__restrict__ cand_idx,
    const float *__restrict__ cand_u, const int32_t *__restrict__ cand_cnt, uint8_t *__restrict__ scratch,
    int64_t scratch_per_cta, int *__restrict__ work_counter, float *__restrict__ energy, int32_t *__restrict__ assign,
    unsigned long long *__restrict__ evaluated)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using SM = DummySmem<KM, NT>;
    SM &sm = *reinterpret_cast<SM *>(smem_raw);
    constexpr int RS = SM::RS, AS = SM::AS, FS = SM::FS, SS = SM::SS;
    constexpr int NW = NT / 32, CT = 4;
    constexpr int TPB = NT / KM, AH = KM / TPB;   // threads per b (and per c), slots a per thread
    constexpr int E = KM, LS = KM + 4;            // slot of eps in the argmin tables, their row stride
    static_assert(TPB == 4, "threads per b");
    const unsigned full = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = p.K, T = p.T;
    const float lam2 = p.lambda2, lam23 = __fmul_rn(p.lambda2, p.lambda3);
    const float ueps = __fmul_rn(p.lambda1, wd);
    const float gmax = lam23 * kGeoMax;
    const int h = tid % TPB, row = tid / TPB, rot = h;
    uint8_t *beta = scratch + (int64_t)blockIdx.x * scratch_per_cta;
    unsigned long long n_eval = 0;
    for (;;) {
        if (tid == 0) sm.unit = atomicAdd(work_counter, 1);
        __syncthreads();
        const int64_t u = sm.unit;
        if (u >= n_units) break;
        const Unit un = units[u];
        const ModelRec md = models[un.model];
        const SceneRec sc = scenes[un.scene];
        const int M = md.M;
        const int32_t *cidx = cand_idx + un.cand;
        const float *cu = cand_u + un.cand;
        const int32_t *ccnt = cand_cnt + un.cand / K;
        for (int q = 1; q <= 3; ++q)
            load_list<KM>(sm.list[(M - q) % 3], sc, cidx + (int64_t)(M - q) * K, cu + (int64_t)(M - q) * K, ccnt[M - q],
                          tid, NT);
        if (tid == 0) {
            sm.geo[(M - 1) & 1] = md.geo[M - 1];
            sm.coin[0] = sm.coin[1] = 0;
            sm.akept[0] = sm.akept[1] = 0u;
            sm.ee[(M - 1) & 1] = ueps;
        }
        __syncthreads();
        {   // the first step's base: alpha_{M+1} == 0 (Eq. 11)
            const List<KM> &LA = sm.list[(M - 1) % 3], &LB = sm.list[(M - 2) % 3];
            const int dt_ab = __float_as_int(sm.geo[(M - 1) & 1].z);
            for (int e = tid; e < KM * KM; e += NT) {
                const int b = e / KM, a = e % KM;
                const bool ok = a < LA.n && b < LB.n && LA.t[a] >= LB.t[b] && LA.idx[a] != LB.idx[b];
                sm.alpha[b * AS + a] = ok ? base_cost(LA.u[a], lam2, dt_ab, LA.t[a], LB.t[b], 0.0f) : kInf;
            }
            if (tid < KM) {
                sm.be((M - 1) & 1, tid) = ueps;
                sm.ea((M - 1) & 1, tid) = LA.u[tid];
            }
        }
        __syncthreads();

        for (int i = M - 1; i >= 2; --i) {
            List<KM> &LA = sm.list[i % 3];
            List<KM> &LB = sm.list[(i - 1) % 3];
            List<KM> &LC = sm.list[(i - 2) % 3];
            const int par = i & 1, npar = par ^ 1;
            const float4 g = sm.geo[par];
            const float A1 = g.x, k2 = g.y;
            const float k2c = wrap_pi(__fsub_rn(k2, kPi));   // a and b at the same position (reading R1)
            const int dt_bc = __float_as_int(g.w);
            const int na = LA.n, nb = LB.n, nc = LC.n;
            uint8_t *bstep = beta + (int64_t)(i - 2) * (KM + 1) * LS;
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
            if (tid == NT - 1 && i >= 3) sm.geo[npar] = md.geo[i - 1];
            auto lower_bound = [](const int32_t *arr, int n, int x) {
                int l = 0;
                while (l < n) {
                    const int mid = (l + n) >> 1;
                    if (arr[mid] < x) l = mid + 1;
                    else n = mid;
                }
                return l;
            };
            const int base_lane = lane & ~(TPB - 1);
            // the a of a time range: those not before frame t0 (range.x) and less than T frames after it (.y)
            auto time_range = [&](int t0, int n) {
                const int x = (h & 1) == 0 ? t0 : (T > 0 && t0 <= INT_MAX - T ? t0 + T : INT_MAX);
                const int f = lower_bound(LA.t, n, x);
                const int l = __shfl_sync(full, f, base_lane), r = __shfl_sync(full, f, base_lane + 1);
                return make_int2(l, T > 0 ? r : n);
            };
            // (value, slot) minimum over the threads of a row, ties to the lower slot
            auto row_min = [&](float &v, int &s) {
#pragma unroll
                for (int off = 1; off < TPB; off <<= 1)
                    argmin_merge(v, s, __shfl_xor_sync(full, v, off), __shfl_xor_sync(full, s, off));
            };

            // ---- phase 1: the kept a list of b = row, and the cell (b, eps)
            {
                const int b = row;
                const bool inb = b < nb;
                float2 pb = make_float2(0.f, 0.f);
                int tb = 0, ib = -1;
                if (inb) { pb = LB.xy[b]; tb = LB.t[b]; ib = LB.idx[b]; }
                const float *arow = sm.alpha + b * AS + AH * h;
                const int2 ra = time_range(tb, inb ? na : 0);
                const int j0 = ra.x - AH * h, jT = ra.y - AH * h, j1 = (inb ? na : 0) - AH * h;
                float v[AH], m1 = kInf, mE = kInf;
                int s1 = 1 << 20, sE = 1 << 20;
#pragma unroll
                for (int k = 0; k < AH; ++k) {
                    const int j = (k + rot) & (AH - 1);
                    const float x = arow[j];
                    v[k] = j >= j0 && j < j1 ? x : kInf;
                    m1 = fminf(m1, v[k]);
                    mE = fminf(mE, j < jT ? v[k] : kInf);
                }
#pragma unroll
                for (int k = 0; k < AH; ++k) {
                    const int j = (k + rot) & (AH - 1), a = AH * h + j;
                    if (v[k] == m1) s1 = min(s1, a);
                    if (v[k] == mE && j < jT) sE = min(sE, a);
                }
                row_min(m1, s1);
                row_min(mE, sE);
                const bool any = m1 < kInf;
                if (!any) s1 = 0;
                const int tw = LA.t[s1], iw = any ? LA.idx[s1] : -2;
                // searches of list C (time order, scene index order), one per lane: c not after b, c too far from the
                // witness, c too far from b, the witness's point
                const int q = h & 3;
                const int x = q == 0 ? tb + 1 : q == 1 ? (T > 0 ? tw - T + 1 : INT_MIN)
                                            : q == 2 ? (T > 0 ? tb - T + 1 : INT_MIN) : iw;
                int f = lower_bound(q < 3 ? LC.t : LC.idx, nc, x);
                if (q == 3 && !(f < nc && LC.idx[f] == x)) f = KM;
                int ccount = __shfl_sync(full, f, base_lane);
                if (!inb) ccount = 0;
                const int nT = min(__shfl_sync(full, f, base_lane + 1), ccount);
                const int nB = min(__shfl_sync(full, f, base_lane + 2), ccount);
                const int pw = __shfl_sync(full, f, base_lane + 3);
                const float beb = inb ? sm.be(par, b) : kInf;
                const bool live = any && ccount > 0;
                float thr = beb;
                {
                    // the open c are those from nB on but b's own point, which is as far from the witness as b is
                    const float lower = m1 + gmax + 1e-6f * fabsf(m1);
                    const bool bad = (T > 0 && tw - tb >= T) || nT > nB || (pw < ccount && pw >= nB);
                    if (lower < thr && !bad) thr = lower;
                }
                thr = live ? fminf(thr, 3.402823466e38f) : -kInf;
                unsigned mk = 0;
#pragma unroll
                for (int k = 0; k < AH; ++k)
                    if (v[k] <= thr) mk |= 1u << k;
                mk = ((mk << rot) | (mk >> (AH - rot))) & ((1u << AH) - 1);
                int pos = 0, kept = __popc(mk);
#pragma unroll
                for (int off = 1; off < TPB; off <<= 1) {
                    const int o = __shfl_xor_sync(full, kept, off);
                    if (h & off) pos += o;
                    kept += o;
                }
                if (mk) {
                    const unsigned long long bits = (unsigned long long)mk << (AH * h);
                    atomicOr(&sm.akept[(AH * h) >> 5], (unsigned)(bits >> ((AH * h) & ~31)));
                }
                for (unsigned m = mk; m; m &= m - 1, ++pos) {
                    const int j = __ffs((int)m) - 1, a = AH * h + j;
                    const float2 pa = LA.xy[a];
                    const bool same = pa.x == pb.x && pa.y == pb.y;
                    if (same) sm.coin[par] = 1;
                    sm.fb[b * FS + pos] = make_float2(arow[j], wrap_pi(__fadd_rn(A1, direction(pb, pa))));
                    sm.fs[b * SS + pos] = (uint8_t)(a | (same ? 0x80 : 0));
                }
                if (h == 0) {
                    const int nt_b = (ccount + CT - 1) / CT;
                    const int key = nt_b > 0 ? ((kept + 1) << 8) | (255 - b) : 0;
                    sm.key(b) = (key << 5) | nt_b;
                    if (inb) {   // the cell (b, eps): base alone; next step's base(a = b, eps) = U(b) + alpha
                        const bool real = mE < kInf && mE <= beb;
                        const float al = real ? mE : beb;
                        sm.ea(npar, b) = i > 2 ? __fadd_rn(LB.u[b], al) : al;
                        bstep[b * LS + E] = (uint8_t)(real ? sE : E);
                    }
                }
            }
            if (pf && tid < pf_n) {
                pf_xy = sc.xy[pf_j];
                pf_t = sc.t[pf_j];
            }
            // the cells (eps, c), c = row: base(a, eps) of the a that may follow c
            const bool inc_c = row < nc;
            const int tc_row = inc_c ? LC.t[row] : 0, ic_row = inc_c ? LC.idx[row] : -3;
            const int2 rc_range = time_range(tc_row, inc_c ? na : 0);
            {
                float m = kInf;
                int s = 1 << 20;
                for (int a = rc_range.x + h; a < rc_range.y; a += TPB) {
                    const float x = sm.ea(par, a);
                    if (LA.idx[a] != ic_row && x < m) { m = x; s = a; }
                }
                row_min(m, s);
                if (h == 0 && inc_c) {
                    const bool real = m < kInf && m <= sm.ee[par];
                    const float al = real ? m : sm.ee[par];
                    sm.be(npar, row) = i > 2 ? __fadd_rn(ueps, al) : al;
                    bstep[E * LS + row] = (uint8_t)(real ? s : E);
                }
            }
            if (warp == NW - 1) {   // the cell (eps, eps)
                float m = kInf;
                int s = 1 << 20;
                for (int a = lane; a < na; a += 32) {
                    const float x = sm.ea(par, a);
                    if (x < m) { m = x; s = a; }
                }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1)
                    argmin_merge(m, s, __shfl_xor_sync(full, m, off), __shfl_xor_sync(full, s, off));
                if (lane == 0) {
                    const bool real = m < kInf && m <= sm.ee[par];
                    const float al = real ? m : sm.ee[par];
                    sm.ee[npar] = i > 2 ? __fadd_rn(ueps, al) : al;
                    bstep[E * LS + E] = (uint8_t)(real ? s : E);
                }
            }
            __syncthreads();

            // theta(a->c) of the kept a, c = row (rows from the first a with t'(a) >= t'(c), as in k_recurse.cu)
            if (inc_c) {
                const unsigned k0 = sm.akept[0], k1 = sm.akept[1];
                if (k0 | k1) {
                    const float2 pc = LC.xy[row];
                    for (int a = rc_range.x + h; a < na; a += TPB) {
                        if (!(((a < 32 ? k0 : k1) >> (a & 31)) & 1u)) continue;
                        sm.r[a * RS + row] = a < rc_range.y && LA.idx[a] != ic_row ? direction(LA.xy[a], pc) : kInf;
                    }
                }
            }
            // tile layout (as in k_recurse.cu)
            {
                const int b = row, wb = sm.key(b), key = wb >> 5, nt_b = wb & 31;
                int before = 0, total = 0;
                for (int b2 = h; b2 < KM; b2 += TPB) {
                    const int w = sm.key(b2);
                    total += w & 31;
                    if ((w >> 5) > key) before += w & 31;
                }
#pragma unroll
                for (int off = 1; off < TPB; off <<= 1) {
                    before += __shfl_xor_sync(full, before, off);
                    total += __shfl_xor_sync(full, total, off);
                }
                if (h == 0) sm.info(b) = before << 12 | max((key >> 8) - 1, 0) << 5 | nt_b;
                for (int t = h; t < nt_b; t += TPB) sm.tile_b(before + t) = (uint8_t)b;
                if (tid == 0) {
                    sm.ntile = total;
                    sm.coin[npar] = 0;
                }
            }
            __syncthreads();

            // list A is not read from here on: its buffer receives list C of the next step
            if (i >= 3 && tid < KM) {
                const bool ok = tid < pf_n;
                LA.idx[tid] = ok ? pf_j : -1;
                LA.xy[tid] = pf_xy;
                LA.t[tid] = pf_t;
                LA.u[tid] = ok ? pf_u : kInf;
                if (tid == 0) {
                    LA.n = pf_n;
                    sm.akept[0] = sm.akept[1] = 0u;
                }
            }
            // ---- phase 3: tiles (b, four consecutive c)
            const int ntile = sm.ntile;
            const bool coin = sm.coin[par] != 0;
            const unsigned long long lamp = pk2(lam23, lam23);
            for (int r0 = 0; r0 < ntile; r0 += NT) {
                const int tile = r0 + (((r0 / NT) & 1) ? NT - 1 - tid : tid);
                if (tile >= ntile) continue;
                const int b = sm.tile_b(tile);
                const int info = sm.info(b);
                const int c0 = (tile - (info >> 12)) * CT;
                const int nf = (info >> 5) & 127;
                const float2 pb = LB.xy[b];
                const int tb = LB.t[b], ib = LB.idx[b];
                const float ub = LB.u[b], beb = sm.be(par, b);
                // a real a of equal cost replaces eps: start just above base(eps, b), but not above +inf (a dear
                // dummy's sums overflow): the next bit pattern is a NaN, which no cost is below
                const float start = __uint_as_float(min(__float_as_uint(beb) + 1u, __float_as_uint(kInf)));
                float best[CT];
                int arg[CT], tcq[CT];
                bool open[CT];
                const int4 t4 = *reinterpret_cast<const int4 *>(&LC.t[c0]);
                const int4 i4 = *reinterpret_cast<const int4 *>(&LC.idx[c0]);
                const int tv[4] = {t4.x, t4.y, t4.z, t4.w}, iv[4] = {i4.x, i4.y, i4.z, i4.w};
#pragma unroll
                for (int q = 0; q < CT; ++q) {
                    tcq[q] = tv[q];
                    open[q] = c0 + q < nc && tv[q] <= tb && iv[q] != ib && (T <= 0 || tb - tv[q] < T);
                    best[q] = open[q] ? start : kInf;
                    arg[q] = open[q] ? E : kNoSlot;
                }
                if (nf > 0) {
                    const float4 xa = *reinterpret_cast<const float4 *>(&LC.xy[c0]);
                    const float4 xb = *reinterpret_cast<const float4 *>(&LC.xy[c0 + 2]);
                    const float2 xv[4] = {make_float2(xa.x, xa.y), make_float2(xa.z, xa.w), make_float2(xb.x, xb.y),
                                          make_float2(xb.z, xb.w)};
                    float q1[CT];
#pragma unroll
                    for (int q = 0; q < CT; ++q) {
                        const float d = direction(pb, xv[q]);   // theta(b->c)
                        q1[q] = open[q] ? d : kInf;
                    }
                    const unsigned long long q1a = pk2(q1[0], q1[1]), q1b = pk2(q1[2], q1[3]);
                    const float2 *fb = sm.fb + b * FS;
                    const uint8_t *fs = sm.fs + b * SS;
                    if constexpr (kCount) n_eval += nf * ((int)open[0] + (int)open[1] + (int)open[2] + (int)open[3]);
#pragma unroll 2
                    for (int k = 0; k < nf; ++k) {
                        const float2 e = fb[k];
                        const int fa = fs[k], a = fa & 0x7f;
                        const float p2 = __fadd_rn(e.y, coin && (fa & 0x80) ? k2c : k2);
                        const float4 r4 = *reinterpret_cast<const float4 *>(sm.r + a * RS + c0);
                        const unsigned long long bp = pk2(e.x, e.x), p1p = pk2(e.y, e.y), p2p = pk2(p2, p2);
                        float v[4];
                        triple_cost2(bp, p1p, p2p, q1a, pk2(r4.x, r4.y), lamp, v[0], v[1]);
                        triple_cost2(bp, p1p, p2p, q1b, pk2(r4.z, r4.w), lamp, v[2], v[3]);
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (v[q] < best[q]) { best[q] = v[q]; arg[q] = a; }
                    }
                }
                uint32_t packed = 0;
#pragma unroll
                for (int q = 0; q < CT; ++q) {
                    const int c = c0 + q;
                    if (arg[q] == E) best[q] = beb;
                    const float al = cell_alpha(best[q], lam2, dt_bc, tb, tcq[q]);
                    const float out = i > 2 ? base_cost(ub, lam2, dt_bc, tb, tcq[q], al) : al;
                    if (c < nc) sm.alpha[c * AS + b] = out;
                    packed |= (uint32_t)arg[q] << (8 * q);
                }
                *reinterpret_cast<uint32_t *>(bstep + b * LS + c0) = packed;   // rows of whole words, eps after them
            }
            if (i == 2) {   // Eq. 13 reads every cell of the last step
                for (int b = warp; b < nb; b += NW) {
                    const int covered = (sm.info(b) & 31) * CT;
                    for (int c = covered + lane; c < nc; c += 32) sm.alpha[c * AS + b] = kInf;
                }
            }
            __syncthreads();
        }

        // Eq. 13 over (z_1 = c, z_2 = b) in C_1 + eps, C_2 + eps: U + U + alpha_3(z_2, z_1); alpha of the cells with
        // eps stands where the step i = 2 left it (parity 1)
        {
            const List<KM> &L0 = sm.list[0], &L1 = sm.list[1];
            const int n0 = L0.n, n1 = L1.n;
            float bv = kInf;
            int bk = 0x7fffffff;
            for (int e = tid; e < (KM + 1) * (KM + 1); e += NT) {
                const int c = e / (KM + 1), b = e % (KM + 1);
                if (!((c < n0 || c == E) && (b < n1 || b == E))) continue;
                const float u1 = c == E ? ueps : L0.u[c], u2 = b == E ? ueps : L1.u[b];
                const float al = c == E ? (b == E ? sm.ee[1] : sm.ea(1, b)) : (b == E ? sm.be(1, c) : sm.alpha[c * AS + b]);
                argmin_merge(bv, bk, __fadd_rn(__fadd_rn(u1, u2), al), e);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1)
                argmin_merge(bv, bk, __shfl_xor_sync(full, bv, off), __shfl_xor_sync(full, bk, off));
            if (lane == 0) { sm.red_v[warp] = bv; sm.red_k[warp] = bk; }
            __syncthreads();
            if (warp == 0) {
                bv = sm.red_v[0];
                bk = sm.red_k[0];
                for (int w = 1; w < NW; ++w) argmin_merge(bv, bk, sm.red_v[w], sm.red_k[w]);
                const bool ok = bv < kInf;
                if (energy && lane == 0) energy[un.out_e] = ok ? bv : kInf;
                if (assign) {   // Eq. 12, as backtrack_unit: every lane walks, the lanes then write 32 points at once
                    int32_t *out = assign + un.out_a;
                    const int z1 = ok ? bk / (KM + 1) : 0, z2 = ok ? bk % (KM + 1) : 0;
                    int s2 = z1, s1 = z2;
                    for (int i0 = 0; i0 < M; i0 += 32) {
                        int mine = kNoSlot;
                        for (int i = i0; i < min(M, i0 + 32) && ok; ++i) {
                            int s0 = i == 0 ? z1 : z2;
                            if (i >= 2) {
                                s0 = beta[((int64_t)(i - 2) * (KM + 1) + s1) * LS + s2];
                                s2 = s1;
                                s1 = s0;
                            }
                            if (i - i0 == lane) mine = s0;
                        }
                        const int i = i0 + lane;
                        if (i < M)
                            out[md.perm[i]] = mine == E ? -2 : mine == kNoSlot ? -1 : sc.perm[cidx[(int64_t)i * K + mine]];
                    }
                }
            }
            __syncthreads();   // tables, lists and the reduction slots are reused by the next unit
        }
    }
    if constexpr (kCount) {
        if (n_eval) atomicAdd(evaluated, n_eval);
    }
}

constexpr int kPerSm64 = 3, kPerSm32 = 4;   // CTAs per SM for lists of up to 64 and 32 candidates

template <int KM, int NT, int MB>
cudaError_t launch_dummy_t(const Unit *units, int64_t n_units, const ModelRec *models, const SceneRec *scenes, Params p,
                           float wd, const int32_t *cand_idx, const float *cand_u, const int32_t *cand_cnt,
                           uint8_t *scratch, int64_t per_cta, int grid, int *work_counter, float *energy,
                           int32_t *assign, unsigned long long *evaluated, cudaStream_t st)
{
    static_assert(MB * (sizeof(DummySmem<KM, NT>) + 1024) <= 228 * 1024, "shared memory exceeds the CTAs' budget");
    const size_t smem = sizeof(DummySmem<KM, NT>);
    auto kern = evaluated ? dummy_recurse_kernel<KM, NT, MB, true> : dummy_recurse_kernel<KM, NT, MB, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaMemsetAsync(work_counter, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    prof_begin(kProfRecurse, st);
    kern<<<(unsigned)std::min<int64_t>(n_units, grid), NT, smem, st>>>(units, n_units, models, scenes, p, wd, cand_idx,
                                                                        cand_u, cand_cnt, scratch, per_cta, work_counter,
                                                                        energy, assign, evaluated);
    e = cudaGetLastError();
    prof_end(kProfRecurse, st);
    return e;
}

int64_t dummy_cta_bytes(int K, int max_M)
{
    const int64_t KM = K <= 32 ? 32 : 64;
    return (std::max(max_M - 2, 1) * (KM + 1) * (KM + 4) + 15) / 16 * 16;
}

}  // namespace

int64_t dummy_scratch_bytes(int K, int max_M, int grid) { return grid * dummy_cta_bytes(K, max_M); }

// As many CTAs as fill the SMs, fewer where a long model's argmin scratch would take more than `room` bytes and more
// than two CTAs per SM with tables of exactly (K+1)^2 would: 450,000 points at K = 4 are 535 MB per CTA, 325 GB in all.
int dummy_grid(int K, int max_M, int64_t room)
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess)
        return 0;
    const int64_t exact = (int64_t)sms * 2 * std::max(max_M - 2, 1) * (K + 1) * (K + 1);
    const int64_t fit = std::max<int64_t>(std::max(room, exact) / dummy_cta_bytes(K, max_M), 1);
    return (int)std::min<int64_t>(fit, sms * (K <= 32 ? kPerSm32 : kPerSm64));
}

cudaError_t launch_recurse_dummy(const Unit *units, int64_t n_units, const ModelRec *models, const SceneRec *scenes,
                                 Params p, float wd, const int32_t *cand_idx, const float *cand_u,
                                 const int32_t *cand_cnt, uint8_t *scratch, int max_M, int grid, int *work_counter,
                                 float *energy, int32_t *assign, unsigned long long *evaluated, cudaStream_t st)
{
    if (n_units <= 0) return cudaSuccess;
    if (p.K > kMaxK) return cudaErrorInvalidValue;
    const int64_t per_cta = dummy_cta_bytes(p.K, max_M);
    if (p.K <= 32)
        return launch_dummy_t<32, 128, kPerSm32>(units, n_units, models, scenes, p, wd, cand_idx, cand_u, cand_cnt, scratch,
                                                 per_cta, grid, work_counter, energy, assign, evaluated, st);
    return launch_dummy_t<64, 256, kPerSm64>(units, n_units, models, scenes, p, wd, cand_idx, cand_u, cand_cnt, scratch,
                                             per_cta, grid, work_counter, energy, assign, evaluated, st);
}

}  // namespace hgm
