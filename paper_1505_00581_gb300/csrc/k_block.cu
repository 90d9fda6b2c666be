// k_block.cu -- the whole-block problem: every scene point is a candidate of every model point (the
// paper's own formulation, Sec. 2.2 and Sec. 3), no time offsets. The trellis of Eq. 10 is S x S per
// step; causality and temporal closeness (Eqs. 7-8) restrict z_{i-2} to the points of the T frames up
// to z_{i-1}'s (the band of Sec. 3.3), and z_i to the frames [t'(z_{i-1}), t'(z_{i-2}) + T) through the
// minnode table (Sec. 3.5).
//
// Two kernels. block_cluster_kernel keeps a pair's whole trellis step in shared memory, split over the CTAs of a
// thread-block cluster where one CTA's share would be too large or most SMs would idle; block_recurse_kernel is
// the general form (bands of any size) with its tables in global memory.
//
// Cells: point b owns the cells (b, c) for c in [lo(b), hi(b)), lo(b) = minnode(t'(b) - T + 1), hi(b) =
// minnode(t'(b) + 1); the cell (b, b) is kept (always +inf) so that a cell's index is cs(b) + c - lo(b). The
// argmin of every cell is stored as a 16-bit offset from minnode(t'(b)).
#include <cooperative_groups.h>

#include "hgm_internal.cuh"
#include "recurse_common.cuh"

namespace hgm {
namespace {

constexpr int kBlockThreads = 256;       // many units: several CTAs per SM
constexpr int kBlockThreadsWide = 1024;  // fewer units than SMs: one wide CTA per unit (latency-bound steps)
constexpr int kBuckets = 64;             // classes of a counts in which cells are ordered
constexpr int kMinShare = 320;           // cells of a cluster's CTA below which a step is mostly the cluster barrier

__global__ void block_cells_kernel(const int64_t *__restrict__ cs, int S, int32_t *__restrict__ cellb)
{
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < S; b += gridDim.x * blockDim.x)
        for (int64_t k = cs[b]; k < cs[b + 1]; ++k) cellb[k] = b;
}

__global__ void block_dirs_kernel(const float2 *__restrict__ xy, const int32_t *__restrict__ lo,
                                  const int64_t *__restrict__ cs, const int32_t *__restrict__ cellb, int64_t cells,
                                  float *__restrict__ dirf, float *__restrict__ dirb)
{
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < cells; k += (int64_t)gridDim.x * blockDim.x) {
        const int b = cellb[k];
        const int c = lo[b] + (int)(k - cs[b]);
        dirf[k] = direction(xy[b], xy[c]);
        dirb[k] = direction(xy[c], xy[b]);
    }
}

struct InitBest {
    float v;
    int c, b;
};

// (v, c, b) ordered by v, then by the slot of z_1 (= c), then of z_2 (= b): Eq. 13 with reading R6.
__device__ __forceinline__ bool init_better(float v, int c, int b, const InitBest &o)
{
    if (v != o.v) return v < o.v;
    if (c != o.c) return c < o.c;
    return b < o.b;
}

// The general form: alpha_{i+1} and alpha_i in a per-CTA global scratch, directions from per-scene band tables.
template <int NT>
__global__ void __launch_bounds__(NT, 1) block_recurse_kernel(
    const BlockUnit *__restrict__ units, int n_units, const ModelRec *__restrict__ models,
    const SceneRec *__restrict__ scenes, const BlockGeo *__restrict__ geos, Params p, uint16_t *__restrict__ beta,
    float *__restrict__ scratch, int64_t scratch_cells, float *__restrict__ energy, int32_t *__restrict__ assign)
{
    __shared__ InitBest red[NT / 32];
    const float lam2 = p.lambda2, lam23 = __fmul_rn(p.lambda2, p.lambda3);
    const float inf = __int_as_float(0x7f800000);
    for (int u = blockIdx.x; u < n_units; u += gridDim.x) {
        const BlockUnit un = units[u];
        const ModelRec md = models[un.model];
        const SceneRec sc = scenes[un.scene];
        const BlockGeo g = geos[un.scene];
        const int64_t C = g.cells;
        float *an = scratch + (int64_t)blockIdx.x * 2 * scratch_cells;
        float *ac = an + scratch_cells;
        const int M = md.M;
        for (int i = M - 1; i >= 2; --i) {
            const float2 mi = md.xy[i], mj = md.xy[i - 1], mk = md.xy[i - 2];
            const float A1 = signed_angle(mj, mi, mk);   // at i-1, from ->i to ->i-2
            const float A2 = signed_angle(mi, mj, mk);   // at i, from ->i-1 to ->i-2
            const int dt1 = md.t[i] - md.t[i - 1], dt2 = md.t[i - 1] - md.t[i - 2];
            const float *Ui = sc.U + (int64_t)(md.urow + i) * sc.upitch;
            uint16_t *bt = beta + un.beta + (int64_t)(i - 2) * C;
            const bool last = i == M - 1;
            for (int64_t cell = threadIdx.x; cell < C; cell += blockDim.x) {
                const int b = g.cellb[cell];
                const int c = g.lo[b] + (int)(cell - g.cs[b]);
                float best = inf;
                int arg = 0xffff;
                if (c != b) {
                    const int tb = sc.t[b], tc = sc.t[c];
                    const int a0 = sc.frame_start[tb];
                    const int a1 = p.T > 0 ? sc.frame_start[min(tc + p.T, sc.n_frames)] : sc.S;
                    const float q1 = g.dirf[cell];                      // theta(b->c)
                    for (int a = a0; a < a1; ++a) {
                        if (a == b || a == c) continue;
                        const int64_t ca = g.cs[a] - g.lo[a];
                        const int64_t cab = ca + b, cac = ca + c;
                        const float alpha = last ? 0.0f : an[cab];
                        const float base = base_cost(__ldg(Ui + a), lam2, dt1, sc.t[a], tb, alpha);
                        const float p1 = __fadd_rn(A1, g.dirb[cab]);     // A1 + theta(b->a)
                        const float p2 = __fadd_rn(A2, g.dirf[cab]);     // A2 + theta(a->b)
                        const float v = triple_cost(base, p1, p2, q1, g.dirf[cac], lam23);
                        if (v < best) {
                            best = v;
                            arg = a - a0;
                        }
                    }
                    if (best < inf) best = cell_alpha(best, lam2, dt2, tb, tc);
                }
                ac[cell] = best;
                bt[cell] = (uint16_t)arg;
            }
            __syncthreads();
            float *tmp = an;
            an = ac;
            ac = tmp;
        }
        // Eq. 13: (z_1, z_2) = argmin U_1(z_1) + U_2(z_2) + alpha_3(z_2, z_1) over the cells (b = z_2, c = z_1)
        const float *U0 = sc.U + (int64_t)md.urow * sc.upitch;
        const float *U1 = U0 + sc.upitch;
        InitBest mine{inf, 0x7fffffff, 0x7fffffff};
        for (int64_t cell = threadIdx.x; cell < C; cell += blockDim.x) {
            const float al = an[cell];
            if (!(al < inf)) continue;
            const int b = g.cellb[cell];
            const int c = g.lo[b] + (int)(cell - g.cs[b]);
            const float v = __fadd_rn(__fadd_rn(__ldg(U0 + c), __ldg(U1 + b)), al);
            if (init_better(v, c, b, mine)) mine = InitBest{v, c, b};
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            InitBest o{__shfl_xor_sync(0xffffffffu, mine.v, off), __shfl_xor_sync(0xffffffffu, mine.c, off),
                       __shfl_xor_sync(0xffffffffu, mine.b, off)};
            if (init_better(o.v, o.c, o.b, mine)) mine = o;
        }
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mine;
        __syncthreads();
        if (threadIdx.x == 0) {
            InitBest best = red[0];
            for (int w = 1; w < NT / 32; ++w)
                if (init_better(red[w].v, red[w].c, red[w].b, best)) best = red[w];
            int32_t *row = assign + un.out_a;
            if (best.v < inf) {
                // Eq. 12: z_i = beta_i(z_{i-1}, z_{i-2})
                int z2 = best.c, z1 = best.b;   // z_{i-2}, z_{i-1}
                row[md.perm[0]] = sc.perm[z2];
                row[md.perm[1]] = sc.perm[z1];
                for (int i = 2; i < M; ++i) {
                    const int64_t cell = g.cs[z1] + (z2 - g.lo[z1]);
                    const int za = sc.frame_start[sc.t[z1]] + beta[un.beta + (int64_t)(i - 2) * C + cell];
                    row[md.perm[i]] = sc.perm[za];
                    z2 = z1;
                    z1 = za;
                }
                energy[un.out_e] = best.v;
            } else {
                for (int i = 0; i < M; ++i) row[i] = -1;
                energy[un.out_e] = inf;
            }
        }
        __syncthreads();   // the reduction slots and the alpha tables are reused by the next unit
    }
}

// ---- the shared-memory form ------------------------------------------------------------------------------------
//
// Rows run forward in time: row b holds the a that may follow b, a in [flo(b), fhi(b)) = [minnode(t'(b)),
// minnode(t'(b) + T)), so that everything the minimum over a of a cell (b, c) reads is contiguous in a:
//   base(a, b) = U(a) + lambda2 Delta(a, b) + alpha_{i+1}(a, b), theta(b->a), theta(a->b) in row b, theta(a->c) in
//   row c, for a in [flo(b), fhi(c)).
// A diagonal entry (a = b) holds +inf in all three tables, which excludes a = b and a = c without a branch, and so
// does a row's padding (one or two entries, to an even length), so that a is taken two at a time. What a
// cell (b, c) produces, alpha_i(b, c), is the next step's entry a = b of row c, so it is turned into that step's
// base at once and stored there; the two base tables alternate. A cell's constants (where its rows start, how many
// a it has, theta(b->c), the time difference, where its result goes) are 16 bytes computed once per pair, in
// decreasing order of the a count: in the cells' own order a warp's lanes differ by up to 10 frames of a, and half
// of them wait. The argmin of a cell is stored at that place, so a warp's stores stay one line.
//
// A cluster's CTAs own consecutive runs of frames with about the same number of cells each. A CTA reads only its
// own rows (and copies of the theta rows of the points up to T frames before its first); a result whose row
// belongs to an earlier CTA is stored there through distributed shared memory, and a cluster barrier ends a step.
//
// Bound by shared memory: per two a of 32 cells three 8-byte and two 4-byte loads of rows that lie apart (about 15
// wavefronts for 43 instructions; two thirds of the cycles on Table 2's scene). Measured with the earlier kernel
// (tables in global memory, five dependent gathers per a, one CTA per pair) and with this one, by CUDA events: 50
// pairs of 10,000 cells (788 points over 723 frames) 1,653 -> 258 us (two CTAs per pair; 46 clusters of three fit the
// chip, not 50), 50 pairs of 1,270 cells (86 points over 60 frames) 282 -> 100 us. Ordering the cells took 31% of the
// instructions and 2% of the time.
struct BlockPt {
    float2 xy;
    int t, flo, fhi, fr, lo, cs;   // fr: first entry of the point's row, cs: its first cell (whole scene)
};

struct BlockShape {                // largest share of a CTA over the call's scenes, and the argmin placement
    int rows, trows, cells, pts;   // entries of its own rows, with the rows before them, cells, points
    int beta;                      // argmin entries kept in shared memory (0: global)
};

__host__ __device__ inline size_t block_smem_bytes(const BlockShape &s)
{
    return (size_t)s.cells * 12 + (size_t)s.pts * sizeof(BlockPt) + ((size_t)s.rows * 3 + s.trows) * 4 +
           ((size_t)s.cells + s.beta) * 2;
}

// Stores v at this CTA's shared address `at`, in the CTA `rank` of the cluster.
__device__ __forceinline__ void store_in_cta(uint32_t at, uint32_t rank, float v)
{
    uint32_t there;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(at), "r"(rank));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(there), "f"(v) : "memory");
}

template <int NT, bool kCluster, bool kSmemBeta>
__global__ void __launch_bounds__(NT, 1024 / NT) block_cluster_kernel(
    const BlockUnit *__restrict__ units, int n_units, const ModelRec *__restrict__ models,
    const SceneRec *__restrict__ scenes, const BlockGeo *__restrict__ geos, Params p, BlockShape shape,
    uint16_t *__restrict__ beta, float *__restrict__ energy, int32_t *__restrict__ assign)
{
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BlockPt *pts = reinterpret_cast<BlockPt *>(smem_raw);
    uint2 *meta = reinterpret_cast<uint2 *>(pts + shape.pts);
    float *base0 = reinterpret_cast<float *>(meta + shape.cells);
    float *thba = base0 + 2 * shape.rows, *thab = thba + shape.rows;
    uint32_t *meta2 = reinterpret_cast<uint32_t *>(thab + shape.trows);
    uint16_t *order = reinterpret_cast<uint16_t *>(meta2 + shape.cells);   // a cell's place in meta
    uint16_t *sbeta = order + shape.cells;
    __shared__ InitBest red[NT / 32 + 8];   // per warp, then (in the first CTA) per CTA of the cluster
    __shared__ float4 consts[2];            // A1, A2 and the frame differences of step i at consts[i & 1]
    __shared__ int path[32];
    __shared__ int bucket[kBuckets];
    // per CTA of the cluster: its first point, the first one it reads, its first cell, its rows' place in thab
    __shared__ int csplit[kMaxCluster + 1], ch0[kMaxCluster], ccs0[kMaxCluster], crow[kMaxCluster];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int rank = 0, csize = 1;
    if constexpr (kCluster) {
        rank = (int)cg::this_cluster().block_rank();
        csize = (int)cg::this_cluster().num_blocks();
    }
    auto sync_all = [&] {
        if constexpr (kCluster) cg::this_cluster().sync();
        else __syncthreads();
    };
    const float lam2 = p.lambda2, lam23 = __fmul_rn(p.lambda2, p.lambda3);
    const float inf = __int_as_float(0x7f800000);
    for (int u = blockIdx.x / csize; u < n_units; u += gridDim.x / csize) {
        const BlockUnit un = units[u];
        const ModelRec md = models[un.model];
        const SceneRec sc = scenes[un.scene];
        const BlockGeo &g = geos[un.scene];
        const int M = md.M;
        // own points [b0, b1); points [h0, e1) are read: the c before them and the a after
        const int b0 = g.split[rank], b1 = g.split[rank + 1];
        const bool some = b1 > b0;
        const int h0 = some ? g.lo[b0] : b0;
        auto row_end = [&](int t) { return p.T > 0 ? sc.frame_start[min(t + p.T, sc.n_frames)] : sc.S; };
        const int e1 = some ? row_end(sc.t[b1 - 1]) : b0;
        const int cs0 = some ? (int)g.cs[b0] : 0, cells = some ? (int)g.cs[b1] - cs0 : 0;
        auto step_consts = [&](int i) {
            const float2 mi = md.xy[i], mj = md.xy[i - 1], mk = md.xy[i - 2];
            // the model angles at i-1 (from ->i to ->i-2) and at i (from ->i-1 to ->i-2)
            return make_float4(signed_angle(mj, mi, mk), signed_angle(mi, mj, mk),
                               __int_as_float(md.t[i] - md.t[i - 1]), __int_as_float(md.t[i - 1] - md.t[i - 2]));
        };
        for (int q = tid; q < e1 - h0; q += NT) {
            const int b = h0 + q, t = sc.t[b];
            pts[q] = BlockPt{sc.xy[b], t, sc.frame_start[t], row_end(t), g.fr[b], g.lo[b], (int)g.cs[b]};
        }
        if (tid == 0) consts[(M - 1) & 1] = step_consts(M - 1);
        if (tid <= csize) csplit[tid] = g.split[tid];
        if (tid < csize) {
            const int b = g.split[tid];
            ch0[tid] = b < sc.S ? g.lo[b] : b;
            ccs0[tid] = (int)g.cs[b];
            crow[tid] = g.split_fr[tid] - (some ? g.fr[h0] : 0);
        }
        __syncthreads();
        // directions of every row read, and the first step's base (alpha_{M+1} = 0, Eq. 11) of the own rows
        const int fr0 = some ? pts[b0 - h0].fr : 0, frh = some ? pts[0].fr : 0;
        {
            const float *Ui = sc.U + (int64_t)(md.urow + M - 1) * sc.upitch;
            const int dt1 = __float_as_int(consts[(M - 1) & 1].z);
            float *bs = base0 + ((M - 1) & 1) * shape.rows;
            for (int q = warp; q < b1 - h0; q += NT / 32) {
                const BlockPt pb = pts[q];
                const int b = h0 + q;
                for (int a = pb.flo + lane; a < pb.flo + block_row(pb.fhi - pb.flo); a += 32) {
                    const bool real = a < pb.fhi && a != b;
                    const BlockPt pa = pts[real ? a - h0 : q];
                    const int e = pb.fr + a - pb.flo;
                    thab[e - frh] = real ? direction(pa.xy, pb.xy) : inf;
                    if (b >= b0) {
                        thba[e - fr0] = real ? direction(pb.xy, pa.xy) : inf;
                        bs[e - fr0] = real ? base_cost(__ldg(Ui + a), lam2, dt1, pa.t, pb.t, 0.0f) : inf;
                        if (a >= pb.fhi) base0[(M & 1) * shape.rows + e - fr0] = inf;   // the other table's padding
                    }
                }
            }
        }
        __syncthreads();
        // the cells' constants: x = row b | a count << 16, y = row c (at a = flo(b)) | b - flo(b) << 16 (the sum
        // is the entry a = b of row c), meta2 = t'(b) - t'(c) | owner of row c << 12 | b << 16. Cells go in decreasing order of
        // their a count (a counting sort, any order within a class), so that a warp's lanes loop alike.
        for (int k = tid; k < kBuckets; k += NT) bucket[k] = 0;
        __syncthreads();
        for (int pass = 0; pass < 2; ++pass) {
            for (int q = b0 - h0 + warp; q < b1 - h0; q += NT / 32) {
                const BlockPt pb = pts[q];
                const int b = h0 + q, nc = (q + 1 < e1 - h0 ? pts[q + 1].cs : cs0 + cells) - pb.cs;
                for (int k = lane; k < nc; k += 32) {
                    const int c = pb.lo + k;
                    const BlockPt pc = pts[c - h0];
                    const int n = c == b ? 0 : max(0, pc.fhi - pb.flo);
                    const int at = atomicAdd(&bucket[max(0, kBuckets - 1 - (n + 1) / 2)], 1);
                    if (pass == 0) continue;
                    int own = rank;
                    if constexpr (kCluster)
                        while (csplit[own] > c) --own;
                    order[pb.cs - cs0 + k] = (uint16_t)at;
                    meta[at] = make_uint2((uint32_t)(pb.fr - fr0) | (uint32_t)n << 16,
                                          (uint32_t)(pc.fr - frh + pb.flo - pc.flo) | (uint32_t)(b - pb.flo) << 16);
                    meta2[at] = (uint32_t)(pb.t - pc.t) | (uint32_t)own << 12 | (uint32_t)q << 16;
                }
            }
            __syncthreads();
            if (pass == 0) {   // first places of the classes
                if (warp == 0) {
                    const int x = bucket[2 * lane], y = bucket[2 * lane + 1];
                    int sum = x + y;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const int o = __shfl_up_sync(0xffffffffu, sum, off);
                        if (lane >= off) sum += o;
                    }
                    bucket[2 * lane] = sum - x - y;
                    bucket[2 * lane + 1] = sum - y;
                }
                __syncthreads();
            }
        }
        sync_all();   // every CTA of the cluster is ready to receive results
        const int64_t scells = g.cells;
        uint16_t *gbeta = beta + un.beta + (int64_t)(M - 3) * scells + cs0;   // the step's argmin row
        uint16_t *lbeta = sbeta + (M - 3) * cells;
        InitBest mine{inf, 0x7fffffff, 0x7fffffff};
        const float *U0 = sc.U + (int64_t)md.urow * sc.upitch;
        const float *Un = U0 + (int64_t)(M - 2) * sc.upitch + h0;               // U(z_{i-1})
        const float *vr0 = thab + (fr0 - frh);
        const unsigned long long lamp = pk2(lam23, lam23);
        for (int i = M - 1; i >= 2; --i, gbeta -= scells, lbeta -= cells, Un -= sc.upitch) {
            const float4 k4 = consts[i & 1];
            const unsigned long long A1p = pk2(k4.x, k4.x), A2p = pk2(k4.y, k4.y);
            const int dt2 = __float_as_int(k4.w);
            const float *bs = base0 + (i & 1) * shape.rows;
            float *next = base0 + ((i - 1) & 1) * shape.rows;
            // dealt back and forth, so that no warp takes the longest of every round
            for (int r0 = 0; r0 < cells; r0 += NT) {
                const int e = r0 + ((r0 / NT) & 1 ? NT - 1 - tid : tid);
                if (e >= cells) continue;
                // the last step needs the cell itself
                const int at = i > 2 ? e : order[e];
                const uint2 m = meta[at];
                const uint32_t mw = meta2[at];
                const int rb = m.x & 0xffff, n = m.x >> 16, td = mw & 0xfff, q = mw >> 16;
                const int row = m.y & 0xffff, entry = row + (int)(m.y >> 16);
                const float ub = __ldg(Un + q);     // U(z_{i-1} = b): the next step's a, or Eq. 13's z_2
                const float *vb = bs + rb, *va = thba + rb, *vr = vr0 + rb, *vc = thab + row;
                const unsigned long long q1p = pk2(thab[entry], thab[entry]);   // theta(b->c)
                float best = inf;
                int arg = 0xffff;
                // two a at a time, packed FP32x2; past an odd count comes row c's padding, +inf
#pragma unroll 2
                for (int k = 0; k < n; k += 2) {
                    const unsigned long long b2 = *reinterpret_cast<const unsigned long long *>(vb + k),
                                             a2 = *reinterpret_cast<const unsigned long long *>(va + k),
                                             r2 = *reinterpret_cast<const unsigned long long *>(vr + k);
                    float v0, v1;
                    triple_cost2(b2, add2(A1p, a2), add2(A2p, r2), q1p, pk2(vc[k], vc[k + 1]), lamp, v0, v1);
                    if (v0 < best) {
                        best = v0;
                        arg = k;
                    }
                    if (v1 < best) {
                        best = v1;
                        arg = k + 1;
                    }
                }
                // alpha_i, +inf where no a is feasible (best is), then the next step's base: the same |Delta| twice
                const float dl = fabsf((float)(dt2 - td));
                const float al = __fmaf_rn(lam2, dl, best);
                (kSmemBeta ? lbeta : gbeta)[at] = (uint16_t)arg;
                if (i > 2) {
                    const float nb = __fadd_rn(__fmaf_rn(lam2, dl, ub), al);
                    if constexpr (kCluster) {
                        const int own = (mw >> 12) & 15;
                        store_in_cta((uint32_t)__cvta_generic_to_shared(next + (entry - crow[own])), own, nb);
                    } else {
                        next[entry] = nb;
                    }
                } else if (al < inf) {
                    const BlockPt pb = pts[q];
                    const int b = h0 + q, c = pb.lo + e - (pb.cs - cs0);
                    const float v = __fadd_rn(__fadd_rn(__ldg(U0 + c), ub), al);
                    if (init_better(v, c, b, mine)) mine = InitBest{v, c, b};
                }
            }
            if (i > 2 && tid == NT - 1) consts[(i - 1) & 1] = step_consts(i - 1);
            sync_all();
        }
        // Eq. 13: (z_1, z_2) = argmin U_1(z_1) + U_2(z_2) + alpha_3(z_2, z_1) over the cells (b = z_2, c = z_1)
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            InitBest o{__shfl_xor_sync(0xffffffffu, mine.v, off), __shfl_xor_sync(0xffffffffu, mine.c, off),
                       __shfl_xor_sync(0xffffffffu, mine.b, off)};
            if (init_better(o.v, o.c, o.b, mine)) mine = o;
        }
        if (lane == 0) red[warp] = mine;
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < NT / 32; ++w)
                if (init_better(red[w].v, red[w].c, red[w].b, mine)) mine = red[w];
            if constexpr (kCluster) *cg::this_cluster().map_shared_rank(&red[NT / 32 + rank], 0) = mine;
        }
        if constexpr (kCluster) sync_all();
        if (rank == 0 && warp == 0) {
            if constexpr (kCluster) {
                mine = red[NT / 32];
                for (int r = 1; r < csize; ++r)
                    if (init_better(red[NT / 32 + r].v, red[NT / 32 + r].c, red[NT / 32 + r].b, mine))
                        mine = red[NT / 32 + r];
            }
            const bool ok = __shfl_sync(0xffffffffu, mine.v, 0) < inf;
            int z2 = mine.c, z1 = mine.b;   // lane 0: z_{i-2}, z_{i-1}
            int32_t *row = assign + un.out_a;
            // Eq. 12: z_i = beta_i(z_{i-1}, z_{i-2}); lane 0 walks, the warp writes 32 points at a time
            for (int i0 = 0; i0 < M; i0 += 32) {
                if (lane == 0 && ok) {
                    for (int i = i0; i < min(M, i0 + 32); ++i) {
                        if (i >= 2) {
                            int za;
                            if (kSmemBeta) {   // the whole scene's points are here (one CTA)
                                const BlockPt pb = pts[z1];
                                za = pb.flo + sbeta[(i - 2) * cells + order[pb.cs + z2 - pb.lo]];
                            } else {
                                // the cell's place and its point are in its owner's tables
                                int own = 0;
                                const uint16_t *po = order;
                                const BlockPt *pp = pts;
                                if constexpr (kCluster) {
                                    while (csplit[own + 1] <= z1) ++own;
                                    po = cg::this_cluster().map_shared_rank(order, own);
                                    pp = cg::this_cluster().map_shared_rank(pts, own);
                                }
                                const BlockPt pb = pp[z1 - ch0[own]];
                                za = pb.flo + __ldcg(beta + un.beta + (int64_t)(i - 2) * g.cells + ccs0[own] +
                                                     po[pb.cs - ccs0[own] + z2 - pb.lo]);
                            }
                            z2 = z1;
                            z1 = za;
                        }
                        path[i - i0] = i == 0 ? z2 : z1;
                    }
                }
                __syncwarp();
                if (i0 + lane < M) row[md.perm[i0 + lane]] = ok ? sc.perm[path[lane]] : -1;
                __syncwarp();
            }
            if (lane == 0) energy[un.out_e] = mine.v;
        }
        sync_all();   // the tables and the reduction slots are reused by the next unit
    }
}

// Clusters of csize CTAs that can run at once (0: none); a property of the device, kept per shape of the launch.
// The callers hold the library's lock.
template <int NT>
int max_clusters(int csize, size_t smem)
{
    struct Known { int dev, csize, n; size_t smem; };
    static Known known[16];
    static int used = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    for (int k = 0; k < std::min(used, 16); ++k)
        if (known[k].dev == dev && known[k].csize == csize && known[k].smem == smem) return known[k].n;
    auto kern = block_cluster_kernel<NT, true, false>;
    int n = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)csize);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)csize;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    known[used % 16] = Known{dev, csize, n, smem};
    ++used;
    return n;
}

}  // namespace

void block_split(const BlockBand &bd, int csize, int32_t *split)
{
    const int64_t cells = bd.cs[bd.S];
    split[0] = 0;
    for (int r = 1; r < csize; ++r) {   // at a frame's first point: a cell's c may share b's frame and follow b
        const int64_t b = std::lower_bound(bd.cs, bd.cs + bd.S, cells * r / csize) - bd.cs;
        split[r] = b < bd.S ? bd.flo[b] : bd.S;
    }
    split[csize] = bd.S;
}

cudaError_t launch_block_geo(const float2 *xy, int S, const int32_t *lo, const int64_t *cs, int64_t cells,
                             int32_t *cellb, float *dirf, float *dirb, cudaStream_t st)
{
    if (S <= 0 || cells <= 0) return cudaSuccess;
    block_cells_kernel<<<(S + 255) / 256, 256, 0, st>>>(cs, S, cellb);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    block_dirs_kernel<<<(unsigned)std::min<int64_t>((cells + 255) / 256, 8192), 256, 0, st>>>(xy, lo, cs, cellb,
                                                                                           cells, dirf, dirb);
    return cudaGetLastError();
}

BlockPlan block_plan(const BlockBand *bands, int n_scenes, int n_units, int max_M, int T)
{
    BlockPlan pl;
    int dev = 0, sms = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return pl;
    const size_t room = (size_t)std::max(optin - 2048, 0);   // less the static arrays
    int64_t max_cells = 0;
    for (int s = 0; s < n_scenes; ++s) {
        max_cells = std::max(max_cells, bands[s].cs[bands[s].S]);
        const int last = bands[s].n_frames - 1, td = T > 0 ? std::min(T - 1, last) : last;
        if (td >= 1 << 12) return pl;   // a cell's time difference has 12 bits
    }
    if (max_cells > (int64_t)kMaxCluster * (int64_t)(room / 16)) return pl;
    auto shape_of = [&](int cl) {
        BlockShape sh{2, 2, 1, 1, 0};
        for (int s = 0; s < n_scenes; ++s) {
            const BlockBand &bd = bands[s];
            int32_t split[kMaxCluster + 1];
            block_split(bd, cl, split);
            for (int r = 0; r < cl; ++r) {
                const int b0 = split[r], b1 = split[r + 1];
                if (b1 <= b0) continue;
                const int h0 = bd.lo[b0], e1 = bd.fhi[b1 - 1];
                sh.rows = std::max(sh.rows, (int)(bd.fr[b1] - bd.fr[b0]));
                sh.trows = std::max(sh.trows, (int)(bd.fr[b1] - bd.fr[h0]));
                sh.cells = std::max(sh.cells, (int)(bd.cs[b1] - bd.cs[b0]));
                sh.pts = std::max(sh.pts, e1 - h0);
            }
        }
        return sh;
    };
    auto threads_of = [](const BlockShape &s) { return s.cells <= 256 ? 256 : s.cells <= 512 ? 512 : 1024; };
    auto at_once = [&](const BlockShape &s, int cl) {
        const size_t b = block_smem_bytes(s);
        const int nt = threads_of(s);
        return nt == 256 ? max_clusters<256>(cl, b) : nt == 512 ? max_clusters<512>(cl, b) : max_clusters<1024>(cl, b);
    };
    // the fewest CTAs whose shared memory holds a pair
    int least = 0;
    BlockShape sh{};
    for (int cl = 1; cl <= kMaxCluster && !least; ++cl) {
        sh = shape_of(cl);
        if (sh.trows < 65536 && sh.cells < 65536 && block_smem_bytes(sh) <= room) least = cl;
    }
    if (!least) return pl;
    // more where SMs would idle, as long as a CTA keeps kMinShare cells and all pairs run at once
    pl.csize = least;
    const int want = (int)std::min<int64_t>(std::min<int64_t>(kMaxCluster, sms / std::max(n_units, 1)), max_cells / kMinShare);
    for (int cl = want; cl > least; --cl) {
        const BlockShape s2 = shape_of(cl);
        if (block_smem_bytes(s2) <= room && at_once(s2, cl) >= n_units) {
            pl.csize = cl;
            sh = s2;
            break;
        }
    }
    if (pl.csize == 1) {
        // the argmin tables of one CTA's pair stay in shared memory where they leave the SM to it or are small
        const int64_t entries = max_cells * std::max(max_M - 2, 1);
        const size_t with = block_smem_bytes(sh) + (size_t)entries * 2;
        if (with <= (n_units <= sms ? room : room / 4)) sh.beta = (int)std::max<int64_t>(entries, 1);
        pl.threads = threads_of(sh);
    } else {
        pl.threads = threads_of(sh);
        const int n = at_once(sh, pl.csize);
        if (n < 1) return BlockPlan{};
        pl.clusters = std::min(n_units, n);
    }
    pl.rows = sh.rows;
    pl.trows = sh.trows;
    pl.cells = sh.cells;
    pl.pts = sh.pts;
    pl.beta = sh.beta;
    pl.shared = true;
    return pl;
}

cudaError_t preload_block()
{
    cudaFuncAttributes a;
    const void *kerns[] = {(const void *)block_cluster_kernel<256, false, false>,
                           (const void *)block_cluster_kernel<256, false, true>,
                           (const void *)block_cluster_kernel<256, true, false>,
                           (const void *)block_cluster_kernel<512, false, false>,
                           (const void *)block_cluster_kernel<512, false, true>,
                           (const void *)block_cluster_kernel<512, true, false>,
                           (const void *)block_cluster_kernel<1024, false, false>,
                           (const void *)block_cluster_kernel<1024, false, true>,
                           (const void *)block_cluster_kernel<1024, true, false>,
                           (const void *)block_recurse_kernel<kBlockThreads>,
                           (const void *)block_recurse_kernel<kBlockThreadsWide>,
                           (const void *)block_cells_kernel,
                           (const void *)block_dirs_kernel};
    for (const void *k : kerns) {
        cudaError_t e = cudaFuncGetAttributes(&a, k);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

bool block_always_shared(int64_t points, int n_frames, int T)
{
    if ((T > 0 ? std::min(T, n_frames) : n_frames) > 1 << 12) return false;
    // a band holds at most points^2 cells, the rows as many entries and their padding
    const int cells = (int)std::min<int64_t>(points * points, 1 << 20), pts = (int)std::min<int64_t>(points, 1 << 20);
    const BlockShape sh{cells + 2 * pts, cells + 2 * pts, cells, pts, 0};
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return false;
    return block_smem_bytes(sh) + 2048 <= (size_t)optin;
}

namespace {
template <int NT>
cudaError_t launch_single(const BlockUnit *units, int n_units, const ModelRec *models, const SceneRec *scenes,
                          const BlockGeo *geos, Params p, const BlockShape &sh, int sms, uint16_t *beta, float *energy,
                          int32_t *assign, cudaStream_t st)
{
    auto kern = sh.beta ? block_cluster_kernel<NT, false, true> : block_cluster_kernel<NT, false, false>;
    const size_t smem = block_smem_bytes(sh);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<std::min(n_units, sms * 8), NT, smem, st>>>(units, n_units, models, scenes, geos, p, sh, beta, energy, assign);
    return cudaGetLastError();
}

template <int NT>
cudaError_t launch_cluster(const BlockUnit *units, int n_units, const ModelRec *models, const SceneRec *scenes,
                           const BlockGeo *geos, Params p, const BlockShape &sh, const BlockPlan &pl, uint16_t *beta,
                           float *energy, int32_t *assign, cudaStream_t st)
{
    auto kern = block_cluster_kernel<NT, true, false>;
    const size_t smem = block_smem_bytes(sh);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(pl.csize * pl.clusters));
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)pl.csize;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, units, n_units, models, scenes, geos, p, sh, beta, energy, assign);
}
}  // namespace

cudaError_t launch_block_recurse(const BlockUnit *units, int n_units, const ModelRec *models, const SceneRec *scenes,
                                 const BlockGeo *geos, Params p, const BlockPlan &pl, int64_t max_cells, uint16_t *beta,
                                 float *scratch, int grid_global, float *energy, int32_t *assign, cudaStream_t st)
{
    if (n_units <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    prof_begin(kProfRecurse, st);
    const BlockShape sh{pl.rows, pl.trows, pl.cells, pl.pts, pl.beta};
    if (pl.shared && pl.csize == 1) {
        e = pl.threads == 256   ? launch_single<256>(units, n_units, models, scenes, geos, p, sh, sms, beta, energy, assign, st)
            : pl.threads == 512 ? launch_single<512>(units, n_units, models, scenes, geos, p, sh, sms, beta, energy, assign, st)
                                : launch_single<1024>(units, n_units, models, scenes, geos, p, sh, sms, beta, energy, assign, st);
    } else if (pl.shared) {
        e = pl.threads == 256   ? launch_cluster<256>(units, n_units, models, scenes, geos, p, sh, pl, beta, energy, assign, st)
            : pl.threads == 512 ? launch_cluster<512>(units, n_units, models, scenes, geos, p, sh, pl, beta, energy, assign, st)
                                : launch_cluster<1024>(units, n_units, models, scenes, geos, p, sh, pl, beta, energy, assign, st);
    } else {
        const bool wide = n_units < sms;
        auto kern = wide ? block_recurse_kernel<kBlockThreadsWide> : block_recurse_kernel<kBlockThreads>;
        kern<<<grid_global, wide ? kBlockThreadsWide : kBlockThreads, 0, st>>>(units, n_units, models, scenes, geos, p,
                                                                                beta, scratch, max_cells, energy,
                                                                                assign);
        e = cudaGetLastError();
    }
    prof_end(kProfRecurse, st);
    return e;
}

}  // namespace hgm
