// k_prop.cu -- the candidate-proposal network: training (forward, backward, Adam) and weights.
//
// Not part of the paper: a small MLP layered on the exact method that scores each
// window candidate so that only the best `keep` enter the recursion (the pruned
// form; the exact recursion stays its fallback and the yardstick of its recall and energy gap). Architecture:
//   x = [f_i, f'_j, dx/100, dy/100, dt/w]  (d_in = 2F + 3)
//   h1 = relu(W1 x + b1), h2 = relu(W2 h1 + b2)  (128 each),  z3 = w3.h2 + b3,  score = sigmoid(z3)
// trained with binary cross-entropy on labels produced by the exact recursion.
//
// A training step is two launches: one pass kernel that takes 128 rows of the batch through the forward and the
// backward pass in one CTA (every contraction on the tensor cores, BF16 operands, FP32 accumulation), and one
// kernel that sums the CTAs' gradient shares and applies Adam. Weights, gradients and moments are FP32.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <vector>

#include "hgm_internal.cuh"
#include "prop.cuh"
#include "tc05.cuh"

namespace hgm {
namespace {

constexpr int H = kPropHidden;

constexpr int TB = 128;                    // batch rows of a tile (MMA M)
constexpr int NT = 512;                    // threads: four warps per 32 rows, each owning 32 of the 128 columns
constexpr int XSLOTS = 3;                  // X chunks of 128 components held at once (F <= 190 stays resident)
constexpr uint32_t kCore = 128;            // bytes of a core matrix (8 x 16 bytes)
constexpr uint32_t kRow = 16 * kCore;      // byte stride of 8 rows of a 128 x 128 BF16 tile
constexpr uint32_t kTile = 16 * kRow;      // 32 KB
constexpr uint32_t kPolls = 1u << 26;      // bounded wait for the tensor core

struct TrainSmem {
    unsigned char x[XSLOTS][kTile];   // X chunks, transposed: row = component j, column = batch row r
    unsigned char w2[kTile];          // W2 [n][k]
    unsigned char p0[kTile];          // W1 chunks (even), then H1 [r][k], then dZ1 [r][n]
    unsigned char p1[kTile];          // W1 chunks (odd), then dZ2 [r][n]
    float b1[H], b2[H], w3[H];
    float zpart[4][TB];               // last layer: sums over 32 columns each
    float csum[3][4][H];              // column sums over 32 rows each: db2, dw3, db1
    float red[2][NT / 32];            // loss and db3 per warp
    uint64_t mbar[3];
    uint32_t tslot;
};

// element (row, col) of a 128 x 128 BF16 tile: core matrices of 8 rows x 8 columns
__device__ __forceinline__ uint32_t tile_at(int row, int col8) { return (uint32_t)(row >> 3) * kRow + (uint32_t)col8 * kCore + (uint32_t)(row & 7) * 16u; }

__device__ __forceinline__ uint4 pack8(const float *v)
{
    __align__(16) __nv_bfloat162 h[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) h[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
    return *reinterpret_cast<uint4 *>(h);
}

// Components [k0, k0 + 128) of W's 128 rows (ld floats, a multiple of 4; C valid) as a [n][j] tile: eight rows on
// consecutive lanes, so a quarter warp stores one whole core matrix.
__device__ __forceinline__ void stage_w(unsigned char *dst, const float *__restrict__ W, int ld, int C, int k0, int tid)
{
#pragma unroll
    for (int e = tid; e < H * 16; e += NT) {
        const int r = (e & 7) | ((e >> 7) << 3), c8 = (e >> 3) & 15, k = k0 + 8 * c8;
        float v[8];
        if (k + 8 <= ld) {   // ld >= C: the padding after C holds zeros
            const float4 *p = reinterpret_cast<const float4 *>(W + (int64_t)r * ld + k);
            const float4 a = p[0], b = p[1];
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = k + q < C ? W[(int64_t)r * ld + k + q] : 0.0f;
        }
        *reinterpret_cast<uint4 *>(dst + tile_at(r, c8)) = pack8(v);
    }
}

// Components [k0, k0 + 128) of batch rows [r0, r0 + 128) as a transposed [j][r] tile: a warp reads 32 consecutive
// components of eight rows (whole lines whatever the row stride) and each lane stores its component's eight rows.
__device__ __forceinline__ void stage_x(unsigned char *dst, const float *__restrict__ X, int64_t ldx, int B, int C, int r0,
                                        int k0, int tid)
{
    const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
    for (int e = warp; e < 64; e += NT / 32) {
        const int j = (e & 3) * 32 + lane, r8 = e >> 2, k = k0 + j;
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int r = r0 + 8 * r8 + q;
            v[q] = (k < C && r < B) ? __ldg(X + (int64_t)r * ldx + k) : 0.0f;
        }
        *reinterpret_cast<uint4 *>(dst + tile_at(j, r8)) = pack8(v);
    }
}

// Sums of v[0..31] over the warp's lanes: lane l receives the sum of v[l] (31 exchanges, fixed order).
__device__ __forceinline__ float column_sum(float (&v)[32], int lane)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int q = 0; q < off; ++q) {
            const float send = up ? v[q] : v[q + off], keep = up ? v[q + off] : v[q];
            v[q] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    return v[0];
}

// One pass over a batch: forward, and with kTrain also the backward pass, of 128 rows at a time in one CTA. Every
// contraction is a tcgen05 product of BF16 operands in shared memory with the FP32 accumulator in tensor memory
// (columns 0: Z1, 128: Z2, 256: dH1, 384: dW2; dW1 later takes 0..383); nothing but the gradients leaves the SM:
//   Z1 = X W1^T + b1, H1 = relu(Z1), Z2 = H1 W2^T + b2, z3 = relu(Z2) . w3 + b3, dz3 = (sigmoid(z3) - y) / B,
//   dZ2 = dz3 w3 [Z2 > 0], dH1 = dZ2 W2, dW2 = dZ2^T H1, dZ1 = dH1 [Z1 > 0], dW1 = dZ1^T X.
// Each operand is stored once: the products that need it transposed read it MN-major. The CTA's share of the
// gradient goes to its own row of `part` (W1 as [j][n], W2 as [k][n], so that a warp's 32 rows are one line),
// summed over CTAs by prop_update_kernel.
//
// Bound by latency (a chain of staging, five products and four epilogues per tile). Measured on 4,096 rows at
// F = 162: 2.28 ms per step with one kernel per operation (the weight gradients were one-CTA products over the
// whole batch, 1.1 ms each, the column sums one-CTA loops, 0.4 ms each), 0.06 ms with this pass, weight transfer
// included. 128 rows per tile because that is the product's M; four warps per 32 rows because a warp reads only
// its quarter of tensor memory and 32 columns leave the epilogue in registers (all but 13 words of the 128 registers
// that 512 threads have).
template <bool kTrain>
__global__ void __launch_bounds__(NT, 1) prop_pass_kernel(PropLayout L, const float *__restrict__ theta,
                                                          const float *__restrict__ X, int64_t ldx,
                                                          const float *__restrict__ y, int B, float *__restrict__ z3out,
                                                          float *__restrict__ part, int *__restrict__ status)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    TrainSmem &sm = *reinterpret_cast<TrainSmem *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int quad = warp & 3, cq = warp >> 2, row = 32 * quad + lane, col0 = 32 * cq;
    if (warp == 0) tc05::tmem_alloc<512>(&sm.tslot);
    if (tid == 0)
        for (int k = 0; k < 3; ++k) tc05::mbar_init(&sm.mbar[k], 1);
    stage_w(sm.w2, theta + L.o_W2, H, H, 0, tid);
    if (tid < H) {
        sm.b1[tid] = theta[L.o_b1 + tid];
        sm.b2[tid] = theta[L.o_b2 + tid];
        sm.w3[tid] = theta[L.o_w3 + tid];
    }
    const float b3 = theta[L.o_b3];
    tc05::fence_proxy_async_smem();
    tc05::fence_before_sync();
    __syncthreads();
    tc05::fence_after_sync();
    const uint32_t tmem = sm.tslot;
    const uint32_t tlane = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)col0;
    constexpr uint32_t kk = tc05::idesc_bf16_f32(TB, H), mk = tc05::idesc_bf16_f32(TB, H, true, false),
                       km = tc05::idesc_bf16_f32(TB, H, false, true), mm = tc05::idesc_bf16_f32(TB, H, true, true);
    // D += A B over 128 K components; K-major tiles advance 16 components by two core matrices, MN-major ones by
    // two groups of eight rows
    auto product = [&](uint32_t d, const unsigned char *a, bool a_mn, const unsigned char *b, bool b_mn, uint32_t idesc,
                       bool acc) {
        const uint32_t a0 = tc05::smem_u32(a), b0 = tc05::smem_u32(b);
        const uint32_t as = a_mn ? 2 * kRow : 2 * kCore, bs = b_mn ? 2 * kRow : 2 * kCore;
        for (int ks = 0; ks < 8; ++ks)
            tc05::mma_bf16(tmem + d,
                           a_mn ? tc05::smem_desc(a0 + ks * as, kRow, kCore) : tc05::smem_desc(a0 + ks * as, kCore, kRow),
                           b_mn ? tc05::smem_desc(b0 + ks * bs, kRow, kCore) : tc05::smem_desc(b0 + ks * bs, kCore, kRow),
                           idesc, acc || ks > 0);
    };
    uint32_t phase = 0;        // bit k: parity of mbar[k]'s next completion
    uint32_t pending = 0;      // bit k: a commit on mbar[k] whose completion was not yet observed
    bool bad = false;
    auto wait = [&](int k) {   // true if the products committed to mbar[k] are done (every thread agrees)
        bool ok = tc05::mbar_wait(&sm.mbar[k], (phase >> k) & 1u, kPolls);
        tc05::fence_before_sync();
        bad = __syncthreads_or(!ok) != 0;
        tc05::fence_after_sync();
        if (!bad) {
            phase ^= 1u << k;
            pending &= ~(1u << k);
        }
        return !bad;
    };
    auto ready = [&] {         // shared-memory operands written by every thread become visible to the products
        tc05::fence_proxy_async_smem();
        tc05::fence_before_sync();
        __syncthreads();
        tc05::fence_after_sync();
    };
    const int nch = (L.d_in + 127) / 128, ntiles = (B + TB - 1) / TB;
    float *mine = part + (int64_t)blockIdx.x * L.n;
    const float rows = (float)B;
    bool first = true;
    for (int tile = blockIdx.x; tile < ntiles && !bad; tile += gridDim.x, first = false) {
        const int r0 = tile * TB;
        // ---- Z1: chunks of 128 components; W1's alternate between p0 and p1, X's take the slots in turn
        for (int ch = 0; ch < nch && !bad; ++ch) {
            if (ch >= 2 && !wait(ch & 1)) break;   // the products that read this W1 buffer (and X slot) are done
            stage_x(sm.x[ch % XSLOTS], X, ldx, B, L.d_in, r0, 128 * ch, tid);
            stage_w(ch & 1 ? sm.p1 : sm.p0, theta + L.o_W1, L.dp, L.d_in, 128 * ch, tid);
            ready();
            if (tid == 0) {
                product(0, sm.x[ch % XSLOTS], true, ch & 1 ? sm.p1 : sm.p0, false, mk, ch > 0);
                tc05::mma_commit(&sm.mbar[ch & 1]);
            }
            pending |= 1u << (ch & 1);
        }
        if (bad || (nch >= 2 && !wait(nch & 1)) || !wait((nch - 1) & 1)) break;
        // ---- H1 (bits of Z1 > 0 kept for the backward mask)
        uint32_t on1 = 0;
        {
            float v[32];
            tc05::tmem_ld32(tlane, v);
#pragma unroll
            for (int q = 0; q < 32; ++q) {
                v[q] += sm.b1[col0 + q];
                on1 |= v[q] > 0.0f ? 1u << q : 0u;
                v[q] = fmaxf(v[q], 0.0f);
            }
#pragma unroll
            for (int g = 0; g < 4; ++g)
                *reinterpret_cast<uint4 *>(sm.p0 + tile_at(row, 4 * cq + g)) = pack8(v + 8 * g);
        }
        ready();
        if (tid == 0) {
            product(128, sm.p0, false, sm.w2, false, kk, false);
            tc05::mma_commit(&sm.mbar[2]);
        }
        pending |= 4u;
        if (!wait(2)) break;
        // ---- Z2, z3, loss, dZ2
        {
            float v[32];
            tc05::tmem_ld32(tlane + 128, v);
            float s = 0.0f;
#pragma unroll
            for (int q = 0; q < 32; ++q) {
                v[q] += sm.b2[col0 + q];
                s = fmaf(fmaxf(v[q], 0.0f), sm.w3[col0 + q], s);
            }
            sm.zpart[cq][row] = s;
            tc05::fence_before_sync();
            __syncthreads();
            tc05::fence_after_sync();
            const float z = ((sm.zpart[0][row] + sm.zpart[1][row]) + (sm.zpart[2][row] + sm.zpart[3][row])) + b3;
            const bool in = r0 + row < B;
            if (!kTrain) {
                if (in && cq == 0) z3out[r0 + row] = z;
                __syncthreads();   // zpart is rewritten by the next tile
                continue;
            }
            const float yy = in ? y[r0 + row] : 0.0f;
            const float sg = 1.0f / (1.0f + expf(-z));
            const float dz = in ? (sg - yy) / rows : 0.0f;
            const float sp = z > 0.0f ? z + log1pf(expf(-z)) : log1pf(expf(z));
            float ls = in && cq == 0 ? sp - yy * z : 0.0f, ds = cq == 0 ? dz : 0.0f;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                ls += __shfl_xor_sync(0xffffffffu, ls, off);
                ds += __shfl_xor_sync(0xffffffffu, ds, off);
            }
            if (lane == 0) {
                sm.red[0][warp] = ls;
                sm.red[1][warp] = ds;
            }
            float g2[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) g2[q] = v[q] > 0.0f ? dz * sm.w3[col0 + q] : 0.0f;
#pragma unroll
            for (int g = 0; g < 4; ++g)
                *reinterpret_cast<uint4 *>(sm.p1 + tile_at(row, 4 * cq + g)) = pack8(g2 + 8 * g);
            sm.csum[0][quad][col0 + lane] = column_sum(g2, lane);
#pragma unroll
            for (int q = 0; q < 32; ++q) v[q] = dz * fmaxf(v[q], 0.0f);
            sm.csum[1][quad][col0 + lane] = column_sum(v, lane);
        }
        ready();
        if (tid == 0) {
            product(256, sm.p1, false, sm.w2, true, km, false);    // dH1 = dZ2 W2
            product(384, sm.p1, true, sm.p0, true, mm, false);     // dW2 = dZ2^T H1
            tc05::mma_commit(&sm.mbar[2]);
        }
        pending |= 4u;
        if (!wait(2)) break;
        // ---- dZ1 (into H1's tile, which the products no longer read)
        {
            float v[32];
            tc05::tmem_ld32(tlane + 256, v);
#pragma unroll
            for (int q = 0; q < 32; ++q) v[q] = (on1 >> q) & 1u ? v[q] : 0.0f;
#pragma unroll
            for (int g = 0; g < 4; ++g)
                *reinterpret_cast<uint4 *>(sm.p0 + tile_at(row, 4 * cq + g)) = pack8(v + 8 * g);
            sm.csum[2][quad][col0 + lane] = column_sum(v, lane);
        }
        // ---- dW1, three chunks at a time; while they run, dW2 and the column sums go out
        for (int g0 = 0; g0 < nch && !bad; g0 += XSLOTS) {
            const int ng = min(XSLOTS, nch - g0);
            if (nch > XSLOTS)
                for (int c = 0; c < ng; ++c) stage_x(sm.x[c], X, ldx, B, L.d_in, r0, 128 * (g0 + c), tid);
            ready();
            if (tid == 0) {
                for (int c = 0; c < ng; ++c) product(128 * c, sm.p0, true, sm.x[c], false, mk, false);
                tc05::mma_commit(&sm.mbar[2]);
            }
            pending |= 4u;
            if (g0 == 0) {
                float v[32];
                tc05::tmem_ld32(tlane + 384, v);   // row = n of dW2, columns k
                float *o = mine + L.o_W2;
#pragma unroll
                for (int q = 0; q < 32; ++q) {
                    float *at = o + (col0 + q) * H + row;
                    *at = first ? v[q] : *at + v[q];
                }
                if (tid < 3 * H) {
                    const int k = tid / H, c = tid - k * H;
                    const float t = (sm.csum[k][0][c] + sm.csum[k][1][c]) + (sm.csum[k][2][c] + sm.csum[k][3][c]);
                    float *at = mine + (k == 0 ? L.o_b2 : k == 1 ? L.o_w3 : L.o_b1) + c;
                    *at = first ? t : *at + t;
                } else if (tid < 3 * H + 2) {      // db3, and beside it the loss
                    const int k = tid - 3 * H;
                    float t = 0.0f;
                    for (int w = 0; w < 4; ++w) t += sm.red[1 - k][w];   // the warps of the first 32 columns
                    float *at = mine + L.o_b3 + k;
                    *at = first ? t : *at + t;
                }
            }
            if (!wait(2)) break;
            for (int c = 0; c < ng; ++c) {
                float v[32];
                tc05::tmem_ld32(tlane + 128 * c, v);
                const int j0 = 128 * (g0 + c) + col0;
#pragma unroll
                for (int q = 0; q < 32; ++q) {
                    if (j0 + q >= L.dp) break;
                    float *at = mine + (int64_t)(j0 + q) * H + row;
                    *at = first ? v[q] : *at + v[q];
                }
            }
            tc05::fence_before_sync();
            __syncthreads();   // accumulators, operand tiles and sums are free for the next group or tile
            tc05::fence_after_sync();
        }
    }
    if (bad) {
        if (tid == 0) atomicExch(status, 1);
        // a wait gave up: the products still in flight get a bounded time before the accumulators are freed
        for (int k = 0; k < 3; ++k)
            if ((pending >> k) & 1u) tc05::mbar_wait(&sm.mbar[k], (phase >> k) & 1u, kPolls);
    }
    tc05::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc05::tmem_dealloc<512>(tmem);
}

struct AdamArgs {
    float *theta, *m, *v;
    float lr, b1, b2, eps, c1, c2;
};

// The gradient from the CTAs' shares (summed in CTA order) into grad, and with kAdam one bias-corrected Adam step.
// A block takes 32 rows n x 8 columns of W1 or W2: the shares are read along n (their layout), the parameters
// written along the columns (theirs). The last block takes the vectors; the loss stands in the padding after b3
// and is scaled to the mean.
template <bool kAdam>
__global__ void __launch_bounds__(256) prop_update_kernel(PropLayout L, const float *__restrict__ part, int nparts,
                                                          float inv_b, float *__restrict__ grad, float *__restrict__ loss,
                                                          AdamArgs ad)
{
    __shared__ float tile[8][33];
    const int tid = threadIdx.x;
    auto sum = [&](int64_t at) {
        float s = 0.0f;
        const float *q = part + at;
#pragma unroll 8
        for (int k = 0; k < nparts; ++k) s += q[(int64_t)k * L.n];
        return s;
    };
    auto apply = [&](int64_t k, float g) {
        grad[k] = g;
        if (kAdam) {
            const float mk = ad.b1 * ad.m[k] + (1.0f - ad.b1) * g;
            const float vk = ad.b2 * ad.v[k] + (1.0f - ad.b2) * g * g;
            ad.m[k] = mk;
            ad.v[k] = vk;
            ad.theta[k] -= ad.lr * (mk / ad.c1) / (sqrtf(vk / ad.c2) + ad.eps);
        }
    };
    const int c1 = (L.dp + 7) / 8, nb1 = 4 * c1, nb2 = 4 * (H / 8);
    const int bk = blockIdx.x;
    if (bk < nb1 + nb2) {
        const bool w1 = bk < nb1;
        const int e = w1 ? bk : bk - nb1, n0 = 32 * (e & 3), j0 = 8 * (e >> 2), cols = w1 ? L.dp : H;
        const int64_t base = w1 ? L.o_W1 : L.o_W2;
        const int jr = tid >> 5, nr = tid & 31;
        if (j0 + jr < cols) tile[jr][nr] = sum(base + (int64_t)(j0 + jr) * H + n0 + nr);
        __syncthreads();
        const int j = tid & 7, n = tid >> 3;
        if (j0 + j < cols) apply(base + (int64_t)(n0 + n) * cols + j0 + j, tile[j][n]);
        return;
    }
    for (int k = tid; k < 3 * H + 2; k += 256) {
        const int64_t at = k < H ? L.o_b1 + k : k < 2 * H ? L.o_b2 + (k - H) : k < 3 * H ? L.o_w3 + (k - 2 * H)
                                                                                        : L.o_b3 + (k - 3 * H);
        const float s = sum(at);
        if (k == 3 * H + 1) *loss = s * inv_b;
        else apply(at, s);
    }
}

// CTAs of a pass over B rows: a tile of 128 rows each, at most one per SM, and at most 256 MB of shares.
int pass_ctas(const PropLayout &L, int B)
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess)
        sms = 1;
    const int64_t cap = std::max<int64_t>(1, ((int64_t)64 << 20) / L.n);
    return (int)std::min<int64_t>(std::min<int64_t>((B + TB - 1) / TB, sms), cap);
}

}  // namespace

// ---- parameter layout ------------------------------------------------------------------------
PropLayout prop_layout(int F)
{
    PropLayout L;
    L.F = F;
    L.d_in = 2 * F + 3;
    L.dp = (L.d_in + 3) & ~3;
    L.o_W1 = 0;
    L.o_b1 = L.o_W1 + (int64_t)H * L.dp;
    L.o_W2 = L.o_b1 + H;
    L.o_b2 = L.o_W2 + (int64_t)H * H;
    L.o_w3 = L.o_b2 + H;
    L.o_b3 = L.o_w3 + H;
    L.n = L.o_b3 + 4;
    L.n_logical = (int64_t)H * L.d_in + H + (int64_t)H * H + H + H + 1;
    return L;
}

// logical (W1 [H x d_in], b1, W2, b2, w3, b3) <-> padded device layout
void prop_pack(const PropLayout &L, const float *logical, std::vector<float> &flat)
{
    flat.assign((size_t)L.n, 0.0f);
    const float *p = logical;
    for (int h = 0; h < H; ++h) std::memcpy(&flat[(size_t)(L.o_W1 + (int64_t)h * L.dp)], p + (int64_t)h * L.d_in,
                                            sizeof(float) * (size_t)L.d_in);
    p += (int64_t)H * L.d_in;
    std::memcpy(&flat[(size_t)L.o_b1], p, sizeof(float) * H);
    p += H;
    std::memcpy(&flat[(size_t)L.o_W2], p, sizeof(float) * H * H);
    p += (int64_t)H * H;
    std::memcpy(&flat[(size_t)L.o_b2], p, sizeof(float) * H);
    p += H;
    std::memcpy(&flat[(size_t)L.o_w3], p, sizeof(float) * H);
    p += H;
    flat[(size_t)L.o_b3] = p[0];
}

void prop_unpack(const PropLayout &L, const float *flat, float *logical)
{
    float *p = logical;
    for (int h = 0; h < H; ++h)
        std::memcpy(p + (int64_t)h * L.d_in, flat + L.o_W1 + (int64_t)h * L.dp, sizeof(float) * (size_t)L.d_in);
    p += (int64_t)H * L.d_in;
    std::memcpy(p, flat + L.o_b1, sizeof(float) * H);
    p += H;
    std::memcpy(p, flat + L.o_W2, sizeof(float) * H * H);
    p += (int64_t)H * H;
    std::memcpy(p, flat + L.o_b2, sizeof(float) * H);
    p += H;
    std::memcpy(p, flat + L.o_w3, sizeof(float) * H);
    p += H;
    p[0] = flat[L.o_b3];
}

void prop_init(const PropLayout &L, uint64_t seed, std::vector<float> &logical)
{
    std::mt19937_64 gen(seed);
    std::normal_distribution<double> nd(0.0, 1.0);
    logical.assign((size_t)L.n_logical, 0.0f);
    float *p = logical.data();
    const double s1 = std::sqrt(2.0 / L.d_in), s2 = std::sqrt(2.0 / H), s3 = std::sqrt(1.0 / H);
    for (int64_t k = 0; k < (int64_t)H * L.d_in; ++k) p[k] = (float)(nd(gen) * s1);
    p += (int64_t)H * L.d_in + H;
    for (int64_t k = 0; k < (int64_t)H * H; ++k) p[k] = (float)(nd(gen) * s2);
    p += (int64_t)H * H + H;
    for (int k = 0; k < H; ++k) p[k] = (float)(nd(gen) * s3);
}

// ---- workspace and launches --------------------------------------------------------------------
cudaError_t PropTrain::ensure(const PropLayout &L, int B)
{
    if (B <= cap && buf) return cudaSuccess;
    if (buf) cudaFree(buf);
    buf = nullptr;
    cap = 0;
    const size_t shares = (size_t)pass_ctas(L, B) * (size_t)L.n;
    const size_t logits = ((size_t)B + 3) & ~(size_t)3;
    cudaError_t e = cudaMalloc(&buf, (shares + logits + 8) * sizeof(float));
    if (e != cudaSuccess) return e;
    float *q = static_cast<float *>(buf);
    part = q;                  // L.n is a multiple of 4: the words after stay aligned
    z3 = q + shares;
    loss = z3 + logits;
    status = reinterpret_cast<int *>(loss + 4);
    cap = B;
    return cudaMemset(status, 0, sizeof(int));
}

cudaError_t prop_forward(const PropLayout &L, const float *theta, PropTrain &w, const float *X, int ldx, int B,
                         float *logits, cudaStream_t st)
{
    const size_t smem = sizeof(TrainSmem);
    cudaError_t e = cudaFuncSetAttribute(prop_pass_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    prop_pass_kernel<false><<<pass_ctas(L, B), NT, smem, st>>>(L, theta, X, ldx, nullptr, B, logits, w.part, w.status);
    return cudaGetLastError();
}

cudaError_t prop_step(const PropLayout &L, float *theta, PropTrain &w, const float *X, int ldx, const float *y, int B,
                      float *grad, float *m, float *v, int64_t t, float lr, cudaStream_t st)
{
    const size_t smem = sizeof(TrainSmem);
    cudaError_t e = cudaFuncSetAttribute(prop_pass_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int ctas = pass_ctas(L, B);
    prop_pass_kernel<true><<<ctas, NT, smem, st>>>(L, theta, X, ldx, y, B, nullptr, w.part, w.status);
    if ((e = cudaGetLastError())) return e;
    const unsigned blocks = (unsigned)(4 * ((L.dp + 7) / 8) + 4 * (H / 8) + 1);
    AdamArgs ad{theta, m, v, lr, 0.9f, 0.999f, 1e-8f, 0.0f, 0.0f};
    if (t > 0) {
        ad.c1 = 1.0f - (float)std::pow(0.9, (double)t);
        ad.c2 = 1.0f - (float)std::pow(0.999, (double)t);
        prop_update_kernel<true><<<blocks, 256, 0, st>>>(L, w.part, ctas, 1.0f / (float)B, grad, w.loss, ad);
    } else {
        prop_update_kernel<false><<<blocks, 256, 0, st>>>(L, w.part, ctas, 1.0f / (float)B, grad, w.loss, ad);
    }
    return cudaGetLastError();
}

}  // namespace hgm
