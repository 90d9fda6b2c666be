// k_select.cu -- candidate lists C_i(o): window + top-K cap.
//
// For unit (model m, scene s, offset o) and model point i, the window is the
// frame range [t_i+o-w, t_i+o+w] clipped to the scene; through the minnode
// table of Sec. 3.4 it is the contiguous sorted-scene range
// [minnode(f0), minnode(f1+1)). If it holds more than K points, the K with
// the smallest unary cost are kept (ties to the lower scene index), and the
// kept points are listed in ascending scene index (hence ascending frame).
//
// One warp per (unit, i). The K-th smallest key is found exactly on the IEEE bit patterns (unary costs are >= 0, so
// the bit pattern orders like the value): 256 equal bins between the window's smallest and largest key, the bin that
// holds rank K, and so on inside it, until the bin is kept whole, holds one value, or the rank is one of its first
// few values, which a warp-wide minimum finds. Costs of a window fill such bins evenly, so one or two rounds decide
// (digits of the bit pattern took three or four, their first one with most keys in a few bins). A final ballot
// pass keeps every key up to that value; only where some of its equals must go does it rank them in index order.
// Integer decisions therefore depend only on the FP32 keys of kernel (a), bit for bit.
// Measured with the digit passes and with this: windows of 210 keys (204,000 lists) 386 -> 202 us, of 560 keys
// (522,000 lists) 1,602 -> 868 us, of 420 with the re-score (237,000 lists) 1,139 -> 651 us, of which the re-score,
// four lists of eight at a time instead of eight lanes of a warp, about a third.
#include "hgm_internal.cuh"
#include "unary_common.cuh"

namespace hgm {
namespace {

constexpr int kWarps = 8;

__device__ __forceinline__ uint32_t lanemask_lt()
{
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

constexpr unsigned kFull = 0xffffffffu;
constexpr int kRescoreMax = kRescore;   // candidates of a list re-scored in the precision mode
static_assert(32 % kRescoreMax == 0, "whole lists fill a warp");

// kKeyRegs keys per lane are held in registers: windows of up to 32 kKeyRegs keys are selected from them,
// longer ones from memory in every pass. The launch picks 8 (three CTAs per SM) when the call's typical
// window (the scenes' mean density over 2w+1 frames) fits 256 keys, else 20 (two CTAs per SM, the registers
// the larger arrays need). At the 80 registers that three CTAs leave, seven words of the first are spilled.
template <int kKeyRegs, int kMinBlocks>
__global__ void __launch_bounds__(kWarps * 32, kMinBlocks) select_kernel(const Unit *__restrict__ units, int64_t n_units,
                                                             const ModelRec *__restrict__ models,
                                                             const SceneRec *__restrict__ scenes, Params p,
                                                             int32_t *__restrict__ cand_idx,
                                                             float *__restrict__ cand_u,
                                                             int32_t *__restrict__ cand_cnt)
{
    __shared__ __align__(16) uint32_t hist[kWarps][256];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int K = p.K;
    const uint32_t lt_mask = lanemask_lt();
    for (int64_t u = blockIdx.x; u < n_units; u += gridDim.x) {
        const Unit un = units[u];
        const ModelRec md = models[un.model];
        const SceneRec sc = scenes[un.scene];
        // precision mode: the re-scores of up to four lists wait until they fill the warp
        int pend = 0, pend_i = 0, pend_slot = -1;
        auto rescore = [&] {
            if (pend_slot >= 0) {
                const int64_t o = un.cand + (int64_t)pend_i * K + pend_slot;
                cand_u[o] = unary_fp32(md.f + (int64_t)pend_i * p.F, sc.f + (int64_t)cand_idx[o] * p.F, p.F, p.lambda1);
            }
            pend = 0;
            pend_slot = -1;
        };
        for (int i = warp; i < md.M; i += kWarps) {
            int32_t *oidx = cand_idx + un.cand + (int64_t)i * K;
            float *ou = cand_u + un.cand + (int64_t)i * K;
            const int ti = md.t[i];
            int f0 = ti + un.offset - p.window, f1 = ti + un.offset + p.window;
            f0 = max(f0, 0);
            f1 = min(f1, sc.n_frames - 1);
            int j0 = 0, n = 0;
            if (f0 <= f1) {
                j0 = sc.frame_start[f0];
                n = sc.frame_start[f1 + 1] - j0;
            }
            const float *key = sc.U + (int64_t)(md.urow + i) * sc.upitch + (j0 - sc.ucol0);
            int kept = n < K ? n : K;
            if (n <= K) {
                for (int e = lane; e < K; e += 32) {
                    oidx[e] = e < n ? j0 + e : -1;
                    ou[e] = e < n ? key[e] : __int_as_float(0x7f800000);
                }
            } else {
                // windows of up to 32 kKeyRegs keys are read once into registers (lane + 32 q), longer ones from
                // memory in every pass; slots past the window hold 0xffffffff, above every key (costs are >= 0, so
                // bit 31 of a key is clear)
                const bool inreg = n <= 32 * kKeyRegs;
                uint32_t kb[kKeyRegs];
#pragma unroll
                for (int q = 0; q < kKeyRegs; ++q) {
                    const int e = lane + 32 * q;
                    kb[q] = inreg && e < n ? __float_as_uint(key[e]) : 0xffffffffu;
                }
                auto each = [&](auto f) {
                    if (inreg) {
#pragma unroll
                        for (int q = 0; q < kKeyRegs; ++q) {
                            if (q % 4 == 0 && 32 * q >= n) break;   // slots past the window are harmless
                            f(kb[q], lane + 32 * q);
                        }
                    } else {
                        for (int c0 = 0; c0 < n; c0 += 32)
                            f(c0 + lane < n ? __float_as_uint(key[c0 + lane]) : 0xffffffffu, c0 + lane);
                    }
                };
                uint32_t lo = 0xffffffffu, hi = 0;
                each([&](uint32_t b, int e) {
                    lo = min(lo, b);
                    hi = max(hi, e < n ? b : 0u);
                });
                lo = __reduce_min_sync(kFull, lo);
                hi = __reduce_max_sync(kFull, hi);
                // the kk-th smallest of the c keys in [lo, hi]; every key below lo is kept. Ends with tau: keys < tau
                // are kept, and the first kk of the neq keys == tau
                int kk = K, c = n, neq = 0;
                uint32_t tau = 0;
                for (;;) {
                    if (kk == c || lo == hi) {   // the whole range, or a range of equals
                        tau = hi;
                        neq = c;
                        break;
                    }
                    if (kk <= 2) {               // one of the range's two smallest values
                        bool done = false;
                        for (uint32_t from = lo; !done;) {
                            uint32_t t = 0xffffffffu;
                            each([&](uint32_t b, int) { t = min(t, b >= from ? b : 0xffffffffu); });
                            t = __reduce_min_sync(kFull, t);
                            int cnt = 0;
                            each([&](uint32_t b, int) { cnt += b == t; });
                            cnt = (int)__reduce_add_sync(kFull, (unsigned)cnt);
                            if (cnt >= kk) {
                                tau = t;
                                neq = cnt;
                                done = true;
                            } else {
                                kk -= cnt;
                                from = t + 1;
                            }
                        }
                        break;
                    }
                    const int shift = max(0, 24 - __clz((int)(hi - lo)));   // (hi - lo) >> shift < 256
                    uint4 *h4 = reinterpret_cast<uint4 *>(hist[warp]) + 2 * lane;
                    h4[0] = h4[1] = make_uint4(0, 0, 0, 0);
                    __syncwarp();
                    each([&](uint32_t b, int) {
                        if (b >= lo && b <= hi) atomicAdd(&hist[warp][(b - lo) >> shift], 1u);
                    });
                    __syncwarp();
                    const uint4 x = h4[0], y = h4[1];
                    const uint32_t cn[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
                    uint32_t sum = 0;
#pragma unroll
                    for (int q = 0; q < 8; ++q) sum += cn[q];
                    uint32_t incl = sum;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const uint32_t v = __shfl_up_sync(kFull, incl, off);
                        if (lane >= off) incl += v;
                    }
                    const bool mine = incl - sum < (uint32_t)kk && (uint32_t)kk <= incl;
                    uint32_t below = incl - sum, in_bin = 0;
                    int bin = 0;
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const bool here = in_bin == 0 && below + cn[q] >= (uint32_t)kk;
                        if (here) {
                            bin = lane * 8 + q;
                            in_bin = cn[q];
                        } else if (in_bin == 0) {
                            below += cn[q];
                        }
                    }
                    const int src = __ffs((int)__ballot_sync(kFull, mine)) - 1;
                    bin = __shfl_sync(kFull, bin, src);
                    kk -= (int)__shfl_sync(kFull, below, src);
                    c = (int)__shfl_sync(kFull, in_bin, src);
                    lo += (uint32_t)bin << shift;
                    hi = min(hi, lo + ((1u << shift) - 1));
                    __syncwarp();
                }
                // keep keys < tau, plus the first kk keys == tau in index order
                int base = 0;
                auto put = [&](bool keep, uint32_t b, int e) {
                    const uint32_t km = __ballot_sync(kFull, keep);
                    if (keep) {
                        const int pos = base + __popc(km & lt_mask);
                        oidx[pos] = j0 + e;
                        ou[pos] = __uint_as_float(b);
                    }
                    base += __popc(km);
                };
                if (kk == neq) {
                    each([&](uint32_t b, int e) { put(b <= tau, b, e); });
                } else {
                    int eqseen = 0;
                    each([&](uint32_t b, int e) {
                        const uint32_t eqm = __ballot_sync(kFull, b == tau);
                        put(b < tau || (b == tau && eqseen + __popc(eqm & lt_mask) < kk), b, e);
                        eqseen += __popc(eqm);
                    });
                }
            }
            if (lane == 0) cand_cnt[un.cand / K + i] = kept;
            if (p.rescore > 0 && kept > 0) {
                // precision mode: the p.rescore smallest approximate costs (ties: lower slot) are
                // recomputed from the FP32 descriptors in the exact kernel's fixed FMA order
                __syncwarp();
                uint32_t k0 = lane < kept ? __float_as_uint(ou[lane]) : 0xffffffffu;
                uint32_t k1 = lane + 32 < kept ? __float_as_uint(ou[lane + 32]) : 0xffffffffu;
                const int rounds = min(min(p.rescore, kRescoreMax), kept);
                for (int q = 0; q < rounds; ++q) {
                    const uint32_t m = __reduce_min_sync(kFull, min(k0, k1));
                    const uint32_t e0 = __ballot_sync(kFull, k0 == m), e1 = __ballot_sync(kFull, k1 == m);
                    const int slot = e0 ? __ffs((int)e0) - 1 : 31 + __ffs((int)e1);
                    if (lane == kRescoreMax * pend + q) {
                        pend_slot = slot;
                        pend_i = i;
                    }
                    if (slot == lane) k0 = 0xffffffffu;
                    if (slot == lane + 32) k1 = 0xffffffffu;
                }
                if (++pend == 32 / kRescoreMax) rescore();
            }
        }
        if (pend) rescore();
    }
}

}  // namespace

cudaError_t launch_select(const Unit *units, int64_t n_units, const ModelRec *models, const SceneRec *scenes,
                          Params p, int max_M, int32_t *cand_idx, float *cand_u, int32_t *cand_cnt,
                          cudaStream_t st)
{
    (void)max_M;
    if (n_units <= 0) return cudaSuccess;
    int64_t blocks = n_units < (int64_t)1 << 20 ? n_units : (int64_t)1 << 20;
    prof_begin(kProfSelect, st);
    if (p.max_window <= 32 * 8)
        select_kernel<8, 3><<<(unsigned)blocks, kWarps * 32, 0, st>>>(units, n_units, models, scenes, p, cand_idx,
                                                                      cand_u, cand_cnt);
    else
        select_kernel<20, 2><<<(unsigned)blocks, kWarps * 32, 0, st>>>(units, n_units, models, scenes, p, cand_idx,
                                                                       cand_u, cand_cnt);
    prof_end(kProfSelect, st);
    return cudaGetLastError();
}

cudaError_t preload_select()
{
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, select_kernel<8, 3>);
    return e == cudaSuccess ? cudaFuncGetAttributes(&a, select_kernel<20, 2>) : e;
}

}  // namespace hgm
