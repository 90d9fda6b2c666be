// k_unary.cu -- kernel (a): the unary look-up table of Sec. 3.3.
//
// U[r][j] = lambda1 * ||A_r - B_j||_2 for every model row r and scene row j
// (Eq. 2, non-dummy branch, with lambda1 of Eq. 1 absorbed). The paper
// pre-computes this S x M table once instead of re-evaluating the distance
// inside every cell of the trellis; here it is one launch per (model set,
// scene), stored row-major with the scene index contiguous so that a model
// point's window [minnode(f0), minnode(f1+1)) is one coalesced segment.
//
// Every output is accumulated in a fixed order: d_k = A_rk - B_jk (FP32),
// s = fma(d_k, d_k, s) for k = 0, 1, ..., then an IEEE square root and an
// FP32 multiply. The value is therefore reproducible bit for bit by any
// IEEE-754 implementation, which makes it usable as the ranking key of the
// top-K candidate cap. Rows are padded with zeros to a multiple of 4
// components; fma(0, 0, s) == s, so padding changes no bit.
//
// Operands go to shared memory as they are, 32 components of every row per stage, by 16-byte asynchronous copies
// several stages ahead of the arithmetic (rows are 16-byte aligned: their width is a multiple of 4). A lane owns
// JT columns (lane + 32 q) and RT rows: per four components RT broadcast and JT conflict-free 16-byte loads for
// 8 RT JT operations. Two tile shapes: 32 x 128 per CTA where the table fills the chip twice, bound by the FP32
// lanes; 16 x 32 with the whole row in flight where it does not, bound by the latency of one round of loads.
// Measured with 32 x 128 tiles staged through registers and two barriers per 16 components before: 16 model x 600
// scene points (F = 162) 21.9 -> 6.5 us, 30 x 9,100 22.8 -> 11.3 us, 1,500 x 870 32.7 -> 29.0 us, 3,264 x 6,000
// 293 -> 273 us (23.5 T lane operations/s, 0.58 of the peak).
#include <algorithm>

#include "hgm_internal.cuh"

namespace hgm {
namespace {

constexpr int KC = 32;        // components per stage
constexpr int LD = KC + 4;    // row stride in shared memory: eight rows' 16-byte reads cover all banks
constexpr int NW = 8;         // warps, each RT rows of the tile

__device__ __forceinline__ void copy16(float *dst, const float *src, bool real)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(real ? 16 : 0) : "memory");
}

template <int RT, int JT, int NS>
__global__ void __launch_bounds__(32 * NW) unary_kernel(const float *__restrict__ A, int R, const float *__restrict__ B,
                                                       int S, int F, float lambda1, float *__restrict__ U, int64_t ldu)
{
    constexpr int BR = NW * RT, BJ = 32 * JT, ROWS = BR + BJ;
    extern __shared__ __align__(16) float sm[];   // NS stages of [BR rows of A | BJ rows of B] x LD
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int r0 = blockIdx.y * BR;
    const int64_t j0 = (int64_t)blockIdx.x * BJ;
    const int nk = (F + KC - 1) / KC;
    auto load = [&](int kc) {   // rows past the end and components past F arrive as zeros: fma(0, 0, s) = s
        if (kc < nk) {
            float *st = sm + (kc % NS) * (ROWS * LD);
#pragma unroll
            for (int e = tid; e < ROWS * (KC / 4); e += 32 * NW) {
                const int row = e / (KC / 4), k = (e % (KC / 4)) * 4, kg = kc * KC + k;
                const bool isa = row < BR;
                const int64_t gr = isa ? r0 + row : j0 + (row - BR);
                const bool real = gr < (isa ? R : S) && kg < F;
                copy16(st + row * LD + k, real ? (isa ? A : B) + gr * F + kg : A, real);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[RT][JT];
#pragma unroll
    for (int a = 0; a < RT; ++a)
#pragma unroll
        for (int b = 0; b < JT; ++b) acc[a][b] = 0.0f;
    for (int kc = 0; kc < NS - 1; ++kc) load(kc);
    for (int kc = 0; kc < nk; ++kc) {
        asm volatile("cp.async.wait_group %0;" ::"n"(NS - 2) : "memory");
        __syncthreads();           // stage kc is here for everyone, and stage kc - 1 is no longer read
        load(kc + NS - 1);
        const float *sa = sm + (kc % NS) * (ROWS * LD) + warp * RT * LD;
        const float *sb = sm + (kc % NS) * (ROWS * LD) + (BR + lane) * LD;
        const int kn = min(KC, F - kc * KC);
#pragma unroll 2
        for (int k = 0; k < kn; k += 4) {
            float4 av[RT], bv[JT];
#pragma unroll
            for (int a = 0; a < RT; ++a) av[a] = *reinterpret_cast<const float4 *>(sa + a * LD + k);
#pragma unroll
            for (int b = 0; b < JT; ++b) bv[b] = *reinterpret_cast<const float4 *>(sb + b * 32 * LD + k);
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int a = 0; a < RT; ++a)
#pragma unroll
                    for (int b = 0; b < JT; ++b) {
                        const float d = __fsub_rn(reinterpret_cast<const float *>(&av[a])[c],
                                                  reinterpret_cast<const float *>(&bv[b])[c]);
                        acc[a][b] = __fmaf_rn(d, d, acc[a][b]);
                    }
        }
    }
#pragma unroll
    for (int a = 0; a < RT; ++a) {
        const int r = r0 + warp * RT + a;
        if (r >= R) continue;
#pragma unroll
        for (int b = 0; b < JT; ++b) {
            const int64_t j = j0 + lane + 32 * b;
            if (j < S) U[(int64_t)r * ldu + j] = __fmul_rn(lambda1, __fsqrt_rn(acc[a][b]));
        }
    }
}

template <int RT, int JT, int NS>
cudaError_t launch_tile(const float *A, int R, const float *B, int S, int F, float lambda1, float *U, int ldu,
                        cudaStream_t st)
{
    constexpr int BR = NW * RT, BJ = 32 * JT;
    constexpr size_t smem = (size_t)NS * (BR + BJ) * LD * sizeof(float);
    auto kern = unary_kernel<RT, JT, NS>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // rows on y: at most 65,535 tiles of rows per launch
    for (int r = 0; r < R; r += BR * 65535) {
        const int n = std::min(R - r, BR * 65535);
        kern<<<dim3((unsigned)((S + BJ - 1) / BJ), (unsigned)((n + BR - 1) / BR)), 32 * NW, smem, st>>>(
            A + (int64_t)r * F, n, B, S, F, lambda1, U + (int64_t)r * ldu, ldu);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_unary(const float *A, int R, const float *B, int S, int F, float lambda1, float *U,
                         int ldu, cudaStream_t st)
{
    if (R <= 0 || S <= 0) return cudaSuccess;
    if ((F & 3) || ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15))
        return cudaErrorMisalignedAddress;   // handles pad rows to a multiple of 4 floats
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    prof_begin(kProfUnary, st);
    if ((int64_t)((S + 127) / 128) * ((R + 31) / 32) >= 2 * sms)
        e = launch_tile<4, 4, 3>(A, R, B, S, F, lambda1, U, ldu, st);
    else
        e = launch_tile<2, 1, 6>(A, R, B, S, F, lambda1, U, ldu, st);
    prof_end(kProfUnary, st);
    return e;
}

cudaError_t preload_unary()
{
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, unary_kernel<4, 4, 3>);
    return e == cudaSuccess ? cudaFuncGetAttributes(&a, unary_kernel<2, 1, 6>) : e;
}

}  // namespace hgm
