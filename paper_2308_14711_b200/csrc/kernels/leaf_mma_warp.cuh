// Grouped leaf evaluation for buckets of a few tokens: one warp per tile of up to 16 tokens of one leaf (bf16, mma.sync,
// float32 accumulate), un-permuting write-back.
//
// Algorithm 1, FORWARD_I, leaf branch:  Y = act(X[T_j] W1_j^T + b1_j) W2_j^T + b2_j  for the tokens T_j of a leaf's list.
//
// With a few tokens per leaf the work is a stream of leaf weights, and the time is how many of them are in flight.  A CTA per
// tile (k_leaf_mma) spends 5 to 7 us on a chain of ring stages, partial sums and barriers however little there is to do, and two
// CTAs per SM make seven rounds of 2048 leaves; here every warp goes its own way, 16 tiles per SM at once, without shared
// memory, barriers or waits:
//   * the operands of both GEMMs are loaded from global memory straight into the registers of the MMAs, 16 bytes per lane:
//     the order of the summands is free, so lane c of a quad takes 8 consecutive columns of its row, four for each of two
//     MMAs, of x and of W1 alike (64 contiguous bytes per row and quad);
//   * the hidden units are numbered so that the accumulators of GEMM1, activated and packed, are the A operand of GEMM2 and
//     lane c's units are consecutive in the rows of W2;
//   * the output columns are numbered so that a lane ends with 8 consecutive outputs of its token: one 16-byte store.
// Bound: latency and HBM (weights).  Measured: see warp_tiles in fff_api.cu.
//
// Leaves of at most 16 neurons: with 32 the fragments of fewer loads fit the registers, and it is level with a CTA per tile.
// Images as in leaf_mma.cuh (LP = 16); D % 8 == 0 (columns past D: zero weights, no loads of x), O % 8 == 0.
#pragma once

#include "common.cuh"
#include "leaf_mma.cuh"
#include "ptx.cuh"

namespace fff {

constexpr int kLWRows = 16;                                // tokens per tile: the rows of one MMA
constexpr int kLWWarps = 8;
constexpr int kLWThreads = kLWWarps * 32;

// Hidden unit of column n of the j-th group of 8 accumulator columns.
__device__ __forceinline__ int warp_tile_unit(int j, int n) { return 4 * (n >> 1) + 2 * j + (n & 1); }

// x [B, D], slots [n_bins][cap] token numbers, counts [n_bins] + [1] CTAs that have finished (all zero again at the end).
// kSplit: the hidden values as sums of two bf16 values (see leaf_umma.cuh).
template <bool kSplit>
__global__ void __launch_bounds__(kLWThreads, 2)
k_leaf_mma_warp(const __nv_bfloat16* __restrict__ x, const int32_t* __restrict__ slots, const __nv_bfloat16* __restrict__ w1img,
                const float* __restrict__ b1img, const unsigned char* __restrict__ w2img, __nv_bfloat16* __restrict__ y, int D, int Dp,
                int O, int act, int32_t* __restrict__ counts, int n_bins, int cap)
{
    constexpr int LP = 16, NT = LP / 8;                    // padded hidden units, accumulator tiles of 8 of them
    constexpr int KU = 4;                                  // 32-column blocks of GEMM1 whose loads are issued together (six spill)
    constexpr int OU = 4;                                  // 32-output blocks of GEMM2, likewise
    constexpr int kStage2 = kNC * LP * 2 + kNC * 4;
    extern __shared__ int s_pre[];                         // [n_bins + 1] tiles before each leaf
    __shared__ int s_wsum[kLWWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;

    pdl_trigger();
    pdl_wait();
    tiles_before_bins([&](int b) { return __ldcg(counts + b); }, n_bins, kLWRows, s_pre, s_wsum, kLWThreads);
    const int n_tiles = s_pre[n_bins];
    const int U2 = (O + kNC - 1) / kNC, w2_bytes = (O / kNC) * kStage2 + (O % kNC) * (LP * 2);

    // this lane's rows of W1 in a 64-column block: byte offset of the 16-byte unit c of its row (columns 32.. : 64 bytes on,
    // modulo the swizzle)
    int w1off[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int n = warp_tile_unit(j, g);
        w1off[j] = n * 128 + ((c ^ (n & 7)) << 4);
    }
    for (int tile = warp * gridDim.x + blockIdx.x; tile < n_tiles; tile += kLWWarps * gridDim.x) {
        const int leaf = bin_of_tile(s_pre, n_bins, tile);
        const int first = (tile - s_pre[leaf]) * kLWRows;
        const int rows = min(kLWRows, __ldcg(counts + leaf) - first);
        const int32_t* list = slots + (int64_t)leaf * cap + first;
        const int64_t tok0 = g < rows ? __ldcg(list + g) : -1, tok1 = g + 8 < rows ? __ldcg(list + g + 8) : -1;
        const unsigned char* w2j = w2img + (int64_t)leaf * U2 * kStage2;
        for (int off = lane * 128; off < w2_bytes; off += 32 * 128)                        // needed after the whole of GEMM1
            asm volatile("prefetch.global.L2 [%0];" ::"l"(w2j + off));

        // ---- GEMM1
        const __nv_bfloat16 *x0 = x + max(tok0, (int64_t)0) * D + 8 * c, *x1 = x + max(tok1, (int64_t)0) * D + 8 * c;
        const unsigned char* w1j = reinterpret_cast<const unsigned char*>(w1img + (int64_t)leaf * LP * Dp);
        float acc[NT][4];
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[j][i] = 0.0f;
        const int blocks = (D + 31) / 32;
        for (int k0 = 0; k0 < blocks; k0 += KU) {
            uint4 a[KU][2], b[KU][NT];
#pragma unroll
            for (int i = 0; i < KU; ++i) {
                const int kb = k0 + i;
                const bool in = kb * 32 + 8 * c < D, any = kb < blocks;
                a[i][0] = in && tok0 >= 0 ? __ldg(reinterpret_cast<const uint4*>(x0 + kb * 32)) : make_uint4(0u, 0u, 0u, 0u);
                a[i][1] = in && tok1 >= 0 ? __ldg(reinterpret_cast<const uint4*>(x1 + kb * 32)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int j = 0; j < NT; ++j)
                    b[i][j] = any ? __ldg(reinterpret_cast<const uint4*>(w1j + (kb >> 1) * (LP * 128) + (w1off[j] ^ ((kb & 1) << 6))))
                                  : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int i = 0; i < KU; ++i)
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    ptx::mma_bf16(acc[j], a[i][0].x, a[i][1].x, a[i][0].y, a[i][1].y, b[i][j].x, b[i][j].y);
                    ptx::mma_bf16(acc[j], a[i][0].z, a[i][1].z, a[i][0].w, a[i][1].w, b[i][j].z, b[i][j].w);
                }
        }
        constexpr int kOps = kSplit ? 2 : 1;
        uint32_t h[kOps][NT][2];
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            const float2 b1 = __ldg(reinterpret_cast<const float2*>(b1img + (int64_t)leaf * LP + warp_tile_unit(j, 2 * c)));
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const float h0 = activate(act, acc[j][2 * r] + b1.x), h1 = activate(act, acc[j][2 * r + 1] + b1.y);
                if constexpr (kSplit) ptx::split_bf16(h0, h1, h[0][j][r], h[1][j][r]);
                else h[0][j][r] = ptx::pack_bf16(h0, h1);
            }
        }

        // ---- GEMM2: column n of group t of a block of 32 outputs is output 8 (n / 2) + 2 t + n % 2 of the block
        for (int o0 = 0; o0 < O; o0 += 32 * OU) {
            uint2 wv[OU][4];                               // per group: four consecutive units of its row
            float4 bias[OU][2];
#pragma unroll
            for (int i = 0; i < OU; ++i) {
                const int ob = min(o0 + 32 * i, (O - 1) & ~31);        // (a block past the end is loaded but not stored)
                const unsigned char* st = w2j + (ob / kNC) * kStage2;
                const int r0 = ob % kNC;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int row = r0 + 8 * (g >> 1) + 2 * t + (g & 1);
                    wv[i][t] = __ldg(reinterpret_cast<const uint2*>(st + ptx::swz128((uint32_t)(row * LP * 2 + 8 * c))));
                }
                const float* bs = reinterpret_cast<const float*>(st + kNC * LP * 2) + r0 + 8 * c;
                bias[i][0] = __ldg(reinterpret_cast<const float4*>(bs));
                bias[i][1] = __ldg(reinterpret_cast<const float4*>(bs + 4));
            }
#pragma unroll
            for (int i = 0; i < OU; ++i) {
                const float bv[8] = {bias[i][0].x, bias[i][0].y, bias[i][0].z, bias[i][0].w, bias[i][1].x, bias[i][1].y, bias[i][1].z, bias[i][1].w};
                uint32_t out0[4], out1[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    float d[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                    for (int op = 0; op < kOps; ++op)
                        ptx::mma_bf16(d, h[op][0][0], h[op][0][1], h[op][1][0], h[op][1][1], wv[i][t].x, wv[i][t].y);
                    out0[t] = ptx::pack_bf16(d[0] + bv[2 * t], d[1] + bv[2 * t + 1]);
                    out1[t] = ptx::pack_bf16(d[2] + bv[2 * t], d[3] + bv[2 * t + 1]);
                }
                const int o = o0 + 32 * i + 8 * c;
                if (o < O) {
                    if (tok0 >= 0) __stcs(reinterpret_cast<uint4*>(y + tok0 * O + o), make_uint4(out0[0], out0[1], out0[2], out0[3]));
                    if (tok1 >= 0) __stcs(reinterpret_cast<uint4*>(y + tok1 * O + o), make_uint4(out1[0], out1[1], out1[2], out1[3]));
                }
            }
        }
    }
    // the last CTA to finish clears the counts (and the word behind them that counts the CTAs) for the next call
    __shared__ int s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(counts + n_bins, 1) == (int)gridDim.x - 1 ? 1 : 0;
    }
    __syncthreads();
    if (s_last)
        for (int b = threadIdx.x; b <= n_bins; b += kLWThreads) counts[b] = 0;
}

}  // namespace fff
