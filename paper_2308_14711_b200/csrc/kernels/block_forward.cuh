// Whole forward pass on CUDA cores in one cooperative launch, for layers without a tensor-core path (float32, or bf16
// shapes outside it) and any batch that gives the leaves a few tokens each.
//
// Algorithm 1, FORWARD_I, both branches.  Weights are fetched for several tokens at a time, which is what a kernel with
// one warp per token cannot do (it pulls its leaf's whole parameters through L2 once per token):
//   phase A  descent.  A warp takes TPW tokens.  The first three levels are the same seven nodes for all of them: a block of
//            TPW x 8 dot products; below, every token has its own path: with four tokens per warp one level at a time, with
//            one token per warp (batches that could not fill the GPU otherwise) the seven nodes of three levels at a time, so
//            that a round trip to L2 decides three levels.  Each token is then filed under its leaf: one atomic add on the
//            leaf's cursor, one store into the leaf's list;
//   barrier  one grid-wide barrier (bounded, like every wait: a CTA that gives up records kDevTimeout and leaves the leaves out);
//   phase B  leaves.  Tiles of up to tile_rows = 8 or 16 tokens of one leaf, derived by every CTA from the counts.  A warp evaluates blocks of
//            4 tokens x 8 hidden units; the output layer runs with one output neuron per thread against the tile's tokens.
// The dot products of a block keep all lanes along the input dimension, so that rows of x and of the weights are read as
// they lie (512 bytes per load instruction, no transposition, no staging), and 4 x 8 products share 12 row loads: 128
// multiply-adds per 12 16-byte loads.  The 32 sums of a block are then added across the lanes with 31 shuffles
// (lane_totals) instead of 5 each.
// Bound: latency, with 16 warps per SM to hide it (float32, 768 -> 768, 256 leaves of 12, 6304 tokens, by counters: issue slots 32 %
// busy, L1 31 %, L2 9 %); a block needs 48 cycles of L1 per 32 cycles of multiply-adds, which is what would bind next.
// Measured: see use_block_forward in fff_api.cu.
//
// float32 accumulation; a token's result depends neither on its position in a block nor on the tokens beside it (the sums
// are added in the same tree wherever they stand), so outputs are bit-reproducible although the lists' order is not.
#pragma once

#include "common.cuh"

namespace fff {

constexpr int kBFWarps = 8;
constexpr int kBFThreads = kBFWarps * 32;
constexpr int kBFTile = 16;                                // most tokens per tile of phase B
constexpr int kBFMaxLeaves = 4096;                         // counts and tile prefix are kept in shared memory

// Sums over the lanes of N = 8, 16 or 32 values at once: while there are values to give away, every lane hands one half to
// the lane `sft` away and adds what it gets to the half it keeps; the remaining steps are plain butterflies.  The total of
// value e ends in all lanes with lane / (32 / N) == e.  Every total is added in the same tree (lanes 16 apart, then 8, ...).
template <int N>
__device__ __forceinline__ float lane_totals(float (&v)[N], int lane) {
    int n = N;
#pragma unroll
    for (int sft = 16; sft >= 1; sft >>= 1) {
        if (n > 1) {
            const bool upper = (lane & sft) != 0;
#pragma unroll
            for (int i = 0; i < N / 2; ++i) {
                if (i < n / 2) {
                    const float send = upper ? v[i] : v[i + n / 2];
                    const float keep = upper ? v[i + n / 2] : v[i];
                    v[i] = keep + __shfl_xor_sync(kFullMask, send, sft);
                }
            }
            n >>= 1;
        } else {
            v[0] += __shfl_xor_sync(kFullMask, v[0], sft);
        }
    }
    return v[0];
}

// acc[t * NW + w] += partial dot products of the rows xr[t] and wr[w] (this lane's share of the columns).
// vec: rows start on 16-byte boundaries and D % kVec == 0.
template <typename T, int NX, int NW>
__device__ __forceinline__ void block_dots(const T* const (&xr)[NX], const T* const (&wr)[NW], int D, bool vec, int lane, float (&acc)[NX * NW])
{
#pragma unroll
    for (int i = 0; i < NX * NW; ++i) acc[i] = 0.0f;
    if (vec) {
        constexpr int V = Elem<T>::kVec;
        auto get = [&](const T* row, int k) { return k < D ? __ldg(reinterpret_cast<const uint4*>(row + k)) : make_uint4(0u, 0u, 0u, 0u); };
        auto multiply = [&](const uint4 (&xq)[NX], uint4 wraw, int w) {
            float wv[V];
            Elem<T>::unpack(wraw, wv);
#pragma unroll
            for (int t = 0; t < NX; ++t) {
                float xv[V];
                Elem<T>::unpack(xq[t], xv);
#pragma unroll
                for (int e = 0; e < V; ++e) acc[t * NW + w] = fmaf(wv[e], xv[e], acc[t * NW + w]);
            }
        };
        if constexpr (NX == 1) {
            // little arithmetic per load: the loads of two steps are issued together
            for (int k = lane * V; k - lane * V < D; k += 64 * V) {
                uint4 xq[2][1], wq[2][NW];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    xq[i][0] = get(xr[0], k + i * 32 * V);
#pragma unroll
                    for (int w = 0; w < NW; ++w) wq[i][w] = get(wr[w], k + i * 32 * V);
                }
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int w = 0; w < NW; ++w) multiply(xq[i], wq[i][w], w);
            }
        } else {
            for (int k = lane * V; k < D; k += 32 * V) {
                uint4 xq[NX], wq[NW];
#pragma unroll
                for (int t = 0; t < NX; ++t) xq[t] = __ldg(reinterpret_cast<const uint4*>(xr[t] + k));
#pragma unroll
                for (int w = 0; w < NW; ++w) wq[w] = __ldg(reinterpret_cast<const uint4*>(wr[w] + k));
#pragma unroll
                for (int w = 0; w < NW; ++w) multiply(xq, wq[w], w);
            }
        }
    } else {
        // (requesting the elements of three steps together costs more registers than it hides: 29 -> 36 us at 990 columns)
#pragma unroll 2
        for (int k = lane; k < D; k += 32) {
            float xv[NX];
#pragma unroll
            for (int t = 0; t < NX; ++t) xv[t] = Elem<T>::to_float(xr[t][k]);
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const float wv = Elem<T>::to_float(wr[w][k]);
#pragma unroll
                for (int t = 0; t < NX; ++t) acc[t * NW + w] = fmaf(wv, xv[t], acc[t * NW + w]);
            }
        }
    }
}

// Node q (breadth-first, q < 7) of the subtree below node n of level m, as a row of the node arrays; rows past the subtree's
// `levels` levels are clamped into it (their results are not used).
__device__ __forceinline__ int64_t subtree_row(int m, int64_t n, int q, int levels) {
    const int lev = q >= 3 ? 2 : q >= 1 ? 1 : 0;
    if (lev >= levels) return (((int64_t)1 << m) - 1) + n;
    return (((int64_t)1 << (m + lev)) - 1) + (n << lev) + (q - ((1 << lev) - 1));
}

// Waits until all CTAs of the (cooperative) launch have arrived; `count` is zero before the launch.  What a CTA wrote before it
// arrived is visible to all after it.  False after kGridWaitCycles: long enough for CTAs that another stream's kernel holds up.
constexpr long long kGridWaitCycles = 1ll << 34;           // about 9 s at 1.9 GHz
__device__ __forceinline__ bool grid_barrier(int* count) {
    __shared__ int s_all;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(count, 1);
        const long long t0 = clock64();
        int seen;
        do {
            asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
        } while (seen < (int)gridDim.x && clock64() - t0 < kGridWaitCycles);
        s_all = seen >= (int)gridDim.x ? 1 : 0;
        __threadfence();
    }
    __syncthreads();
    return s_all != 0;
}

// slots: [n_leaves][cap] token numbers, cursor: [n_leaves] counts + [1] CTAs that have finished + [1] CTAs at the barrier; cursor is
// zero on entry and again when the launch has ended (the last CTA clears it).  leaf_out, leaf_out2 (optional): leaf of every token.
template <typename T, int TPW>
__global__ void __launch_bounds__(kBFThreads, 2)
k_block_forward(const T* __restrict__ x, const T* __restrict__ node_w, const T* __restrict__ node_b, const T* __restrict__ w1,
                const T* __restrict__ b1, const T* __restrict__ w2, const T* __restrict__ b2, T* __restrict__ y, int32_t* __restrict__ leaf_out,
                int32_t* __restrict__ leaf_out2, int32_t* slots, int32_t* cursor, int cap, int D, int O, int depth, int l, int act, int B,
                bool vec, int n_leaves, int tile_rows, int* __restrict__ status)
{
    static_assert(TPW == 1 || TPW == 4, "tokens per warp in the descent");
    extern __shared__ __align__(16) int smem_bf[];
    int* s_pre = smem_bf;                                   // [n_leaves + 1] tiles before each leaf
    float* hs = reinterpret_cast<float*>(smem_bf + ((n_leaves + 1 + 3) & ~3));      // [l][kBFTile]
    __shared__ int s_wsum[kBFWarps];
    __shared__ int s_tok[kBFTile];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    pdl_trigger();
    pdl_wait();

    // ---- phase A
    const int n_groups = (B + TPW - 1) / TPW;
    for (int g = blockIdx.x + warp * gridDim.x; g < n_groups; g += gridDim.x * kBFWarps) {
        const T* xr[TPW];
        int64_t n[TPW];
#pragma unroll
        for (int t = 0; t < TPW; ++t) {
            xr[t] = x + (int64_t)min(g * TPW + t, B - 1) * D;
            n[t] = 0;
        }
        int m = 0;
        if (depth > 0) {
            // the seven nodes of the first three levels, for all tokens
            const int levels = min(3, depth);
            const T* wr[8];
            float acc[TPW * 8];
#pragma unroll
            for (int q = 0; q < 8; ++q) wr[q] = node_w + subtree_row(0, 0, min(q, 6), levels) * D;
            block_dots<T, TPW, 8>(xr, wr, D, vec, lane, acc);
            float z = lane_totals<TPW * 8>(acc, lane);
            const int mine = lane / (32 / (TPW * 8));       // the value this lane holds: token mine / 8, node mine % 8
            z += Elem<T>::to_float(node_b[subtree_row(0, 0, min(mine & 7, 6), levels)]);
            const unsigned right = __ballot_sync(kFullMask, z >= 0.0f);
#pragma unroll
            for (int t = 0; t < TPW; ++t) {
                int p = 0;
                for (int i = 0; i < levels; ++i) {
                    const int bit = (int)(right >> ((t * 8 + p) * (32 / (TPW * 8)))) & 1;
                    p = 2 * p + 1 + bit;
                    n[t] = 2 * n[t] + bit;
                }
            }
            m = levels;
        }
        if constexpr (TPW == 1) {
            for (; m < depth; m += 3) {
                const int levels = min(3, depth - m);
                const T* wr[8];
                float acc[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) wr[q] = node_w + subtree_row(m, n[0], min(q, 6), levels) * D;
                block_dots<T, 1, 8>(xr, wr, D, vec, lane, acc);
                const int mine = lane >> 2;
                const float bias = Elem<T>::to_float(node_b[subtree_row(m, n[0], min(mine, 6), levels)]);
                const float z = lane_totals<8>(acc, lane) + bias;
                const unsigned right = __ballot_sync(kFullMask, z >= 0.0f);
                int p = 0;
                for (int i = 0; i < levels; ++i) {
                    const int bit = (int)(right >> (p * 4)) & 1;
                    p = 2 * p + 1 + bit;
                    n[0] = 2 * n[0] + bit;
                }
            }
        } else {
            for (; m < depth; ++m) {
                const int64_t row0 = ((int64_t)1 << m) - 1;
                float acc[8];                               // (four sums and four zeros: lane_totals takes eight)
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i] = 0.0f;
                const T* wr[TPW];
#pragma unroll
                for (int t = 0; t < TPW; ++t) wr[t] = node_w + (row0 + n[t]) * D;
                if (vec) {
                    constexpr int V = Elem<T>::kVec;
                    for (int k = lane * V; k - lane * V < D; k += 64 * V) {
                        uint4 xq[2][TPW], wq[2][TPW];
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int t = 0; t < TPW; ++t) {
                                const bool in = k + i * 32 * V < D;
                                wq[i][t] = in ? __ldg(reinterpret_cast<const uint4*>(wr[t] + k + i * 32 * V)) : make_uint4(0u, 0u, 0u, 0u);
                                xq[i][t] = in ? __ldg(reinterpret_cast<const uint4*>(xr[t] + k + i * 32 * V)) : make_uint4(0u, 0u, 0u, 0u);
                            }
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int t = 0; t < TPW; ++t) {
                                float wv[V], xv[V];
                                Elem<T>::unpack(wq[i][t], wv);
                                Elem<T>::unpack(xq[i][t], xv);
#pragma unroll
                                for (int e = 0; e < V; ++e) acc[t] = fmaf(wv[e], xv[e], acc[t]);
                            }
                    }
                } else {
                    for (int k = lane; k < D; k += 32)
#pragma unroll
                        for (int t = 0; t < TPW; ++t) acc[t] = fmaf(Elem<T>::to_float(wr[t][k]), Elem<T>::to_float(xr[t][k]), acc[t]);
                }
                float z = lane_totals<8>(acc, lane);        // token t's sum in the lanes 4t .. 4t + 3
                const int t_mine = min(lane >> 2, TPW - 1);
                int64_t n_mine = n[0];
#pragma unroll
                for (int t = 1; t < TPW; ++t) n_mine = t_mine == t ? n[t] : n_mine;
                z += Elem<T>::to_float(node_b[row0 + n_mine]);
                const unsigned right = __ballot_sync(kFullMask, z >= 0.0f);
#pragma unroll
                for (int t = 0; t < TPW; ++t) n[t] = 2 * n[t] + (int)((right >> (t * 4)) & 1u);
            }
        }
        if (lane < TPW && g * TPW + lane < B) {
            const int tok = g * TPW + lane;
            int64_t leaf = n[0];
#pragma unroll
            for (int t = 1; t < TPW; ++t) leaf = lane == t ? n[t] : leaf;
            if (leaf_out) leaf_out[tok] = (int32_t)leaf;
            if (leaf_out2) leaf_out2[tok] = (int32_t)leaf;
            slots[leaf * cap + atomicAdd(cursor + leaf, 1)] = tok;
        }
    }
    const bool all_filed = grid_barrier(cursor + n_leaves + 1);
    if (!all_filed && tid == 0) atomicExch(status, kDevTimeout);

    // ---- tiles of every leaf and their running sum, by every CTA for itself
    tiles_before_bins([&](int j) { return __ldcg(cursor + j); }, n_leaves, tile_rows, s_pre, s_wsum, kBFThreads);
    const int n_tiles = all_filed ? s_pre[n_leaves] : 0;

    // ---- phase B
    // threads per group of outputs and tokens per thread in the output layer: narrow layers share a tile's tokens out
    int og = 32;
    while (og < kBFThreads && og < O) og <<= 1;
    const int tpt = kBFTile / min(kBFThreads / og, kBFTile);             // 16, 8, 4 or 2
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const int lo = bin_of_tile(s_pre, n_leaves, tile);
        const int64_t leaf = lo;
        const int first = (tile - s_pre[lo]) * tile_rows;
        const int rows = min(tile_rows, __ldcg(cursor + lo) - first);
        if (tid < kBFTile) s_tok[tid] = __ldcg(slots + leaf * cap + first + min(tid, rows - 1));
        __syncthreads();
        const T* w1j = w1 + leaf * (int64_t)l * D;
        const int tb = (rows + 3) / 4, ub = (l + 7) / 8;    // blocks of tokens and of hidden units
        for (int task = warp; task < tb * ub; task += kBFWarps) {
            const int t0 = (task % tb) * 4, u0 = (task / tb) * 8;
            const T *xr[4], *wr[8];
#pragma unroll
            for (int t = 0; t < 4; ++t) xr[t] = x + (int64_t)s_tok[t0 + t] * D;
#pragma unroll
            for (int u = 0; u < 8; ++u) wr[u] = w1j + (int64_t)min(u0 + u, l - 1) * D;
            float acc[32];
            block_dots<T, 4, 8>(xr, wr, D, vec, lane, acc);
            const int u = u0 + (lane & 7);
            const float bias = u < l ? Elem<T>::to_float(b1[leaf * l + u]) : 0.0f;
            const float sum = lane_totals<32>(acc, lane) + bias;
            if (u < l) hs[u * kBFTile + t0 + (lane >> 3)] = activate(act, sum);
        }
        __syncthreads();
        // output layer
        const T* w2j = w2 + leaf * (int64_t)O * l;
        auto outputs = [&](auto tokens_per_thread) {
            constexpr int TPT = decltype(tokens_per_thread)::value;
            const int ts = (tid / og) * TPT;                // this thread's tokens of the tile
            if (ts >= rows) return;
            // two outputs at a time share the loads of the hidden values
            for (int o = tid % og; o < O; o += 2 * og) {
                const int o2 = o + og < O ? o + og : o;
                const T *wr0 = w2j + (int64_t)o * l, *wr1 = w2j + (int64_t)o2 * l;
                const float bias0 = Elem<T>::to_float(b2[leaf * O + o]), bias1 = Elem<T>::to_float(b2[leaf * O + o2]);
                float acc[2][TPT];
#pragma unroll
                for (int t = 0; t < TPT; ++t) { acc[0][t] = bias0; acc[1][t] = bias1; }
                auto step = [&](int u, float w0, float w1v) {
                    const float* hu = hs + u * kBFTile + ts;
                    constexpr int VH = TPT >= 4 ? 4 : 2;
#pragma unroll
                    for (int t = 0; t < TPT; t += VH) {
                        float hv[VH];
                        if constexpr (VH == 4) {
                            const float4 q = *reinterpret_cast<const float4*>(hu + t);
                            hv[0] = q.x; hv[1] = q.y; hv[2] = q.z; hv[3] = q.w;
                        } else {
                            const float2 q = *reinterpret_cast<const float2*>(hu + t);
                            hv[0] = q.x; hv[1] = q.y;
                        }
#pragma unroll
                        for (int i = 0; i < VH; ++i) {
                            acc[0][t + i] = fmaf(w0, hv[i], acc[0][t + i]);
                            acc[1][t + i] = fmaf(w1v, hv[i], acc[1][t + i]);
                        }
                    }
                };
                if (l % 4 == 0) {                           // rows start on 16-byte (float32) or 8-byte (bf16) boundaries
#pragma unroll 2
                    for (int u = 0; u < l; u += 4) {
                        float wv[2][4];
#pragma unroll
                        for (int r = 0; r < 2; ++r) {
                            const T* wrow = (r ? wr1 : wr0) + u;
                            if constexpr (sizeof(T) == 4) {
                                const float4 q = __ldg(reinterpret_cast<const float4*>(wrow));
                                wv[r][0] = q.x; wv[r][1] = q.y; wv[r][2] = q.z; wv[r][3] = q.w;
                            } else {
                                const uint2 q = __ldg(reinterpret_cast<const uint2*>(wrow));
                                wv[r][0] = __uint_as_float(q.x << 16); wv[r][1] = __uint_as_float(q.x & 0xffff0000u);
                                wv[r][2] = __uint_as_float(q.y << 16); wv[r][3] = __uint_as_float(q.y & 0xffff0000u);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) step(u + i, wv[0][i], wv[1][i]);
                    }
                } else {
#pragma unroll 4
                    for (int u = 0; u < l; ++u) step(u, Elem<T>::to_float(wr0[u]), Elem<T>::to_float(wr1[u]));
                }
#pragma unroll
                for (int t = 0; t < TPT; ++t)
                    if (ts + t < rows) {
                        T* yt = y + (int64_t)s_tok[ts + t] * O;
                        yt[o] = Elem<T>::from_float(acc[0][t]);
                        if (o2 != o) yt[o2] = Elem<T>::from_float(acc[1][t]);
                    }
            }
        };
        if (tpt == 16) outputs(std::integral_constant<int, 16>{});
        else if (tpt == 8) outputs(std::integral_constant<int, 8>{});
        else if (tpt == 4) outputs(std::integral_constant<int, 4>{});
        else outputs(std::integral_constant<int, 2>{});
        __syncthreads();
    }

    // the last CTA to finish clears the counts for the next call
    __syncthreads();
    __shared__ int s_last;
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(cursor + n_leaves, 1) == (int)gridDim.x - 1 ? 1 : 0;
    }
    __syncthreads();
    if (s_last)
        for (int j = tid; j <= n_leaves + 1; j += kBFThreads) cursor[j] = 0;
}

}  // namespace fff
