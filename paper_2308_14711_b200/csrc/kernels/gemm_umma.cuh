// Dense bf16 GEMMs on the fifth-generation tensor cores for FORWARD_T.
//
// Algorithm 1, FORWARD_T: the training-time forward pass evaluates EVERY node and EVERY leaf for every
// token and mixes the leaf outputs with the products of the node choices along the root paths.  Unlike
// hard inference this is a true dense contraction.  It runs as three GEMMs with fused epilogues:
//   nodes    mix[t, j]   = product along leaf j's root path of c or 1 - c, c = sigmoid(<x_t, w_r> + b_r), and the
//                          batch sums of the entropies of c                            (k_train_nodes, depth <= 8)
//   hidden   h'[t, q]    = mix[t, leaf(q)] * act(<x_t, W1_q> + b1_q)      for all 2^d l hidden neurons q
//   output   y[t, o]     = sum_q h'[t, q] W2[o, q] + sum_j mix[t, j] b2[j, o]
// (the mixture of the output biases rides in 2^d extra columns of the K dimension of the last GEMM).  Trees deeper
// than 8 levels take the node choices from k_gemm_pair<kGemmNodes> and the products from k_mixture_weights.
//
// Hidden neurons are kept in an order of their own: blocks of G = min(32, 2^d) leaves, inside a block unit-major, so
// that 32 consecutive columns belong to the leaves g G .. g G + 31 in order (or repeat all leaves when 2^d < 32).  The
// mixture weights of 32 columns are then 32 consecutive floats and no column has to look up which leaf it belongs to;
// with leaf-major columns that look-up was more than half of the epilogue's instructions (50 per value, now 12).
//
// All of them work on pairs of CTAs (cta_group::2): a tile is 256 rows x BN columns, each CTA holds its own 128 rows
// of A and half of the rows of B, which cuts the bytes pulled from L2 into the SMs per multiply-add by a third against
// single CTAs (48 -> 32 KB per CTA and K-block at BN = 256); that traffic is what bounds these kernels.  BN = 256 unless
// the tiles would not fill the GPU.  Per CTA: one warp issues the tensor-map loads of the K-blocks (64 columns) into a
// ring of shared-memory stages, one (first CTA) the four tcgen05.mma (M = 256, N = BN, K = 16) per stage into one of
// two accumulators, sixteen warps read finished accumulators (four per lane quarter, BN / 4 columns each), apply the
// epilogue and hand 32-row pieces to the copy engine through a 4 KB staging tile per warp: a register store of one row
// per lane touches 32 cache lines per instruction, and these stores alone would take as long as the MMAs.
// Tiles that share their rows of A are neighbours in the schedule, so A is read from DRAM once.
//
// 50 432 tokens, D = O = 768, 2^8 leaves of 12, us, before (single CTAs, leaf-major columns, register stores) and now:
// nodes 66 + products 61 + entropies 8 -> 42; hidden 388 -> 243; output 195 -> 195; the whole call, in a loop that the power
// limit slows down, 796 -> 562.  Output runs at the rate of the library's large GEMMs; hidden is bound by power and shared
// memory: its MMAs alone take 180 us, its epilogue alone 145, and forms of the epilogue with fewer loads, fewer instructions
// or direct stores all ended between 245 and 254.
//
// Every wait is bounded (see ptx.cuh); tensor memory is released on every exit path.
// Requirements: bf16, K % 64 == 0, A and B 16-byte aligned with row pitches that are multiples of 16 bytes.
#pragma once

#include <cooperative_groups.h>
#include <cuda.h>      // CUtensorMap

#include "common.cuh"
#include "ptx.cuh"

namespace fff {

using ptx::swz_rows;

constexpr int kGM = 256;                 // rows of C per tile: 128 per CTA of the pair
constexpr int kGRows = 128;
constexpr int kGKB = 64;                 // K-block: 128 bytes, one swizzle line
constexpr int kGMaxStages = 8;
constexpr int kGEpiWarps = 16;           // four per tensor-memory lane quarter: a lone warp per scheduler cannot hide the
                                         // latency of the epilogue arithmetic
constexpr int kGProducerWarp = kGEpiWarps, kGMmaWarp = kGEpiWarps + 1;
constexpr int kGMixWarp = kGEpiWarps + 2;                            // hidden GEMM: mixture weights and biases of the coming tiles
constexpr int kGThreads = (kGEpiWarps + 2) * 32;
constexpr int kGPairThreads = kGThreads + 32;
constexpr int kGWarpStage = 4096;        // staging tile of an epilogue warp: 32 rows of 128 bytes
constexpr int kGSmemMax = 227 * 1024;

enum : int { kGemmNodes = 0, kGemmHidden = 1, kGemmOutput = 2 };

constexpr int kGMixSlots = 2;
constexpr int kGMixBytes = kGRows * 128;                     // a block of mixture weights: 128 rows x 32 leaves, float32

template <int MODE, int BN> struct GemmLayout {
    static_assert(BN == 128 || BN == 256, "columns of a tile");
    static constexpr int kABytes = kGRows * kGKB * 2;
    static constexpr int kBBytes = (BN / 2) * kGKB * 2;                      // this CTA's half of the rows of B
    static constexpr int kStageBytes = kABytes + kBBytes;                    // a multiple of 1024
    static constexpr int kMixBytes = MODE == kGemmHidden ? kGMixSlots * (kGMixBytes + BN * 4) : 0;    // + biases of a tile
    static constexpr int kBarrierBytes = 512;
    static constexpr int kFixed = kGEpiWarps * kGWarpStage + kMixBytes + kBarrierBytes;
    static constexpr int kStages = (kGSmemMax - kFixed) / kStageBytes < kGMaxStages ? (kGSmemMax - kFixed) / kStageBytes : kGMaxStages;
    static constexpr int kSmemBytes = kFixed + kStages * kStageBytes;
    static constexpr int kTmemCols = 2 * BN;                                 // two accumulators (per CTA)
    static constexpr int kColsPerWarp = BN / (kGEpiWarps / 4);               // 64 or 32
};

// Entropy in nats of a Bernoulli choice with probability c, 0 ln 0 = 0.
// (Branch-free: the logarithms take their arguments clamped to the smallest normal float, so that c = 0 and c = 1 give
// 0 x a finite number = 0; with branches the unrolled epilogue would evaluate its 32 values one after the other.)
__device__ __forceinline__ float bernoulli_entropy(float c) {
    const float tiny = 1.17549435e-38f;
    const float d = 1.0f - c;
    return -(c * __logf(fmaxf(c, tiny)) + d * __logf(fmaxf(d, tiny)));
}

// Sums over the warp's 32 rows of all 32 columns at once: in step s every lane hands one half of its values to the
// lane s away and adds what it gets to the half it keeps, so that lane j ends with the total of column j in v[0]
// (31 shuffles instead of 5 per column); the order is fixed.
__device__ __forceinline__ float column_totals(float (&v)[32], int lane) {
#pragma unroll
    for (int sft = 16; sft >= 1; sft >>= 1) {
        const bool upper = (lane & sft) != 0;
#pragma unroll
        for (int i = 0; i < sft; ++i) {
            const float send = upper ? v[i] : v[i + sft];
            const float keep = upper ? v[i + sft] : v[i];
            v[i] = keep + __shfl_xor_sync(kFullMask, send, sft);
        }
    }
    return v[0];
}

// Where the nodes of a tree of DEPTH <= 8 levels sit among the NP >= 2^DEPTH columns of the node GEMM: the tree is cut
// below its first T = min(3, DEPTH) levels into 2^T subtrees of S = DEPTH - T levels; part p owns the 2^S columns from
// p 2^S on: the 2^S - 1 nodes of its subtree in breadth-first order, then, in the last one, top node p (breadth-first).
struct TrainNodeColumns {
    int T, S;
    __host__ __device__ explicit TrainNodeColumns(int depth) : T(depth < 3 ? depth : 3), S(depth - (depth < 3 ? depth : 3)) {}
    // node (index into node_w) of a column, -1 for the columns that hold none
    __host__ __device__ int node(int col) const {
        const int p = col >> S, i = col & ((1 << S) - 1);
        if (p >= (1 << T)) return -1;
        if (i == (1 << S) - 1) return p < (1 << T) - 1 ? p : -1;
        int r = 0;
        while (((2 << r) - 1) <= i) ++r;
        return (1 << (T + r)) - 1 + (p << r) + (i - ((1 << r) - 1));
    }
};

struct GemmEpilogueArgs {
    // kGemmNodes: bias_bf16 = node biases [N], out_f32 = c [M, ld_out]; ent_part (optional) = [m tiles of 128 * 4][N]
    // sums of the entropies over each warp's 32 rows.
    // kGemmHidden: bias = hidden biases in the order of the columns, padded with zeros to whole tiles, mix = [M, n_leaves]
    // float32, l = neurons per leaf, out_bf16 = h' [M, ld_out] (through tmap_c); ent_part / ent_out (optional): the node
    // entropies are finished here from the ent_rows partial sums k_train_nodes left (see there).
    // kGemmOutput: out_bf16 = y [M, ld_out], through tmap_c when tma_out != 0.
    const __nv_bfloat16* bias_bf16;
    const float* bias;
    const float* mix;
    float* out_f32;
    __nv_bfloat16* out_bf16;
    float* ent_part;
    float* ent_out;
    int ent_rows, ent_depth;
    int ld_out, n_leaves, l, act, tma_out;
};

// The roles that the GEMM kernels share: ring of K-blocks, MMAs of the pair.
// smem: [stages][A | B half], barriers as below.
template <int STAGE_BYTES, int A_BYTES>
__device__ __forceinline__ bool pair_produce(unsigned char* ring, uint64_t* full, uint64_t* empty, int stages, const CUtensorMap* ta,
                                             const CUtensorMap* tb, int a_row, int b_row, int KB, int& stage, uint32_t& phase, int lane)
{
    bool ok = true;
    for (int kb = 0; kb < KB; ++kb) {
        if (ok && !ptx::mbar_wait(empty + stage, phase ^ 1)) ok = false;
        if (lane == 0) {
            unsigned char* st = ring + stage * STAGE_BYTES;
            const uint32_t bar = ptx::map_to_cta(ptx::smem_addr(full + stage), 0);
            ptx::mbar_arrive_expect_tx_cluster(bar, (uint32_t)STAGE_BYTES);
            ptx::tma_load_2d_pair(st, ta, kb * kGKB, a_row, bar);
            ptx::tma_load_2d_pair(st + A_BYTES, tb, kb * kGKB, b_row, bar);
        }
        __syncwarp();
        if (++stage == stages) { stage = 0; phase ^= 1; }
    }
    return ok;
}

template <int STAGE_BYTES, int A_BYTES>
__device__ __forceinline__ bool pair_multiply(unsigned char* ring, uint64_t* full, uint64_t* empty, uint64_t* acc_full, int stages,
                                              uint32_t acc, uint32_t idesc, int KB, int& stage, uint32_t& phase, int lane)
{
    bool ok = true;
    for (int kb = 0; kb < KB; ++kb) {
        if (ok && !ptx::mbar_wait(full + stage, phase)) ok = false;
        ptx::tc_fence_after_sync();
        if (lane == 0) {
            const uint32_t xs = ptx::smem_addr(ring + stage * STAGE_BYTES);
            const uint64_t ad = ptx::umma_desc_k128(xs), bd = ptx::umma_desc_k128(xs + A_BYTES);
#pragma unroll
            for (int j = 0; j < kGKB / 16; ++j) ptx::umma_bf16_pair(acc, ad + 2 * j, bd + 2 * j, idesc, (kb | j) != 0 ? 1u : 0u);
            const uint32_t e0 = ptx::smem_addr(empty + stage);
            ptx::umma_commit_pair(ptx::map_to_cta(e0, 0));
            ptx::umma_commit_pair(ptx::map_to_cta(e0, 1));
            if (kb == KB - 1) {
                const uint32_t f0 = ptx::smem_addr(acc_full);
                ptx::umma_commit_pair(ptx::map_to_cta(f0, 0));
                ptx::umma_commit_pair(ptx::map_to_cta(f0, 1));
            }
        }
        __syncwarp();
        if (++stage == stages) { stage = 0; phase ^= 1; }
    }
    return ok;
}

template <int MODE, int BN>
__global__ void __launch_bounds__(kGPairThreads, 1)
k_gemm_pair(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
            const __grid_constant__ CUtensorMap tmap_c, const __grid_constant__ CUtensorMap tmap_mix, int M, int N, int K,
            GemmEpilogueArgs ep, int* __restrict__ status)
{
    namespace cg = cooperative_groups;
    using L = GemmLayout<MODE, BN>;
    extern __shared__ __align__(1024) unsigned char smem_pair[];
    unsigned char* ring = smem_pair;
    unsigned char* staging = ring + L::kStages * L::kStageBytes;                  // [kGEpiWarps][kGWarpStage]
    unsigned char* mix_ring = staging + kGEpiWarps * kGWarpStage;                 // [kGMixSlots][kGMixBytes]   (hidden GEMM)
    float* bias_ring = reinterpret_cast<float*>(mix_ring + kGMixSlots * kGMixBytes);      // [kGMixSlots][BN]
    uint64_t* full = reinterpret_cast<uint64_t*>(mix_ring + L::kMixBytes);        // used in the first CTA only
    uint64_t* empty = full + kGMaxStages;
    uint64_t* acc_full = empty + kGMaxStages;
    uint64_t* acc_empty = acc_full + 2;                                           // used in the first CTA only
    uint64_t* mix_full = acc_empty + 2;
    uint64_t* mix_empty = mix_full + kGMixSlots;
    uint64_t* bias_full = mix_empty + kGMixSlots;
    uint64_t* bias_empty = bias_full + kGMixSlots;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bias_empty + kGMixSlots);

    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank();            // 0: issues the MMAs
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_mt = (M + kGM - 1) / kGM, n_nt = (N + BN - 1) / BN;
    const int n_tiles = n_mt * n_nt;
    // tiles of this pair.  Hidden GEMM: a run of neighbours, so that a block of mixture weights (rows x 32 leaves) serves
    // all the tiles it reaches into.  Output GEMM: pairs take neighbours at the same time, which read the same rows of h'
    // while they are in L2 (h' is far larger than L2; x is not).
    const int n_pairs = gridDim.x >> 1, pair = blockIdx.x >> 1;
    const int tile0 = MODE == kGemmHidden ? (int)((int64_t)n_tiles * pair / n_pairs) : pair;
    const int tile_end = MODE == kGemmHidden ? (int)((int64_t)n_tiles * (pair + 1) / n_pairs) : n_tiles;
    const int tile_stride = MODE == kGemmHidden ? 1 : n_pairs;
    const int KB = K / kGKB;
    // hidden GEMM, 32 leaves or more: the blocks of 32 leaves that the columns of a tile belong to
    const bool blocks = MODE == kGemmHidden && ep.n_leaves >= 32;
    const int gcols = MODE == kGemmHidden ? 32 * ep.l : 1, g_max = MODE == kGemmHidden ? ep.n_leaves / 32 - 1 : 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < L::kStages; ++s) {
            ptx::mbar_init(full + s, 2);                   // one arrival (with its byte count) per CTA
            ptx::mbar_init(empty + s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            ptx::mbar_init(acc_full + a, 1);
            ptx::mbar_init(acc_empty + a, 2 * kGEpiWarps);
        }
        for (int m = 0; m < kGMixSlots; ++m) {
            ptx::mbar_init(mix_full + m, 1);
            ptx::mbar_init(mix_empty + m, kGEpiWarps);
            ptx::mbar_init(bias_full + m, 1);
            ptx::mbar_init(bias_empty + m, kGEpiWarps);
        }
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_a);
        ptx::prefetch_tensormap(&tmap_b);
    }
    if (warp == kGMmaWarp) {
        ptx::tmem_alloc_pair(tmem_slot, L::kTmemCols);
        ptx::tmem_relinquish_alloc_permit_pair();
    }
    ptx::tc_fence_before_sync();
    pdl_trigger();
    cluster.sync();                                        // both CTAs' barriers exist before anything arrives on them
    ptx::tc_fence_after_sync();
    pdl_wait();
    const uint32_t tmem_base = *tmem_slot;

    bool timed_out = false;
    if (warp == kGProducerWarp) {
        // ------------------------------------------------------------------ producer (each CTA: its rows of A, its half of B)
        int stage = 0;
        uint32_t phase = 0;
        for (int tile = tile0; tile < tile_end && !timed_out; tile += tile_stride)
            if (!pair_produce<L::kStageBytes, L::kABytes>(ring, full, empty, L::kStages, &tmap_a, &tmap_b,
                                                          (tile / n_nt) * kGM + (int)rank * kGRows,
                                                          (tile % n_nt) * BN + (int)rank * (BN / 2), KB, stage, phase, lane))
                timed_out = true;
    } else if (warp == kGMmaWarp) {
        // ------------------------------------------------------------------ MMA issuer (first CTA only)
        if (rank == 0) {
            constexpr uint32_t idesc = ptx::umma_idesc_bf16(kGM, BN);
            int stage = 0;
            uint32_t phase = 0;
            int it = 0;
            for (int tile = tile0; tile < tile_end && !timed_out; tile += tile_stride, ++it) {
                const int a = it & 1;
                if (!ptx::mbar_wait(acc_empty + a, ((it >> 1) & 1) ^ 1)) timed_out = true;
                ptx::tc_fence_after_sync();
                if (!pair_multiply<L::kStageBytes, L::kABytes>(ring, full, empty, acc_full + a, L::kStages, tmem_base + a * BN, idesc, KB,
                                                               stage, phase, lane))
                    timed_out = true;
            }
        }
    } else if (warp == kGMixWarp) {
        // ------------------------------------------------------------------ mixture weights and biases of the coming tiles
        if (MODE == kGemmHidden) {
            int slot = 0, it = 0, last_mt = -1, last_g = -1;
            uint32_t phase = 1;
            for (int tile = tile0; tile < tile_end && !timed_out; ++tile, ++it) {
                const int mt = tile / n_nt, c0 = (tile % n_nt) * BN;
                if (!ptx::mbar_wait_relaxed(bias_empty + (it & 1), ((it >> 1) & 1) ^ 1)) timed_out = true;
                if (lane == 0) {
                    ptx::mbar_arrive_expect_tx(bias_full + (it & 1), BN * 4);
                    ptx::bulk_g2s(bias_ring + (it & 1) * BN, ep.bias + c0, BN * 4, bias_full + (it & 1));
                }
                if (!blocks) continue;
                const int g1 = min((c0 + BN - 1) / gcols, g_max);
                for (int g = min(c0 / gcols, g_max); g <= g1 && !timed_out; ++g) {
                    if (mt == last_mt && g == last_g) continue;
                    last_mt = mt;
                    last_g = g;
                    if (!ptx::mbar_wait_relaxed(mix_empty + slot, phase)) timed_out = true;
                    if (lane == 0) {
                        ptx::mbar_arrive_expect_tx(mix_full + slot, kGMixBytes);
                        ptx::tma_load_2d(mix_ring + slot * kGMixBytes, &tmap_mix, g * 32, mt * kGM + (int)rank * kGRows, mix_full + slot);
                    }
                    __syncwarp();
                    if (++slot == kGMixSlots) { slot = 0; phase ^= 1; }
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue: one row of C and one quarter of
        // the tile's columns per thread (warps w, w + 4, w + 8, w + 12 share the lanes of quarter w % 4)
        const int quarter = warp & 3, cpart = warp >> 2;
        constexpr int CP = L::kColsPerWarp;
        unsigned char* my_stage = staging + warp * kGWarpStage;
        int mix_mt = -1, mix_g = 0, mix_slot = kGMixSlots - 1;         // the block of mixture weights in use
        uint32_t mix_phase = 1;
        int it = 0;
        if (MODE == kGemmHidden && ep.ent_out && warp < 4) {
            // node entropies: batch means from the per-CTA sums, added in a fixed order (lane i takes the sums i, i + 32, ...)
            const TrainNodeColumns cols(ep.ent_depth);
            const int np = 1 << ep.ent_depth;
            for (int col = blockIdx.x * 4 + warp; col < np; col += gridDim.x * 4) {
                const int node = cols.node(col);
                if (node < 0) continue;
                float s = 0.0f;
                for (int i = lane; i < ep.ent_rows; i += 32) s += ep.ent_part[(int64_t)i * np + col];
                s = warp_sum(s);
                if (lane == 0) ep.ent_out[node] = s / (float)M;
            }
        }
        for (int tile = tile0; tile < tile_end; tile += tile_stride, ++it) {
            const int a = it & 1;
            const int row0 = (tile / n_nt) * kGM + (int)rank * kGRows + quarter * 32;      // of this warp
            const int col0 = (tile % n_nt) * BN + cpart * CP;
            const int row = row0 + lane;
            const bool row_ok = row < M;
            const bool valid = row0 < M && col0 < N;                                        // warp-uniform
            // on to the block (mt, g) of mixture weights, through the ones before it: they come tile by tile in the order of
            // their columns, a block that the next tile starts with once
            const int mt = tile / n_nt, g_first = min(((tile % n_nt) * BN) / gcols, g_max);
            auto take_block = [&](int g) {
                while (mix_mt != mt || mix_g != g) {
                    __syncwarp();
                    if (mix_mt >= 0 && lane == 0) ptx::mbar_arrive(mix_empty + mix_slot);
                    mix_g = mix_mt == mt ? mix_g + 1 : g_first;
                    mix_mt = mt;
                    if (++mix_slot == kGMixSlots) { mix_slot = 0; mix_phase ^= 1; }
                    if (!timed_out && !ptx::mbar_wait(mix_full + mix_slot, mix_phase)) timed_out = true;
                }
            };
            if (!timed_out && !ptx::mbar_wait(acc_full + a, (it >> 1) & 1)) timed_out = true;
            ptx::tc_fence_after_sync();
            const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + a * BN + cpart * CP;
            if (valid) {
                if (MODE == kGemmNodes) {
#pragma unroll 1
                    for (int c = 0; c < CP / 32; ++c) {
                        const int cc = col0 + c * 32;
                        if (cc >= N) break;
                        uint32_t v[32];
                        ptx::tmem_ld32(taddr + c * 32, v);
                        ptx::tmem_ld_wait();
                        const int nv = min(32, N - cc);
                        float* out = ep.out_f32 + (int64_t)row * ep.ld_out + cc;
                        float cv[32];
#pragma unroll
                        for (int e = 0; e < 32; ++e) {
                            const float logit = __uint_as_float(v[e]) + (e < nv ? __bfloat162float(ep.bias_bf16[cc + e]) : 0.0f);
                            cv[e] = 1.0f / (1.0f + __expf(-logit));
                        }
                        if (row_ok) {
                            if (nv == 32 && (ep.ld_out & 3) == 0) {
#pragma unroll
                                for (int q = 0; q < 8; ++q)
                                    *reinterpret_cast<float4*>(out + 4 * q) = make_float4(cv[4 * q], cv[4 * q + 1], cv[4 * q + 2], cv[4 * q + 3]);
                            } else {
#pragma unroll
                                for (int e = 0; e < 32; ++e)
                                    if (e < nv) out[e] = cv[e];
                            }
                        }
                        if (ep.ent_part) {
#pragma unroll
                            for (int e = 0; e < 32; ++e) cv[e] = (row_ok && e < nv) ? bernoulli_entropy(cv[e]) : 0.0f;
                            const float total = column_totals(cv, lane);
                            if (lane < nv) ep.ent_part[(int64_t)(row0 / 32) * N + cc + lane] = total;
                        }
                    }
                } else {
                    uint32_t packed[CP / 2];
                    if (MODE == kGemmHidden) {
                        const float* mrow = ep.mix + (int64_t)(row_ok ? row : 0) * ep.n_leaves;
                        const float* bt = bias_ring + (it & 1) * BN + cpart * CP;
                        if (!timed_out && !ptx::mbar_wait(bias_full + (it & 1), (it >> 1) & 1)) timed_out = true;
                        with_activation(ep.act, [&](auto act) {
                            constexpr int kAct = decltype(act)::value;
#pragma unroll
                            for (int c = 0; c < CP / 32; ++c) {
                                if (blocks) take_block(min((col0 + c * 32) / gcols, g_max));
                                const unsigned char* wp = mix_ring + mix_slot * kGMixBytes + (quarter * 32 + lane) * 128;
                                uint32_t v[32];
                                ptx::tmem_ld32(taddr + c * 32, v);
                                ptx::tmem_ld_wait();
                                auto weighted = [&](auto in_blocks) {
#pragma unroll
                                    for (int q = 0; q < 8; ++q) {
                                        float4 w;
                                        if (decltype(in_blocks)::value) {
                                            w = *reinterpret_cast<const float4*>(wp + ((q ^ (lane & 7)) << 4));
                                        } else {
                                            const int mk = ep.n_leaves - 1;
                                            w = make_float4(mrow[(4 * q) & mk], mrow[(4 * q + 1) & mk], mrow[(4 * q + 2) & mk], mrow[(4 * q + 3) & mk]);
                                        }
                                        const float4 b = *reinterpret_cast<const float4*>(bt + c * 32 + 4 * q);
                                        const f32x2 h0 = activate_bf16x2<kAct>(add2(pack2u(v[4 * q], v[4 * q + 1]), pack2(b.x, b.y)));
                                        const f32x2 h1 = activate_bf16x2<kAct>(add2(pack2u(v[4 * q + 2], v[4 * q + 3]), pack2(b.z, b.w)));
                                        packed[c * 16 + 2 * q] = to_bf16x2(mul2(h0, pack2(w.x, w.y)));
                                        packed[c * 16 + 2 * q + 1] = to_bf16x2(mul2(h1, pack2(w.z, w.w)));
                                    }
                                };
                                if (blocks) weighted(std::true_type{});
                                else weighted(std::false_type{});
                            }
                        });
                    } else {
#pragma unroll
                        for (int c = 0; c < CP / 32; ++c) {
                            uint32_t v[32];
                            ptx::tmem_ld32(taddr + c * 32, v);
                            ptx::tmem_ld_wait();
#pragma unroll
                            for (int e = 0; e < 16; ++e) packed[c * 16 + e] = ptx::pack_bf16(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1]));
                        }
                    }
                    ptx::tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive_cluster(ptx::map_to_cta(ptx::smem_addr(acc_empty + a), 0));
                    if (MODE == kGemmHidden || ep.tma_out) {
                        // rows of CP bf16 (128 or 64 bytes) in the swizzle of that width, then one tensor-map store per warp
                        if (lane == 0) ptx::bulk_store_wait_read();       // (the store of the tile before)
                        __syncwarp();
#pragma unroll
                        for (int q = 0; q < CP / 8; ++q)
                            *reinterpret_cast<uint4*>(my_stage + swz_rows((uint32_t)(lane * CP * 2 + q * 16), CP * 2)) =
                                make_uint4(packed[4 * q], packed[4 * q + 1], packed[4 * q + 2], packed[4 * q + 3]);
                        ptx::fence_proxy_async();
                        __syncwarp();
                        if (lane == 0) ptx::tma_store_2d(&tmap_c, my_stage, col0, row0);
                    } else if (row_ok) {
                        __nv_bfloat16* out = ep.out_bf16 + (int64_t)row * ep.ld_out + col0;
#pragma unroll
                        for (int e = 0; e < CP; ++e)
                            if (col0 + e < N) out[e] = __ushort_as_bfloat16((unsigned short)((packed[e / 2] >> ((e & 1) * 16)) & 0xffffu));
                    }
                }
            }
            if (!valid || MODE == kGemmNodes) {
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_cluster(ptx::map_to_cta(ptx::smem_addr(acc_empty + a), 0));
            }
            if (MODE == kGemmHidden) {
                // every warp passes all blocks of the tile, so that the releases count up
                if (blocks) take_block(min(((tile % n_nt) * BN + BN - 1) / gcols, g_max));
                if (!valid && !timed_out && !ptx::mbar_wait(bias_full + (it & 1), (it >> 1) & 1)) timed_out = true;
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bias_empty + (it & 1));
            }
        }
        if (lane == 0) ptx::bulk_store_wait_all();
    }
    if (timed_out) {
        if (lane == 0) atomicExch(status, kDevTimeout);
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);     // let copies and MMAs still in flight finish before exit
    }
    ptx::tc_fence_before_sync();
    cluster.sync();                                        // nothing of the pair is in flight any more
    if (warp == kGMmaWarp) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, L::kTmemCols);
    }
}

// Node choices, mixture weights and entropy sums of a tree of 1 <= DEPTH <= 8 levels in one pass over x: the node
// logits of 256 tokens are one tile of the pair, and a thread turns the 2^S columns of a part of its token's row into
// that part's leaf weights in registers.  (With the choices written to memory and the products made by a second kernel
// the two took 66 + 61 us for 50 432 tokens and 255 nodes, plus 8 us for the entropies; the bytes the path cannot do
// without, x in and the weights out as float32 and bf16, are 24 us.)
// tmap_w: rows = columns of TrainNodeColumns in order (NP rows, the absent ones zero), bias [NP] likewise.
// mix [B, 2^d] float32; the same weights as bf16 go to the columns `hidden` .. of h' (row pitch ld_hp); tmap_mix / tmap_tail
// describe both for boxes of one part x 32 rows (kStaged only).
// ent_part (optional): [gridDim.x][2^DEPTH] sums over the CTA's tokens, added in a fixed order.
template <int DEPTH> struct TrainNodesLayout {
    static constexpr int T = DEPTH < 3 ? DEPTH : 3, S = DEPTH - T, kPart = 1 << S;
    static constexpr int NP = (1 << DEPTH) < 32 ? 32 : (1 << DEPTH);
    static constexpr int kABytes = kGRows * kGKB * 2;
    static constexpr int kBBytes = (NP / 2) * kGKB * 2;
    static constexpr int kStageBytes = kABytes + kBBytes;                    // a multiple of 1024
    // with 16 or 32 leaves per part the weights leave through staging tiles (float32 rows, then bf16 rows) and tensor-map
    // stores, one of each per warp and part: as register stores, one row per lane, they took longer than the loads of a tile
    static constexpr bool kStaged = kPart >= 16;
    static constexpr int kWarpStage = kStaged ? 32 * kPart * 6 : 0;
    static constexpr int kFixed = 1024 + 512 + NP * 4 + kGEpiWarps * kWarpStage;
    static constexpr int kStages = (kGSmemMax - kFixed) / kStageBytes < kGMaxStages ? (kGSmemMax - kFixed) / kStageBytes : kGMaxStages;
    static constexpr int kSmemBytes = kFixed + kStages * kStageBytes;
    // columns that one load brings of a part (of a narrow one more than it has), and tensor memory for all that the loads of the
    // last part of the second accumulator touch: with 2 NP columns, those of trees of 5 and 6 levels ended 12 and 8 columns past it
    static constexpr int kLoadCols = kPart == 32 ? 32 : 16;
    static constexpr int kTouched = NP + ((1 << T) - 1) * kPart + kLoadCols;
    static constexpr int kTmemCols = kTouched <= 64 ? 64 : kTouched <= 128 ? 128 : kTouched <= 256 ? 256 : 512;
    static_assert(kTouched <= kTmemCols && 2 * NP <= kTmemCols, "both accumulators and every load lie inside the allocation");
    static_assert(4 * NP * 4 <= kStages * kStageBytes, "the entropy sums take the ring's place at the end");
};

template <int DEPTH>
__global__ void __launch_bounds__(kGThreads, 1)
k_train_nodes(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w,
              const __grid_constant__ CUtensorMap tmap_mix, const __grid_constant__ CUtensorMap tmap_tail, const float* __restrict__ bias,
              float* __restrict__ mix, __nv_bfloat16* __restrict__ hp, int ld_hp, int hidden, float* __restrict__ ent_part, int B, int D,
              int* __restrict__ status)
{
    namespace cg = cooperative_groups;
    using L = TrainNodesLayout<DEPTH>;
    constexpr int NP = L::NP, PART = L::kPart, T = L::T;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char* staging = ring + L::kStages * L::kStageBytes;                  // [kGEpiWarps][kWarpStage]
    uint64_t* full = reinterpret_cast<uint64_t*>(staging + kGEpiWarps * L::kWarpStage);
    uint64_t* empty = full + kGMaxStages;
    uint64_t* acc_full = empty + kGMaxStages;
    uint64_t* acc_empty = acc_full + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
    float* s_bias = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(full) + 512);     // [NP]
    float* s_ent = reinterpret_cast<float*>(ring);                                // [4 quarters][NP], once the last MMA is done

    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_tiles = (B + kGM - 1) / kGM;
    const int tile0 = blockIdx.x >> 1, tile_stride = gridDim.x >> 1;
    const int KB = D / kGKB;

    if (threadIdx.x == 0) {
        for (int s = 0; s < L::kStages; ++s) {
            ptx::mbar_init(full + s, 2);
            ptx::mbar_init(empty + s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            ptx::mbar_init(acc_full + a, 1);
            ptx::mbar_init(acc_empty + a, 2 * kGEpiWarps);
        }
        ptx::fence_mbar_init();
        ptx::prefetch_tensormap(&tmap_x);
        ptx::prefetch_tensormap(&tmap_w);
    }
    if (warp == kGMmaWarp) {
        ptx::tmem_alloc_pair(tmem_slot, L::kTmemCols);
        ptx::tmem_relinquish_alloc_permit_pair();
    }
    for (int i = threadIdx.x; i < NP; i += kGThreads) s_bias[i] = bias[i];
    ptx::tc_fence_before_sync();
    pdl_trigger();
    cluster.sync();
    ptx::tc_fence_after_sync();
    pdl_wait();
    const uint32_t tmem_base = *tmem_slot;

    bool timed_out = false;
    if (warp == kGProducerWarp) {
        int stage = 0;
        uint32_t phase = 0;
        for (int tile = tile0; tile < n_tiles && !timed_out; tile += tile_stride)
            if (!pair_produce<L::kStageBytes, L::kABytes>(ring, full, empty, L::kStages, &tmap_x, &tmap_w, tile * kGM + (int)rank * kGRows,
                                                          (int)rank * (NP / 2), KB, stage, phase, lane))
                timed_out = true;
    } else if (warp == kGMmaWarp) {
        if (rank == 0) {
            constexpr uint32_t idesc = ptx::umma_idesc_bf16(kGM, NP);
            int stage = 0;
            uint32_t phase = 0;
            int it = 0;
            for (int tile = tile0; tile < n_tiles && !timed_out; tile += tile_stride, ++it) {
                const int a = it & 1;
                if (!ptx::mbar_wait(acc_empty + a, ((it >> 1) & 1) ^ 1)) timed_out = true;
                ptx::tc_fence_after_sync();
                if (!pair_multiply<L::kStageBytes, L::kABytes>(ring, full, empty, acc_full + a, L::kStages, tmem_base + a * NP, idesc, KB,
                                                               stage, phase, lane))
                    timed_out = true;
            }
        }
    } else {
        const int quarter = warp & 3, cw = warp >> 2;
        constexpr int PARTS = 1 << T, PER_WARP = PARTS > 4 ? 2 : 1;      // parts of a thread: cw (and cw + 4)
        unsigned char* my_stage = staging + warp * L::kWarpStage;
        float ent_acc[PER_WARP];
#pragma unroll
        for (int i = 0; i < PER_WARP; ++i) ent_acc[i] = 0.0f;
        int it = 0;
        for (int tile = tile0; tile < n_tiles; tile += tile_stride, ++it) {
            const int a = it & 1;
            const int row = tile * kGM + (int)rank * kGRows + quarter * 32 + lane;
            const bool row_ok = row < B;
            if (!timed_out && !ptx::mbar_wait(acc_full + a, (it >> 1) & 1)) timed_out = true;
            ptx::tc_fence_after_sync();
            const uint32_t tq = tmem_base + ((uint32_t)(quarter * 32) << 16) + a * NP;
#pragma unroll
            for (int i = 0; i < PER_WARP; ++i) {
                const int p = cw + 4 * i;
                if (p >= PARTS) continue;                                 // warp-uniform
                // the logits of the part's own columns, and of the top nodes on its path
                float z[32];
                {
                    uint32_t v[32];
                    if (L::kLoadCols == 32) ptx::tmem_ld32(tq + p * PART, v);
                    else {
                        uint32_t v16[16];
                        ptx::tmem_ld16(tq + p * PART, v16);               // (columns past the part are not used)
#pragma unroll
                        for (int e = 0; e < 16; ++e) v[e] = v16[e];
                    }
                    uint32_t top[3] = {0u, 0u, 0u};
#pragma unroll
                    for (int m = 0; m < T; ++m) {
                        const int node = (1 << m) - 1 + (p >> (T - m));
                        ptx::tmem_ld1(tq + node * PART + PART - 1, top[m]);
                    }
                    ptx::tmem_ld_wait();
                    if (i == PER_WARP - 1 || p + 4 >= PARTS) {
                        // last read of this accumulator by the warp
                        ptx::tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive_cluster(ptx::map_to_cta(ptx::smem_addr(acc_empty + a), 0));
                    }
#pragma unroll
                    for (int e = 0; e < 32; ++e) z[e] = e < PART ? __uint_as_float(v[e < PART ? e : 0]) + s_bias[p * PART + e] : 0.0f;
                    // path product down to the part's subtree (the same order as the recursion: root first)
                    float w[PART];
                    w[0] = 1.0f;
#pragma unroll
                    for (int m = 0; m < T; ++m) {
                        const int node = (1 << m) - 1 + (p >> (T - m));
                        float right, left, h;
                        node_choice(__uint_as_float(top[m]) + s_bias[node * PART + PART - 1], right, left, h);
                        w[0] *= ((p >> (T - m - 1)) & 1) ? right : left;
                    }
                    // the subtree, level by level; z becomes the entropies
#pragma unroll
                    for (int r = 0; r < L::S; ++r) {
#pragma unroll
                        for (int n = 0; n < 16; ++n) {
                            if (n >= (1 << r)) continue;
                            constexpr int kLast = PART - 1;                // (keeps the indices of the skipped iterations in range)
                            const int j = (1 << r) - 1 - n, c = ((1 << r) - 1 + j) & kLast;
                            float right, left, h;
                            node_choice(z[c], right, left, h);
                            z[c] = h;
                            const float q = w[j & kLast];
                            w[(2 * j + 1) & kLast] = q * right;
                            w[(2 * j) & kLast] = q * left;
                        }
                    }
                    if (ent_part) {
                        float right, left, h;
                        node_choice(z[PART - 1], right, left, h);         // top node p (the last part's column holds none: ignored below)
                        z[PART - 1] = h;
#pragma unroll
                        for (int e = 0; e < 32; ++e) z[e] = (row_ok && e < PART) ? z[e] : 0.0f;
                        ent_acc[i] += column_totals(z, lane);
                    }
                    if constexpr (L::kStaged) {
                        float* fs = reinterpret_cast<float*>(my_stage);
                        unsigned char* bs = my_stage + 32 * PART * 4;
                        if (lane == 0) ptx::bulk_store_wait_read();
                        __syncwarp();
#pragma unroll
                        for (int q = 0; q < PART / 4; ++q)
                            *reinterpret_cast<float4*>(reinterpret_cast<unsigned char*>(fs) + swz_rows((uint32_t)(lane * PART * 4 + q * 16), PART * 4)) =
                                make_float4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
#pragma unroll
                        for (int q = 0; q < PART / 8; ++q)
                            *reinterpret_cast<uint4*>(bs + swz_rows((uint32_t)(lane * PART * 2 + q * 16), PART * 2)) =
                                make_uint4(ptx::pack_bf16(w[8 * q], w[8 * q + 1]), ptx::pack_bf16(w[8 * q + 2], w[8 * q + 3]),
                                           ptx::pack_bf16(w[8 * q + 4], w[8 * q + 5]), ptx::pack_bf16(w[8 * q + 6], w[8 * q + 7]));
                        ptx::fence_proxy_async();
                        __syncwarp();
                        if (lane == 0 && row < B) {                       // (lane 0 carries the warp's first row)
                            ptx::tma_store_2d(&tmap_mix, my_stage, p * PART, row);
                            ptx::tma_store_2d(&tmap_tail, bs, p * PART, row);
                        }
                    } else if (row_ok) {
                        float* mo = mix + (int64_t)row * (1 << DEPTH) + p * PART;
                        __nv_bfloat16* ho = hp + (int64_t)row * ld_hp + hidden + p * PART;
#pragma unroll
                        for (int e = 0; e < PART; ++e) {
                            mo[e] = w[e];
                            ho[e] = __float2bfloat16_rn(w[e]);
                        }
                    }
                }
            }
            if (cw >= PARTS) {                                            // (fewer parts than column warps)
                ptx::tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive_cluster(ptx::map_to_cta(ptx::smem_addr(acc_empty + a), 0));
            }
        }
        if (L::kStaged && lane == 0) ptx::bulk_store_wait_all();
        if (ent_part) {
#pragma unroll
            for (int i = 0; i < PER_WARP; ++i)
                if (cw + 4 * i < PARTS && lane < PART) s_ent[quarter * NP + (cw + 4 * i) * PART + lane] = ent_acc[i];
        }
    }
    if (timed_out) {
        if (lane == 0) atomicExch(status, kDevTimeout);
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    }
    ptx::tc_fence_before_sync();
    cluster.sync();
    if (ent_part)
        for (int c = threadIdx.x; c < (1 << DEPTH); c += kGThreads)
            ent_part[(int64_t)blockIdx.x * (1 << DEPTH) + c] = (s_ent[c] + s_ent[NP + c]) + (s_ent[2 * NP + c] + s_ent[3 * NP + c]);
    if (warp == kGMmaWarp) {
        ptx::tc_fence_after_sync();
        ptx::tmem_dealloc_pair(tmem_base, L::kTmemCols);
    }
}

// The products along the root path of leaf j for kMixTokens tokens at once, for a tree of DEPTH levels (ct[u] = token
// u's node choices, nullptr = no token): all loads are independent of each other and are issued before the products
// start (with a run-time depth the loop stays rolled and every level waits for its own load: DEPTH round trips to L2
// per value, one token at a time).
constexpr int kMixTokens = 4;
template <int DEPTH>
__device__ __forceinline__ void path_products(const float* const (&ct)[kMixTokens], int j, float (&p)[kMixTokens]) {
    float cv[kMixTokens][DEPTH];
#pragma unroll
    for (int u = 0; u < kMixTokens; ++u)
#pragma unroll
        for (int m = 0; m < DEPTH; ++m) cv[u][m] = ct[u] ? ct[u][(1 << m) - 1 + (j >> (DEPTH - m))] : 0.0f;
#pragma unroll
    for (int u = 0; u < kMixTokens; ++u) {
        float q = 1.0f;
#pragma unroll
        for (int m = 0; m < DEPTH; ++m) q *= ((j >> (DEPTH - m - 1)) & 1) ? cv[u][m] : 1.0f - cv[u][m];
        p[u] = q;
    }
}

// Mixture weights of FORWARD_T from the node choices: unrolling the recursion of Algorithm 1, leaf j enters the
// output with the product over its root path of c (where the path turns right) or 1 - c (left).
// c: [B, ldc] float32 (node r in column r);  mix: [B, 2^d] float32 (optional: mix_user, a second copy);
// hp_tail: the same weights as bf16 in the last 2^d used columns of the rows of h' (row pitch ld_hp), where
// the output GEMM multiplies them with the output biases; the padding columns up to ld_hp are zeroed.
// A block takes kMixTokens tokens at a time, a thread one column of each (no 64-bit divisions in the loop).
__global__ void __launch_bounds__(256)
k_mixture_weights(const float* __restrict__ c, int ldc, float* __restrict__ mix, float* __restrict__ mix_user,
                  __nv_bfloat16* __restrict__ hp, int ld_hp, int hidden, int depth, int64_t B)
{
    const int nl = 1 << depth;
    const int tail = ld_hp - hidden;                          // >= nl: mixture columns, then zero padding
    for (int64_t t0 = (int64_t)blockIdx.x * kMixTokens; t0 < B; t0 += (int64_t)gridDim.x * kMixTokens)
    for (int j = threadIdx.x; j < tail; j += blockDim.x) {
        float p[kMixTokens];
#pragma unroll
        for (int u = 0; u < kMixTokens; ++u) p[u] = 0.0f;
        if (j < nl) {
            const float* ct[kMixTokens];
#pragma unroll
            for (int u = 0; u < kMixTokens; ++u) ct[u] = t0 + u < B ? c + (t0 + u) * ldc : nullptr;
            switch (depth) {            // (the same multiplications in the same order in every case)
                case 9: path_products<9>(ct, j, p); break;
                case 10: path_products<10>(ct, j, p); break;
                case 11: path_products<11>(ct, j, p); break;
                case 12: path_products<12>(ct, j, p); break;
                default:
#pragma unroll
                    for (int u = 0; u < kMixTokens; ++u) {
                        if (!ct[u]) continue;
                        float q = 1.0f;
                        for (int m = 0; m < depth; ++m) {
                            const float cv = ct[u][(1 << m) - 1 + (j >> (depth - m))];
                            q *= ((j >> (depth - m - 1)) & 1) ? cv : 1.0f - cv;
                        }
                        p[u] = q;
                    }
            }
        }
#pragma unroll
        for (int u = 0; u < kMixTokens; ++u) {
            const int64_t t = t0 + u;
            if (t >= B) break;
            if (j < nl) {
                mix[t * nl + j] = p[u];
                if (mix_user) mix_user[t * nl + j] = p[u];
            }
            hp[t * ld_hp + hidden + j] = __float2bfloat16_rn(p[u]);
        }
    }
}

// Batch means of the node entropies from the per-warp partial sums of the node GEMM, added in a fixed order:
// one warp per node, lane i adds the parts i, i + 32, ... in order, then the lanes' sums are added by a fixed tree.
// Blocks of 8 warps.
__global__ void __launch_bounds__(256)
k_entropy_reduce(const float* __restrict__ part, int n_parts, int n_nodes, int64_t B, float* __restrict__ ent)
{
    const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= n_nodes) return;
    float s = 0.0f;
    for (int p = lane; p < n_parts; p += 32) s += part[(int64_t)p * n_nodes + r];
    s = warp_sum(s);
    if (lane == 0) ent[r] = s / (float)B;
}

// Position of hidden neuron (leaf j, unit u) among the columns of h' (see the top of this file).
__host__ __device__ __forceinline__ int64_t train_column(int64_t j, int u, int n_leaves, int l) {
    const int G = n_leaves < 32 ? n_leaves : 32;
    return (j / G) * ((int64_t)G * l) + (int64_t)u * G + j % G;
}

// Columns of h' that the hidden neurons take: whole 16-byte units (a tensor-map store whose last unit crosses the end of
// its matrix writes that unit whole, and the mixture weights follow right behind).
__host__ __device__ __forceinline__ int train_hidden_columns(int n_leaves, int l) { return (n_leaves * l + 7) & ~7; }

// B operand of the output GEMM: w2t [O][Kp] bf16, column train_column(j, u) = W2[j][o][u], then from column
// train_hidden_columns on b2[j][o], all other columns zero.
template <typename T>
__global__ void k_pack_w2_transposed(const T* __restrict__ w2, const T* __restrict__ b2, __nv_bfloat16* __restrict__ w2t,
                                     int n_leaves, int l, int O, int Kp)
{
    const int64_t total = (int64_t)O * Kp;
    const int hidden = n_leaves * l, tail = train_hidden_columns(n_leaves, l), G = n_leaves < 32 ? n_leaves : 32;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t o = i / Kp;
        const int q = (int)(i % Kp);
        float v = 0.0f;
        if (q < hidden) {
            const int64_t j = (int64_t)(q / (G * l)) * G + q % G;
            v = Elem<T>::to_float(w2[(j * O + o) * l + (q % (G * l)) / G]);
        } else if (q >= tail && q < tail + n_leaves && b2) {
            v = Elem<T>::to_float(b2[(int64_t)(q - tail) * O + o]);
        }
        w2t[i] = __float2bfloat16_rn(v);
    }
}

// B operand and biases of the hidden GEMM in the order of train_column: w1t [train_hidden_columns][D] bf16, b1t [padded]
// float32; rows without a neuron are zero.
template <typename T>
__global__ void k_pack_train_hidden(const T* __restrict__ w1, const T* __restrict__ b1, __nv_bfloat16* __restrict__ w1t, float* __restrict__ b1t,
                                    int n_leaves, int l, int D, int padded)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int hidden = n_leaves * l, G = n_leaves < 32 ? n_leaves : 32, units = D / 8;      // 16-byte units of a row (D % 64 == 0)
    for (int64_t i = t0; i < (int64_t)train_hidden_columns(n_leaves, l) * units; i += stride) {
        const int q = (int)(i / units);
        if (q >= hidden) {
            reinterpret_cast<uint4*>(w1t)[i] = make_uint4(0u, 0u, 0u, 0u);
            continue;
        }
        const int64_t j = (int64_t)(q / (G * l)) * G + q % G;
        const int u = (q % (G * l)) / G;
        reinterpret_cast<uint4*>(w1t)[i] = reinterpret_cast<const uint4*>(w1)[(j * l + u) * units + i % units];
    }
    for (int64_t q = t0; q < padded; q += stride) {
        float v = 0.0f;
        if (q < hidden && b1) v = Elem<T>::to_float(b1[((q / (G * l)) * G + q % G) * l + (q % (G * l)) / G]);
        b1t[q] = v;
    }
}

// B operand and biases of k_train_nodes: rows in the order of TrainNodeColumns, the columns without a node zero.
template <typename T>
__global__ void k_pack_train_nodes(const T* __restrict__ node_w, const T* __restrict__ node_b, __nv_bfloat16* __restrict__ wn,
                                   float* __restrict__ bn, int depth, int NP, int D)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const TrainNodeColumns cols(depth);
    for (int64_t i = t0; i < (int64_t)NP * D; i += stride) {
        const int node = cols.node((int)(i / D));
        wn[i] = node < 0 ? __float2bfloat16_rn(0.0f) : __float2bfloat16_rn(Elem<T>::to_float(node_w[(int64_t)node * D + i % D]));
    }
    for (int64_t c = t0; c < NP; c += stride) {
        const int node = cols.node((int)c);
        bn[c] = node < 0 || !node_b ? 0.0f : Elem<T>::to_float(node_b[node]);
    }
}

}  // namespace fff
