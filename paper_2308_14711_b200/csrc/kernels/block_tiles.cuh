// k_block_forward for float32 layers whose operands fit an SM's shared memory in pieces: the same cooperative launch (descent, grid
// barrier, tiles of a leaf's tokens), the same sums in the same order, with every matrix brought into shared memory by bulk copies.
//
// What bound k_block_forward (float32, 768 -> 768, 256 leaves of 12, 6304 tokens; clock stamps of one launch): the registers hold the
// loads of one step of 128 columns, so a block of dot products was a chain of six round trips of 1.5 us and a tile two such chains:
// hidden layer 9.6 us, output layer 7, two tiles per CTA, of 57 us in all.  Bulk copies cost no registers: a tile's rows of x and its
// leaf's W1 and W2, in blocks of up to a ring slot, are sent for as far ahead as the ring holds, across tiles, each by the warp that was
// the last to read what lay there (hidden layer 3.5 to 4, output layer 4).  Which batches it is taken for and what it measured: block_tiles_plan in
// fff_api.cu.
// Bound: in the descent the rows of the nodes below the first three levels, 130 KB per SM and level from L2 (12 us of 48); in the hidden
// layer shared memory (48 cycles of loads per 32 of multiply-adds).  The top four levels in shared memory changed nothing.
//   phase A  a warp takes kTok = 1 to 4 neighbouring tokens, so many that the batch is one pass where it can be, and copies
//            their rows; the seven nodes of the first three levels are in shared memory too, shared by all warps.  Below, node rows
//            are read from L2 as in k_block_forward: three levels at a time with one token per warp, else one.
//   phase B  tiles of up to tile_rows = 8, 16 or 32 tokens of one leaf.  Hidden layer: warps share out blocks of 4 tokens x 8 hidden
//            units.  Output layer: from W2 transposed ([l][O], an image of the library's own), so that neighbouring
//            threads read neighbouring weights; a thread keeps up to 4 outputs of up to 16 tokens in registers over all units.
// 16 warps share one CTA per SM: a leaf's weights are fetched once per 32 tokens.
// Rows that do not start on 16-byte boundaries (D or O no multiple of 4) are copied from the boundary before them; the up to three
// values past the last whole 16 bytes of x are fetched one by one.
#pragma once

#include "block_forward.cuh"
#include "ptx.cuh"

namespace fff {

constexpr int kBTWarps = 16;
constexpr int kBTThreads = kBTWarps * 32;
constexpr int kBTTile = 32;                                // most tokens per tile
constexpr int kBTMaxTok = 4;                               // most tokens per warp in phase A
constexpr int kBTMaxSlots = 8;
constexpr int kBTMaxOut = 1024;                            // most outputs (4 per thread of 256)
constexpr int kBTTop = 7;                                  // nodes of the first three levels

// Shared memory, in floats; every part starts on 16 bytes.  A part that holds n values from an arbitrary start is n + 3 rounded up
// to 4 long: the copy begins at the 16-byte boundary before the first of them.
struct BlockTilesLayout {
    int x_pitch;                      // a staged row of x
    int slot;                         // a ring slot
    int w1_units;                     // hidden units per W1 block, a multiple of 8
    int w2_units;                     // units (rows of W2 transposed) per W2 block
    int slots, tile_rows, tok;
    int hs_at, pre_at, bar_at;        // offsets of the parts behind x and the ring; those of phase A (nodes, rows) start at 0
    int total_bytes;
    __host__ __device__ static int part(int n) { return (n + 3 + 3) & ~3; }
    // false: does not fit `budget` bytes.  tok: tokens per warp in phase A, lowered to what fits.
    __host__ bool plan(int D, int O, int l, int n_leaves, int tile_rows_, int tok_, int budget) {
        tile_rows = tile_rows_;
        x_pitch = part(D);
        const int row_bytes = D * 4;
        int groups = (24 * 1024) / (8 * row_bytes);                        // blocks of about 24 KB, of 8 units at least
        if (groups < 1) groups = 1;
        if (groups > (l + 7) / 8) groups = (l + 7) / 8;
        w1_units = 8 * groups;
        const int w1_rows = w1_units < l ? w1_units : l;
        int payload = w1_rows * D;
        if (payload < O) payload = O;
        w2_units = payload / O < l ? payload / O : l;
        slot = part(payload);
        const int tail = ((l * kBTTile + 3) & ~3) + ((2 * n_leaves + 1 + 3) & ~3) + 2 * (kBTMaxSlots + kBTWarps + 2);
        const int room = budget / 4 - tail;
        const int x_area = tile_rows * x_pitch;
        slots = (room - x_area) / slot;
        if (slots > kBTMaxSlots) slots = kBTMaxSlots;
        if (slots < 2) return false;
        int front = x_area + slots * slot;
        // phase A lies over the same floats
        const int top = part(kBTTop * D);
        tok = tok_;
        while (tok > 1 && top + kBTWarps * part(tok * D) > room) --tok;
        const int a = top + kBTWarps * part(tok * D);
        if (a > room) return false;
        if (front < a) front = a;
        hs_at = front;
        pre_at = hs_at + ((l * kBTTile + 3) & ~3);
        bar_at = pre_at + ((2 * n_leaves + 1 + 3) & ~3);
        total_bytes = 4 * (front + tail);
        return true;
    }
};

// Copies n floats from `src` (any 4-byte boundary) to dst + head, head = the floats between the 16-byte boundary before src and src;
// up to `slack` floats past the end may be read (3: an allocation of the library's own, rounded up; else 0: then the floats past the
// last whole 16 bytes are left to copy_rest).  Returns the bytes that `bar` will count.
__device__ __forceinline__ uint32_t bulk_floats(float* dst, const float* src, int n, bool slack, uint64_t* bar) {
    const int head = (int)((reinterpret_cast<uintptr_t>(src) >> 2) & 3);
    const int whole = slack ? (head + n + 3) & ~3 : (head + n) & ~3;
    if (whole > 0) ptx::bulk_g2s(dst, src - head, (uint32_t)whole * 4, bar);
    return (uint32_t)whole * 4;
}
__device__ __forceinline__ int head_of(const float* src) { return (int)((reinterpret_cast<uintptr_t>(src) >> 2) & 3); }

// acc[t * NW + w] = partial dot products of the rows xr[t] and wr[w] in shared memory (this lane's share of the columns, in the order
// of block_dots).  vec: rows on 16-byte boundaries, D % 4 == 0.
template <int NX, int NW>
__device__ __forceinline__ void shared_dots(const float* const (&xr)[NX], const float* const (&wr)[NW], int D, bool vec, int lane,
                                            float (&acc)[NX * NW])
{
#pragma unroll
    for (int i = 0; i < NX * NW; ++i) acc[i] = 0.0f;
    if (vec) {
        for (int k = lane * 4; k < D; k += 128) {
            float4 xq[NX];
#pragma unroll
            for (int t = 0; t < NX; ++t) xq[t] = *reinterpret_cast<const float4*>(xr[t] + k);
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const float4 wq = *reinterpret_cast<const float4*>(wr[w] + k);
#pragma unroll
                for (int t = 0; t < NX; ++t) {
                    float a = acc[t * NW + w];
                    a = fmaf(wq.x, xq[t].x, a);
                    a = fmaf(wq.y, xq[t].y, a);
                    a = fmaf(wq.z, xq[t].z, a);
                    acc[t * NW + w] = fmaf(wq.w, xq[t].w, a);
                }
            }
        }
    } else {
#pragma unroll 2
        for (int k = lane; k < D; k += 32) {
            float xv[NX];
#pragma unroll
            for (int t = 0; t < NX; ++t) xv[t] = xr[t][k];
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const float wv = wr[w][k];
#pragma unroll
                for (int t = 0; t < NX; ++t) acc[t * NW + w] = fmaf(wv, xv[t], acc[t * NW + w]);
            }
        }
    }
}

// The walk of kTok tokens (rows xr in shared memory): node numbers of level `depth` in n.  top: the first seven node rows.
template <int kTok>
__device__ __forceinline__ void walk_staged(const float* const (&xr)[kTok], const float* top, const float* __restrict__ node_w,
                                            const float* __restrict__ node_b, int D, int depth, bool vec, int lane, int (&n)[kTok])
{
    constexpr int kPad = kTok == 1 ? 1 : kTok == 2 ? 2 : 4;              // (lane_totals takes 8, 16 or 32 values)
#pragma unroll
    for (int t = 0; t < kTok; ++t) n[t] = 0;
    if (depth == 0) return;
    {
        const int levels = min(3, depth);
        const float* wr[8];
        float acc[kTok * 8], v[kPad * 8];
#pragma unroll
        for (int q = 0; q < 8; ++q) wr[q] = top + subtree_row(0, 0, min(q, 6), levels) * D;
        const int mine = lane / (32 / (kPad * 8));                       // the value this lane will hold: token mine / 8, node mine % 8
        const float bias = __ldg(node_b + subtree_row(0, 0, min(mine & 7, 6), levels));
        shared_dots<kTok, 8>(xr, wr, D, vec, lane, acc);
#pragma unroll
        for (int i = 0; i < kPad * 8; ++i) v[i] = i < kTok * 8 ? acc[i] : 0.0f;
        const float z = lane_totals<kPad * 8>(v, lane) + bias;
        const unsigned right = __ballot_sync(kFullMask, z >= 0.0f);
#pragma unroll
        for (int t = 0; t < kTok; ++t) {
            int p = 0;
            for (int i = 0; i < levels; ++i) {
                const int bit = (int)(right >> ((t * 8 + p) * (32 / (kPad * 8)))) & 1;
                p = 2 * p + 1 + bit;
                n[t] = 2 * n[t] + bit;
            }
        }
    }
    auto get = [&](const float* row, int k) { return k < D ? __ldg(reinterpret_cast<const float4*>(row + k)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f); };
    auto add = [](float a, const float4& w, const float4& x) {
        a = fmaf(w.x, x.x, a);
        a = fmaf(w.y, x.y, a);
        a = fmaf(w.z, x.z, a);
        return fmaf(w.w, x.w, a);
    };
    if constexpr (kTok == 1) {
        // three levels at a time: a round trip decides three
        for (int m = 3; m < depth; m += 3) {
            const int levels = min(3, depth - m);
            const float* wr[7];
            float acc[8];
#pragma unroll
            for (int q = 0; q < 7; ++q) wr[q] = node_w + subtree_row(m, n[0], q, levels) * D;
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] = 0.0f;
            const int mine = min(lane >> 2, 6);
            const float bias = __ldg(node_b + subtree_row(m, n[0], mine, levels));
            if (vec) {
                for (int k = lane * 4; k - lane * 4 < D; k += 256) {
                    float4 wq[2][7];
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int q = 0; q < 7; ++q) wq[i][q] = get(wr[q], k + i * 128);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        if (k + i * 128 >= D) break;
                        const float4 xq = *reinterpret_cast<const float4*>(xr[0] + k + i * 128);
#pragma unroll
                        for (int q = 0; q < 7; ++q) acc[q] = add(acc[q], wq[i][q], xq);
                    }
                }
            } else {
#pragma unroll 4
                for (int k = lane; k < D; k += 32) {
                    const float xv = xr[0][k];
#pragma unroll
                    for (int q = 0; q < 7; ++q) acc[q] = fmaf(__ldg(wr[q] + k), xv, acc[q]);
                }
            }
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
        for (int m = 3; m < depth; ++m) {
            const int64_t row0 = ((int64_t)1 << m) - 1;
            const float* wr[kTok];
            float acc[8];                                    // (sums and zeros: lane_totals takes eight)
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[i] = 0.0f;
#pragma unroll
            for (int t = 0; t < kTok; ++t) wr[t] = node_w + (row0 + n[t]) * D;
            const int t_mine = min(lane >> 2, kTok - 1);
            int n_mine = n[0];
#pragma unroll
            for (int t = 1; t < kTok; ++t) n_mine = t_mine == t ? n[t] : n_mine;
            const float bias = __ldg(node_b + row0 + n_mine);
            if (vec) {
                constexpr int kAhead = kTok == 2 ? 8 : kTok == 3 ? 6 : 4;      // steps of 128 columns whose loads are issued together (64 or 72 registers)
                for (int k = lane * 4; k - lane * 4 < D; k += kAhead * 128) {
                    float4 wq[kAhead][kTok];
#pragma unroll
                    for (int i = 0; i < kAhead; ++i)
#pragma unroll
                        for (int t = 0; t < kTok; ++t) wq[i][t] = get(wr[t], k + i * 128);
#pragma unroll
                    for (int i = 0; i < kAhead; ++i) {
                        if (k + i * 128 < D) {
#pragma unroll
                            for (int t = 0; t < kTok; ++t) acc[t] = add(acc[t], wq[i][t], *reinterpret_cast<const float4*>(xr[t] + k + i * 128));
                        }
                    }
                }
            } else {
#pragma unroll 4
                for (int k = lane; k < D; k += 32)
#pragma unroll
                    for (int t = 0; t < kTok; ++t) acc[t] = fmaf(__ldg(wr[t] + k), xr[t][k], acc[t]);
            }
            const float z = lane_totals<8>(acc, lane) + bias;       // token t's sum in the lanes 4t .. 4t + 3
            const unsigned right = __ballot_sync(kFullMask, z >= 0.0f);
#pragma unroll
            for (int t = 0; t < kTok; ++t) n[t] = 2 * n[t] + (int)((right >> (t * 4)) & 1u);
        }
    }
}

// w2t: [n_leaves][l][O].  node_w, w1 and w2t are allocations whose size is rounded up to 16 bytes.  slots, cursor: as in
// k_block_forward.  lay: see BlockTilesLayout.
__global__ void __launch_bounds__(kBTThreads, 1)
k_block_tiles(const float* __restrict__ x, const float* __restrict__ node_w, const float* __restrict__ node_b, const float* __restrict__ w1,
              const float* __restrict__ b1, const float* __restrict__ w2t, const float* __restrict__ b2, float* __restrict__ y,
              int32_t* __restrict__ leaf_out, int32_t* __restrict__ leaf_out2, int32_t* lists, int32_t* cursor, int cap, int D, int O,
              int depth, int l, int act, int B, int n_leaves, const BlockTilesLayout lay, int* __restrict__ status)
{
    extern __shared__ __align__(16) float smem_bt[];
    float* hs = smem_bt + lay.hs_at;                        // [l][kBTTile]
    int* s_pre = reinterpret_cast<int*>(smem_bt + lay.pre_at);           // [n_leaves + 1] tiles before each leaf
    int* s_cnt = s_pre + n_leaves + 1;                      // [n_leaves] its tokens
    uint64_t* full = reinterpret_cast<uint64_t*>(smem_bt + lay.bar_at);
    uint64_t* rows_full = full + kBTMaxSlots;               // [kBTWarps] phase A: a warp's rows
    uint64_t* top_full = rows_full + kBTWarps;
    uint64_t* x_full = top_full + 1;
    __shared__ int s_wsum[kBTWarps];
    __shared__ int s_tok[2][kBTTile], s_leaf[2], s_rows[2];
    __shared__ int s_done[kBTMaxSlots], s_last;             // warps that are through with a slot
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool vec = (D & 3) == 0;
    float* top = smem_bt;                                   // phase A: seven node rows, then the warps' rows of x
    const int top_part = BlockTilesLayout::part(kBTTop * D);

    if (tid == 0) {
        for (int s = 0; s < kBTMaxSlots; ++s) {
            ptx::mbar_init(full + s, 1);
            s_done[s] = 0;
        }
        for (int w = 0; w < kBTWarps; ++w) ptx::mbar_init(rows_full + w, 1);
        ptx::mbar_init(top_full, 1);
        ptx::mbar_init(x_full, kBTWarps);
        ptx::fence_mbar_init();
        if (depth > 0) {                                    // parameters, not a predecessor's output
            const int rows = depth == 1 ? 1 : depth == 2 ? 3 : kBTTop;
            ptx::mbar_arrive_expect_tx(top_full, (uint32_t)((rows * D + 3) & ~3) * 4);
            bulk_floats(top, node_w, rows * D, true, top_full);
        }
    }
    pdl_trigger();
    __syncthreads();
    pdl_wait();
    bool timed_out = false;

    // ---- phase A
    {
        float* buf = smem_bt + top_part + warp * BlockTilesLayout::part(lay.tok * D);
        bool top_here = false;
        uint32_t phase = 0;
        const int n_groups = (B + lay.tok - 1) / lay.tok;
        for (int g = blockIdx.x + warp * gridDim.x; g < n_groups; g += gridDim.x * kBTWarps, phase ^= 1) {
            const int t0 = g * lay.tok, count = min(lay.tok, B - t0);
            const float* src = x + (int64_t)t0 * D;
            const int head = head_of(src), len = head + count * D;
            if (lane == 0) {
                // (the warp has read the rows of the round before: the sums are known)
                const uint32_t bytes = bulk_floats(buf, src, count * D, false, rows_full + warp);
                ptx::mbar_arrive_expect_tx(rows_full + warp, bytes);
            }
            if (lane < (len & 3)) buf[(len & ~3) + lane] = src[(len & ~3) + lane - head];
            if (!top_here && depth > 0 && !timed_out && !ptx::mbar_wait(top_full, 0)) timed_out = true;
            top_here = true;
            if (!timed_out && !ptx::mbar_wait(rows_full + warp, phase)) timed_out = true;
            __syncwarp();
            const float* row = buf + head;
            int leaf = 0;
            auto walk = [&](auto tokens) {
                constexpr int kTok = decltype(tokens)::value;
                const float* xr[kTok];
                int n[kTok];
#pragma unroll
                for (int t = 0; t < kTok; ++t) xr[t] = row + min(t, count - 1) * D;
                walk_staged<kTok>(xr, top, node_w, node_b, D, depth, vec, lane, n);
                leaf = n[0];
#pragma unroll
                for (int t = 1; t < kTok; ++t) leaf = lane == t ? n[t] : leaf;
            };
            if (lay.tok == 1) walk(std::integral_constant<int, 1>{});
            else if (lay.tok == 2) walk(std::integral_constant<int, 2>{});
            else if (lay.tok == 3) walk(std::integral_constant<int, 3>{});
            else walk(std::integral_constant<int, 4>{});
            if (lane < count) {
                const int tok = t0 + lane;
                if (leaf_out) leaf_out[tok] = leaf;
                if (leaf_out2) leaf_out2[tok] = leaf;
                lists[(int64_t)leaf * cap + atomicAdd(cursor + leaf, 1)] = tok;
            }
            if (!vec) ptx::fence_proxy_async();             // values stored one by one, before a copy comes to lie over them
            __syncwarp();
        }
        // the copy of the nodes has landed before phase B writes over them (a warp without tokens has not looked)
        if (!top_here && depth > 0 && !timed_out && !ptx::mbar_wait(top_full, 0)) timed_out = true;
    }
    const bool all_filed = grid_barrier(cursor + n_leaves + 1);
    if (!all_filed && tid == 0) atomicExch(status, kDevTimeout);

    // ---- tiles of every leaf and their running sum, by every CTA for itself
    tiles_before_bins([&](int j) { return s_cnt[j] = __ldcg(cursor + j); }, n_leaves, lay.tile_rows, s_pre, s_wsum, kBTThreads);
    const int n_tiles = all_filed ? s_pre[n_leaves] : 0;

    // ---- phase B
    // A tile's blocks (W1, then W2) are numbered through all tiles of the CTA; block k goes into slot k % slots once the last warp
    // is through with block k - slots: that warp sends for it.  The rows of the next tile follow once the hidden layer has read this one's, two
    // per warp (a warp sends one request per 70 cycles: 32 from one warp were 1.2 us in which the others waited).
    float* xs = smem_bt;
    float* ring = smem_bt + lay.tile_rows * lay.x_pitch;
    const int blocks1 = (l + lay.w1_units - 1) / lay.w1_units, blocks = blocks1 + (l + lay.w2_units - 1) / lay.w2_units;
    constexpr int kPerWarp = kBTTile / kBTWarps;            // rows of a tile that each warp sends for
    static_assert(kBTTile == 32 && kPerWarp == 2 && kBTMaxSlots <= kBTWarps, "a lane per row");
    auto send_block = [&](int k) {                          // one lane
        const int tile = blockIdx.x + k / blocks * gridDim.x, j = k % blocks, slot = k % lay.slots;
        if (tile >= n_tiles) return;
        const int64_t unit0 = (int64_t)bin_of_tile(s_pre, n_leaves, tile) * l;
        const bool first = j < blocks1;
        const int u = first ? j * lay.w1_units : (j - blocks1) * lay.w2_units;
        const float* src = first ? w1 + (unit0 + u) * D : w2t + (unit0 + u) * O;
        const int n = first ? min(lay.w1_units, l - u) * D : min(lay.w2_units, l - u) * O;
        ptx::mbar_arrive_expect_tx(full + slot, (uint32_t)((head_of(src) + n + 3) & ~3) * 4);
        bulk_floats(ring + slot * lay.slot, src, n, true, full + slot);
    };
    auto tile_token = [&](int tile, int& leaf, int& rows) { // this lane's token of a tile (its last one past the end)
        leaf = bin_of_tile(s_pre, n_leaves, tile);
        const int first = (tile - s_pre[leaf]) * lay.tile_rows;
        rows = min(lay.tile_rows, s_cnt[leaf] - first);
        return __ldcg(lists + (int64_t)leaf * cap + first + min(lane, rows - 1));
    };
    auto send_rows = [&](int it, int leaf, int rows, int tok) {          // all warps
        if (warp == 0) {
            s_tok[it & 1][lane] = tok;
            if (lane == 0) {
                s_leaf[it & 1] = leaf;
                s_rows[it & 1] = rows;
            }
        }
        if (!vec) ptx::fence_proxy_async();                 // (as in phase A)
        uint32_t bytes = 0;
        if (lane / kPerWarp == warp && lane < rows) {
            const float* src = x + (int64_t)tok * D;
            float* dst = xs + lane * lay.x_pitch;
            bytes = bulk_floats(dst, src, D, false, x_full);
            const int head = head_of(src), len = head + D;
            for (int i = len & ~3; i < len; ++i) dst[i] = src[i - head];
        }
#pragma unroll
        for (int o = 1; o < kPerWarp; o <<= 1) bytes += __shfl_xor_sync(kFullMask, bytes, o);
        __syncwarp();
        if (lane == warp * kPerWarp) ptx::mbar_arrive_expect_tx(x_full, bytes);
    };
    auto last_one = [&](int* count) {                       // one lane of every warp: is it the last?
        int before;
        asm volatile("atom.acq_rel.cta.shared::cta.add.s32 %0, [%1], 1;" : "=r"(before) : "r"(ptx::smem_addr(count)) : "memory");
        if (before != kBTWarps - 1) return false;
        *count = 0;
        return true;
    };
    if (blockIdx.x < n_tiles) {
        int leaf, rows;
        const int tok = tile_token(blockIdx.x, leaf, rows);
        send_rows(0, leaf, rows, tok);
        if (lane == 0 && warp < lay.slots) send_block(warp);
    }
    // threads per group of outputs, outputs per thread, tokens per thread in the output layer
    int og = 32;
    while (og < 256 && og < O) og <<= 1;
    const int per = (O + og - 1) / og, groups = kBTThreads / og;
    const int tpt = max(2, lay.tile_rows / groups);         // 16, 8, 4 or 2
    int slot = 0, it = 0, block = 0;
    uint32_t phase = 0;
    auto next_slot = [&]() {
        __syncwarp();
        if (lane == 0 && last_one(s_done + slot)) send_block(block + lay.slots);
        ++block;
        if (++slot == lay.slots) { slot = 0; phase ^= 1; }
    };
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++it) {
        int next_leaf = 0, next_rows = 0, next_tok = 0;
        if (tile + (int)gridDim.x < n_tiles) next_tok = tile_token(tile + gridDim.x, next_leaf, next_rows);
        if (!timed_out && !ptx::mbar_wait(x_full, (uint32_t)it & 1)) timed_out = true;
        const int* toks = s_tok[it & 1];
        const int leaf = s_leaf[it & 1], rows = s_rows[it & 1];
        // hidden layer: blocks of 4 tokens x 8 units, dealt to the warps in turn
        const int tb = (rows + 3) / 4;
        int dealt = 0;
        for (int ub = 0; ub < l; ub += lay.w1_units) {
            const int units = min(lay.w1_units, l - ub), tasks = tb * ((units + 7) / 8);
            if (!timed_out && !ptx::mbar_wait(full + slot, phase)) timed_out = true;
            const float* w = ring + slot * lay.slot + head_of(w1 + ((int64_t)leaf * l + ub) * D);
            for (int task = (warp - dealt) & (kBTWarps - 1); task < tasks; task += kBTWarps) {
                const int t0 = (task % tb) * 4, u0 = (task / tb) * 8;
                const float* xr[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int r = min(t0 + t, rows - 1);
                    xr[t] = xs + r * lay.x_pitch + (vec ? 0 : head_of(x + (int64_t)toks[r] * D));
                }
                auto block_of = [&](auto width) {
                    constexpr int NW = decltype(width)::value;
                    const float* wr[NW];
#pragma unroll
                    for (int u = 0; u < NW; ++u) wr[u] = w + min(u0 + u, units - 1) * D;
                    constexpr int kLanes = 32 / (4 * NW);                // lanes that end with the same sum
                    const int mine = lane / kLanes, u = u0 + mine % NW;
                    const float bias = __ldg(b1 + (int64_t)leaf * l + ub + min(u, units - 1));
                    float acc[4 * NW];
                    shared_dots<4, NW>(xr, wr, D, vec, lane, acc);
                    const float sum = lane_totals<4 * NW>(acc, lane) + bias;
                    if (u < units && lane % kLanes == 0) hs[(ub + u) * kBTTile + t0 + mine / NW] = activate(act, sum);
                };
                if (units - u0 > 4) block_of(std::integral_constant<int, 8>{});
                else block_of(std::integral_constant<int, 4>{});
            }
            dealt += tasks;
            next_slot();
        }
        float bias2[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) bias2[i] = __ldg(b2 + (int64_t)leaf * O + min(tid % og + i * og, O - 1));
        __syncthreads();                                    // H is complete, x is free
        if (next_rows > 0) send_rows(it + 1, next_leaf, next_rows, next_tok);
        // output layer
        auto outputs = [&](auto outs, auto tokens) {
            constexpr int NO = decltype(outs)::value, NT = decltype(tokens)::value;
            const int o0 = tid % og, ts = (tid / og) * NT;
            float acc[NO][NT];
#pragma unroll
            for (int i = 0; i < NO; ++i) {
#pragma unroll
                for (int t = 0; t < NT; ++t) acc[i][t] = bias2[i];
            }
            const bool busy = ts < rows;
            for (int ub = 0; ub < l; ub += lay.w2_units) {
                const int units = min(lay.w2_units, l - ub);
                if (!timed_out && !ptx::mbar_wait(full + slot, phase)) timed_out = true;
                const float* w = ring + slot * lay.slot + head_of(w2t + ((int64_t)leaf * l + ub) * O);
                if (busy) {
#pragma unroll 2
                    for (int u = 0; u < units; ++u) {
                        float wv[NO];
#pragma unroll
                        for (int i = 0; i < NO; ++i) wv[i] = w[u * O + min(o0 + i * og, O - 1)];
                        const float* hu = hs + (ub + u) * kBTTile + ts;
                        constexpr int VH = NT >= 4 ? 4 : 2;
#pragma unroll
                        for (int t = 0; t < NT; t += VH) {
                            float hv[VH];
                            if constexpr (VH == 4) {
                                const float4 q = *reinterpret_cast<const float4*>(hu + t);
                                hv[0] = q.x; hv[1] = q.y; hv[2] = q.z; hv[3] = q.w;
                            } else {
                                const float2 q = *reinterpret_cast<const float2*>(hu + t);
                                hv[0] = q.x; hv[1] = q.y;
                            }
#pragma unroll
                            for (int j = 0; j < VH; ++j)
#pragma unroll
                                for (int i = 0; i < NO; ++i) acc[i][t + j] = fmaf(wv[i], hv[j], acc[i][t + j]);
                        }
                    }
                }
                next_slot();
            }
            if (busy) {
#pragma unroll
                for (int t = 0; t < NT; ++t)
                    if (ts + t < rows) {
                        float* yt = y + (int64_t)toks[ts + t] * O;
#pragma unroll
                        for (int i = 0; i < NO; ++i)
                            if (o0 + i * og < O) yt[o0 + i * og] = acc[i][t];
                    }
            }
        };
        auto with_tokens = [&](auto outs) {
            if (tpt == 16) outputs(outs, std::integral_constant<int, 16>{});
            else if (tpt == 8) outputs(outs, std::integral_constant<int, 8>{});
            else if (tpt == 4) outputs(outs, std::integral_constant<int, 4>{});
            else outputs(outs, std::integral_constant<int, 2>{});
        };
        if (per == 1) with_tokens(std::integral_constant<int, 1>{});
        else if (per == 2) with_tokens(std::integral_constant<int, 2>{});
        else if (per == 3) with_tokens(std::integral_constant<int, 3>{});
        else with_tokens(std::integral_constant<int, 4>{});
        __syncthreads();                                    // H may be written again
    }
    if (timed_out) {
        if (lane == 0) atomicExch(status, kDevTimeout);
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);   // let copies still in flight finish before exit
    }

    // the last CTA to finish clears the counts for the next call
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(cursor + n_leaves, 1) == (int)gridDim.x - 1 ? 1 : 0;
    }
    __syncthreads();
    if (s_last)
        for (int j = tid; j <= n_leaves + 1; j += kBTThreads) cursor[j] = 0;
}

// W2 transposed: [n_leaves][O][l] -> [n_leaves][l][O].
__global__ void k_pack_w2_columns(const float* __restrict__ w2, float* __restrict__ w2t, int64_t n_leaves, int l, int O)
{
    const int64_t total = n_leaves * l * O;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int o = (int)(i % O), u = (int)((i / O) % l);
        w2t[i] = w2[(i / ((int64_t)O * l) * O + o) * l + u];
    }
}

}  // namespace fff
