// Whole forward pass of a few tokens in one launch: one CTA walks one token down the tree and evaluates its leaf.
//
// Algorithm 1, FORWARD_I, both branches, for batches so small that nothing can be shared between tokens and the time is
// a chain of memory latencies: launches, the dependent levels of the walk, the two layers of the leaf.  What shortens
// the chain:
//   * three levels per step: the seven nodes of the subtree below the current node are evaluated at once, one warp per
//     node, so that a step costs one round trip for three decisions (2.3 times the weight rows of the plain walk);
//   * all loads of a warp's rows are issued before the first multiply-add;
//   * the leaf's output weights are on their way to shared memory while its hidden layer is evaluated.
// 768 -> 768, 2^8 leaves of 12, bf16: see use_token_block in fff_api.cu for the batches it is taken for and the times.
//
// float32 accumulation, any D, l, O, both element types.
#pragma once

#include "common.cuh"
#include "ptx.cuh"

namespace fff {

constexpr int kTBWarps = 8;
constexpr int kTBThreads = kTBWarps * 32;
constexpr int kTBLevels = 3;                               // levels per step of the walk: 2^3 - 1 nodes, one per warp
constexpr int kTBW2Bytes = 32 * 1024;                      // output weights staged at a time

// Shared memory: the token row, the hidden activations, the staged output weights.
struct TokenBlockLayout {
    int D, l, esize;
    __host__ __device__ size_t x_bytes() const { return ((size_t)D * esize + 15) & ~(size_t)15; }
    __host__ __device__ size_t h_bytes() const { return ((size_t)l * 4 + 15) & ~(size_t)15; }
    __host__ __device__ size_t total() const { return x_bytes() + h_bytes() + kTBW2Bytes; }
};

// Dot products of N weight rows (nullptr = none) with the token row in shared memory, by one warp; every lane returns the
// sums.  vec: rows start on 16-byte boundaries and D % kVec == 0.
template <typename T> constexpr int kTBAhead = sizeof(T) == 2 ? 4 : 8;      // vectors of a row in flight: 1024 columns
template <typename T, int N>
__device__ __forceinline__ void token_dots(const T* const (&rows)[N], const T* __restrict__ xs, int D, bool vec, int lane, float (&out)[N])
{
    constexpr int V = Elem<T>::kVec;
    constexpr int U = kTBAhead<T>;
#pragma unroll
    for (int n = 0; n < N; ++n) out[n] = 0.0f;
    if (vec) {
        for (int k0 = lane * V; k0 < D; k0 += 32 * V * U) {
            uint4 w[N][U];
#pragma unroll
            for (int n = 0; n < N; ++n)
#pragma unroll
                for (int u = 0; u < U; ++u)
                    w[n][u] = rows[n] && k0 + u * 32 * V < D ? __ldg(reinterpret_cast<const uint4*>(rows[n] + k0 + u * 32 * V)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (k0 + u * 32 * V >= D) break;
                float xv[V];
                Elem<T>::unpack(*reinterpret_cast<const uint4*>(xs + k0 + u * 32 * V), xv);
#pragma unroll
                for (int n = 0; n < N; ++n) {
                    float wv[V];
                    Elem<T>::unpack(w[n][u], wv);
#pragma unroll
                    for (int e = 0; e < V; ++e) out[n] = fmaf(wv[e], xv[e], out[n]);
                }
            }
        }
    } else {
        constexpr int S = 8;
        for (int k0 = lane; k0 < D; k0 += 32 * S) {
            T w[N][S];
#pragma unroll
            for (int n = 0; n < N; ++n)
#pragma unroll
                for (int u = 0; u < S; ++u)
                    if (rows[n] && k0 + u * 32 < D) w[n][u] = rows[n][k0 + u * 32];
#pragma unroll
            for (int u = 0; u < S; ++u) {
                if (k0 + u * 32 >= D) break;
                const float xv = Elem<T>::to_float(xs[k0 + u * 32]);
#pragma unroll
                for (int n = 0; n < N; ++n)
                    if (rows[n]) out[n] = fmaf(Elem<T>::to_float(w[n][u]), xv, out[n]);
            }
        }
    }
#pragma unroll
    for (int n = 0; n < N; ++n) out[n] = warp_sum(out[n]);
}

// leaf_out / leaf_out2 (optional): leaf of every token.
template <typename T>
__global__ void __launch_bounds__(kTBThreads, sizeof(T) == 2 ? 4 : 2)
k_token_block(const T* __restrict__ x, const T* __restrict__ node_w, const T* __restrict__ node_b, const T* __restrict__ w1,
              const T* __restrict__ b1, const T* __restrict__ w2, const T* __restrict__ b2, T* __restrict__ y,
              int32_t* __restrict__ leaf_out, int32_t* __restrict__ leaf_out2, int D, int O, int depth, int l, int act, int B, bool vec)
{
    extern __shared__ __align__(16) unsigned char smem_tb[];
    const TokenBlockLayout L{D, l, (int)sizeof(T)};
    T* xs = reinterpret_cast<T*>(smem_tb);
    float* h = reinterpret_cast<float*>(smem_tb + L.x_bytes());
    unsigned char* w2s = smem_tb + L.x_bytes() + L.h_bytes();
    __shared__ float s_logit[2][8];
    constexpr int V = Elem<T>::kVec;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // rows of W2 staged at a time: whole 16-byte groups, none if the leaves' matrices are not 16-byte aligned
    const int row_bytes = l * (int)sizeof(T);
    const int stage_rows = ((int64_t)O * row_bytes) % 16 == 0 ? (kTBW2Bytes / row_bytes) & ~15 : 0;

    // The first step's nodes are the same for every token, and parameters: their rows are sent for before the kernel waits for its
    // predecessor, and arrive while x does: one image of 768 columns 8.6 -> 7.9 us, 102 float32 tokens of 832 7.9 -> 7.35.  Rows of up to the
    // 1024 columns that stay in registers.
    constexpr int U = kTBAhead<T>;
    const bool ahead = vec && D <= 32 * V * U, has_top = ahead && warp < (1 << min(kTBLevels, depth)) - 1;
    uint4 top_row[U];
    float top_bias = 0.0f;
    if (has_top) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = (u * 32 + lane) * V;
            top_row[u] = k < D ? __ldg(reinterpret_cast<const uint4*>(node_w + (int64_t)warp * D + k)) : make_uint4(0u, 0u, 0u, 0u);
        }
        top_bias = Elem<T>::to_float(node_b[warp]);
    }
    pdl_trigger();
    pdl_wait();
    const int t = blockIdx.x;                           // (a CTA per token)
    const T* xt = x + (int64_t)t * D;
    if (vec) {
        for (int i = tid; i < D / V; i += kTBThreads) reinterpret_cast<uint4*>(xs)[i] = __ldg(reinterpret_cast<const uint4*>(xt) + i);
    } else {
        for (int i = tid; i < D; i += kTBThreads) xs[i] = xt[i];
    }
    __syncthreads();

    // ---- the walk
    int64_t n = 0;
    if (has_top) {                                      // (summed as in token_dots)
        float sum = 0.0f;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int k = (u * 32 + lane) * V;
            if (k >= D) break;
            float xv[V], wv[V];
            Elem<T>::unpack(*reinterpret_cast<const uint4*>(xs + k), xv);
            Elem<T>::unpack(top_row[u], wv);
#pragma unroll
            for (int e = 0; e < V; ++e) sum = fmaf(wv[e], xv[e], sum);
        }
        sum = warp_sum(sum);
        if (lane == 0) s_logit[0][warp] = sum + top_bias;
    }
    for (int m = 0, buf = 0; m < depth; m += kTBLevels, buf ^= 1) {
        const int r = min(kTBLevels, depth - m);
        if (warp < (1 << r) - 1 && !(m == 0 && ahead)) {
            const int lev = 31 - __clz(warp + 1);
            const int64_t row = (((int64_t)1 << (m + lev)) - 1) + (n << lev) + (warp + 1 - (1 << lev));
            const T* rows[1] = {node_w + row * D};
            const float bias = Elem<T>::to_float(node_b[row]);
            float sum[1];
            token_dots<T, 1>(rows, xs, D, vec, lane, sum);
            if (lane == 0) s_logit[buf][warp] = sum[0] + bias;
        }
        __syncthreads();
        int p = 0;
        for (int i = 0; i < r; ++i) {
            const int right = s_logit[buf][p] >= 0.0f ? 1 : 0;
            p = 2 * p + 1 + right;
            n = 2 * n + right;
        }
    }
    if (tid == 0) {
        if (leaf_out) leaf_out[t] = (int32_t)n;
        if (leaf_out2) leaf_out2[t] = (int32_t)n;
    }

    // ---- the leaf: its output weights start to arrive, then the hidden layer, two units per warp at a time
    const T* w2j = w2 + n * (int64_t)O * l;
    const T* b2j = b2 + n * (int64_t)O;
    auto stage = [&](int r0) {
        const int bytes = min(stage_rows, O - r0) * row_bytes;          // (the last group may be cut: O * row_bytes is whole groups)
        const unsigned char* src = reinterpret_cast<const unsigned char*>(w2j) + (int64_t)r0 * row_bytes;
        for (int i = tid * 16; i < bytes; i += kTBThreads * 16) ptx::cp_async16(w2s + i, src + i);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (stage_rows > 0) stage(0);
    float b2r[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) b2r[i] = tid + i * kTBThreads < O ? Elem<T>::to_float(b2j[tid + i * kTBThreads]) : 0.0f;
    const T* w1j = w1 + n * (int64_t)l * D;
    for (int i0 = warp; i0 < l; i0 += 2 * kTBWarps) {
        const int i1 = i0 + kTBWarps;
        const T* rows[2] = {w1j + (int64_t)i0 * D, i1 < l ? w1j + (int64_t)i1 * D : nullptr};
        const float bias0 = Elem<T>::to_float(b1[n * l + i0]), bias1 = i1 < l ? Elem<T>::to_float(b1[n * l + i1]) : 0.0f;
        float sum[2];
        token_dots<T, 2>(rows, xs, D, vec, lane, sum);
        if (lane == 0) {
            h[i0] = activate(act, sum[0] + bias0);
            if (i1 < l) h[i1] = activate(act, sum[1] + bias1);
        }
    }

    // ---- output layer: one output neuron per thread
    T* yt = y + (int64_t)t * O;
    auto outputs = [&](int r0, int r1, const unsigned char* base) {      // rows r0 .. r1 - 1, row r0 at `base`
        for (int o = r0 + tid; o < r1; o += kTBThreads) {
            const int bi = (o - tid) / kTBThreads;
            float acc = (o - tid) % kTBThreads == 0 && bi < 4 ? (bi == 0 ? b2r[0] : bi == 1 ? b2r[1] : bi == 2 ? b2r[2] : b2r[3])
                                                              : Elem<T>::to_float(b2j[o]);
            const unsigned char* row = base + (int64_t)(o - r0) * row_bytes;
            int q = 0;
            if (row_bytes % 16 == 0 && (reinterpret_cast<uintptr_t>(base) & 15) == 0) {
                for (; q < l; q += V) {
                    float wv[V];
                    Elem<T>::unpack(*reinterpret_cast<const uint4*>(row + q * sizeof(T)), wv);
#pragma unroll
                    for (int e = 0; e < V; ++e) acc = fmaf(wv[e], h[q + e], acc);
                }
            } else if (row_bytes % 8 == 0 && (reinterpret_cast<uintptr_t>(base) & 7) == 0) {
                for (; q < l; q += V / 2) {
                    const uint2 raw = *reinterpret_cast<const uint2*>(row + q * sizeof(T));
                    float wv[V];
                    Elem<T>::unpack(make_uint4(raw.x, raw.y, 0u, 0u), wv);
#pragma unroll
                    for (int e = 0; e < V / 2; ++e) acc = fmaf(wv[e], h[q + e], acc);
                }
            } else {
                for (; q < l; ++q) acc = fmaf(Elem<T>::to_float(reinterpret_cast<const T*>(row)[q]), h[q], acc);
            }
            yt[o] = Elem<T>::from_float(acc);
        }
    };
    if (stage_rows > 0) {
        for (int r0 = 0; r0 < O; r0 += stage_rows) {
            if (r0 > 0) {
                __syncthreads();
                stage(r0);
            }
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            outputs(r0, min(O, r0 + stage_rows), w2s);
        }
    } else {
        __syncthreads();
        outputs(0, O, reinterpret_cast<const unsigned char*>(w2j));
    }
}

}  // namespace fff
