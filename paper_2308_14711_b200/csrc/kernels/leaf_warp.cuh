// Grouped leaf evaluation on CUDA cores with un-permuting write-back.
//
// Algorithm 1, FORWARD_I, leaf branch: the token returns N_{d,j}(x), the
// <D, l, O> feedforward network of its leaf:  y = W2_j act(W1_j x + b1_j) + b2_j.
//
// One warp evaluates one token.  Warps walk the tokens in bucket order
// (perm), so the warps of a CTA mostly work on the same leaf and share its
// weights through L1/L2.  The row of y is written straight to the token's
// original position, which is the un-permute step.
//
// The kernel can also finish the descent first (tail_levels > 0): the warp walks the last levels of the tree
// from the position the staged descent reached, exactly as k_descent_warp would (same dot product, same
// comparison), records the leaf index and goes on with that leaf.  With a token per warp and no bucketing in
// between, this saves a kernel and one pass over x.
//
// General path: any D, l, O, both element types, float32 accumulation.  It is
// the path for float32 layers, for very thin leaves and for buckets of a few
// tokens, where the work is a gather of weights rather than a contraction.
#pragma once

#include "common.cuh"

namespace fff {

constexpr int kLeafWarps = 8;
constexpr int kLeafHiddenUnroll = 4;

// Starts to bring the 128-byte lines of [p, p + bytes) into L2, at most four per lane.
__device__ __forceinline__ void prefetch_lines(const void* p, int64_t bytes, int lane) {
    const char* c = reinterpret_cast<const char*>(p);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t off = ((int64_t)i * 32 + lane) * 128;
        if (off < bytes) asm volatile("prefetch.global.L2 [%0];" ::"l"(c + off));
    }
}

// N = 4, 8 or 16 bytes as one access (both addresses aligned to N).
template <int N>
__device__ __forceinline__ void copy_bytes(void* dst, const void* src) {
    static_assert(N == 4 || N == 8 || N == 16, "one access");
    if constexpr (N == 16) *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
    else if constexpr (N == 8) *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(src);
    else *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(src);
}

// Dynamic shared memory: kLeafWarps * l floats (hidden activations per warp).
// kTail: walk tail_levels levels of the descent first (a separate instantiation keeps the plain kernel lean).
// FORM: kLeafWide the general form; kLeafDense the same at six CTAs per SM; kLeafThin for leaves of one, two or four neurons with
// rows in 16-byte vectors, six CTAs per SM (35.5 -> 31.9 us on the layer named below; eight: 32.3) and the output weights sent for
// early.  The line is drawn in run_leaf (fff_api.cu).
enum : int { kLeafWide = 0, kLeafDense = 1, kLeafThin = 2 };
template <typename T, bool kTail, int FORM>
__global__ void __launch_bounds__(kLeafWarps * 32, FORM == kLeafWide ? 0 : 6)
k_leaf_warp(const T* __restrict__ x, const int32_t* __restrict__ leaf_idx, const int32_t* __restrict__ perm,
            const T* __restrict__ w1, const T* __restrict__ b1, const T* __restrict__ w2, const T* __restrict__ b2,
            T* __restrict__ y, int D, int O, int l, int act, int64_t B, bool vec,
            const T* __restrict__ node_w, const T* __restrict__ node_b, int tail_level0, int tail_levels,
            const int32_t* __restrict__ tail_pos, int32_t* __restrict__ leaf_out)
{
    extern __shared__ float s_h[];
    pdl_trigger();
    pdl_wait();
    constexpr int V = Elem<T>::kVec;
    constexpr int U = kLeafHiddenUnroll;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    float* h = s_h + (size_t)wib * l;
    const int64_t warp0 = (int64_t)blockIdx.x * kLeafWarps + wib;
    const int64_t nwarps = (int64_t)gridDim.x * kLeafWarps;

    for (int64_t i = warp0; i < B; i += nwarps) {
        const int64_t t = perm ? perm[i] : i;
        const T* xt = x + t * D;
        int64_t j;
        if (kTail) {
            // the walk starts at node N_{tail_level0, tail_pos[t]} (position 0 without tail_pos)
            int64_t n = tail_pos ? tail_pos[t] : 0;
            for (int m = tail_level0; m < tail_level0 + tail_levels; ++m) {
                const int64_t row = ((int64_t)1 << m) - 1 + n;
                const float logit = warp_dot<T>(node_w + row * D, xt, D, vec, lane) + Elem<T>::to_float(node_b[row]);
                n = 2 * n + (logit >= 0.0f ? 1 : 0);
            }
            j = n;
            if (lane == 0) leaf_out[t] = (int32_t)n;
        } else {
            j = leaf_idx[t];
        }
        const T* w1j = w1 + j * (int64_t)l * D;
        const T* b1j = b1 + j * (int64_t)l;
        // With about a token per leaf these weights come from DRAM: the output layer's lines are sent for now, so that they
        // arrive in L2 while the hidden layer is evaluated (15 levels, 768 columns, l = 1, 16 384 tokens: 36.8 -> 35.5 us).
        if constexpr (FORM == kLeafThin) {
            prefetch_lines(w2 + j * (int64_t)O * l, (int64_t)O * l * (int)sizeof(T), lane);
            prefetch_lines(b2 + j * (int64_t)O, (int64_t)O * (int)sizeof(T), lane);
        }

        // hidden layer: U neurons at a time share the loads of x
        for (int i0 = 0; i0 < l; i0 += U) {
            float acc[U];
#pragma unroll
            for (int u = 0; u < U; ++u) acc[u] = 0.0f;
            if (vec) {
                for (int k = lane * V; k < D; k += 32 * V) {
                    float fx[V];
                    Elem<T>::load_vec(xt + k, fx);
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (i0 + u < l) {
                            float fw[V];
                            Elem<T>::load_vec(w1j + (int64_t)(i0 + u) * D + k, fw);
#pragma unroll
                            for (int e = 0; e < V; ++e) acc[u] = fmaf(fw[e], fx[e], acc[u]);
                        }
                    }
                }
            } else {
                for (int k = lane; k < D; k += 32) {
                    const float fx = Elem<T>::to_float(xt[k]);
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (i0 + u < l) acc[u] = fmaf(Elem<T>::to_float(w1j[(int64_t)(i0 + u) * D + k]), fx, acc[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float s = warp_sum(acc[u]);
                if (lane == 0 && i0 + u < l) h[i0 + u] = activate(act, s + Elem<T>::to_float(b1j[i0 + u]));
            }
        }
        __syncwarp();

        // output layer.  Thin leaves (l = 1, 2 or 4): a 16-byte vector of W2 holds the rows of kVec / l consecutive outputs,
        // which one lane evaluates and stores together (with one output per lane and element-wise loads the output layer
        // of a leaf of two neurons took as long as its walk through the tree: 256 columns, 2016 tokens 26 us, now 13).
        // Otherwise one output neuron per lane, four rows in flight.
        const T* w2j = w2 + j * (int64_t)O * l;
        const T* b2j = b2 + j * (int64_t)O;
        T* yt = y + t * O;
        auto thin = [&](auto width) {
            constexpr int W = decltype(width)::value, N = V / W;       // outputs per vector
            float hv[W];
#pragma unroll
            for (int q = 0; q < W; ++q) hv[q] = h[q];
#pragma unroll 4
            for (int o = lane * N; o < O; o += 32 * N) {
                float fw[V];
                Elem<T>::load_vec(w2j + (int64_t)o * W, fw);
                alignas(16) T bias[N];
                alignas(16) T out[N];
                copy_bytes<N * (int)sizeof(T)>(bias, b2j + o);
#pragma unroll
                for (int e = 0; e < N; ++e) {
                    float acc = Elem<T>::to_float(bias[e]);
#pragma unroll
                    for (int q = 0; q < W; ++q) acc = fmaf(fw[e * W + q], hv[q], acc);
                    out[e] = Elem<T>::from_float(acc);
                }
                copy_bytes<N * (int)sizeof(T)>(yt + o, out);
            }
        };
        if (FORM == kLeafThin && l == 1) {
            thin(std::integral_constant<int, 1>{});
        } else if (FORM == kLeafThin && l == 2) {
            thin(std::integral_constant<int, 2>{});
        } else if (FORM == kLeafThin && l == 4) {
            thin(std::integral_constant<int, 4>{});
        } else if (FORM != kLeafThin && l == 1 && vec && O % V == 0) {
            const float h0 = h[0];
            for (int o = lane * V; o < O; o += 32 * V) {
                float fw[V], fb[V];
                Elem<T>::load_vec(w2j + o, fw);
                Elem<T>::load_vec(b2j + o, fb);
                alignas(16) T out[V];
#pragma unroll
                for (int e = 0; e < V; ++e) out[e] = Elem<T>::from_float(fmaf(fw[e], h0, fb[e]));
                *reinterpret_cast<uint4*>(yt + o) = *reinterpret_cast<const uint4*>(out);
            }
        } else {
#pragma unroll 4
            for (int o = lane; o < O; o += 32) {
                const T* row = w2j + (int64_t)o * l;
                float acc = Elem<T>::to_float(b2j[o]);
                for (int q = 0; q < l; ++q) acc = fmaf(Elem<T>::to_float(row[q]), h[q], acc);
                yt[o] = Elem<T>::from_float(acc);
            }
        }
        __syncwarp();
    }
}

}  // namespace fff
