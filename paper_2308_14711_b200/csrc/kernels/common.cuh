// Shared device helpers for the FFF inference kernels (sm_100a).
#pragma once

#include <type_traits>

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace fff {

constexpr unsigned kFullMask = 0xffffffffu;

enum : int { kActRelu = 0, kActGelu = 1, kActGeluTanh = 2, kActSilu = 3 };

// Values written to the per-handle device status word by kernels.
enum : int { kDevOk = 0, kDevTimeout = 1 };

// A tile of the grouped kernels: up to a fixed number of consecutive perm entries of one bin
// (a leaf, or a node position during a staged descent).
struct Tile {
    int bin, start, rows, pad;
};

// Programmatic dependent launch.  pdl_trigger: the next kernel in the stream may be scheduled from now
// on.  pdl_wait: block until the previous kernel in the stream has completed and its writes are
// visible; must precede the first read of anything that kernel produced.  Both are no-ops for a
// kernel that was launched the ordinary way.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename T> struct Elem;


template <> struct Elem<float> {
    static constexpr int kVec = 4;   // elements per 16-byte load
    __device__ __forceinline__ static float to_float(float v) { return v; }
    __device__ __forceinline__ static float from_float(float v) { return v; }
    __device__ __forceinline__ static void unpack(uint4 v, float (&out)[4]) {
        out[0] = __uint_as_float(v.x); out[1] = __uint_as_float(v.y); out[2] = __uint_as_float(v.z); out[3] = __uint_as_float(v.w);
    }
    __device__ __forceinline__ static void load_vec(const float* p, float (&out)[4]) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p));
        out[0] = v.x; out[1] = v.y; out[2] = v.z; out[3] = v.w;
    }
};

template <> struct Elem<__nv_bfloat16> {
    static constexpr int kVec = 8;
    __device__ __forceinline__ static float to_float(__nv_bfloat16 v) { return __bfloat162float(v); }
    __device__ __forceinline__ static __nv_bfloat16 from_float(float v) { return __float2bfloat16_rn(v); }
    __device__ __forceinline__ static void load_vec(const __nv_bfloat16* p, float (&out)[8]) {
        unpack(__ldg(reinterpret_cast<const uint4*>(p)), out);
    }
    __device__ __forceinline__ static void unpack(uint4 v, float (&out)[8]) {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            out[2 * i] = __uint_as_float(w[i] << 16);              // low half = even element
            out[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);  // high half = odd element
        }
    }
};

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFullMask, v, o);
    return v;
}

// The leaf's hidden activation (create-time parameter; the paper's Definition leaves it open): ReLU, GELU in
// the exact erf form, GELU in the published tanh form v/2 (1 + tanh(sqrt(2/pi) (v + 0.044715 v^3))), SiLU
// v sigmoid(v).  All four map 0 to 0, which the zero-padded hidden units of the tensor-core images rely on.
__device__ __forceinline__ float activate(int act, float v) {
    if (act == kActRelu) return fmaxf(v, 0.0f);
    if (act == kActGeluTanh) return 0.5f * v * (1.0f + tanhf(0.79788456080286535588f * (v + 0.044715f * v * v * v)));
    if (act == kActSilu) return v / (1.0f + expf(-v));
    return 0.5f * v * (1.0f + erff(v * 0.70710678118654752440f));
}

__device__ __forceinline__ float exp2_approx(float v) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float rcp_approx(float v) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float max_nan(float a, float b) {      // NaN if either is
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// GELU for results that are rounded to bf16 right away: v Phi(v) = max(v, 0) - |v| Q(|v|) with the normal tail
// Q = 1 - Phi evaluated as 2^P(|v|).  log2 Q is so nearly quadratic that a polynomial of degree 6 is enough: its
// coefficients are a least-squares fit on [0, 6], reweighted until the error of |v| Q is level, which leaves at most
// 5.1e-8 (7.6e-8 with float32 arithmetic; the formula 7.1.26 of Abramowitz & Stegun that stood here before: 2.1e-7).
// One exponential and no division.  |v| is cut off at 10, where Q < 2^-74.  kGeluP: coefficients in -|v|.
constexpr float kGeluCut = -10.0f;
constexpr float kGeluP0 = -0.9999930609869272f, kGeluP1 = 1.1512017022737409f, kGeluP2 = -0.45877097266965633f,
                kGeluP3 = 0.05341210482228353f, kGeluP4 = 0.008080716673348184f, kGeluP5 = 0.0007692196373495289f,
                kGeluP6 = 3.309279284094074e-05f;

// The activations for kernels whose result is rounded to bf16 right away.
__device__ __forceinline__ float activate_bf16(int act, float v) {
    if (act == kActRelu) return fmaxf(v, 0.0f);
    if (act == kActGeluTanh) {
        // v / 2 (1 + tanh u) = v / (1 + e^(-2u))
        const float m = -2.0f * 1.44269504088896340736f * 0.79788456080286535588f;
        return v * rcp_approx(1.0f + exp2_approx(v * fmaf(m * 0.044715f, v * v, m)));
    }
    if (act == kActSilu) return v * rcp_approx(1.0f + exp2_approx(-1.44269504088896340736f * fmaxf(v, -80.0f)));
    const float a = max_nan(-fabsf(v), kGeluCut);
    float p = fmaf(kGeluP6, a, kGeluP5);
    p = fmaf(p, a, kGeluP4);
    p = fmaf(p, a, kGeluP3);
    p = fmaf(p, a, kGeluP2);
    p = fmaf(p, a, kGeluP1);
    p = fmaf(p, a, kGeluP0);
    return fmaf(a, exp2_approx(p), fmaxf(v, 0.0f));
}

// Calls f(std::integral_constant<int, act>) with the activation as a compile-time constant.  Code that applies the
// activation to many values in an unrolled loop goes through this: with a run-time `act` every value carries the
// branches between the four forms, which keeps the values' dependency chains from overlapping.
template <class F>
__device__ __forceinline__ void with_activation(int act, F&& f) {
    switch (act) {
        case kActRelu: f(std::integral_constant<int, kActRelu>{}); break;
        case kActGeluTanh: f(std::integral_constant<int, kActGeluTanh>{}); break;
        case kActSilu: f(std::integral_constant<int, kActSilu>{}); break;
        default: f(std::integral_constant<int, kActGelu>{}); break;
    }
}

// Two float32 values in one 64-bit register: the packed instructions (add / mul / fma .f32x2) do both in one issue slot,
// each rounded as its scalar form.
struct f32x2 { unsigned long long r; };
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d.r) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ f32x2 pack2u(uint32_t lo, uint32_t hi) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d.r) : "r"(lo), "r"(hi));
    return d;
}
__device__ __forceinline__ void unpack2(f32x2 a, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.r)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d.r) : "l"(a.r), "l"(b.r));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d.r) : "l"(a.r), "l"(b.r));
    return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d.r) : "l"(a.r), "l"(b.r), "l"(c.r));
    return d;
}
__device__ __forceinline__ f32x2 splat2(float v) { return pack2(v, v); }
__device__ __forceinline__ uint32_t to_bf16x2(f32x2 a) {
    float lo, hi;
    unpack2(a, lo, hi);
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

// activate_bf16 for two values at once.
template <int kAct>
__device__ __forceinline__ f32x2 activate_bf16x2(f32x2 v) {
    float v0, v1;
    unpack2(v, v0, v1);
    if (kAct == kActGelu) {
        float p0, p1;
        const f32x2 a = pack2(max_nan(-fabsf(v0), kGeluCut), max_nan(-fabsf(v1), kGeluCut));
        f32x2 p = fma2(splat2(kGeluP6), a, splat2(kGeluP5));
        p = fma2(p, a, splat2(kGeluP4));
        p = fma2(p, a, splat2(kGeluP3));
        p = fma2(p, a, splat2(kGeluP2));
        p = fma2(p, a, splat2(kGeluP1));
        p = fma2(p, a, splat2(kGeluP0));
        unpack2(p, p0, p1);
        return fma2(a, pack2(exp2_approx(p0), exp2_approx(p1)), pack2(fmaxf(v0, 0.0f), fmaxf(v1, 0.0f)));
    }
    return pack2(activate_bf16(kAct, v0), activate_bf16(kAct, v1));
}

// One node's choice from its logit: right = sigmoid(z), left = 1 - right (each from the exponential of -|z|, so that the
// small one keeps its relative accuracy), h = the entropy -right ln right - left ln left = ln(1 + e^-|z|) + |z| min(right, left).
__device__ __forceinline__ void node_choice(float z, float& right, float& left, float& h) {
    const float a = fabsf(z);
    const float e = exp2_approx(a * -1.44269504088896340736f);
    const float d = 1.0f + e;
    const float big = rcp_approx(d), small = e * big;
    right = z >= 0.0f ? big : small;
    left = z >= 0.0f ? small : big;
    h = fmaf(fminf(a, 128.0f), small, __logf(d));          // (beyond 128 the small one is 0; keeps 0 x inf out)
}

// <a, b> over n elements, evaluated by one warp; every lane returns the sum.
// `vec` says both rows start on 16-byte boundaries and n is a multiple of kVec.
template <typename T>
__device__ __forceinline__ float warp_dot(const T* __restrict__ a, const T* __restrict__ b, int n, bool vec, int lane) {
    constexpr int V = Elem<T>::kVec;
    float acc = 0.0f;
    if (vec) {
        for (int k = lane * V; k < n; k += 32 * V) {
            float fa[V], fb[V];
            Elem<T>::load_vec(a + k, fa);
            Elem<T>::load_vec(b + k, fb);
#pragma unroll
            for (int i = 0; i < V; ++i) acc = fmaf(fa[i], fb[i], acc);
        }
    } else {
        for (int k = lane; k < n; k += 32) acc = fmaf(Elem<T>::to_float(a[k]), Elem<T>::to_float(b[k]), acc);
    }
    return warp_sum(acc);
}

// Tiles of up to tile_rows entries of every bin, from the bins' counts: s_pre[b] = tiles before bin b, s_pre[n_bins] = all of
// them.  By all `n_threads` threads of a CTA (thread i takes a run of bins); s_wsum: one int per warp.  `count(b)` reads a count.
// Index: int, or uint16_t where the caller knows that there are fewer than 65536 tiles.
template <class Index, class Count>
__device__ __forceinline__ void tiles_before_bins(Count&& count, int n_bins, int tile_rows, Index* s_pre, int* s_wsum, int n_threads) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (n_bins + n_threads - 1) / n_threads;
    const int b0 = min(tid * per, n_bins), b1 = min(b0 + per, n_bins);
    int mine = 0;
#pragma unroll 4
    for (int b = b0; b < b1; ++b) {
        const int t = (count(b) + tile_rows - 1) / tile_rows;
        s_pre[b] = (Index)t;
        mine += t;
    }
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(kFullMask, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) s_wsum[warp] = incl;
    __syncthreads();
    int run = incl - mine;
    for (int w = 0; w < warp; ++w) run += s_wsum[w];
    for (int b = b0; b < b1; ++b) {
        const int t = s_pre[b];
        s_pre[b] = (Index)run;
        run += t;
    }
    if (tid == n_threads - 1) s_pre[n_bins] = (Index)run;
    __syncthreads();
}

// The bin of tile `idx`: s_pre[bin] <= idx < s_pre[bin + 1].
template <class Index>
__device__ __forceinline__ int bin_of_tile(const Index* s_pre, int n_bins, int idx) {
    int lo = 0, hi = n_bins;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (s_pre[mid] <= idx) lo = mid;
        else hi = mid;
    }
    return lo;
}

}  // namespace fff
