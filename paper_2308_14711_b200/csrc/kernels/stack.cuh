// Glue between the FFF layers of a stack (Section "Fast feedforward layers as building blocks": an FFF layer in
// place of each feedforward layer of a transformer, i.e. behind a layer normalisation and inside a residual
// connection).  Per token, for block k:
//     x_k   = x_{k-1} + y_{k-1}                      (residual of the previous block; skipped for k = 0)
//     z_k   = (x_k - mean) / sqrt(var + eps) * gamma + beta         (mean, population variance over the D features)
// and z_k is what the block's FFF layer reads.  Both are stored in the stack's element type; the statistics are
// taken in float32 from the stored x_k (two passes: mean, then squared deviations).
// One warp per token.  Rows of up to kStackVecs 16-byte vectors per lane (1024 columns in bf16) stay in registers between the
// sum, the statistics and the normalised row, with all loads of a row issued at once (12 608 rows of 768: 20 -> 14 us;
// read again from L1 / L2 for each of them, as longer and unaligned rows still are, a row was a chain of four round trips).
// These are plain element-wise passes bound by HBM bandwidth: 1-2 reads and 1-2 writes of a [B, D] matrix.
#pragma once

#include "common.cuh"

namespace fff {

constexpr int kStackWarps = 8;
template <typename T> constexpr int kStackVecs = 32 / Elem<T>::kVec;       // 32 values of a row per lane

template <typename T>
__global__ void __launch_bounds__(kStackWarps * 32)
k_stack_glue_rows(const T* __restrict__ x_prev, const T* __restrict__ y_prev, T* __restrict__ x_out, T* __restrict__ z,
                  const T* __restrict__ gamma, const T* __restrict__ beta, float eps, int D, int64_t B)
{
    pdl_trigger();
    pdl_wait();
    constexpr int V = Elem<T>::kVec, NV = kStackVecs<T>;
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (int64_t)blockIdx.x * kStackWarps + (threadIdx.x >> 5), nwarps = (int64_t)gridDim.x * kStackWarps;
    for (int64_t t = warp0; t < B; t += nwarps) {
        uint4 a[NV], b[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int k = (i * 32 + lane) * V;
            a[i] = b[i] = make_uint4(0u, 0u, 0u, 0u);
            if (k < D) {
                a[i] = *reinterpret_cast<const uint4*>(x_prev + t * D + k);
                if (y_prev) b[i] = *reinterpret_cast<const uint4*>(y_prev + t * D + k);
            }
        }
        float v[NV][V];
        float sum = 0.0f;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int k = (i * 32 + lane) * V;
            Elem<T>::unpack(a[i], v[i]);
            if (y_prev) {
                float w[V];
                Elem<T>::unpack(b[i], w);
                __align__(16) T r[V];
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    r[e] = Elem<T>::from_float(v[i][e] + w[e]);
                    v[i][e] = Elem<T>::to_float(r[e]);             // the statistics are those of the stored row
                }
                if (k < D) *reinterpret_cast<uint4*>(x_out + t * D + k) = *reinterpret_cast<const uint4*>(r);
            }
#pragma unroll
            for (int e = 0; e < V; ++e) sum += v[i][e];            // (vectors past the row are zero)
        }
        if (!z) continue;
        const float mean = warp_sum(sum) / (float)D;
        float sq = 0.0f;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            if ((i * 32 + lane) * V >= D) continue;
#pragma unroll
            for (int e = 0; e < V; ++e) {
                const float d = v[i][e] - mean;
                sq = fmaf(d, d, sq);
            }
        }
        const float rstd = 1.0f / sqrtf(warp_sum(sq) / (float)D + eps);
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int k = (i * 32 + lane) * V;
            if (k >= D) continue;
            float g[V], bt[V];
            if (gamma) Elem<T>::load_vec(gamma + k, g);
            if (beta) Elem<T>::load_vec(beta + k, bt);
            __align__(16) T out[V];
#pragma unroll
            for (int e = 0; e < V; ++e) {
                float q = (v[i][e] - mean) * rstd;
                if (gamma) q *= g[e];
                if (beta) q += bt[e];
                out[e] = Elem<T>::from_float(q);
            }
            *reinterpret_cast<uint4*>(z + t * D + k) = *reinterpret_cast<const uint4*>(out);
        }
    }
}

// x_out (optional, needs y_prev) = x_prev + y_prev;  z (optional) = LayerNorm(x_out or x_prev).
template <typename T>
__global__ void __launch_bounds__(kStackWarps * 32)
k_stack_glue(const T* __restrict__ x_prev, const T* __restrict__ y_prev, T* x_out, T* __restrict__ z,
             const T* __restrict__ gamma, const T* __restrict__ beta, float eps, int D, int64_t B, bool vec)
{
    pdl_trigger();
    pdl_wait();
    constexpr int V = Elem<T>::kVec;
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (int64_t)blockIdx.x * kStackWarps + (threadIdx.x >> 5), nwarps = (int64_t)gridDim.x * kStackWarps;
    for (int64_t t = warp0; t < B; t += nwarps) {
        const T* xp = x_prev + t * D;
        const T* cur = xp;
        float sum = 0.0f;
        if (y_prev) {
            const T* yp = y_prev + t * D;
            T* xo = x_out + t * D;
            if (vec) {
                for (int k = lane * V; k < D; k += 32 * V) {
                    float a[V], b[V];
                    Elem<T>::load_vec(xp + k, a);
                    Elem<T>::load_vec(yp + k, b);
                    __align__(16) T r[V];
#pragma unroll
                    for (int e = 0; e < V; ++e) {
                        r[e] = Elem<T>::from_float(a[e] + b[e]);
                        sum += Elem<T>::to_float(r[e]);
                    }
                    *reinterpret_cast<uint4*>(xo + k) = *reinterpret_cast<const uint4*>(r);
                }
            } else {
                for (int k = lane; k < D; k += 32) {
                    const T r = Elem<T>::from_float(Elem<T>::to_float(xp[k]) + Elem<T>::to_float(yp[k]));
                    xo[k] = r;
                    sum += Elem<T>::to_float(r);
                }
            }
            cur = xo;
        } else if (z) {
            if (vec) {
                for (int k = lane * V; k < D; k += 32 * V) {
                    float a[V];
                    Elem<T>::load_vec(xp + k, a);
#pragma unroll
                    for (int e = 0; e < V; ++e) sum += a[e];
                }
            } else {
                for (int k = lane; k < D; k += 32) sum += Elem<T>::to_float(xp[k]);
            }
        }
        if (!z) continue;
        __syncwarp();          // the row just written is read back below, in scalar mode by other lanes than wrote it
        const float mean = warp_sum(sum) / (float)D;
        // (plain loads: `cur` may be the row this warp has just written)
        float sq = 0.0f;
        if (vec) {
            for (int k = lane * V; k < D; k += 32 * V) {
                const uint4 raw = *reinterpret_cast<const uint4*>(cur + k);
                const T* r = reinterpret_cast<const T*>(&raw);
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    const float d = Elem<T>::to_float(r[e]) - mean;
                    sq = fmaf(d, d, sq);
                }
            }
        } else {
            for (int k = lane; k < D; k += 32) {
                const float d = Elem<T>::to_float(cur[k]) - mean;
                sq = fmaf(d, d, sq);
            }
        }
        const float rstd = 1.0f / sqrtf(warp_sum(sq) / (float)D + eps);
        T* zo = z + t * D;
        if (vec) {
            for (int k = lane * V; k < D; k += 32 * V) {
                const uint4 raw = *reinterpret_cast<const uint4*>(cur + k);
                const T* r = reinterpret_cast<const T*>(&raw);
                __align__(16) T out[V];
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    float v = (Elem<T>::to_float(r[e]) - mean) * rstd;
                    if (gamma) v *= Elem<T>::to_float(gamma[k + e]);
                    if (beta) v += Elem<T>::to_float(beta[k + e]);
                    out[e] = Elem<T>::from_float(v);
                }
                *reinterpret_cast<uint4*>(zo + k) = *reinterpret_cast<const uint4*>(out);
            }
        } else {
            for (int k = lane; k < D; k += 32) {
                float v = (Elem<T>::to_float(cur[k]) - mean) * rstd;
                if (gamma) v *= Elem<T>::to_float(gamma[k]);
                if (beta) v += Elem<T>::to_float(beta[k]);
                zo[k] = Elem<T>::from_float(v);
            }
        }
    }
}

}  // namespace fff
