// Device helpers: FP32 dot products and thresholded cosine decisions whose
// outcome is exact in FP64.
#pragma once

#include "ms_internal.cuh"

namespace ms {

// Sequential FP32 dot product, k = 0..Dp-1, one fused multiply-add per term.
template <int Dp>
__device__ __forceinline__ float dot_seq(const float* a, const float* b) {
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < Dp; ++k) s = fmaf(a[k], b[k], s);
    return s;
}

// Cosine (Eq. 1) in FP64 of two FP32 vectors of length n.
__device__ __forceinline__ double cos64(const float* a, const float* b, int n) {
    double ab = 0.0, aa = 0.0, bb = 0.0;
    for (int k = 0; k < n; ++k) {
        const double x = a[k], y = b[k];
        ab += x * y;
        aa += x * x;
        bb += y * y;
    }
    return ab / (sqrt(aa) * sqrt(bb));
}

// cos(a, b) >= thr for unit-length FP32 vectors: decided from the FP32 dot
// product when it clears thr by more than kEpsF32, else recomputed in FP64.
template <int Dp>
__device__ __forceinline__ bool cos_at_least(const float* a, const float* b, float thr_f, double thr) {
    const float s = dot_seq<Dp>(a, b);
    if (s >= thr_f + kEpsF32) return true;
    if (s < thr_f - kEpsF32) return false;
    return cos64(a, b, Dp) >= thr;
}

// Mean-shift update of one seed (Eq. 5 with the flat kernel) from its window
// sums (fixed point, 2^-36 units) and count, which are set back to zero: x <-
// normalise(sum), *conv when the FP64 step norm is below tol, *fail when the
// window is empty. True when the seed moves on.
// Every load comes before the first store: a store between two loads of the
// same array keeps them in order, and the 33 loads of a seed then cost a memory
// round trip each (18 us a launch instead of 4).
template <int Dp>
__device__ __forceinline__ bool finalize_seed(unsigned long long* a, float* x, uint8_t* state, int32_t* support,
                                              double tol, bool* conv, bool* fail) {
    long long sum[Dp + 1];
    float4 x4[Dp / 4];
#pragma unroll
    for (int k = 0; k <= Dp; ++k) sum[k] = (long long)a[k];
#pragma unroll
    for (int k = 0; k < Dp / 4; ++k) x4[k] = reinterpret_cast<const float4*>(x)[k];
    const long long cnt = sum[Dp];
    double y[Dp];
    double ss = 0.0;
#pragma unroll
    for (int k = 0; k < Dp; ++k) {
        y[k] = (double)sum[k] * (1.0 / 68719476736.0);
        ss += y[k] * y[k];
    }
#pragma unroll
    for (int k = 0; k <= Dp; ++k) a[k] = 0ull;
    if (cnt == 0) {
        *fail = true;
        *state = kFailed;
        return false;
    }
    const double inv = 1.0 / sqrt(ss);
    double dd = 0.0;
#pragma unroll
    for (int k = 0; k < Dp; k += 4) {
        float4 xn;
        xn.x = (float)(y[k] * inv);
        xn.y = (float)(y[k + 1] * inv);
        xn.z = (float)(y[k + 2] * inv);
        xn.w = (float)(y[k + 3] * inv);
        const float4 xo = x4[k / 4];
        const double d0 = (double)xn.x - (double)xo.x, d1 = (double)xn.y - (double)xo.y,
                     d2 = (double)xn.z - (double)xo.z, d3 = (double)xn.w - (double)xo.w;
        dd += d0 * d0;
        dd += d1 * d1;
        dd += d2 * d2;
        dd += d3 * d3;
        reinterpret_cast<float4*>(x)[k / 4] = xn;
    }
    *support = (int32_t)cnt;
    if (sqrt(dd) < tol) {
        *conv = true;
        *state = kConverged;
        return false;
    }
    return true;
}

}  // namespace ms
