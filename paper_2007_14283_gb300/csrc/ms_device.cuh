// Device helpers: FP32 dot products and thresholded cosine decisions whose
// outcome is exact in FP64.
#pragma once

#include "ms_internal.cuh"

namespace ms {

// Let the stream's next kernel start its blocks (launch_after): they run up to
// their own grid_wait.
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Wait until the work ahead on the stream has ended and its writes are visible;
// returns at once in a kernel that was launched the ordinary way.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Few seeds of a selection are put in pixel order by the CTA that took them,
// instead of by a pass over every pixel of the frame (1 ms for a batched frame of
// 4 million pixels, 80 us for a single one): counted into kFewThreads ranges of
// pixels, and ranked among those of their own range.
constexpr int kFewThreads = 1024;
constexpr int kFewSeeds = 2 * kFewThreads;

struct FewSeeds {
    int32_t pix[kFewSeeds];   // in draw order
    int32_t list[kFewSeeds];  // by range, unordered within one
    int32_t count[kFewThreads];
    int32_t first[kFewThreads];
    int32_t warp[32];
};

// Ranks in pixel order of the frame's n of the pixels pix[tid] and pix[tid +
// kFewThreads] among pix[0..m), m <= kFewSeeds, all distinct (where there are such
// two). Every thread of the CTA calls it, with pix written.
__device__ __forceinline__ void few_ranks(FewSeeds& s, int m, int n, int rank[2]) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int sh = n > kFewThreads ? 32 - __clz((n - 1) / kFewThreads) : 0;  // (n - 1) >> sh < kFewThreads
    s.count[tid] = 0;
    __syncthreads();
    int32_t p[2], at[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int i = tid + k * kFewThreads;
        p[k] = i < m ? s.pix[i] : -1;
        if (p[k] >= 0) at[k] = atomicAdd(&s.count[p[k] >> sh], 1);
    }
    __syncthreads();
    const int c = s.count[tid];
    int incl = c;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s.warp[wid] = incl;
    __syncthreads();
    int before = lane < wid ? s.warp[lane] : 0;
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    s.first[tid] = before + incl - c;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (p[k] >= 0) s.list[s.first[p[k] >> sh] + at[k]] = p[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (p[k] < 0) continue;
        const int q0 = s.first[p[k] >> sh], q1 = q0 + s.count[p[k] >> sh];
        int r = q0;
        for (int q = q0; q < q1; ++q) r += s.list[q] < p[k];
        rank[k] = r;
    }
}

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

// Squared step norms that an FP32 evaluation settles: below `lo` the seed has
// converged, from `hi` on it moves; between them FP64 decides. The FP32 value's
// relative error is at most (d + 5) 2^-24 < 3e-6 (differences, products and
// sums of non-negative terms each round once), the lines lie 1e-5 apart from
// tol^2, and below 1e-30, where products underflow, FP64 always decides.
struct StepBand {
    float lo, hi;
};
inline StepBand step_band(double tol) {
    const double t2 = tol * tol;
    StepBand b;
    b.lo = t2 < 1e-30 ? -1.0f : (float)(t2 * (1.0 - 1e-5));
    b.hi = t2 < 1e-30 ? 1e-30f : (float)(t2 * (1.0 + 1e-5));
    return b;
}

struct SeedEnd {
    bool conv, fail, move;
};

// Mean-shift update (Eq. 5 with the flat kernel) of the 8 seeds of a warp, four
// lanes a seed: lane 8 q + s holds dimensions [q Dp/4, (q+1) Dp/4) of seed s.
// The seed's window sums (fixed point, 2^-36 units) and count are set back to
// zero: x <- normalise(sum), conv when the FP64 step norm is below tol, fail
// when the window is empty, move when the seed moves on (the same on all four
// lanes); lanes that are not `live` only take part in the shuffles.
// Bound by the FP64 pipe: a warp's FP64 instruction takes about 64 clocks here,
// and one thread per seed was 219 of them (5.6 us a launch of few seeds). Four
// lanes a seed, no scaling by 2^-36 (a power of two moves through every step of
// the normalisation unchanged) and the step norm in FP32 outside the band leave
// 78. The sums over dimensions pass from lane to lane in the order of the
// dimensions, so every bit is that of one thread's loop.
// Every load comes before the first store: a store between two loads of the
// same array keeps them in order, and each load then costs a memory round trip.
template <int Dp>
__device__ __forceinline__ SeedEnd finalize_seed(bool live, unsigned long long* a, float* x, uint8_t* state,
                                                 int32_t* support, double tol, StepBand band) {
    constexpr int kPer = Dp / 4;
    const int lane = threadIdx.x & 31, q = lane >> 3, sl = lane & 7;
    long long sum[kPer], cnt = 0;
    float4 xo[kPer / 4];
#pragma unroll
    for (int k = 0; k < kPer; ++k) sum[k] = 0;
#pragma unroll
    for (int k = 0; k < kPer / 4; ++k) xo[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (live) {
#pragma unroll
        for (int k = 0; k < kPer; ++k) sum[k] = (long long)a[q * kPer + k];
        if (q == 0) cnt = (long long)a[Dp];
#pragma unroll
        for (int k = 0; k < kPer / 4; ++k) xo[k] = reinterpret_cast<const float4*>(x)[q * (kPer / 4) + k];
    }
    double y[kPer], ss = 0.0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) y[k] = (double)sum[k];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        double t = ss;
#pragma unroll
        for (int k = 0; k < kPer; ++k) t += y[k] * y[k];
        ss = __shfl_sync(0xffffffffu, t, 8 * g + sl);
    }
    cnt = __shfl_sync(0xffffffffu, cnt, sl);
    if (live) {
#pragma unroll
        for (int k = 0; k < kPer; ++k) a[q * kPer + k] = 0ull;
        if (q == 0) a[Dp] = 0ull;
    }
    const double inv = 1.0 / sqrt(ss);
    float xn[kPer];
    float dd32 = 0.f;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        xn[k] = (float)(y[k] * inv);
        const float d = xn[k] - reinterpret_cast<const float*>(xo)[k];
        dd32 = fmaf(d, d, dd32);
    }
    dd32 += __shfl_xor_sync(0xffffffffu, dd32, 8);
    dd32 += __shfl_xor_sync(0xffffffffu, dd32, 16);
    bool conv = dd32 <= band.lo;
    const bool settled = conv || dd32 >= band.hi || cnt == 0;
    if (__any_sync(0xffffffffu, live && !settled)) {
        double dd = 0.0;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            double t = dd;
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                const double d = (double)xn[k] - (double)reinterpret_cast<const float*>(xo)[k];
                t += d * d;
            }
            dd = __shfl_sync(0xffffffffu, t, 8 * g + sl);
        }
        conv = sqrt(dd) < tol;
    }
    if (!live) return SeedEnd{false, false, false};
    if (cnt == 0) {
        if (q == 0) *state = kFailed;
        return SeedEnd{false, true, false};
    }
#pragma unroll
    for (int k = 0; k < kPer / 4; ++k)
        reinterpret_cast<float4*>(x)[q * (kPer / 4) + k] =
            make_float4(xn[4 * k], xn[4 * k + 1], xn[4 * k + 2], xn[4 * k + 3]);
    if (q == 0) {
        *support = (int32_t)cnt;
        if (conv) *state = kConverged;
    }
    return SeedEnd{conv, false, !conv};
}

}  // namespace ms
