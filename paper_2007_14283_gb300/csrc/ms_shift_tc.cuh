// What the tensor-core shift kernels (ms_shift_tc.cu: BF16 form,
// ms_shift_f32_tc.cu: FP32 form) share: the seed operand of GEMM1, the bound of
// its scores, the roles' waits, and what a work item is.
#pragma once

#include "ms_batch.cuh"
#include "ms_tc.cuh"

namespace ms {
namespace {

using namespace tc;

constexpr int kTileBytes = 128 * 128;        // 128 rows x 128 bytes
constexpr float kFixScale = 68719476736.0f;  // 2^36

// Half-width of the recheck band of the scores S' = Xh.Ph + Xh.Pm + Xl.Ph - c:
// above their bound (dropped terms 4.64e-5 and accumulation (3 * D + 3) * 2^-22
// = 1.2e-5 or 2.4e-5; derived in ms_shift_tc.cu).
template <int D>
constexpr float kScoreBand = D == 16 ? 6.103515625e-05f : 7.5e-05f;  // 2^-14 for d = 16

// Bounded wait that ignores the abort flag (used while draining).
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - t0 > kWaitCycles) return;
}

// Seed `slot` of X (D components; slot < 0: zeros). X is written by the kernel
// ahead, so its pointer promises nothing: all loads come before whatever the caller
// stores, or each would wait for the one before it (1.2 us a launch).
template <int D>
__device__ __forceinline__ void load_seed_row(const float* X, int slot, float (&x)[D]) {
#pragma unroll
    for (int k = 0; k < D; k += 4) {
        const float4 v = slot >= 0 ? *reinterpret_cast<const float4*>(X + (int64_t)slot * D + k)
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
        x[k] = v.x; x[k + 1] = v.y; x[k + 2] = v.z; x[k + 3] = v.w;
    }
}

// Row r of one 16-dimensional half of a seed operand tile:
// [Xh | Xl | -c split, 0 | unused] for the first half, [Xh | Xl | unused] for
// the second (the -c column is added once), 128-byte swizzle.
__device__ __forceinline__ void write_a1_half(uint8_t* A1, int r, const float* x, float c_f, bool with_c) {
    uint32_t wh[8], wl[8];
#pragma unroll
    for (int k = 0; k < 16; k += 2) {
        const float h0 = bf16_round(x[k]), h1 = bf16_round(x[k + 1]);
        wh[k / 2] = pack_bf16(h0, h1);
        wl[k / 2] = pack_bf16(x[k] - h0, x[k + 1] - h1);
    }
    *reinterpret_cast<uint4*>(A1 + sw128_offset(r, 0)) = make_uint4(wh[0], wh[1], wh[2], wh[3]);
    *reinterpret_cast<uint4*>(A1 + sw128_offset(r, 1)) = make_uint4(wh[4], wh[5], wh[6], wh[7]);
    *reinterpret_cast<uint4*>(A1 + sw128_offset(r, 2)) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
    *reinterpret_cast<uint4*>(A1 + sw128_offset(r, 3)) = make_uint4(wl[4], wl[5], wl[6], wl[7]);
    if (with_c) {
        const float c_hi = bf16_round(c_f);
        const float c_mid = bf16_round(c_f - c_hi);
        const float c_lo = (c_f - c_hi) - c_mid;
        *reinterpret_cast<uint4*>(A1 + sw128_offset(r, 4)) =
            make_uint4(pack_bf16(-c_hi, -c_mid), pack_bf16(-c_lo, 0.f), 0u, 0u);
        *reinterpret_cast<uint4*>(A1 + sw128_offset(r, 5)) = make_uint4(0u, 0u, 0u, 0u);
    }
}

// FP32 value of pixel row `row` of a 16-dimensional pixel stage, rebuilt
// exactly from its three BF16 parts (h + m) + l: the split of an FP32 value
// into three round-to-nearest BF16 terms is exact, and so is this sum.
__device__ __forceinline__ void stage_pixel16(const uint8_t* stage, int row, float (&p)[16]) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const uint4 hv = *reinterpret_cast<const uint4*>(stage + sw128_offset(row, c));
        const uint4 mv = *reinterpret_cast<const uint4*>(stage + sw128_offset(row, c + 2));
        const uint4 lv = *reinterpret_cast<const uint4*>(stage + sw128_offset(row, c + 4));
        const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w}, mw[4] = {mv.x, mv.y, mv.z, mv.w},
                       lw[4] = {lv.x, lv.y, lv.z, lv.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            p[c * 8 + 2 * k] = __fadd_rn(__fadd_rn(__uint_as_float(hw[k] << 16), __uint_as_float(mw[k] << 16)),
                                         __uint_as_float(lw[k] << 16));
            p[c * 8 + 2 * k + 1] =
                __fadd_rn(__fadd_rn(__uint_as_float(hw[k] & 0xFFFF0000u), __uint_as_float(mw[k] & 0xFFFF0000u)),
                          __uint_as_float(lw[k] & 0xFFFF0000u));
        }
    }
}

// Dot product, in FP32 with one FMA per component in component order (the
// FP32 form's dot_seq, bit for bit), of seed x (D floats in shared memory)
// with pixel row `row` of a pixel stage (D / 16 tiles of 16 dimensions). The
// pixel is rebuilt exactly from its three BF16 parts (h + m) + l: the split of
// an FP32 value into three round-to-nearest BF16 terms is exact, and so is
// this sum.
template <int D>
__device__ __forceinline__ float stage_dot(const uint8_t* stage, int row, const float* x) {
    float acc = 0.f;
#pragma unroll
    for (int hf = 0; hf < D / 16; ++hf) {
        const uint8_t* t = stage + hf * kTileBytes;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const uint4 hv = *reinterpret_cast<const uint4*>(t + sw128_offset(row, c));
            const uint4 mv = *reinterpret_cast<const uint4*>(t + sw128_offset(row, c + 2));
            const uint4 lv = *reinterpret_cast<const uint4*>(t + sw128_offset(row, c + 4));
            const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w}, mw[4] = {mv.x, mv.y, mv.z, mv.w},
                           lw[4] = {lv.x, lv.y, lv.z, lv.w};
            const float4 x0 = *reinterpret_cast<const float4*>(x + 16 * hf + c * 8);
            const float4 x1 = *reinterpret_cast<const float4*>(x + 16 * hf + c * 8 + 4);
            const float xv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float p0 = __fadd_rn(__fadd_rn(__uint_as_float(hw[k] << 16), __uint_as_float(mw[k] << 16)),
                                           __uint_as_float(lw[k] << 16));
                const float p1 =
                    __fadd_rn(__fadd_rn(__uint_as_float(hw[k] & 0xFFFF0000u), __uint_as_float(mw[k] & 0xFFFF0000u)),
                              __uint_as_float(lw[k] & 0xFFFF0000u));
                acc = fmaf(xv[2 * k], p0, acc);
                acc = fmaf(xv[2 * k + 1], p1, acc);
            }
        }
    }
    return acc;
}

// What a work item covers, in the frame it belongs to.
struct TcItem {
    const int32_t* active;  // seed slots of the frame's active list
    int n_active;           // length of that list
    int seed0;              // list position of the item's first seed
    int pt0, pt1;           // the frame's 128-pixel tiles [pt0, pt1)
    int pk_row0;            // Pk row of the frame's pixel 0 and acc row of its slot 0 (multiple of 128)
    int64_t pix0;           // the frame's slot 0
    int n;                  // the frame's pixel count
};

// Warp-uniform bounded wait: every lane polls, all lanes get the same answer.
// The first look has no time limit to set up: the issuing warps run one
// dependent chain per tile, in which reading the clock before every wait cost
// more than the wait (a wait on a completed phase took 190 clocks).
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort));
}

// Both of two waits; b1 is looked at only once b0's phase is over. (Two
// independent try_waits may be resolved in either order: the first can be held
// back until its phase completes while the second is answered at once.)
__device__ __forceinline__ bool warp_wait2(uint64_t* b0, uint32_t p0, uint64_t* b1, uint32_t p1, volatile int* abort) {
    if (__all_sync(0xffffffffu, mbar_try_wait(b0, p0)) && __all_sync(0xffffffffu, mbar_try_wait(b1, p1))) return true;
    return __all_sync(0xffffffffu, mbar_wait(b0, p0, abort) && mbar_wait(b1, p1, abort));
}

// Bounded wait of a converged warp for four counters in shared memory to reach
// n. Counters, not a barrier: the warps that wait for items may skip items in
// which they have no tile, and a barrier's parity tells only two phases apart.
__device__ __forceinline__ bool seq_wait4(volatile int* seq, int n, volatile int* abort) {
    volatile int* mine = seq + (threadIdx.x & 3);
    if (*mine < n) {
        const long long t0 = clock64();
        while (*mine < n) {
            if (*abort) break;
            if (clock64() - t0 > kWaitCycles) {
                *abort = 1;
                break;
            }
        }
    }
    const bool ok = __all_sync(0xffffffffu, *mine >= n);
    __threadfence_block();
    return ok;
}

// Position in a ring of N slots, with the parity of the current lap.
template <int N>
struct Ring {
    int i = 0;
    uint32_t par = 0;
    __device__ __forceinline__ void advance(int by) {  // by <= N
        i += by;
        if (i >= N) {
            i -= N;
            par ^= 1u;
        }
    }
};

}  // namespace
}  // namespace ms
