// Batched form: B frames of uneven size clustered together, every frame's
// OSOP control on the device (a per-frame state machine advanced by one CUDA
// graph whose body runs until all frames finish).
#pragma once

#include "ms_internal.cuh"

namespace ms {

// Per-frame phase of the OSOP loop.
enum BPhase : int32_t { kNeedSeed = 0, kIterating = 1, kRoundDone = 2, kFinished = 3 };

// Per-frame constants, fixed after set-up. Frame f owns the rows
// [pix0, pix0 + n) of every per-pixel, per-seed, per-candidate and per-mode
// array, and the rows [pk_row0, pk_row0 + pk_rows) of Pk and of acc. As in a
// context (ms_ctx), Pk shares its memory with the earlier modes' split rows and
// the conflict lists (candidate a's at row pk_row0 + a), acc with the split rows of
// candidates and of modes (split_row0), and the modes with Xr.
struct BFrame {
    int64_t pix0;
    int64_t n_pixels;   // input pixels
    int32_t n;          // foreground pixels
    int32_t n_ptiles;   // ceil(n / 128)
    int32_t pk_row0;
    int32_t pad;
    uint64_t perm_a, perm_b;
    const float* emb;   // borrowed input [n_pixels, d]
    const uint8_t* mask;
};

// The frame's padded rows.
__host__ __device__ inline int pk_rows(const BFrame& fr) { return (int)((fr.n_pixels + 127) / 128 * 128); }

// The frame's first 128-byte row in acc, read as split rows: its first acc row lies
// pk_row0 * (Dp + 1) * 8 bytes in, a whole number of them as pk_row0 is a multiple
// of 128. Its share holds Dp / 16 arrays of pk_rows split rows.
__host__ __device__ inline int split_row0(const BFrame& fr, int Dp) { return fr.pk_row0 / 16 * (Dp + 1); }

// Per-frame state, advanced only by device code.
struct BState {
    DevCounters dc;
    int64_t N;          // seeds requested next round (Sec. 3.2.4)
    int32_t phase;
    int32_t rounds;
    int32_t k0;         // kept modes before the current merge
    int32_t iters_total;
    int64_t seeds_total;
    int64_t cands_total;
    int64_t dropped_total;
};

// Work split of the current iteration, computed on the device.
// item_off / seed_off: exclusive prefix sums over frames (B + 1 entries).
struct BPlan {
    int32_t* item_off;
    int32_t* seed_off;
    int32_t* chunks;    // per frame
    int32_t* tpc;       // per frame: pixel tiles (TC) or pixels (FP32) per chunk
};

// Tensor-core shift over all iterating frames (ms_shift_tc.cu).
ms_status tc_batch_setup(int D, int shape);
ms_status launch_shift_tc_batch(const CUtensorMap& pmap, const CUtensorMap& pmap1, int D,
                                const float* X, unsigned long long* acc, float c_f, const BFrame* frames,
                                const BState* states, BPlan plan, const int32_t* act0, const int32_t* act1, int nf,
                                int* status, unsigned long long* band, int grid, int shape, cudaStream_t st);
// FP32 form's shift over all iterating frames (ms_shift_f32_tc.cu).
ms_status launch_shift_f32_tc_batch(const CUtensorMap& pmap, const CUtensorMap& pmap1, int Dp, const float* X,
                                    unsigned long long* acc, float c, const BFrame* frames, const BState* states,
                                    BPlan plan, const int32_t* act0, const int32_t* act1, int nf, int* status,
                                    int num_sms, cudaStream_t st);

// Index of the frame whose [off[f], off[f+1]) holds i (off has nf + 1 entries).
__device__ __forceinline__ int locate(const int32_t* off, int nf, int i) {
    int lo = 0, hi = nf;  // invariant: off[lo] <= i < off[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= i) lo = mid; else hi = mid;
    }
    return lo;
}

// Scratch of the tensor-core labelling: the near-tie queue (capacity: the
// foreground pixels) and, in batch form, the per-frame item offsets (B + 1).
struct LabelTcScratch {
    int2* fix;
    int* fix_count;
    int32_t* off;
};

ms_status label_tc_setup();
// Labelling on the tensor cores (Dp = 16 or 32): exact FP64-argmax labels,
// near-ties decided by FP32 scores, then FP64. pmap1: the
// pixels' dimensions 16-31 (Dp = 32); Mk holds the modes' split rows, for
// Dp = 32 followed by a second array of n_pad (mk_rows) rows.
ms_status launch_label_tc_single(const CUtensorMap& pmap, const CUtensorMap& pmap1, void* Mk, int64_t n_pad, int Dp,
                                 const float* modes, int K, int n, const float* P32, const int32_t* pix,
                                 const float* emb, int d, int32_t* labels, LabelTcScratch sc, int grid, int* status,
                                 cudaStream_t st);
// Coverage against one frame's new modes [k0, k1) on the tensor cores, after the
// first `taken` rows of Pk (second array pk_half rows on) are the pixels' again:
// exact decisions.
ms_status launch_cover_tc_single(const CUtensorMap& pmap, const CUtensorMap& pmap1, void* Pk, int64_t pk_half,
                                 int taken, void* Mk, int64_t n_pad, int Dp, const float* modes, int k0, int k1, int n,
                                 const float* P32, const int32_t* pix, const float* emb, int d, double c,
                                 uint8_t* covered, int* n_uncovered, int grid, int* status, cudaStream_t st);
// The same for the frames of a batch whose round ended (tile_off: their pixel
// tiles, from k_b_blocks with 128 pixels per block). amap: the split rows in acc.
ms_status launch_cover_tc_batch(const CUtensorMap& pmap, const CUtensorMap& pmap1, const CUtensorMap& amap, void* Pk,
                                int64_t pk_half, void* Mk, int Dp, const BFrame* frames, BState* states, int B,
                                int max_pk_rows, const float* modes, const float* P32, const int32_t* pix, int d,
                                double c, uint8_t* covered, const int32_t* tile_off, int grid, int* status,
                                cudaStream_t st);
// The merge's two contractions on the tensor cores for the frames whose round
// ended (tile_off: their candidates in blocks of 128): the candidates in rank
// order (Xr, packed into Ck) against their earlier modes (packed into Pk), then
// against one another; exact decisions (merge_cos), the near-threshold pairs decided
// by the FP32-then-FP64 test. Sets removed_r and cand_state and fills the conflict
// lists.
ms_status launch_merge_tc_batch(const CUtensorMap& pmap, const CUtensorMap& pmap1, const CUtensorMap& amap, void* Pk,
                                int64_t pk_half, void* Ck, int Dp, const BFrame* frames, BState* states, int B,
                                int max_pk_rows, const float* modes, const int32_t* rank_cand, uint8_t* cand_state,
                                uint8_t* removed_r, int32_t* conf_deg, int32_t* conf, float thr_f, double thr,
                                const int32_t* tile_off, int grid, int* status, cudaStream_t st);
// The same for one frame: k candidates (Xr) against its K_old earlier modes, then
// against one another.
ms_status launch_merge_tc_single(const CUtensorMap& pmap, const CUtensorMap& pmap1, void* Pk, int64_t pk_half,
                                 void* Ck, int64_t n_pad, int Dp, int k, int K_old, const float* Xr,
                                 const float* modes, const int32_t* rank_cand, uint8_t* cand_state, uint8_t* removed_r,
                                 int32_t* conf_deg, int32_t* conf, float thr_f, double thr, int grid, int* status,
                                 cudaStream_t st);
ms_status launch_label_tc_batch(const CUtensorMap& pmap, const CUtensorMap& pmap1, const CUtensorMap& amap, void* Mk,
                                int Dp, const BFrame* frames, const BState* states, int B, int max_pk_rows,
                                const float* modes, const float* P32, const int32_t* pix, int d,
                                int32_t* const* labels, LabelTcScratch sc, int grid, int* status, cudaStream_t st);

// Pixel tiles per chunk when a frame's seed tiles (128 seeds each) are cut
// into tiles x chunks work items for the tensor-core shift. The plain rule
// spreads `target` items over the seed tiles. With grid > 0 the items are
// also fitted to the launch's CTAs, which each take items in turn: among the
// chunk counts that fill 2..8 whole waves of the grid (at least two items per
// CTA, so one item's pipeline fill overlaps the previous item's drain) and the
// plain rule's,
// the one with the smallest makespan waves x (tiles per item + 2 tiles of
// per-item overhead) wins (ties: the earlier candidate). Integer arithmetic
// only, so every caller with the same arguments cuts a frame the same way.
__host__ __device__ inline int tc_tiles_per_chunk(int tiles, int n_ptiles, int target, int grid) {
    if (tiles <= 0 || n_ptiles <= 0) return 1;
    int ch = (target + tiles - 1) / tiles;
    ch = ch < 1 ? 1 : (ch > n_ptiles ? n_ptiles : ch);
    int best = (n_ptiles + ch - 1) / ch;
    if (grid <= 0) return best;
    auto cost = [&](int tpc) {
        const long long items = (long long)tiles * ((n_ptiles + tpc - 1) / tpc);
        return ((items + grid - 1) / grid) * (long long)(tpc + 2);
    };
    long long best_cost = cost(best);
    for (int w = 2; w <= 8; ++w) {
        int c = (int)((long long)w * grid / tiles);
        if (c < 1) continue;
        c = c > n_ptiles ? n_ptiles : c;
        const int tpc = (n_ptiles + c - 1) / c;
        const long long k = cost(tpc);
        if (k < best_cost) {
            best_cost = k;
            best = tpc;
        }
    }
    return best;
}

#ifdef __CUDACC__
// tc_tiles_per_chunk by a converged warp, a candidate per lane (the divisions
// of one thread took 3.5 us at the start of every shift launch).
__device__ inline int tc_tiles_per_chunk_warp(int tiles, int n_ptiles, int target, int grid) {
    if (tiles <= 0 || n_ptiles <= 0) return 1;
    const int lane = threadIdx.x & 31;
    const unsigned T = (unsigned)tiles, P = (unsigned)n_ptiles, G = (unsigned)(grid > 0 ? grid : 1);
    // lane 0: the plain rule; lanes 1..7: 2..8 waves
    unsigned c = lane == 0 ? ((unsigned)target + T - 1) / T : (unsigned)(lane + 1) * G / T;
    const bool valid = lane == 0 || (lane < 8 && grid > 0 && c >= 1);
    c = c < 1 ? 1 : (c > P ? P : c);
    const unsigned tpc = (P + c - 1) / c;
    const unsigned long long items = (unsigned long long)T * ((P + tpc - 1) / tpc);
    const unsigned long long waves =
        items + G <= 0xffffffffull ? ((unsigned)items + G - 1) / G : (items + G - 1) / G;
    unsigned long long key = valid ? (waves * (tpc + 2)) << 3 | (unsigned)lane : ~0ull;
    for (int o = 4; o > 0; o >>= 1) {
        const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
        key = k2 < key ? k2 : key;
    }
    key = __shfl_sync(0xffffffffu, key, 0);
    return (int)__shfl_sync(0xffffffffu, tpc, (int)(key & 7));
}

// Item i of a frame's seed tiles x chunks, heaviest first: a seed tile's
// windows lie mostly in the chunks around its own place in pixel order (both
// run in pixel order), so the items go from that diagonal outwards, chunk
// offsets 0, +1, -1, +2, ... Items are dealt to the CTAs in turn, so every CTA
// gets its share of heavy ones.
__device__ __forceinline__ void tc_item_place(int i, int tiles, int chunks, int* tile, int* chunk) {
    const int delta = i / tiles, t = i - delta * tiles;
    int ch = (int)((unsigned)(2 * t + 1) * (unsigned long long)chunks / (2u * (unsigned)tiles));
    ch += (delta & 1) ? (delta + 1) / 2 : -(delta / 2);
    ch = ch < 0 ? ch + chunks : (ch >= chunks ? ch - chunks : ch);
    *tile = t;
    *chunk = ch;
}
#endif

}  // namespace ms
