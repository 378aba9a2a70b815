// Shift iteration, BF16 tensor-core form (the shift loop of Algorithm 2; Eq. 6-8, 11).
//
// One work item = 128 seeds x a chunk of 128-pixel tiles. Per pixel tile:
//   GEMM1  S' = Xh.Ph + Xh.Pm + Xl.Ph - c       (4 tcgen05 MMAs, FP32 in TMEM)
//          x ~ Xh + Xl and p = Ph + Pm + Pl are round-to-nearest BF16 splits
//          of the FP32 vectors (p's exact) and -c is split into three BF16
//          terms against a ones column, so S' = x.p - c up to the dropped
//          terms (at most 3.04 * 2^-16 = 4.64e-5 for unit vectors: a BF16
//          residual is at most 2^-8 of what it splits) and the tensor cores'
//          FP32 accumulation (at most 51 * 2^-22 = 1.2e-5 for d = 16 even for
//          an adder that truncates; measured <= 6e-6): 5.9e-5 < kBand.
//   scan   every 32 x 32 piece of S' (32 seeds, 32 pixels) whose largest value
//          is below -kBand = -2^-14 holds no pair of any window. That maximum
//          comes with the TMEM load (tcgen05.ld.red max), so such a piece
//          costs one load and one compare and has no further work.
//   mask   the other pieces: a pair is in the window when S' >= 0 (sign bit
//          clear). Pairs with |S'| < kBand are re-decided with the same
//          sequential FP32 dot product as the FP32 form, against the pixel's
//          exact FP32 value rebuilt from its BF16 parts in the shared-memory
//          tile, so every decision equals the FP32 form's, whose dot product
//          is within 1e-6 of x.p. Whether a warp holds such a pair comes with
//          the second TMEM load (ld.red min.abs), so the mask costs a byte
//          permute and a logic op per two pixels and nothing else.
//   GEMM2  Y += Mask . [Ph | Pm | Pl | 1]    (mask exact in BF16; a ones
//          column, 0 in the rows that pad the last tile, yields the window
//          size), 2 tcgen05 MMAs for each 32-pixel
//          piece that holds a mask, with the lanes (seeds) of pieces without
//          one disabled. A skipped product would have added zeros, so the
//          sums are those of the full product, bit for bit.
// The seed-by-pixel matrix lives only in TMEM and registers. After the item's
// last tile the Y sums are added to the per-seed fixed-point accumulators
// shared with the FP32 form, and the same finalize kernel normalises the seeds
// and tests convergence in FP64.
//
// What this rests on: a window is a small part of a frame (0.5% on 512 x 512
// frames of 60 cells), and the active seeds of a round are kept in pixel order
// (ms_seed.cu), so the 128 seeds of an item come from the same few cells, and
// so do 128 consecutive pixels: on such a frame 22% of the 128 x 128 tiles hold a
// pair of any window for 4096 active seeds (99% with the seeds in draw order).
// One launch of 32768 seeds on a 512 x 512 frame: 0.56 ms against 1.06 ms for
// the form that built every mask and ran every product; 4096 seeds: 0.10
// against 0.149 ms. What bounds it now: the issuing and scanning warps' chains
// per tile (about 400 clocks; the tensor pipe needs 256 of them), and tiles
// that hold windows, whose S buffer stays taken through mask and GEMM2.
//
// Warp roles (one CTA per SM): the mask warps read S and build masks (each
// reaches the TMEM lanes 32 * (warp % 4) + 0..31), in groups that take the
// pixel tiles in turn; then a TMA producer (a ring of pixel tiles), the GEMM1
// issuer, which owns TMEM (three S buffers and Y), and the GEMM2 issuer. A mask is written over the
// columns of S it was made from, where GEMM2 reads it as its A operand: the
// buffer is free for GEMM1 again once the tile's mask warps are done and its
// GEMM2, if any, has completed. The
// issuing warps run their loops with all 32 lanes and let one elected lane
// issue each MMA and commit: a loop run by lane 0 alone issues the MMAs about
// 1.5x slower. Seed operands (A1) are double-buffered, Y is single (one item
// at a time; the next item's GEMM2 waits for the epilogue's read). All waits
// are bounded; a timeout raises the CTA's abort flag, drains what is in
// flight, frees TMEM and reports MS_ERR_TIMEOUT through the frame's status
// word.
#include <cudaTypedefs.h>

#include "ms_batch.cuh"
#include "ms_device.cuh"
#include "ms_shift_tc.cuh"
#include "ms_tc.cuh"

#include <type_traits>

namespace ms {
namespace {

using namespace tc;

// Warp arrangement of a CTA (what the autotuner chooses among). MW mask warps
// form G groups that take the pixel tiles in turn (group k has the tiles g with
// g % G == k); each warp of a group scans 128 / (MW / G / 4) pixels of its
// tiles for its 32 seeds. NS S buffers of 128 TMEM columns let GEMM1 run ahead
// of the groups.
template <int MW, int G, int NS>
struct TcShape {
    static constexpr int kGroups = G;
    static constexpr int kGroupWarps = MW / G;      // mask warps per tile
    static constexpr int kSBufs = NS;
    static constexpr int kPxPerWarp = 4 * 128 / kGroupWarps;  // pixels of a tile per mask warp
    static constexpr int kSub = kPxPerWarp / 32;    // 32-pixel pieces per mask warp and tile
    static constexpr int kWarpTma = MW;
    static constexpr int kWarpG1 = MW + 1;
    static constexpr int kWarpG2 = MW + 3;
    static constexpr int kThreads = (MW + 4) * 32;
    static_assert(MW % G == 0 && kGroupWarps % 4 == 0 && kPxPerWarp % 32 == 0 && kPxPerWarp >= 32,
                  "each group's mask warps cover the four TMEM quadrants evenly");
    static_assert(NS == 2 || NS == 3, "two or three S buffers");
    // a group that waits for tile g has seen tile g - G, so S buffer phases up
    // to tile g - NS are over and the parity it waits for is the next one
    static_assert(G <= NS, "a group's tiles are at most NS apart");
};
// Index = ms_config.tc_shape.
using TcShape0 = TcShape<8, 2, 3>;
using TcShape1 = TcShape<16, 1, 3>;
using TcShape2 = TcShape<4, 1, 3>;
using TcShape3 = TcShape<8, 1, 3>;
using TcShape4 = TcShape<16, 2, 3>;
using TcShape5 = TcShape<12, 3, 3>;
using TcShape6 = TcShape<16, 2, 2>;
using TcShape7 = TcShape<8, 2, 2>;
constexpr uint32_t kTmemCols = 512;
constexpr int kMaxSBufs = 3;
constexpr uint32_t kColS = 0;          // S accumulators (and the masks built in place), 384 columns
constexpr uint32_t kColY = 384;        // Y accumulators: 64 columns per 16-dimensional half

// Layout for embedding dimension D: 16, or 32 as two 16-dimensional halves,
// each with its own seed-operand tile, pixel tile (a second Pk array) and Y
// block.
template <int D>
struct TcDim {
    static_assert(D == 16 || D == 32, "embedding dimension 16 or 32");
    static constexpr int kHalves = D / 16;
    static constexpr int kStages = D == 16 ? 10 : 4;              // pixel-tile ring, more than the S buffers
    static constexpr int kStageBytes = kHalves * kTileBytes;
    static constexpr int kOffA1 = 0;                              // 2 items x kHalves x 16 KB
    static constexpr int kOffP = 2 * kHalves * kTileBytes;        // kStages stages
    static constexpr int kOffX = kOffP + kStages * kStageBytes;   // 2 x 128 x D floats: the item's seeds
    static constexpr int kOffBar = kOffX + 2 * 128 * D * 4;
    static constexpr int kNumBars = 3 * kStages + kMaxSBufs + 2 + 3;
    static constexpr int kOffHit = (kOffBar + kNumBars * 8 + 15) / 16 * 16;  // kStages x 16 bytes
    static constexpr int kSmemBytes = kOffHit + kStages * 16 + 32 + 1024;    // + TMEM slot, flags, alignment slack
    static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
    static_assert(kStages % 2 == 0, "a GEMM1 issuer of alternate tiles has seen its stage's previous phase");
    static_assert(kStages > kMaxSBufs, "GEMM1 of a tile never waits for a stage that its own GEMM2 order holds");
};

struct TcSplit {
    int tiles, chunks, tpc;  // seed tiles, pixel chunks, pixel tiles per chunk
};

__device__ __forceinline__ TcSplit tc_split(int n_active, int n_ptiles, int target, int grid) {
    TcSplit s;
    s.tiles = (n_active + 127) / 128;
    if (s.tiles == 0 || n_ptiles == 0) {
        s.chunks = 0;
        s.tpc = 1;
        return s;
    }
    s.tpc = tc_tiles_per_chunk_warp(s.tiles, n_ptiles, target, grid);
    s.chunks = (n_ptiles + s.tpc - 1) / s.tpc;
    return s;
}

// Bytes {0,1} = sign of a, {2,3} = sign of b, replicated: 0xFFFF per negative half.
__device__ __forceinline__ uint32_t sign_halves(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, 0xFFBB;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// Row r of an item's seed operand (one 16 KB tile per 16-dimensional half)
// and of its FP32 seed tile in shared memory, for seed slot `slot` of X
// (D components; a padding row, slot < 0: zeros).
template <int D>
__device__ __forceinline__ void write_seed_rows(uint8_t* A1, float* Xs, int r, const float* X, int slot, float c_f) {
    float x[D];
    load_seed_row<D>(X, slot, x);
#pragma unroll
    for (int k = 0; k < D; k += 4)
        *reinterpret_cast<float4*>(Xs + r * D + k) = make_float4(x[k], x[k + 1], x[k + 2], x[k + 3]);
#pragma unroll
    for (int hf = 0; hf < D / 16; ++hf) write_a1_half(A1 + hf * kTileBytes, r, x + 16 * hf, c_f, hf == 0);
}

// Work items of one frame: seed tiles of 128 x chunks of 128-pixel tiles.
struct TcSingleMap {
    const int32_t* active;
    const DevCounters* dc;
    int n, n_ptiles, target;
    int n_active;
    TcSplit sp;
    __device__ __forceinline__ bool init() {
        if (dc->done) return false;
        n_active = dc->n_active;
        sp = tc_split(n_active, n_ptiles, target, (int)gridDim.x);
        return true;
    }
    __device__ __forceinline__ int total() const { return sp.tiles * sp.chunks; }
    __device__ __forceinline__ TcItem item(int i) const {
        int t, ch;
        tc_item_place(i, sp.tiles, sp.chunks, &t, &ch);
        const int pt0 = ch * sp.tpc;
        TcItem it;
        it.active = active;
        it.n_active = n_active;
        it.seed0 = t * 128;
        it.pt0 = pt0;
        it.pt1 = min(n_ptiles, pt0 + sp.tpc);
        it.pk_row0 = 0;
        it.pix0 = 0;
        it.n = n;
        return it;
    }
};

template <class Shape, int kD, bool kDebug, class Map>
__global__ void __launch_bounds__(Shape::kThreads, 1)
k_shift_tc(const __grid_constant__ CUtensorMap pmap, const __grid_constant__ CUtensorMap pmap1,
           const float* X, unsigned long long* __restrict__ acc, float c_f, Map map, int* status,
           unsigned long long* band_ctr, float* __restrict__ dbg_S, int64_t dbg_stride) {
    using L = TcDim<kD>;
    constexpr int kHalves = L::kHalves, kStages = L::kStages, kStageBytes = L::kStageBytes;
    constexpr int kGroups = Shape::kGroups, kGroupWarps = Shape::kGroupWarps, kSBufs = Shape::kSBufs;
    constexpr int kPxPerWarp = Shape::kPxPerWarp, kSub = Shape::kSub;
    constexpr float kBand = kScoreBand<kD>;
    constexpr int kWarpTma = Shape::kWarpTma, kWarpG1 = Shape::kWarpG1, kWarpG2 = Shape::kWarpG2;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* A1 = smem + L::kOffA1;               // [item buffer][half] 16 KB tiles
    uint8_t* Pst = smem + L::kOffP;
    float* Xs = (float*)(smem + L::kOffX);        // [2][128][kD] seeds of an item (FP32 re-decisions)
    uint64_t* bars = (uint64_t*)(smem + L::kOffBar);
    uint64_t* full = bars;                        // [kStages] pixel tile landed
    uint64_t* done = full + kStages;              // [kStages] the tile's mask warps have read S and written their masks
    uint64_t* empty = done + kStages;             // [kStages] pixel tile no longer needed
    uint64_t* s_full = empty + kStages;           // [kSBufs] GEMM1 of a tile done
    uint64_t* d_full = s_full + kMaxSBufs;        // Y of an item complete
    uint64_t* d_empty = d_full + 1;               // Y read by the epilogue and set to zero
    uint64_t* aux = d_empty + 1;                  // [3] drain barriers of the MMA issuers
    uint8_t* hits = smem + L::kOffHit;            // [kStages][quadrant][piece] 1: a mask was written
    uint32_t* tmem_slot = (uint32_t*)(hits + kStages * 16);
    volatile int* abort = (volatile int*)(tmem_slot + 1);
    volatile int* a1_seq = (volatile int*)(tmem_slot + 4);  // [4] items whose rows of A1 a lead warp has written

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&done[s], kGroupWarps);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < kSBufs; ++b) mbar_init(&s_full[b], 1);
        mbar_init(d_full, 1);
        mbar_init(d_empty, 128);
        for (int k = 0; k < 3; ++k) mbar_init(&aux[k], 1);
        *abort = 0;
        for (int k = 0; k < 4; ++k) a1_seq[k] = 1;  // the first item's are written before the roles start
        fence_mbar_init();
    }
    if (warp == kWarpTma && lane == 0) {
        tma_prefetch_desc(&pmap);
        if (kHalves > 1) tma_prefetch_desc(&pmap1);
    }
    if (warp == kWarpG1) {
        tmem_alloc(tmem_slot, kTmemCols);
        tmem_relinquish();
    }
    __syncthreads();
    grid_release();  // TMEM is held
    grid_wait();
    const int items = map.init() ? map.total() : 0;
    if (warp < 4 && (int)blockIdx.x < items) {  // the first item's seeds, while the rest is set up
        const TcItem ii = map.item(blockIdx.x);
        const int pos = ii.seed0 + warp * 32 + lane;
        write_seed_rows<kD>(A1, Xs, warp * 32 + lane, X, pos < ii.n_active ? ii.active[pos] : -1, c_f);
        fence_proxy_async();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == kWarpTma) {
        // ------------------------------------------------ TMA producer
        // The issuing warps run their loops with all 32 lanes (waits are
        // warp-uniform) and one lane issues; see mma_bf16_warp.
        Ring<kStages> st;
        int g = 0;
        bool ok = true;
        for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
            const TcItem ii = map.item(item);
            for (int pt = ii.pt0; pt < ii.pt1; ++pt, ++g, st.advance(1)) {
                const int s = st.i;
                if (g >= kStages && !(ok = warp_wait(&empty[s], st.par ^ 1u, abort))) break;
                if (lane == 0) {
                    mbar_arrive_expect_tx(&full[s], kStageBytes);
                    tma_load_2d(Pst + s * kStageBytes, &pmap, 0, ii.pk_row0 + pt * 128, &full[s]);
                    if (kHalves > 1)
                        tma_load_2d(Pst + s * kStageBytes + kTileBytes, &pmap1, 0, ii.pk_row0 + pt * 128, &full[s]);
                }
                __syncwarp();
            }
        }
        if (lane == 0 && *abort)
            for (int q = max(0, g - kStages); q < g; ++q) drain_wait(&full[q % kStages], (q / kStages) & 1);
    } else if (warp >= kWarpG1 && warp < kWarpG2) {
        // ------------------------------------------------ GEMM1 issuers
        // Two warps take alternate tiles (a warp's chain of waits, address
        // arithmetic, issue and commit takes 400 clocks), up to kSBufs tiles
        // ahead of the mask warps. The S buffer of tile g - kSBufs is free when
        // its pixel stage is: its mask warps are done and its GEMM2, if any,
        // has completed. Descriptors are built once; moving an operand by b
        // bytes adds b >> 4 to the descriptor's start-address field (no carry:
        // shared addresses stay below 2^18).
        const int par = warp - kWarpG1;
        const uint64_t dA1 = desc_sw128(smem_u32(A1), 16, 1024);           // seed operand, K-major
        const uint64_t dP1 = desc_sw128(smem_u32(Pst), 16, 1024);          // pixel tile, K-major
        constexpr uint32_t id1 = idesc_bf16(128, 128, 0, 0);
        constexpr uint64_t kT = kTileBytes >> 4;
        Ring<kStages> st, old;   // stages of tile g and of tile g - kSBufs
        Ring<kSBufs> sb;
        st.advance(par);
        sb.advance(par);
        old.advance((kSBufs ^ par) & 1);  // tile g - kSBufs of the warp's first g >= kSBufs
        bool ok = true;
        int g = par, g0 = 0, it = 0;
        for (int item = blockIdx.x; item < items && ok; item += gridDim.x, ++it) {
            const TcItem ii = map.item(item);
            const int g1 = g0 + ii.pt1 - ii.pt0;
            if (g < g1 && !(ok = seq_wait4(a1_seq, it + 1, abort))) break;
            const uint64_t a = dA1 + (uint64_t)(it & 1) * kHalves * kT;
            for (; g < g1; g += 2, st.advance(2), sb.advance(2)) {
                const bool reuse = g >= kSBufs;  // (the first tiles find their S buffers free)
                if (!(ok = warp_wait2(&full[st.i], st.par, reuse ? &empty[old.i] : &full[st.i],
                                      reuse ? old.par : st.par, abort)))
                    break;
                if (reuse) old.advance(2);
                tc_fence_after();
                const uint32_t tS = tmem + kColS + sb.i * 128;
                const uint64_t pb = dP1 + (uint64_t)st.i * kHalves * kT;
                mma_bf16_split3c_warp(tS, a, pb, id1);                            // Xh.Ph + Xh.Pm + Xl.Ph - c
                if (kHalves > 1) mma_bf16_split3_warp(tS, a + kT, pb + kT, id1);  // dimensions 16..31
                mma_commit_warp(&s_full[sb.i]);
            }
            g0 = g1;
        }
        if (__any_sync(0xffffffffu, *abort)) {
            mma_commit_warp(&aux[par]);
            drain_wait(&aux[par], 0);
        }
    } else if (warp == kWarpG2) {
        // ------------------------------------------------ GEMM2 issuer
        // Y += Mask . P for the pieces that hold a mask; the pixel stage is
        // released when those MMAs complete, or at once when there are none.
        const uint64_t dP2 = desc_sw128(smem_u32(Pst), kTileBytes, 1024);  // pixel tile, MN-major
        constexpr uint32_t id2 = idesc_bf16(128, 64, 0, 1);
        constexpr uint64_t kT = kTileBytes >> 4;
        Ring<kStages> st;
        Ring<kSBufs> sb;
        bool ok = true;
        int it = 0;
        for (int item = blockIdx.x; item < items && ok; item += gridDim.x, ++it) {
            const TcItem ii = map.item(item);
            if (!(ok = warp_wait(d_empty, it & 1, abort))) break;
            for (int pt = ii.pt0; pt < ii.pt1; ++pt, st.advance(1), sb.advance(1)) {
                if (!(ok = warp_wait(&done[st.i], st.par, abort))) break;
                const uint4 hm = *reinterpret_cast<const uint4*>(hits + st.i * 16);
                if (hm.x | hm.y | hm.z | hm.w) {
                    tc_fence_after();
                    const uint32_t tM = tmem + kColS + sb.i * 128;
#pragma unroll
                    for (int pc = 0; pc < 4; ++pc) {
                        const uint32_t byte = 0xffu << (8 * pc);
                        if (!((hm.x | hm.y | hm.z | hm.w) & byte)) continue;
                        const uint32_t off0 = (hm.x & byte) ? 0u : 0xffffffffu, off1 = (hm.y & byte) ? 0u : 0xffffffffu,
                                       off2 = (hm.z & byte) ? 0u : 0xffffffffu, off3 = (hm.w & byte) ? 0u : 0xffffffffu;
#pragma unroll
                        for (int hf = 0; hf < kHalves; ++hf) {
                            const uint32_t tY = tmem + kColY + 64 * hf;
                            const uint64_t pb = dP2 + (uint64_t)(st.i * kHalves + hf) * kT;
                            mma_bf16_ts2_lanes_warp(tY, tM + 32 * pc, pb + 2 * pc * 128, id2, off0, off1, off2, off3);
                        }
                    }
                    mma_commit_warp(&empty[st.i]);
                } else if (lane == 0) {
                    mbar_arrive(&empty[st.i]);
                }
            }
            if (!ok) break;
            mma_commit_warp(d_full);
        }
        if (__any_sync(0xffffffffu, *abort)) {
            mma_commit_warp(&aux[2]);
            drain_wait(&aux[2], 0);
        }
    } else {
        // ------------------------------------------------ mask warps
        // Group grp of kGroups takes the tiles g with g % kGroups == grp; in a
        // group, warp w reaches TMEM lanes 32 * (w % 4) + 0..31 (its seeds) and
        // scans kPxPerWarp pixels of the tile.
        const int grp = warp / kGroupWarps;
        const int q = warp & 3;                         // TMEM lane quadrant
        const int h = (warp % kGroupWarps) >> 2;        // which kPxPerWarp pixels of a tile
        const bool lead = warp < 4;                     // writes the seed operand and reads Y
        const int r = q * 32 + lane;                    // seed row
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        long long band_local = 0;
        int my = grp, g0 = 0, it = 0;
        Ring<kStages> st;
        Ring<kSBufs> sb;
        Ring<kStages> old;  // stage of tile my - kSBufs, from the first such tile on
        st.advance(grp);
        sb.advance(grp);
        old.advance((kGroups - kSBufs % kGroups + grp) % kGroups);
        if (lead) {  // Y starts from zero
#pragma unroll
            for (int k = 0; k < 4 * kHalves; ++k) tmem_zero16(tmem + kColY + lane_base + 16 * k);
            tmem_st_wait();
            tc_fence_before();
            mbar_arrive(d_empty);
        }
        for (int item = blockIdx.x; item < items; item += gridDim.x, ++it) {
            if (__any_sync(0xffffffffu, *abort)) break;
            const TcItem ii = map.item(item);
            const int pt0 = ii.pt0, pt1 = ii.pt1;
            const int pos = ii.seed0 + r;
            const int slot = pos < ii.n_active ? ii.active[pos] : -1;
            if (lead) {
                // A1 for the next item (the first item's was written at the
                // start). Its buffer was last read by the GEMM1s of item it-1,
                // all complete before this warp saw that item's d_full.
                const int nitem = item + gridDim.x;
                if (nitem < items) {
                    const TcItem ni = map.item(nitem);
                    const int npos = ni.seed0 + r;
                    write_seed_rows<kD>(A1 + ((it + 1) & 1) * kHalves * kTileBytes, Xs + ((it + 1) & 1) * 128 * kD, r, X,
                                        npos < ni.n_active ? ni.active[npos] : -1, c_f);
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) {
                        __threadfence_block();
                        a1_seq[warp] = it + 2;
                    }
                }
            }
            bool ok = true;
            const float* xs = Xs + (it & 1) * 128 * kD + r * kD;
            // my: the group's next tile, counted over all items
            for (; my < g0 + pt1 - pt0 && ok; my += kGroups, st.advance(kGroups), sb.advance(kGroups)) {
                const int pt = pt0 + my - g0, s = st.i;
                // The buffer's previous phase has to be over before the parity
                // of this tile's means anything. A group that took tile
                // g - kSBufs (one group, or as many as buffers) knows; else the
                // release of that tile says so (it comes before GEMM1 of this
                // one, so the wait is over by then, and its barrier is not a
                // phase ahead before this tile is done).
                if constexpr (kGroups > 1 && kGroups != kSBufs) {
                    const bool reuse = my >= kSBufs;
                    if (!(ok = warp_wait2(reuse ? &empty[old.i] : &s_full[sb.i], reuse ? old.par : sb.par,
                                          &s_full[sb.i], sb.par, abort)))
                        break;
                    if (reuse) old.advance(kGroups);
                } else {
                    if (!(ok = warp_wait(&s_full[sb.i], sb.par, abort))) break;
                }
                tc_fence_after();
                const uint32_t tS = tmem + kColS + sb.i * 128 + lane_base + h * kPxPerWarp;
                // Which pieces may hold a pair of a window (a NaN seed's scores
                // are all NaN: not below the threshold). Their scores are
                // loaded again below, so that none stays in registers here.
                uint32_t need = 0u;
                {
                    float mx[kSub];
                    uint32_t v[32];
#pragma unroll
                    for (int p = 0; p < kSub; ++p) tmem_ld32_max(tS + 32 * p, v, &mx[p]);
                    tmem_ld_wait();
                    bool near[kSub], any = false;
#pragma unroll
                    for (int p = 0; p < kSub; ++p) any |= near[p] = !(mx[p] < -kBand);
                    if (__any_sync(0xffffffffu, any)) {
#pragma unroll
                        for (int p = 0; p < kSub; ++p)
                            if (__any_sync(0xffffffffu, near[p])) need |= 1u << p;
                    }
                }
                if (kDebug) {
                    for (int j = 0; j < kSub; ++j) {
                        uint32_t v[32];
                        tmem_ld32(tS + j * 32, v);
                        tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            dbg_S[(int64_t)r * dbg_stride + pt * 128 + h * kPxPerWarp + j * 32 + i] =
                                __uint_as_float(v[i]);
                    }
                }
                // The masks of those pieces. Pairs near the boundary are noted
                // (bit 31 - i: pair i is near / S' < 0) and decided below, once
                // for all pieces: a decision that differs from the sign is rare.
                uint32_t hit = 0u, bandp = 0u;
                uint32_t bandm[kSub], negm[kSub];
#pragma unroll
                for (int p = 0; p < kSub; ++p) bandm[p] = negm[p] = 0u;
                while (need) {
                    const int j = __ffs(need) - 1;
                    need &= need - 1u;
                    uint32_t v[32], w[16];
                    float mn;
                    tmem_ld32_minabs(tS + j * 32, v, &mn);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 16; ++i) w[i] = ~sign_halves(v[2 * i], v[2 * i + 1]) & 0x3F803F80u;
                    tmem_st16(tS + j * 32, w);
                    hit |= 1u << (8 * j);
                    if (__any_sync(0xffffffffu, mn < kBand)) {
                        uint32_t bm[4] = {0u, 0u, 0u, 0u}, nm[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                        for (int i = 0; i < 8; ++i)
#pragma unroll
                            for (int e = 0; e < 4; ++e) {  // four chains of eight
                                const uint32_t vi = v[8 * e + i];
                                bm[e] = __funnelshift_l(__float_as_uint(fabsf(__uint_as_float(vi)) - kBand), bm[e], 1);
                                nm[e] = __funnelshift_l(vi, nm[e], 1);
                            }
                        const uint32_t b4 = (bm[0] << 24) | (bm[1] << 16) | (bm[2] << 8) | bm[3];
                        const uint32_t n4 = (nm[0] << 24) | (nm[1] << 16) | (nm[2] << 8) | nm[3];
#pragma unroll
                        for (int p = 0; p < kSub; ++p)
                            if (p == j) {
                                bandm[p] = b4;
                                negm[p] = n4;
                            }
                        bandp |= 1u << j;
                    }
                }
                if (bandp) {
                    // Re-decide near-boundary pairs with the FP32 form's dot
                    // product against the exact FP32 pixel rebuilt from the
                    // tile in shared memory. The tile and the item's seeds
                    // landed long ago; these waits make them visible here (the
                    // barrier cannot be a phase ahead: this tile is not done).
                    ok = seq_wait4(a1_seq, it + 1, abort) && mbar_wait(&full[s], st.par, abort);
                    if (!ok) *abort = 1;
                    const uint8_t* stage = Pst + s * kStageBytes;
                    uint32_t flip[kSub];
                    bool flips = false;
#pragma unroll
                    for (int p = 0; p < kSub; ++p) {
                        uint32_t todo = ok ? bandm[p] : 0u;
                        flip[p] = 0u;
                        while (todo) {
                            const int i = __clz(todo);
                            const uint32_t bit = 0x80000000u >> i;
                            todo &= ~bit;
                            const int row = h * kPxPerWarp + p * 32 + i;
                            bool in = false;  // a padding pixel is in no window
                            if (pt * 128 + row < ii.n) {
                                ++band_local;
                                in = stage_dot<kD>(stage, row, xs) >= c_f;  // xs: the seed (a padding row: zeros)
                            }
                            if (in == ((negm[p] & bit) != 0u)) flip[p] |= bit;
                        }
                        flips |= flip[p] != 0u;
                    }
                    __syncwarp();
                    if (__any_sync(0xffffffffu, flips)) {
#pragma unroll 1
                        for (int j = 0; j < kSub; ++j) {
                            if (!((bandp >> j) & 1u)) continue;
                            uint32_t f = flip[0];
#pragma unroll
                            for (int p = 1; p < kSub; ++p)
                                if (p == j) f = flip[p];
                            uint32_t w[16];
                            tmem_st_wait();
                            tmem_ld16(tS + j * 32, w);
                            tmem_ld_wait();
#pragma unroll
                            for (int k = 0; k < 16; ++k) {
                                if (f & (0x80000000u >> (2 * k))) w[k] ^= 0x3F80u;
                                if (f & (0x40000000u >> (2 * k))) w[k] ^= 0x3F800000u;
                            }
                            tmem_st16(tS + j * 32, w);
                        }
                    }
                    if (!(ok = __all_sync(0xffffffffu, ok))) break;
                }
                if (hit) tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    uint8_t* hw = hits + s * 16 + q * 4 + h * kSub;
                    if constexpr (kSub == 1) *hw = (uint8_t)hit;
                    else if constexpr (kSub == 2) *reinterpret_cast<uint16_t*>(hw) = (uint16_t)hit;
                    else *reinterpret_cast<uint32_t*>(hw) = hit;
                    mbar_arrive(&done[s]);
                }
            }
            if (!ok) break;
            g0 += pt1 - pt0;
            if (lead) {
                if (!warp_wait(d_full, it & 1, abort)) break;
                tc_fence_after();
                // Y: per half [sum ph | sum pm | sum pl | count] (the count in
                // half 0), set back to zero once read; Y is handed back after
                // the last half, the sums go out as fixed-point reductions half
                // by half
                const uint32_t ty = tmem + kColY + lane_base;
                bool live = false;
#pragma unroll
                for (int hf = 0; hf < kHalves; ++hf) {
                    uint32_t yh[16], ym[16], yl[16];
                    tmem_ld16(ty + 64 * hf, yh);
                    tmem_ld16(ty + 64 * hf + 16, ym);
                    tmem_ld16(ty + 64 * hf + 32, yl);
                    float cntf = 0.f;
                    if (hf == 0) {
                        uint32_t yc[16];
                        tmem_ld16(ty + 48, yc);
                        tmem_ld_wait();
                        cntf = __uint_as_float(yc[kCountCol - 48]);
                        live = slot >= 0 && cntf > 0.f;
                    } else {
                        tmem_ld_wait();
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) tmem_zero16(ty + 64 * hf + 16 * k);
                    if (hf == kHalves - 1) {
                        tmem_st_wait();
                        tc_fence_before();
                        mbar_arrive(d_empty);
                    }
                    if (live) {
                        unsigned long long* a = acc + (slot - ii.pix0 + ii.pk_row0) * (kD + 1);
#pragma unroll
                        for (int k = 0; k < 16; ++k) {
                            const float y = __uint_as_float(yh[k]) + __uint_as_float(ym[k]) + __uint_as_float(yl[k]);
                            atomicAdd(a + 16 * hf + k, (unsigned long long)__float2ll_rn(y * kFixScale));
                        }
                        if (hf == 0) atomicAdd(a + kD, (unsigned long long)__float2ll_rn(cntf));
                    }
                }
            }
        }
        if (band_local) atomicAdd(band_ctr, (unsigned long long)band_local);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kWarpG1) tmem_dealloc(tmem, kTmemCols);
    if (threadIdx.x == 0 && *abort) atomicOr(status, 2);
}

// Pixels as BF16 splits for the tensor cores: row i = [Ph | Pm | Pl | 1 1 1 1 0..0]
// (64 values, 128 bytes) with p = Ph + Pm + Pl; rows from the foreground count
// n (read on the device) up to `rows` hold three ones only, so they score
// S' = -c and add nothing to a window's sums or size (pack_split_row). For
// D = 32 a second array of `rows` rows follows, holding dimensions 16..31 the
// same way without the ones.
__global__ void k_pack_bf16(const float* __restrict__ P32, const DevCounters* __restrict__ dc, int rows, int D,
                            uint4* __restrict__ Pk) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows) return;
    const bool fg = i < dc->n_fg;
    pack_split_row(fg ? P32 + (int64_t)i * D : nullptr, Pk + (int64_t)i * 8);
    if (D == 32) pack_split_row(fg ? P32 + (int64_t)i * D + 16 : nullptr, Pk + ((int64_t)rows + i) * 8, false);
}

ms_status encode_pmap(void* Pk, int n_pad, CUtensorMap* map) {
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        cudaDriverEntryPointQueryResult qr;
        void* fn = nullptr;
        MS_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &qr));
        if (qr != cudaDriverEntryPointSuccess || !fn)
            return set_error(MS_ERR_CUDA, "cuTensorMapEncodeTiled is unavailable");
        encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    }
    const cuuint64_t dims[2] = {64, (cuuint64_t)n_pad};
    const cuuint64_t strides[1] = {128};
    const cuuint32_t box[2] = {64, 128};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Pk, dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(MS_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    return MS_OK;
}

// Calls fn with a value of the shape type that `shape` (ms_config.tc_shape) names.
template <class Fn>
ms_status with_tc_shape(int shape, Fn&& fn) {
    switch (shape) {
        case 0: return fn(TcShape0{});
        case 1: return fn(TcShape1{});
        case 2: return fn(TcShape2{});
        case 3: return fn(TcShape3{});
        case 4: return fn(TcShape4{});
        case 5: return fn(TcShape5{});
        case 6: return fn(TcShape6{});
        case 7: return fn(TcShape7{});
        default: return set_error(MS_ERR_INVALID_ARG, "unknown tile shape %d", shape);
    }
}

template <class Map, int D>
ms_status allow_smem(int shape) {
    return with_tc_shape(shape, [](auto sh) -> ms_status {
        MS_CUDA(cudaFuncSetAttribute(k_shift_tc<decltype(sh), D, false, Map>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, TcDim<D>::kSmemBytes));
        return MS_OK;
    });
}

}  // namespace

int tc_smem_bytes(int D) { return D == 32 ? TcDim<32>::kSmemBytes : TcDim<16>::kSmemBytes; }

ms_status tc_pack_async(ms_ctx* ctx) {
    const int rows = (int)((ctx->n_pixels + 127) / 128 * 128);
    if (rows == 0) return MS_OK;
    k_pack_bf16<<<(unsigned)((rows + 255) / 256), 256, 0, ctx->stream>>>(ctx->P32, ctx->dc, rows, (int)ctx->Dp,
                                                                         (uint4*)ctx->Pk);
    MS_LAUNCH("k_pack_bf16");
    ctx->launches += 1;
    return MS_OK;
}

ms_status tc_finish(ms_ctx* ctx) {
    ms_status st = ctx->cfg.precision == MS_FP32 ? f32_tc_setup(ctx->Dp)
                   : ctx->Dp == 32               ? allow_smem<TcSingleMap, 32>(ctx->cfg.tc_shape)
                                                 : allow_smem<TcSingleMap, 16>(ctx->cfg.tc_shape);
    if (st != MS_OK) return st;
    ctx->tc_grid = ctx->num_sms;  // one CTA per SM: it owns all 512 TMEM columns
    if (ms_status ls = label_tc_setup(); ls != MS_OK) return ls;
    // the packed rows use the padding of the workspace (n_pixels rounded up to 128)
    const int64_t rows = (ctx->n_pixels + 127) / 128 * 128;
    if ((st = encode_pmap(ctx->Pk, (int)ctx->n_pad, &ctx->pmap)) != MS_OK) return st;
    if (ctx->Dp == 32) return encode_pmap((uint8_t*)ctx->Pk + rows * 128, (int)ctx->n_pad, &ctx->pmap1);
    ctx->pmap1 = ctx->pmap;
    return MS_OK;
}

ms_status launch_shift_tc(ms_ctx* ctx, const int32_t* active, int grid, int target_items, float* dbg_S) {
    const float c = ceil_to_float(ctx->cfg.bandwidth_cos);
    TcSingleMap map;
    map.active = active;
    map.dc = ctx->dc;
    map.n = (int)ctx->n;
    map.n_ptiles = (int)(ctx->n_pad / 128);
    map.target = target_items;
    unsigned long long* band = (unsigned long long*)&ctx->dc->band_pairs;
    return with_tc_shape(ctx->cfg.tc_shape, [&](auto sh) -> ms_status {
        using Sh = decltype(sh);
        if (ctx->Dp == 32) {
            if (dbg_S) return set_error(MS_ERR_INVALID_ARG, "the score dump is for d <= 16");
            MS_CUDA(launch_after(k_shift_tc<Sh, 32, false, TcSingleMap>, grid, Sh::kThreads, TcDim<32>::kSmemBytes,
                                 ctx->stream, ctx->pmap, ctx->pmap1, ctx->X, ctx->acc, c, map, &ctx->dc->status, band,
                                 nullptr, 0));
        } else if (dbg_S) {
            MS_CUDA(cudaFuncSetAttribute(k_shift_tc<Sh, 16, true, TcSingleMap>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, TcDim<16>::kSmemBytes));
            k_shift_tc<Sh, 16, true, TcSingleMap><<<grid, Sh::kThreads, TcDim<16>::kSmemBytes, ctx->stream>>>(
                ctx->pmap, ctx->pmap1, ctx->X, ctx->acc, c, map, &ctx->dc->status, band, dbg_S, ctx->n_pad);
        } else {
            MS_CUDA(launch_after(k_shift_tc<Sh, 16, false, TcSingleMap>, grid, Sh::kThreads, TcDim<16>::kSmemBytes,
                                 ctx->stream, ctx->pmap, ctx->pmap1, ctx->X, ctx->acc, c, map, &ctx->dc->status, band,
                                 nullptr, 0));
        }
        MS_LAUNCH("k_shift_tc");
        return MS_OK;
    });
}

// ------------------------------------------------------------ batched form
// Work items of every iterating frame: frame f contributes
// item_off[f+1] - item_off[f] items (seed tiles of 128 x chunks).
struct TcBatchMap {
    const BFrame* frames;
    const BState* states;
    BPlan plan;
    const int32_t* act0;
    const int32_t* act1;
    int nf;
    int total_;
    __device__ __forceinline__ bool init() {
        total_ = plan.item_off[nf];
        return total_ > 0;
    }
    __device__ __forceinline__ int total() const { return total_; }
    __device__ __forceinline__ TcItem item(int i) const {
        const int f = locate(plan.item_off, nf, i);
        const int local = i - plan.item_off[f];
        const int chunks = plan.chunks[f], tpc = plan.tpc[f];
        const int n_active = states[f].dc.n_active;
        int t, ch;
        tc_item_place(local, (n_active + 127) / 128, chunks, &t, &ch);
        const BFrame& fr = frames[f];
        TcItem it;
        it.active = ((states[f].dc.iters & 1) ? act1 : act0) + fr.pix0;
        it.n_active = n_active;
        it.seed0 = t * 128;
        it.pt0 = ch * tpc;
        it.pt1 = min(fr.n_ptiles, it.pt0 + tpc);
        it.pk_row0 = fr.pk_row0;
        it.pix0 = fr.pix0;
        it.n = fr.n;
        return it;
    }
};

ms_status tc_batch_setup(int D, int shape) {
    return D == 32 ? allow_smem<TcBatchMap, 32>(shape) : allow_smem<TcBatchMap, 16>(shape);
}

ms_status launch_shift_tc_batch(const CUtensorMap& pmap, const CUtensorMap& pmap1, int D,
                                const float* X, unsigned long long* acc, float c_f, const BFrame* frames,
                                const BState* states, BPlan plan, const int32_t* act0, const int32_t* act1, int nf,
                                int* status, unsigned long long* band, int grid, int shape, cudaStream_t st) {
    TcBatchMap map;
    map.frames = frames;
    map.states = states;
    map.plan = plan;
    map.act0 = act0;
    map.act1 = act1;
    map.nf = nf;
    map.total_ = 0;
    return with_tc_shape(shape, [&](auto sh) -> ms_status {
        using Sh = decltype(sh);
        if (D == 32)
            k_shift_tc<Sh, 32, false, TcBatchMap><<<grid, Sh::kThreads, TcDim<32>::kSmemBytes, st>>>(
                pmap, pmap1, X, acc, c_f, map, status, band, nullptr, 0);
        else
            k_shift_tc<Sh, 16, false, TcBatchMap><<<grid, Sh::kThreads, TcDim<16>::kSmemBytes, st>>>(
                pmap, pmap1, X, acc, c_f, map, status, band, nullptr, 0);
        MS_LAUNCH("k_shift_tc(batch)");
        return MS_OK;
    });
}

ms_status encode_pk_map(void* Pk, int rows, CUtensorMap* map) { return encode_pmap(Pk, rows, map); }

}  // namespace ms
