// Shift iteration, FP32 form (the shift loop of Algorithm 2; Eq. 6-8, 11): the
// window decisions and the sums of the plain FP32 kernel, bit for bit, with the
// tensor cores left to find where windows can be.
//
// One work item = 128 seeds x a chunk of pixels, the chunks of the plain form
// (shift_split). Per 128-pixel tile:
//   scan   S' = Xh.Ph + Xh.Pm + Xl.Ph - c by 4 tcgen05 MMAs into TMEM, as in
//          the BF16 form (ms_shift_tc.cu, with the bound of S'); a 32 x 32
//          piece whose maximum is below -kBand holds no pair of any window.
//   decide in the other pieces a pair is in the window when S' >= 0, and pairs
//          with |S'| < kBand are decided by the sequential FP32 dot product
//          against c, which the bound makes the decision of every pair.
//   sum    each lane owns a seed and adds its window's pixels in FP32 in pixel
//          order: over the pixels that any of the warp's 32 seeds takes, one
//          multiply-add by 0 or 1 per component (x + 1 p rounds as x + p does,
//          x + 0 p is x). The pixels are rebuilt from the tile's BF16 parts
//          (exactly) into a small shared buffer and read as broadcasts.
// Seed by seed these are the additions of the plain kernel in its order, so the
// fixed-point sums are the same words.
//
// A 512 x 512 frame (310,092 seed-iterations over 131,072 pixels): 15.0 ms in 138
// launches against 41.9 ms for the plain kernel, which ran at 80% of the FP32
// FMA rate over all pairs. What bounds it: the additions over the pixels that
// any of a warp's seeds takes, and the issuing warps' chain per tile.
//
// Roles (192 threads, two CTAs per SM for d <= 16, so that one CTA's sums and
// waits overlap the other's): warps 0-3 scan, decide and sum, each for the 32
// seeds of its TMEM lane quadrant; warp 4 issues TMA loads of pixel tiles; warp
// 5 owns TMEM and issues the MMAs into S buffers of 128 columns. Waits are
// bounded as in the BF16 form.
#include "ms_batch.cuh"
#include "ms_device.cuh"
#include "ms_shift_tc.cuh"
#include "ms_tc.cuh"

namespace ms {
namespace {

constexpr int kFWarpTma = 4, kFWarpG1 = 5, kFThreads = 6 * 32;

template <int D>
struct FDim {
    static constexpr int kHalves = D / 16;
    static constexpr int kCtas = D == 16 ? 2 : 1;                 // per SM
    static constexpr int kStages = 3;                             // pixel-tile ring
    static constexpr int kSBufs = 2;                              // S buffers
    static constexpr int kStageBytes = kHalves * kTileBytes;
    static constexpr int kPxStride = D + 4;                       // floats of a rebuilt pixel (bank spread)
    static constexpr int kOffA1 = 0;                              // 2 items x kHalves x 16 KB
    static constexpr int kOffP = 2 * kHalves * kTileBytes;
    static constexpr int kOffPx = kOffP + kStages * kStageBytes;  // per warp 32 rebuilt pixels
    static constexpr int kOffX = kOffPx + 4 * 32 * kPxStride * 4;  // 2 x 128 x D floats: the item's seeds
    static constexpr int kOffBar = kOffX + 2 * 128 * D * 4;
    static constexpr int kNumBars = 2 * kStages + kSBufs + 1;
    static constexpr int kSmemBytes = kOffBar + kNumBars * 8 + 32 + 1024;  // + TMEM slot, flags, alignment slack
    static_assert(kCtas * (kSmemBytes + 1024) <= 228 * 1024, "shared memory budget");
};

__device__ __forceinline__ unsigned long long pack2(float a, float b) {
    return (unsigned long long)__float_as_uint(a) | (unsigned long long)__float_as_uint(b) << 32;
}
// Both halves of y: y + m * p, rounded once each.
__device__ __forceinline__ void fma2(unsigned long long& y, unsigned long long m, unsigned long long p) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(y) : "l"(m), "l"(p));
}

template <int kD, class Map>
__global__ void __launch_bounds__(kFThreads, FDim<kD>::kCtas)
k_shift_f32_tc(const __grid_constant__ CUtensorMap pmap, const __grid_constant__ CUtensorMap pmap1,
               const float* X, unsigned long long* __restrict__ acc, float c_f, Map map, int* status) {
    using L = FDim<kD>;
    constexpr int kHalves = L::kHalves, kStages = L::kStages, kStageBytes = L::kStageBytes, kSBufs = L::kSBufs;
    constexpr float kBand = kScoreBand<kD>;
    constexpr uint32_t kCols = 128 * kSBufs;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* A1 = smem + L::kOffA1;
    uint8_t* Pst = smem + L::kOffP;
    uint64_t* bars = (uint64_t*)(smem + L::kOffBar);
    uint64_t* full = bars;                   // [kStages] pixel tile landed
    uint64_t* empty = full + kStages;        // [kStages] the tile's four warps are done with it and its S buffer
    uint64_t* s_full = empty + kStages;      // [kSBufs] scores of a tile complete
    uint64_t* aux = s_full + kSBufs;         // drain barrier of the MMA issuer
    uint32_t* tmem_slot = (uint32_t*)(bars + L::kNumBars);
    volatile int* abort = (volatile int*)(tmem_slot + 1);
    volatile int* a1_seq = (volatile int*)(tmem_slot + 4);  // [4] items whose rows of A1 a warp has written

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 4);
        }
        for (int b = 0; b < kSBufs; ++b) mbar_init(&s_full[b], 1);
        mbar_init(aux, 1);
        *abort = 0;
        for (int k = 0; k < 4; ++k) a1_seq[k] = 0;
        fence_mbar_init();
    }
    if (warp == kFWarpTma && lane == 0) {
        tma_prefetch_desc(&pmap);
        if (kHalves > 1) tma_prefetch_desc(&pmap1);
    }
    if (warp == kFWarpG1) {
        tmem_alloc(tmem_slot, kCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    grid_release();  // TMEM is held
    grid_wait();
    const int items = map.init() ? map.total() : 0;

    if (warp == kFWarpTma) {
        // ------------------------------------------------ TMA producer
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
    } else if (warp == kFWarpG1) {
        // ------------------------------------------------ MMA issuer
        const uint64_t dA1 = desc_sw128(smem_u32(A1), 16, 1024);
        const uint64_t dP1 = desc_sw128(smem_u32(Pst), 16, 1024);
        constexpr uint32_t id1 = idesc_bf16(128, 128, 0, 0);
        constexpr uint64_t kT = kTileBytes >> 4;
        Ring<kStages> st, old;  // stages of tile g and of tile g - kSBufs
        Ring<kSBufs> sb;
        bool ok = true;
        int g = 0, it = 0;
        for (int item = blockIdx.x; item < items && ok; item += gridDim.x, ++it) {
            const TcItem ii = map.item(item);
            if (!(ok = seq_wait4(a1_seq, it + 1, abort))) break;
            const uint64_t a = dA1 + (uint64_t)(it & 1) * kHalves * kT;
            for (int pt = ii.pt0; pt < ii.pt1; ++pt, ++g, st.advance(1), sb.advance(1)) {
                if (!(ok = warp_wait(&full[st.i], st.par, abort))) break;
                if (g >= kSBufs) {
                    if (!(ok = warp_wait(&empty[old.i], old.par, abort))) break;
                    old.advance(1);
                }
                tc_fence_after();
                const uint32_t tS = tmem + sb.i * 128;
                const uint64_t pb = dP1 + (uint64_t)st.i * kHalves * kT;
                mma_bf16_split3c_warp(tS, a, pb, id1);                            // Xh.Ph + Xh.Pm + Xl.Ph - c
                if (kHalves > 1) mma_bf16_split3_warp(tS, a + kT, pb + kT, id1);  // dimensions 16..31
                mma_commit_warp(&s_full[sb.i]);
            }
        }
        if (__any_sync(0xffffffffu, *abort)) {
            mma_commit_warp(aux);
            drain_wait(aux, 0);
        }
    } else {
        // ------------------------------------------------ seeds
        const int r = warp * 32 + lane;  // seed row
        const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
        float* px = reinterpret_cast<float*>(smem + L::kOffPx) + warp * 32 * L::kPxStride;
        Ring<kStages> st;
        Ring<kSBufs> sb;
        float* Xs = reinterpret_cast<float*>(smem + L::kOffX) + r * kD;  // [2][128][kD]
        int slot = -1, slot_n = -1, it = 0;
        // the lane's row of the seed operand of item number n (buffer n & 1)
        // and the seed's FP32 value
        auto load_seed = [&](int item, int n) {
            const TcItem ni = map.item(item);
            const int pos = ni.seed0 + r;
            slot_n = pos < ni.n_active ? ni.active[pos] : -1;
            float x[kD];
            load_seed_row<kD>(X, slot_n, x);
#pragma unroll
            for (int k = 0; k < kD; k += 4)
                *reinterpret_cast<float4*>(Xs + (n & 1) * 128 * kD + k) =
                    make_float4(x[k], x[k + 1], x[k + 2], x[k + 3]);
#pragma unroll
            for (int hf = 0; hf < kHalves; ++hf)
                write_a1_half(A1 + ((n & 1) * kHalves + hf) * kTileBytes, r, x + 16 * hf, c_f, hf == 0);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
                __threadfence_block();
                a1_seq[warp] = n + 1;
            }
        };
        if ((int)blockIdx.x < items) load_seed(blockIdx.x, 0);
        for (int item = blockIdx.x; item < items; item += gridDim.x, ++it) {
            if (__any_sync(0xffffffffu, *abort)) break;
            const TcItem ii = map.item(item);
            slot = slot_n;
            const float* x = Xs + (it & 1) * 128 * kD;
            // the next item's buffer: this warp saw every score of the item
            // that used it last
            if (item + (int)gridDim.x < items) load_seed(item + gridDim.x, it + 1);
            unsigned long long y[kD / 2];
            float cnt = 0.f;
#pragma unroll
            for (int k = 0; k < kD / 2; ++k) y[k] = 0ull;
            bool ok = true;
            for (int pt = ii.pt0; pt < ii.pt1; ++pt, st.advance(1), sb.advance(1)) {
                if (!(ok = warp_wait(&s_full[sb.i], sb.par, abort))) break;
                tc_fence_after();
                const uint32_t tS = tmem + sb.i * 128 + lane_base;
                const uint8_t* stage = Pst + st.i * kStageBytes;
                uint32_t need = 0u;
                {
                    float mx[4];
                    uint32_t v[32];
#pragma unroll
                    for (int p = 0; p < 4; ++p) tmem_ld32_max(tS + 32 * p, v, &mx[p]);
                    tmem_ld_wait();
                    if (__any_sync(0xffffffffu, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) >= -kBand)) {
#pragma unroll
                        for (int p = 0; p < 4; ++p)
                            if (__any_sync(0xffffffffu, mx[p] >= -kBand)) need |= 1u << p;
                    }
                }
                if (need) {
                    // the tile landed long ago; this wait makes it visible here
                    if (!(ok = warp_wait(&full[st.i], st.par, abort))) break;
                    do {
                        const int j = __ffs(need) - 1;
                        need &= need - 1u;
                        uint32_t v[32];
                        float mn;
                        tmem_ld32_minabs(tS + j * 32, v, &mn);
                        tmem_ld_wait();
                        // win: bit 31 - i: pixel i of the piece is in this lane's
                        // window (four chains of eight sign bits; a NaN score,
                        // whose sign is clear, is none)
                        uint32_t nm[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                        for (int i = 0; i < 8; ++i)
#pragma unroll
                            for (int e = 0; e < 4; ++e) nm[e] = __funnelshift_l(v[8 * e + i], nm[e], 1);
                        uint32_t win = ~((nm[0] << 24) | (nm[1] << 16) | (nm[2] << 8) | nm[3]);
                        if (!(fabsf(__uint_as_float(v[0])) <= INFINITY)) win = 0u;
                        if (__any_sync(0xffffffffu, mn < kBand)) {
                            uint32_t bm[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                            for (int i = 0; i < 8; ++i)
#pragma unroll
                                for (int e = 0; e < 4; ++e)
                                    bm[e] = __funnelshift_l(
                                        __float_as_uint(fabsf(__uint_as_float(v[8 * e + i])) - kBand), bm[e], 1);
                            uint32_t todo = (bm[0] << 24) | (bm[1] << 16) | (bm[2] << 8) | bm[3];
                            while (todo) {
                                const int i = __clz(todo);
                                const uint32_t bit = 0x80000000u >> i;
                                todo &= ~bit;
                                win = stage_dot<kD>(stage, j * 32 + i, x) >= c_f ? win | bit : win & ~bit;
                            }
                            __syncwarp();
                        }
                        const int left = ii.n - (pt * 128 + j * 32);  // pixels of the frame from this piece on
                        if (left < 32) win &= left > 0 ? 0xffffffffu << (32 - left) : 0u;
                        uint32_t any = __reduce_or_sync(0xffffffffu, win);
                        if (any == 0u) continue;
                        // the piece's pixels: lane i rebuilds pixel i
#pragma unroll
                        for (int hf = 0; hf < kHalves; ++hf) {
                            float p[16];
                            stage_pixel16(stage + hf * kTileBytes, j * 32 + lane, p);
#pragma unroll
                            for (int k = 0; k < 16; k += 4)
                                *reinterpret_cast<float4*>(px + lane * L::kPxStride + 16 * hf + k) =
                                    make_float4(p[k], p[k + 1], p[k + 2], p[k + 3]);
                        }
                        __syncwarp();
                        cnt += (float)__popc(win);
                        while (any) {
                            const int i = __clz(any);
                            any &= ~(0x80000000u >> i);
                            const float m = (win << i) & 0x80000000u ? 1.f : 0.f;
                            const unsigned long long mm = pack2(m, m);
                            const ulonglong2* pp = reinterpret_cast<const ulonglong2*>(px + i * L::kPxStride);
#pragma unroll
                            for (int k = 0; k < kD / 4; ++k) {
                                const ulonglong2 q = pp[k];
                                fma2(y[2 * k], mm, q.x);
                                fma2(y[2 * k + 1], mm, q.y);
                            }
                        }
                        __syncwarp();  // px is read before the next piece's is written
                    } while (need);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[st.i]);
            }
            if (!ok) break;
            if (slot >= 0 && cnt > 0.f) {
                unsigned long long* a = acc + (slot - ii.pix0 + ii.pk_row0) * (kD + 1);
#pragma unroll
                for (int k = 0; k < kD; ++k) {
                    const float yk = __uint_as_float((uint32_t)(y[k / 2] >> (32 * (k & 1))));
                    atomicAdd(a + k, (unsigned long long)__float2ll_rn(yk * kFixScale));
                }
                atomicAdd(a + kD, (unsigned long long)cnt);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kFWarpG1) tmem_dealloc(tmem, kCols);
    if (threadIdx.x == 0 && *abort) atomicOr(status, 2);
}

// Work items of one frame: seed tiles of 128 x the plain form's pixel chunks.
struct FSingleMap {
    const int32_t* active;
    const DevCounters* dc;
    int n, target;
    int n_active, tiles;
    ShiftSplit sp;
    __device__ __forceinline__ bool init() {
        if (dc->done) return false;
        n_active = dc->n_active;
        tiles = (n_active + 127) / 128;
        sp = shift_split(n_active, n, target);
        return true;
    }
    __device__ __forceinline__ int total() const { return tiles * sp.chunks; }
    __device__ __forceinline__ TcItem item(int i) const {
        int t, ch;
        tc_item_place(i, tiles, sp.chunks, &t, &ch);
        TcItem it;
        it.active = active;
        it.n_active = n_active;
        it.seed0 = t * 128;
        it.pt0 = ch * (sp.chunk_len / 128);
        it.pt1 = min((n + 127) / 128, it.pt0 + sp.chunk_len / 128);
        it.pk_row0 = 0;
        it.pix0 = 0;
        it.n = n;
        return it;
    }
};

// Work items of every iterating frame (tpc: pixels per chunk).
struct FBatchMap {
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
        const int n_active = states[f].dc.n_active, tpc = plan.tpc[f] / 128;
        int t, ch;
        tc_item_place(i - plan.item_off[f], (n_active + 127) / 128, plan.chunks[f], &t, &ch);
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

template <int D>
ms_status f32_tc_allow() {
    MS_CUDA(cudaFuncSetAttribute(k_shift_f32_tc<D, FSingleMap>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 FDim<D>::kSmemBytes));
    MS_CUDA(cudaFuncSetAttribute(k_shift_f32_tc<D, FBatchMap>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 FDim<D>::kSmemBytes));
    return MS_OK;
}

}  // namespace

ms_status f32_tc_setup(int D) { return D == 32 ? f32_tc_allow<32>() : f32_tc_allow<16>(); }

ms_status launch_shift_f32_tc(ms_ctx* ctx, const int32_t* active, float c) {
    FSingleMap map;
    map.active = active;
    map.dc = ctx->dc;
    map.n = (int)ctx->n;
    map.target = ctx->target_items;
    int* status = &ctx->dc->status;
    if (ctx->Dp == 32)
        MS_CUDA(launch_after(k_shift_f32_tc<32, FSingleMap>, ctx->num_sms * FDim<32>::kCtas, kFThreads,
                             FDim<32>::kSmemBytes, ctx->stream, ctx->pmap, ctx->pmap1, ctx->X, ctx->acc, c, map, status));
    else
        MS_CUDA(launch_after(k_shift_f32_tc<16, FSingleMap>, ctx->num_sms * FDim<16>::kCtas, kFThreads,
                             FDim<16>::kSmemBytes, ctx->stream, ctx->pmap, ctx->pmap1, ctx->X, ctx->acc, c, map, status));
    return MS_OK;
}

ms_status launch_shift_f32_tc_batch(const CUtensorMap& pmap, const CUtensorMap& pmap1, int Dp, const float* X,
                                    unsigned long long* acc, float c, const BFrame* frames, const BState* states,
                                    BPlan plan, const int32_t* act0, const int32_t* act1, int nf, int* status,
                                    int num_sms, cudaStream_t st) {
    FBatchMap map;
    map.frames = frames;
    map.states = states;
    map.plan = plan;
    map.act0 = act0;
    map.act1 = act1;
    map.nf = nf;
    map.total_ = 0;
    if (Dp == 32)
        k_shift_f32_tc<32, FBatchMap><<<num_sms * FDim<32>::kCtas, kFThreads, FDim<32>::kSmemBytes, st>>>(
            pmap, pmap1, X, acc, c, map, status);
    else
        k_shift_f32_tc<16, FBatchMap><<<num_sms * FDim<16>::kCtas, kFThreads, FDim<16>::kSmemBytes, st>>>(
            pmap, pmap1, X, acc, c, map, status);
    MS_LAUNCH("k_shift_f32_tc(batch)");
    return MS_OK;
}

}  // namespace ms
