// OSOP seed selection (the seed-selection step of Algorithm 2): the next `want` uncovered
// positions of the frame's fixed seed order pi(j) = (b + a j) mod n.
//
// The batch is the first `want` uncovered positions in seed order, exactly as
// a sequential scan would take them, and each seed keeps its rank in that
// order (seed_order; the merge's ties use it). Its slot, though, is its rank
// in pixel order: neighbouring slots are neighbouring pixels, so a shift
// item's 128 seeds come from the same few cells and most of its pixel tiles
// hold no pair of any window (ms_shift_tc.cu).
//
// Four passes, each over blocks of 1024 positions or pixels: count the
// uncovered positions, take them (block prefix from the counts), count the
// taken pixels, write their slots. Up to kFewSeeds seeds that are found within
// few positions are one CTA's work: it needs no pass over the pixels, as its
// seeds are ranked among themselves.
#include "ms_device.cuh"
#include "ms_internal.cuh"

namespace ms {
namespace {

constexpr int kSelThreads = 1024;
constexpr uint8_t kTaken = 2;       // covered[]: drawn by the running selection
static_assert(kSelThreads == kFewThreads, "blocks of one size");

// Exclusive prefix of `flag` over the block's threads; *total: the block's count.
__device__ __forceinline__ int block_rank(bool flag, int* total) {
    __shared__ int32_t s_cnt[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned bal = __ballot_sync(0xffffffffu, flag);
    __syncthreads();
    if (lane == 0) s_cnt[wid] = __popc(bal);
    __syncthreads();
    const int c = s_cnt[lane];
    int incl = c;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    *total = __shfl_sync(0xffffffffu, incl, 31);
    return __shfl_sync(0xffffffffu, incl - c, wid) + __popc(bal & ((1u << lane) - 1u));
}

// Sum of counts[0..m) by the whole block (every thread gets it).
__device__ __forceinline__ int block_sum(const int32_t* __restrict__ counts, int m) {
    __shared__ int32_t s_sum[32];
    int v = 0;
    for (int i = threadIdx.x; i < m; i += kSelThreads) v += counts[i];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = v;
    __syncthreads();
    v = s_sum[threadIdx.x & 31];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

struct SelArgs {
    int32_t n;
    uint64_t a, b;
    int32_t want;
    int Dp;
    const float* P32;
    uint8_t* covered;
    int32_t* order_of;   // [n] draw number of a taken pixel (scratch)
    int32_t* counts;     // per block of 1024 (scratch)
    float* X;
    unsigned long long* acc;
    int32_t* seed_order;
    int32_t* active0;
    uint8_t* sstate;
    int32_t* seed_log;
    DevCounters* dc;
};

__device__ __forceinline__ int32_t sel_pixel(const SelArgs& s, int32_t pos) {
    return (int32_t)((s.b + s.a * (uint64_t)pos) % (uint64_t)s.n);
}

// Position pos takes draw r of this batch when it is uncovered and r < want.
__device__ __forceinline__ void sel_take(const SelArgs& s, int32_t p, int32_t pos, int32_t r, int32_t drawn) {
    s.covered[p] = kTaken;
    s.order_of[p] = drawn + r;
    s.seed_log[drawn + r] = p;
    if (r == s.want - 1) s.dc->cursor_next = pos + 1;
}

__device__ __forceinline__ void sel_write(const SelArgs& s, int32_t p, int32_t slot, int32_t order) {
    s.covered[p] = 1;
    s.seed_order[slot] = order;
    s.active0[slot] = slot;
    s.sstate[slot] = kMoving;
    const float4* src = reinterpret_cast<const float4*>(s.P32 + (int64_t)p * s.Dp);
    float4* dst = reinterpret_cast<float4*>(s.X + (int64_t)slot * s.Dp);
    for (int k = 0; k < s.Dp / 4; ++k) dst[k] = src[k];
}

// The block clears the window sums of slots [first, first + count).
__device__ __forceinline__ void sel_clear(const SelArgs& s, int32_t first, int32_t count) {
    unsigned long long* a = s.acc + (int64_t)first * (s.Dp + 1);
    for (int64_t i = threadIdx.x; i < (int64_t)count * (s.Dp + 1); i += kSelThreads) a[i] = 0ull;
}

__device__ __forceinline__ void sel_finish(const SelArgs& s, int32_t taken) {
    DevCounters* dc = s.dc;
    dc->cursor = taken == s.want ? dc->cursor_next : s.n;
    dc->drawn += taken;
    dc->n_seeded = taken;
    dc->m_round = taken;
    dc->n_active = taken;
    dc->n_next = 0;
    dc->conv_new = 0;
    dc->conv_total = 0;
    dc->fail_total = 0;
    dc->iters = 0;
    dc->done = taken == 0;
    dc->n_uncovered -= taken;
}

__global__ void __launch_bounds__(kSelThreads) k_seed_count(SelArgs s) {
    const int32_t pos = s.dc->cursor + blockIdx.x * kSelThreads + threadIdx.x;
    const int c = __syncthreads_count(pos < s.n && s.covered[sel_pixel(s, pos)] == 0);
    if (threadIdx.x == 0) s.counts[blockIdx.x] = c;
}

__global__ void __launch_bounds__(kSelThreads) k_seed_take(SelArgs s) {
    const int32_t drawn = s.dc->drawn;
    const int32_t pos = s.dc->cursor + blockIdx.x * kSelThreads + threadIdx.x;
    const int before = block_sum(s.counts, blockIdx.x);
    if (before >= s.want) return;
    int32_t p = -1;
    bool flag = false;
    if (pos < s.n) {
        p = sel_pixel(s, pos);
        flag = s.covered[p] == 0;
    }
    int total;
    const int r = before + block_rank(flag, &total);
    if (flag && r < s.want) sel_take(s, p, pos, r, drawn);
}

__global__ void __launch_bounds__(kSelThreads) k_slot_count(SelArgs s) {
    const int32_t p = blockIdx.x * kSelThreads + threadIdx.x;
    const int c = __syncthreads_count(p < s.n && s.covered[p] == kTaken);
    if (threadIdx.x == 0) s.counts[blockIdx.x] = c;
}

__global__ void __launch_bounds__(kSelThreads) k_slot_write(SelArgs s) {
    const int32_t p = blockIdx.x * kSelThreads + threadIdx.x;
    const int before = block_sum(s.counts, blockIdx.x);
    const bool flag = p < s.n && s.covered[p] == kTaken;
    int total;
    const int r = before + block_rank(flag, &total);
    if (flag) sel_write(s, p, r, s.order_of[p]);
    sel_clear(s, before, total);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) sel_finish(s, before + total);
}

// Up to kFewSeeds seeds: one CTA takes the positions 1024 at a time and ranks
// what it took.
__global__ void __launch_bounds__(kFewThreads) k_seed_few(SelArgs s) {
    __shared__ FewSeeds few;
    const int32_t cursor = s.dc->cursor, drawn = s.dc->drawn;
    int32_t taken = 0;
    for (int32_t base = cursor; base < s.n && taken < s.want; base += kFewThreads) {
        const int32_t pos = base + threadIdx.x;
        int32_t p = -1;
        bool flag = false;
        if (pos < s.n) {
            p = sel_pixel(s, pos);
            flag = s.covered[p] == 0;
        }
        int total;
        const int r = taken + block_rank(flag, &total);
        if (flag && r < s.want) {
            few.pix[r] = p;
            s.seed_log[drawn + r] = p;
            if (r == s.want - 1) s.dc->cursor_next = pos + 1;
        }
        taken = min(taken + total, s.want);
    }
    __syncthreads();
    int rank[2];
    few_ranks(few, taken, s.n, rank);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int t = threadIdx.x + k * kFewThreads;
        if (t < taken) sel_write(s, few.pix[t], rank[k], drawn + t);
    }
    sel_clear(s, 0, taken);
    if (threadIdx.x == 0) sel_finish(s, taken);
}

// Whether k_seed_few is the shorter form. A call with its readback takes about 17
// us and 9 us per 1024 seeds, and 1 to 1.5 us per 1024 positions, of which as many
// are expected as the uncovered share of the positions left says; the four passes
// take about 30 us and 1 us per 61,000 pixels. (128 seeds of 131,072 pixels, nothing
// covered: 18 us against 31; of 4 million 23 against 98; with all but 1% covered
// 30 against 32 and 41 against 94; 1024 seeds then 114 against 33.)
bool few_seeds(const ms_ctx* ctx, int32_t want) {
    if (want > kFewSeeds || ctx->uncovered <= 0) return false;
    const int64_t left = ctx->n - ctx->hc->cursor;
    return 4 * (int64_t)want + want * left / ctx->uncovered <= 8192 + ctx->n / 96;
}

}  // namespace

ms_status launch_seed_select(ms_ctx* ctx, int32_t want) {
    const SelArgs s{(int32_t)ctx->n, (uint64_t)ctx->perm_a, (uint64_t)ctx->perm_b, want, ctx->Dp, ctx->P32,
                    ctx->covered, ctx->cand_rank, ctx->block_tmp, ctx->X, ctx->acc, ctx->seed_order,
                    ctx->active[0], ctx->sstate, ctx->seed_log, ctx->dc};
    if (few_seeds(ctx, want)) {
        k_seed_few<<<1, kFewThreads, 0, ctx->stream>>>(s);
        MS_LAUNCH("k_seed_few");
        ctx->launches += 1;
        return MS_OK;
    }
    const unsigned nb = (unsigned)((ctx->n + kSelThreads - 1) / kSelThreads);
    k_seed_count<<<nb, kSelThreads, 0, ctx->stream>>>(s);
    MS_LAUNCH("k_seed_count");
    k_seed_take<<<nb, kSelThreads, 0, ctx->stream>>>(s);
    MS_LAUNCH("k_seed_take");
    k_slot_count<<<nb, kSelThreads, 0, ctx->stream>>>(s);
    MS_LAUNCH("k_slot_count");
    k_slot_write<<<nb, kSelThreads, 0, ctx->stream>>>(s);
    MS_LAUNCH("k_slot_write");
    ctx->launches += 4;
    return MS_OK;
}

}  // namespace ms
