// Prune/merge of converged modes (the prune/merge step of Algorithm 2) and OSOP coverage.
//
// Merge rule: candidates (the round's converged seeds) are visited in order of
// support descending, then seed order ascending; a candidate is kept when its
// cosine to every mode kept so far is < merge_cos. Each decision is the FP64
// one: FP32 dot products decide pairs that clear the threshold by more than
// kEpsF32 and the rest are recomputed in FP64.
//
// The sequential greedy is evaluated in parallel as the lexicographically
// first independent set of the conflict graph: candidates that conflict with a
// previously kept mode are removed up front; then, sweep by sweep, a candidate
// is removed as soon as a higher-ranked conflicting candidate is kept, and kept
// as soon as every higher-ranked conflicting candidate is removed. This fixed
// point equals the sequential greedy result; a single-warp sequential pass
// finishes any candidates still undecided after a bounded number of sweeps.
#include "ms_batch.cuh"
#include "ms_device.cuh"

namespace ms {
namespace {

constexpr int kMT = 128;  // threads per merge block
constexpr int kMergeOne = 4096;  // candidates that one block resolves and appends
constexpr int kMergeScan = 1024; // the same with more conflicts than are stored
constexpr int kVT = 64;   // vectors per shared-memory tile

__global__ void k_collect(const uint8_t* __restrict__ sstate, int m, int32_t* __restrict__ cand,
                          DevCounters* dc) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    const bool c = s < m && sstate[s] == kConverged;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned b = __ballot_sync(0xffffffffu, c);
    int base = 0;
    if (lane == 0 && b) base = atomicAdd(&dc->n_cand, __popc(b));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (c) cand[base + __popc(b & ((1u << lane) - 1u))] = s;
}

// Rank of every candidate in (support desc, seed order asc): the count of
// candidates ahead of it. Block (x, y) counts candidate block x against slice y
// of all candidates and adds its partial count (ranks start at 0). A candidate
// is ahead of another exactly when its key support * 2^32 + (2^32 - 1 - order)
// is larger (seed orders are distinct within a frame).
__device__ __forceinline__ unsigned long long rank_key(int32_t support, int32_t order) {
    return ((unsigned long long)(uint32_t)support << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)order);
}

__global__ void k_rank(const int32_t* __restrict__ cand, int k, const int32_t* __restrict__ support,
                       const int32_t* __restrict__ order, int32_t* __restrict__ cand_rank) {
    __shared__ unsigned long long s_key[256];
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned long long ka = a < k ? rank_key(support[cand[a]], order[cand[a]]) : 0ull;
    const int lo = (int)((int64_t)blockIdx.y * k / gridDim.y), hi = (int)((int64_t)(blockIdx.y + 1) * k / gridDim.y);
    int r = 0;
    for (int base = lo; base < hi; base += 256) {
        const int b = base + threadIdx.x;
        if (b < hi) s_key[threadIdx.x] = rank_key(support[cand[b]], order[cand[b]]);
        __syncthreads();
        const int lim = min(256, hi - base);
        for (int j = 0; j < lim; ++j) r += s_key[j] > ka;
        __syncthreads();
    }
    if (a < k && r) atomicAdd(&cand_rank[a], r);
}

// rank_cand inverts cand_rank; each candidate's position is copied to its
// rank's row of Xr (the merge reads the candidates in rank order).
template <int Dp>
__global__ void k_rank_invert_xr(const int32_t* __restrict__ cand_rank, int k, const int32_t* __restrict__ cand,
                                 const float* __restrict__ X, int32_t* __restrict__ rank_cand, float* __restrict__ Xr) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= k) return;
    const int r = cand_rank[a];
    rank_cand[r] = a;
    const float4* src = reinterpret_cast<const float4*>(X + (int64_t)cand[a] * Dp);
    float4* dst = reinterpret_cast<float4*>(Xr + (int64_t)r * Dp);
#pragma unroll
    for (int q = 0; q < Dp / 4; ++q) dst[q] = src[q];
}

template <int Dp>
__device__ __forceinline__ void load_vec(float* dst, const float* src) {
#pragma unroll
    for (int k = 0; k < Dp; k += 4) {
        const float4 v = *reinterpret_cast<const float4*>(src + k);
        dst[k] = v.x; dst[k + 1] = v.y; dst[k + 2] = v.z; dst[k + 3] = v.w;
    }
}

// What a look at a candidate's stored conflicts says of it: removed when a kept
// one is among them, kept when all are removed, else still undecided.
__device__ __forceinline__ uint8_t merge_look(const int32_t* conf, int deg, const volatile uint8_t* st) {
    bool all_removed = true;
    for (int j = 0; j < deg; ++j) {
        const uint8_t s = st[conf[j]];
        if (s == kKept) return kRemoved;
        if (s == kUndecided) all_removed = false;
    }
    return all_removed ? kKept : kUndecided;
}

// The same for a candidate, of rank r, with more conflicts than were stored: the
// candidates ranked above it are tested again, in rank order. Threads take
// candidates by rank: a warp's then read the same few higher ranks, whose positions
// lie in a row in Xr (by candidate, in pixel order, that look took four times as
// long: 2.8 ms for 4096 candidates of one cell).
template <int Dp>
__device__ __forceinline__ uint8_t merge_look_all(int r, const float* Xr, const int32_t* __restrict__ rank_cand,
                                                  const volatile uint8_t* st, float thr_f, double thr) {
    bool all_removed = true;
    float x[Dp];
    load_vec<Dp>(x, Xr + (int64_t)r * Dp);
    for (int rb = 0; rb < r; ++rb) {
        const uint8_t s = st[rank_cand[rb]];
        if (s == kRemoved) continue;
        if (!cos_at_least<Dp>(x, Xr + (int64_t)rb * Dp, thr_f, thr)) continue;
        if (s == kKept) return kRemoved;
        all_removed = false;
    }
    return all_removed ? kKept : kUndecided;
}

template <int Dp>
__global__ void __launch_bounds__(kMT)
k_merge_resolve(const float* __restrict__ Xr, int k, const int32_t* __restrict__ rank_cand, uint8_t* cand_state,
                const int32_t* __restrict__ conf_deg, const int32_t* __restrict__ conf,
                float thr_f, double thr, DevCounters* dc) {
    const int r = blockIdx.x * kMT + threadIdx.x;
    if (r >= k) return;
    const int a = rank_cand[r];
    volatile uint8_t* st = cand_state;
    if (st[a] != kUndecided) return;
    const int deg = conf_deg[a];
    const uint8_t d = deg <= kMergeCap ? merge_look(conf + (int64_t)a * kMergeCap, deg, st)
                                       : merge_look_all<Dp>(r, Xr, rank_cand, st, thr_f, thr);
    if (d != kUndecided)
        st[a] = d;
    else
        atomicAdd(&dc->undecided, 1);
}

// Exact sequential greedy for whatever is still undecided (one warp).
template <int Dp>
__global__ void k_merge_sequential(const float* __restrict__ X, const int32_t* __restrict__ cand,
                                   int k, const int32_t* __restrict__ rank_cand, uint8_t* cand_state,
                                   float thr_f, double thr) {
    volatile uint8_t* st = cand_state;
    const int lane = threadIdx.x;
    for (int r = 0; r < k; ++r) {
        const int a = rank_cand[r];
        if (st[a] != kUndecided) continue;
        const float* xa = X + (int64_t)cand[a] * Dp;
        bool hit = false;
        for (int rb = lane; rb < r && !hit; rb += 32) {
            const int b = rank_cand[rb];
            if (st[b] == kKept && cos_at_least<Dp>(xa, X + (int64_t)cand[b] * Dp, thr_f, thr)) hit = true;
        }
        const bool any = __any_sync(0xffffffffu, hit);
        if (lane == 0) st[a] = any ? kRemoved : kKept;
        __syncwarp();
    }
}

// Kept candidates are appended to the mode list in rank order, by a block of
// 1024 threads.
template <int Dp>
__device__ __forceinline__ void merge_append(const float* __restrict__ X, const int32_t* __restrict__ cand,
                                             const int32_t* __restrict__ rank_cand, int k,
                                             const volatile uint8_t* cand_state, const int32_t* __restrict__ support,
                                             float* modes, int32_t* __restrict__ mode_support, DevCounters* dc) {
    __shared__ int32_t warp_excl[32];
    __shared__ int32_t s_total;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int base = dc->n_kept;
    int carry = 0;
    for (int r0 = 0; r0 < k; r0 += 1024) {
        const int r = r0 + tid;
        const int a = r < k ? rank_cand[r] : -1;
        const bool flag = a >= 0 && cand_state[a] == kKept;
        const unsigned bal = __ballot_sync(0xffffffffu, flag);
        if (lane == 0) warp_excl[wid] = __popc(bal);
        __syncthreads();
        if (wid == 0) {
            const int w = warp_excl[lane];
            int incl = w;
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            warp_excl[lane] = incl - w;
            if (lane == 31) s_total = incl;
        }
        __syncthreads();
        if (flag) {
            const int dst = base + carry + warp_excl[wid] + __popc(bal & ((1u << lane) - 1u));
            const int slot = cand[a];
            const float4* src = reinterpret_cast<const float4*>(X + (int64_t)slot * Dp);
            float4* out = reinterpret_cast<float4*>(modes + (int64_t)dst * Dp);
            for (int q = 0; q < Dp / 4; ++q) out[q] = src[q];
            mode_support[dst] = support[slot];
        }
        carry += s_total;
        __syncthreads();
    }
    if (tid == 0) dc->n_kept = base + carry;
}

template <int Dp>
__global__ void __launch_bounds__(1024)
k_merge_append(const float* __restrict__ X, const int32_t* __restrict__ cand,
               const int32_t* __restrict__ rank_cand, int k, const uint8_t* __restrict__ cand_state,
               const int32_t* __restrict__ support, float* __restrict__ modes,
               int32_t* __restrict__ mode_support, DevCounters* dc) {
    merge_append<Dp>(X, cand, rank_cand, k, cand_state, support, modes, mode_support, dc);
}

// The whole resolution and the append in one block, for up to kMergeOne
// candidates. Sweeps until nothing is undecided: each decides at least the
// undecided candidate of the lowest rank, so k of them always suffice (two to
// four do). With eight sweeps in launches of their own, each with its counter's
// reset, the host's look at the count and the append's launch, a round's merge
// and coverage took 131 to 158 us for 128 to 2048 candidates; so 89 to 108 us. A
// block's sweep grows with k / 1024 (139 against 183 us at 4096 candidates, no
// gain expected at 8192), so larger rounds keep the launches.
// Of candidates with more conflicts than are stored the line is kMergeScan: a look
// at one of them tests the candidates ranked above it one by one. 947 candidates of
// six cells: 302 us here, 363 us in launches; 3880: 2.0 ms here, 0.89 ms in launches
// over all SMs. The block leaves such a round undecided (dc->undecided = k).
// Xr lies in the modes' rows that the append writes, after the last look.
template <int Dp>
__global__ void __launch_bounds__(1024)
k_merge_one(const float* __restrict__ X, const float* Xr, const int32_t* __restrict__ cand, int k,
            const int32_t* __restrict__ rank_cand, uint8_t* cand_state, const int32_t* __restrict__ conf_deg,
            const int32_t* __restrict__ conf, float thr_f, double thr, const int32_t* __restrict__ support,
            float* modes, int32_t* __restrict__ mode_support, DevCounters* dc) {
    volatile uint8_t* st = cand_state;
    bool over = false;
    if (k > kMergeScan) {
        for (int a = threadIdx.x; a < k; a += 1024) over |= conf_deg[a] > kMergeCap;
        over = __syncthreads_or(over);
    }
    if (threadIdx.x == 0) dc->undecided = over ? k : 0;
    if (over) return;
    for (int sweep = 0; sweep < k; ++sweep) {
        bool open = false;
        for (int r = threadIdx.x; r < k; r += 1024) {
            const int a = rank_cand[r];
            if (st[a] != kUndecided) continue;
            const int deg = conf_deg[a];
            const uint8_t d = deg <= kMergeCap ? merge_look(conf + (int64_t)a * kMergeCap, deg, st)
                                               : merge_look_all<Dp>(r, Xr, rank_cand, st, thr_f, thr);
            if (d != kUndecided) st[a] = d;
            else open = true;
        }
        if (!__syncthreads_or(open)) break;
    }
    merge_append<Dp>(X, cand, rank_cand, k, st, support, modes, mode_support, dc);
}

// Slices of an O(outer x inner) loop so that the grid fills about four waves
// of the GPU: the candidate blocks alone are often fewer than the SMs.
unsigned inner_slices(int outer_blocks, int inner, int num_sms) {
    int sl = (4 * num_sms + outer_blocks - 1) / outer_blocks;
    const int max_sl = (inner + kVT - 1) / kVT;
    sl = sl > max_sl ? max_sl : sl;
    sl = sl > 64 ? 64 : sl;
    return (unsigned)(sl < 1 ? 1 : sl);
}

// The candidates' positions in rank order: in the modes' rows that are still free.
float* merge_xr(const ms_ctx* ctx) { return ctx->modes + (int64_t)ctx->n_kept * ctx->Dp; }

template <int Dp>
ms_status merge_prepare_t(ms_ctx* ctx, int32_t k) {
    const float thr_f = (float)ctx->cfg.merge_cos;
    const double thr = ctx->cfg.merge_cos;
    const unsigned g256 = (unsigned)((k + 255) / 256);
    MS_CUDA(cudaMemsetAsync(ctx->cand_rank, 0, sizeof(int32_t) * (size_t)k, ctx->stream));
    MS_CUDA(cudaMemsetAsync(ctx->cand_state, kUndecided, (size_t)k, ctx->stream));
    MS_CUDA(cudaMemsetAsync(ctx->conf_deg, 0, sizeof(int32_t) * (size_t)k, ctx->stream));
    k_rank<<<dim3(g256, inner_slices((int)g256, k, ctx->num_sms)), 256, 0, ctx->stream>>>(
        ctx->cand, k, ctx->support, ctx->seed_order, ctx->cand_rank);
    MS_LAUNCH("k_rank");
    MS_CUDA(cudaMemsetAsync(ctx->removed_r, 0, (size_t)k, ctx->stream));
    float* Xr = merge_xr(ctx);
    k_rank_invert_xr<Dp><<<g256, 256, 0, ctx->stream>>>(ctx->cand_rank, k, ctx->cand, ctx->X, ctx->rank_cand, Xr);
    MS_LAUNCH("k_rank_invert_xr");
    const ms_status s = launch_merge_tc_single(ctx->pmap, ctx->pmap1, ctx->Pk, pk_half_rows(ctx), ctx->Ck, ctx->n_pad,
                                               Dp, k, ctx->n_kept, Xr, ctx->modes, ctx->rank_cand, ctx->cand_state,
                                               ctx->removed_r, ctx->conf_deg, ctx->conf, thr_f, thr, ctx->num_sms,
                                               &ctx->dc->status, ctx->stream);
    ctx->launches += 4 + (ctx->n_kept > 0 ? 1 : 0);
    return s;
}

}  // namespace

ms_status launch_collect(ms_ctx* ctx) {
    MS_CUDA(cudaMemsetAsync(&ctx->dc->n_cand, 0, sizeof(int32_t), ctx->stream));
    if (ctx->m_round <= 0) return MS_OK;
    k_collect<<<(unsigned)((ctx->m_round + 255) / 256), 256, 0, ctx->stream>>>(ctx->sstate, ctx->m_round,
                                                                             ctx->cand, ctx->dc);
    MS_LAUNCH("k_collect");
    ctx->launches += 1;
    return MS_OK;
}

ms_status launch_merge_prepare(ms_ctx* ctx, int32_t k) {
    if (k <= 0) return MS_OK;
    return ctx->Dp == 16 ? merge_prepare_t<16>(ctx, k) : merge_prepare_t<32>(ctx, k);
}

ms_status launch_merge_resolve(ms_ctx* ctx, int32_t k, int sweeps) {
    if (k <= 0) return MS_OK;
    const float thr_f = (float)ctx->cfg.merge_cos;
    const double thr = ctx->cfg.merge_cos;
    const unsigned gm = (unsigned)((k + kMT - 1) / kMT);
    for (int s = 0; s < sweeps; ++s) {
        MS_CUDA(cudaMemsetAsync(&ctx->dc->undecided, 0, sizeof(int32_t), ctx->stream));
        if (ctx->Dp == 16)
            k_merge_resolve<16><<<gm, kMT, 0, ctx->stream>>>(merge_xr(ctx), k, ctx->rank_cand, ctx->cand_state,
                                                             ctx->conf_deg, ctx->conf, thr_f, thr, ctx->dc);
        else
            k_merge_resolve<32><<<gm, kMT, 0, ctx->stream>>>(merge_xr(ctx), k, ctx->rank_cand, ctx->cand_state,
                                                             ctx->conf_deg, ctx->conf, thr_f, thr, ctx->dc);
        MS_LAUNCH("k_merge_resolve");
        ctx->launches += 1;
    }
    return MS_OK;
}

ms_status launch_merge_sequential(ms_ctx* ctx, int32_t k) {
    if (k <= 0) return MS_OK;
    const float thr_f = (float)ctx->cfg.merge_cos;
    const double thr = ctx->cfg.merge_cos;
    if (ctx->Dp == 16)
        k_merge_sequential<16><<<1, 32, 0, ctx->stream>>>(ctx->X, ctx->cand, k, ctx->rank_cand,
                                                          ctx->cand_state, thr_f, thr);
    else
        k_merge_sequential<32><<<1, 32, 0, ctx->stream>>>(ctx->X, ctx->cand, k, ctx->rank_cand,
                                                          ctx->cand_state, thr_f, thr);
    MS_LAUNCH("k_merge_sequential");
    ctx->launches += 1;
    return MS_OK;
}

bool merge_in_one(int32_t k) { return k <= kMergeOne; }

ms_status launch_merge_one(ms_ctx* ctx, int32_t k) {
    if (k <= 0) return MS_OK;
    const float thr_f = (float)ctx->cfg.merge_cos;
    const double thr = ctx->cfg.merge_cos;
    if (ctx->Dp == 16)
        k_merge_one<16><<<1, 1024, 0, ctx->stream>>>(ctx->X, merge_xr(ctx), ctx->cand, k, ctx->rank_cand,
                                                     ctx->cand_state, ctx->conf_deg, ctx->conf, thr_f, thr,
                                                     ctx->support, ctx->modes, ctx->mode_support, ctx->dc);
    else
        k_merge_one<32><<<1, 1024, 0, ctx->stream>>>(ctx->X, merge_xr(ctx), ctx->cand, k, ctx->rank_cand,
                                                     ctx->cand_state, ctx->conf_deg, ctx->conf, thr_f, thr,
                                                     ctx->support, ctx->modes, ctx->mode_support, ctx->dc);
    MS_LAUNCH("k_merge_one");
    ctx->launches += 1;
    return MS_OK;
}

ms_status launch_merge_append(ms_ctx* ctx, int32_t k) {
    if (k <= 0) return MS_OK;
    if (ctx->Dp == 16)
        k_merge_append<16><<<1, 1024, 0, ctx->stream>>>(ctx->X, ctx->cand, ctx->rank_cand, k,
                                                        ctx->cand_state, ctx->support, ctx->modes,
                                                        ctx->mode_support, ctx->dc);
    else
        k_merge_append<32><<<1, 1024, 0, ctx->stream>>>(ctx->X, ctx->cand, ctx->rank_cand, k,
                                                        ctx->cand_state, ctx->support, ctx->modes,
                                                        ctx->mode_support, ctx->dc);
    MS_LAUNCH("k_merge_append");
    ctx->launches += 1;
    return MS_OK;
}

ms_status launch_cover(ms_ctx* ctx, int32_t k, int32_t k0, int32_t k1) {
    if (k <= 0 || ctx->n == 0) return MS_OK;
    const ms_status s = launch_cover_tc_single(ctx->pmap, ctx->pmap1, ctx->Pk, pk_half_rows(ctx), k > k0 ? k : k0,
                                               ctx->Mk, ctx->n_pad, ctx->Dp, ctx->modes, k0, k1, (int)ctx->n, ctx->P32,
                                               ctx->pix, ctx->emb, ctx->d, ctx->cfg.bandwidth_cos, ctx->covered,
                                               &ctx->dc->n_uncovered, ctx->num_sms, &ctx->dc->status, ctx->stream);
    ctx->launches += k1 > k0 ? 2 : 1;
    return s;
}

}  // namespace ms
