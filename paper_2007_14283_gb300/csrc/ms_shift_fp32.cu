// Shift iteration, plain FP32 form (the shift loop of Algorithm 2; Eq. 6-8, 11).
//
// For every active seed x: y = sum of p_i over the window {i : x.p_i >= c},
// cnt = |window|; then x' = y / ||y|| and the FP64 norm ||x' - x|| decides
// convergence. Sec. 3.2.1's dense form is used (every pixel is tested against
// the kernel, no neighbour search), but the seed-by-pixel matrix is never
// materialised: pixels stream through shared memory and each thread keeps its
// seeds' sums in registers.
//
// Launch shape: a persistent grid. Each launch reads the active-seed count on
// the device and splits the work into (seed tile of 256) x (pixel chunk)
// items, so successive iterations can be queued without reading counts back.
// Each item adds its FP32 window sums into per-seed 64-bit fixed-point
// accumulators (units of 2^-36). Integer addition is associative, so the
// totals do not depend on the order in which items finish: runs are
// deterministic, and the finalize step reads one word per component.
#include "ms_batch.cuh"
#include "ms_device.cuh"

namespace ms {
namespace {

constexpr float kFixScale = 68719476736.0f;      // 2^36

// What a work item covers: a tile of the frame's active seeds and the pixel
// rows [p_begin, p_end) of P32.
struct F32Item {
    const int32_t* active;
    int n_active;
    int seed0;
    int64_t p_begin, p_end;
};

// Work items of one frame: seed tiles of 256 x pixel chunks.
struct F32SingleMap {
    const int32_t* active;
    const DevCounters* dc;
    int n, target;
    int n_active;
    ShiftSplit sp;
    __device__ __forceinline__ bool init() {
        if (dc->done) return false;
        n_active = dc->n_active;
        sp = shift_split(n_active, n, target);
        return true;
    }
    __device__ __forceinline__ int total() const { return sp.tiles * sp.chunks; }
    __device__ __forceinline__ F32Item item(int i) const {
        const int t = i / sp.chunks, ch = i - t * sp.chunks;
        F32Item it;
        it.active = active;
        it.n_active = n_active;
        it.seed0 = t * kSeedsPerTile;
        it.p_begin = (int64_t)ch * sp.chunk_len;
        it.p_end = min((int64_t)n, it.p_begin + sp.chunk_len);
        return it;
    }
};

template <int Dp, class Map>
__global__ void __launch_bounds__(kShiftThreads)
k_shift_fp32(const float* __restrict__ P32, const float* __restrict__ X, unsigned long long* __restrict__ acc,
             float c, Map map) {
    if (!map.init()) return;
    const int items = map.total();
    __shared__ __align__(16) float tile[kPixTile * Dp];
    const int tid = threadIdx.x;
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
        const F32Item ii = map.item(item);
        const int pos0 = ii.seed0 + tid;
        const int pos1 = pos0 + kShiftThreads;
        const int s0 = pos0 < ii.n_active ? ii.active[pos0] : -1;
        const int s1 = pos1 < ii.n_active ? ii.active[pos1] : -1;
        float x0[Dp], x1[Dp], y0[Dp], y1[Dp];
        float c0 = 0.f, c1 = 0.f;
#pragma unroll
        for (int k = 0; k < Dp; k += 4) {
            float4 a = s0 >= 0 ? *reinterpret_cast<const float4*>(X + (int64_t)s0 * Dp + k)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 b = s1 >= 0 ? *reinterpret_cast<const float4*>(X + (int64_t)s1 * Dp + k)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
            x0[k] = a.x; x0[k + 1] = a.y; x0[k + 2] = a.z; x0[k + 3] = a.w;
            x1[k] = b.x; x1[k + 1] = b.y; x1[k + 2] = b.z; x1[k + 3] = b.w;
        }
#pragma unroll
        for (int k = 0; k < Dp; ++k) y0[k] = y1[k] = 0.f;
        const int64_t p_begin = ii.p_begin, p_end = ii.p_end;
        for (int64_t pb = p_begin; pb < p_end; pb += kPixTile) {
            const int cnt = (int)min((int64_t)kPixTile, p_end - pb);
            __syncthreads();
            const float4* src = reinterpret_cast<const float4*>(P32 + (int64_t)pb * Dp);
            float4* dst = reinterpret_cast<float4*>(tile);
            for (int q = tid; q < cnt * (Dp / 4); q += kShiftThreads) dst[q] = src[q];
            __syncthreads();
            for (int j = 0; j < cnt; ++j) {
                float p[Dp];
#pragma unroll
                for (int k = 0; k < Dp; k += 4) {
                    float4 v = *reinterpret_cast<const float4*>(tile + j * Dp + k);
                    p[k] = v.x; p[k + 1] = v.y; p[k + 2] = v.z; p[k + 3] = v.w;
                }
                float d0 = 0.f, d1 = 0.f;
#pragma unroll
                for (int k = 0; k < Dp; ++k) {
                    d0 = fmaf(x0[k], p[k], d0);
                    d1 = fmaf(x1[k], p[k], d1);
                }
                const bool in0 = d0 >= c, in1 = d1 >= c;
                if (__any_sync(0xffffffffu, in0 || in1)) {
                    if (in0) {
#pragma unroll
                        for (int k = 0; k < Dp; ++k) y0[k] += p[k];
                        c0 += 1.f;
                    }
                    if (in1) {
#pragma unroll
                        for (int k = 0; k < Dp; ++k) y1[k] += p[k];
                        c1 += 1.f;
                    }
                }
            }
        }
        if (s0 >= 0 && c0 > 0.f) {
            unsigned long long* a = acc + (int64_t)s0 * (Dp + 1);
#pragma unroll
            for (int k = 0; k < Dp; ++k) atomicAdd(a + k, (unsigned long long)__float2ll_rn(y0[k] * kFixScale));
            atomicAdd(a + Dp, (unsigned long long)c0);
        }
        if (s1 >= 0 && c1 > 0.f) {
            unsigned long long* a = acc + (int64_t)s1 * (Dp + 1);
#pragma unroll
            for (int k = 0; k < Dp; ++k) atomicAdd(a + k, (unsigned long long)__float2ll_rn(y1[k] * kFixScale));
            atomicAdd(a + Dp, (unsigned long long)c1);
        }
    }
}

// End of an iteration: every active seed's update, the next active list and
// the early stop (Sec. 3.2.3: the round ends once more than gamma of its seeds
// have converged, when none is still moving, or at max_iter).
// The last block to finish writes the list, the moving seeds in the order of
// the current one (the pixel order that the selection gave them; appending them
// as blocks finish would mix the cells of an item's seeds). A second kernel for
// that cost a launch per iteration; one block's pass over the masks of a few
// thousand seeds is shorter.
// Launched before the shift has ended (launch_after), and the next shift before
// this has: launches and set-up overlap the work ahead. A BF16 frame of 131072
// pixels (146 iterations) took 17.2 ms with two kernels, one thread a seed and
// ordinary launches, 14.6 ms now; a 64 x 64 FP32 frame 3.25 and 2.69 ms.
template <int Dp>
__global__ void __launch_bounds__(kFinThreads)
k_finalize(unsigned long long* __restrict__ acc, const int32_t* active_in,
           int32_t* __restrict__ active_out, float* __restrict__ X, uint8_t* __restrict__ sstate,
           int32_t* __restrict__ support, double tol, StepBand band, uint32_t* __restrict__ moving, DevCounters* dc,
           double gamma, int max_iter) {
    grid_wait();
    grid_release();
    if (dc->done) return;
    const int n_active = dc->n_active;
    const int nb = (n_active + kFinSeeds - 1) / kFinSeeds;
    if ((int)blockIdx.x >= nb) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __shared__ int s_last;
    __shared__ uint32_t s_part[kFinThreads / 32];
    {
        const int pos = blockIdx.x * kFinSeeds + wid * 8 + (lane & 7);
        const bool live = pos < n_active;
        const int64_t slot = live ? active_in[pos] : 0;
        const SeedEnd e = finalize_seed<Dp>(live, acc + slot * (Dp + 1), X + slot * Dp, sstate + slot, support + slot,
                                            tol, band);
        const bool first = lane < 8;  // one lane per seed
        const uint32_t mv = __ballot_sync(0xffffffffu, first && e.move);
        if (lane == 0) s_part[wid] = mv;
        const int mc = __syncthreads_count(first && e.conv), mf = __syncthreads_count(first && e.fail);
        if (threadIdx.x == 0) {
            moving[blockIdx.x] = s_part[0] | s_part[1] << 8 | s_part[2] << 16 | s_part[3] << 24;
            if (mc) atomicAdd(&dc->conv_new, mc);
            if (mf) atomicAdd(&dc->fail_total, mf);
            __threadfence();
            s_last = atomicAdd(&dc->ticket, 1) == nb - 1;
        }
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // Tiles of one mask per thread: prefix sums over the block, then each warp
    // copies every fourth mask's seeds.
    __shared__ uint32_t s_mask[kFinThreads];
    __shared__ int s_off[kFinThreads];
    int next = 0;
    for (int b0 = 0; b0 < nb; b0 += kFinThreads) {
        const int b = b0 + threadIdx.x;
        const uint32_t m = b < nb ? __ldcg(moving + b) : 0u;
        int incl = __popc(m);
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        __syncthreads();
        if (lane == 31) s_part[wid] = (uint32_t)incl;
        __syncthreads();
        int before = next;
#pragma unroll
        for (int w = 0; w < kFinThreads / 32; ++w) {
            if (w < wid) before += (int)s_part[w];
            next += (int)s_part[w];
        }
        s_mask[threadIdx.x] = m;
        s_off[threadIdx.x] = before + incl - __popc(m);
        __syncthreads();
        const int nw = min(kFinThreads, nb - b0);
#pragma unroll 4
        for (int w = wid; w < nw; w += kFinThreads / 32) {
            const uint32_t bits = s_mask[w];
            if ((bits >> lane) & 1u)
                active_out[s_off[w] + __popc(bits & ((1u << lane) - 1u))] = active_in[(b0 + w) * kFinSeeds + lane];
        }
    }
    if (threadIdx.x != 0) return;
    const int conv = dc->conv_total + *(volatile int32_t*)&dc->conv_new, iters = dc->iters + 1;
    dc->ticket = 0;
    dc->seed_iters += n_active;
    dc->conv_total = conv;
    dc->conv_new = 0;
    dc->n_active = next;
    dc->iters = iters;
    if ((double)conv > gamma * (double)dc->m_round || next == 0 || iters >= max_iter) dc->done = 1;
}

template <int Dp>
ms_status shift_iteration_t(ms_ctx* ctx, int t, int max_iter, cudaEvent_t e0, cudaEvent_t e1) {
    const int32_t* a_in = ctx->active[t & 1];
    int32_t* a_out = ctx->active[(t + 1) & 1];
    const float c = ceil_to_float(ctx->cfg.bandwidth_cos);
    const double gamma = ctx->cfg.all_seeds ? 1.0 : ctx->cfg.gamma;
    const unsigned fin_blocks = (unsigned)((ctx->m_round + kFinSeeds - 1) / kFinSeeds);
    if (e0) MS_CUDA(cudaEventRecord(e0, ctx->stream));
    if (ctx->cfg.precision == MS_BF16) {
        ms_status s = launch_shift_tc(ctx, a_in, ctx->tc_grid, 2 * ctx->tc_grid, nullptr);
        if (s != MS_OK) return s;
    } else {
        ms_status s = launch_shift_f32_tc(ctx, a_in, c);
        if (s != MS_OK) return s;
    }
    if (e1) MS_CUDA(cudaEventRecord(e1, ctx->stream));
    MS_CUDA(launch_after(k_finalize<Dp>, fin_blocks, kFinThreads, 0, ctx->stream, ctx->acc, a_in, a_out, ctx->X,
                         ctx->sstate, ctx->support, ctx->cfg.tol, step_band(ctx->cfg.tol), ctx->moving, ctx->dc, gamma,
                         max_iter));
    ctx->launches += 2;
    return MS_OK;
}

}  // namespace

float ceil_to_float(double c) {
    float f = (float)c;
    if ((double)f < c) f = nextafterf(f, 2.0f);
    return f;
}

int shift_blocks_per_sm() {
    int b16 = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b16, k_shift_fp32<16, F32SingleMap>, kShiftThreads, 0);
    return b16 > 0 ? b16 : 1;
}

ms_status launch_window_sums_fp32(const float* P32, int32_t n, const int32_t* active, const float* X,
                                  unsigned long long* acc, float c, const DevCounters* dc,
                                  cudaStream_t stream) {
    int per_sm = shift_blocks_per_sm();
    int dev = 0, sms = 1;
    MS_CUDA(cudaGetDevice(&dev));
    MS_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int grid = sms * per_sm;
    F32SingleMap map;
    map.active = active;
    map.dc = dc;
    map.n = n;
    map.target = 2 * grid;
    k_shift_fp32<16, F32SingleMap><<<grid, kShiftThreads, 0, stream>>>(P32, X, acc, c, map);
    MS_LAUNCH("k_shift_fp32");
    return MS_OK;
}

ms_status launch_shift_iteration(ms_ctx* ctx, int t, int max_iter, cudaEvent_t e0, cudaEvent_t e1) {
    if (ctx->m_round <= 0) return MS_OK;
    return ctx->Dp == 16 ? shift_iteration_t<16>(ctx, t, max_iter, e0, e1)
                         : shift_iteration_t<32>(ctx, t, max_iter, e0, e1);
}

}  // namespace ms
