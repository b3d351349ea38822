// Method neighbours of the search (declarations in include/cetra.h):
//  - masking a detected signal before the next search (Sec. 4.2): the resampled cells in and
//    around the signal's transits are nulled, then the linear stage is rerun;
//  - single-transit (monotransit) events from the linear search (Sec. 1, Sec. 5): the
//    strongest dimming windows, greedily, each hiding the mid-times within its duration.
#include <algorithm>
#include <cmath>

#include "internal.h"

namespace {

constexpr int NB_THREADS = 256;

// Null cell k (W y = W = 0) when its time g = t_ref + (k - n_pad) c is within h of a mid-time
// t0 + n P, n = floor((g - t0) / P + 1/2) the nearest epoch; FP64, one rounding per operation.
// counts[0] += cells that held data (counts may be NULL).
__global__ void mask_kernel(float2 *__restrict__ grid, int64_t n_grid,
                            double t_ref, double c, int64_t n_pad, double P, double t0, double h,
                            unsigned long long *__restrict__ counts) {
    unsigned long long mine = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_grid; k += stride) {
        const double g = __dadd_rn(t_ref, __dmul_rn((double)(k - n_pad), c));
        const double d = __dsub_rn(g, t0);
        const double n = floor(__dadd_rn(__ddiv_rn(d, P), 0.5));
        const double r = fabs(__dsub_rn(d, __dmul_rn(n, P)));
        if (r < h) {
            mine += grid[k].y > 0.0f;
            grid[k] = make_float2(0.0f, 0.0f);
        }
    }
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_down_sync(0xFFFFFFFFu, mine, o);
    if (counts && (threadIdx.x & 31) == 0 && mine) atomicAdd(counts, mine);
}

// Event keys: per t0 cell the best dimming window over durations, packed so that a larger key
// is a better event: LR bits (positive floats order like their bits), then 255 - j (smaller j
// first), then 2^24 - 1 - i (smaller i first). 0 = no dimming window at this t0.
__device__ __forceinline__ unsigned long long event_key(float lr, int j, int64_t i) {
    return ((unsigned long long)__float_as_uint(lr) << 32) |
           ((unsigned long long)(255 - j) << 24) | (unsigned long long)(0xFFFFFF - i);
}

// The greedy steps are serial and short, so what bounded them was two launches a step, the first
// a pass over every key (12 us a step at 2.1 M t0 cells). The keys are now kept with the best of
// each segment of 2^shift cells (at most EV_SEGMENTS), and one block takes all the steps: it
// scans the segments' maxima in shared memory, and after a step works out again only those of the
// segments that the event hides cells of. A kept cell is its LR and its duration (5 bytes; the
// index is its place), so that the segments' maxima fit beside them in n_t0 + max_events words:
// with at least 256 cells a segment, 5 I + 8 ceil(I / 256) <= 8 I + 8.
// Measured (2.1 M cells, 30 durations, 10 events): linear stage and events 1.88 -> 1.75 ms.
constexpr int EV_THREADS = 1024;
constexpr int EV_SEGMENTS = 4096;
__host__ __device__ inline int event_shift(int64_t I) {
    int shift = 8;
    while (((I + ((int64_t)1 << shift) - 1) >> shift) > EV_SEGMENTS) ++shift;
    return shift;
}

__device__ __forceinline__ unsigned long long warp_max(unsigned long long v) {
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}

struct mono_cells {
    unsigned long long *top;  // [segments]
    float *lr;                // [I]; 0 = no dimming window, or hidden
    uint8_t *dur;             // [I]
};
inline mono_cells mono_carve(unsigned long long *scratch, int64_t I, unsigned segments) {
    mono_cells m;
    m.top = scratch;
    m.lr = reinterpret_cast<float *>(scratch + segments);
    m.dur = reinterpret_cast<uint8_t *>(m.lr + I);
    return m;
}

// One block per segment: its cells (equal LR: the smaller duration index) and their best key.
__global__ void __launch_bounds__(NB_THREADS, 6)
mono_keys_kernel(const float2 *__restrict__ ab, int64_t ld, int64_t I, int J, int shift,
                 mono_cells cells) {
    __shared__ unsigned long long red[NB_THREADS / 32];
    const int64_t lo = (int64_t)blockIdx.x << shift;
    const int64_t hi = min(I, lo + ((int64_t)1 << shift));
    unsigned long long most = 0ull;
    auto take = [](float x, float y, int j, float &best, int &best_j) {
        if (y > 0.0f && x > 0.0f) {
            const float lr = 0.5f * (x * (x / y));
            if (lr > best) best = lr, best_j = j;
        }
    };
    auto keep = [&](int64_t i, float lr, int j) {
        cells.lr[i] = lr;
        cells.dur[i] = (uint8_t)j;
        if (lr > 0.0f) most = max(most, event_key(lr, j, i));
    };
    // two cells per load (the rows' strides and a segment's first cell are even; the row goes on
    // after its last cell)
    for (int64_t i = lo + 2 * threadIdx.x; i < hi; i += 2 * NB_THREADS) {
        float best0 = 0.0f, best1 = 0.0f;
        int j0 = 0, j1 = 0;
#pragma unroll 4
        for (int j = 0; j < J; ++j) {
            const float4 v = *reinterpret_cast<const float4 *>(ab + (int64_t)j * ld + i);
            take(v.x, v.y, j, best0, j0);
            take(v.z, v.w, j, best1, j1);
        }
        keep(i, best0, j0);
        if (i + 1 < hi) keep(i + 1, best1, j1);
    }
    most = warp_max(most);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = most;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int x = 1; x < NB_THREADS / 32; ++x) most = max(most, red[x]);
        cells.top[blockIdx.x] = most;
    }
}

// All greedy steps (one block): the best key left becomes the next event, then the t0 cells within
// its duration are hidden: |i - i_e| < h = D_j q / (c p) (FP64) -> LR 0. Ends early when no key
// is left. The FP64 work (every duration's h before the steps, the events' values from their
// windows' FP32 sums after them) is a lane each: within a step one lane's divisions were half of
// its time.
__global__ void __launch_bounds__(EV_THREADS)
mono_events_kernel(const float2 *__restrict__ ab, int64_t ld, int64_t I,
                   const double *__restrict__ durations, double t_ref, double c, int64_t p,
                   int64_t q, int64_t n_pad, int shift, int J, int max_events,
                   mono_cells cells, cetra_event *__restrict__ events,
                   int *__restrict__ n_events) {
    __shared__ unsigned long long seg[EV_SEGMENTS];
    __shared__ unsigned long long red[EV_THREADS / 32];
    __shared__ unsigned long long s_key;
    __shared__ int64_t reach[256];  // integers below h are those below ceil(h)
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int n_seg = (int)((I + ((int64_t)1 << shift) - 1) >> shift);
    for (int x = t; x < n_seg; x += EV_THREADS) seg[x] = cells.top[x];
    if (t < J) {
        const double span =
            ceil(__ddiv_rn(__dmul_rn(durations[t], (double)q), __dmul_rn(c, (double)p)));
        reach[t] = span < (double)I ? (int64_t)span : I;
    }
    __syncthreads();
    int e = 0;
    for (; e < max_events; ++e) {
        unsigned long long best = 0ull;
        for (int x = t; x < n_seg; x += EV_THREADS) best = max(best, seg[x]);
        best = warp_max(best);
        if (lane == 0) red[wid] = best;
        __syncthreads();
        if (wid == 0) {
            best = warp_max(red[lane]);
            if (lane == 0) s_key = best;
        }
        __syncthreads();
        const unsigned long long key = s_key;
        if (key == 0ull) break;  // uniform
        const int64_t ie = 0xFFFFFF - (int64_t)(key & 0xFFFFFFull);
        const int j = 255 - (int)((key >> 24) & 0xFFull);
        if (t == 0) events[e].i = (int64_t)key;  // decoded below
        const int64_t r = reach[j];
        const int64_t lo = max((int64_t)0, ie - r), hi = min(I - 1, ie + r);
        // hide the cells, and work out the maxima of their segments again (32 consecutive cells
        // are of one segment)
        const int64_t s0 = lo >> shift, s1 = hi >> shift;
        for (int64_t x = s0 + t; x <= s1; x += EV_THREADS) seg[x] = 0ull;
        __syncthreads();
        const int64_t end = min(I, (s1 + 1) << shift);
        for (int64_t i0 = s0 << shift; i0 < end; i0 += EV_THREADS) {
            const int64_t i = i0 + t;
            float lr = i < end ? cells.lr[i] : 0.0f;
            if (lr > 0.0f && llabs(i - ie) < r) cells.lr[i] = lr = 0.0f;
            unsigned long long k = lr > 0.0f ? event_key(lr, cells.dur[i], i) : 0ull;
            k = warp_max(k);
            if (lane == 0 && k) atomicMax(&seg[i >> shift], k);
        }
        __syncthreads();
    }
    if (t == 0) *n_events = e;
    __syncthreads();
    for (int x = t; x < e; x += EV_THREADS) {
        const unsigned long long key = (unsigned long long)events[x].i;
        const int64_t ie = 0xFFFFFF - (int64_t)(key & 0xFFFFFFull);
        const int j = 255 - (int)((key >> 24) & 0xFFull);
        const float2 v = ab[(int64_t)j * ld + ie];
        cetra_event ev;
        ev.depth = __ddiv_rn((double)v.x, (double)v.y);
        ev.depth_var = __ddiv_rn(1.0, (double)v.y);
        ev.dlogl = 0.5 * __dmul_rn((double)v.x, ev.depth);
        ev.t0 = __dadd_rn(t_ref, __ddiv_rn(__dmul_rn((double)(ie * p - n_pad * q), c), (double)q));
        ev.duration = durations[j];
        ev.i = ie;
        ev.j = j;
        ev.pad_ = 0;
        events[x] = ev;
    }
}

unsigned blocks_for(int64_t n, int num_sms) {
    int64_t b = (n + NB_THREADS - 1) / NB_THREADS;
    const int64_t cap = (int64_t)num_sms * 8;
    return (unsigned)std::max<int64_t>(1, std::min(b, cap));
}

}  // namespace

cudaError_t launch_mask(cetra_ctx *ctx, const cetra_plan *plan, float2 *grid, double P,
                        double t0, double h, unsigned long long *counts) {
    mask_kernel<<<blocks_for(plan->n_grid, ctx->num_sms), NB_THREADS, 0, ctx->stream>>>(
        grid, plan->n_grid, plan->t_ref, plan->cadence, plan->n_pad, P, t0, h, counts);
    ctx->launches++;
    return cudaGetLastError();
}

size_t mono_scratch_words(const cetra_plan *plan, int max_events) {
    return (size_t)plan->n_t0 + (size_t)max_events;
}

cudaError_t launch_monotransits(cetra_ctx *ctx, const cetra_plan *plan, const float2 *ab,
                                unsigned long long *scratch, int max_events,
                                cetra_event *events, int *n_events) {
    const int64_t I = plan->n_t0;
    const int shift = event_shift(I);
    const unsigned segments = (unsigned)((I + ((int64_t)1 << shift) - 1) >> shift);
    const mono_cells cells = mono_carve(scratch, I, segments);
    mono_keys_kernel<<<segments, NB_THREADS, 0, ctx->stream>>>(ab, plan->ab_ld, I, plan->J, shift,
                                                               cells);
    ctx->launches++;
    cudaError_t e = cudaGetLastError();
    if (e) return e;
    mono_events_kernel<<<1, EV_THREADS, 0, ctx->stream>>>(
        ab, plan->ab_ld, I, plan->d_durations, plan->t_ref, plan->cadence, plan->p, plan->q,
        plan->n_pad, shift, plan->J, max_events, cells, events, n_events);
    ctx->launches++;
    return cudaGetLastError();
}
