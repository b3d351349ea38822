// Learned period-interval proposal (not in the paper; a deployment aid for the periodic
// search of Sec. 2.3): a 1-D CNN reads the max-pooled linear-search likelihood ratios of a
// curve ([durations][bins]) and marks the bins that hold transits; a comb over that map
// scores log-spaced period intervals, and the fold then evaluates the best intervals first.
//
// Network: log1p(features) -> conv(Cin -> 32, k 9) ReLU -> conv(32 -> 32) ReLU ->
// conv(32 -> 32) ReLU -> conv(32 -> 1) -> logit per bin. Weights are kept in FP32 (the
// training copy) and used in BF16 (rounded to nearest even) by every kernel; sums are FP32.
// Training: binary cross-entropy with logits against per-bin transit labels (positive
// weight w+), Adam. All kernels are written here; nothing calls a library.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <random>
#include <vector>

#include "device.cuh"
#include "internal.h"

namespace {

constexpr int CNN_K = 9;           // kernel width
constexpr int CNN_C = 32;          // hidden channels
constexpr int CNN_LAYERS = 4;
constexpr size_t kCombSmemMax = 98 * 1024;  // maps up to 24,576 bins (+ 512 cells) are staged

// ------------------------------------------------------------------------------- kernels

// ------------------------------------------------------------------------- fused forward pass
//
// All four layers of NET_OUT bins of one curve per tile, on the tensor cores (tcgen05), without
// the activations leaving the SM (training also stores them). Conv as GEMM: D[bin][co] +=
// X[bin + k][ci] W[k][ci][co] for the 9 taps k: the activations sit in shared memory as rows
// (bins) of 8-channel units of 16 bytes, every row 16 bytes after the one before it, so a tap is
// a row offset of the operand's start address and nothing is gathered. M = 128 bins, N = 32
// channels, K = 16 channels per instruction.
//
// Precision: the weights are BF16 values; an FP32 activation is the exact sum of three BF16
// parts (its leading 8, middle 8 and last 8 bits), so three products with the same weight give
// the FP32 product exactly. The tensor core's accumulator truncates, so a sum is kept in four
// accumulators (net_layer_mma; each takes its last and middle parts first), which are added in
// FP32 with the mean of what truncation took off (net_sums). Measured error of the probabilities
// against 64 bits: 6.4e-8 (FP32 kernels: 1.1e-7).
//
// Measured (256 curves, 16 durations, 4,096 bins): 2,347 us as log1p, four FP32 conv kernels and
// a sigmoid with every activation in memory, 260 us as this kernel (three parts' products alone:
// 76 us at the measured BF16 rate). Bound: the instructions' reads of the activation operand from
// shared memory (4 KB each, 150 per tile at 16 durations) and the epilogues (splitting the next
// layer's input), in turn: two blocks per SM, so that one's epilogue runs under the other's
// instructions.
//
// Halo: layer l's row r is bin t0 - 16 + 4 l + r. A tile computes NET_ROWS = 254 rows of the
// first three layers in place (rows past the last valid one are never used): 254, 246, 238
// valid rows, then NET_OUT = 230 logits. Rows outside [0, T) are zero (zero padding).
constexpr int NET_BLOCK = 127;             // rows a block of 128 completes (see net_layer_mma)
constexpr int NET_ROWS = 2 * NET_BLOCK;    // rows computed per layer
constexpr int NET_XROWS = 264;             // rows held: 8 more for the last tap, whole groups of 8
constexpr int NET_OUT = NET_ROWS - 24;     // logits per tile
constexpr int NET_THREADS = 256;
constexpr int NET_GRP = 4;                 // accumulators of a sum
constexpr int NET_AHEAD = 2;               // input items a thread reads ahead (any tile has as many)
constexpr int NET_UNIT = NET_XROWS * 16;   // bytes of one 8-channel unit of all rows
constexpr int NET_PART = 4 * NET_UNIT;     // bytes of one BF16 part (32 channels)
constexpr int NET_ACT3_LD = 260;           // floats per channel row of the last activation
constexpr int NET_TMEM_COLS = 2 * NET_GRP * CNN_C;  // 256
constexpr int NET_PLD = 256;               // partial logits per channel group
constexpr float NET_SHORT = 5.0e-8f;       // what truncation takes off a sum (see net_sums)
static_assert(3 * NET_PART >= CNN_C * NET_ACT3_LD * 4 + 4 * NET_PLD * 4, "activation reuse");

__host__ __device__ constexpr int net_units(int cin) { return (cin + 15) / 16 * 2; }
// bytes of the BF16 weights of a layer with `units` input units: taps 0-7 in pairs
// [pair][unit][tap of the pair][co][8 ci], then tap 8 [unit][co][8 ci]
__host__ __device__ constexpr int net_wbytes(int units) { return CNN_K * units * CNN_C * 16; }
inline size_t net_smem(int cin) {
    return (size_t)3 * NET_PART + net_wbytes(net_units(cin)) + 2 * net_wbytes(4) +
           (CNN_C * CNN_K + 4 * CNN_C) * sizeof(float);
}

// Place of weight (tap k, unit u, co, element e) in them.
__device__ __forceinline__ int net_wplace(int units, int k, int u, int co, int e) {
    return k < 8 ? (((k >> 1) * units + u) * 64 + (k & 1) * CNN_C + co) * 8 + e
                 : (4 * units * 64 + u * CNN_C + co) * 8 + e;
}

// Words of a network on the device that its kernels leave beside their outputs.
struct net_words {
    double loss;
    int next[CNN_LAYERS];  // tiles of the weight gradients handed out
    int status;            // 0, or CETRA_ETIMEOUT: a bounded wait gave up
    int lost;              // not 0: a wait of the last gradient's launches gave up
};

// Bounded waits of a launch: a wait gives up after `limit` SM clocks, is recorded in the status
// word, and the block's remaining outputs are NaN. The self-test leaves the matrix instructions
// of tile `skip` out (-1: none), so that the waits for them run out.
struct net_waits {
    int *status;
    long long limit;
    int skip;
};

struct net_layers {
    const __nv_bfloat16 *w[CNN_LAYERS];  // [co][ci][9], BF16
    const float *bias[CNN_LAYERS];
    float *act[CNN_LAYERS + 1];          // training: log1p(features), the activations, the logits
    net_waits wait;
};

// Matrix descriptor of a K-major operand without swizzle: rows 16 bytes apart, 8-row groups 128
// bytes apart (high word), the second 8-element unit of K `unit_bytes` after the first. The low
// word; an offset of the start address adds its 16-byte units to it.
__device__ __forceinline__ uint32_t net_desc_lo(uint32_t addr, uint32_t unit_bytes) {
    return ((addr >> 4) & 0x3FFFu) | ((unit_bytes >> 4) << 16);
}

// kind::f16: FP32 accumulator, BF16 operands, both K-major, M = 128, N = 32 or 64.
__host__ __device__ constexpr uint32_t net_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n / 8) << 17) | ((128u / 16) << 24);
}

__device__ __forceinline__ void net_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                        bool add) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)add)
        : "memory");
}
// The matrix instructions of one layer for one block of 128 rows (one thread): a_lo, w are the
// low word of the activations' descriptor at tap 0, unit 0, part 0, and the weights' address.
//
// Reading the activations is the bound, so an instruction takes two taps: N = 64 are the 32
// output channels of taps 2 p and 2 p + 1, both on the rows of tap 2 p, and the second tap's sums
// belong one row further down: out[r] = E0[r] + E1[r + 1] (net_sums). A block of 128 rows
// therefore completes 127. 256 curves x 16 durations: 260 us; one tap per instruction: 26 us more.
// Accumulators: E0 and E1 of pairs 0-1 and of pairs 2-4 (columns 0, 32, 64, 96), four partial
// sums of every output. Consecutive instructions go to different ones, and every offset is a
// constant of the unrolled code (worked out in a loop, one accumulator after the other, the
// instructions were three times further apart).
template <int UNITS>
__device__ __forceinline__ void net_layer_mma(uint32_t d, uint32_t a_lo, uint32_t w) {
    constexpr uint32_t hi = (128u >> 4) | (1u << 14);
    const uint32_t b64 = net_desc_lo(w, 64 * 16);
    const uint32_t b32 = net_desc_lo(w + 4 * UNITS * 64 * 16, CNN_C * 16);
#pragma unroll
    for (int q = 2; q >= 0; --q)
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int u = 0; u < UNITS; u += 2)
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    if (g == 0 && j == 2) continue;  // pairs 0, 1 and 2, 3, 4 (tap 8 alone)
                    const int pair = g == 0 ? j : 2 + j;
                    const uint64_t a = ((uint64_t)hi << 32) |
                                       (a_lo + (q * NET_PART + u * NET_UNIT + 2 * pair * 16) / 16);
                    const bool add = q < 2 || j > 0 || u > 0;
                    if (pair < 4)
                        net_mma(d + g * 64, a,
                                ((uint64_t)hi << 32) | (b64 + (pair * UNITS + u) * 64 * 16 / 16),
                                net_idesc(64), add);
                    else
                        net_mma(d + g * 64, a,
                                ((uint64_t)hi << 32) | (b32 + u * CNN_C * 16 / 16),
                                net_idesc(CNN_C), add);
                }
}
__device__ __forceinline__ void net_commit(uint64_t *bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void net_tmem_load(float (&v)[16], uint32_t taddr) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}
// Wait for the warp's loads; the operands tie the uses of the loaded values to the wait.
__device__ __forceinline__ void net_tmem_wait(float (&v)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]),
                   "+f"(v[6]), "+f"(v[7]), "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]),
                   "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15])
                 :
                 : "memory");
}

// The first row's E1 of every warp of a block, for the last lane of the warp before it (called by
// the four warps of the block; xch: [3][32] floats of the block, barrier id 1 or 2).
__device__ __forceinline__ void net_exchange(uint32_t taddr, float *xch, int warp4, int barrier) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float v[16], o[16];
        net_tmem_load(v, taddr + 32 + h * 16);
        net_tmem_load(o, taddr + 96 + h * 16);
        net_tmem_wait(v);
        net_tmem_wait(o);
        if (warp4 > 0 && lane == 0)
#pragma unroll
            for (int c = 0; c < 16; ++c) xch[(warp4 - 1) * 32 + h * 16 + c] = v[c] + o[c];
    }
    asm volatile("bar.sync %0, 128;" ::"r"(barrier) : "memory");
}

// Sixteen channels (half h) of the lane's row: E0 + E1 of the next row, and what truncation took
// off them on average. An accumulator loses up to a unit in the last place per instruction,
// always towards zero; a mean over many bins (the loss, a weight's gradient) does not average
// that out, as it does rounding to nearest. As truncated multipliers add back the expected value
// of the columns they leave out (Schulte and Swartzlander 1993), the sum is raised by its mean
// shortfall, measured against 64-bit sums of the same operands: 4.0e-8 to 6.4e-8 of the sum by
// layer, network and direction (7.7e-8 in a first layer of 32 channels), 5.0e-8 taken. The
// term goes into the smaller addend before the last rounding: that keeps it from rounding away.
// Measured (16 durations; with it, without, FP32 kernels): mean signed error of the logits by
// their mean size 1.3e-8, -1.45e-7, -1.2e-8; of the loss 1.5e-8, -3.3e-8, 6e-9; a layer's
// gradient at 2 curves off by at most 1.5e-7, 3.2e-7, 2.1e-7 of its largest.
__device__ __forceinline__ void net_sums(float (&v)[16], uint32_t taddr, const float *xch,
                                         int warp4, int h) {
    const int lane = threadIdx.x & 31;
    float o[16];
    net_tmem_load(v, taddr + 32 + h * 16);
    net_tmem_load(o, taddr + 96 + h * 16);
    net_tmem_wait(v);
    net_tmem_wait(o);
#pragma unroll
    for (int c = 0; c < 16; c += 2) {
        float2 e1 = make_float2(v[c], v[c + 1]);
        add2(e1, make_float2(o[c], o[c + 1]));
        v[c] = __shfl_down_sync(0xFFFFFFFFu, e1.x, 1);
        v[c + 1] = __shfl_down_sync(0xFFFFFFFFu, e1.y, 1);
        if (lane == 31) {
            v[c] = warp4 < 3 ? xch[warp4 * 32 + h * 16 + c] : 0.0f;
            v[c + 1] = warp4 < 3 ? xch[warp4 * 32 + h * 16 + c + 1] : 0.0f;
        }
    }
    float w[16];
    net_tmem_load(w, taddr + h * 16);
    net_tmem_load(o, taddr + 64 + h * 16);
    net_tmem_wait(w);
    net_tmem_wait(o);
    // (packed pairs: v += t + NET_SHORT (v + t) with t = w + o)
#pragma unroll
    for (int c = 0; c < 16; c += 2) {
        float2 t = make_float2(w[c], w[c + 1]), r = make_float2(v[c], v[c + 1]);
        add2(t, make_float2(o[c], o[c + 1]));
        float2 s = r;
        add2(s, t);
        fma2(t, s, make_float2(NET_SHORT, NET_SHORT));
        add2(r, t);
        v[c] = r.x;
        v[c + 1] = r.y;
    }
}

// Eight channels of one row as three BF16 parts (the leading, middle and last 8 bits of each
// value: exact) into the 16-byte slot at `at` of every part.
__device__ __forceinline__ void net_store_row(uint32_t at, const float *v) {
    uint32_t p[3][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t part[3][2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float x = v[2 * k + e];
            const uint32_t hi = __float_as_uint(x) & 0xFFFF0000u;
            float r = x - __uint_as_float(hi);
            if (!(fabsf(x) < INFINITY)) r = 0.0f;  // an infinity or NaN is its leading part
            const uint32_t mid = __float_as_uint(r) & 0xFFFF0000u;
            part[0][e] = hi;
            part[1][e] = mid;
            part[2][e] = __float_as_uint(r - __uint_as_float(mid));
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) p[q][k] = __byte_perm(part[q][0], part[q][1], 0x7632);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at + q * NET_PART),
                     "r"(p[q][0]), "r"(p[q][1]), "r"(p[q][2]), "r"(p[q][3])
                     : "memory");
}

template <bool STORE>
__global__ void __launch_bounds__(NET_THREADS, 2)
cnn_net_kernel(const float *__restrict__ features, net_layers net, float *__restrict__ prob,
               int cin, int T, int n_tiles, int tiles_per_curve) {
    extern __shared__ __align__(128) unsigned char net_raw[];
    __shared__ uint64_t done[2];  // matrix instructions of row block 0 / 1 complete
    __shared__ float xch[2][96];
    __shared__ uint32_t s_tmem;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int units1 = net_units(cin);
    const uint32_t x0 = smem_u32(net_raw);
    unsigned char *wraw = net_raw + 3 * NET_PART;
    const uint32_t w0 = x0 + 3 * NET_PART;
    const int wsize1 = net_wbytes(units1);
    float *w4 = reinterpret_cast<float *>(wraw + wsize1 + 2 * net_wbytes(4));  // [co][9]
    float *bias = w4 + CNN_C * CNN_K;                                          // [4][32]
    float *act3 = reinterpret_cast<float *>(net_raw);    // [32][NET_ACT3_LD], after layer 3
    float *part = act3 + CNN_C * NET_ACT3_LD;            // [4][NET_PLD]

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&s_tmem)),
                     "n"(NET_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        mbar_init(&done[0], 1);
        mbar_init(&done[1], 1);
        fence_mbar_init();
    }
    // weights (channels past the layer's own are zero)
    for (int l = 0; l < 3; ++l) {
        const int ci_n = l == 0 ? cin : CNN_C, units = l == 0 ? units1 : 4;
        __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(
            wraw + (l == 0 ? 0 : wsize1 + (l - 1) * net_wbytes(4)));
        const int n = CNN_K * units * CNN_C * 8;
        for (int i = tid; i < n; i += NET_THREADS) {
            const int e = i & 7, co = (i >> 3) & 31, ku = i >> 8;
            const int u = ku % units, ci = u * 8 + e, k = ku / units;
            dst[net_wplace(units, k, u, co, e)] =
                ci < ci_n ? net.w[l][(co * ci_n + ci) * CNN_K + k] : __float2bfloat16(0.0f);
        }
    }
    for (int i = tid; i < CNN_C * CNN_K; i += NET_THREADS) w4[i] = __bfloat162float(net.w[3][i]);
    for (int i = tid; i < 3 * CNN_C + 1; i += NET_THREADS) bias[i] = net.bias[i / CNN_C][i % CNN_C];
    fence_proxy_async();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm = s_tmem;

    // item `it` of a tile's input: row it % NET_XROWS (bin t0 - 16 + row), channels 8 u .. 8 u + 7,
    // u = it / NET_XROWS
    auto read_item = [&](int tile, int it, float (&v)[8]) {
        const int b = tile / tiles_per_curve, u = it / NET_XROWS;
        const int t = (tile - b * tiles_per_curve) * NET_OUT - 16 + it - u * NET_XROWS;
        const float *fb = features + (int64_t)b * cin * T + t;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int ci = u * 8 + e;
            v[e] = t >= 0 && t < T && ci < cin ? fb[(int64_t)ci * T] : 0.0f;
        }
    };
    const int items = NET_XROWS * units1;
    float ahead[NET_AHEAD][8];  // the first items of the next tile, read under the last layer
    if (blockIdx.x < n_tiles)
#pragma unroll
        for (int x = 0; x < NET_AHEAD; ++x) read_item(blockIdx.x, tid + x * NET_THREADS, ahead[x]);
    uint32_t phase = 0;
    bool failed = false;
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const int b = tile / tiles_per_curve;
        const int t0 = (tile - b * tiles_per_curve) * NET_OUT;
        // layer 0: log1p of the features
        auto put_item = [&](int it, float (&v)[8]) {
            const int u = it / NET_XROWS, i = it - u * NET_XROWS;
            const int t = t0 - 16 + i;
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = log1pf(fmaxf(v[e], 0.0f));
            if (STORE && t >= t0 && t < T && t < t0 + NET_OUT)
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (u * 8 + e < cin)
                        net.act[0][((int64_t)b * cin + u * 8 + e) * T + t] = v[e];
            net_store_row(x0 + (uint32_t)(u * NET_UNIT + i * 16), v);
        };
#pragma unroll
        for (int x = 0; x < NET_AHEAD; ++x) put_item(tid + x * NET_THREADS, ahead[x]);
        for (int it = tid + NET_AHEAD * NET_THREADS; it < items; it += NET_THREADS) {
            float v[8];
            read_item(tile, it, v);
            put_item(it, v);
        }
        fence_proxy_async();
        __syncthreads();
        for (int l = 0; l < 3; ++l) {
            const int units = l == 0 ? units1 : 4;
            const uint32_t wl = w0 + (l == 0 ? 0 : wsize1 + (l - 1) * net_wbytes(4));
            if (tid == 0 && tile != net.wait.skip) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                for (int mb = 0; mb < 2; ++mb) {
                    const uint32_t d = tm + (uint32_t)(mb * NET_GRP * CNN_C);
                    const uint32_t a_lo =
                        net_desc_lo(x0 + (uint32_t)(mb * NET_BLOCK * 16), NET_UNIT);
                    if (units == 2)
                        net_layer_mma<2>(d, a_lo, wl);
                    else
                        net_layer_mma<4>(d, a_lo, wl);
                    net_commit(&done[mb]);
                }
            }
            __syncwarp();
            if (l == 2 && tile + (int)gridDim.x < n_tiles)
#pragma unroll
                for (int x = 0; x < NET_AHEAD; ++x)
                    read_item(tile + gridDim.x, tid + x * NET_THREADS, ahead[x]);
            // epilogue: warps 0-3 the rows of block 0, warps 4-7 of block 1 (in place: the other
            // block's instructions read no row of this one). The last layer's FP32 activations
            // overlay the parts, so it waits for both blocks.
            const int mb = warp >> 2, warp4 = warp & 3, r = mb * NET_BLOCK + warp4 * 32 + lane;
            bool ok = mbar_wait(&done[mb], phase, net.wait.limit);
            if (l == 2) {
                ok = mbar_wait(&done[mb ^ 1], phase, net.wait.limit) && ok;
                __syncthreads();
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int t = t0 - 12 + 4 * l + r;
            const bool mine = warp4 * 32 + lane < NET_BLOCK;  // the block's last lane has no row
            const bool inside = t >= 0 && t < T;
            const bool own = STORE && mine && inside && t >= t0 && t < t0 + NET_OUT;
            const uint32_t src = tm + (uint32_t)(mb * NET_GRP * CNN_C) + ((uint32_t)(warp & 3) << 21);
            net_exchange(src, xch[mb], warp4, 1 + mb);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float v[16];
                net_sums(v, src, xch[mb], warp4, h);
#pragma unroll
                for (int c = 0; c < 16; c += 2) {
                    float2 a = make_float2(v[c], v[c + 1]);
                    add2(a, *reinterpret_cast<const float2 *>(&bias[l * CNN_C + h * 16 + c]));
                    v[c] = inside ? fmaxf(a.x, 0.0f) : 0.0f;
                    v[c + 1] = inside ? fmaxf(a.y, 0.0f) : 0.0f;
                }
                if (own)
#pragma unroll
                    for (int c = 0; c < 16; ++c)
                        net.act[l + 1][((int64_t)b * CNN_C + h * 16 + c) * T + t] = v[c];
                if (l < 2 && mine) {
                    net_store_row(x0 + (uint32_t)(2 * h * NET_UNIT + r * 16), v);
                    net_store_row(x0 + (uint32_t)((2 * h + 1) * NET_UNIT + r * 16), v + 8);
                } else if (mine) {
#pragma unroll
                    for (int c = 0; c < 16; ++c) act3[(h * 16 + c) * NET_ACT3_LD + r] = v[c];
                }
            }
            phase ^= 1u;
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            fence_proxy_async();
            failed = __syncthreads_or(!ok);
            if (failed) break;
        }
        if (failed) {  // a wait gave up: this and the block's later tiles are NaN
            if (tid == 0) atomicExch(net.wait.status, CETRA_ETIMEOUT);
            mbar_wait(&done[0], phase ^ 1u, net.wait.limit);  // before the tensor memory goes
            mbar_wait(&done[1], phase ^ 1u, net.wait.limit);
            float *out = STORE ? net.act[CNN_LAYERS] : prob;
            for (; tile < n_tiles; tile += gridDim.x) {
                const int bb = tile / tiles_per_curve;
                const int at = (tile - bb * tiles_per_curve) * NET_OUT;
                for (int o = tid; o < NET_OUT && at + o < T; o += NET_THREADS)
                    out[(int64_t)bb * T + at + o] = __int_as_float(0x7fc00000);
            }
            break;
        }
        // layer 4 (one output channel, FP32): 4 bins x 8 input channels per thread
        {
            const int q = tid & 63, cg = tid >> 6;
            if (q < (NET_OUT + 3) / 4) {
                float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int ci = cg * 8 + c;
                    float xv[12];
#pragma unroll
                    for (int m = 0; m < 3; ++m) {
                        const float4 f =
                            *reinterpret_cast<const float4 *>(&act3[ci * NET_ACT3_LD + 4 * q + 4 * m]);
                        xv[4 * m] = f.x;
                        xv[4 * m + 1] = f.y;
                        xv[4 * m + 2] = f.z;
                        xv[4 * m + 3] = f.w;
                    }
#pragma unroll
                    for (int k = 0; k < CNN_K; ++k) {
                        const float wk = w4[ci * CNN_K + k];
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[e] = fmaf(wk, xv[e + k], acc[e]);
                    }
                }
                *reinterpret_cast<float4 *>(&part[cg * NET_PLD + 4 * q]) =
                    make_float4(acc[0], acc[1], acc[2], acc[3]);
            }
            __syncthreads();
            for (int o = tid; o < NET_OUT && t0 + o < T; o += NET_THREADS) {
                const float z = (part[o] + part[NET_PLD + o]) +
                                (part[2 * NET_PLD + o] + part[3 * NET_PLD + o]) +
                                bias[3 * CNN_C];
                if (STORE)
                    net.act[CNN_LAYERS][(int64_t)b * T + t0 + o] = z;
                else
                    prob[(int64_t)b * T + t0 + o] = 1.0f / (1.0f + expf(-z));
            }
            __syncthreads();  // act3 and part are read before the next tile's rows
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm),
                     "n"(NET_TMEM_COLS));
}

// ------------------------------------------------------------------------- backward pass
//
// Weighted binary cross-entropy with logits, mean over bins:
// l = w+ y softplus(-z) + (1 - y) softplus(z);  dl/dz = (sigmoid(z) (w+ y + 1 - y) - w+ y) / n.
__device__ __forceinline__ float bce_grad(float z, float y, float wpos, float inv) {
    const float s = 1.0f / (1.0f + expf(-z));
    return (s * (wpos * y + 1.0f - y) - wpos * y) * inv;
}
__device__ __forceinline__ float bce_loss(float z, float y, float wpos) {
    const float sp_pos = fmaxf(z, 0.0f) + log1pf(expf(-fabsf(z)));  // softplus(z)
    return wpos * y * (sp_pos - z) + (1.0f - y) * sp_pos;            // softplus(-z) = sp_pos - z
}

// Gradients G_l of the pre-activations of layers 2, 1 and 0 (and the loss) for BACK_OUT bins of
// one curve per tile, in one kernel: the gradient of a layer's input is a conv of its output's
// gradient with the flipped, transposed weights, so the same tensor-core tiles as the forward
// pass run in reverse: G_3 (one channel) -> G_2 in FP32, G_2 -> G_1 -> G_0 as matrix
// instructions, each masked where the layer's activation is not positive (ReLU). Rows: G_2's
// row i is bin t0 - 8 + i, G_1's row r bin t0 - 4 + r, G_0's row r bin t0 + r.
// Measured (32 curves, 16 durations): a training step took 940 us when each layer's gradient was a
// transpose, an FP32 conv and a mask kernel and the weight gradients met in atomics (the forward
// pass fused already); with this kernel (44 us) and the weight gradients below (152 us), 302 us.
constexpr int BACK_OUT = NET_ROWS - 8;
constexpr int BACK_G4 = NET_XROWS + 8;  // bins of G_3 a tile needs
inline size_t back_smem() {
    return (size_t)3 * NET_PART + 2 * net_wbytes(4) + (CNN_C * CNN_K + BACK_G4) * sizeof(float);
}
struct back_args {
    const __nv_bfloat16 *w1, *w2, *w3;       // layers 1, 2, 3: [co][ci][9]
    const float *logits, *labels;            // [B][T]
    const float *act1, *act2, *act3;         // outputs of layers 0, 1, 2: [B][32][T]
    float *g0, *g1, *g2;                     // [B][32][T]
    double *loss;
    float wpos;
    int64_t n;                               // bins of the batch
    net_waits wait;
};

__global__ void __launch_bounds__(NET_THREADS, 2)
cnn_back_kernel(back_args ar, int T, int n_tiles, int tiles_per_curve) {
    extern __shared__ __align__(128) unsigned char net_raw[];
    __shared__ uint64_t done[2];
    __shared__ float xch[2][96];
    __shared__ uint32_t s_tmem;
    __shared__ double s_loss[NET_THREADS / 32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t x0 = smem_u32(net_raw), w0 = x0 + 3 * NET_PART;
    unsigned char *wraw = net_raw + 3 * NET_PART;
    float *w3 = reinterpret_cast<float *>(wraw + 2 * net_wbytes(4));  // [ci][9]
    float *g3 = w3 + CNN_C * CNN_K;                                   // [BACK_G4]
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&s_tmem)),
                     "n"(NET_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        mbar_init(&done[0], 1);
        mbar_init(&done[1], 1);
        fence_mbar_init();
    }
    // flipped, transposed weights of layers 2 and 1 (units of co, rows of ci)
    for (int l = 0; l < 2; ++l) {
        const __nv_bfloat16 *w = l == 0 ? ar.w2 : ar.w1;
        __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(wraw + l * net_wbytes(4));
        for (int i = tid; i < CNN_K * 4 * CNN_C * 8; i += NET_THREADS) {
            const int e = i & 7, ci = (i >> 3) & 31, u = (i >> 8) & 3, k = i >> 10;
            dst[net_wplace(4, k, u, ci, e)] =
                w[((u * 8 + e) * CNN_C + ci) * CNN_K + (CNN_K - 1 - k)];
        }
    }
    for (int i = tid; i < CNN_C * CNN_K; i += NET_THREADS) w3[i] = __bfloat162float(ar.w3[i]);
    fence_proxy_async();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm = s_tmem;
    const float inv = 1.0f / (float)ar.n;
    double loss = 0.0;
    uint32_t phase = 0;
    bool failed = false;
    for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
        const int b = tile / tiles_per_curve;
        const int t0 = (tile - b * tiles_per_curve) * BACK_OUT;
        const int own_end = min(T, t0 + BACK_OUT);
        for (int i = tid; i < BACK_G4; i += NET_THREADS) {  // G_3 and the loss, bin t0 - 12 + i
            const int t = t0 - 12 + i;
            float g = 0.0f;
            if (t >= 0 && t < T) {
                const float z = ar.logits[(int64_t)b * T + t], y = ar.labels[(int64_t)b * T + t];
                g = bce_grad(z, y, ar.wpos, inv);
                if (t >= t0 && t < own_end) loss += (double)bce_loss(z, y, ar.wpos);
            }
            g3[i] = g;
        }
        __syncthreads();
        for (int it = tid; it < NET_XROWS * 4; it += NET_THREADS) {
            const int u = it / NET_XROWS, i = it - u * NET_XROWS;
            const int t = t0 - 8 + i;
            const bool inside = t >= 0 && t < T;
            const int64_t at = ((int64_t)b * CNN_C + u * 8) * T + t;
            float a[8], v[8], g[CNN_K];
#pragma unroll
            for (int e = 0; e < 8; ++e) a[e] = inside ? ar.act3[at + (int64_t)e * T] : 0.0f;
#pragma unroll
            for (int k = 0; k < CNN_K; ++k) g[k] = g3[i + 8 - k];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                float sum = 0.0f;
#pragma unroll
                for (int k = 0; k < CNN_K; ++k)
                    sum = fmaf(g[k], w3[(u * 8 + e) * CNN_K + k], sum);
                v[e] = a[e] > 0.0f ? sum : 0.0f;
                if (inside && t >= t0 && t < own_end) ar.g2[at + (int64_t)e * T] = v[e];
            }
            net_store_row(x0 + (uint32_t)(u * NET_UNIT + i * 16), v);
        }
        fence_proxy_async();
        __syncthreads();
        for (int l = 0; l < 2; ++l) {
            if (tid == 0 && tile != ar.wait.skip) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                for (int mb = 0; mb < 2; ++mb) {
                    net_layer_mma<4>(tm + (uint32_t)(mb * NET_GRP * CNN_C),
                                     net_desc_lo(x0 + (uint32_t)(mb * NET_BLOCK * 16), NET_UNIT),
                                     w0 + (uint32_t)(l * net_wbytes(4)));
                    net_commit(&done[mb]);
                }
            }
            __syncwarp();
            const int mb = warp >> 2, warp4 = warp & 3, r = mb * NET_BLOCK + warp4 * 32 + lane;
            const int t = t0 - 4 + 4 * l + r;
            const bool mine = warp4 * 32 + lane < NET_BLOCK;  // the block's last lane has no row
            const bool inside = mine && t >= 0 && t < T;
            const bool own = inside && t >= t0 && t < own_end;
            const int64_t at = (int64_t)b * CNN_C * T + t;
            const float *act = l == 0 ? ar.act2 : ar.act1;
            float *out = l == 0 ? ar.g1 : ar.g0;
            uint32_t mask = 0u;  // channels whose activation is positive, read under the instructions
            if (inside)
#pragma unroll
                for (int c = 0; c < CNN_C; ++c)
                    mask |= (act[at + (int64_t)c * T] > 0.0f ? 1u : 0u) << c;
            const bool ok = mbar_wait(&done[mb], phase, ar.wait.limit);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t src = tm + (uint32_t)(mb * NET_GRP * CNN_C) + ((uint32_t)(warp & 3) << 21);
            net_exchange(src, xch[mb], warp4, 1 + mb);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float v[16];
                net_sums(v, src, xch[mb], warp4, h);
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    v[c] = (mask >> (h * 16 + c)) & 1u ? v[c] : 0.0f;
                    if (own) out[at + (int64_t)(h * 16 + c) * T] = v[c];
                }
                if (l == 0 && mine) {
                    net_store_row(x0 + (uint32_t)(2 * h * NET_UNIT + r * 16), v);
                    net_store_row(x0 + (uint32_t)((2 * h + 1) * NET_UNIT + r * 16), v + 8);
                }
            }
            phase ^= 1u;
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            fence_proxy_async();
            failed = __syncthreads_or(!ok);
            if (failed) break;
        }
        if (failed) {  // a wait gave up: the loss is NaN, and the gradient by the status word
            if (tid == 0) atomicExch(ar.wait.status, CETRA_ETIMEOUT);
            mbar_wait(&done[0], phase ^ 1u, ar.wait.limit);  // before the tensor memory goes
            mbar_wait(&done[1], phase ^ 1u, ar.wait.limit);
            loss = __longlong_as_double(0x7ff8000000000000ll);
            break;
        }
    }
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_down_sync(0xFFFFFFFFu, loss, o);
    if (lane == 0) s_loss[warp] = loss;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (tid == 0) {
        for (int x = 1; x < NET_THREADS / 32; ++x) loss += s_loss[x];
        atomicAdd(ar.loss, loss / (double)ar.n);
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm),
                     "n"(NET_TMEM_COLS));
}

// Weight and bias gradients of every layer in one launch:
// dW[co][ci][k] = sum_{b,t} G[b][co][t] x[b][ci][t + k - 4],  db[co] = sum_{b,t} G[b][co][t].
// Each layer has its share of the blocks; a block goes through its tiles of bins with the sums in
// registers and leaves one partial gradient, which cnn_grad_sum_kernel adds over the blocks (no
// atomics: 4.7 M scattered ones per layer were most of the time of the kernel this replaces,
// 150 us for a 32 -> 32 layer of 32 curves). Thread: one input channel x 8 output channels x 9
// taps over WG_SUB bins of the tile: 36 packed FP32x2 multiply-adds per bin on the pair (G of two
// output channels) x (x, x), so the FMA pipe is the bound (55 % busy, 153 us for 32 curves); the
// 9-wide input window rotates through registers, G comes as broadcast 16-byte loads. Tiles are
// staged by asynchronous copies, the next one under the arithmetic of this one, and handed out as
// blocks come free (206 us with plain loads and a fixed share).
constexpr int WG_THREADS = 256;
constexpr int WG_SUB = 63;   // bins per thread and tile (a multiple of the taps: the window's rotation)
constexpr int WG_LDG = 36;   // floats per bin of the staged G (16-byte aligned, few bank conflicts)
constexpr int WG_LAST = 128; // bins per tile of the last layer
struct wgrad_job {
    const float *x, *g;  // input [B][cin][T], gradient [B][32][T] (last layer: from the logits)
    float *part;         // [blocks][size] partial gradients: W then b
    int cin, cout, first, blocks, size;
};
struct wgrad_args {
    wgrad_job job[CNN_LAYERS];
    const float *logits, *labels;  // [B][T]
    int *next;                     // [layer] tiles handed out beyond each block's first (zeroed)
    const int *status;             // not 0: a wait gave up, the gradient is NaN
    int *lost;                     // the status word at the time of the gradient
    float wpos;
    int64_t n;
    int B, T;
};
// Input channels as lanes hold them (16 or 32), thread groups along the bins, bins per tile.
__host__ __device__ constexpr int wg_cinp(int cin) { return cin <= 16 ? 16 : 32; }
__host__ __device__ constexpr int wg_subs(int cin) { return WG_THREADS / 4 / wg_cinp(cin); }
__host__ __device__ constexpr int wg_tile(int cin) { return wg_subs(cin) * WG_SUB; }
constexpr int WG_STAGE = 16 * (4 * WG_SUB + 9) + 4 * WG_SUB * WG_LDG;  // floats of a staged tile
constexpr size_t WG_SMEM = (size_t)2 * WG_STAGE * sizeof(float);
static_assert(WG_STAGE >= 32 * (2 * WG_SUB + 9) + 2 * WG_SUB * WG_LDG && WG_STAGE % 4 == 0 &&
                  2 * WG_STAGE >= 72 * 128 && 2 * WG_STAGE >= CNN_C * (WG_LAST + 9) + WG_LAST,
              "weight gradient staging");

// Asynchronous copy of one float (zero when !ok: nothing is read then).
__device__ __forceinline__ void copy_float(float *dst, const float *src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(ok ? 4 : 0)
                 : "memory");
}

// Stage one tile of a layer's input and output gradient (asynchronous; one commit group).
__device__ __forceinline__ void wgrad_stage(const wgrad_job &jb, int tile, int per, int tile_n,
                                            int cinp, int T, float *xs, float *gs) {
    const int b = tile / per, t0 = (tile - b * per) * tile_n, XS = tile_n + 9;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float *xb = jb.x + (int64_t)b * jb.cin * T, *gb = jb.g + (int64_t)b * CNN_C * T;
    for (int c = warp; c < cinp; c += WG_THREADS / 32)
        for (int u = lane; u < tile_n + 8; u += 32) {
            const int t = t0 - 4 + u;
            const bool ok = c < jb.cin && t >= 0 && t < T;
            copy_float(&xs[c * XS + u], ok ? xb + (int64_t)c * T + t : jb.x, ok);
        }
    for (int c = warp; c < CNN_C; c += WG_THREADS / 32)
        for (int u = lane; u < tile_n; u += 32) {
            const bool ok = t0 + u < T;
            copy_float(&gs[u * WG_LDG + c], ok ? gb + (int64_t)c * T + t0 + u : jb.g, ok);
        }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ void wgrad_last(const wgrad_args &ar, const wgrad_job &jb, float *smem) {
    constexpr int XS = WG_LAST + 9;
    float *xs = smem, *gs = smem + CNN_C * XS;
    const int tid = threadIdx.x, ci = tid & 31, warp = tid >> 5;
    const int T = ar.T, per = (T + WG_LAST - 1) / WG_LAST;
    const float inv = 1.0f / (float)ar.n;
    float acc[CNN_K], db = 0.0f;
#pragma unroll
    for (int k = 0; k < CNN_K; ++k) acc[k] = 0.0f;
    for (int tile = blockIdx.x - jb.first; tile < per * ar.B; tile += jb.blocks) {
        const int b = tile / per, t0 = (tile - b * per) * WG_LAST;
        __syncthreads();
        for (int c = warp; c < CNN_C; c += WG_THREADS / 32)  // (in flight together)
            for (int u = ci; u < WG_LAST + 8; u += 32) {
                const int t = t0 - 4 + u;
                const bool ok = t >= 0 && t < T;
                copy_float(&xs[c * XS + u], ok ? jb.x + ((int64_t)b * CNN_C + c) * T + t : jb.x,
                           ok);
            }
        asm volatile("cp.async.commit_group;" ::: "memory");
        for (int u = tid; u < WG_LAST; u += WG_THREADS) {
            const int64_t at = (int64_t)b * T + t0 + u;
            gs[u] = t0 + u < T ? bce_grad(ar.logits[at], ar.labels[at], ar.wpos, inv) : 0.0f;
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const int u0 = warp * (WG_LAST / 8);
        for (int u = u0; u < u0 + WG_LAST / 8; ++u) {
            const float g = gs[u];
            db += g;
#pragma unroll
            for (int k = 0; k < CNN_K; ++k) acc[k] = fmaf(g, xs[ci * XS + u + k], acc[k]);
        }
    }
    __syncthreads();
    float *red = smem;  // [8 warps][32][9], then [8] biases
#pragma unroll
    for (int k = 0; k < CNN_K; ++k) red[(warp * CNN_C + ci) * CNN_K + k] = acc[k];
    if (ci == 0) red[8 * CNN_C * CNN_K + warp] = db;
    __syncthreads();
    float *out = jb.part + (int64_t)(blockIdx.x - jb.first) * jb.size;
    for (int i = tid; i < CNN_C * CNN_K; i += WG_THREADS) {
        float v = 0.0f;
        for (int w = 0; w < 8; ++w) v += red[w * CNN_C * CNN_K + i];
        out[i] = v;
    }
    if (tid == 0) {
        float v = 0.0f;
        for (int w = 0; w < 8; ++w) v += red[8 * CNN_C * CNN_K + w];
        out[CNN_C * CNN_K] = v;
    }
}

__global__ void __launch_bounds__(WG_THREADS, 2) cnn_wgrad_kernel(wgrad_args ar) {
    extern __shared__ __align__(16) float wg_smem[];
    int l = 0;
    while (l < CNN_LAYERS - 1 && (int)blockIdx.x >= ar.job[l].first + ar.job[l].blocks) ++l;
    const wgrad_job jb = ar.job[l];
    if (l == CNN_LAYERS - 1) {  // uniform over the block
        wgrad_last(ar, jb, wg_smem);
        return;
    }
    const int tid = threadIdx.x, cin = jb.cin, T = ar.T;
    const int cinp = wg_cinp(cin), subs = wg_subs(cin), tile_n = wg_tile(cin), XS = tile_n + 9;
    const int g_at = (cinp * XS + 3) & ~3;  // G after the input, in each of the two stages
    const int ci = tid % cinp, rest = tid / cinp, cg = rest & 3, sub = rest >> 2;
    const int per = (T + tile_n - 1) / tile_n;
    unsigned long long acc[4][CNN_K];  // (output channels 2 p, 2 p + 1 of the thread's eight)
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int k = 0; k < CNN_K; ++k) acc[p][k] = 0ull;
    float db = 0.0f;
    // tiles after a block's first are handed out as blocks come free: an SM may hold blocks of
    // layers of different length
    __shared__ int s_next;
    const int n_tiles = per * ar.B;
    int tile = blockIdx.x - jb.first, stage = 0;
    if (tid == 0) s_next = jb.blocks + atomicAdd(&ar.next[l], 1);
    if (tile < n_tiles) wgrad_stage(jb, tile, per, tile_n, cinp, T, wg_smem, wg_smem + g_at);
    __syncthreads();
    for (int after; tile < n_tiles; tile = after, stage ^= 1) {
        // the next tile lands in the other stage while this one is used
        float *xs = wg_smem + stage * WG_STAGE, *gs = xs + g_at;
        float *xn_s = wg_smem + (stage ^ 1) * WG_STAGE;
        after = s_next;
        if (after < n_tiles) {
            wgrad_stage(jb, after, per, tile_n, cinp, T, xn_s, xn_s + g_at);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        if (tid == 0 && after < n_tiles) s_next = jb.blocks + atomicAdd(&ar.next[l], 1);
        const float *xr = xs + ci * XS + sub * WG_SUB, *gr = gs + sub * WG_SUB * WG_LDG + cg * 8;
        unsigned long long win[CNN_K];
#pragma unroll
        for (int k = 0; k < CNN_K; ++k) win[k] = pack2(make_float2(xr[k], xr[k]));
        for (int it = 0; it < WG_SUB; it += CNN_K)
#pragma unroll
            for (int s = 0; s < CNN_K; ++s) {
                const ulonglong2 ga = *reinterpret_cast<const ulonglong2 *>(gr + (it + s) * WG_LDG);
                const ulonglong2 gc =
                    *reinterpret_cast<const ulonglong2 *>(gr + (it + s) * WG_LDG + 4);
                const unsigned long long g[4] = {ga.x, ga.y, gc.x, gc.y};
                const float xn = xr[it + s + CNN_K];
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int k = 0; k < CNN_K; ++k)
                        asm("fma.rn.f32x2 %0, %1, %2, %0;"
                            : "+l"(acc[p][k])
                            : "l"(g[p]), "l"(win[(s + k) % CNN_K]));
                win[s] = pack2(make_float2(xn, xn));
            }
        for (int u = tid >> 5; u < tile_n; u += WG_THREADS / 32) db += gs[u * WG_LDG + (tid & 31)];
        __syncthreads();  // the stage is read before the next copies into it
    }
    // the thread groups' sums of each weight, then this block's partial gradient
    float *red = wg_smem;  // [72][128]
    const int slot = cg * cinp + ci;
    for (int x = 1; x < subs; ++x) {
        __syncthreads();
        if (sub == x)
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int k = 0; k < CNN_K; ++k) {
                    const float2 v = unpack2(acc[p][k]);
                    red[((p * CNN_K + k) * 2) * 128 + slot] = v.x;
                    red[((p * CNN_K + k) * 2 + 1) * 128 + slot] = v.y;
                }
        __syncthreads();
        if (sub == 0)
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int k = 0; k < CNN_K; ++k) {
                    float2 v = unpack2(acc[p][k]);
                    v.x += red[((p * CNN_K + k) * 2) * 128 + slot];
                    v.y += red[((p * CNN_K + k) * 2 + 1) * 128 + slot];
                    acc[p][k] = pack2(v);
                }
    }
    float *out = jb.part + (int64_t)(blockIdx.x - jb.first) * jb.size;
    if (sub == 0 && ci < cin)
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int k = 0; k < CNN_K; ++k) {
                const float2 v = unpack2(acc[p][k]);
                const int co = cg * 8 + 2 * p;
                out[(co * cin + ci) * CNN_K + k] = v.x;
                out[((co + 1) * cin + ci) * CNN_K + k] = v.y;
            }
    __syncthreads();
    red[tid] = db;
    __syncthreads();
    if (tid < CNN_C) {
        float v = 0.0f;
        for (int w = 0; w < WG_THREADS / 32; ++w) v += red[w * 32 + tid];
        out[CNN_C * cin * CNN_K + tid] = v;
    }
}

// The gradient: the blocks' partial gradients of each layer, added by 8 thread rows of 4 sums each
// (one thread per weight waited 13 us for its chain of loads).
constexpr int GS_ROWS = 8;
__global__ void __launch_bounds__(32 * GS_ROWS)
cnn_grad_sum_kernel(wgrad_args ar, float *__restrict__ grads) {
    __shared__ float red[GS_ROWS][32];
    const wgrad_job jb = ar.job[blockIdx.y];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (i < jb.size) {
        int x = row;
        for (; x + 3 * GS_ROWS < jb.blocks; x += 4 * GS_ROWS)
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] += jb.part[(int64_t)(x + k * GS_ROWS) * jb.size + i];
        for (; x < jb.blocks; x += GS_ROWS) v[0] += jb.part[(int64_t)x * jb.size + i];
    }
    red[row][lane] = (v[0] + v[1]) + (v[2] + v[3]);
    __syncthreads();
    if (row == 0 && i < jb.size) {
        float sum = red[0][lane];
#pragma unroll
        for (int r = 1; r < GS_ROWS; ++r) sum += red[r][lane];
        int64_t off = 0;
        for (int l = 0; l < (int)blockIdx.y; ++l) off += ar.job[l].size;
        const int status = *ar.status;
        grads[off + i] = status == 0 ? sum : __int_as_float(0x7fc00000);
        if (i == 0 && blockIdx.y == 0) *ar.lost = status;
    }
}

__global__ void cnn_round_kernel(const float *__restrict__ w, __nv_bfloat16 *__restrict__ wb,
                                 int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) wb[i] = __float2bfloat16_rn(w[i]);
}

// Adam on the FP32 training copy. Nothing changes when a wait of the gradient's launches gave up.
__global__ void cnn_adam_kernel(float *__restrict__ w, const float *__restrict__ g,
                                float *__restrict__ m, float *__restrict__ v, int64_t n, float lr,
                                float b1, float b2, float eps, float c1, float c2,
                                const int *__restrict__ lost) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || *lost != 0) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Proposal map: m[b][t] = p[b][t] max_j max(f[b][j][t], 0), the network's transit
// probability times the best window LR of the bin (Sec. 2.2). (Measured against p times the
// window SNR and p^2 times the SNR: this weighting recovers the most injected planets.)
__global__ void cnn_map_kernel(const float *__restrict__ prob, const float *__restrict__ f,
                               int J, int T, int64_t n, float *__restrict__ out) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += stride) {
        const int64_t b = x / T, t = x % T;
        const float *fb = f + b * J * T + t;
        float m = 0.0f;
        for (int j = 0; j < J; ++j) m = fmaxf(m, fb[(int64_t)j * T]);
        out[x] = prob[x] * m;
    }
}

// Period comb over per-bin maps p[b][t]: curve b has V = n_valid[b] valid bins of bw[b] days.
// Interval q has log-spaced edges lo = p_lo (p_hi / p_lo)^(q / n_int), hi = the same at q + 1
// (days), or blo, bhi in bins. Its trial periods are Pb_m = blo + (bhi - blo)(m + 1/2) / nP,
// m < nP = max(1, ceil((bhi - blo) V / blo)), so that the phase of the last epoch drifts by at
// most about one bin between neighbouring trials; trials below 1 bin or above V / 2 are
// skipped. Epochs run in 32.32 fixed point: F = floor(Pb 2^32 + 1/2), and for each phase
// ph < ceil(Pb) the epochs are t_e = (ph 2^32 + e F + 2^31) >> 32 < V; the score is
// sum_e p[t_e] / sqrt(E). The interval's score is the best of those, and 0 if none is positive.
//
// An epoch's offset o_e = (e F + 2^31) >> 32 is the same for every phase of a trial (t_e = ph +
// o_e, phases being whole bins), so a warp takes a trial and up to COMB_ROWS x 32 of its phases:
// the offset is worked out once per epoch for the warp, and each lane adds one map cell per row
// (consecutive lanes read consecutive cells). Bound: the shared-memory loads, 32 cells per clock
// and SM; with the epoch arithmetic in every lane it was issue.
//
// One block per interval and `cpb` curves. The interval's edges (two FP64 powers) are worked out
// by two lanes once per block, and a curve's interval in bins by one lane: every FP64
// instruction of a warp holds the SM's FP64 pipe for 16 clocks, and with all the warps of a
// block per (interval, curve) doing it that was two thirds of the time. A curve's map is staged in
// shared memory when it fits; the trials' own FP64 arithmetic (Pb, F, phase count) is done once
// per trial into shared memory, COMB_CHUNK trials at a time.
// Measured (256 curves, 4,096 bins, 512 intervals): 5.3 ms; 15.8 ms with a block per (interval,
// curve) and a lane per (trial, phase). The shared loads alone: 2.2 ms.
constexpr int COMB_CHUNK = 256;
constexpr int COMB_ROWS = 16;
constexpr int COMB_THREADS = 256;

// The larger of `best` and the best score of phases ph0 + lane + 32 r (r < R, below nph) of one
// trial. Phases of equal epoch counts are compared by their sums (a rounded division by the same
// number keeps their order), and the square root and the division are taken only where they may
// beat `best`: m / sqrt(n) > best needs m^2 > best^2 n (1 - 2^-17), whose left side and right
// side are rounded by far less (below 1e-15 the squares might not be normal). PAD: cells up to
// 32 R past the last valid one may be read (a phase that has no further epoch is done with, so
// what is added to it does not matter).
// Short trials (nph <= 16, R = 1) share a warp: `mine` is the lane's phase and F its own trial's.
template <int R, bool PAD>
__device__ __forceinline__ float comb_unit(const float *__restrict__ src, uint32_t V,
                                           unsigned long long F, uint32_t ph0, uint32_t mine,
                                           uint32_t nph, float best) {
    const float *cell = src + mine;
    const uint32_t top = ph0 + 32 * R - 1;
    float s[R];
#pragma unroll
    for (int r = 0; r < R; ++r) s[r] = 0.0f;
    unsigned long long acc = 1ull << 31;
    uint32_t o = 0;
    int n = 0;
    // epochs that every phase has, four at a time (an epoch is at most `step` cells on)
    const uint32_t step = (uint32_t)(F >> 32) + 1u;
    for (const uint32_t last = top + 4 * step; o + last < V; n += 4) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
#pragma unroll
            for (int r = 0; r < R; ++r) s[r] += cell[o + 32 * r];
            acc += F;
            o = (uint32_t)(acc >> 32);
        }
    }
    for (; o + top < V; ++n) {
#pragma unroll
        for (int r = 0; r < R; ++r) s[r] += cell[o + 32 * r];
        acc += F;
        o = (uint32_t)(acc >> 32);
    }
    for (uint32_t have = nph;; ++n) {  // phases below `have` have n epochs or more
        const uint32_t lim = o < V ? V - o : 0u;  // phases below lim have the next one too
        float m = 0.0f;
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (mine + 32 * r >= lim && mine + 32 * r < have) m = fmaxf(m, s[r]);
        const float fn = (float)n;
        if (m > 0.0f && !(best > 1e-15f && m * m < best * best * fn * (1.0f - 1.0f / 131072.0f)))
            best = fmaxf(best, m / sqrtf(fn));
        if (lim <= ph0) return best;
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (PAD || o + mine + 32 * r < V) s[r] += cell[o + 32 * r];
        have = min(have, lim);
        acc += F;
        o = (uint32_t)(acc >> 32);
    }
}

template <bool PAD>
__device__ __forceinline__ float comb_rows(int rows, const float *__restrict__ src, uint32_t V,
                                           unsigned long long F, uint32_t ph0, uint32_t nph,
                                           float best) {
    const uint32_t mine = ph0 + (threadIdx.x & 31);
    switch (rows) {
        case 1: return comb_unit<1, PAD>(src, V, F, ph0, mine, nph, best);
        case 2: return comb_unit<2, PAD>(src, V, F, ph0, mine, nph, best);
        case 3: return comb_unit<3, PAD>(src, V, F, ph0, mine, nph, best);
        case 4: return comb_unit<4, PAD>(src, V, F, ph0, mine, nph, best);
        case 6: return comb_unit<6, PAD>(src, V, F, ph0, mine, nph, best);
        case 8: return comb_unit<8, PAD>(src, V, F, ph0, mine, nph, best);
        case 12: return comb_unit<12, PAD>(src, V, F, ph0, mine, nph, best);
        default: return comb_unit<16, PAD>(src, V, F, ph0, mine, nph, best);
    }
}

template <bool SMEM>
__global__ void __launch_bounds__(COMB_THREADS, 3)
cnn_comb_kernel(const float *__restrict__ p, const double *__restrict__ bw,
                const int *__restrict__ n_valid, int T, int B, int cpb, double p_lo, double p_hi,
                int n_int, float *__restrict__ scores) {
    extern __shared__ float cmap[];
    __shared__ unsigned long long trial_F[COMB_CHUNK];
    __shared__ uint32_t trial_nph[COMB_CHUNK];
    __shared__ double edge[2], s_blo, s_bhi;
    __shared__ int64_t s_nP;  // trials of the interval, 0: none
    __shared__ uint32_t s_nph;
    __shared__ float red[COMB_THREADS / 32];
    const int q = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid < 2) edge[tid] = p_lo * pow(p_hi / p_lo, (double)(q + tid) / n_int);
    const int b1 = min(B, ((int)blockIdx.y + 1) * cpb);
    for (int b = blockIdx.y * cpb; b < b1; ++b) {
        const int V = n_valid ? min(max(n_valid[b], 0), T) : T;
        const float *pb = p + (int64_t)b * T;
        __syncthreads();  // the edges, or the previous curve's shared values
        if (SMEM)
            for (int t = tid; t < V; t += COMB_THREADS) cmap[t] = pb[t];
        if (tid == 0) {
            const double w = bw[b];
            const double blo = w > 0.0 ? edge[0] / w : 0.0, bhi = w > 0.0 ? edge[1] / w : 0.0;
            const bool any = w > 0.0 && V > 0 && bhi >= 1.0 && blo <= 0.5 * (double)V;
            s_nP = any ? max((int64_t)1, (int64_t)ceil((bhi - blo) * (double)V / blo)) : 0;
            // phases of the longest trial (<= V / 2 < 2^30)
            s_nph = any ? (uint32_t)ceil(fmin(bhi, 0.5 * (double)V)) : 0u;
            s_blo = blo;
            s_bhi = bhi;
        }
        __syncthreads();
        const float *src = SMEM ? cmap : pb;
        float best = 0.0f;
        const int64_t nP = s_nP;
        if (nP > 0) {  // uniform over the block
            const double blo = s_blo, bhi = s_bhi;
            // phases of a trial in `parts` equal units of `rows` x 32 (1 to 4, 6, 8, 12 or 16
            // rows), or several trials of few phases in a warp
            const uint32_t nrow = (s_nph + 31) / 32, parts = (nrow + COMB_ROWS - 1) / COMB_ROWS;
            uint32_t rows = (nrow + parts - 1) / parts;
            if (rows > 4) rows = rows <= 8 ? (rows + 1) & ~1u : (rows + 3) & ~3u;
            const int share = s_nph <= 4 ? 8 : s_nph <= 8 ? 4 : s_nph <= 16 ? 2 : 1;
            for (int64_t m0 = 0; m0 < nP; m0 += COMB_CHUNK) {
                const int cnt = (int)min((int64_t)COMB_CHUNK, nP - m0);
                __syncthreads();  // the previous chunk's trials are no longer read
                for (int i = tid; i < cnt; i += COMB_THREADS) {
                    const double Pb = blo + (bhi - blo) * ((double)(m0 + i) + 0.5) / (double)nP;
                    const bool ok = Pb >= 1.0 && Pb <= 0.5 * (double)V;
                    trial_F[i] = ok ? (unsigned long long)floor(Pb * 4294967296.0 + 0.5) : 0ull;
                    trial_nph[i] = ok ? (uint32_t)ceil(Pb) : 0u;
                }
                __syncthreads();
                if (share > 1) {
                    const int width = 32 / share;
                    for (int m0w = wid * share; m0w < cnt; m0w += COMB_THREADS / 32 * share) {
                        const int m = m0w + lane / width;
                        const uint32_t nph = m < cnt ? trial_nph[m] : 0u;
                        if (nph)
                            best = comb_unit<1, SMEM>(src, V, trial_F[m], 0u,
                                                      (uint32_t)(lane % width), nph, best);
                    }
                    continue;
                }
                for (int m = wid; m < cnt; m += COMB_THREADS / 32) {
                    const uint32_t nph = trial_nph[m];
                    const unsigned long long F = trial_F[m];
                    for (uint32_t ph0 = 0; ph0 < nph; ph0 += rows * 32)
                        best = comb_rows<SMEM>((int)rows, src, V, F, ph0, nph, best);
                }
            }
        }
        for (int o = 16; o > 0; o >>= 1)
            best = fmaxf(best, __shfl_down_sync(0xFFFFFFFFu, best, o));
        if (lane == 0) red[wid] = best;
        __syncthreads();
        if (tid == 0) {
            float mx = 0.0f;
            for (int i = 0; i < COMB_THREADS / 32; ++i) mx = fmaxf(mx, red[i]);
            scores[(int64_t)b * n_int + q] = mx;
        }
    }
}

unsigned grid_for(int64_t n, int threads, int num_sms) {
    int64_t blocks = (n + threads - 1) / threads;
    if (blocks > (int64_t)num_sms * 32) blocks = (int64_t)num_sms * 32;
    return (unsigned)std::max<int64_t>(blocks, 1);
}

}  // namespace

// ------------------------------------------------------------------------------- host side

struct cetra_cnn {
    int device = 0;
    int cin = 0, T = 0, max_batch = 0;
    int ch_in[CNN_LAYERS], ch_out[CNN_LAYERS];
    int64_t w_off[CNN_LAYERS], b_off[CNN_LAYERS], n_params = 0;
    float *d_params = nullptr, *d_grads = nullptr, *d_m = nullptr, *d_v = nullptr;
    __nv_bfloat16 *d_wb = nullptr;  // BF16 weights
    float *d_act[CNN_LAYERS + 1] = {};  // act[0] = log1p(features), act[l + 1] = layer l output
    float *d_g[CNN_LAYERS - 1] = {};  // gradients of layers 0 .. 2 [max_batch][32][T]
    float *d_part = nullptr;          // partial weight gradients of the blocks
    net_words *d_words = nullptr;
    void *d_mem = nullptr;
    int adam_step = 0;
    long long wait_limit = FT_WAIT_CYCLES;
    int skip[2] = {-1, -1};  // self-test: tiles of the forward and the gradient pass left out
};

namespace {

int cnn_fail(cetra_ctx *ctx, cudaError_t e, const char *what) {
    return set_error(ctx, CETRA_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// Blocks of the weight-gradient launch (two per SM), and the largest partial gradient.
int wgrad_blocks(int num_sms) { return 2 * num_sms; }
constexpr size_t WG_PART = (size_t)CNN_C * CNN_C * CNN_K + CNN_C;

// The forward pass: probabilities of B curves into prob, or (prob NULL, training) the layers'
// activations and the logits into the network's buffers.
cudaError_t forward(cetra_ctx *ctx, cetra_cnn *n, const float *features, int B, float *prob) {
    net_layers net;
    for (int l = 0; l < CNN_LAYERS; ++l) {
        net.w[l] = n->d_wb + n->w_off[l];
        net.bias[l] = n->d_params + n->b_off[l];
    }
    for (int l = 0; l <= CNN_LAYERS; ++l) net.act[l] = n->d_act[l];
    net.wait = {&n->d_words->status, n->wait_limit, n->skip[0]};
    const int per = (n->T + NET_OUT - 1) / NET_OUT;
    const int64_t tiles = (int64_t)per * B;
    if (tiles > 2147483647) return cudaErrorInvalidConfiguration;
    const unsigned blocks = (unsigned)std::min<int64_t>(tiles, 2 * (int64_t)ctx->num_sms);
    auto kern = prob ? cnn_net_kernel<false> : cnn_net_kernel<true>;
    kern<<<blocks, NET_THREADS, net_smem(n->cin), ctx->stream>>>(features, net, prob, n->cin, n->T,
                                                               (int)tiles, per);
    ctx->launches++;
    return cudaGetLastError();
}

cudaError_t round_weights(cetra_ctx *ctx, cetra_cnn *n) {
    cnn_round_kernel<<<(unsigned)((n->n_params + 255) / 256), 256, 0, ctx->stream>>>(
        n->d_params, n->d_wb, n->n_params);
    ctx->launches++;
    return cudaGetLastError();
}

}  // namespace

int *cnn_status_word(cetra_cnn *n) { return &n->d_words->status; }

extern "C" {

int cetra_cnn_create(cetra_ctx *ctx, int in_channels, int n_bins, int max_batch, uint64_t seed,
                     cetra_cnn **out) {
    if (!ctx || !out) return set_error(ctx, CETRA_EINVAL, "cnn_create: NULL argument");
    *out = nullptr;
    if (in_channels < 1 || in_channels > CNN_C || n_bins < 256 || n_bins % 256 ||
        max_batch < 1)
        return set_error(ctx, CETRA_EINVAL,
                         "cnn_create: need 1 <= in_channels <= 32, n_bins a multiple of 256, max_batch >= 1");
    cetra_cnn *n = new (std::nothrow) cetra_cnn;
    if (!n) return set_error(ctx, CETRA_ENOMEM, "cnn_create: host allocation");
    n->device = ctx->device;
    n->cin = in_channels;
    n->T = n_bins;
    n->max_batch = max_batch;
    int64_t off = 0;
    for (int l = 0; l < CNN_LAYERS; ++l) {
        n->ch_in[l] = l == 0 ? in_channels : CNN_C;
        n->ch_out[l] = l == CNN_LAYERS - 1 ? 1 : CNN_C;
        n->w_off[l] = off;
        off += (int64_t)n->ch_out[l] * n->ch_in[l] * CNN_K;
        n->b_off[l] = off;
        off += n->ch_out[l];
    }
    n->n_params = off;
    // He-normal weights, zero biases, from a seeded generator
    std::vector<float> init((size_t)off, 0.0f);
    std::mt19937_64 rng(seed);
    std::normal_distribution<float> nd(0.0f, 1.0f);
    for (int l = 0; l < CNN_LAYERS; ++l) {
        const float sd = std::sqrt(2.0f / (float)(n->ch_in[l] * CNN_K));
        for (int64_t i = 0; i < (int64_t)n->ch_out[l] * n->ch_in[l] * CNN_K; ++i)
            init[(size_t)(n->w_off[l] + i)] = sd * nd(rng);
    }
    const size_t P = (size_t)off;
    const size_t act = (size_t)max_batch * CNN_C * n_bins;
    const size_t logits = (size_t)max_batch * n_bins;
    const size_t part = (size_t)wgrad_blocks(ctx->num_sms) * WG_PART;
    const size_t bytes = P * sizeof(float) * 4 + P * sizeof(__nv_bfloat16) + 256 * 16 +
                         (act * (CNN_LAYERS + CNN_LAYERS - 1) + logits + part) * sizeof(float);
    device_guard dguard(ctx->device);
    cudaError_t e = dguard.status;
    if (!e) e = cudaMalloc(&n->d_mem, bytes);
    if (e) {
        delete n;
        return set_error(ctx, CETRA_ENOMEM, "cnn_create: device allocation");
    }
    char *p = static_cast<char *>(n->d_mem);
    auto take = [&](size_t nb) {
        char *r = p;
        p += (nb + 255) & ~(size_t)255;
        return r;
    };
    n->d_params = reinterpret_cast<float *>(take(P * 4));
    n->d_grads = reinterpret_cast<float *>(take(P * 4));
    n->d_m = reinterpret_cast<float *>(take(P * 4));
    n->d_v = reinterpret_cast<float *>(take(P * 4));
    n->d_wb = reinterpret_cast<__nv_bfloat16 *>(take(P * 2));
    n->d_words = reinterpret_cast<net_words *>(take(sizeof(net_words)));
    for (int l = 0; l < CNN_LAYERS; ++l) n->d_act[l] = reinterpret_cast<float *>(take(act * 4));
    n->d_act[CNN_LAYERS] = reinterpret_cast<float *>(take(logits * 4));
    for (float *&g : n->d_g) g = reinterpret_cast<float *>(take(act * 4));
    n->d_part = reinterpret_cast<float *>(take(part * 4));
    e = cudaMemcpy(n->d_params, init.data(), P * 4, cudaMemcpyHostToDevice);
    if (!e) e = cudaMemset(n->d_m, 0, P * 4);
    if (!e) e = cudaMemset(n->d_v, 0, P * 4);
    if (!e) e = cudaMemset(n->d_words, 0, sizeof(net_words));
    for (auto fn : {cnn_net_kernel<false>, cnn_net_kernel<true>})
        if (!e)
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)net_smem(CNN_C));
    if (!e)
        e = cudaFuncSetAttribute(cnn_back_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)back_smem());
    if (!e)
        e = cudaFuncSetAttribute(cnn_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)WG_SMEM);
    if (!e) e = round_weights(ctx, n);
    if (!e) e = cudaStreamSynchronize(ctx->stream);
    if (e) {
        cudaFree(n->d_mem);
        delete n;
        return cnn_fail(ctx, e, "cnn_create");
    }
    *out = n;
    return CETRA_OK;
}

void cetra_cnn_destroy(cetra_cnn *n) {
    if (!n) return;
    device_guard dguard(n->device);
    cudaFree(n->d_mem);
    delete n;
}

int64_t cetra_cnn_param_count(const cetra_cnn *n) { return n ? n->n_params : 0; }

int cetra_cnn_shape(const cetra_cnn *n, int *in_channels, int *n_bins, int *max_batch) {
    if (!n) return CETRA_EINVAL;
    if (in_channels) *in_channels = n->cin;
    if (n_bins) *n_bins = n->T;
    if (max_batch) *max_batch = n->max_batch;
    return CETRA_OK;
}

int cetra_cnn_get_params(cetra_ctx *ctx, const cetra_cnn *n, float *host) {
    if (!ctx || !n || !host) return set_error(ctx, CETRA_EINVAL, "cnn_get_params: NULL argument");
    device_guard dguard(ctx->device);
    cudaError_t e = dguard.status;
    if (!e) e = cudaMemcpyAsync(host, n->d_params, (size_t)n->n_params * 4,
                                    cudaMemcpyDeviceToHost, ctx->stream);
    if (!e) e = cudaStreamSynchronize(ctx->stream);
    return e ? cnn_fail(ctx, e, "cnn_get_params") : CETRA_OK;
}

int cetra_cnn_set_params(cetra_ctx *ctx, cetra_cnn *n, const float *host) {
    if (!ctx || !n || !host) return set_error(ctx, CETRA_EINVAL, "cnn_set_params: NULL argument");
    device_guard dguard(ctx->device);
    cudaError_t e = dguard.status;
    if (!e) e = cudaMemcpyAsync(n->d_params, host, (size_t)n->n_params * 4,
                                    cudaMemcpyHostToDevice, ctx->stream);
    if (!e) e = round_weights(ctx, n);
    // new parameters start a new optimisation: clear Adam's moments and step count
    if (!e) e = cudaMemsetAsync(n->d_m, 0, (size_t)n->n_params * 4, ctx->stream);
    if (!e) e = cudaMemsetAsync(n->d_v, 0, (size_t)n->n_params * 4, ctx->stream);
    if (!e) e = cudaStreamSynchronize(ctx->stream);
    n->adam_step = 0;
    return e ? cnn_fail(ctx, e, "cnn_set_params") : CETRA_OK;
}

int cetra_cnn_forward(cetra_ctx *ctx, cetra_cnn *n, const float *d_features, int B,
                      float *d_prob) {
    if (!ctx || !n || !d_features || !d_prob || B < 1 || B > n->max_batch)
        return set_error(ctx, CETRA_EINVAL, "cnn_forward: bad argument");
    device_guard dguard(ctx->device);
    cudaError_t e = dguard.status;
    // One kernel reads the features (a halo of 16 bins per tile too) and writes the probabilities:
    // where the two overlap, these go to the network's own buffer first.
    const size_t rows = (size_t)B * n->T;
    const uintptr_t f0 = reinterpret_cast<uintptr_t>(d_features);
    const uintptr_t p0 = reinterpret_cast<uintptr_t>(d_prob);
    const bool overlap = p0 < f0 + rows * n->cin * sizeof(float) && f0 < p0 + rows * sizeof(float);
    float *prob = overlap ? n->d_act[CNN_LAYERS] : d_prob;
    if (!e) e = forward(ctx, n, d_features, B, prob);
    if (!e && overlap)
        e = cudaMemcpyAsync(d_prob, prob, rows * sizeof(float), cudaMemcpyDeviceToDevice,
                            ctx->stream);
    return e ? cnn_fail(ctx, e, "cnn_forward") : CETRA_OK;
}

int cetra_cnn_backward(cetra_ctx *ctx, cetra_cnn *n, const float *d_features,
                       const float *d_labels, int B, float pos_weight, double *loss,
                       float *host_grads) {
    if (!ctx || !n || !d_features || !d_labels || B < 1 || B > n->max_batch)
        return set_error(ctx, CETRA_EINVAL, "cnn_backward: bad argument");
    const int T = n->T;
    device_guard dguard(ctx->device);
    cudaError_t e = dguard.status;
    if (!e) e = cudaMemsetAsync(n->d_words, 0, sizeof(net_words), ctx->stream);
    if (!e) e = forward(ctx, n, d_features, B, nullptr);
    if (!e) {
        back_args ar{};
        ar.w1 = n->d_wb + n->w_off[1];
        ar.w2 = n->d_wb + n->w_off[2];
        ar.w3 = n->d_wb + n->w_off[3];
        ar.logits = n->d_act[CNN_LAYERS];
        ar.labels = d_labels;
        ar.act1 = n->d_act[1];
        ar.act2 = n->d_act[2];
        ar.act3 = n->d_act[3];
        ar.g0 = n->d_g[0];
        ar.g1 = n->d_g[1];
        ar.g2 = n->d_g[2];
        ar.loss = &n->d_words->loss;
        ar.wait = {&n->d_words->status, n->wait_limit, n->skip[1]};
        ar.wpos = pos_weight;
        ar.n = (int64_t)B * T;
        const int per = (T + BACK_OUT - 1) / BACK_OUT;
        if ((int64_t)per * B > 2147483647) e = cudaErrorInvalidConfiguration;
        const unsigned blocks =
            (unsigned)std::min<int64_t>((int64_t)per * B, 2 * (int64_t)ctx->num_sms);
        if (!e) {
            cnn_back_kernel<<<blocks, NET_THREADS, back_smem(), ctx->stream>>>(ar, T, per * B, per);
            ctx->launches++;
            e = cudaGetLastError();
        }
    }
    if (!e) {
        // every layer's share of the blocks by its multiply-adds (the last layer is bound by
        // reading its input: as a 32 -> 8 layer)
        wgrad_args ar{};
        ar.logits = n->d_act[CNN_LAYERS];
        ar.labels = d_labels;
        ar.next = n->d_words->next;
        ar.status = &n->d_words->status;
        ar.lost = &n->d_words->lost;
        ar.wpos = pos_weight;
        ar.n = (int64_t)B * T;
        ar.B = B;
        ar.T = T;
        const int slots = wgrad_blocks(ctx->num_sms);
        double weight[CNN_LAYERS], total = 0.0;
        for (int l = 0; l < CNN_LAYERS; ++l)
            total += weight[l] = l == CNN_LAYERS - 1 ? 8.0 : wg_cinp(n->ch_in[l]);
        int first = 0;
        float *part = n->d_part;
        for (int l = 0; l < CNN_LAYERS; ++l) {
            wgrad_job &jb = ar.job[l];
            jb.x = n->d_act[l];
            jb.g = l < CNN_LAYERS - 1 ? n->d_g[l] : nullptr;
            jb.cin = n->ch_in[l];
            jb.cout = n->ch_out[l];
            jb.size = jb.cout * jb.cin * CNN_K + jb.cout;
            const int tile = l < CNN_LAYERS - 1 ? wg_tile(jb.cin) : WG_LAST;
            const int64_t tiles = (int64_t)((T + tile - 1) / tile) * B;
            if (tiles > 2147483647) e = cudaErrorInvalidConfiguration;
            jb.first = first;
            jb.blocks = (int)std::max<int64_t>(
                1, std::min<int64_t>(tiles, (int64_t)(slots * weight[l] / total)));
            jb.part = part;
            part += (size_t)jb.blocks * jb.size;
            first += jb.blocks;
        }
        if (!e) {
            cnn_wgrad_kernel<<<first, WG_THREADS, WG_SMEM, ctx->stream>>>(ar);
            ctx->launches++;
            e = cudaGetLastError();
        }
        if (!e) {
            dim3 grid((unsigned)((WG_PART + 31) / 32), CNN_LAYERS);
            cnn_grad_sum_kernel<<<grid, 32 * GS_ROWS, 0, ctx->stream>>>(ar, n->d_grads);
            ctx->launches++;
            e = cudaGetLastError();
        }
    }
    net_words words{};
    if (!e && (loss || host_grads))
        e = cudaMemcpyAsync(&words, n->d_words, sizeof(words), cudaMemcpyDeviceToHost, ctx->stream);
    if (!e && host_grads)
        e = cudaMemcpyAsync(host_grads, n->d_grads, (size_t)n->n_params * 4,
                            cudaMemcpyDeviceToHost, ctx->stream);
    if (!e && (loss || host_grads)) e = cudaStreamSynchronize(ctx->stream);
    if (e) return cnn_fail(ctx, e, "cnn_backward");
    if (loss) *loss = words.loss;
    return words.status ? set_error(ctx, words.status, "cnn_backward: a device wait timed out")
                        : CETRA_OK;
}

int cetra_cnn_status(cetra_ctx *ctx, cetra_cnn *n, int *status) {
    if (!ctx || !n || !status) return set_error(ctx, CETRA_EINVAL, "cnn_status: NULL argument");
    device_guard dguard(ctx->device);
    int v = 0;
    cudaError_t e = dguard.status;
    if (!e) e = cudaMemcpyAsync(&v, &n->d_words->status, sizeof(int), cudaMemcpyDeviceToHost,
                                ctx->stream);
    if (!e) e = cudaMemsetAsync(&n->d_words->status, 0, sizeof(int), ctx->stream);
    if (!e) e = cudaStreamSynchronize(ctx->stream);
    if (e) return cnn_fail(ctx, e, "cnn_status");
    *status = v;
    return CETRA_OK;
}

int cetra_selftest_cnn_waits(cetra_cnn *n, int forward_tile, int gradient_tile,
                             int64_t wait_cycles) {
    if (!n || wait_cycles < 0) return CETRA_EINVAL;
    n->skip[0] = std::max(-1, forward_tile);
    n->skip[1] = std::max(-1, gradient_tile);
    n->wait_limit = wait_cycles ? wait_cycles : FT_WAIT_CYCLES;
    return CETRA_OK;
}

int cetra_cnn_adam(cetra_ctx *ctx, cetra_cnn *n, float lr, float beta1, float beta2, float eps) {
    if (!ctx || !n) return set_error(ctx, CETRA_EINVAL, "cnn_adam: NULL argument");
    device_guard dguard(ctx->device);
    if (dguard.status) return cnn_fail(ctx, dguard.status, "cnn_adam");
    n->adam_step++;
    const float c1 = 1.0f - std::pow(beta1, (float)n->adam_step);
    const float c2 = 1.0f - std::pow(beta2, (float)n->adam_step);
    cnn_adam_kernel<<<(unsigned)((n->n_params + 255) / 256), 256, 0, ctx->stream>>>(
        n->d_params, n->d_grads, n->d_m, n->d_v, n->n_params, lr, beta1, beta2, eps, c1, c2,
        &n->d_words->lost);
    ctx->launches++;
    cudaError_t e = cudaGetLastError();
    if (!e) e = round_weights(ctx, n);
    return e ? cnn_fail(ctx, e, "cnn_adam") : CETRA_OK;
}

int cetra_cnn_map(cetra_ctx *ctx, const float *d_prob, const float *d_features, int B,
                  int n_dur, int n_bins, float *d_map) {
    if (!ctx || !d_prob || !d_features || !d_map || B < 1 || n_dur < 1 || n_bins < 1)
        return set_error(ctx, CETRA_EINVAL, "cnn_map: bad argument");
    device_guard dguard(ctx->device);
    if (dguard.status) return cnn_fail(ctx, dguard.status, "cnn_map");
    const int64_t n = (int64_t)B * n_bins;
    cnn_map_kernel<<<grid_for(n, 256, ctx->num_sms), 256, 0, ctx->stream>>>(d_prob, d_features,
                                                                           n_dur, n_bins, n, d_map);
    ctx->launches++;
    cudaError_t e = cudaGetLastError();
    return e ? cnn_fail(ctx, e, "cnn_map") : CETRA_OK;
}

int cetra_cnn_comb(cetra_ctx *ctx, const float *d_prob, int B, int n_bins,
                   const double *d_bin_days, const int *d_n_valid, double p_lo, double p_hi,
                   int n_intervals, float *d_scores) {
    if (!ctx || !d_prob || !d_bin_days || !d_scores || B < 1 || B > 65535 || n_bins < 1 ||
        n_bins > (1 << 30) || n_intervals < 1 || !(p_lo > 0.0) || !(p_hi > p_lo))
        return set_error(ctx, CETRA_EINVAL, "cnn_comb: bad argument");
    device_guard dguard(ctx->device);
    if (dguard.status) return cnn_fail(ctx, dguard.status, "cnn_comb");
    // curves per block: as many as leave 32 blocks per SM (four waves), 16 at most
    const int64_t want = (int64_t)ctx->num_sms * 32;
    const int cpb =
        (int)std::max<int64_t>(1, std::min<int64_t>(16, (int64_t)B * n_intervals / want));
    dim3 grid((unsigned)n_intervals, (unsigned)((B + cpb - 1) / cpb));
    const size_t smem = ((size_t)n_bins + 32 * COMB_ROWS) * sizeof(float);
    cudaError_t e = cudaSuccess;
    if (smem <= kCombSmemMax) {
        e = cudaFuncSetAttribute(cnn_comb_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem);
        if (!e)
            cnn_comb_kernel<true><<<grid, COMB_THREADS, smem, ctx->stream>>>(
                d_prob, d_bin_days, d_n_valid, n_bins, B, cpb, p_lo, p_hi, n_intervals, d_scores);
    } else {
        cnn_comb_kernel<false><<<grid, COMB_THREADS, 0, ctx->stream>>>(
            d_prob, d_bin_days, d_n_valid, n_bins, B, cpb, p_lo, p_hi, n_intervals, d_scores);
    }
    ctx->launches++;
    if (!e) e = cudaGetLastError();
    return e ? cnn_fail(ctx, e, "cnn_comb") : CETRA_OK;
}

}  // extern "C"
