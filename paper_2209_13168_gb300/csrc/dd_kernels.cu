// GB300 (sm_103a) kernels of the exact divergence estimator:
//   ingest   validate + counting-sort events by (polarity plane, time bucket,
//            row), per window
//   eval     point contrast (Eqs. 11-13) and interval bound (Eqs. 14-19) on
//            shared-memory IWE tiles: a resident grid takes (job, row band)
//            units, a job being one task (or one split of it) of one window
//   keys     per-task integer keys from the per-task sums
//   control  Algorithm 1 on the device, one block per window: incumbent,
//            priority queue, pruning, the next round's jobs
//
// Arithmetic contract.  The warp is evaluated in IEEE binary32 with one
// rounding per operation, in this order, with no contraction into FMA:
//     g = 1/(1 - D*t_ref);  s = (1 - D*t)*g;  cell = floor((FOE + d*s) + 1/2),
// t_ref = tau (the window's end, the paper's warp) or 0 (its start).
// __fmul_rn/__fadd_rn/__fsub_rn/__frcp_rn are never contracted.  The pixel a
// warped event lands in is an integer decided by that arithmetic, and all
// later work (counts, sums of squares, keys) is exact integer arithmetic, so
// results do not depend on thread, block or launch order.
#include "dd_internal.cuh"
#include "../../include/dd.h"

#include <cfloat>
#include <math_constants.h>
#include <mutex>

namespace dd {

// ------------------------------------------------------------ warp (Eq. 11)

__device__ __forceinline__ float warp_g(float D, float tau) {
    return __frcp_rn(__fsub_rn(1.0f, __fmul_rn(D, tau)));
}
__device__ __forceinline__ float warp_s(float D, float t, float g) {
    return __fmul_rn(__fsub_rn(1.0f, __fmul_rn(D, t)), g);
}

// --------------------------------------------------- paired binary32 arithmetic

// Two binary32 values in one 64-bit register pair.  sm_103a adds and
// multiplies both halves in one instruction (add/mul.f32x2), each half
// rounded as the scalar operation is, so a warp's pair of offsets, scales or
// cells costs one issue slot instead of two; k_eval is bound by issue slots.
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pair(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float lo_of(f32x2 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi_of(f32x2 v) { return __uint_as_float((uint32_t)(v >> 32)); }
// A product as a fused multiply-add onto +0, which rounds once, to the
// product (a product of -0 becomes +0; no cell depends on that sign).  The
// plain mul.rn.f32x2 will not do: the assembler contracts it with a following
// add.rn.f32x2 into one rounding (measured: 39% of FOE + d s differ from the
// two scalar operations; none with this form).
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(0ull));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// Biased cells: for |v| < 2^22, v + 1.5 x 2^23 rounded towards minus infinity
// is floor(v) + 1.5 x 2^23 exactly, whose bit pattern is CELL0 + floor(v).
// Cells stay below 2^22 in magnitude: scales are at most 65 (D tau >= -64)
// and 4 (D tau <= 3/4), offsets at most 4096.  The conversion instruction
// this replaces runs at a sixteenth of the add's rate.
constexpr uint32_t CELL0 = 0x4B400000u;
__device__ constexpr float CELL0_F = 12582912.0f;
__device__ __forceinline__ f32x2 floor2(f32x2 v) {
    f32x2 r;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(v), "l"(pair(CELL0_F, CELL0_F)));
    return r;
}
// Eq. (12), pixel u covers [u - 1/2, u + 1/2): floor((foe + d s) + 1/2), biased,
// of one coordinate and of a pair.
__device__ __forceinline__ uint32_t cell1(float foe, float d, float s) {
    return __float_as_uint(__fadd_rd(__fadd_rn(__fadd_rn(foe, __fmul_rn(d, s)), 0.5f), CELL0_F));
}
__device__ __forceinline__ f32x2 cells2(f32x2 foe, f32x2 d, f32x2 s) {
    return floor2(add2(add2(foe, mul2(d, s)), pair(0.5f, 0.5f)));
}
// An event's biased pixel (x, y) at scale s.
__device__ __forceinline__ uint2 pixel_of(f32x2 foe, f32x2 d, float s) {
    const f32x2 c = cells2(foe, d, pair(s, s));
    return make_uint2((uint32_t)c, (uint32_t)(c >> 32));
}

// Relative widening of the per-event scale range (binary32 s(D) is monotone
// in D only up to a few ulps; 2^-19 covers the error for D*tau <= 3/4).
__device__ constexpr float WIDEN_DN = 1.0f - 0x1p-19f;
__device__ constexpr float WIDEN_UP = 1.0f + 0x1p-19f;
// Half a pixel plus a 2^-8 px margin (above the cell rounding error).
__device__ constexpr float HALF_PLUS = 0.50390625f;

// Checked builds (-DDD_CHECKED, the stand-in for a memory checker): every
// index into a shared tile, a window's events, a split accumulator or the
// sorted-event output is tested first; an index out of range sets a bit of
// g_dd_check and the access is skipped (nothing traps).  Bits: 1 point and
// one-pixel tile cells, 2 segment tile cells, 4 event indices, 8 ingest
// positions, 16 accumulator and image cells.  Other builds compile the tests
// away.
#ifdef DD_CHECKED
__device__ unsigned int g_dd_check;
__device__ __forceinline__ bool dd_in(long long i, long long n, unsigned bit) {
    if (i >= 0 && i < n) return true;
    atomicOr(&g_dd_check, bit);
    return false;
}
#define DD_IN(i, n, bit) dd_in((long long)(i), (long long)(n), (bit))
#else
#define DD_IN(i, n, bit) true
#endif

// Warp sum of 64-bit values as three 32-bit warp reductions (20, 20 and 24
// bits per part: 32 of each add up within 32 bits).
__device__ __forceinline__ unsigned long long warp_total(unsigned long long v) {
    const uint32_t a = __reduce_add_sync(0xffffffffu, (uint32_t)v & 0xFFFFFu);
    const uint32_t b = __reduce_add_sync(0xffffffffu, (uint32_t)(v >> 20) & 0xFFFFFu);
    const uint32_t c = __reduce_add_sync(0xffffffffu, (uint32_t)(v >> 40));
    return (unsigned long long)a + ((unsigned long long)b << 20) + ((unsigned long long)c << 40);
}

// Inclusive prefix sum over the warp.
__device__ __forceinline__ int warp_incl_scan(int v) {
    const int lane = threadIdx.x & 31;
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// ------------------------------------------------------------------ ingest

constexpr int INGEST_THREADS = 512;
// Blocks per ingest chunk: each takes CHUNK / INGEST_SUB consecutive events,
// so that a window of a few chunks still spreads over many SMs.
constexpr int INGEST_SUB = 8;
static_assert(CHUNK % INGEST_SUB == 0, "sub-chunks tile a chunk");
constexpr int MAX_BINS = 4096;

__device__ __forceinline__ bool event_ok(int xi, int yi, float ti, float tr, float tau, int W, int H) {
    return isfinite(ti) && tr >= 0.0f && tr <= tau && xi >= 0 && xi < W && yi >= 0 && yi < H;
}

// Sort key of an event: (polarity plane, time bucket, row).  Bucket b holds
// the events with t*scale in [b, b+1) (binary32 product), scale = n_tb/tau.
__device__ __forceinline__ int event_key(const Geom& g, int yi, float tr, float bscale, int plane) {
    int b = __float2int_rd(__fmul_rn(tr, bscale));
    b = min(max(b, 0), g.n_tb - 1);
    return (plane * g.n_tb + b) * g.H + yi;
}

// Plane of event i: 1 for polarity p <= 0 when the planes are split.
__device__ __forceinline__ int plane_of(const Geom& g, const WinIn& win, int64_t i) {
    return g.planes > 1 && win.p[i] <= 0 ? 1 : 0;
}

// Events [i0, i1) of the sub-chunk that block b ingests: sub-chunk
// b % INGEST_SUB of chunk b / INGEST_SUB, within that chunk's window.
__device__ __forceinline__ void sub_chunk(const WinIn& win, int chunk, int sub, int64_t& i0, int64_t& i1) {
    constexpr int SUB_EVENTS = CHUNK / INGEST_SUB;
    i0 = min(win.n, (int64_t)(chunk - win.chunk0) * CHUNK + (int64_t)sub * SUB_EVENTS);
    i1 = min(win.n, i0 + SUB_EVENTS);
}

// Block b counts its sub-chunk of its window into a shared histogram of the
// window's bins, then adds it to the window's global counts.
__global__ void __launch_bounds__(INGEST_THREADS) k_row_hist(Geom g, const WinIn* __restrict__ wins,
                                                             const int32_t* __restrict__ chunk_win,
                                                             int32_t* row_count, int32_t* err) {
    __shared__ int32_t h[MAX_BINS];
    const int chunk = blockIdx.x / INGEST_SUB;
    const int w = chunk_win[chunk];
    const WinIn win = wins[w];
    const int bins = bins_of(g);
    const float bscale = __fdiv_rn((float)g.n_tb, win.tau);
    for (int r = threadIdx.x; r < bins; r += blockDim.x) h[r] = 0;
    __syncthreads();
    int64_t i0, i1;
    sub_chunk(win, chunk, blockIdx.x % INGEST_SUB, i0, i1);
    int bad = 0;
    for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        const int xi = win.x[i], yi = win.y[i];
        const float ti = win.t[i];
        const float tr = __fsub_rn(ti, win.t0);
        if (!event_ok(xi, yi, ti, tr, win.tau, g.W, g.H)) { bad = 1; continue; }
        atomicAdd(&h[event_key(g, yi, tr, bscale, plane_of(g, win, i))], 1);
    }
    if (bad) atomicOr(&err[w], 1);
    __syncthreads();
    int32_t* rc = row_count + (size_t)w * bins;
    for (int r = threadIdx.x; r < bins; r += blockDim.x)
        if (h[r]) atomicAdd(&rc[r], h[r]);
}

// Exclusive scan of one window's bin counts (at most 4096 bins), block = window.
// Leaves the counts zero for the next call.
__global__ void __launch_bounds__(1024) k_row_scan(int bins, int32_t* row_count, int32_t* row_off, int32_t* cursor) {
    __shared__ int32_t wsum[32];
    const int w = blockIdx.x;
    row_count += (size_t)w * bins;
    cursor += (size_t)w * bins;
    row_off += (size_t)w * (bins + 1);
    const int per = (bins + 1023) / 1024;
    int base = threadIdx.x * per;
    int local[4];
    int tot = 0;
    for (int k = 0; k < per; k++) {
        int r = base + k;
        local[k] = r < bins ? row_count[r] : 0;
        if (r < bins) row_count[r] = 0;
        tot += local[k];
    }
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int v = tot;
    for (int o = 1; o < 32; o <<= 1) {
        int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) wsum[wid] = v;
    __syncthreads();
    if (wid == 0) {
        int s = wsum[lane];
        for (int o = 1; o < 32; o <<= 1) {
            int u = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += u;
        }
        wsum[lane] = s;
    }
    __syncthreads();
    int excl = v - tot + (wid ? wsum[wid - 1] : 0);
    for (int k = 0; k < per; k++) {
        int r = base + k;
        if (r < bins) { row_off[r] = excl; cursor[r] = excl; }
        excl += local[k];
    }
    if (threadIdx.x == 1023) row_off[bins] = excl;
}

// Scatter each valid event of the block's sub-chunk to its bin (offsets
// within the window); a block reserves one range per bin, so the global
// atomics are per (block, bin).  Also stores the reciprocal of the event's
// larger offset from the FOE (used by the bound's cell walk).
__global__ void __launch_bounds__(INGEST_THREADS) k_row_scatter(Geom g, const WinIn* __restrict__ wins,
                                                                const int32_t* __restrict__ chunk_win,
                                                                int32_t* cursor, Ev* __restrict__ out) {
    __shared__ int32_t h[MAX_BINS];
    __shared__ int32_t base[MAX_BINS];
    const int chunk = blockIdx.x / INGEST_SUB;
    const int w = chunk_win[chunk];
    const WinIn win = wins[w];
    const int bins = bins_of(g);
    const float bscale = __fdiv_rn((float)g.n_tb, win.tau);
    int64_t i0, i1;
    sub_chunk(win, chunk, blockIdx.x % INGEST_SUB, i0, i1);
    int32_t* cur = cursor + (size_t)w * bins;
    Ev* o = out + win.ev_off;
    for (int r = threadIdx.x; r < bins; r += blockDim.x) h[r] = 0;
    __syncthreads();
    for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        const int xi = win.x[i], yi = win.y[i];
        const float ti = win.t[i];
        const float tr = __fsub_rn(ti, win.t0);
        if (event_ok(xi, yi, ti, tr, win.tau, g.W, g.H))
            atomicAdd(&h[event_key(g, yi, tr, bscale, plane_of(g, win, i))], 1);
    }
    __syncthreads();
    for (int r = threadIdx.x; r < bins; r += blockDim.x) {
        base[r] = h[r] ? atomicAdd(&cur[r], h[r]) : 0;
        h[r] = 0;
    }
    __syncthreads();
    for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        const int xi = win.x[i], yi = win.y[i];
        const float ti = win.t[i];
        const float tr = __fsub_rn(ti, win.t0);
        if (!event_ok(xi, yi, ti, tr, win.tau, g.W, g.H)) continue;
        const int key = event_key(g, yi, tr, bscale, plane_of(g, win, i));
        const int pos = base[key] + atomicAdd(&h[key], 1);
        if (!DD_IN(pos, win.n, 8u)) continue;
        Ev e;
        e.dx = __fsub_rn((float)xi, g.fx);
        e.dy = __fsub_rn((float)yi, g.fy);
        e.t = tr;
        e.rm = __frcp_rn(fabsf(e.dx) >= fabsf(e.dy) ? e.dx : e.dy);
        o[pos] = e;
    }
}

// The whole ingest of one window of at most CHUNK events by one block: each
// thread keeps its events in registers from the count (which gives an event
// its place in its bin) over the scan to the store.  A small window's ingest
// is three dependent launches otherwise (a search of 4,000 events 310 -> 293
// us, of 3,000 325 -> 315 us).
constexpr int SMALL_THREADS = 1024;
__global__ void __launch_bounds__(SMALL_THREADS) k_ingest_small(Geom g, const WinIn* __restrict__ wins,
                                                                int32_t* row_off, Ev* __restrict__ out, int32_t* err) {
    constexpr int PER = CHUNK / SMALL_THREADS;
    __shared__ int32_t h[MAX_BINS];
    __shared__ int32_t wsum[SMALL_THREADS / 32];
    const WinIn win = wins[0];
    const int bins = bins_of(g), tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const float bscale = __fdiv_rn((float)g.n_tb, win.tau);
    for (int r = tid; r < bins; r += SMALL_THREADS) h[r] = 0;
    int xi[PER], yi[PER], key[PER], rank[PER];
    float tr[PER];
    bool bad = false;
#pragma unroll
    for (int k = 0; k < PER; k++) {
        const int64_t i = tid + (int64_t)k * SMALL_THREADS;
        key[k] = -1;
        if (i < win.n) {
            xi[k] = win.x[i];
            yi[k] = win.y[i];
            const float ti = win.t[i];
            tr[k] = __fsub_rn(ti, win.t0);
            if (event_ok(xi[k], yi[k], ti, tr[k], win.tau, g.W, g.H))
                key[k] = event_key(g, yi[k], tr[k], bscale, plane_of(g, win, i));
            else
                bad = true;
        }
    }
    if (bad) atomicOr(err, 1);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; k++)
        if (key[k] >= 0) rank[k] = atomicAdd(&h[key[k]], 1);
    __syncthreads();
    // exclusive scan of the bins, four consecutive ones per thread
    constexpr int BINS_PER = MAX_BINS / SMALL_THREADS;
    int local[BINS_PER], tot = 0;
#pragma unroll
    for (int k = 0; k < BINS_PER; k++) {
        const int r = BINS_PER * tid + k;
        local[k] = r < bins ? h[r] : 0;
        tot += local[k];
    }
    const int incl = warp_incl_scan(tot);
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    if (wid == 0) wsum[lane] = warp_incl_scan(wsum[lane]);
    __syncthreads();
    int excl = incl - tot + (wid ? wsum[wid - 1] : 0);
#pragma unroll
    for (int k = 0; k < BINS_PER; k++) {
        const int r = BINS_PER * tid + k;
        if (r < bins) {
            h[r] = excl;
            row_off[r] = excl;
        }
        excl += local[k];
    }
    if (tid == SMALL_THREADS - 1) row_off[bins] = excl;
    __syncthreads();
    Ev* o = out + win.ev_off;
#pragma unroll
    for (int k = 0; k < PER; k++) {
        if (key[k] < 0) continue;
        const int pos = h[key[k]] + rank[k];
        if (!DD_IN(pos, win.n, 8u)) continue;
        Ev e;
        e.dx = __fsub_rn((float)xi[k], g.fx);
        e.dy = __fsub_rn((float)yi[k], g.fy);
        e.t = tr[k];
        e.rm = __frcp_rn(fabsf(e.dx) >= fabsf(e.dy) ? e.dx : e.dy);
        o[pos] = e;
    }
}

cudaError_t launch_ingest(const Geom& g, const WinIn* wins_dev, int32_t n_windows, const int32_t* chunk_win_dev,
                          int32_t n_chunks, Ev* out, int32_t* row_count, int32_t* row_off,
                          int32_t* cursor, int32_t* err, cudaStream_t s, bool clear, int* launches) {
    const int bins = bins_of(g);
    if (n_windows <= 0) return cudaSuccess;
    if (clear) {
        cudaError_t e = cudaMemsetAsync(row_count, 0, sizeof(int32_t) * bins * (size_t)n_windows, s);
        if (e != cudaSuccess) return e;
        e = cudaMemsetAsync(err, 0, sizeof(int32_t) * (size_t)n_windows, s);
        if (e != cudaSuccess) return e;
    }
    if (n_windows == 1 && n_chunks == 1) {
        k_ingest_small<<<1, SMALL_THREADS, 0, s>>>(g, wins_dev, row_off, out, err);
        if (launches) *launches = 1;
        return cudaGetLastError();
    }
    if (launches) *launches = n_chunks > 0 ? 3 : 1;
    const unsigned blocks = (unsigned)n_chunks * INGEST_SUB;
    if (n_chunks > 0) k_row_hist<<<blocks, INGEST_THREADS, 0, s>>>(g, wins_dev, chunk_win_dev, row_count, err);
    k_row_scan<<<n_windows, 1024, 0, s>>>(bins, row_count, row_off, cursor);
    if (n_chunks > 0) k_row_scatter<<<blocks, INGEST_THREADS, 0, s>>>(g, wins_dev, chunk_win_dev, cursor, out);
    return cudaGetLastError();
}

// ------------------------------------------------------------------- eval

// Events of time bucket b that can reach tile rows [y0, y1) for D in
// [Dl, Dh]: the scale s(D, t) = (1 - D t)/(1 - D tau) is monotone in D and in
// t, so over the bucket's time range its extremes are at the four corners.
// An event at row y can reach the rows only if (y - FOE_y) s meets them for
// some s in that range; the rows that can are a contiguous range of the
// bucket's row-sorted events.  Binary32, each operation correctly rounded
// (relative error 2^-24; quotients as products with rounded reciprocals):
// every scale has relative error below 12 x 2^-24 on the domain
// -64 <= D tau <= 3/4, the bucket's time edges below 3 x 2^-24, and the row
// bounds (at most 4096 px) below 3 x 2^-24, all far under the margins: 1e-4
// relative on s, 1e-3 of a bucket in t (an event of bucket b has t bscale in
// [b (1 - 2^-24), (b + 1)(1 + 2^-24)), b < 8), 1/16 pixel on the band's
// edges.  A superset.
__device__ void bucket_event_range(const Geom& g, const int32_t* row_off, float Dl, float Dh, float tau,
                                   float bscale, int b, int y0, int y1, int& e0, int& e1) {
    const float rb = __frcp_rn(bscale);
    const float tl = fmaxf(0.0f, __fmul_rn((float)b - 1e-3f, rb));
    const float th = fminf(tau, __fmul_rn((float)b + 1.001f, rb));
    const float tref = warp_tref(g, tau);
    const float gl = __frcp_rn(1.0f - Dl * tref), gh = __frcp_rn(1.0f - Dh * tref);
    float smin = 3.0e38f, smax = -3.0e38f;
    for (int i = 0; i < 4; i++) {
        const float D = (i & 1) ? Dh : Dl, t = (i & 2) ? th : tl;
        const float s = (1.0f - D * t) * ((i & 1) ? gh : gl);
        smin = fminf(smin, s);
        smax = fmaxf(smax, s);
    }
    smin *= 1.0f - 1e-4f;
    smax *= 1.0f + 1e-4f;
    const float A = (float)y0 - 0.5625f - g.fy;
    const float B = (float)(y1 - 1) + 0.5625f - g.fy;
    const float dylo = A * __frcp_rn(A >= 0.0f ? smax : smin);
    const float dyhi = B * __frcp_rn(B >= 0.0f ? smin : smax);
    // The margins above exceed the few-ulp error of this arithmetic, and
    // rounding a bound that is off by less than a row outward to an integer
    // row never drops a row the exact bound admits.
    const float rl = floorf(g.fy + dylo), rh = ceilf(g.fy + dyhi);
    if (rh < 0.0f || rl > (float)(g.H - 1)) {
        e0 = e1 = 0;
        return;
    }
    const int rlo = rl < 0.0f ? 0 : (int)rl;
    const int rhi = rh > (float)(g.H - 1) ? g.H - 1 : (int)rh;
    e0 = row_off[b * g.H + rlo];
    e1 = row_off[b * g.H + rhi + 1];
}

// A unit's candidate events: one run of consecutive events per time bucket,
// taken in chunks of 32 (a run's last chunk may be partial), so that a warp
// works on one run at a time and finds it with a uniform test.  Run b holds
// chunks [next of run b - 1, next of run b); chunk c's events are
// 32 c + first + lane, below end.
constexpr int MAX_TB = 8;         // time buckets of the event sort

struct __align__(16) Run {
    int first, end, next, pad;
};
constexpr Run NO_RUN = {0, INT32_MIN, INT32_MAX, 0};   // after the last run: chunks without events

// One unit -- a job's row band -- as the block's last warp prepares it in
// shared memory for the others: everything that is the same for all threads is worked out once.
enum UnitKind : int { UNIT_NONE = 0, UNIT_POINT, UNIT_BOUND, UNIT_DENSE, UNIT_FUSED };

struct __align__(16) Unit {
    Run run[MAX_TB + 1];     // candidate events (an event split: its share of them), then NO_RUN
    int chunks;              // of all runs
    int kind;
    int y0, rows;            // tile rows [y0, y0 + rows) of the frame
    float D_lo, D_hi, D_c, tau;  // D_c: a fused job's centre
    int win, task, left;     // left: a fused job's left half
    int tile;                // the job's band over both planes, and its plane
    int plane;
    int split, splits;       // event splits (1: none; a split by rows is a unit of its own rows)
    const Ev* ev;            // the window's sorted events
#ifdef DD_CHECKED
    int64_t n_ev;            // the window's event count
#endif
};

// Chunk-to-event cursor of one warp; visited chunks increase.
struct Cursor {
    const Run* at;
    Run r;
    __device__ __forceinline__ explicit Cursor(const Unit& u) : at(u.run), r(u.run[0]) {}
    __device__ __forceinline__ int event(int chunk, int lane) {   // the lane's event; none if >= r.end
        while (chunk >= r.next) r = *++at;
        return 32 * chunk + r.first + lane;
    }
};

// Prepares unit `id` (job id / (n_tiles slices), band, slice of it) in `un`:
// one warp, one time bucket per lane.  The jobs' rows or events are divided
// here, so no other thread divides.
__device__ __forceinline__ void prepare_unit(const Geom& g, const EvalArgs& a, const Job* jobs, int id, int n_units,
                                             int slices, Unit& un) {
    const int lane = threadIdx.x & 31;
    if (id >= n_units) {
        if (lane == 0) un.kind = UNIT_NONE;
        return;
    }
    const int bands = slices > 1 ? id / slices : id, slice = id - bands * slices;
    const int j = bands / g.n_tiles, ti = bands - j * g.n_tiles;
    const Job jb = jobs[j];
    const WinIn* win = a.wins + jb.win;
    const int64_t ev_off = win->ev_off;
    const float tau = win->tau, Dl = jb.D_lo, Dh = jb.D_hi;
    const bool fused = jb.splits < 0;             // one expanded interval: its three tasks together
    const float cells = bound_cells(g, Dl, Dh, tau);
    const int kind = fused ? UNIT_FUSED : (jb.kind == TASK_POINT ? UNIT_POINT
                                                                 : (cells >= DENSE_CELLS ? UNIT_DENSE : UNIT_BOUND));
    const int plane = ti >= g.plane_tiles ? 1 : 0, band = ti - plane * g.plane_tiles;
    int splits = fused ? 1 : max(1, jb.splits);
    int y0 = band * g.band_rows, rows = min(g.band_rows, g.H - y0);
    if (splits > 1 && (!a.mg.acc || cells < SPLIT_ROWS_CELLS || win->n < SPLIT_ROWS_EVENTS)) {    // split by rows: its own rows
        const int r0 = (int)((uint32_t)(rows * jb.split) / (uint32_t)splits);
        rows = (int)((uint32_t)(rows * (jb.split + 1)) / (uint32_t)splits) - r0;
        y0 += r0;
        splits = 1;
    }
    if (slices > 1) {                             // an event split stays whole: its first slice has every row
        const int r0 = splits > 1 ? (slice ? rows : 0) : rows * slice / slices;
        rows = (splits > 1 ? rows : rows * (slice + 1) / slices) - r0;
        y0 += r0;
        if (splits > 1 && slice) splits = 1;      // without rows: nothing to count or to merge
    }
    const int32_t* row_off = a.row_off + (size_t)jb.win * (bins_of(g) + 1) + (size_t)plane * g.n_tb * g.H;
    int e0 = 0, e1 = 0;
    if (lane < g.n_tb && rows > 0)
        bucket_event_range(g, row_off, Dl, Dh, tau, __fdiv_rn((float)g.n_tb, tau), lane, y0, y0 + rows, e0, e1);
    int n = (e1 - e0 + 31) >> 5, incl = warp_incl_scan(n);
    if (splits > 1) {                             // this split's share of the chunks of all runs
        const uint32_t all = (uint32_t)__shfl_sync(0xffffffffu, incl, 31);
        const int c0 = (int)(all * (uint32_t)jb.split / (uint32_t)splits);
        const int c1 = (int)(all * (uint32_t)(jb.split + 1) / (uint32_t)splits);
        const int a0 = incl - n, b0 = max(a0, c0), b1 = min(incl, c1);
        e1 = min(e1, e0 + 32 * (b1 - a0));
        e0 += 32 * (b0 - a0);
        n = max(b1 - b0, 0);
        incl = warp_incl_scan(n);
    }
    if (lane <= g.n_tb) {
        Run r = NO_RUN;
        if (lane < g.n_tb) {
            r.first = e0 - 32 * (incl - n);
            r.end = e1;
            r.next = incl;
        }
        un.run[lane] = r;
    }
    const int chunks = __shfl_sync(0xffffffffu, incl, 31);
    if (lane == 0) {
        un.chunks = chunks;
        un.kind = kind;
        un.y0 = y0;
        un.rows = rows;
        un.D_lo = Dl;
        un.D_hi = Dh;
        un.D_c = jb.D_c;
        un.tau = tau;
        un.win = jb.win;
        un.task = jb.task;
        un.left = jb.split;
        un.tile = ti;
        un.plane = plane;
        un.split = jb.split;
        un.splits = splits;
        un.ev = a.ev + ev_off;
#ifdef DD_CHECKED
        un.n_ev = win->n;
#endif
    }
}

// ----------------------------------------------------- passes over the events

constexpr int MAX_WARPS = 16;     // working warps of a k_eval block (at most 512 threads)
// A block of k_eval: working warps and one more that prepares their units.
__device__ __forceinline__ int work_threads() { return (int)blockDim.x - 32; }
__device__ __forceinline__ int work_warps() { return ((int)blockDim.x >> 5) - 1; }
__device__ __forceinline__ void work_sync() {     // a barrier of the working warps
    __barrier_sync_count(1, work_threads());
}

// Shared scratch of one working warp (WARP_WORDS words of dynamic shared
// memory after the tile): the ring of a sparse bound's queued events, the
// segment descriptors of a dense bound's walks, or the warp's list of a fused
// unit's unstable events.
constexpr int WARP_WORDS = EVAL_WARP_WORDS;
constexpr int RUN = 7;            // major cells of a segment that one lane walks at a time (odd)
constexpr int RING = 64;          // queued events per warp (a power of two, >= 63)

// Dynamic shared memory of a k_eval block: the band tile (rounded up to 16
// bytes) and its warps' scratch.
__host__ __device__ inline int eval_tile_words(const Geom& g) { return (g.band_rows * tile_pitch(g) + 3) & ~3; }
__host__ __device__ inline size_t eval_smem_bytes(const Geom& g, int threads) {
    return sizeof(uint32_t) * ((size_t)eval_tile_words(g) + (size_t)WARP_WORDS * (threads / 32));
}

// The block's tile and what every pass needs of the unit: rows [row0, row0 +
// rows) of the frame (biased), pitch P.
struct Tile {
    uint32_t* cell;
    uint32_t base;           // shared-memory address of biased pixel (0, 0) if the tile reached it
    uint32_t pitch;          // bytes
    uint32_t idle;           // shared-memory address of the lane's own word outside the tile
    uint32_t row0, rows, W;
    __device__ __forceinline__ uint32_t first() const {           // address of the tile's first cell
        return base + row0 * pitch + 4u * CELL0;
    }
};

// Increments of a tile cell.  Sparse images: the sum of squares grows by
// 2v + 1 from the cell's previous count v, so S = 2 sum(v) + (increments).
// Dense images (many increments per cell) add without an answer; their sums
// are taken from the tile afterwards.  A fused unit keeps the images of its
// three tasks in three 10-bit fields of one cell.
enum Field : int { FIELD_P = 0, FIELD_L = 10, FIELD_R = 20, FIELD_ALL = 30, WHOLE = 32, DENSE = 33 };
constexpr uint32_t FIELD_MAX = 1023;

template <int F>
__device__ __forceinline__ uint32_t field_inc() {
    return F >= WHOLE ? 1u : (F == FIELD_ALL ? 0x00100401u : 1u << (F & 31));
}
// The previous count in an atomic's answer (0 if it was not issued): into V,
// and into top, their maximum (a field that held FIELD_MAX has run over into
// the next one).
template <int F, class Sum>
__device__ __forceinline__ void take(uint32_t old, Sum& V, uint32_t& top) {
    if (F == WHOLE) {
        V += old;
    } else if (F != DENSE) {
        const uint32_t v = (old >> (F == FIELD_ALL ? 0 : F & 31)) & FIELD_MAX;
        V += v;
        top = max(top, v);
    }
}

// One atomic increment at shared-memory address `at`; a lane that has none
// (`here` false) adds to a word of its own instead.  A predicated atomic is
// compiled to a branch around it (measured: about five control instructions
// per atomic, a third of a wide bound's instructions); an address that is
// always valid takes none.
template <int F, class Sum>
__device__ __forceinline__ void bump(const Tile& T, uint32_t at, bool here, Sum& V, uint32_t& top) {
    const uint32_t to = here ? at : T.idle;
    if (F == DENSE) {
        asm volatile("red.shared.add.u32 [%0], 1;" : : "r"(to) : "memory");
    } else {
        uint32_t old;
        asm volatile("atom.shared.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(to), "r"(field_inc<F>()) : "memory");
        take<F>(here ? old : 0u, V, top);
    }
}

// Adds one to the field of biased pixel c if it is in the tile (and `also`
// holds); n counts the increments.
template <int F, class Sum>
__device__ __forceinline__ void bump_pixel(const Tile& T, uint2 c, Sum& V, uint32_t& n, uint32_t& top,
                                           bool also = true) {
    const uint32_t r = c.y - T.row0, x = c.x - CELL0, at = T.base + c.y * T.pitch + 4u * c.x;
    bool here = (r < T.rows) & (x < T.W) & also;
#ifdef DD_CHECKED
    here = here && DD_IN((int)(at - T.first()), T.rows * T.pitch, 1u);
#endif
    bump<F>(T, at, here, V, top);
    n += here;
}

// An event's widened scale range over an interval and its end pixels (biased).
struct Span {
    float sa, sb;
    uint2 a, b;
};
__device__ __forceinline__ Span span_of(f32x2 foe, f32x2 d, float s1, float s2, f32x2 widen) {
    const f32x2 w = mul2(pair(fminf(s1, s2), fmaxf(s1, s2)), widen);
    Span s;
    s.sa = lo_of(w);
    s.sb = hi_of(w);
    s.a = pixel_of(foe, d, s.sa);
    s.b = pixel_of(foe, d, s.sb);
    return s;
}
// Both scales of an event at time t: (1 - D t) g for the pair of D.
__device__ __forceinline__ f32x2 scales2(f32x2 minus_D, f32x2 gg, float t) {
    return mul2(add2(pair(1.0f, 1.0f), mul2(minus_D, pair(t, t))), gg);
}
// Every covered cell lies between the end pixels (each coordinate is monotone
// in s): does that box meet the tile?
__device__ __forceinline__ bool meets(const Tile& T, const Span& s) {
    return max(s.a.y, s.b.y) >= T.row0 && min(s.a.y, s.b.y) < T.row0 + T.rows && max(s.a.x, s.b.x) >= CELL0 &&
           min(s.a.x, s.b.x) < CELL0 + T.W;
}
// Eq. (19): both end pixels in the frame; counted by the tile of row a.y.
__device__ __forceinline__ bool counts_full(const Geom& g, const Tile& T, const Span& s) {
    return s.a.x - CELL0 < T.W && s.b.x - CELL0 < T.W && s.b.y - CELL0 < (uint32_t)g.H && s.a.y - T.row0 < T.rows;
}
// End pixels side by side: one coordinate is constant and the other takes two
// adjacent values, so the segment covers exactly those two pixels.
__device__ __forceinline__ bool adjacent(const Span& s) {
    return abs((int)(s.a.x - s.b.x)) + abs((int)(s.a.y - s.b.y)) == 1;
}

// Eq. (16), the cells of one longer segment.  It is walked along its major
// axis (the larger offset from the FOE, ties to x): major cell k takes the
// s-range in which the major coordinate rounds to k, widened by 2^-8 px and
// clipped to [s_a, s_b], and covers the minor cells between the ends of that
// range.  walk_range gives the major cells whose runs can reach the tile (a
// superset: the runs are cut to the tile's rows and the frame's columns);
// their number can be negative.  Major y: the rows in the tile.  Major x: the
// columns at the scales at which the minor coordinate is within the tile's
// rows (half a pixel and the margin beyond, which exceeds the error of the
// approximate reciprocal, 2^-22 of at most 4096 px), 2^-6 px farther than the
// event's own positions there (a column's s-range reaches 2^-8 px beyond it,
// rounding far less).  A minor offset of 0 makes those scales infinite or not
// a number, which the minimum and maximum ignore: any scale will do.  One
// straight line of code: a warp has events of both axes.
__device__ __forceinline__ int walk_range(const Geom& g, const Tile& T, float4 v, const Span& s, bool major_x,
                                          uint32_t& k) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v.y));
    const float y0 = __uint_as_float(T.row0) - CELL0_F, y1 = __uint_as_float(T.row0 + T.rows - 1) - CELL0_F;
    const float b0 = __fmul_rn(__fsub_rn(__fsub_rn(y0, g.fy), HALF_PLUS), r);
    const float b1 = __fmul_rn(__fadd_rn(__fsub_rn(y1, g.fy), HALF_PLUS), r);
    const float lo = fmaxf(fminf(b0, b1), s.sa), hi = fminf(fmaxf(b0, b1), s.sb);
    const float x0 = __fadd_rn(g.fx, __fmul_rn(v.x, lo)), x1 = __fadd_rn(g.fx, __fmul_rn(v.x, hi));
    const uint32_t c0 = __float_as_uint(__fadd_rd(__fadd_rn(fminf(x0, x1), 0.5f - 0x1p-6f), CELL0_F));
    const uint32_t c1 = __float_as_uint(__fadd_rd(__fadd_rn(fmaxf(x0, x1), 0.5f + 0x1p-6f), CELL0_F));
    const uint32_t ea = major_x ? s.a.x : s.a.y, eb = major_x ? s.b.x : s.b.y;
    const uint32_t a = max(min(ea, eb), major_x ? max(c0, CELL0) : T.row0);
    const uint32_t b = min(max(ea, eb), major_x ? min(c1, CELL0 + T.W - 1) : T.row0 + T.rows - 1);
    k = a;
    return major_x && lo > hi ? 0 : (int)(b - a) + 1;
}

// `n` consecutive major cells of a segment from k (biased) on, by one lane:
// each covers the run of minor cells between the ends of its s-range, cut to
// the tile's rows and the frame's columns.  dn, rm: the minor offset and the
// major one's reciprocal.  A run has at most three cells: its s-range spans
// 1.008 major cells and the slope is at most 1.
template <int F, class Sum>
__device__ __forceinline__ void walk_cells(const Geom& g, const Tile& T, bool mx, uint32_t k, int n, float dn, float rm,
                                           float sa, float sb, Sum& V, uint32_t& C, uint32_t& top) {
    const float fm = mx ? g.fx : g.fy, fn = mx ? g.fy : g.fx;
    const float h = copysignf(HALF_PLUS, rm);     // so that lo is the smaller end
    const uint32_t jmin = mx ? T.row0 : CELL0, jmax = mx ? T.row0 + T.rows - 1 : CELL0 + T.W - 1;
    const uint32_t sk = mx ? 4u : T.pitch, sj = mx ? T.pitch : 4u;
    uint32_t at_k = T.base + k * sk;
    float kf = __fsub_rn(__uint_as_float(k), CELL0_F);
#pragma unroll 2
    for (; n > 0; n--) {
        const float e = __fsub_rn(kf, fm);
        const float lo = fmaxf(__fmul_rn(__fsub_rn(e, h), rm), sa), hi = fminf(__fmul_rn(__fadd_rn(e, h), rm), sb);
        const uint32_t c0 = cell1(fn, dn, lo), c1 = cell1(fn, dn, hi);
        const uint32_t j0 = max(min(c0, c1), jmin), jn = min(max(c0, c1), jmax);
        const uint32_t at = at_k + j0 * sj;
        bool some = lo <= hi;                     // an empty s-range covers nothing
#ifdef DD_CHECKED
        if (some && j0 <= jn)
            some = DD_IN(jn - j0, 3, 2u) && DD_IN((int)(at - T.first()), T.rows * T.pitch, 2u) &&
                   DD_IN((int)(at + (jn - j0) * sj - T.first()), T.rows * T.pitch, 2u);
#endif
        bump<F>(T, at, some & (j0 <= jn), V, top);
        bump<F>(T, at + sj, some & (j0 < jn), V, top);
        if (some & (j0 + 1 < jn)) bump<F>(T, at + 2 * sj, true, V, top);     // rare: slopes near 1
        if (F != DENSE) C += some & (j0 <= jn) ? jn - j0 + 1 : 0u;
        kf = __fadd_rn(kf, 1.0f);
        at_k += sk;
    }
}

// A short segment walked by its own lane.
template <int F, class Sum>
__device__ __forceinline__ void walk_lane(const Geom& g, const Tile& T, float4 v, const Span& s, Sum& V,
                                          uint32_t& C, uint32_t& top) {
    const bool mx = fabsf(v.x) >= fabsf(v.y);
    uint32_t k;
    const int n = walk_range(g, T, v, s, mx, k);
    walk_cells<F>(g, T, mx, k, n, mx ? v.y : v.x, v.w, s.sa, s.sb, V, C, top);
}

// The segments of a warp's events (`here`: the lane has one that meets the
// tile).  If none has more than RUN major cells in the tile, each lane walks
// its own; otherwise they are cut into runs of RUN cells that are spread over
// the lanes: the segments put their descriptors in shared memory in lane
// order, and 32 runs at a time find their owners from the bit mask of the
// segments whose runs start among them.  RUN is odd, so that the runs of one
// segment lie in different shared-memory banks.
template <int F>
__device__ __forceinline__ void walk_warp(const Geom& g, const Tile& T, float4 v, const Span& s, bool here,
                                          uint32_t* scratch, unsigned long long& V, uint32_t& C, uint32_t& top) {
    const int lane = threadIdx.x & 31;
    const bool mx = fabsf(v.x) >= fabsf(v.y);
    uint32_t k;
    const int cells = walk_range(g, T, v, s, mx, k), n = here ? max(cells, 0) : 0;
    const int longest = __reduce_max_sync(0xffffffffu, n);
    if (longest == 0) return;
    const float dn = mx ? v.y : v.x;
    if (longest <= RUN) {
        walk_cells<F>(g, T, mx, k, n, dn, v.w, s.sa, s.sb, V, C, top);
        return;
    }
    float4* desc = reinterpret_cast<float4*>(scratch);            // [32] rm, dn, s_a, s_b
    uint2* key = reinterpret_cast<uint2*>(scratch + 128);         // [32] first cell (top bit: major y), cells << 16 | first run
    const int runs = (n + RUN - 1) / RUN, incl = warp_incl_scan(runs), excl = incl - runs;
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    const unsigned act = __ballot_sync(0xffffffffu, n > 0);
    if (n > 0) {
        const int r = __popc(act & ((1u << lane) - 1u));
        desc[r] = make_float4(v.w, dn, s.sa, s.sb);
        key[r] = make_uint2(k | (mx ? 0u : 0x80000000u), (uint32_t)n << 16 | (uint32_t)excl);
    }
    __syncwarp();
    const unsigned upto = 0xffffffffu >> (31 - lane);             // lanes 0..lane
    int seen = -1;
    for (int c0 = 0; c0 < total; c0 += 32) {
        const uint32_t rel = (uint32_t)(excl - c0);
        const unsigned starts = __reduce_or_sync(0xffffffffu, n > 0 && rel < 32u ? 1u << rel : 0u);
        const int r = seen + __popc(starts & upto);
        seen += __popc(starts);
        if (c0 + lane < total) {
            const float4 q = desc[r];
            const uint2 w = key[r];
            const int i = RUN * (c0 + lane - (int)(w.y & 0xffffu));
            walk_cells<F>(g, T, (int)w.x >= 0, (w.x & 0x7fffffffu) + (uint32_t)i, min(RUN, (int)(w.y >> 16) - i), q.y, q.x,
                          q.z, q.w, V, C, top);
        }
    }
    __syncwarp();                                 // read before the scratch is written again
}

// The walks of a dense bound: segments are cut into runs of at most DENSE_RUN
// major cells, queued in the warp's ring (a segment's lane puts them there one
// at a time, with all that a walk needs), and every 32 queued runs are walked
// together, one per lane, across chunks of events: no lane waits for a longer
// segment and only the last run of a segment is short.  A ring entry is five
// words: 1/major offset, minor offset, s_a, s_b, and the first cell (12 bits),
// the axis and the cells.  Runs of 3, 4, 5 and 7 cells: 337, 339, 304, 292 us
// for 60 bounds of width 1/2, 143, 152, 139, 141 us of width 1/8 (320 and 153
// us with each chunk of events walked by itself).
constexpr int DENSE_RUN = 7;
struct RunRing {
    uint32_t* mem;                                // [64] float4, then [64] words
    int head, count;
    __device__ __forceinline__ void walk(const Geom& g, const Tile& T, bool valid) {
        const int lane = threadIdx.x & 31, i = (head + lane) & (RING - 1);
        __syncwarp();                             // the queued runs are visible to the warp
        const float4 q = reinterpret_cast<const float4*>(mem)[i];
        const uint32_t w = mem[4 * RING + i];
        __syncwarp();                             // read before their places are written again
        unsigned long long V = 0;
        uint32_t C = 0, top = 0;
        walk_cells<DENSE>(g, T, !(w & 0x1000u), CELL0 + (w & 0xfffu), valid ? (int)(w >> 13) : 0, q.y, q.x, q.z, q.w, V,
                          C, top);
    }
    // Each lane's segment: n major cells from k (biased); n <= 0: none.
    __device__ __forceinline__ void add(const Geom& g, const Tile& T, float4 v, const Span& s, bool mx, uint32_t k,
                                        int n) {
        const unsigned below = (1u << (threadIdx.x & 31)) - 1u;
        for (unsigned m; (m = __ballot_sync(0xffffffffu, n > 0)) != 0;) {
            if (n > 0) {
                const int i = (head + count + __popc(m & below)) & (RING - 1);
                reinterpret_cast<float4*>(mem)[i] = make_float4(v.w, mx ? v.y : v.x, s.sa, s.sb);
                mem[4 * RING + i] = (k - CELL0) | (mx ? 0u : 0x1000u) | (uint32_t)min(n, DENSE_RUN) << 13;
                k += DENSE_RUN;
                n -= DENSE_RUN;
            }
            count += __popc(m);
            if (count >= 32) {
                walk(g, T, true);
                head += 32;
                count -= 32;
            }
        }
    }
    __device__ __forceinline__ void flush(const Geom& g, const Tile& T) {
        if (count > 0) walk(g, T, (int)(threadIdx.x & 31) < count);
        count = 0;
    }
};

__device__ __forceinline__ float4 load_event(const float4* ev, int e) {
    return __ldg(ev + e);                         // dx, dy, t, 1/major offset
}
// The lane's event of a chunk; a lane without one gets offsets that are not
// numbers, whose biased pixel lies in no tile and at every scale is the same.
__device__ __forceinline__ float4 chunk_event(const Unit& un, const float4* ev, Cursor& cur, int chunk, int lane,
                                              int& e) {
    e = cur.event(chunk, lane);
    float4 v = make_float4(CUDART_NAN_F, CUDART_NAN_F, 0.0f, 0.0f);
    if (e < cur.r.end && DD_IN(e, un.n_ev, 4u)) v = load_event(ev, e);
    return v;
}

// Eqs. (11)-(12) at D: each event of the unit's chunks into the tile.  V and
// C collect the previous counts and the increments.  Four chunks are loaded
// before any is used, so that a warp waits for one L2 round trip per 128
// events.
__device__ __forceinline__ void point_pass(const Geom& g, const Unit& un, const Tile& T, float D,
                                           unsigned long long& V, unsigned long long& C) {
    constexpr int U = 4;
    const int lane = threadIdx.x & 31, nw = work_warps(), chunks = un.chunks;
    const float4* ev = reinterpret_cast<const float4*>(un.ev);
    const float gg = warp_g(D, warp_tref(g, un.tau));
    const f32x2 foe = pair(g.fx, g.fy);
    uint32_t n = 0, top = 0;                      // increments: at most one per event
    Cursor cur(un);
    for (int ch = (int)(threadIdx.x >> 5); ch < chunks; ch += U * nw) {
        float4 v[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            int e;
            v[u] = chunk_event(un, ev, cur, ch + u * nw, lane, e);
        }
#pragma unroll
        for (int u = 0; u < U; u++)
            bump_pixel<WHOLE>(T, pixel_of(foe, pair(v[u].x, v[u].y), warp_s(D, v[u].z, gg)), V, n, top);
    }
    C += n;
}

// Eqs. (16) and (19) over [Dl, Dh] for the unit's chunks: Hbar into the tile,
// N_full into F, and (sparse) the previous counts and increments into V and C.
// An event whose end pixels coincide covers that pixel only.  Sparse bounds
// (few such segments are longer) queue the others, so that full warps handle
// them; dense bounds cut them into runs (RunRing).
template <bool IS_DENSE>
__device__ __forceinline__ void bound_pass(const Geom& g, const Unit& un, const Tile& T, float Dl, float Dh,
                                           uint32_t* scratch, unsigned long long& V, unsigned long long& C,
                                           unsigned long long& F) {
    constexpr int U = IS_DENSE ? 1 : 2;
    const int lane = threadIdx.x & 31, nw = work_warps(), chunks = un.chunks;
    const float4* ev = reinterpret_cast<const float4*>(un.ev);
    const float tref = warp_tref(g, un.tau);
    const f32x2 foe = pair(g.fx, g.fy), minus_D = pair(-Dl, -Dh), gg = pair(warp_g(Dl, tref), warp_g(Dh, tref));
    const f32x2 widen = pair(WIDEN_DN, WIDEN_UP);
    uint32_t one = 0, full = 0, top = 0;
    int head = 0, tail = 0;
    RunRing runs = {scratch, 0, 0};
    auto span = [&](float4 v) {
        const f32x2 s2 = scales2(minus_D, gg, v.z);
        return span_of(foe, pair(v.x, v.y), lo_of(s2), hi_of(s2), widen);
    };
    auto queued = [&](bool valid) {               // up to 32 queued events, one per lane
        __syncwarp();                             // the queued events are visible to the warp
        float4 v = make_float4(CUDART_NAN_F, CUDART_NAN_F, 0.0f, 0.0f);
        if (valid) v = load_event(ev, (int)scratch[(head + lane) & (RING - 1)]);
        __syncwarp();                             // read before the next chunk overwrites them
        const Span s = span(v);
        full += (uint32_t)(valid & counts_full(g, T, s));
        const bool two = adjacent(s);
        uint32_t more = 0;
        bump_pixel<WHOLE>(T, s.a, V, more, top, two);
        bump_pixel<WHOLE>(T, s.b, V, more, top, two);
        walk_warp<WHOLE>(g, T, v, s, valid & !two & meets(T, s), scratch + RING, V, more, top);
        C += more;
    };
    Cursor cur(un);
    for (int ch = (int)(threadIdx.x >> 5); ch < chunks; ch += U * nw) {
        float4 v[U];
        int e[U];
#pragma unroll
        for (int u = 0; u < U; u++) v[u] = chunk_event(un, ev, cur, ch + u * nw, lane, e[u]);
#pragma unroll
        for (int u = 0; u < U; u++) {
            const Span s = span(v[u]);
            const bool single = s.a.x == s.b.x && s.a.y == s.b.y;
            bump_pixel<IS_DENSE ? DENSE : WHOLE>(T, s.a, V, one, top, single);
            const unsigned m = __ballot_sync(0xffffffffu, !single);
            if (!m) continue;
            if (IS_DENSE) {
                full += (uint32_t)(!single & counts_full(g, T, s));
                // Adjacent end pixels need no walk, from two such events in the
                // chunk on (60 bounds of width 1/32: 92 -> 84 us; of width 1/2,
                // where they are rare, 300 -> 297 us).
                bool walk = !single;
                const bool two = adjacent(s);
                if (__popc(__ballot_sync(0xffffffffu, two)) >= 2) {
                    uint32_t more = 0;            // not used: counted from the tile
                    bump_pixel<DENSE>(T, s.a, V, more, top, two);
                    bump_pixel<DENSE>(T, s.b, V, more, top, two);
                    walk = walk && !two;
                }
                const bool mx = fabsf(v[u].x) >= fabsf(v[u].y);
                uint32_t k;
                const int n = walk_range(g, T, v[u], s, mx, k);
                runs.add(g, T, v[u], s, mx, k, walk ? n : 0);
            } else {
                if (!single) scratch[(tail + __popc(m & ((1u << lane) - 1u))) & (RING - 1)] = (uint32_t)e[u];
                tail += __popc(m);
                if (tail - head >= 32) {
                    queued(true);
                    head += 32;
                }
            }
        }
    }
    if (IS_DENSE) runs.flush(g, T);
    else queued(lane < tail - head);
    C += one;
    F += (unsigned long long)one + full;
}

// One fused unit: the three tasks of one expanded interval [lo, hi] with
// centre c -- the contrast at c (Eqs. 11-13) and the bounds over [lo, c] and
// [c, hi] (Eqs. 14-19) -- with one pass over the events.  Per event, the
// range [min(s_lo, s_hi)(1 - 2^-18), max(s_lo, s_hi)(1 + 2^-18)] contains
// every scale the three tasks use: the binary32 scale at any D of the
// interval is within 2^-19 of the range of its end scales, so s_c and the
// halves' ends, widened by 2^-19, are within 2^-18.  Each cell coordinate is
// monotone in s, so when both ends of that range fall in one pixel, every
// task puts the event in that pixel and nowhere else: a stable event, added
// to the cell's three fields at once (its previous count, the same in all
// three, goes to V[0]).  Each warp lists the others, and once every stable
// event is in, each task adds the listed events to its own field (V[1..3]):
// one pass instead of five (with the increments of two tasks taken back
// between them) and one barrier instead of five.  The sums of squares, 2 sum(v) +
// increments, are those of three separate passes.  Returns false if the list
// or a field overflowed: then the tile holds nothing of use.  *s_over is 1
// after an overflow before the first barrier and 2 after one between the two:
// a warp that reads it late after the first barrier must not take another
// warp's overflow of the listed events for one of the first part, leave early
// and stay a barrier ahead of its block (two words instead of two values: 256
// uneven windows 49.1 -> 51.2 ms, a 1280x720 stream 56.2 -> 59.2 ms).
//
// With few candidates a unit's fixed instructions count (16 windows of
// 1280x720, 70 chunks a unit: 13,155 warp instructions), so a warp's sums stay
// within 32 bits and take one warp reduction each: previous counts are at most
// 1022, a warp has at most FUSED_CHUNKS chunks (2^16 x 32 x 1022 < 2^31) or
// WARP_WORDS listed events of at most 3 x 4096 cells (320 x 12,288 x 1022 <
// 2^32).
constexpr int FUSED_CHUNKS = 1 << 16;             // per warp
struct FusedSums {
    uint32_t V[4];                                // previous counts: stable, centre, left, right
    uint32_t n, C[3], F[2];                       // stable increments; each task's own; the halves' N_full
};

template <int F>
__device__ __forceinline__ void fused_half(const Geom& g, const Tile& T, float4 v, f32x2 foe, float s1, float s2,
                                           uint32_t& V, uint32_t& C, uint32_t& full, uint32_t& top) {
    const Span s = span_of(foe, pair(v.x, v.y), s1, s2, pair(WIDEN_DN, WIDEN_UP));
    full += counts_full(g, T, s);
    const bool single = s.a.x == s.b.x && s.a.y == s.b.y, two = adjacent(s);
    bump_pixel<F>(T, s.a, V, C, top, single | two);
    bump_pixel<F>(T, s.b, V, C, top, two);
    if (!single && !two && meets(T, s)) walk_lane<F>(g, T, v, s, V, C, top);
}

__device__ __forceinline__ bool fused_pass(const Geom& g, const Unit& un, const Tile& T, uint32_t* list,
                                           int* s_over, FusedSums& q) {
    constexpr int U = 2;
    const int lane = threadIdx.x & 31, nw = work_warps(), chunks = un.chunks;
    const float4* ev = reinterpret_cast<const float4*>(un.ev);
    const float tref = warp_tref(g, un.tau), lo = un.D_lo, hi = un.D_hi;
    const f32x2 foe = pair(g.fx, g.fy), minus_D = pair(-lo, -hi), gg = pair(warp_g(lo, tref), warp_g(hi, tref));
    const f32x2 widen = pair(1.0f - 0x1p-18f, 1.0f + 0x1p-18f);
    uint32_t top = 0;
    int listed = 0;
    Cursor cur(un);
    for (int ch = (int)(threadIdx.x >> 5); ch < chunks; ch += U * nw) {
        float4 v[U];
        int e[U];
#pragma unroll
        for (int u = 0; u < U; u++) v[u] = chunk_event(un, ev, cur, ch + u * nw, lane, e[u]);
#pragma unroll
        for (int u = 0; u < U; u++) {
            const f32x2 s2 = scales2(minus_D, gg, v[u].z);
            const Span s = span_of(foe, pair(v[u].x, v[u].y), lo_of(s2), hi_of(s2), widen);
            const bool single = s.a.x == s.b.x && s.a.y == s.b.y;
            bump_pixel<FIELD_ALL>(T, s.a, q.V[0], q.n, top, single);
            const unsigned m = __ballot_sync(0xffffffffu, !single);
            const int at = listed + __popc(m & ((1u << lane) - 1u));
            if (!single && at < WARP_WORDS) list[at] = (uint32_t)e[u];
            listed += __popc(m);
        }
    }
    if (top >= FIELD_MAX || listed > WARP_WORDS || chunks > FUSED_CHUNKS * nw) *s_over = 1;
    work_sync();
    if (*s_over == 1) return false;
    const float c = un.D_c, gc = warp_g(c, tref);
    for (int k = lane; k < listed; k += 32) {
        const float4 v = load_event(ev, (int)list[k]);
        const f32x2 s2 = scales2(minus_D, gg, v.z);
        const float sc = warp_s(c, v.z, gc);
        bump_pixel<FIELD_P>(T, pixel_of(foe, pair(v.x, v.y), sc), q.V[1], q.C[0], top);
        fused_half<FIELD_L>(g, T, v, foe, lo_of(s2), sc, q.V[2], q.C[1], q.F[0], top);
        fused_half<FIELD_R>(g, T, v, foe, sc, hi_of(s2), q.V[3], q.C[2], q.F[1], top);
    }
    if (top >= FIELD_MAX) *s_over = 2;
    work_sync();
    return !*s_over;
}

// ------------------------------------------------------------------- units

// Zeroes the tile: one instruction of one thread (bulk store of zeros),
// ordered by the block's next barrier like any store of that thread.
__device__ __forceinline__ void clear_tile(uint32_t* tile, int words) {
    asm volatile("st.bulk.weak.shared::cta [%0], %1, 0;"
                 :
                 : "r"((uint32_t)__cvta_generic_to_shared(tile)), "l"((unsigned long long)words * 4ull)
                 : "memory");
}

// A band of a bound split by events: this split's tile added into the band's
// L2 accumulator (each addition of u onto a count w adds (w + u)^2 - w^2 to S,
// so the splits' sums add up to the band's), the tile zeroed on the way; the
// last split to finish copies the image, clears the accumulated band and adds
// the band's sums to the task's.
__device__ __noinline__ void merge_split(const Geom& g, const EvalArgs& a, const Unit& un, const Tile& T, Partial* part,
                                         uint32_t* out, unsigned long long F, unsigned long long (*red)[MAX_WARPS],
                                         int* s_last) {
    const size_t task_cells = (size_t)g.planes * g.W * g.H, plane_off = (size_t)un.plane * g.W * g.H;
    const int W = g.W, P = tile_pitch(g), rows = un.rows;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = work_warps();
    uint32_t* acc = a.mg.acc + (size_t)un.task * task_cells + plane_off + (size_t)un.y0 * W;
    const size_t ti = (size_t)un.task * g.n_tiles + un.tile;
    Partial* sums = a.mg.sums + ti;
    // Splits of one band finish together: each starts its pass at its own row
    // so that they add into different words at a time.
    const int rot = (int)((uint32_t)(rows * un.split) / (uint32_t)un.splits);
    unsigned long long S = 0, C = 0;
    // Four columns per lane at a time: their additions are issued before any
    // returned count is used, so the L2 round trips overlap.
    constexpr int MERGE_COLS = 4;
    for (int q = wid; q < rows; q += nw) {
        const int r = q + rot < rows ? q + rot : q + rot - rows;
        for (int c0 = lane; c0 < W; c0 += 32 * MERGE_COLS) {
            uint32_t v[MERGE_COLS], w[MERGE_COLS];
#pragma unroll
            for (int k = 0; k < MERGE_COLS; k++) {
                const int c = c0 + 32 * k;
                v[k] = c < W ? T.cell[r * P + c] : 0u;
            }
#pragma unroll
            for (int k = 0; k < MERGE_COLS; k++) {
                const int c = c0 + 32 * k;
                w[k] = 0u;
                if (v[k]) {
                    T.cell[r * P + c] = 0u;
                    if (DD_IN(r * W + c, rows * W, 16u)) w[k] = atomicAdd(&acc[r * W + c], v[k]);
                    else v[k] = 0u;
                }
            }
#pragma unroll
            for (int k = 0; k < MERGE_COLS; k++) {
                S += (2ull * w[k] + v[k]) * v[k];
                C += v[k];
            }
        }
    }
    __threadfence();                              // this thread's additions, before the count below
    S = warp_total(S);
    C = warp_total(C);
    F = warp_total(F);
    if (lane == 0) {
        red[0][wid] = S;
        red[1][wid] = C;
        red[2][wid] = F;
    }
    work_sync();
    if (threadIdx.x == 0) {
        S = C = F = 0;
        for (int w = 0; w < nw; w++) {
            S += red[0][w];
            C += red[1][w];
            F += red[2][w];
        }
        atomicAdd(&sums->S, S);
        atomicAdd(&sums->cells[0], C);
        if (F) atomicAdd(&sums->full[0], F);
        __threadfence();
        *s_last = atomicAdd(&a.mg.done[ti], 1) == un.splits - 1;
    }
    work_sync();
    if (!*s_last) return;                         // another split finishes the band
    __threadfence();                              // every split's additions are visible now
    for (int i = threadIdx.x; i < rows * W; i += work_threads()) {
        if (out) out[i] = __ldcg(&acc[i]);
        acc[i] = 0u;
    }
    if (threadIdx.x == 0) {
        S = atomicExch(&sums->S, 0ull);
        C = atomicExch(&sums->cells[0], 0ull);
        F = atomicExch(&sums->full[0], 0ull);
        a.mg.done[ti] = 0;
        if (S) atomicAdd(&part->S, S);
        if (C) atomicAdd(&part->cells[un.plane], C);
        if (F) atomicAdd(&part->full[un.plane], F);
    }
}

// A unit's sums in shared memory, one entry per warp: [0..2] S, cells and
// N_full of the point, the bound or a fused unit's centre, [3..5] and [6..8]
// of its left and right halves.
constexpr int UNIT_SUMS = 9;

// Adds n of the warps' sums (rows 0.. of `red`) to the tasks' sums k0.. (per
// plane), the warps taking one each: nine by one warp took 0.4 us.
__device__ __forceinline__ void add_sums(const EvalArgs& a, const Unit& un, unsigned long long (*red)[MAX_WARPS],
                                         int n, int k0 = 0) {
    const int lane = threadIdx.x & 31, nw = work_warps();
    Partial* wp = a.part + (size_t)un.win * a.task_stride;
    for (int k = k0 + (int)(threadIdx.x >> 5); k < k0 + n; k += nw) {
        const unsigned long long t = warp_total(lane < nw ? red[k - k0][lane] : 0ull);
        if (lane == 0 && t) {
            Partial* q = wp + (k < 3 ? un.task : un.left + (k >= 6));
            const int f = k % 3;
            atomicAdd(f == 0 ? &q->S : (f == 1 ? &q->cells[un.plane] : &q->full[un.plane]), t);
        }
    }
}

// The pass of a point or bound unit and its warps' sums.  Images and dense
// sums are read from the finished tile.  Ends before the barrier after which
// the sums may be read and the tile cleared.  A window has at most 2^30
// events, so a warp's points and full events add up in 32 bits; a sparse
// bound's cells do in units of at most SPARSE_CHUNKS chunks: an event covers at
// most three cells in each of 4096 columns or rows (its estimate is well below
// that, but no bound on it: far from the reference time it falls short).
constexpr int SPARSE_CHUNKS = 1 << 13;
static_assert(SPARSE_CHUNKS * 32ull * 3 * 4096 <= 0xffffffffull, "a sparse unit's cells fit 32 bits");
__device__ __forceinline__ void single_unit(const Geom& g, const EvalArgs& a, const Unit& un, const Tile& T, int kind,
                                            float Dl, float Dh, uint32_t* scratch, uint32_t* out,
                                            unsigned long long (*red)[MAX_WARPS], int* s_last) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = work_warps();
    unsigned long long V = 0, C = 0, F = 0, S;
    if (kind == UNIT_POINT) point_pass(g, un, T, Dl, V, C);
    else if (kind == UNIT_DENSE) bound_pass<true>(g, un, T, Dl, Dh, scratch, V, C, F);
    else bound_pass<false>(g, un, T, Dl, Dh, scratch, V, C, F);
    S = 2 * V + C;
    if (un.splits > 1) {
        work_sync();
        merge_split(g, a, un, T, a.part + (size_t)un.win * a.task_stride + un.task, out, F, red, s_last);
        return;
    }
    if (out) {
        // Tile rows have pitch P, frame rows pitch W: warps take rows, lanes
        // take columns.
        work_sync();
        for (int r = wid; r < un.rows; r += nw)
            for (int c = lane; c < g.W; c += 32)
                if (DD_IN(r * g.W + c, un.rows * g.W, 16u)) out[r * g.W + c] = T.cell[r * tile_pitch(g) + c];
    }
    if (kind == UNIT_DENSE) {
        // The band's rows are contiguous in the tile (the padding column of an
        // odd pitch stays zero): 16-byte words, then the tail.
        work_sync();
        const int words = un.rows * tile_pitch(g), quads = words >> 2;
        const uint4* t4 = reinterpret_cast<const uint4*>(T.cell);
        S = C = 0;
        for (int i = threadIdx.x; i < quads; i += work_threads()) {
            const uint4 v = t4[i];
            S += (unsigned long long)v.x * v.x + (unsigned long long)v.y * v.y + (unsigned long long)v.z * v.z +
                 (unsigned long long)v.w * v.w;
            C += (unsigned long long)v.x + v.y + v.z + v.w;
        }
        for (int i = 4 * quads + threadIdx.x; i < words; i += work_threads()) {
            const uint32_t v = T.cell[i];
            S += (unsigned long long)v * v;
            C += v;
        }
    }
    S = warp_total(S);
    const bool wide = kind == UNIT_DENSE || (kind == UNIT_BOUND && un.chunks > SPARSE_CHUNKS);
    C = wide ? warp_total(C) : __reduce_add_sync(0xffffffffu, (uint32_t)C);
    if (kind != UNIT_POINT) F = __reduce_add_sync(0xffffffffu, (uint32_t)F);
    if (lane == 0) {
        red[0][wid] = S;
        red[1][wid] = C;
        red[2][wid] = F;
    }
}

// A fused unit and its warps' sums; if its list or a field overflows, its
// three tasks run as ordinary units over the same candidates.  Returns the
// number of sums left in `red`.
__device__ __forceinline__ int fused_unit(const Geom& g, const EvalArgs& a, const Unit& un, const Tile& T,
                                          int tile_words, uint32_t* scratch, unsigned long long (*red)[MAX_WARPS],
                                          int* s_over, int* s_last) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    FusedSums q = {};
    if (fused_pass(g, un, T, scratch, s_over, q)) {
        auto total = [](uint32_t x) { return __reduce_add_sync(0xffffffffu, x); };
        const uint32_t n = total(q.n), v0 = total(q.V[0]);
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const uint32_t v = total(q.V[k + 1]), c = total(q.C[k]), f = k ? n + total(q.F[k - 1]) : 0u;
            if (lane == 0) {
                red[3 * k][wid] = 2 * ((unsigned long long)v0 + v) + n + c;
                red[3 * k + 1][wid] = n + c;
                red[3 * k + 2][wid] = f;
            }
        }
        return 9;
    }
    const int kind = bound_cells(g, un.D_lo, un.D_hi, un.tau) >= DENSE_CELLS ? UNIT_DENSE : UNIT_BOUND;
    for (int k = 0; k < 3; k++) {
        work_sync();
        if (threadIdx.x == 0) clear_tile(T.cell, tile_words);
        work_sync();
        single_unit(g, a, un, T, k == 0 ? UNIT_POINT : kind, k == 1 ? un.D_lo : un.D_c, k == 1 ? un.D_c : un.D_hi,
                    scratch, nullptr, red, s_last);
        work_sync();
        add_sums(a, un, red, 3, 3 * k);
    }
    return 0;
}

// IWE evaluation of the round's job list.  A grid of resident blocks takes
// units (job, row band).  The last warp of a block only prepares units, one
// ahead of the others: a unit's preparation is a chain of dependent L2 loads
// (its number, job, window, bin offsets) that takes longer than a small unit's
// pass over its events.  Per unit there is one barrier of the whole block
// (the unit is prepared, the tile is clear) and one of the working warps (the
// pass is done), after which the sums go to the tasks and the tile is cleared
// by different warps.  Block b starts with unit b; later units come from a
// counter, which numbers them from the number of blocks on.  Block 0 clears the other
// parity's list and counter for the control blocks of this round.
//
// What bounds it: with many units, issue slots (60 bounds of 100,000 events:
// 70-84% of the cycles issue, DRAM under 1%), so the passes are written for
// few instructions per event and cell; with few units, the latency of a unit
// (its preparation 2.7 us, two barriers, one L2 round trip per four chunks).
// Two blocks of 480 + 32 threads per SM with 64 registers a thread and tiles
// of up to 91 KB: three of 256 + 32 with smaller tiles are 4% faster on
// 640-pixel frames in late rounds but 29% slower on 1280-pixel ones, where
// the lower tile re-reads more events.  Against one thread deciding each
// unit's split, candidates and sums in every warp (512 threads, 3 blocks of 40
// registers): 129 points of 100,000 events 74 -> 50 us, 60 bounds of width
// 1/2 569 -> 340 us, of width 1/32 124 -> 90 us; 256 uneven windows 97.8 ->
// 64.2 ms, 96 windows of a 1280x720 stream 112.0 -> 66.2 ms.
struct EvalShared {
    Unit un[2];
    unsigned long long red[UNIT_SUMS][MAX_WARPS];
    uint32_t idle[32];
    int last;
    int over;                // a fused unit's overflow (fused_pass)
};

// The share of block `block` of `blocks` in a round of n_units units.  The tile arrives clear and
// leaves clear; ends with a barrier of the whole block.
__device__ __forceinline__ void eval_round(const Geom& g, const EvalArgs& a, const Job* jobs, int32_t* work, int n_units,
                                           int slices, int block, int blocks, uint32_t* tile, EvalShared& sm) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = work_warps();
    if (wid == nw) {                              // the preparing warp
        int id = block;
        for (int b = 0;; b ^= 1) {
            prepare_unit(g, a, jobs, id, n_units, slices, sm.un[b]);
            __syncthreads();
            if (id >= n_units) return;
            id = n_units;
            if (lane == 0 && n_units > blocks) id = blocks + atomicAdd(work, 1);
            id = __shfl_sync(0xffffffffu, id, 0);
        }
    }
    const int tile_words = eval_tile_words(g);
    uint32_t* scratch = tile + tile_words + WARP_WORDS * wid;
    for (int b = 0;; b ^= 1) {
        __syncthreads();                          // unit b is prepared, the tile is clear
        const Unit& un = sm.un[b];
        if (un.kind == UNIT_NONE) return;
        Tile T;
        T.cell = tile;
        T.pitch = 4u * (uint32_t)tile_pitch(g);
        T.idle = (uint32_t)__cvta_generic_to_shared(sm.idle + lane);
        T.row0 = CELL0 + (uint32_t)un.y0;
        T.base = (uint32_t)__cvta_generic_to_shared(tile) - T.row0 * T.pitch - 4u * CELL0;
        T.rows = (uint32_t)un.rows;
        T.W = (uint32_t)g.W;
        int sums = 3;
        if (un.kind == UNIT_FUSED) {
            sums = fused_unit(g, a, un, T, tile_words, scratch, sm.red, &sm.over, &sm.last);
        } else {
            uint32_t* out = a.iwe_out ? a.iwe_out + ((size_t)un.task * g.planes + un.plane) * g.W * g.H + (size_t)un.y0 * g.W
                                      : nullptr;
            single_unit(g, a, un, T, un.kind, un.D_lo, un.D_hi, scratch, out, sm.red, &sm.last);
            if (un.splits > 1) sums = 0;
        }
        work_sync();                              // the pass is done
        if (threadIdx.x == 0) {
            clear_tile(tile, tile_words);
            sm.over = 0;
        }
        add_sums(a, un, sm.red, sums);
    }
}

__global__ void __launch_bounds__(EVAL_THREADS + 32, 2) k_eval(const __grid_constant__ Geom g,
                                                               const __grid_constant__ EvalArgs a) {
    extern __shared__ __align__(16) uint32_t tile[];
    __shared__ EvalShared sm;
    Sched* sch = a.sch;
    const int par = sch->round & 1;
    const int n_units = sch->n_jobs[par] * g.n_tiles * a.slices;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sch->n_jobs[par ^ 1] = 0;
        sch->work[par ^ 1] = 0;
    }
    if ((int)blockIdx.x >= n_units) return;
    if (threadIdx.x == 0) {
        clear_tile(tile, eval_tile_words(g));
        sm.over = 0;
    }
    eval_round(g, a, a.jobs + (size_t)par * a.job_stride, &sch->work[par], n_units, a.slices, blockIdx.x, gridDim.x, tile,
               sm);
}

// The checked-build error word (always 0 in other builds); reset clears it.
cudaError_t check_flags(uint32_t* flags, int32_t* checked, bool reset) {
#ifdef DD_CHECKED
    cudaError_t e = cudaMemcpyFromSymbol(flags, g_dd_check, sizeof(uint32_t));
    if (e == cudaSuccess && reset) {
        const uint32_t zero = 0;
        e = cudaMemcpyToSymbol(g_dd_check, &zero, sizeof(uint32_t));
    }
    *checked = 1;
    return e;
#else
    (void)reset;
    *flags = 0;
    *checked = 0;
    return cudaSuccess;
#endif
}

int eval_resident_blocks(const Geom& g, int threads) {
    int per_sm = 0, dev = 0, sms = 0;
    const size_t smem = eval_smem_bytes(g, threads);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_eval, threads + 32, smem) != cudaSuccess) return 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return per_sm * sms;
}

cudaError_t launch_eval(const Geom& g, const EvalArgs& a, int threads, int grid_blocks, cudaStream_t s) {
    if (grid_blocks <= 0) return cudaErrorInvalidValue;
    k_eval<<<grid_blocks, threads + 32, eval_smem_bytes(g, threads), s>>>(g, a);
    return cudaGetLastError();
}

// ------------------------------------------------------------------- keys

__global__ void k_keys(Geom g, const Task* tasks, int32_t n_tasks, Partial* part, i128* key,
                       unsigned long long* S_out, unsigned long long* C_out, unsigned long long* F_out,
                       const int32_t* err, int32_t* err_out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0 && err_out) *err_out = *err;
    if (t >= n_tasks) return;
    const Partial p = part[t];
    part[t] = Partial{};                          // cleared for the next evaluation
    const int64_t M = (int64_t)g.W * g.H;
    key[t] = partial_key(M, p, tasks[t].kind == TASK_POINT);
    S_out[t] = p.S;
    C_out[t] = p.cells[0] + p.cells[1];
    F_out[t] = p.full[0] + p.full[1];
}

cudaError_t launch_keys(const Geom& g, const Task* tasks, int32_t n_tasks, Partial* part, i128* key,
                        unsigned long long* S, unsigned long long* cells, unsigned long long* full,
                        cudaStream_t s, const int32_t* err, int32_t* err_out) {
    if (n_tasks <= 0) return cudaSuccess;
    k_keys<<<(n_tasks + 63) / 64, 64, 0, s>>>(g, tasks, n_tasks, part, key, S, cells, full, err, err_out);
    return cudaGetLastError();
}

constexpr int Q_STAGE = 256;   // queued intervals staged in shared memory for the merge

// Shared memory of one control step (one block of k_control per window).
struct __align__(16) CtlShared {
    SolveState s;
    i128 key[3 * MAX_POP];
    unsigned long long cells[3 * MAX_POP];
    Node kids[2 * MAX_POP + 1];
    Node sorted_kids[2 * MAX_POP + 1];
    Node q_stage[Q_STAGE];
    Node q_head[MAX_POP];               // the merged queue's first entries, for the dequeue
    float4 t_iv[3 * MAX_POP];           // per next-round task: its interval, and its centre (points)
    int16_t t_fuse[3 * MAX_POP];        // per next-round task: 0 own jobs, -1 part of a fused
                                        // job, k > 0 the centre of a fused job (left half k - 1)
    int8_t t_dense[3 * MAX_POP];        // per next-round task: a dense bound that may be split
    int16_t t_jobs[3 * MAX_POP];        // per next-round task, in job order: its number of jobs
    int16_t t_at[3 * MAX_POP];          // and the place of its first one in the window's jobs
    uint4 pop_mask[2];                  // per 32 dequeued: to split, fused, dense left and right halves
    int pop_fail[2];                    // first that fails the gap test
    int s_nk, s_stop, s_base, s_total;
    int q_shared;                       // resident: the queue is in the block's shared memory
};

__device__ __forceinline__ float centre(float lo, float hi) {
    return __fadd_rn(lo, __fmul_rn(0.5f, __fsub_rn(hi, lo)));
}

// One block per window w0 + b: the search state, the first tasks (the centre
// of the domain and the bound of the domain) and their jobs in the list the
// next evaluation reads.  `sharers`: the searches that share the rounds
// (their bound tasks split to fill 1/sharers of the grid; 0: never split).
__global__ void k_init(Geom g, int32_t sharers, int32_t w0, SolveState* st_all, Task* tasks_all,
                       int32_t task_stride, Partial* part_all, const WinIn* wins, const WinParams* params,
                       Job* jobs_all, int32_t job_stride, Sched* sch, int32_t K_pop, int32_t qcap,
                       int64_t max_rounds, int32_t trace_cap) {
    const int w = w0 + blockIdx.x;
    for (int i = threadIdx.x; i < task_stride; i += blockDim.x)   // the window's task sums start at zero
        part_all[(size_t)w * task_stride + i] = Partial{};
    if (threadIdx.x != 0) return;
    const int par = sch->round & 1;
    Job* jobs = jobs_all + (size_t)par * job_stride;
    SolveState* st = st_all + w;
    Task* tasks = tasks_all + (size_t)w * task_stride;
    const WinParams pr = params[w];
    const float tau = wins[w].tau;
    st->gamma_K = pr.gamma_K;
    st->M = (int64_t)g.W * g.H;
    st->max_rounds = max_rounds;
    st->D_lo = pr.D_lo;
    st->D_hi = pr.D_hi;
    st->tol = pr.tol;
    st->tau = tau;
    st->K_pop = K_pop;
    st->qcap = qcap;
    st->trace_cap = trace_cap;
    st->K_hat = 0;
    st->leaf_max = 0;
    st->stop_kb = 0;
    st->warm = pr.warm;
    st->D_warm = 0.0f;
    st->w_warm = 0.0f;
    // The pieces the domain enters the queue as: the domain itself, or with
    // a warm start the pieces of positive width cut at guess -/+ half-width.
    float cut[4] = {pr.D_lo, pr.D_hi, pr.D_hi, pr.D_hi};
    int n_cut = 2;
    if (pr.warm) {
        float d = pr.D_warm;                      // the guess, clamped into the domain
        if (!(d >= pr.D_lo)) d = pr.D_lo;
        if (d > pr.D_hi) d = pr.D_hi;
        float a = __fsub_rn(d, pr.w_warm), b = __fadd_rn(d, pr.w_warm);
        if (!(a >= pr.D_lo)) a = pr.D_lo;
        if (!(b <= pr.D_hi)) b = pr.D_hi;
        cut[1] = a;
        cut[2] = b;
        n_cut = 4;
        st->D_hat = d;                            // incumbent = the guess
        st->D_warm = d;
        st->w_warm = pr.w_warm;
    } else {
        st->D_hat = centre(pr.D_lo, pr.D_hi);     // incumbent = centre of the domain
    }
    st->phase = PH_INIT;
    st->status = DD_OK;
    st->cancel = 0;
    st->n_pop = 0;
    st->q_n = 0;
    st->q_start = 0;
    st->q_cur = 0;
    st->have_leaf = 0;
    st->have_stop = 0;
    st->nodes_expanded = st->point_evals = st->bound_evals = st->cells = st->bcells = 0;
    st->rounds = st->max_queue = st->trace_len = 0;
    Task a;
    a.D_lo = a.D_hi = st->D_hat;
    a.kind = TASK_POINT;
    a.splits = 1;
    tasks[0] = a;
    int nt = 1, n_jobs = 1;
    int n_pieces = 0, n_dense = 0, rank = 0;
    for (int i = 0; i + 1 < n_cut; i++)
        if (cut[i] < cut[i + 1]) {
            n_pieces++;
            n_dense += bound_cells(g, cut[i], cut[i + 1], tau) >= DENSE_CELLS;
        }
    for (int i = 0; i + 1 < n_cut; i++) {
        if (!(cut[i] < cut[i + 1])) continue;
        Task b;                                   // bound of one piece
        b.D_lo = cut[i];
        b.D_hi = cut[i + 1];
        b.kind = TASK_BOUND;
        const bool dense = bound_cells(g, b.D_lo, b.D_hi, tau) >= DENSE_CELLS;
        b.splits = sharers > 0 && dense ? fill_splits(g, g.split_target / sharers, (1 + n_pieces) * g.n_tiles,
                                                      n_dense, rank++)
                                        : 1;
        tasks[nt++] = b;
        n_jobs += b.splits;
    }
    st->n_tasks = nt;
    const int base = atomicAdd(&sch->n_jobs[par], n_jobs);
    int o = base;
    for (int t = 1; t < nt; t++)                  // bounds first (heavier)
        for (int s = 0; s < tasks[t].splits; s++) {
            Job j;
            j.win = w;
            j.task = t;
            j.split = s;
            j.splits = tasks[t].splits;
            j.D_lo = tasks[t].D_lo;
            j.D_hi = tasks[t].D_hi;
            j.D_c = 0.0f;
            j.kind = TASK_BOUND;
            jobs[o++] = j;
        }
    Job j;
    j.win = w;
    j.task = 0;
    j.split = 0;
    j.splits = 1;
    j.D_lo = j.D_hi = j.D_c = tasks[0].D_lo;
    j.kind = TASK_POINT;
    jobs[o] = j;
}

cudaError_t launch_init(const Geom& g, int32_t n_windows, SolveState* st, Task* tasks, int32_t task_stride,
                        Partial* part, const WinIn* wins, const WinParams* params, Job* jobs, int32_t job_stride,
                        Sched* sch, int32_t K_pop, int32_t qcap, int64_t max_rounds, int32_t trace_cap,
                        cudaStream_t s, int32_t w0, int32_t sharers) {
    if (sharers < 0) sharers = n_windows;
    k_init<<<n_windows, 32, 0, s>>>(g, sharers, w0, st, tasks, task_stride, part, wins, params, jobs, job_stride,
                                    sch, K_pop, qcap, max_rounds, trace_cap);
    return cudaGetLastError();
}

// Priority order of the queue: larger Kbar first, ties to the smaller D_lo.
// Distinct queued intervals have distinct D_lo, so the order is total.
__device__ __forceinline__ bool better(const Node& a, const Node& b) {
    return a.kb > b.kb || (a.kb == b.kb && a.lo < b.lo);
}

// Number of entries of the sorted array q[0..n) that come before e.
__device__ __forceinline__ int rank_in(const Node* q, int n, const Node& e) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (better(q[mid], e)) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

constexpr int CTL_THREADS = 256;

// Warp maximum of non-negative 128-bit values, word by word from the top (a
// lane without a value passes 0); `at`: the lanes that hold it.
__device__ __forceinline__ i128 warp_max_i128(i128 v, bool valid, unsigned& at) {
    uint32_t w[4], m[4];
    for (int k = 0; k < 4; k++) w[k] = (uint32_t)((unsigned __int128)v >> (32 * k));
    bool in = valid;
    for (int k = 3; k >= 0; k--) {
        m[k] = __reduce_max_sync(0xffffffffu, in ? w[k] : 0u);
        in = in && w[k] == m[k];
    }
    at = __ballot_sync(0xffffffffu, in);
    return (i128)(((unsigned __int128)((unsigned long long)m[3] << 32 | m[2]) << 64) |
                  ((unsigned long long)m[1] << 32 | m[0]));
}

// One block per window.  Consumes the keys of the round just evaluated
// (Algorithm 1: incumbent update, leaves, child bounds and their insertion),
// then dequeues the next batch (dequeue and gap test) and writes its tasks
// and jobs, or finishes.  The search state is staged in shared memory.  The
// queue is kept sorted in priority order in one of two buffers: insertion is
// a parallel merge into the other buffer, a dequeue takes a prefix.  The last
// block to finish counts the windows still searching, advances the round and
// sets the graph loop condition (with one window, its block does so
// directly).
//
// Nothing here is much work (at most 64 intervals and 128 children): its time
// is the chain of dependent steps, so the steps are as wide as the data allows
// (a thread per task, child, queued interval or dequeued interval; the sums
// and maxima of a round by different warps) and a block barrier apart.  Per
// round of one window, in k_search: 6.5 -> 4 us.
//
// RESIDENT (the control block of k_search): the state stays in `sm` from round
// to round, and so does the queue while it has at most q_cap entries (two
// buffers of q_cap at q_mem); the state reaches global memory when the search
// ends, the queue when it grows beyond that.  FEW: its launch has several
// windows.
template <bool RESIDENT, bool FEW = false>
__device__ __forceinline__ void control_body(const Geom& g, const CtlArgs& c, int w, CtlShared& sm, int par,
                                             Node* q_mem = nullptr, int q_cap = 0) {
    SolveState& s = sm.s;
    i128* key = sm.key;
    unsigned long long* cells = sm.cells;
    Sched* sch = c.sch;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nwarps = (int)blockDim.x >> 5;
    // searches still running after the last round
    const int running = !RESIDENT ? sch->running : (FEW ? __ldcg(&sch->running) : 1);
    SolveState* st = c.st_all + w;
    Task* tasks = c.tasks_all + (size_t)w * c.task_stride;
    Partial* part = c.part_all + (size_t)w * c.task_stride;
    Job* jobs = c.jobs_all + (size_t)(par ^ 1) * c.job_stride;
    static_assert(sizeof(SolveState) % 16 == 0, "state is copied as int4");
    if (!RESIDENT) {
        for (int i = tid; i < (int)(sizeof(SolveState) / 16); i += blockDim.x)
            reinterpret_cast<int4*>(&s)[i] = reinterpret_cast<const int4*>(st)[i];
        __syncthreads();
    }
    const int phase = s.phase;                    // read before a barrier: one thread changes it
    if (phase != PH_DONE) {
    Node* qa = c.queues + (size_t)w * 2 * s.qcap;
    Node* qb = qa + s.qcap;
    const int64_t M = s.M;
    const int n_tasks = s.n_tasks, np0 = s.n_pop, n_points = phase == PH_INIT ? 1 : np0;   // points come first

    // Each task's sums (accumulated by the evaluation over its row bands, in
    // L2), read and cleared for the next round.
    for (int t = tid; t < n_tasks; t += blockDim.x) {
        Partial q;
        q.S = __ldcg(&part[t].S);
        for (int k = 0; k < 2; k++) {
            q.cells[k] = __ldcg(&part[t].cells[k]);
            q.full[k] = __ldcg(&part[t].full[k]);
        }
        part[t] = Partial{};
        key[t] = partial_key(M, q, t < n_points);
        cells[t] = q.cells[0] + q.cells[1];
    }
    if (tid == 0) {
        sm.s_nk = 0;
        sm.s_stop = 0;
        if (!RESIDENT || phase == PH_INIT) {
            if (c.err_all[w]) {                   // malformed events
                s.status = DD_ERR_ARG;
                sm.s_stop = 1;
            } else if (s.cancel) {                // the host cancelled the search between rounds
                s.status = DD_ERR_CANCELLED;
                sm.s_stop = 1;
            }
        }
    }
    __syncthreads();
    int stop = sm.s_stop;

    // The incumbent, the counters and the leaves, each by a warp of its own.
    if (!stop && phase == PH_INIT) {
        if (tid == 0) {
            s.K_hat = key[0];
            s.point_evals = 1;
            s.bound_evals = n_tasks - 1;
            s.cells = (int64_t)cells[0];
            s.bcells = 0;
            for (int t = 1; t < n_tasks; t++) {
                s.cells += (int64_t)cells[t];
                s.bcells += (int64_t)cells[t];
            }
            s.phase = PH_RUN;
        }
    } else if (!stop) {
        if (wid == 0) {
            // Incumbent update in dequeue order (a centre with K >= K_hat
            // wins): per chunk of 32, the chunk maximum wins if it reaches
            // the running incumbent, at the last lane attaining it.
            i128 K_hat = s.K_hat;
            int best = -1;
            for (int base = 0; base < np0; base += 32) {
                const bool v = base + lane < np0;
                unsigned at;
                const i128 m = warp_max_i128(v ? key[base + lane] : (i128)0, v, at);
                if (m >= K_hat) {
                    K_hat = m;
                    best = base + 31 - __clz(at);
                }
            }
            if (lane == 0) {
                s.K_hat = K_hat;
                if (best >= 0) s.D_hat = s.pop[best].c;
            }
        }
        if (wid == (nwarps > 2 ? 1 : 0)) {        // cells of the points and of all tasks
            unsigned long long pc = 0, all = 0;
            for (int t = lane; t < n_tasks; t += 32) {
                if (t < np0) pc += cells[t];
                all += cells[t];
            }
            pc = warp_total(pc);
            all = warp_total(all);
            if (lane == 0) {
                s.nodes_expanded += np0;
                s.point_evals += np0;
                s.bound_evals += n_tasks - np0;
                s.cells += (int64_t)all;
                s.bcells += (int64_t)(all - pc);
            }
        }
        if (wid == (nwarps > 2 ? 2 : 1)) {        // the largest bound among the leaves
            bool any = false;
            i128 lmax = 0;
            for (int base = 0; base < np0; base += 32) {
                const bool v = base + lane < np0 && s.pop[base + lane].leaf;
                unsigned at;
                const i128 m = warp_max_i128(v ? s.pop[base + lane].kb : (i128)0, v, at);
                if (at && (!any || m > lmax)) lmax = m;
                any |= at != 0;
            }
            if (lane == 0 && any) {
                if (!s.have_leaf || lmax > s.leaf_max) s.leaf_max = lmax;
                s.have_leaf = 1;
            }
        }
        if (c.trace && w == 0)
            for (int j = tid; j < np0; j += blockDim.x)
                if (s.trace_len + j < s.trace_cap) {
                    const Popped& p = s.pop[j];
                    TraceRec r;
                    r.D_lo = p.lo;
                    r.D_hi = p.hi;
                    r.D_c = p.c;
                    r.leaf = p.leaf;
                    r.Kbar = p.kb;
                    r.K_c = key[p.t_point];
                    c.trace[s.trace_len + j] = r;
                }
    }
    __syncthreads();

    // Children (or the first pieces) that reach the end-of-round incumbent,
    // one thread each, in any order: they are sorted next.
    const i128 K_hat = s.K_hat;
    if (!stop) {
        const int nc = phase == PH_INIT ? n_tasks - 1 : 2 * np0;
        for (int k = tid; k < nc; k += blockDim.x) {
            Node nd;
            nd.pad0 = nd.pad1 = 0;
            bool in;
            if (phase == PH_INIT) {
                // the domain is queued unconditionally; warm-start pieces
                // when their bound reaches the incumbent, as children are
                nd.lo = tasks[1 + k].D_lo;
                nd.hi = tasks[1 + k].D_hi;
                nd.kb = key[1 + k];
                in = !s.warm || nd.kb >= K_hat;
            } else {
                const Popped& p = s.pop[k >> 1];
                const bool right = k & 1;
                nd.lo = right ? p.c : p.lo;
                nd.hi = right ? p.hi : p.c;
                nd.kb = p.leaf ? (i128)0 : key[right ? p.t_right : p.t_left];
                in = !p.leaf && nd.kb >= K_hat;
            }
            if (in) sm.kids[atomicAdd(&sm.s_nk, 1)] = nd;
        }
    }
    __syncthreads();
    const int nk = sm.s_nk, a = s.q_n;
    if (!stop && a + nk > s.qcap) stop = 2;       // (the same for every thread)
    if (stop == 2 && tid == 0) s.status = DD_ERR_QUEUE_OVERFLOW;

    if (!stop) {
        // Sort the new children, then merge them with the queued intervals; a
        // queue in global memory that fits is staged in shared memory first,
        // so that the children's ranks are searched there.
        const bool in_shared = RESIDENT && sm.q_shared, to_shared = RESIDENT && a + nk <= q_cap;
        const Node* src = (in_shared ? q_mem + (s.q_cur ? q_cap : 0) : (s.q_cur ? qb : qa)) + s.q_start;
        Node* dst = to_shared ? q_mem + (s.q_cur ? 0 : q_cap) : (s.q_cur ? qa : qb);
        const bool staged = !in_shared && a <= Q_STAGE;
        // A child's rank among the children (they are distinct: popped
        // intervals are disjoint) counted by `per` threads, each over every
        // per-th child, summed within the thread group.
        int per = 1, lg = 0;
        while (nk > 8 && per < 32 && 2 * per * nk <= (int)blockDim.x) {
            per *= 2;
            lg++;
        }
        for (int base = 0; base < nk * per; base += blockDim.x) {
            const int i = (base + tid) >> lg, p = (base + tid) & (per - 1);
            int r = 0;
            if (i < nk)
                for (int j = p; j < nk; j += per) r += better(sm.kids[j], sm.kids[i]);
            for (int o = per / 2; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
            if (i < nk && p == 0) sm.sorted_kids[r] = sm.kids[i];
        }
        if (staged)
            for (int i = tid; i < a; i += blockDim.x) sm.q_stage[i] = src[i];
        __syncthreads();
        const Node* qs = staged ? sm.q_stage : src;
        // Children from the last thread down, queued intervals from the first
        // up: one pass of different warps.
        for (int i = tid; i < a; i += blockDim.x) {
            const Node e = qs[i];
            const int at = i + rank_in(sm.sorted_kids, nk, e);
            dst[at] = e;
            if (at < MAX_POP) sm.q_head[at] = e;
        }
        for (int j = (int)blockDim.x - 1 - tid; j < nk; j += blockDim.x) {
            const Node e = sm.sorted_kids[j];
            const int at = j + rank_in(qs, a, e);
            dst[at] = e;
            if (at < MAX_POP) sm.q_head[at] = e;
        }
        __syncthreads();
        if (tid == 0) {
            s.q_cur ^= 1;
            s.q_start = 0;
            s.q_n = a + nk;
            sm.q_shared = to_shared;
            s.trace_len += phase == PH_INIT ? 0 : np0;
            if (s.q_n > s.max_queue) s.max_queue = s.q_n;
        }
    }

    // Dequeue up to K_pop intervals, one thread each (two warps): the gap
    // test, the centre and the bisection, and which tasks the interval will
    // need; the first that fails the gap test ends the batch.
    const int lim = stop ? 0 : min(s.K_pop, a + nk);
    Popped p;
    bool split = false, fuse = false, dense_l = false, dense_r = false;
    if (wid < 2) {
        const bool v = tid < lim;
        bool pass = false;
        if (v) {
            const Node nd = sm.q_head[tid];
            pass = nd.kb - K_hat > s.gamma_K;     // gap test
            p.lo = nd.lo;
            p.hi = nd.hi;
            p.kb = nd.kb;
            p.c = centre(p.lo, p.hi);
            const float wd = __fsub_rn(p.hi, p.lo);
            p.leaf = !(wd > s.tol) || !(p.c > p.lo) || !(p.c < p.hi);
            split = !p.leaf;
            // narrow intervals: centre and halves evaluated by one fused job
            fuse = split && g.fuse_cells > 0.0f && bound_cells(g, p.lo, p.hi, s.tau) - 1.0f <= g.fuse_cells;
            // dense bounds (splittable when the round is small)
            const bool own = split && !fuse && c.split_ok;
            dense_l = own && bound_cells(g, p.lo, p.c, s.tau) >= DENSE_CELLS;
            dense_r = own && bound_cells(g, p.c, p.hi, s.tau) >= DENSE_CELLS;
        }
        const unsigned fail = __ballot_sync(0xffffffffu, v && !pass);
        const unsigned ms = __ballot_sync(0xffffffffu, split), mf = __ballot_sync(0xffffffffu, fuse);
        const unsigned ml = __ballot_sync(0xffffffffu, dense_l), mr = __ballot_sync(0xffffffffu, dense_r);
        if (lane == 0) {
            sm.pop_fail[wid] = fail ? 32 * wid + __ffs(fail) - 1 : MAX_POP;
            sm.pop_mask[wid] = make_uint4(ms, mf, ml, mr);
        }
    }
    __syncthreads();
    const int first = min(sm.pop_fail[0], sm.pop_fail[1]), np = min(lim, first);
    const unsigned in0 = np >= 32 ? 0xffffffffu : (1u << np) - 1u;
    const unsigned in1 = np >= 64 ? 0xffffffffu : (np > 32 ? (1u << (np - 32)) - 1u : 0u);
    const uint4 m0 = sm.pop_mask[0], m1 = sm.pop_mask[1];
    const int n_split = __popc(m0.x & in0) + __popc(m1.x & in1);
    const int nt = np + 2 * n_split, n_fused = __popc(m0.y & in0) + __popc(m1.y & in1);
    const int nd = __popc(m0.z & in0) + __popc(m1.z & in1) + __popc(m0.w & in0) + __popc(m1.w & in1);
    const bool late = np > 0 && s.rounds + 1 > s.max_rounds, done = np == 0 || late;
    if (wid < 2 && tid < np) {
        const unsigned below = (1u << lane) - 1u;
        p.t_point = tid;
        p.t_left = p.t_right = -1;
        p.pad = 0;
        sm.t_iv[tid] = make_float4(p.lo, p.hi, p.c, 0.0f);
        sm.t_fuse[tid] = 0;
        sm.t_dense[tid] = 0;
        if (split) {
            const int l = np + 2 * (__popc((wid ? m1.x : m0.x) & below) + (wid ? __popc(m0.x) : 0));
            p.t_left = l;
            p.t_right = l + 1;
            sm.t_fuse[tid] = fuse ? (int16_t)(l + 1) : (int16_t)0;
            sm.t_fuse[l] = sm.t_fuse[l + 1] = fuse ? (int16_t)-1 : (int16_t)0;
            sm.t_dense[l] = dense_l;
            sm.t_dense[l + 1] = dense_r;
            sm.t_iv[l] = make_float4(p.lo, p.c, 0.0f, 0.0f);
            sm.t_iv[l + 1] = make_float4(p.c, p.hi, 0.0f, 0.0f);
        }
        s.pop[tid] = p;
    }
    __syncthreads();                              // the state above is read, the tasks' kinds are known
    if (tid == 0) {
        if (!stop && first == 0 && lim > 0) {     // the search ends here
            s.have_stop = 1;
            s.stop_kb = sm.q_head[0].kb;
        }
        s.q_start = np;
        s.q_n -= np;
        s.n_pop = done ? 0 : np;
        s.n_tasks = done ? 0 : nt;
        if (np > 0) s.rounds++;
        if (late) {
            s.status = DD_ERR_TIMEOUT;
            s.stop_kb = 0;
            s.n_pop = np;
        } else if (done) {
            i128 top = K_hat;
            if (s.have_leaf && s.leaf_max > top) top = s.leaf_max;
            if (s.have_stop && s.stop_kb > top) top = s.stop_kb;
            s.stop_kb = top - K_hat;              // the certificate gap_K
        }
        if (done) s.phase = PH_DONE;
    }
    // Jobs of the next round, bound tasks first: a task of `splits` splits
    // contributes that many jobs (fill_splits for the dense bounds, ranked in
    // this loop's order; every other task has one split).
    if (wid == 0 && !done) {
        const int units = (nt - 2 * n_fused) * g.n_tiles;    // one per job and band before any split
        // the window's share of the grid: the searches still running after
        // the last round share it (all of them before the first)
        const int sharers = c.n_windows == 1 ? 1 : (running > 0 ? running : c.n_windows);
        const int target = sharers == 1 ? g.split_target : g.split_target / sharers;
        const bool extra = nd > 0 && target - units >= g.n_tiles;
        int total = 0, seen = 0;
        for (int c0 = 0; c0 < nt; c0 += 32) {     // jobs per task, counted once
            const int q = c0 + lane, t = nt - 1 - q;
            int n = q < nt && sm.t_fuse[t] >= 0 ? 1 : 0;
            int before;
            if (extra) {
                const bool d = q < nt && sm.t_dense[t];
                const unsigned db = __ballot_sync(0xffffffffu, d);
                if (d) n = fill_splits(g, target, units, nd, seen + __popc(db & ((1u << lane) - 1u)));
                seen += __popc(db);
                const int incl = warp_incl_scan(n);
                before = total + incl - n;
                total += __shfl_sync(0xffffffffu, incl, 31);
            } else {                              // one job or none each
                const unsigned b = __ballot_sync(0xffffffffu, n);
                before = total + __popc(b & ((1u << lane) - 1u));
                total += __popc(b);
            }
            if (q < nt) {
                sm.t_jobs[q] = (int16_t)n;
                sm.t_at[q] = (int16_t)before;
            }
        }
        if (lane == 0) {
            sm.s_total = total;
            if (c.n_windows == 1) {               // the only block: the list is its own
                if (!RESIDENT) sch->n_jobs[par ^ 1] = total;
                sm.s_base = 0;
            } else {
                sm.s_base = atomicAdd(&sch->n_jobs[par ^ 1], total);
            }
        }
    }
    __syncthreads();
    if (!done)                                    // the jobs, written by the whole block
        for (int q = tid; q < nt; q += blockDim.x) {
            const int n = sm.t_jobs[q], t = nt - 1 - q;
            if (n == 0) continue;
            const int fz = (int)sm.t_fuse[t];
            Job* out = jobs + sm.s_base + sm.t_at[q];
            Job j;
            j.win = w;
            j.task = t;
            j.kind = t < np ? TASK_POINT : TASK_BOUND;
            const float4 iv = sm.t_iv[t];         // a point's: its centre and, to be fused, its interval
            j.D_lo = fz > 0 ? iv.x : (t < np ? iv.z : iv.x);
            j.D_hi = fz > 0 ? iv.y : (t < np ? iv.z : iv.y);
            j.D_c = iv.z;
            for (int k = 0; k < n; k++) {
                j.split = fz > 0 ? fz - 1 : k;
                j.splits = fz > 0 ? -1 : n;
                out[k] = j;
            }
        }
    if (!RESIDENT || done)
        for (int i = tid; i < (int)(sizeof(SolveState) / 16); i += blockDim.x)
            reinterpret_cast<int4*>(st)[i] = reinterpret_cast<const int4*>(&s)[i];
    } // phase != PH_DONE at entry
    if (RESIDENT) return;
    __syncthreads();
    if (tid == 0 && c.phase_out) c.phase_out[w] = s.phase;
    if (tid == 0 && c.n_windows == 1) {           // the only block is the last: no ticket
        const int active = s.phase != PH_DONE ? 1 : 0;
        sch->running = active;
        sch->round += 1;
        if (c.use_loop) cudaGraphSetConditional(c.loop, active ? 1u : 0u);
    } else if (tid == 0) {
        __threadfence();
        if (s.phase != PH_DONE) atomicAdd(&sch->active, 1);
        if (atomicAdd(&sch->ticket, 1) == c.n_windows - 1) {  // the last block of the round
            __threadfence();
            const int active = atomicAdd(&sch->active, 0);
            sch->running = active;
            sch->active = 0;
            sch->ticket = 0;
            sch->round += 1;
            if (c.use_loop) cudaGraphSetConditional(c.loop, active > 0 ? 1u : 0u);
        }
    }
}

__global__ void __launch_bounds__(CTL_THREADS) k_control(Geom g, CtlArgs c) {
    __shared__ CtlShared sm;
    control_body<false>(g, c, blockIdx.x, sm, c.sch->round & 1);
}


// A polled 64-bit word: the round it announces in the high half, that round's
// jobs in the low half (none: the search has ended).
__device__ __forceinline__ unsigned long long load_acquire(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int32_t load_acquire(const int32_t* p) {
    int32_t v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void store_release(unsigned long long* p, unsigned long long v) {
    // cumulative: the block's writes before its last barrier come with it
    asm volatile("st.release.gpu.global.u64 [%0], %1;" : : "l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void add_release(int32_t* p, int32_t v) {
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" : : "l"(p), "r"(v) : "memory");
}

// Polls for the announcement of `round`, and for the reports of `all` blocks;
// 0 (no jobs) or false after `limit` polls.
__device__ __forceinline__ unsigned long long wait_go(const unsigned long long* go, uint32_t round, int limit) {
    unsigned long long v;
    while ((uint32_t)((v = load_acquire(go)) >> 32) != round)
        if (--limit <= 0) return 0;
    return v;
}
__device__ __forceinline__ bool wait_all(const int32_t* ticket, int32_t all, int limit) {
    while (load_acquire(ticket) != all)
        if (--limit <= 0) return false;
    return true;
}

// Window w's control block of k_search: waits for the `others` evaluating
// blocks and runs the window's control step; the last window's block to finish
// announces the next round (or, with no search left, the end).
template <bool FEW>
__device__ __noinline__ void control_rounds(const Geom& g, const CtlArgs& c, int window, CtlShared& sm, Node* q_mem, int q_cap,
                                            int others) {
    Sched* sch = c.sch;
    const int w = FEW ? window : 0, nw = FEW ? c.n_windows : 1;
    for (int i = threadIdx.x; i < (int)(sizeof(SolveState) / 16); i += blockDim.x)
        reinterpret_cast<int4*>(&sm.s)[i] = reinterpret_cast<const int4*>(c.st_all + w)[i];
    if (threadIdx.x == 0) sm.q_shared = 1;        // empty
    __syncthreads();
    for (uint32_t round = 0;; round++) {
        const int par = (int)(round & 1);
        if (threadIdx.x == 0) {
            const int32_t all = (int32_t)((round + 1) * (uint32_t)others);   // wraps as the count does
            sm.s_stop = !wait_all(&sch->ticket, all, __ldcg(&sch->polls));
        }
        __syncthreads();
        if (sm.s_stop) return;                    // given up: the search stays unfinished
        __syncthreads();
        control_body<true, FEW>(g, c, w, sm, par, q_mem, q_cap);
        __syncthreads();                          // the round's tasks and jobs are written
        const bool done = sm.s.phase == PH_DONE;
        const unsigned long long next = (unsigned long long)(round + 1) << 32;
        if (!FEW) {
            if (threadIdx.x == 0) store_release(&sch->go, next | (done ? 0u : (uint32_t)sm.s_total));
            if (done) return;
            continue;
        }
        if (threadIdx.x == 0) {
            __threadfence();
            if (!done) atomicAdd(&sch->active, 1);
            if (atomicAdd(&sch->controls, 1) == (int32_t)((round + 1) * (uint32_t)nw - 1)) {   // the round's last window
                __threadfence();
                const int active = atomicExch(&sch->active, 0);
                const int jobs = atomicAdd(&sch->n_jobs[par ^ 1], 0);
                sch->running = active;
                sch->n_jobs[par] = 0;             // every block has read its round's count
                store_release(&sch->go, next | (active ? (uint32_t)jobs : 0u));
            }
            sm.s_stop = (uint32_t)wait_go(&sch->go, round + 1, __ldcg(&sch->polls)) == 0;  // given up, or all have ended
        }
        __syncthreads();
        if (sm.s_stop) return;
        __syncthreads();
    }
}

// All rounds of a few windows' searches in one cooperative launch.  Block w runs
// window w's control steps, with its state and queue in shared memory;
// the others evaluate a round's units as k_eval does, count themselves in
// sch->ticket and poll sch->go for the next round.  A search of few events is
// bound by the latency of its rounds, and a round of two graph nodes, the
// loop's condition and a control step that reads and writes its state in L2
// costs about 10 us beside the evaluation.  A kernel of its own for one window
// (FEW false): with the window and their number read at run time its searches
// took 1-5% longer (30,000 events, one interval a round: 3.34 / 3.50 ms).
template <bool FEW>
__global__ void __launch_bounds__(EVAL_THREADS + 32, 2) k_search(const __grid_constant__ Geom g,
                                                                 const __grid_constant__ EvalArgs a,
                                                                 const __grid_constant__ CtlArgs c, int q_cap) {
    extern __shared__ __align__(16) uint32_t tile[];
    __shared__ EvalShared sm;
    __shared__ unsigned long long s_go;
    __shared__ int s_polls;
    Sched* sch = a.sch;
    const int nw = FEW ? c.n_windows : 1;
    if ((int)blockIdx.x < nw) {
        CtlShared& ctl = *reinterpret_cast<CtlShared*>(tile);
        control_rounds<FEW>(g, c, blockIdx.x, ctl, reinterpret_cast<Node*>(&ctl + 1), q_cap, (int)gridDim.x - nw);
        return;
    }
    if (threadIdx.x == 0) {
        clear_tile(tile, eval_tile_words(g));
        sm.over = 0;
        s_go = (unsigned long long)(uint32_t)sch->n_jobs[0];
        s_polls = sch->polls;
    }
    __syncthreads();
    const int block = (int)blockIdx.x - nw, blocks = (int)gridDim.x - nw;
    for (uint32_t round = 0;; round++) {
        const int par = round & 1, n_jobs = (int)(uint32_t)s_go;
        const int slices = round_slices(g, n_jobs), n_units = n_jobs * g.n_tiles * slices;
        if (block == 0 && threadIdx.x == 0) sch->work[par ^ 1] = 0;
        if (block < n_units)
            eval_round(g, a, a.jobs + (size_t)par * a.job_stride, &sch->work[par], n_units, slices, block, blocks, tile, sm);
        __syncthreads();                          // the block's sums are on their way; s_go has been read
        if (threadIdx.x == 0) {
            add_release(&sch->ticket, 1);
            s_go = wait_go(&sch->go, round + 1, s_polls);     // 0 if given up: no more jobs
        }
        __syncthreads();
        if ((uint32_t)s_go == 0) return;
    }
}

CtlArgs control_args(int32_t n_windows, SolveState* st, Node* queues, Task* tasks, int32_t task_stride, Partial* part,
                     const int32_t* err, TraceRec* trace, Job* jobs, int32_t job_stride, Sched* sch,
                     cudaGraphConditionalHandle loop, int32_t use_loop, int32_t split_ok, int32_t* phase_out) {
    CtlArgs c;
    c.n_windows = n_windows;
    c.st_all = st;
    c.queues = queues;
    c.tasks_all = tasks;
    c.task_stride = task_stride;
    c.part_all = part;
    c.err_all = err;
    c.trace = trace;
    c.jobs_all = jobs;
    c.job_stride = job_stride;
    c.sch = sch;
    c.loop = loop;
    c.use_loop = use_loop;
    c.split_ok = split_ok < 0 ? 1 : split_ok;
    c.phase_out = phase_out;
    return c;
}

cudaError_t launch_control(const Geom& g, int32_t n_windows, SolveState* st, Node* queues, Task* tasks,
                           int32_t task_stride, Partial* part, const int32_t* err, TraceRec* trace,
                           Job* jobs, int32_t job_stride, Sched* sch, cudaGraphConditionalHandle loop,
                           int32_t use_loop, cudaStream_t s, int32_t split_ok, int32_t* phase_out) {
    const CtlArgs c = control_args(n_windows, st, queues, tasks, task_stride, part, err, trace, jobs, job_stride, sch,
                                   loop, use_loop, split_ok, phase_out);
    k_control<<<n_windows, CTL_THREADS, 0, s>>>(g, c);
    return cudaGetLastError();
}

// The dynamic shared memory of a k_search block holds the tile and scratch of
// the evaluation or, in the control block, the search's state and as much of
// its queue (two buffers) as fits, up to SEARCH_QUEUE entries.
constexpr int SEARCH_QUEUE = 1024;
static size_t search_smem_bytes(const Geom& g, int threads) {
    const size_t e = eval_smem_bytes(g, threads);
    return e > sizeof(CtlShared) ? e : sizeof(CtlShared);
}
static int search_queue(const Geom& g, int threads) {
    const size_t n = (search_smem_bytes(g, threads) - sizeof(CtlShared)) / (2 * sizeof(Node));
    return n < SEARCH_QUEUE ? (int)n : SEARCH_QUEUE;
}

int search_resident_blocks(const Geom& g, int threads) {
    int per_sm = 0, dev = 0, sms = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return 0;
    int one = 0;
    const size_t bytes = search_smem_bytes(g, threads);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&one, k_search<false>, threads + 32, bytes) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_search<true>, threads + 32, bytes) != cudaSuccess)
        return 0;
    if (one < per_sm) per_sm = one;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return per_sm * sms;
}

cudaError_t launch_search(const Geom& g, const EvalArgs& a, const CtlArgs& c, int threads, int grid_blocks,
                          cudaStream_t s) {
    if (grid_blocks <= c.n_windows) return cudaErrorInvalidValue; // no block would evaluate
    int q_cap = search_queue(g, threads);
    void* args[] = {const_cast<Geom*>(&g), const_cast<EvalArgs*>(&a), const_cast<CtlArgs*>(&c), &q_cap};
    const void* kernel = c.n_windows == 1 ? (const void*)k_search<false> : (const void*)k_search<true>;
    return cudaLaunchCooperativeKernel(kernel, dim3(grid_blocks), dim3(threads + 32), args, search_smem_bytes(g, threads),
                                       s);
}

// Function attributes are per device: the carveout and the dynamic
// shared-memory limit of k_eval and k_search are set on the current device the first time
// it is used, and the limit only ever raised, under one lock (contexts of
// several host threads and devices share these records).
constexpr int SMEM_MAX_DEVICES = 64;
static std::mutex g_smem_mu;
static bool g_carveout[SMEM_MAX_DEVICES];
static int g_smem_bytes[SMEM_MAX_DEVICES];

cudaError_t eval_smem_setup(const Geom& g) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= SMEM_MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_smem_mu);
    if (!g_carveout[dev]) {
        // One shared-memory carveout for every kernel of the library, so that
        // consecutive launches never wait for an L1 / shared reconfiguration.
        const void* fns[] = {(const void*)k_eval, (const void*)k_control, (const void*)k_init,
                             (const void*)k_keys, (const void*)k_search<false>, (const void*)k_search<true>,
                             (const void*)k_ingest_small, (const void*)k_row_hist, (const void*)k_row_scan,
                             (const void*)k_row_scatter};
        for (const void* f : fns) {
            e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     (int)cudaSharedmemCarveoutMaxShared);
            if (e != cudaSuccess) return e;
        }
        g_carveout[dev] = true;
    }
    const int bytes = (int)search_smem_bytes(g, EVAL_THREADS);   // any block size
    if (bytes <= g_smem_bytes[dev]) return cudaSuccess;
    e = cudaFuncSetAttribute(k_eval, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_search<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_search<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) g_smem_bytes[dev] = bytes;
    return e;
}

}  // namespace dd
