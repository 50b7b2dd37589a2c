// Learned warm start: window features, the 128-128-128-2 network (forward,
// backward, Adam), and the kernel that turns a window's features into the
// guess its search starts from.
//
// The paper starts Algorithm 1 from the centre of the domain; this network,
// trained on windows solved exactly, proposes a guess and a half-width
// instead (include/dd.h states the contract).  Everything here is small next
// to the search: the features are one pass over the window's sorted events
// (16 bytes per event), the network 66k multiply-adds per window.  It runs
// on CUDA cores in binary32 with a fixed summation order (each unit adds
// weight * input for inputs 0..127 in turn onto its bias), so a window's
// guess is reproducible bit for bit.
#include "dd_internal.cuh"
#include "../../include/dd.h"

#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include <cuda_bf16.h>

namespace dd {

namespace {

constexpr int P_W1 = 0;
constexpr int P_B1 = P_W1 + MLP_H * FEATURES;
constexpr int P_W2 = P_B1 + MLP_H;
constexpr int P_B2 = P_W2 + MLP_H * MLP_H;
constexpr int P_W3 = P_B2 + MLP_H;
constexpr int P_B3 = P_W3 + MLP_OUT * MLP_H;
constexpr int N_PARAMS = P_B3 + MLP_OUT;
static_assert(N_PARAMS == DD_MLP_PARAMS, "dd.h states the parameter count");
static_assert(FEATURES == DD_MLP_FEATURES && FEATURES == MLP_H, "one thread per feature and per unit");

constexpr float LOG2E = 1.44269504f;

__device__ __forceinline__ float bf(uint16_t b) { return __uint_as_float((uint32_t)b << 16); }

// The 128 bfloat16 weights of one unit as sixteen 16-byte loads, independent of
// one another.  How many are in flight is the compiler's choice: a row is 64
// registers, and the kernels have 98 (k_sample, one sample), 102 (four) and 36
// (k_fwd, k_warm): about one layer's loads, and not half of one's in the last
// two.  The hidden layers' matrices are stored in groups of
// eight inputs, [in / 8][unit][8], so that a warp's load is 512 consecutive
// bytes (with contiguous rows each load touched 32 lines: a gradient of 256
// samples 28.6 us, then 21.6; of 2,048 43.1 and 34.9).  The output layer's two
// rows of 128 are each contiguous (UNITS = 1).
constexpr int IN_GROUP = 8;
__host__ __device__ __forceinline__ int grouped(int unit, int in) {
    return (in / IN_GROUP * MLP_H + unit) * IN_GROUP + in % IN_GROUP;
}
struct Row {
    uint4 q[MLP_H / IN_GROUP];
};
template <int UNITS = MLP_H>
__device__ __forceinline__ Row load_row(const uint16_t* __restrict__ w, int unit) {
    Row r;
#pragma unroll
    for (int k = 0; k < MLP_H / IN_GROUP; k++) {
        const uint4* q = reinterpret_cast<const uint4*>(w) + (UNITS > 1 ? k * UNITS + unit : unit * (MLP_H / IN_GROUP) + k);
        r.q[k] = __ldg(q);
    }
    return r;
}
template <class F>
__device__ __forceinline__ void each_weight(const Row& r, F&& f) {   // f(input, weight) for inputs 0..127 in turn
#pragma unroll
    for (int k = 0; k < MLP_H / 8; k++) {
        const uint32_t w[4] = {r.q[k].x, r.q[k].y, r.q[k].z, r.q[k].w};
#pragma unroll
        for (int i = 0; i < 4; i++) {
            f(8 * k + 2 * i, __uint_as_float(w[i] << 16));
            f(8 * k + 2 * i + 1, __uint_as_float(w[i] & 0xffff0000u));
        }
    }
}

// A dense layer's unit for S samples x[s][in] in shared memory: weight * input
// for inputs 0..127 in turn onto the bias.
template <int S>
__device__ __forceinline__ void unit(const Row& w, float bias, const float (*x)[MLP_H], float (&acc)[S]) {
#pragma unroll
    for (int s = 0; s < S; s++) acc[s] = bias;
    each_weight(w, [&](int k, float v) {
#pragma unroll
        for (int s = 0; s < S; s++) acc[s] = __fadd_rn(acc[s], __fmul_rn(v, x[s][k]));
    });
}

// The forward pass of S samples by a block of 128 threads; x, h1, h2 and out
// in shared memory.  Both hidden layers' weights are asked for before the first
// layer, the output layer's (and, `ahead` of it, what the caller needs next)
// before the second, so that loads may run ahead of the layer that uses them.
// Every thread returns after the last barrier.
template <int S, class Ahead>
__device__ __forceinline__ void forward(const MlpDev& m, const float (*x)[MLP_H], float (*h1)[MLP_H], float (*h2)[MLP_H],
                                        float (*out)[MLP_OUT], Ahead&& ahead) {
    const int j = threadIdx.x;
    float a[S];
    const Row w1 = load_row(m.w1, j), w2 = load_row(m.w2, j);
    const float b1 = m.b1[j], b2 = m.b2[j];
    unit<S>(w1, b1, x, a);
#pragma unroll
    for (int s = 0; s < S; s++) h1[s][j] = a[s] > 0.0f ? a[s] : 0.0f;
    const Row w3 = load_row<1>(m.w3, j % MLP_OUT);
    __syncthreads();
    unit<S>(w2, b2, h1, a);
    ahead();
#pragma unroll
    for (int s = 0; s < S; s++) h2[s][j] = a[s] > 0.0f ? a[s] : 0.0f;
    __syncthreads();
    if (j < MLP_OUT * S) {
        const int o = j % MLP_OUT;
        float v[1];
        unit<1>(w3, m.b3[o], h2 + j / MLP_OUT, v);
        out[j / MLP_OUT][o] = v[0];
    }
    __syncthreads();
}

// ------------------------------------------------------------ features

constexpr int FEAT_THREADS = 256;

// Block c counts chunk c of its window's sorted events into the window's
// 16 x 8 bins (radial bin from the squared distance to the FOE relative to
// the farthest corner pixel centre; temporal bin from (t - t0)/tau).
__global__ void __launch_bounds__(FEAT_THREADS) k_features(Geom g, const WinIn* __restrict__ wins,
                                                           const int32_t* __restrict__ chunk_win,
                                                           const Ev* __restrict__ ev, int32_t* counts) {
    __shared__ int32_t h[FEATURES];
    for (int k = threadIdx.x; k < FEATURES; k += blockDim.x) h[k] = 0;
    __syncthreads();
    const int w = chunk_win[blockIdx.x];
    const WinIn win = wins[w];
    const float ax = g.fx, bx = __fsub_rn((float)(g.W - 1), g.fx);
    const float ay = g.fy, by = __fsub_rn((float)(g.H - 1), g.fy);
    const float cx = ax > bx ? ax : bx, cy = ay > by ? ay : by;
    const float R2 = __fadd_rn(__fmul_rn(cx, cx), __fmul_rn(cy, cy));
    const float tsc = __fdiv_rn((float)FEAT_T, win.tau);
    const int64_t i0 = (int64_t)(blockIdx.x - win.chunk0) * CHUNK, i1 = min(win.n, i0 + CHUNK);
    const Ev* e = ev + win.ev_off;
    for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        const Ev v = e[i];
        const float dx = v.dx, dy = v.dy;
        const float r2 = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
        const float u = R2 > 0.0f ? __fdiv_rn(r2, R2) : 0.0f;
        int rb = (int)floorf(__fmul_rn(__fsqrt_rn(u), (float)FEAT_R));
        rb = rb > FEAT_R - 1 ? FEAT_R - 1 : rb;
        int tb = (int)floorf(__fmul_rn(v.t, tsc));
        tb = tb < 0 ? 0 : (tb > FEAT_T - 1 ? FEAT_T - 1 : tb);
        atomicAdd(&h[rb * FEAT_T + tb], 1);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < FEATURES; k += blockDim.x)
        if (h[k]) atomicAdd(&counts[(size_t)w * FEATURES + k], h[k]);
}

// Block w: if window w asks for the model's warm start, its features, the
// network, and the guess and half-width written into its search parameters.
__global__ void __launch_bounds__(MLP_H) k_warm(int32_t n_windows, const int32_t* __restrict__ counts,
                                                const WinIn* __restrict__ wins, WinParams* params, MlpDev m) {
    __shared__ __align__(16) float x[1][FEATURES], h1[1][MLP_H], h2[1][MLP_H];
    __shared__ float out[1][MLP_OUT];
    const int w = blockIdx.x;
    if (w >= n_windows || params[w].warm != DD_WARM_MODEL) return;
    const int j = threadIdx.x;
    const int64_t n = wins[w].n;
    x[0][j] = n > 0 ? __fdiv_rn((float)(counts[(size_t)w * FEATURES + j] * FEATURES), (float)n) : 0.0f;
    __syncthreads();
    forward<1>(m, x, h1, h2, out, [] {});
    if (j == 0) {
        const float tau = wins[w].tau;
        float v = __fadd_rn(__fmul_rn(out[0][1], LOG2E), 0.5f);
        if (!(v >= -20.0f)) v = -20.0f;
        if (v > 1.0f) v = 1.0f;
        const int e = (int)floorf(v);
        params[w].D_warm = __fdiv_rn(out[0][0], tau);
        params[w].w_warm = __fdiv_rn(__uint_as_float((uint32_t)(e + 127) << 23), tau);
        params[w].warm = 1;
    }
}

// feat[w][k] = 128 counts[w][k] / n_w, as the warm-start kernel forms its input.
__global__ void __launch_bounds__(FEATURES) k_feature_norm(const int32_t* __restrict__ counts,
                                                           const WinIn* __restrict__ wins, float* feat) {
    const int w = blockIdx.x, j = threadIdx.x;
    const int64_t n = wins[w].n;
    feat[(size_t)w * FEATURES + j] =
        n > 0 ? __fdiv_rn((float)(counts[(size_t)w * FEATURES + j] * FEATURES), (float)n) : 0.0f;
}

// -------------------------------------------------------------- training

// Block b: the outputs of sample b.
__global__ void __launch_bounds__(MLP_H) k_fwd(MlpDev m, const float* __restrict__ X, float* outg) {
    __shared__ __align__(16) float x[1][FEATURES], h1[1][MLP_H], h2[1][MLP_H];
    __shared__ float out[1][MLP_OUT];
    const int b = blockIdx.x, j = threadIdx.x;
    x[0][j] = X[(size_t)b * FEATURES + j];
    __syncthreads();
    forward<1>(m, x, h1, h2, out, [] {});
    if (j < MLP_OUT) outg[(size_t)b * MLP_OUT + j] = out[0][j];
}

// What the weight gradients need of every sample, and its loss.
struct Acts {
    float *h1, *h2, *g1, *g2;    // [B][128]
    float *gout;                 // [B][2]
    float *loss;                 // [B]
};

// Block b: forward and backward pass of samples S b .. S b + S - 1: the hidden
// activations, the loss and its gradient with respect to the outputs and to
// the hidden units (through the ReLUs, with the bfloat16 weights).
// A sample's gradient depends on the others only through 1/B.  One sample a
// block while that fits one wave of the device, else SAMPLES, which share the
// weights' loads (1,684 samples: the four-launch form 208 us in all).
constexpr int SAMPLES = 4;
template <int S>
__global__ void __launch_bounds__(MLP_H) k_sample(MlpDev m, const uint16_t* __restrict__ w2t, int32_t B,
                                                  const float* __restrict__ X, const float* __restrict__ u_star,
                                                  Acts a) {
    __shared__ __align__(16) float x[S][FEATURES], h1[S][MLP_H], h2[S][MLP_H], g2[S][MLP_H];
    __shared__ float out[S][MLP_OUT], go[S][MLP_OUT];
    const int b0 = S * blockIdx.x, k = threadIdx.x;
#pragma unroll
    for (int s = 0; s < S; s++) x[s][k] = b0 + s < B ? X[(size_t)(b0 + s) * FEATURES + k] : 0.0f;
    __syncthreads();
    Row wk;                                       // of hidden unit k to each unit of the next layer
    forward<S>(m, x, h1, h2, out, [&] { wk = load_row(w2t, k); });
    if (k < S && b0 + k < B) {
        const float inv = 1.0f / (float)B;
        const float u = out[k][0], l = out[k][1];
        const float e = u_star[b0 + k] - u;
        const float q = 9.0f * expf(-2.0f * l);
        a.loss[b0 + k] = 0.5f * q * e * e + l;
        go[k][0] = -q * e * inv;
        go[k][1] = (1.0f - q * e * e) * inv;
        a.gout[2 * (size_t)(b0 + k)] = go[k][0];
        a.gout[2 * (size_t)(b0 + k) + 1] = go[k][1];
    }
    __syncthreads();
    const float wa = bf(m.w3[k]), wb = bf(m.w3[MLP_H + k]);
#pragma unroll
    for (int s = 0; s < S; s++) {
        if (b0 + s >= B) break;
        const float v = h2[s][k] > 0.0f ? wa * go[s][0] + wb * go[s][1] : 0.0f;
        g2[s][k] = v;
        a.g2[(size_t)(b0 + s) * MLP_H + k] = v;
        a.h1[(size_t)(b0 + s) * MLP_H + k] = h1[s][k];
        a.h2[(size_t)(b0 + s) * MLP_H + k] = h2[s][k];
    }
    __syncthreads();
    float acc[S][2] = {};                         // even and odd units
    each_weight(wk, [&](int j, float v) {
#pragma unroll
        for (int s = 0; s < S; s++) acc[s][j & 1] = __fmaf_rn(v, g2[s][j], acc[s][j & 1]);
    });
#pragma unroll
    for (int s = 0; s < S; s++)
        if (b0 + s < B) a.g1[(size_t)(b0 + s) * MLP_H + k] = h1[s][k] > 0.0f ? acc[s][0] + acc[s][1] : 0.0f;
}

// Weight gradients of WG_CHUNK samples (blockIdx.y): blocks 0-15 and 16-31 a
// 32 x 32 tile of the first two layers (four outputs a thread), blocks 32-35
// 32 columns of the output layer and of the biases, block 36, once, the mean
// loss.  Every block first stages its operands in shared memory, all loads in
// flight at once, so it waits for memory once; one block for the output layer
// and all biases that read memory sample by sample took 7 us longer than the
// tiles (gradient of 256 samples 21.6 -> 14.6 us, of 2,048 34.9 -> 28.8).
// Each chunk writes its own partial gradient; they are added in order
// (k_wsum), so the result does not depend on the launch.  With one thread per
// parameter over the whole batch in turn, the chain of B loads and additions
// was most of a training step (256 samples: 45 us in all).
constexpr int WG_CHUNK = 64, WG_TILE = 32, WG_THREADS = 256, WG_COLS = MLP_H / WG_TILE;
constexpr int WG_TILES = 2 * WG_COLS * WG_COLS;
__global__ void __launch_bounds__(WG_THREADS) k_wgrad(int32_t B, const float* __restrict__ X, Acts a, float* part,
                                                      float* loss) {
    __shared__ __align__(16) float G[WG_CHUNK][WG_TILE];
    __shared__ float A[WG_CHUNK][WG_TILE], G1[WG_CHUNK][WG_TILE], go[WG_CHUNK][MLP_OUT];
    const int t = threadIdx.x, b0 = blockIdx.y * WG_CHUNK, n = min(WG_CHUNK, B - b0);
    float* out = part + (size_t)blockIdx.y * N_PARAMS;
    if (blockIdx.x < WG_TILES) {
        const int tile = blockIdx.x % (WG_TILES / 2), j0 = tile / 4 * WG_TILE, i0 = tile % 4 * WG_TILE;
        const bool first = blockIdx.x < WG_TILES / 2;
        const float* g = (first ? a.g1 : a.g2) + (size_t)b0 * MLP_H + j0;
        const float* v = (first ? X : a.h1) + (size_t)b0 * MLP_H + i0;
#pragma unroll
        for (int q = 0; q < WG_CHUNK * WG_TILE / WG_THREADS; q++) {
            const int r = t / WG_TILE + q * (WG_THREADS / WG_TILE), c = t % WG_TILE;
            G[r][c] = r < n ? g[(size_t)r * MLP_H + c] : 0.0f;
            A[r][c] = r < n ? v[(size_t)r * MLP_H + c] : 0.0f;
        }
        __syncthreads();
        const int i = t % WG_TILE, j = 4 * (t / WG_TILE);
        float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, s3 = 0.0f;
#pragma unroll 16
        for (int r = 0; r < WG_CHUNK; r++) {
            const float4 q = *reinterpret_cast<const float4*>(&G[r][j]);
            const float x = A[r][i];
            s0 = __fmaf_rn(q.x, x, s0);
            s1 = __fmaf_rn(q.y, x, s1);
            s2 = __fmaf_rn(q.z, x, s2);
            s3 = __fmaf_rn(q.w, x, s3);
        }
        float* o = out + (first ? P_W1 : P_W2) + (size_t)(j0 + j) * MLP_H + i0 + i;
        o[0] = s0;
        o[MLP_H] = s1;
        o[2 * MLP_H] = s2;
        o[3 * MLP_H] = s3;
        return;
    }
    if (blockIdx.x == WG_TILES + WG_COLS) {       // the mean loss, summed in a fixed order
        if (blockIdx.y || !loss) return;
        float* sum = &A[0][0];
        float acc = 0.0f;
        for (int b = t; b < B; b += WG_THREADS) acc += a.loss[b];
        sum[t] = acc;
        __syncthreads();
        for (int o = WG_THREADS / 2; o > 0; o >>= 1) {
            if (t < o) sum[t] += sum[t + o];
            __syncthreads();
        }
        if (t == 0) *loss = sum[0] * (1.0f / (float)B);
        return;
    }
    // 32 columns of W3 [2][128] and of both hidden biases; b3
    const int i0 = (blockIdx.x - WG_TILES) * WG_TILE;
#pragma unroll
    for (int q = 0; q < WG_CHUNK * WG_TILE / WG_THREADS; q++) {
        const int r = t / WG_TILE + q * (WG_THREADS / WG_TILE), c = t % WG_TILE;
        const size_t k = (size_t)(b0 + r) * MLP_H + i0 + c;
        A[r][c] = r < n ? a.h2[k] : 0.0f;
        G1[r][c] = r < n ? a.g1[k] : 0.0f;
        G[r][c] = r < n ? a.g2[k] : 0.0f;
    }
    if (t < MLP_OUT * n) go[t / MLP_OUT][t % MLP_OUT] = a.gout[MLP_OUT * (size_t)b0 + t];
    __syncthreads();
    const int i = t % WG_TILE, o = t / WG_TILE % 2;
    float s = 0.0f;
    if (t < 2 * WG_TILE) {
#pragma unroll 16
        for (int r = 0; r < n; r++) s = __fmaf_rn(go[r][o], A[r][i], s);
        out[P_W3 + o * MLP_H + i0 + i] = s;
    } else if (t < 4 * WG_TILE) {
#pragma unroll 16
        for (int r = 0; r < n; r++) s += o ? G[r][i] : G1[r][i];
        out[(o ? P_B2 : P_B1) + i0 + i] = s;
    } else if (t < 4 * WG_TILE + MLP_OUT && i0 == 0) {
        for (int r = 0; r < n; r++) s += go[r][i];
        out[P_B3 + i] = s;
    }
}

// The chunks' partial gradients added in order.
__global__ void __launch_bounds__(256) k_wsum(int32_t chunks, const float* __restrict__ part, float* grad) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N_PARAMS) return;
    float acc = 0.0f;
#pragma unroll 8
    for (int c = 0; c < chunks; c++) acc += part[(size_t)c * N_PARAMS + p];
    grad[p] = acc;
}

__device__ __forceinline__ bool is_weight(int p, int* layer, int* o, int* i) {
    if (p < P_B1) { *layer = 0; *o = p / FEATURES; *i = p % FEATURES; return true; }
    if (p >= P_W2 && p < P_B2) { *layer = 1; *o = (p - P_W2) / MLP_H; *i = (p - P_W2) % MLP_H; return true; }
    if (p >= P_W3 && p < P_B3) { *layer = 2; *o = (p - P_W3) / MLP_H; *i = (p - P_W3) % MLP_H; return true; }
    return false;
}

struct Weights {
    uint16_t *w1, *w2, *w3;      // w1, w2 grouped; w3 [out][in]
    uint16_t* w2t;               // w2 transposed, grouped, for the backward pass
};

__device__ __forceinline__ void store_weight(const Weights& wb, int layer, int o, int i, float v) {
    const uint16_t h = __bfloat16_as_ushort(__float2bfloat16_rn(v));
    if (layer == 0) wb.w1[grouped(o, i)] = h;
    else if (layer == 1) { wb.w2[grouped(o, i)] = h; wb.w2t[grouped(i, o)] = h; }
    else wb.w3[o * MLP_H + i] = h;
}

// One thread per parameter: an Adam step on the binary32 master value
// (lr_t carries the bias corrections), then the bfloat16 copies.
__global__ void __launch_bounds__(256) k_adam(float lr_t, const float* __restrict__ grad, float* master, float* mom,
                                              float* vel, Weights wb) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N_PARAMS) return;
    const float g = grad[p];
    const float m1 = 0.9f * mom[p] + 0.1f * g;
    const float v1 = 0.999f * vel[p] + 0.001f * g * g;
    mom[p] = m1;
    vel[p] = v1;
    const float v = master[p] - lr_t * m1 / (sqrtf(v1) + 1e-8f);
    master[p] = v;
    int layer, o, i;
    if (is_weight(p, &layer, &o, &i)) store_weight(wb, layer, o, i, v);
}

// bfloat16 copies of the master weights; with `export_` non-null also the
// parameters as the network evaluates them.
__global__ void __launch_bounds__(256) k_sync(const float* __restrict__ master, Weights wb, float* export_) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N_PARAMS) return;
    const float v = master[p];
    int layer, o, i;
    const bool w = is_weight(p, &layer, &o, &i);
    if (w) store_weight(wb, layer, o, i, v);
    if (export_) export_[p] = w ? __bfloat162float(__float2bfloat16_rn(v)) : v;
}

}  // namespace

cudaError_t launch_features(const Geom& g, const WinIn* wins, const int32_t* chunk_win, int32_t n_chunks,
                            const Ev* ev, int32_t* counts, cudaStream_t s) {
    if (n_chunks <= 0) return cudaSuccess;
    k_features<<<n_chunks, FEAT_THREADS, 0, s>>>(g, wins, chunk_win, ev, counts);
    return cudaGetLastError();
}

cudaError_t launch_feature_norm(int32_t n_windows, const int32_t* counts, const WinIn* wins, float* feat,
                                cudaStream_t s) {
    if (n_windows <= 0) return cudaSuccess;
    k_feature_norm<<<n_windows, FEATURES, 0, s>>>(counts, wins, feat);
    return cudaGetLastError();
}

cudaError_t launch_warm(const Geom& g, int32_t n_windows, const int32_t* counts, const WinIn* wins,
                        WinParams* params, const MlpDev& m, cudaStream_t s) {
    (void)g;
    if (n_windows <= 0) return cudaSuccess;
    k_warm<<<n_windows, MLP_H, 0, s>>>(n_windows, counts, wins, params, m);
    return cudaGetLastError();
}

}  // namespace dd

// ------------------------------------------------------------------ model

struct dd_mlp {
    int device = 0;
    cudaStream_t stream = nullptr;
    float* master = nullptr;        // binary32 parameters ([out][in] matrices)
    float* mom = nullptr;           // Adam moments
    float* vel = nullptr;
    float* grad = nullptr;
    float* exp = nullptr;           // export buffer (get_params)
    float* loss = nullptr;
    dd::Weights wb{};
    int64_t step = 0;
    // training activations for up to cap samples
    int32_t cap = 0;
    dd::Acts act{};
    float* part = nullptr;          // partial gradients per chunk of samples
};

namespace {

constexpr int NP = DD_MLP_PARAMS;
constexpr int B_MAX = 4096;
constexpr int ONE_SAMPLE_MAX = 608;   // samples up to which each has a block of its own (four per SM)

template <class T>
void release(T*& p) {
    if (p) cudaFree(p);
    p = nullptr;
}

int chunks_of(int32_t B) { return (B + dd::WG_CHUNK - 1) / dd::WG_CHUNK; }

void free_acts(dd_mlp* m) {
    release(m->act.h1);
    release(m->act.h2);
    release(m->act.g1);
    release(m->act.g2);
    release(m->act.gout);
    release(m->act.loss);
    release(m->part);
    m->cap = 0;
}

int ensure_acts(dd_mlp* m, int32_t B) {
    if (B <= m->cap) return DD_OK;
    free_acts(m);
    const size_t n = (size_t)B;
    if (cudaMalloc((void**)&m->act.h1, sizeof(float) * n * dd::MLP_H) != cudaSuccess ||
        cudaMalloc((void**)&m->act.h2, sizeof(float) * n * dd::MLP_H) != cudaSuccess ||
        cudaMalloc((void**)&m->act.g1, sizeof(float) * n * dd::MLP_H) != cudaSuccess ||
        cudaMalloc((void**)&m->act.g2, sizeof(float) * n * dd::MLP_H) != cudaSuccess ||
        cudaMalloc((void**)&m->act.gout, sizeof(float) * n * dd::MLP_OUT) != cudaSuccess ||
        cudaMalloc((void**)&m->act.loss, sizeof(float) * n) != cudaSuccess ||
        cudaMalloc((void**)&m->part, sizeof(float) * (size_t)chunks_of(B) * NP) != cudaSuccess) {
        free_acts(m);
        return DD_ERR_OOM;
    }
    m->cap = B;
    return DD_OK;
}

dd::MlpDev view(const dd_mlp* m) {
    dd::MlpDev v;
    v.w1 = m->wb.w1;
    v.w2 = m->wb.w2;
    v.w3 = m->wb.w3;
    v.b1 = m->master + dd::P_B1;
    v.b2 = m->master + dd::P_B2;
    v.b3 = m->master + dd::P_B3;
    return v;
}

int sync_weights(dd_mlp* m, float* export_) {
    dd::k_sync<<<(NP + 255) / 256, 256, 0, m->stream>>>(m->master, m->wb, export_);
    return cudaGetLastError() == cudaSuccess ? DD_OK : DD_ERR_CUDA;
}

void destroy(dd_mlp* m) {
    release(m->master);
    release(m->mom);
    release(m->vel);
    release(m->grad);
    release(m->exp);
    release(m->loss);
    release(m->wb.w1);
    release(m->wb.w2);
    release(m->wb.w3);
    release(m->wb.w2t);
    free_acts(m);
    delete m;
}

// SplitMix64 (Steele, Lea and Flood, OOPSLA 2014) for the initial weights.
uint64_t splitmix(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

int upload(dd_mlp* m, const float* host) {
    if (cudaMemcpyAsync(m->master, host, sizeof(float) * NP, cudaMemcpyHostToDevice, m->stream) != cudaSuccess ||
        cudaMemsetAsync(m->mom, 0, sizeof(float) * NP, m->stream) != cudaSuccess ||
        cudaMemsetAsync(m->vel, 0, sizeof(float) * NP, m->stream) != cudaSuccess)
        return DD_ERR_CUDA;
    int rc = sync_weights(m, nullptr);
    if (rc) return rc;
    return cudaStreamSynchronize(m->stream) == cudaSuccess ? DD_OK : DD_ERR_CUDA;
}

int grad_impl(dd_mlp* m, const float* X, const float* u_star, int32_t B, float* grad, float* loss) {
    if (B < 1 || B > B_MAX || !X || !u_star || !grad) return DD_ERR_ARG;
    int rc = ensure_acts(m, B);
    if (rc) return rc;
    const dd::MlpDev v = view(m);
    if (B <= ONE_SAMPLE_MAX)
        dd::k_sample<1><<<B, dd::MLP_H, 0, m->stream>>>(v, m->wb.w2t, B, X, u_star, m->act);
    else
        dd::k_sample<dd::SAMPLES><<<(B + dd::SAMPLES - 1) / dd::SAMPLES, dd::MLP_H, 0, m->stream>>>(
            v, m->wb.w2t, B, X, u_star, m->act);
    const int chunks = chunks_of(B);
    float* part = chunks == 1 ? grad : m->part;
    dd::k_wgrad<<<dim3(dd::WG_TILES + dd::WG_COLS + 1, chunks), dd::WG_THREADS, 0, m->stream>>>(B, X, m->act, part, loss);
    if (chunks > 1) dd::k_wsum<<<(NP + 255) / 256, 256, 0, m->stream>>>(chunks, m->part, grad);
    return cudaGetLastError() == cudaSuccess ? DD_OK : DD_ERR_CUDA;
}

}  // namespace

namespace dd {
bool mlp_device_view(const ::dd_mlp* m, MlpDev* out, int* device) {
    if (!m) return false;
    *out = view(m);
    *device = m->device;
    return true;
}
}  // namespace dd

extern "C" {

int dd_mlp_create(uint64_t seed, dd_mlp** out) {
    if (!out) return DD_ERR_ARG;
    int dev = 0;
    cudaDeviceProp prop;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceProperties(&prop, dev) != cudaSuccess ||
        !(prop.major == 10 && prop.minor == 3))
        return DD_ERR_NO_DEVICE;
    dd_mlp* m = new (std::nothrow) dd_mlp();
    if (!m) return DD_ERR_OOM;
    m->device = dev;
    bool ok = cudaMalloc((void**)&m->master, sizeof(float) * NP) == cudaSuccess &&
              cudaMalloc((void**)&m->mom, sizeof(float) * NP) == cudaSuccess &&
              cudaMalloc((void**)&m->vel, sizeof(float) * NP) == cudaSuccess &&
              cudaMalloc((void**)&m->grad, sizeof(float) * NP) == cudaSuccess &&
              cudaMalloc((void**)&m->exp, sizeof(float) * NP) == cudaSuccess &&
              cudaMalloc((void**)&m->loss, sizeof(float)) == cudaSuccess &&
              cudaMalloc((void**)&m->wb.w1, 2 * dd::MLP_H * dd::FEATURES) == cudaSuccess &&
              cudaMalloc((void**)&m->wb.w2, 2 * dd::MLP_H * dd::MLP_H) == cudaSuccess &&
              cudaMalloc((void**)&m->wb.w2t, 2 * dd::MLP_H * dd::MLP_H) == cudaSuccess &&
              cudaMalloc((void**)&m->wb.w3, 2 * dd::MLP_OUT * dd::MLP_H) == cudaSuccess;
    if (!ok) {
        destroy(m);
        return DD_ERR_OOM;
    }
    // Uniform in +-sqrt(6 / fan_in) (fan_in = 128 for every layer); biases 0,
    // except the log half-width's, which starts at log(0.05).
    std::vector<float> p(NP, 0.0f);
    uint64_t s = seed;
    const float a = std::sqrt(6.0f / 128.0f);
    for (int i = 0; i < NP; i++) {
        const bool bias = (i >= dd::P_B1 && i < dd::P_W2) || (i >= dd::P_B2 && i < dd::P_W3) || i >= dd::P_B3;
        if (bias) continue;
        const float u = (float)(splitmix(s) >> 40) * (1.0f / 16777216.0f);
        p[i] = (2.0f * u - 1.0f) * a;
    }
    p[dd::P_B3 + 1] = std::log(0.05f);
    const int rc = upload(m, p.data());
    if (rc) {
        destroy(m);
        return rc;
    }
    *out = m;
    return DD_OK;
}

void dd_mlp_destroy(dd_mlp* m) {
    if (m) destroy(m);
}

int dd_mlp_set_stream(dd_mlp* m, void* stream) {
    if (!m) return DD_ERR_ARG;
    m->stream = (cudaStream_t)stream;
    return DD_OK;
}

int dd_mlp_get_params(dd_mlp* m, float* params, int64_t n) {
    if (!m || !params || n != NP) return DD_ERR_ARG;
    int rc = sync_weights(m, m->exp);
    if (rc) return rc;
    if (cudaMemcpyAsync(params, m->exp, sizeof(float) * NP, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
        cudaStreamSynchronize(m->stream) != cudaSuccess)
        return DD_ERR_CUDA;
    return DD_OK;
}

int dd_mlp_set_params(dd_mlp* m, const float* params, int64_t n) {
    if (!m || !params || n != NP) return DD_ERR_ARG;
    for (int64_t i = 0; i < n; i++)
        if (!std::isfinite(params[i])) return DD_ERR_ARG;
    m->step = 0;
    return upload(m, params);
}

int dd_mlp_save(dd_mlp* m, const char* path) {
    if (!m || !path) return DD_ERR_ARG;
    std::vector<float> p(NP);
    if (cudaMemcpyAsync(p.data(), m->master, sizeof(float) * NP, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
        cudaStreamSynchronize(m->stream) != cudaSuccess)
        return DD_ERR_CUDA;
    unsigned char hdr[32];
    std::memset(hdr, 0, sizeof(hdr));
    std::memcpy(hdr, "DDMLP001", 8);
    const int64_t np = NP, st = m->step;
    std::memcpy(hdr + 8, &np, 8);
    std::memcpy(hdr + 16, &st, 8);
    FILE* f = std::fopen(path, "wb");
    if (!f) return DD_ERR_ARG;
    const bool ok = std::fwrite(hdr, 1, 32, f) == 32 && std::fwrite(p.data(), sizeof(float), NP, f) == (size_t)NP;
    return (std::fclose(f) == 0 && ok) ? DD_OK : DD_ERR_ARG;
}

int dd_mlp_load(dd_mlp* m, const char* path) {
    if (!m || !path) return DD_ERR_ARG;
    FILE* f = std::fopen(path, "rb");
    if (!f) return DD_ERR_ARG;
    unsigned char hdr[32];
    std::vector<float> p(NP);
    bool ok = std::fread(hdr, 1, 32, f) == 32;
    int64_t np = 0, st = 0;
    if (ok) {
        std::memcpy(&np, hdr + 8, 8);
        std::memcpy(&st, hdr + 16, 8);
        ok = std::memcmp(hdr, "DDMLP001", 8) == 0 && np == NP &&
             std::fread(p.data(), sizeof(float), NP, f) == (size_t)NP;
    }
    std::fclose(f);
    if (!ok) return DD_ERR_ARG;
    for (float v : p)
        if (!std::isfinite(v)) return DD_ERR_ARG;
    const int rc = upload(m, p.data());
    if (rc == DD_OK) m->step = st;
    return rc;
}

int dd_mlp_forward(dd_mlp* m, const float* X, int32_t B, float* out) {
    if (!m || B < 0 || (B > 0 && (!X || !out))) return DD_ERR_ARG;
    if (B == 0) return DD_OK;
    dd::k_fwd<<<B, dd::MLP_H, 0, m->stream>>>(view(m), X, out);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(m->stream) != cudaSuccess) return DD_ERR_CUDA;
    return DD_OK;
}

int dd_mlp_grad(dd_mlp* m, const float* X, const float* u_star, int32_t B, float* grad, float* loss) {
    if (!m || !loss) return DD_ERR_ARG;
    return grad_impl(m, X, u_star, B, grad, loss);
}

int dd_mlp_train_step(dd_mlp* m, const float* X, const float* u_star, int32_t B, float lr, float* loss) {
    if (!m || !std::isfinite(lr) || !(lr > 0.0f)) return DD_ERR_ARG;
    int rc = grad_impl(m, X, u_star, B, m->grad, loss);
    if (rc) return rc;
    m->step++;
    const double t = (double)m->step;
    const float lr_t = (float)(lr * std::sqrt(1.0 - std::pow(0.999, t)) / (1.0 - std::pow(0.9, t)));
    dd::k_adam<<<(NP + 255) / 256, 256, 0, m->stream>>>(lr_t, m->grad, m->master, m->mom, m->vel, m->wb);
    return cudaGetLastError() == cudaSuccess ? DD_OK : DD_ERR_CUDA;
}

}  // extern "C"
