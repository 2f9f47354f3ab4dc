// Cost model of the variant tuner: a 3-layer MLP (tanh, tanh, linear) with its forward pass,
// back-propagation and Adam update as hand-written FP32 CUDA kernels.
//
// The network is small (input ~30 features, width 64, a few thousand samples), so each
// kernel gives one thread one output element and loops over the reduction index in a fixed
// order: deterministic results, no atomics.  The weight gradients sum over the samples in two
// fixed-order levels: chunks of kChunk samples in parallel, then the chunk partials in order.
//
// Flat parameter layout: W1 (H x d, row-major), b1 (H), W2 (H x H), b2 (H), W3 (1 x H), b3 (1).
// Workspace for n samples (floats): h1 (n H), h2 (n H), y (n), dy (n), dz2 (n H), dz1 (n H),
// grad (P), loss (1), the Adam step counter (one int), small networks: what rounding left out of
// the parameters (P), the weight-gradient chunk partials
// (ceil(n / kChunk) x H x (max(d, H) + 1)) or, for small networks, the CTAs' gradients and losses.
//
// Networks of at most 64 inputs and 64 hidden units (the cost model's) train in two launches per
// epoch: mlp_tile_kernel takes tiles of 32 samples through forward pass, loss and
// back-propagation in shared memory and leaves each CTA's weight gradients; mlp_update_kernel sums
// them in CTA order and applies Adam.  The thirteen launches of the general kernels took 174 us an
// epoch (4200 records, 35 inputs, width 64), most of it in gathers and launches; the two take
// about 9.  The general kernels serve wider networks.
//
// There training replays captured epochs: the Adam step number lives in the workspace (the loss
// kernel advances it, the Adam kernel derives its bias corrections from it), so one epoch's
// launches are the same every epoch and a CUDA graph of kEpochsPerGraph epochs is replayed.
#include <math.h>
#include <string.h>

#include "../../include/hydro.h"
#include "hydro_internal.h"

namespace {

constexpr int kThreads = 256;
constexpr int kChunk = 128;  // samples per partial sum of the weight gradients

constexpr int kEpochsPerGraph = 16;

struct Sizes {
    long long P, h1, h2, y, dy, dz2, dz1, grad, loss, stepc, rest, part, total;  // float offsets
};

constexpr int kSmall = 64;       // most inputs and hidden units of the two-launch epoch
constexpr int kTile = 32;        // samples of a tile
constexpr int kTileCtas = 152;   // most CTAs of the tile kernel (one per SM of a GB300)
constexpr int kRow = kTile + 4;  // floats of a shared row of a tile (rows on distinct banks)
constexpr int kWRow = kSmall + 1;  // and of a weight matrix (its transposing stores conflict-free)

bool small_net(int d, int H) { return d <= kSmall && H <= kSmall; }
long long tile_ctas(long long n) {
    const long long t = (n + kTile - 1) / kTile;
    return t < kTileCtas ? t : kTileCtas;
}

Sizes sizes(int d, int H, long long n) {
    Sizes S;
    S.P = (long long)H * d + H + (long long)H * H + H + H + 1;
    long long o = 0;
    S.h1 = o; o += n * H;
    S.h2 = o; o += n * H;
    S.y = o; o += n;
    S.dy = o; o += n;
    S.dz2 = o; o += n * H;
    S.dz1 = o; o += n * H;
    S.grad = o; o += S.P;
    S.loss = o; o += 1;
    S.stepc = o; o += 1;
    S.rest = o; o += small_net(d, H) ? S.P : 0;
    S.part = o;
    const long long chunks = (n + kChunk - 1) / kChunk * (long long)H * ((d > H ? d : H) + 1);
    const long long tiles = small_net(d, H) ? tile_ctas(n) * (S.P + 1) : 0;
    o += chunks > tiles ? chunks : tiles;
    S.total = o;
    return S;
}

// out[s][j] = act(b[j] + sum_i in[s][i] W[j][i])
template <bool TANH>
__global__ void __launch_bounds__(kThreads) dense_forward(const float *in, int din, const float *W,
                                                          const float *b, int dout, long long n,
                                                          float *out) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * dout) return;
    const long long s = idx / dout;
    const int j = (int)(idx % dout);
    float acc = b[j];
    for (int i = 0; i < din; ++i) acc = fmaf(in[s * din + i], W[(long long)j * din + i], acc);
    out[idx] = TANH ? tanhf(acc) : acc;
}

// dy[s] = 2 (y[s] - t[s]) / n; loss = (1/n) sum_s (y[s] - t[s])^2 (one CTA, fixed order).
// Training (stepc non-null): also record the loss in hist[*stepc - step0] and advance the Adam
// step counter *stepc, which the Adam kernel of the same epoch reads.
__global__ void __launch_bounds__(kThreads) mse_kernel(const float *y, const float *t, long long n,
                                                       float *dy, float *loss, int *stepc = nullptr,
                                                       int step0 = 0, float *hist = nullptr) {
    __shared__ float s[kThreads];
    float acc = 0.0f;
    for (long long i = threadIdx.x; i < n; i += kThreads) {
        const float e = y[i] - t[i];
        dy[i] = 2.0f * e / (float)n;
        acc = fmaf(e, e, acc);
    }
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int w = kThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        *loss = s[0] / (float)n;
        if (stepc) {
            if (hist) hist[*stepc - step0] = s[0] / (float)n;
            *stepc += 1;
        }
    }
}

// dz[s][i] = (sum_j delta[s][j] W[j][i]) (1 - h[s][i]^2): back through a dense layer and tanh
__global__ void __launch_bounds__(kThreads) dense_backward(const float *delta, int dout,
                                                           const float *W, const float *h, int din,
                                                           long long n, float *dz) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * din) return;
    const long long s = idx / din;
    const int i = (int)(idx % din);
    float acc = 0.0f;
    for (int j = 0; j < dout; ++j) acc = fmaf(delta[s * dout + j], W[(long long)j * din + i], acc);
    const float hv = h[idx];
    dz[idx] = acc * (1.0f - hv * hv);
}

// Chunk partials of the weight gradient: part[c][j][i] = sum over samples s of chunk c of
// delta[s][j] in[s][i] (i = din: delta[s][j] alone, the bias), s in increasing order.
__global__ void __launch_bounds__(kThreads) dense_wgrad_part(const float *delta, int dout,
                                                             const float *in, int din, long long n,
                                                             float *part) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long per = (long long)dout * (din + 1);
    if (idx >= per) return;
    const int j = (int)(idx / (din + 1));
    const int i = (int)(idx % (din + 1));
    const long long s0 = (long long)blockIdx.y * kChunk;
    const long long s1 = s0 + kChunk < n ? s0 + kChunk : n;
    float acc = 0.0f;
    if (i < din) {
        for (long long s = s0; s < s1; ++s) acc = fmaf(delta[s * dout + j], in[s * din + i], acc);
    } else {
        for (long long s = s0; s < s1; ++s) acc += delta[s * dout + j];
    }
    part[blockIdx.y * per + idx] = acc;
}

// gW[j][i] = sum_c part[c][j][i] in chunk order; gb[j] = the same for i = din
__global__ void __launch_bounds__(kThreads) dense_wgrad_sum(const float *part, int dout, int din,
                                                            int nchunks, float *gW, float *gb) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long per = (long long)dout * (din + 1);
    if (idx >= per) return;
    float acc = 0.0f;
    for (int c = 0; c < nchunks; ++c) acc += part[c * per + idx];
    const int j = (int)(idx / (din + 1));
    const int i = (int)(idx % (din + 1));
    if (i < din)
        gW[(long long)j * din + i] = acc;
    else
        gb[j] = acc;
}

// Adam with the step number t = *stepc read on the device (bias corrections 1 - b^t)
__global__ void __launch_bounds__(kThreads) adam_kernel_dev(float *p, float *m, float *v,
                                                            const float *g, long long count,
                                                            float lr, float b1, float b2, float eps,
                                                            const int *stepc) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const float t = (float)*stepc;
    const float c1 = 1.0f - powf(b1, t), c2 = 1.0f - powf(b2, t);
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

__global__ void set_step_kernel(int *stepc, int value) { *stepc = value; }

__global__ void __launch_bounds__(kThreads) adam_kernel(float *p, float *m, float *v, const float *g,
                                                        long long count, float lr, float b1,
                                                        float b2, float eps, float c1, float c2) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// ---- the two-launch epoch -------------------------------------------------------------------

// Shared memory of the tile kernel (floats): the weights padded to 64 x 64 with zeros, W1 and W2
// with the input index first for the forward pass, W2 with the output index first for the
// backward one; a tile's inputs, hidden states and deltas, the sample index last.
struct TileSmem {
    float w1[kSmall * kWRow], w2[kSmall * kWRow], w2t[kSmall * kWRow];
    float b1[kSmall], b2[kSmall], w3[kSmall];
    float x[kSmall * kRow], h1[kSmall * kRow], h2[kSmall * kRow], z1[kSmall * kRow], z2[kSmall * kRow];
    float dy[kTile], loss[kTile];
};

// acc[s] += sum_i w[i][j] in[i][8 g + s], i < n in order, for the thread's unit j and eight samples
__device__ __forceinline__ void tile_dense(const float *w, const float *in, int n, int j, int g,
                                           float (&acc)[8]) {
    for (int i = 0; i < n; ++i) {
        const float c = w[i * kWRow + j];
        const float4 a = *reinterpret_cast<const float4 *>(in + i * kRow + 8 * g);
        const float4 b = *reinterpret_cast<const float4 *>(in + i * kRow + 8 * g + 4);
        acc[0] = fmaf(a.x, c, acc[0]);
        acc[1] = fmaf(a.y, c, acc[1]);
        acc[2] = fmaf(a.z, c, acc[2]);
        acc[3] = fmaf(a.w, c, acc[3]);
        acc[4] = fmaf(b.x, c, acc[4]);
        acc[5] = fmaf(b.y, c, acc[5]);
        acc[6] = fmaf(b.z, c, acc[6]);
        acc[7] = fmaf(b.w, c, acc[7]);
    }
}
__device__ __forceinline__ void put8(float *row, int g, const float (&v)[8]) {
    *reinterpret_cast<float4 *>(row + 8 * g) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4 *>(row + 8 * g + 4) = make_float4(v[4], v[5], v[6], v[7]);
}
// acc[a][b] += sum over the tile's samples of delta[j0 + 16 a] in[i0 + 16 b], samples in order
__device__ __forceinline__ void tile_wgrad(const float *delta, const float *in, int j0, int i0,
                                           float (&acc)[4][4]) {
#pragma unroll 2
    for (int s = 0; s < kTile; s += 4) {
        float4 u[4], v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            u[q] = *reinterpret_cast<const float4 *>(delta + (j0 + 16 * q) * kRow + s);
            v[q] = *reinterpret_cast<const float4 *>(in + (i0 + 16 * q) * kRow + s);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                acc[a][b] = fmaf(u[a].x, v[b].x, acc[a][b]);
                acc[a][b] = fmaf(u[a].y, v[b].y, acc[a][b]);
                acc[a][b] = fmaf(u[a].z, v[b].z, acc[a][b]);
                acc[a][b] = fmaf(u[a].w, v[b].w, acc[a][b]);
            }
    }
}

// Forward pass, loss and back-propagation of tiles b, b + gridDim.x, ... of 32 samples; the CTA's
// gradients (the parameters' layout) and its share of the summed squared error go to
// part[b (P + 1)].  Thread t: unit t % 64, samples 8 (t / 64) ... + 7 in the passes; a 4 x 4 block
// of each weight gradient.  Training (stepc non-null): CTA 0 advances the Adam step counter, which
// the update kernel after it reads.
__global__ void __launch_bounds__(kThreads) mlp_tile_kernel(const float *p, int d, int H,
                                                            const float *X, const float *t,
                                                            long long n, float *part, int *stepc) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TileSmem &M = *reinterpret_cast<TileSmem *>(smem_raw);
    const int tid = threadIdx.x, j = tid & 63, g = tid >> 6;
    const int P = H * d + H + H * H + H + H + 1;
    const float *W1 = p, *b1 = W1 + H * d, *W2 = b1 + H, *b2 = W2 + H * H, *W3 = b2 + H, *b3 = W3 + H;
    if (stepc && blockIdx.x == 0 && tid == 0) *stepc += 1;
    for (int q = tid; q < kSmall * kWRow; q += kThreads) M.w1[q] = M.w2[q] = M.w2t[q] = 0.0f;
    for (int q = tid; q < kSmall * kRow; q += kThreads) M.x[q] = 0.0f;
    __syncthreads();
    for (int q = tid; q < H * d; q += kThreads) M.w1[(q % d) * kWRow + q / d] = W1[q];
    for (int q = tid; q < H * H; q += kThreads) {
        const float w = W2[q];
        M.w2[(q % H) * kWRow + q / H] = w;
        M.w2t[(q / H) * kWRow + q % H] = w;
    }
    if (tid < kSmall) {
        M.b1[tid] = tid < H ? b1[tid] : 0.0f;
        M.b2[tid] = tid < H ? b2[tid] : 0.0f;
        M.w3[tid] = tid < H ? W3[tid] : 0.0f;
    }
    const int j0 = tid >> 4, i0 = tid & 15;
    float g1[4][4] = {}, g2[4][4] = {};  // gradients of W1 and W2
    float gb1 = 0.0f, gb2 = 0.0f, gw3 = 0.0f, gb3 = 0.0f, loss = 0.0f;
    const float bias3 = b3[0];
    const long long tiles = (n + kTile - 1) / kTile;
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long long s0 = tile * kTile;
        const int ns = n - s0 < kTile ? (int)(n - s0) : kTile;
        __syncthreads();  // the weights are there; the previous tile's rows are free
        for (int q = tid; q < kTile * d; q += kThreads) {
            const int s = q / d, i = q - s * d;
            M.x[i * kRow + s] = s < ns ? X[s0 * d + q] : 0.0f;
        }
        __syncthreads();
        float acc[8];
#pragma unroll
        for (int s = 0; s < 8; ++s) acc[s] = M.b1[j];
        tile_dense(M.w1, M.x, d, j, g, acc);
#pragma unroll
        for (int s = 0; s < 8; ++s) acc[s] = tanhf(acc[s]);
        put8(M.h1 + j * kRow, g, acc);
        __syncthreads();
#pragma unroll
        for (int s = 0; s < 8; ++s) acc[s] = M.b2[j];
        tile_dense(M.w2, M.h1, H, j, g, acc);
#pragma unroll
        for (int s = 0; s < 8; ++s) acc[s] = tanhf(acc[s]);
        put8(M.h2 + j * kRow, g, acc);
        __syncthreads();
        if (tid < kTile) {  // output and loss of one sample
            float y = bias3;
            for (int i = 0; i < H; ++i) y = fmaf(M.h2[i * kRow + tid], M.w3[i], y);
            const float e = tid < ns ? y - t[s0 + tid] : 0.0f;
            M.dy[tid] = 2.0f * e / (float)n;
            loss = fmaf(e, e, loss);
        }
        __syncthreads();
        {  // back through the output layer: h2 still in acc
            float z[8];
#pragma unroll
            for (int s = 0; s < 8; ++s)
                z[s] = fmaf(M.dy[8 * g + s], M.w3[j], 0.0f) * (1.0f - acc[s] * acc[s]);
            put8(M.z2 + j * kRow, g, z);
        }
        __syncthreads();
        {  // back through the second layer
            float z[8] = {};
            tile_dense(M.w2t, M.z2, H, j, g, z);
            const float4 a = *reinterpret_cast<const float4 *>(M.h1 + j * kRow + 8 * g);
            const float4 b = *reinterpret_cast<const float4 *>(M.h1 + j * kRow + 8 * g + 4);
            const float h[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
            for (int s = 0; s < 8; ++s) z[s] = z[s] * (1.0f - h[s] * h[s]);
            put8(M.z1 + j * kRow, g, z);
        }
        __syncthreads();
        tile_wgrad(M.z1, M.x, j0, i0, g1);
        tile_wgrad(M.z2, M.h1, j0, i0, g2);
        if (g == 0)
            for (int s = 0; s < kTile; ++s) gb1 += M.z1[j * kRow + s];
        if (g == 1)
            for (int s = 0; s < kTile; ++s) gb2 += M.z2[j * kRow + s];
        if (g == 2)
            for (int s = 0; s < kTile; ++s) gw3 = fmaf(M.dy[s], M.h2[j * kRow + s], gw3);
        if (tid == 255)
            for (int s = 0; s < kTile; ++s) gb3 += M.dy[s];
    }
    float *out = part + (long long)blockIdx.x * (P + 1);
    float *o1 = out + H * d, *o2 = o1 + H, *o3 = o2 + H * H, *o4 = o3 + H, *o5 = o4 + H;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int r = j0 + 16 * a, c = i0 + 16 * b;
            if (r < H && c < d) out[r * d + c] = g1[a][b];
            if (r < H && c < H) o2[r * H + c] = g2[a][b];
        }
    if (j < H) {
        if (g == 0) o1[j] = gb1;
        if (g == 1) o3[j] = gb2;
        if (g == 2) o4[j] = gw3;
    }
    if (tid == 255) o5[0] = gb3;
    if (tid < kTile) M.loss[tid] = loss;
    __syncthreads();
    if (tid == 0) {
        float e = 0.0f;
        for (int s = 0; s < kTile; ++s) e += M.loss[s];
        out[P] = e;
    }
}

constexpr int kUpdateParams = 32;  // parameters of an update CTA, eight threads each

// grad = the sum of the tile CTAs' gradients, eight runs of CTAs in parallel, the runs in order;
// then, training (stepc non-null), the Adam update of adam_kernel_dev, with what rounding a
// parameter to FP32 leaves out carried to its next update (rest; TwoSum): an update of about lr is
// 1e-3 of a parameter, and without that 200 updates' roundings are most of the result's error.
// The thread of index P sums the losses.
__global__ void __launch_bounds__(kThreads)
    mlp_update_kernel(const float *part, int ctas, int P, long long n, float *grad, float *loss_out,
                      float *p, float *m, float *v, float *rest, float lr, float b1, float b2,
                      float eps, const int *stepc, int step0, float *hist) {
    __shared__ float run[8][kUpdateParams];
    const int q = threadIdx.x & (kUpdateParams - 1), r = threadIdx.x / kUpdateParams;
    const int i = blockIdx.x * kUpdateParams + q;
    const int c0 = ctas * r / 8, c1 = ctas * (r + 1) / 8;
    float acc = 0.0f;
    if (i <= P) {
#pragma unroll 8
        for (int c = c0; c < c1; ++c) acc += part[(long long)c * (P + 1) + i];
    }
    run[r][q] = acc;
    __syncthreads();
    if (r != 0 || i > P) return;
#pragma unroll
    for (int k = 1; k < 8; ++k) acc += run[k][q];
    if (i == P) {
        const float loss = acc / (float)n;
        *loss_out = loss;
        if (stepc && hist) hist[*stepc - 1 - step0] = loss;
        return;
    }
    grad[i] = acc;
    if (!stepc) return;
    const float t = (float)*stepc;
    const float k1 = 1.0f - powf(b1, t), k2 = 1.0f - powf(b2, t);
    const float mi = b1 * m[i] + (1.0f - b1) * acc;
    const float vi = b2 * v[i] + (1.0f - b2) * acc * acc;
    m[i] = mi;
    v[i] = vi;
    const float q0 = p[i], y = __fadd_rn(rest[i], -(lr * (mi / k1) / (sqrtf(vi / k2) + eps)));
    const float q1 = __fadd_rn(q0, y), back = __fadd_rn(q1, -q0);
    rest[i] = __fadd_rn(__fadd_rn(q0, -__fadd_rn(q1, -back)), __fadd_rn(y, -back));
    p[i] = q1;
}

// One small-network epoch (or, with m null, the gradient alone).
cudaError_t small_epoch(float *p, float *m, float *v, int d, int H, const float *X, const float *t,
                        long long n, float *ws, const Sizes &S, float lr, int *stepc, int step0,
                        float *hist, cudaStream_t st) {
    const int ctas = (int)tile_ctas(n), P = (int)S.P;
    float *part = ws + S.part;
    mlp_tile_kernel<<<ctas, kThreads, sizeof(TileSmem), st>>>(p, d, H, X, t, n, part, stepc);
    mlp_update_kernel<<<(P + 1 + kUpdateParams - 1) / kUpdateParams, kThreads, 0, st>>>(
        part, ctas, P, n, ws + S.grad, ws + S.loss, p, m, v, ws + S.rest, lr, 0.9f, 0.999f, 1e-8f,
        stepc, step0, hist);
    return cudaGetLastError();
}
cudaError_t small_prepare() {
    static hydro::PerDevice attribute;
    return attribute.once([] {
        return cudaFuncSetAttribute(mlp_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sizeof(TileSmem));
    });
}

unsigned blocks(long long work) { return (unsigned)((work + kThreads - 1) / kThreads); }

// gW, gb of a dense layer (delta: n x dout, in: n x din) through the chunk partials
void dense_wgrad(const float *delta, int dout, const float *in, int din, long long n, float *part,
                 float *gW, float *gb, cudaStream_t st) {
    const int nchunks = (int)((n + kChunk - 1) / kChunk);
    const long long per = (long long)dout * (din + 1);
    dense_wgrad_part<<<dim3(blocks(per), (unsigned)nchunks), kThreads, 0, st>>>(delta, dout, in,
                                                                                din, n, part);
    dense_wgrad_sum<<<blocks(per), kThreads, 0, st>>>(part, dout, din, nchunks, gW, gb);
}

cudaError_t forward_all(const float *p, int d, int H, const float *X, long long n, float *ws,
                        const Sizes &S, cudaStream_t st) {
    const float *W1 = p, *b1 = W1 + (long long)H * d, *W2 = b1 + H, *b2 = W2 + (long long)H * H;
    const float *W3 = b2 + H, *b3 = W3 + H;
    dense_forward<true><<<blocks(n * H), kThreads, 0, st>>>(X, d, W1, b1, H, n, ws + S.h1);
    dense_forward<true><<<blocks(n * H), kThreads, 0, st>>>(ws + S.h1, H, W2, b2, H, n, ws + S.h2);
    dense_forward<false><<<blocks(n), kThreads, 0, st>>>(ws + S.h2, H, W3, b3, 1, n, ws + S.y);
    return cudaGetLastError();
}

// Forward, loss and back-propagation into ws + S.grad.  Training: stepc/step0/hist as in
// mse_kernel.
cudaError_t gradient_all(const float *p, int d, int H, const float *X, const float *t, long long n,
                         float *ws, const Sizes &S, cudaStream_t st, int *stepc = nullptr,
                         int step0 = 0, float *hist = nullptr) {
    cudaError_t e = forward_all(p, d, H, X, n, ws, S, st);
    if (e != cudaSuccess) return e;
    const float *W2 = p + (long long)H * d + H, *W3 = W2 + (long long)H * H + H;
    float *g = ws + S.grad;
    float *gW1 = g, *gb1 = gW1 + (long long)H * d, *gW2 = gb1 + H, *gb2 = gW2 + (long long)H * H;
    float *gW3 = gb2 + H, *gb3 = gW3 + H;
    mse_kernel<<<1, kThreads, 0, st>>>(ws + S.y, t, n, ws + S.dy, ws + S.loss, stepc, step0, hist);
    // output layer (linear): delta = dy
    float *part = ws + S.part;
    dense_wgrad(ws + S.dy, 1, ws + S.h2, H, n, part, gW3, gb3, st);
    dense_backward<<<blocks(n * H), kThreads, 0, st>>>(ws + S.dy, 1, W3, ws + S.h2, H, n, ws + S.dz2);
    dense_wgrad(ws + S.dz2, H, ws + S.h1, H, n, part, gW2, gb2, st);
    dense_backward<<<blocks(n * H), kThreads, 0, st>>>(ws + S.dz2, H, W2, ws + S.h1, H, n, ws + S.dz1);
    dense_wgrad(ws + S.dz1, H, X, d, n, part, gW1, gb1, st);
    return cudaGetLastError();
}

bool dims_ok(int d, int H, long long n) {
    return d >= 1 && d <= 4096 && H >= 1 && H <= 4096 && n >= 1 && n <= 65535LL * kChunk;
}

}  // namespace

extern "C" {

int hydro_mlp_sizes(int32_t d, int32_t hidden, int64_t n, int64_t *param_count,
                    size_t *workspace_bytes) {
    if (!dims_ok(d, hidden, n)) return HYDRO_EINVAL;
    const Sizes S = sizes(d, hidden, n);
    if (param_count) *param_count = S.P;
    if (workspace_bytes) *workspace_bytes = sizeof(float) * (size_t)S.total;
    return HYDRO_OK;
}

int hydro_mlp_forward(const float *params, int32_t d, int32_t hidden, const float *X, int64_t n,
                      float *y_out, void *workspace, void *stream) {
    if (!params || !X || !y_out || !workspace || !dims_ok(d, hidden, n)) return HYDRO_EINVAL;
    const Sizes S = sizes(d, hidden, n);
    float *ws = static_cast<float *>(workspace);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = forward_all(params, d, hidden, X, n, ws, S, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(y_out, ws + S.y, sizeof(float) * (size_t)n, cudaMemcpyDeviceToDevice, st);
    return e == cudaSuccess ? HYDRO_OK : hydro::record_cuda_error(e, "hydro_mlp_forward");
}

int hydro_mlp_gradient(const float *params, int32_t d, int32_t hidden, const float *X,
                       const float *t, int64_t n, void *workspace, float *grad_out,
                       float *loss_out, void *stream) {
    if (!params || !X || !t || !workspace || !dims_ok(d, hidden, n)) return HYDRO_EINVAL;
    const Sizes S = sizes(d, hidden, n);
    float *ws = static_cast<float *>(workspace);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaSuccess;
    if (small_net(d, hidden)) {
        e = small_prepare();
        if (e == cudaSuccess)  // (the parameters are only read: no step counter)
            e = small_epoch(const_cast<float *>(params), nullptr, nullptr, d, hidden, X, t, n, ws, S,
                            0.0f, nullptr, 0, nullptr, st);
    } else {
        e = gradient_all(params, d, hidden, X, t, n, ws, S, st);
    }
    if (e == cudaSuccess && grad_out)
        e = cudaMemcpyAsync(grad_out, ws + S.grad, sizeof(float) * (size_t)S.P,
                            cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess && loss_out)
        e = cudaMemcpyAsync(loss_out, ws + S.loss, sizeof(float), cudaMemcpyDeviceToDevice, st);
    return e == cudaSuccess ? HYDRO_OK : hydro::record_cuda_error(e, "hydro_mlp_gradient");
}

int hydro_mlp_adam(float *params, float *m, float *v, const float *grad, int64_t count,
                   int32_t step, float lr, float beta1, float beta2, float eps, void *stream) {
    if (!params || !m || !v || !grad || count < 1 || step < 1) return HYDRO_EINVAL;
    const float c1 = 1.0f - powf(beta1, (float)step);
    const float c2 = 1.0f - powf(beta2, (float)step);
    adam_kernel<<<blocks(count), kThreads, 0, static_cast<cudaStream_t>(stream)>>>(
        params, m, v, grad, count, lr, beta1, beta2, eps, c1, c2);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? HYDRO_OK : hydro::record_cuda_error(e, "hydro_mlp_adam");
}

int hydro_mlp_train(float *params, float *m, float *v, int32_t d, int32_t hidden, const float *X,
                    const float *t, int64_t n, int32_t epochs, int32_t step0, float lr,
                    void *workspace, float *loss_out, void *stream) {
    if (!params || !m || !v || !X || !t || !workspace || epochs < 0 || step0 < 0 ||
        !dims_ok(d, hidden, n))
        return HYDRO_EINVAL;
    const Sizes S = sizes(d, hidden, n);
    float *ws = static_cast<float *>(workspace);
    int *stepc = reinterpret_cast<int *>(ws + S.stepc);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // one epoch: forward, loss (advances the step counter), back-propagation, Adam
    auto epoch = [&](cudaStream_t s) -> cudaError_t {
        cudaError_t e = gradient_all(params, d, hidden, X, t, n, ws, S, s, stepc, step0, loss_out);
        if (e != cudaSuccess) return e;
        adam_kernel_dev<<<blocks(S.P), kThreads, 0, s>>>(params, m, v, ws + S.grad, S.P, lr, 0.9f,
                                                         0.999f, 1e-8f, stepc);
        return cudaGetLastError();
    };
    set_step_kernel<<<1, 1, 0, st>>>(stepc, step0);
    cudaError_t e = cudaGetLastError();
    if (small_net(d, hidden)) {  // two launches an epoch: the GPU, not the launches, sets the pace
        if (e == cudaSuccess) e = small_prepare();
        if (e == cudaSuccess) e = cudaMemsetAsync(ws + S.rest, 0, sizeof(float) * (size_t)S.P, st);
        for (int k = 0; k < epochs && e == cudaSuccess; ++k)
            e = small_epoch(params, m, v, d, hidden, X, t, n, ws, S, lr, stepc, step0, loss_out, st);
        return e == cudaSuccess ? HYDRO_OK : hydro::record_cuda_error(e, "hydro_mlp_train");
    }
    const int per = epochs < kEpochsPerGraph ? epochs : kEpochsPerGraph;
    const int reps = per > 0 ? epochs / per : 0;
    if (e == cudaSuccess && reps > 1) {
        // capture `per` epochs on a private stream and replay them on the caller's
        cudaStream_t cap = nullptr;
        cudaGraph_t g = nullptr;
        cudaGraphExec_t x = nullptr;
        e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            cudaError_t ec = cudaSuccess;
            for (int k = 0; k < per && ec == cudaSuccess; ++k) ec = epoch(cap);
            e = cudaStreamEndCapture(cap, &g);
            if (e == cudaSuccess) e = ec;
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&x, g, 0);
        for (int r = 0; r < reps && e == cudaSuccess; ++r) e = cudaGraphLaunch(x, st);
        if (x) cudaGraphExecDestroy(x);
        if (g) cudaGraphDestroy(g);
        if (cap) cudaStreamDestroy(cap);
        for (int k = reps * per; k < epochs && e == cudaSuccess; ++k) e = epoch(st);
    } else {
        for (int k = 0; k < epochs && e == cudaSuccess; ++k) e = epoch(st);
    }
    return e == cudaSuccess ? HYDRO_OK : hydro::record_cuda_error(e, "hydro_mlp_train");
}

}  // extern "C"
