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
// grad (P), loss (1), the Adam step counter (one int), the weight-gradient chunk partials
// (ceil(n / kChunk) x H x (max(d, H) + 1), or x P for small networks).
//
// Networks of at most 64 inputs and 64 hidden units (the cost model's) train in two launches per
// epoch: mlp_chunk_kernel takes a chunk of samples through forward pass and back-propagation in
// the shared memory of a thread-block cluster and leaves the chunk's weight gradients;
// mlp_update_kernel sums them in chunk order and applies Adam.  The thirteen launches of the
// general kernels took 174 us an epoch (4200 records, 35 inputs, width 64), most of it in gathers
// and launches; the two take 23.4, with equal bits.  The general kernels serve wider networks.
//
// There training replays captured epochs: the Adam step number lives in the workspace (the loss
// kernel advances it, the Adam kernel derives its bias corrections from it), so one epoch's
// launches are the same every epoch and a CUDA graph of kEpochsPerGraph epochs is replayed.
#include <cooperative_groups.h>
#include <math.h>
#include <string.h>

#include "../../include/hydro.h"
#include "hydro_internal.h"

namespace {

namespace cg = cooperative_groups;

constexpr int kThreads = 256;
constexpr int kChunk = 128;  // samples per partial sum of the weight gradients

constexpr int kEpochsPerGraph = 16;

struct Sizes {
    long long P, h1, h2, y, dy, dz2, dz1, grad, loss, stepc, part, total;  // float offsets
};

constexpr int kSmall = 64;                // most inputs and hidden units of the two-launch epoch
constexpr int kTile = 32;                 // samples of a CTA's tile
constexpr int kTiles = kChunk / kTile;    // CTAs of a cluster
constexpr int kUnits = kSmall / kTiles;   // units whose gradients a CTA sums
constexpr int kPass = 512;                // threads of the passes: a unit, four samples each
constexpr int kChunkThreads = kPass + 32;
constexpr int kRow = kTile + 4;           // floats of a shared row of a tile,
constexpr int kCRow = kChunk + 4;         // of a chunk (rows on distinct banks)
constexpr int kWRow = kSmall + 1;         // and of a weight matrix (either index conflict-free)

bool small_net(int d, int H) { return d <= kSmall && H <= kSmall; }

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
    S.part = o;
    const long long per = (long long)H * ((d > H ? d : H) + 1);
    o += (n + kChunk - 1) / kChunk * (small_net(d, H) && S.P > per ? S.P : per);
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

// The sum of the CTA's kThreads values by halving, in thread 0
__device__ __forceinline__ float block_sum(float (&s)[kThreads], float value) {
    s[threadIdx.x] = value;
    __syncthreads();
    for (int w = kThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
        __syncthreads();
    }
    return s[0];
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
    const float sum = block_sum(s, acc);
    if (threadIdx.x == 0) {
        *loss = sum / (float)n;
        if (stepc) {
            if (hist) hist[*stepc - step0] = sum / (float)n;
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

// Adam's step number t for parameter i of gradient gi (bias corrections 1 - b^t)
__device__ __forceinline__ void adam_step(float *p, float *m, float *v, long long i, float gi,
                                          float lr, float b1, float b2, float eps, float t) {
    const float c1 = 1.0f - powf(b1, t), c2 = 1.0f - powf(b2, t);
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Adam with the step number read on the device
__global__ void __launch_bounds__(kThreads) adam_kernel_dev(float *p, float *m, float *v,
                                                            const float *g, long long count,
                                                            float lr, float b1, float b2, float eps,
                                                            const int *stepc) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    adam_step(p, m, v, i, g[i], lr, b1, b2, eps, (float)*stepc);
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

// Shared memory of the chunk kernel (floats).  Weights with the input index first; a tile's own
// rows (z2, h2) of 32 samples; rows of the chunk's 128 samples, the sample index last: the inputs
// and first hidden states of all units, and for the CTA's 16 units the deltas and second states.
struct ChunkSmem {
    float w1[kSmall * kWRow], w2[kSmall * kWRow];
    float b1[kSmall], b2[kSmall], w3[kSmall];
    float x[kSmall * kCRow], h1[kSmall * kCRow];
    float h2[kSmall * kRow], z2[kSmall * kRow];
    float z1c[kUnits * kCRow], z2c[kUnits * kCRow], h2c[kUnits * kCRow];
    float dy[kChunk];
};

// Asynchronous copy of one float to shared memory; zero where !valid (`from` is readable anyway)
__device__ __forceinline__ void copy4(float *to, const float *from, bool valid = true) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(to)),
                 "l"(from), "r"(valid ? 4 : 0)
                 : "memory");
}

// acc[s] += sum_i w[i stride] in[i ROW + s], i < n in order: one unit, four samples
template <int ROW>
__device__ __forceinline__ void tile_dense(const float *w, int stride, const float *in, int n,
                                           float (&acc)[4]) {
#pragma unroll 8
    for (int i = 0; i < n; ++i) {
        const float c = w[i * stride];
        const float4 a = *reinterpret_cast<const float4 *>(in + i * ROW);
        acc[0] = fmaf(a.x, c, acc[0]);
        acc[1] = fmaf(a.y, c, acc[1]);
        acc[2] = fmaf(a.z, c, acc[2]);
        acc[3] = fmaf(a.w, c, acc[3]);
    }
}
__device__ __forceinline__ void put4(float *at, const float (&v)[4]) {
    *reinterpret_cast<float4 *>(at) = make_float4(v[0], v[1], v[2], v[3]);
}
// acc[a][b] += sum_s z[8 a][s] in[16 b][s], bias[a] += sum_s z[8 a][s], s < ns in order
__device__ __forceinline__ void chunk_wgrad(const float *z, const float *in, int ns,
                                            float (&acc)[2][2], float (&bias)[2]) {
    int s = 0;
#pragma unroll 4
    for (; s + 4 <= ns; s += 4) {
        float4 u[2], v[2];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            u[a] = *reinterpret_cast<const float4 *>(z + 8 * a * kCRow + s);
            v[a] = *reinterpret_cast<const float4 *>(in + 16 * a * kCRow + s);
        }
#pragma unroll
        for (int a = 0; a < 2; ++a) {
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                acc[a][b] = fmaf(u[a].x, v[b].x, acc[a][b]);
                acc[a][b] = fmaf(u[a].y, v[b].y, acc[a][b]);
                acc[a][b] = fmaf(u[a].z, v[b].z, acc[a][b]);
                acc[a][b] = fmaf(u[a].w, v[b].w, acc[a][b]);
            }
            bias[a] = bias[a] + u[a].x;
            bias[a] = bias[a] + u[a].y;
            bias[a] = bias[a] + u[a].z;
            bias[a] = bias[a] + u[a].w;
        }
    }
    for (; s < ns; ++s)
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const float u = z[8 * a * kCRow + s];
#pragma unroll
            for (int b = 0; b < 2; ++b) acc[a][b] = fmaf(u, in[16 * b * kCRow + s], acc[a][b]);
            bias[a] += u;
        }
}

// Forward pass, back-propagation and weight-gradient sums of one chunk of kChunk samples by a
// cluster of four CTAs: each takes a tile of 32 samples through the passes (thread t < 512: unit
// t % 64, samples 4 (t / 64) ... + 3; warp 16: the output layer) and leaves its hidden states and
// deltas in the shared memory of the CTAs that need them; then each sums the gradients of 16 units
// over all 128 samples, so that every sum runs in the order of the general kernels above and the
// results equal theirs bit for bit (training amplifies a last bit by orders of magnitude over 200
// epochs).  The errors y - t go to err, the chunk's sums (the parameters' layout) to
// part[chunk P].  Training (stepc non-null): CTA 0 advances the Adam step counter, which the update
// kernel after it reads.  Bound by shared-memory accesses (the LSU's wavefronts 60 % of its peak) along a
// chain of five dependent passes; 17.6 us of the epoch under a profiler with cold caches.
__global__ void __cluster_dims__(kTiles, 1, 1) __launch_bounds__(kChunkThreads)
    mlp_chunk_kernel(const float *p, int d, int H, const float *X, const float *t, long long n,
                     float *err, float *part, int *stepc) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ChunkSmem &M = *reinterpret_cast<ChunkSmem *>(smem_raw);
    const cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), tid = threadIdx.x;
    const int P = H * d + H + H * H + H + H + 1;
    const float *W1 = p, *b1 = W1 + H * d, *W2 = b1 + H, *b2 = W2 + H * H, *W3 = b2 + H, *b3 = W3 + H;
    const long long chunk = blockIdx.x / kTiles, s0 = chunk * kChunk;
    const int ns = n - s0 < kChunk ? (int)(n - s0) : kChunk;  // samples of the chunk
    if (stepc && blockIdx.x == 0 && tid == 0) *stepc += 1;
    // (Units from H up and inputs from d up are never summed: their rows keep whatever is there.)
    // Asynchronous copies, a warp per row: plain loads in a loop wait for one another (an epoch of
    // 27.5 us instead of 25.4 with them).
    const int lane = tid & 31, warp = tid >> 5;
    for (int r = warp; r < kChunk; r += kChunkThreads / 32)
        for (int i = lane; i < d; i += 32)
            copy4(&M.x[i * kCRow + r], X + (s0 + (r < ns ? r : 0)) * d + i, r < ns);
    for (int r = warp; r < H; r += kChunkThreads / 32) {
        for (int i = lane; i < d; i += 32) copy4(&M.w1[i * kWRow + r], W1 + r * d + i);
        for (int i = lane; i < H; i += 32) copy4(&M.w2[i * kWRow + r], W2 + r * H + i);
    }
    if (tid < H) {
        copy4(&M.b1[tid], b1 + tid);
        copy4(&M.b2[tid], b2 + tid);
        copy4(&M.w3[tid], W3 + tid);
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    const bool unit = tid < kPass;
    const int j = tid & 63, g = (tid >> 6) & 7;
    const int col = kTile * rank + 4 * g;  // the thread's samples in the chunk
    // What other CTAs need goes to them from shared memory, eight lanes per row of 128 B: stores of
    // a unit per lane are 32 separate packets each (an epoch of 25.4 us instead of 23.4).
    const int row = tid >> 3, at = 4 * (tid & 7), seat = (row % kUnits) * kCRow + kTile * rank + at;
    const int seat_rank = (row / kUnits) % kTiles;
    cluster.sync();  // the weights and inputs are there; every CTA of the cluster runs
    float acc[4];
    if (unit) {
#pragma unroll
        for (int s = 0; s < 4; ++s) acc[s] = M.b1[j];
        tile_dense<kCRow>(M.w1 + j, kWRow, M.x + col, d, acc);
#pragma unroll
        for (int s = 0; s < 4; ++s) acc[s] = tanhf(acc[s]);
        put4(M.h1 + j * kCRow + col, acc);
    }
    __syncthreads();
    if (unit) {
        const int o = row * kCRow + kTile * rank + at;
        const float4 h = *reinterpret_cast<const float4 *>(M.h1 + o);
#pragma unroll
        for (int r = 1; r < kTiles; ++r)
            *reinterpret_cast<float4 *>(cluster.map_shared_rank(M.h1, (rank + r) % kTiles) + o) = h;
#pragma unroll
        for (int s = 0; s < 4; ++s) acc[s] = M.b2[j];
        tile_dense<kCRow>(M.w2 + j, kWRow, M.h1 + col, H, acc);
#pragma unroll
        for (int s = 0; s < 4; ++s) acc[s] = tanhf(acc[s]);
        put4(M.h2 + j * kRow + 4 * g, acc);
    }
    __syncthreads();
    if (!unit) {  // output and error of one sample
        float y = b3[0];
#pragma unroll 8
        for (int i = 0; i < H; ++i) y = fmaf(M.h2[i * kRow + lane], M.w3[i], y);
        const int s = kTile * rank + lane;
        float e = 0.0f;
        if (s < ns) {
            e = y - t[s0 + s];
            err[s0 + s] = e;
        }
        const float dy = 2.0f * e / (float)n;
#pragma unroll
        for (int r = 0; r < kTiles; ++r) cluster.map_shared_rank(M.dy, r)[s] = dy;
    }
    __syncthreads();
    if (unit) {  // back through the output layer: h2 still in acc
        *reinterpret_cast<float4 *>(cluster.map_shared_rank(M.h2c, seat_rank) + seat) =
            *reinterpret_cast<const float4 *>(M.h2 + row * kRow + at);
        float z[4];
#pragma unroll
        for (int s = 0; s < 4; ++s)
            z[s] = fmaf(M.dy[col + s], M.w3[j], 0.0f) * (1.0f - acc[s] * acc[s]);
        put4(M.z2 + j * kRow + 4 * g, z);
    }
    __syncthreads();
    if (unit) {  // back through the second layer
        *reinterpret_cast<float4 *>(cluster.map_shared_rank(M.z2c, seat_rank) + seat) =
            *reinterpret_cast<const float4 *>(M.z2 + row * kRow + at);
        float z[4] = {};
        tile_dense<kRow>(M.w2 + j * kWRow, 1, M.z2 + 4 * g, H, z);
        const float *h = M.h1 + j * kCRow + col;
#pragma unroll
        for (int s = 0; s < 4; ++s) z[s] = z[s] * (1.0f - h[s] * h[s]);
        put4(M.h2 + j * kRow + 4 * g, z);  // (h2 is no longer read)
    }
    __syncthreads();
    if (unit)
        *reinterpret_cast<float4 *>(cluster.map_shared_rank(M.z1c, seat_rank) + seat) =
            *reinterpret_cast<const float4 *>(M.h2 + row * kRow + at);
    cluster.sync();  // the chunk's states and deltas are there
    float *out = part + chunk * P;
    float *o1 = out + H * d, *o2 = o1 + H, *o3 = o2 + H * H, *o4 = o3 + H, *o5 = o4 + H;
    if (unit) {  // threads 0-255: W1 and b1; 256-511: W2 and b2; two units, two inputs each
        const bool first = tid < kPass / 2;
        const int cols = first ? d : H;
        const int j0 = (tid >> 4) & 7, i0 = (tid & 15) + (tid & 128) / 4;
        if (i0 < cols) {
            float gw[2][2] = {}, gb[2] = {};
            chunk_wgrad((first ? M.z1c : M.z2c) + j0 * kCRow, (first ? M.x : M.h1) + i0 * kCRow, ns,
                        gw, gb);
            float *ow = first ? out : o2, *ob = first ? o1 : o3;
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const int r = kUnits * rank + j0 + 8 * a;
                if (r >= H) continue;
#pragma unroll
                for (int b = 0; b < 2; ++b)
                    if (i0 + 16 * b < cols) ow[r * cols + i0 + 16 * b] = gw[a][b];
                if (i0 == 0) ob[r] = gb[a];
            }
        }
    } else if (lane <= kUnits) {  // W3; b3
        const int r = kUnits * rank + lane;
        float sum = 0.0f;
        if (lane < kUnits) {
#pragma unroll 8
            for (int s = 0; s < ns; ++s) sum = fmaf(M.dy[s], M.h2c[lane * kCRow + s], sum);
            if (r < H) o4[r] = sum;
        } else if (rank == 0) {
#pragma unroll 8
            for (int s = 0; s < ns; ++s) sum += M.dy[s];
            o5[0] = sum;
        }
    }
}

// grad = the chunks' sums added in chunk order; then, training (stepc non-null), the Adam update.
// The last CTA adds up the loss as mse_kernel does.
__global__ void __launch_bounds__(kThreads)
    mlp_update_kernel(const float *part, const float *err, int chunks, int P, long long n,
                      float *grad, float *loss_out, float *p, float *m, float *v, float lr,
                      float b1, float b2, float eps, const int *stepc, int step0, float *hist) {
    if (blockIdx.x == gridDim.x - 1) {
        __shared__ float s[kThreads];
        float acc = 0.0f;
#pragma unroll 8
        for (long long i = threadIdx.x; i < n; i += kThreads) acc = fmaf(err[i], err[i], acc);
        const float sum = block_sum(s, acc);
        if (threadIdx.x == 0) {
            *loss_out = sum / (float)n;
            if (stepc && hist) hist[*stepc - 1 - step0] = sum / (float)n;
        }
        return;
    }
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i >= P) return;
    float acc = 0.0f;
#pragma unroll 32
    for (int c = 0; c < chunks; ++c) acc += part[(long long)c * P + i];
    grad[i] = acc;
    if (stepc) adam_step(p, m, v, i, acc, lr, b1, b2, eps, (float)*stepc);
}

// One small-network epoch (or, with m null, the gradient alone).
cudaError_t small_epoch(float *p, float *m, float *v, int d, int H, const float *X, const float *t,
                        long long n, float *ws, const Sizes &S, float lr, int *stepc, int step0,
                        float *hist, cudaStream_t st) {
    const int chunks = (int)((n + kChunk - 1) / kChunk), P = (int)S.P;
    float *part = ws + S.part, *err = ws + S.y;
    mlp_chunk_kernel<<<chunks * kTiles, kChunkThreads, sizeof(ChunkSmem), st>>>(p, d, H, X, t, n,
                                                                                err, part, stepc);
    mlp_update_kernel<<<(P + kThreads - 1) / kThreads + 1, kThreads, 0, st>>>(
        part, err, chunks, P, n, ws + S.grad, ws + S.loss, p, m, v, lr, 0.9f, 0.999f, 1e-8f, stepc,
        step0, hist);
    return cudaGetLastError();
}
cudaError_t small_prepare() {
    static hydro::PerDevice attribute;
    return attribute.once([] {
        return cudaFuncSetAttribute(mlp_chunk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sizeof(ChunkSmem));
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
