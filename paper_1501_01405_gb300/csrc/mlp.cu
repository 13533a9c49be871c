// Learned control variate, network stages: a d_in -> 64 -> 64 -> 1 ReLU
// network (d_in = 8 for the tandem queue, 6 for the forest fire) trained on
// replications the engine generates, used as a control variate.  The paper
// has no learned component; its estimator (the replication mean, Section 1)
// stays the fallback and the yardstick the control variate is checked against.
//
// Arithmetic: parameters are FP32 masters; every matmul takes BF16 operands
// (round to nearest even from FP32) and accumulates in FP32:
//   forward  z1 = x~ W1~^T + b1, h1 = relu(z1); z2 = h1~ W2~^T + b2, h2 = relu(z2);
//            yhat = h2~ . W3~ + b3
//   backward dyhat = 2 (yhat - y) / B; dW3 = sum dyhat h2~; dz2 = dyhat W3~ [z2 > 0];
//            dW2 = dz2~^T h1~; dz1 = (dz2~ W2~) [z1 > 0]; dW1 = dz1~^T x~;
//            bias gradients are FP32 sums of the unrounded dz.
// The matrices are 64 wide, so the passes are latency- not throughput-bound:
// a CTA takes a tile of 32 samples with the BF16-rounded weights staged in
// shared memory (both orientations of W2, so every inner product reads
// consecutive words), and writes its per-parameter partial sums; a second
// kernel adds the partials of all CTAs in a fixed order (deterministic) and,
// during training, applies Adam in the same pass.  These serve the stage
// entry points; the control-variate driver trains in one launch on the
// tensor cores (mlp_train_tc_kernel).
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <numeric>
#include <vector>

#include "common.cuh"
#include "model.cuh"
#include "tc.cuh"

namespace mrip {

namespace {

constexpr int H = 64;
constexpr int kTile = 32;        // samples per CTA
constexpr int kGradThreads = 256;
constexpr int kMaxIn = 8;

__host__ __device__ constexpr long long off_b1(int d) { return static_cast<long long>(H) * d; }
__host__ __device__ constexpr long long off_w2(int d) { return off_b1(d) + H; }
__host__ __device__ constexpr long long off_b2(int d) { return off_w2(d) + H * H; }
__host__ __device__ constexpr long long off_w3(int d) { return off_b2(d) + H; }
__host__ __device__ constexpr long long off_b3(int d) { return off_w3(d) + H; }
__host__ __device__ constexpr long long n_params(int d) { return off_b3(d) + 1; }

__device__ __forceinline__ float bf(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// He-uniform weights from stream tag 3: element e of (W1, W2, W3) reads words
// 2(e mod 2), 2(e mod 2)+1 of block (c0 = e div 2, c1 = 0, rep 0, dp 0).
__global__ void mlp_init_kernel(int d_in, const __grid_constant__ RoundKeys rk, float* theta) {
    const long long n_w = static_cast<long long>(H) * d_in + H * H + H;
    const long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    if (e < n_w) {
        const uint4 b = philox(static_cast<uint32_t>(e >> 1), 0u, 0u, stream_word(3u, 0u), rk);
        const double u = (e & 1) ? u53(b.z, b.w) : u53(b.x, b.y);
        long long dst;
        double fan;
        if (e < static_cast<long long>(H) * d_in) {
            dst = e;
            fan = d_in;
        } else if (e < static_cast<long long>(H) * d_in + H * H) {
            dst = off_w2(d_in) + (e - static_cast<long long>(H) * d_in);
            fan = H;
        } else {
            dst = off_w3(d_in) + (e - static_cast<long long>(H) * d_in - H * H);
            fan = H;
        }
        theta[dst] = static_cast<float>((2.0 * u - 1.0) * sqrt(6.0 / fan));
    }
    // biases
    if (e < H) {
        theta[off_b1(d_in) + e] = 0.0f;
        theta[off_b2(d_in) + e] = 0.0f;
    }
    if (e == 0) theta[off_b3(d_in)] = 0.0f;
}

// Which sample sits at batch position i.
struct SampleMap {
    const int64_t* idx;   // explicit indices, or null
    unsigned long long a, b, n;  // affine permutation (a i + b) mod n when n > 0
    long long off;        // batch offset within the epoch
};

__device__ __forceinline__ long long sample_of(const SampleMap& m, long long i) {
    if (m.idx) return m.idx[i];
    const unsigned long long k = static_cast<unsigned long long>(m.off + i);
    if (m.n > 0) return static_cast<long long>((m.a * k + m.b) % m.n);
    return static_cast<long long>(k);
}

constexpr int HP = H + 4;

struct GradSmem {
    alignas(16) float w1t[kMaxIn][H];  // [k][u]
    alignas(16) float w2t[H][H];       // [u][v]
    alignas(16) float w2[H][H];        // [v][u]
    float w3[H], b1[H], b2[H];
    float b3;
    float xt[kTile][kMaxIn];
    // per-sample rows padded to HP words: samples 4 apart in a warp sit in
    // different banks, and rows stay 16-byte aligned for float4 loads
    alignas(16) float h1[kTile][HP];
    alignas(16) float h1t[kTile][HP];
    alignas(16) float h2[kTile][HP];
    alignas(16) float h2t[kTile][HP];
    alignas(16) float dz2[kTile][HP];
    alignas(16) float dz2t[kTile][HP];
    alignas(16) float dz1[kTile][HP];
    float dy[kTile];
    float ys[kTile];
};

// Stage the BF16-rounded weights (and FP32 biases) of theta (global or
// shared) into S.
__device__ void stage_weights(GradSmem& S, const float* theta, int d_in) {
    const int t = threadIdx.x;
    for (int i = t; i < H * d_in; i += kGradThreads) {
        const int u = i / d_in, k = i - u * d_in;
        S.w1t[k][u] = bf(theta[i]);
    }
    for (int i = t; i < H * H; i += kGradThreads) {
        const int v = i / H, u = i - v * H;
        const float w = bf(theta[off_w2(d_in) + i]);
        S.w2[v][u] = w;
        S.w2t[u][v] = w;
    }
    for (int i = t; i < H; i += kGradThreads) {
        S.w3[i] = bf(theta[off_w3(d_in) + i]);
        S.b1[i] = theta[off_b1(d_in) + i];
        S.b2[i] = theta[off_b2(d_in) + i];
    }
    if (t == 0) S.b3 = theta[off_b3(d_in)];
}

// Stage samples at batch positions pos0 .. pos0 + n_valid - 1 (n_valid <= kTile;
// the rest of the tile is zero and contributes nothing).
__device__ void stage_tile(GradSmem& S, int d_in, const float* __restrict__ X, long long n_total,
                           const float* __restrict__ Y, const SampleMap& map, long long pos0, int n_valid) {
    const int t = threadIdx.x;
    for (int i = t; i < kTile * kMaxIn; i += kGradThreads) {
        const int s = i / kMaxIn, k = i - s * kMaxIn;
        float v = 0.0f;
        if (s < n_valid && k < d_in) {
            const long long smp = sample_of(map, pos0 + s);
            if (MRIP_CHECK(smp >= 0 && smp < n_total, 403, smp)) v = bf(X[k * n_total + smp]);
        }
        S.xt[s][k] = v;
    }
    if (t < kTile) {
        float y = 0.0f;
        if (t < n_valid) {
            const long long smp = sample_of(map, pos0 + t);
            if (MRIP_CHECK(smp >= 0 && smp < n_total, 404, smp)) y = Y[smp];
        }
        S.ys[t] = y;
    }
}

// Forward and backward passes of the staged tile (batch size B_scale for the
// loss gradient 2 r / B).  Leaves h1, h2, dz1, dz2, dy and the squared
// residuals (in ys) in S.
__device__ void tile_passes(GradSmem& S, int d_in, int n_valid, float B_scale) {
    const int t = threadIdx.x;
    const int s = t >> 3;  // sample of this thread for the per-sample passes
    const int g = t & 7;   // its slice of units: g, g + 8, ..., g + 56
    // layer 1
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int u = g + 8 * i;
        float acc = 0.0f;
        for (int k = 0; k < d_in; ++k) acc = fmaf(S.xt[s][k], S.w1t[k][u], acc);
        const float h = fmaxf(acc + S.b1[u], 0.0f);
        S.h1[s][u] = h;
        S.h1t[s][u] = bf(h);
    }
    __syncthreads();
    // layer 2: thread = 2 samples x 4 units, operands read once per 8 FMAs
    {
        const int v0 = 4 * (t & 15), s0 = 2 * (t >> 4);
        float acc[2][4] = {};
#pragma unroll 8
        for (int u = 0; u < H; ++u) {
            const float a0 = S.h1t[s0][u], a1 = S.h1t[s0 + 1][u];
            const float4 w = *reinterpret_cast<const float4*>(&S.w2t[u][v0]);
            acc[0][0] = fmaf(a0, w.x, acc[0][0]);
            acc[0][1] = fmaf(a0, w.y, acc[0][1]);
            acc[0][2] = fmaf(a0, w.z, acc[0][2]);
            acc[0][3] = fmaf(a0, w.w, acc[0][3]);
            acc[1][0] = fmaf(a1, w.x, acc[1][0]);
            acc[1][1] = fmaf(a1, w.y, acc[1][1]);
            acc[1][2] = fmaf(a1, w.z, acc[1][2]);
            acc[1][3] = fmaf(a1, w.w, acc[1][3]);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float h = fmaxf(acc[j][i] + S.b2[v0 + i], 0.0f);
                S.h2[s0 + j][v0 + i] = h;
                S.h2t[s0 + j][v0 + i] = bf(h);
            }
    }
    __syncthreads();
    // output and residual (8 threads per sample, lanes 8s'..8s'+7 of a warp)
    {
        float part = 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i) part = fmaf(S.h2t[s][g + 8 * i], S.w3[g + 8 * i], part);
        part += __shfl_xor_sync(0xFFFFFFFFu, part, 1);
        part += __shfl_xor_sync(0xFFFFFFFFu, part, 2);
        part += __shfl_xor_sync(0xFFFFFFFFu, part, 4);
        if (g == 0) {
            const bool valid = s < n_valid;
            const float r = valid ? (part + S.b3) - S.ys[s] : 0.0f;
            S.dy[s] = valid ? 2.0f * r / B_scale : 0.0f;
            S.ys[s] = r * r;  // reuse: squared residual
        }
    }
    __syncthreads();
    // dz2 = dyhat W3~ [z2 > 0]
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int v = g + 8 * i;
        const float d = S.h2[s][v] > 0.0f ? S.dy[s] * S.w3[v] : 0.0f;
        S.dz2[s][v] = d;
        S.dz2t[s][v] = bf(d);
    }
    __syncthreads();
    // dz1 = (dz2~ W2~) [z1 > 0], same blocking
    {
        const int u0 = 4 * (t & 15), s0 = 2 * (t >> 4);
        float acc[2][4] = {};
#pragma unroll 8
        for (int v = 0; v < H; ++v) {
            const float a0 = S.dz2t[s0][v], a1 = S.dz2t[s0 + 1][v];
            const float4 w = *reinterpret_cast<const float4*>(&S.w2[v][u0]);
            acc[0][0] = fmaf(a0, w.x, acc[0][0]);
            acc[0][1] = fmaf(a0, w.y, acc[0][1]);
            acc[0][2] = fmaf(a0, w.z, acc[0][2]);
            acc[0][3] = fmaf(a0, w.w, acc[0][3]);
            acc[1][0] = fmaf(a1, w.x, acc[1][0]);
            acc[1][1] = fmaf(a1, w.y, acc[1][1]);
            acc[1][2] = fmaf(a1, w.z, acc[1][2]);
            acc[1][3] = fmaf(a1, w.w, acc[1][3]);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                S.dz1[s0 + j][u0 + i] = S.h1[s0 + j][u0 + i] > 0.0f ? acc[j][i] : 0.0f;
    }
    __syncthreads();
}

// The tile's gradient into out[0 .. P) and its squared-residual sum into
// *loss (every parameter has one owner thread).
__device__ void tile_write(const GradSmem& S, int d_in, float* out, float* loss) {
    const int t = threadIdx.x;
    {  // dW2: thread = 4 x 4 block, two float4 loads per 16 FMAs
        const int v0 = 4 * (t >> 4), u0 = 4 * (t & 15);
        float acc[4][4] = {};
#pragma unroll 4
        for (int q = 0; q < kTile; ++q) {
            const float4 a = *reinterpret_cast<const float4*>(&S.dz2t[q][v0]);
            const float4 b = *reinterpret_cast<const float4*>(&S.h1t[q][u0]);
            const float av[4] = {a.x, a.y, a.z, a.w};
            const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                out[off_w2(d_in) + (v0 + i) * H + u0 + j] = acc[i][j];
            }
    }
    for (int i = t; i < H * d_in; i += kGradThreads) {
        const int u = i / d_in, k = i - u * d_in;
        float acc = 0.0f;
        for (int q = 0; q < kTile; ++q) acc = fmaf(bf(S.dz1[q][u]), S.xt[q][k], acc);
        out[i] = acc;
    }
    if (t < H) {
        float a3 = 0.0f, a2 = 0.0f, a1 = 0.0f;
        for (int q = 0; q < kTile; ++q) {
            a3 = fmaf(S.dy[q], S.h2t[q][t], a3);
            a2 += S.dz2[q][t];
            a1 += S.dz1[q][t];
        }
        out[off_w3(d_in) + t] = a3;
        out[off_b2(d_in) + t] = a2;
        out[off_b1(d_in) + t] = a1;
    }
    if (t == H) {
        float a = 0.0f, l = 0.0f;
        for (int q = 0; q < kTile; ++q) {
            a += S.dy[q];
            l += S.ys[q];
        }
        out[off_b3(d_in)] = a;
        *loss = l;
    }
}

// Forward + backward of one tile of kTile samples; partial[blockIdx][p] gets
// the tile's gradient, partial_loss[blockIdx] its sum of squared residuals.
__global__ void __launch_bounds__(kGradThreads) mlp_grad_kernel(
    const float* __restrict__ theta, int d_in, const float* __restrict__ X, long long n_total,
    const float* __restrict__ Y, SampleMap map, long long B, float* __restrict__ partial,
    float* __restrict__ partial_loss) {
    extern __shared__ unsigned char smem_raw[];
    GradSmem& S = *reinterpret_cast<GradSmem*>(smem_raw);
    const long long base = static_cast<long long>(blockIdx.x) * kTile;
    const int n_valid = static_cast<int>(min(static_cast<long long>(kTile), B - base));
    stage_weights(S, theta, d_in);
    stage_tile(S, d_in, X, n_total, Y, map, base, n_valid);
    __syncthreads();
    tile_passes(S, d_in, n_valid, static_cast<float>(B));
    tile_write(S, d_in, partial + static_cast<long long>(blockIdx.x) * n_params(d_in),
                      partial_loss + blockIdx.x);
}

// grad[p] = sum over CTAs of partial[c][p] (fixed order); optionally Adam.
template <bool kAdam>
__global__ void mlp_reduce_kernel(const float* __restrict__ partial, const float* __restrict__ partial_loss,
                                  int n_cta, long long P, long long B, float* __restrict__ grad,
                                  float* __restrict__ loss, float* __restrict__ theta, float* __restrict__ m,
                                  float* __restrict__ v, float lr, float beta1, float beta2, float eps,
                                  float bc1, float bc2) {
    const long long p = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    if (p < P) {
        float acc = 0.0f;
        for (int c = 0; c < n_cta; ++c) acc += partial[static_cast<long long>(c) * P + p];
        if (grad) grad[p] = acc;
        if (kAdam) {
            const float mi = beta1 * m[p] + (1.0f - beta1) * acc;
            const float vi = beta2 * v[p] + (1.0f - beta2) * acc * acc;
            m[p] = mi;
            v[p] = vi;
            const float mhat = mi / bc1;
            const float vhat = vi / bc2;
            theta[p] = theta[p] - lr * mhat / (sqrtf(vhat) + eps);
        }
    }
    if (p == 0 && loss) {
        float l = 0.0f;
        for (int c = 0; c < n_cta; ++c) l += partial_loss[c];
        *loss = l / static_cast<float>(B);
    }
}

__global__ void adam_kernel(float* __restrict__ theta, float* __restrict__ m, float* __restrict__ v,
                            const float* __restrict__ g, long long n, float lr, float beta1, float beta2,
                            float eps, float bc1, float bc2) {
    const long long p = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
    if (p >= n) return;
    const float gi = g[p];
    const float mi = beta1 * m[p] + (1.0f - beta1) * gi;
    const float vi = beta2 * v[p] + (1.0f - beta2) * gi * gi;
    m[p] = mi;
    v[p] = vi;
    theta[p] = theta[p] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
}

// ---------------------------------------------------------------------------
// Whole training run in one launch (mlp_train_tc_kernel below): a cluster of
// CTAs keeps the network in shared memory for all epochs.
// ---------------------------------------------------------------------------
struct TrainArgs {
    const float* X;  // standardised features, d_in planes of n_tr
    const float* Y;
    long long n_tr, B, steps_per_epoch;
    int epochs, d_in;
    const unsigned long long* ab;  // per epoch: the affine order (a, b)
    const float* bc;               // per step: the bias corrections (1 - beta1^t, 1 - beta2^t)
    float lr, beta1, beta2, eps;
    float* theta;   // in: initial parameters; out: trained (the best epoch's with validation)
    float* losses;  // per step: mean squared residual of the minibatch (may be null)
    long long max_steps;  // > 0: stop after this many steps
    float* grad;    // may be null: the gradient of the last step
    float* m_out;   // may be null: Adam's first moment after the last step
    float* v_out;   // may be null: Adam's second moment after the last step
    const float* Xv;  // validation features, d_in planes of n_val (n_val = 0: none)
    const float* Yv;
    long long n_val;
    int patience;       // > 0: stop after this many epochs without a lower validation loss
    float* val_losses;  // per epoch (may be null)
    int* info;          // may be null: epochs run, epoch kept, steps run
    const float* m_in;  // may be null (zero): Adam's moments to resume from
    const float* v_in;
    float best0;        // validation loss to beat (+inf: none yet)
    int bad0;           // epochs without a lower validation loss so far
    const float* theta_in;  // may be null (= theta): the parameters to start from
    float* theta_last;      // may be null: the parameters after the last step run
};

// ---------------------------------------------------------------------------
// Training with the five contractions of a step on the tensor cores (tcgen05,
// FP32 accumulators in tensor memory).  A cluster of kTcCluster CTAs keeps the
// BF16 operands of the weights in every CTA's shared memory and the FP32
// parameters with Adam's moments in registers, spread over the cluster; per
// step each CTA takes 1/kTcCluster of the minibatch in tiles of 128 samples
// (sample m = TMEM lane m, its 64 columns split over 4 of the 512 workers):
//   Z1  = X~ W1~^T        (M 128, N 64, K 16: the d_in features, zero-padded)
//   Z2  = H1~ W2~^T       (K 64)
//   dH1 = dZ2~ W2~        (K 64, W2~ read MN-major)
//   dW2 = dZ2~^T H1~      (K = the 128 samples, both read MN-major)
//   dW1 = dZ1~^T X~       (N 16, likewise)
// Activations and deltas are written once, as rows (16-byte stores), and read
// by the tensor cores along either index; the last two products are taken at
// M = 128, whose rows 64.. read neighbouring bytes and are not used.  Each
// worker turns its 16 columns of a row of Z1 / Z2 / dH1 into activations,
// residual and deltas (FP32, rounded to BF16 where the next contraction reads
// them; a unit is off where its BF16 activation has its sign set, see relu_signed).  The bias and W3 gradients are FP32 column
// sums over the tile in a fixed order (chunks of 16 samples, then the chunks
// in order), taken while the products run.  Four more warps: one issues the
// products, one adds the output deltas and the squared residuals one after
// the other, two fetch samples.
//
// CTA r owns hidden units 8r .. 8r + 7 of both layers: a CTA's gradient lies in
// shared memory as one block per owner and is sent to the owners' shared memory
// as bulk copies that complete on the owner's mbarrier; a thread of the owner adds its
// one word over the 8 CTAs in rank order, applies Adam and writes the new value
// as the operand it is used as, again into one block, which is sent to the other
// CTAs in the same way.  No cluster barrier is needed in a step: an owner sends
// the weights of a step only once every CTA's gradient has arrived, so nothing of
// the old weights is still read, and a CTA starts the next step only once every
// owner's weights have arrived, so nothing of its gradient or of the owners'
// receive buffers is still read.
//
// What bounds it: a step is a chain of latencies on 8 SMs (three products, one
// after the other, and two exchanges in the cluster; the gradient of a step
// needs the weights of the one before, and the order of additions is kept, so
// more SMs would not shorten it), so everything that can leaves the chain: the
// samples are copied behind the products (loads into registers were waited for
// at the next loop), the sums run behind the products, the next tile's operand
// is built while the weights are under way.  The kernel before, at 13.0 us a
// step, held two transposed operand copies (4,000 of 24,000 cycles), additions of
// the gradient in shared memory with 32-way bank conflicts (2,600), rounding of
// all weights by every CTA (1,850), remote loads and stores of single words and
// two cluster barriers (6,500), the samples' loads (2,500) and a serial sum
// (1,900).  Measured, 94,208 samples of 8 inputs in minibatches of 1,024 and 12,288
// validation samples, one epoch: 1.21 -> 0.63 ms (6.5 us a step).
//
// Every wait has an iteration limit; on a timeout a thread stops waiting, no
// more products are issued, everything runs on to the same barriers (so no peer
// waits forever), waits once more, with the limit, for what is in flight, and
// *err reports it.
// ---------------------------------------------------------------------------
constexpr int kTcCluster = 8;
constexpr int kTcWorkers = 512;              // 4 threads per sample row, 16 columns each
constexpr int kTcThreads = kTcWorkers + 128;  // and the issuing, the adding and two fetching warps
constexpr int kTcRows = 128;
constexpr int kTcChunks = kTcWorkers / H;    // row chunks of the column sums
constexpr int kTcWait = 1 << 22;
constexpr int kTcUnits = H / kTcCluster;     // hidden units per owner
constexpr int kRowF = H + 4, kRowB = H + 8;  // row strides of the FP32 and BF16 tiles: 16-byte stores of
                                             // eight neighbouring rows fall on different banks
static_assert(kTcUnits == 8, "an owner's rows are one group of core matrices");

// An owner's part of the weights, as it is used.
struct TcWeights {
    unsigned char w2[kTcUnits * H * 2];   // W2~ [v][u], one row group of core matrices
    unsigned char w1[kTcUnits * 16 * 2];  // W1~ [u][k], k padded to 16
    float b1[kTcUnits], b2[kTcUnits];
    float w3[kTcUnits];                   // rounded to BF16
    float b3;                             // (owner 0)
    float pad[7];
};
constexpr uint32_t kWStride = sizeof(TcWeights);
static_assert(kWStride == 1408 && kWStride % 128 == 0, "row groups of the weight operands lie kWStride apart");

// An owner's part of the gradient: W2 as 8 rows of 65 words, W1 as 8 rows of
// d + 1 (odd strides: the rows of a warp's lanes fall on different banks, also
// across owners, kGradWords being 8 modulo 32), b1, b2, W3, then (owner 0) b3
// and the sum of squared residuals.
constexpr int kGradWords = 648;
__host__ __device__ constexpr int grad_w1() { return kTcUnits * (H + 1); }
__host__ __device__ constexpr int grad_b1(int d) { return grad_w1() + kTcUnits * (d + 1); }
__host__ __device__ constexpr int grad_b3(int d) { return grad_b1(d) + 3 * kTcUnits; }
__host__ __device__ constexpr int grad_loss(int d) { return grad_b3(d) + 1; }
static_assert(grad_loss(kMaxIn) < kGradWords && grad_loss(kMaxIn) <= kTcThreads, "a block, and the threads, hold its words");

struct TcSmem {
    alignas(1024) unsigned char a1[kTcRows * 16 * 2];      // X~ rows, 16 columns
    alignas(1024) unsigned char a2[kTcRows * H * 2];       // H1~ rows
    alignas(1024) unsigned char a3[kTcRows * H * 2];       // dZ2~ rows
    alignas(1024) unsigned char a4[kTcRows * H * 2];       // dZ1~ rows
    alignas(128) TcWeights w[kTcCluster];
    alignas(16) float dz1[kTcRows][kRowF];                 // dZ1, FP32
    alignas(16) __nv_bfloat16 h2t[kTcRows][kRowB];         // H2~ rows (for dW3)
    alignas(16) float part[kTcCluster][kGradWords];        // this CTA's gradient, by owner
    alignas(16) float recv[kTcCluster][kGradWords];        // this owner's gradient, by CTA
    float ypart[4][kTcRows];                               // output partials per column block
    float colpart[3][kTcChunks][H];                        // column sums per row chunk
    alignas(16) float dy[kTcRows];
    alignas(16) float r2[kTcRows];
    float vsum;                                            // validation: this CTA's squared residuals
    uint64_t bar, bar_w2, bar_grad, bar_weights;
    float rows[4][kMaxIn + 1][kTcRows];                    // samples fetched: features, target; two tiles of
                                                           // a step and two of the validation samples
    float bc[2][2];                                        // Adam's bias corrections of this step and the next
    uint32_t tmem;
};
static_assert(sizeof(TcSmem) <= 227 * 1024, "fits a CTA's shared memory");

// What word e of owner r's gradient block belongs to: the parameter's index (-1:
// padding), the byte it is used at within TcWeights and how.
enum ParamUse { kUseBf16, kUseRounded, kUseFp32 };
__device__ __forceinline__ int owned_param(int e, int r, int d, uint32_t& at, ParamUse& use) {
    at = 0;
    use = kUseBf16;
    if (e < grad_w1()) {
        const int row = e / (H + 1), u = e % (H + 1);
        if (u == H) return -1;
        at = static_cast<uint32_t>(offsetof(TcWeights, w2)) + tc::core_offset(row, u, H);
        return static_cast<int>(off_w2(d)) + (kTcUnits * r + row) * H + u;
    }
    if (e < grad_b1(d)) {
        const int row = (e - grad_w1()) / (d + 1), k = (e - grad_w1()) % (d + 1);
        if (k == d) return -1;
        at = static_cast<uint32_t>(offsetof(TcWeights, w1)) + tc::core_offset(row, k, 16);
        return (kTcUnits * r + row) * d + k;
    }
    use = kUseFp32;
    if (e < grad_b3(d)) {
        const int i = e - grad_b1(d), unit = i % kTcUnits;
        const int which = i / kTcUnits;
        at = static_cast<uint32_t>(which == 0 ? offsetof(TcWeights, b1) : which == 1 ? offsetof(TcWeights, b2)
                                                                                     : offsetof(TcWeights, w3)) +
             4u * unit;
        if (which == 2) use = kUseRounded;
        return static_cast<int>(which == 0 ? off_b1(d) : which == 1 ? off_b2(d) : off_w3(d)) + kTcUnits * r + unit;
    }
    at = static_cast<uint32_t>(offsetof(TcWeights, b3));
    return e == grad_b3(d) && r == 0 ? static_cast<int>(off_b3(d)) : -1;
}

__device__ __forceinline__ void put_weight(TcWeights& w, uint32_t at, ParamUse use, float v) {
    unsigned char* dst = reinterpret_cast<unsigned char*>(&w) + at;
    if (use == kUseBf16)
        *reinterpret_cast<__nv_bfloat16*>(dst) = __float2bfloat16_rn(v);
    else
        *reinterpret_cast<float*>(dst) = use == kUseRounded ? bf(v) : v;
}

// max(x, 0), zero with a sign where the unit is off: BF16 rounds 0 < x <= 2^-134 to zero
// too, but such a unit is on.
__device__ __forceinline__ float relu_signed(float x) { return x > 0.0f ? x : -0.0f; }

// Eight FP32 values rounded to BF16 (nearest even), the first at the lowest
// address: one core-matrix row of 16 bytes.
__device__ __forceinline__ uint4 pack_bf16x8(const float* w) {
    uint32_t r[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const __nv_bfloat162 p = __floats2bfloat162_rn(w[2 * q], w[2 * q + 1]);
        r[q] = *reinterpret_cast<const uint32_t*>(&p);
    }
    return make_uint4(r[0], r[1], r[2], r[3]);
}

__global__ void __cluster_dims__(kTcCluster, 1, 1) __launch_bounds__(kTcThreads, 1)
    mlp_train_tc_kernel(TrainArgs ta, int* err) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(1024) unsigned char tc_raw[];
    TcSmem& S = *reinterpret_cast<TcSmem*>(tc_raw);
    const int d_in = ta.d_in;
    const int rank = static_cast<int>(cluster.block_rank());
    const int t = threadIdx.x, lane = t & 31;
    const int warp = __shfl_sync(0xFFFFFFFFu, t >> 5, 0);  // (known to be the same in a warp)
    const bool worker = t < kTcWorkers;
    const bool issuer = warp == kTcWorkers / 32;    // the warp that issues products
    const bool sends = warp < kTcCluster && warp != rank && lane == 0;  // blocks to CTA `warp` (a warp each: 60 cycles)
    const bool fetcher = warp >= kTcWorkers / 32 + 2;  // the two warps that fetch samples
    const bool summer = warp == kTcWorkers / 32 + 1 && lane < 2;  // lane 0 adds the outputs' deltas, 1 the squared residuals
    const int quarter = warp & 3, cb = warp >> 2;   // TMEM lane quarter, column block
    const int m = 32 * quarter + lane;              // this worker's sample row / TMEM lane
    const int c0 = 16 * cb;                         // its 16 columns
    constexpr uint32_t kIdesc = tc::idesc_bf16(kTcRows, H);
    constexpr uint32_t kIdescH1 = tc::idesc_bf16(kTcRows, H, false, true);
    constexpr uint32_t kIdescW2 = tc::idesc_bf16(kTcRows, H, true, true);
    constexpr uint32_t kIdescW1 = tc::idesc_bf16(kTcRows, 16, true, true);
    // (debug build: the layout must fit the launch's shared memory; every CTA
    // of the cluster leaves together, before any cluster barrier or
    // tensor-memory allocation)
    if (!MRIP_CHECK(sizeof(TcSmem) <= dynamic_smem_bytes(), 402, sizeof(TcSmem))) {
        if (t == 0 && rank == 0) atomicExch(err, 1);
        return;
    }

    if (warp == 0) tc::tmem_alloc(&S.tmem, 256);
    if (t == 0) {
        tc::mbar_init(&S.bar);
        tc::mbar_init(&S.bar_w2);
        tc::mbar_init(&S.bar_grad);
        tc::mbar_init(&S.bar_weights);
    }
    for (int i = t; i < kTcRows * 16 * 2 / 16; i += kTcThreads)
        reinterpret_cast<uint4*>(S.a1)[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int i = t; i < static_cast<int>(sizeof(S.w) / 16); i += kTcThreads)
        reinterpret_cast<uint4*>(S.w)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    const float* th_src = ta.theta_in ? ta.theta_in : ta.theta;
    for (int i = t; i < kTcCluster * grad_loss(d_in); i += kTcThreads) {
        uint32_t at;
        ParamUse use;
        const int r = i / grad_loss(d_in);
        const int p = owned_param(i - r * grad_loss(d_in), r, d_in, at, use);
        if (p >= 0) put_weight(S.w[r], at, use, th_src[p]);
    }
    // this thread's parameter: word t of the owner's block
    uint32_t at = 0;
    ParamUse use = kUseFp32;
    const int par = t <= grad_b3(d_in) ? owned_param(t, rank, d_in, at, use) : -1;
    float th = par >= 0 ? th_src[par] : 0.0f;
    float mom = (ta.m_in && par >= 0) ? ta.m_in[par] : 0.0f;
    float vel = (ta.v_in && par >= 0) ? ta.v_in[par] : 0.0f;
    tc::fence_smem_async();
    tc::fence_before_sync();
    cluster.sync();
    tc::fence_after_sync();
    const uint32_t tm = S.tmem;
    const uint32_t lane_base = static_cast<uint32_t>(32 * quarter) << 16;
    uint32_t phase = 0, phase_w2 = 0, phase_grad = 0, phase_weights = 0;
    bool ok = true;  // of this thread

    auto wait_on = [&](uint64_t* bar, uint32_t& ph) {
        if (ok && !tc::mbar_wait(bar, ph, kTcWait)) {
            ok = false;
            atomicExch(err, 1);
        }
        ph ^= 1u;
    };
    auto wait_mma = [&]() {
        wait_on(&S.bar, phase);
        tc::fence_after_sync();
    };
    auto sync_for_mma = [&]() {
        tc::fence_smem_async();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
    };
    // the same without the fetching warps, which may be waiting for memory
    auto sync_for_mma_tile = [&]() {
        tc::fence_smem_async();
        tc::fence_before_sync();
        tc::sync_threads(2, kTcThreads - 64);
        tc::fence_after_sync();
    };
    bool pending = false;  // weights on their way
    auto settle = [&]() {
        if (pending) wait_on(&S.bar_weights, phase_weights);
        pending = false;
    };
    // a block of this CTA to `dst` in CTA `to`, completing on its mbarrier `bar`
    auto send = [&](const void* src, uint32_t bytes, const void* dst, uint64_t* bar, int to) {
        tc::bulk_to_cta(tc::cluster_addr(tc::smem_addr(dst), to), tc::smem_addr(src), bytes,
                        tc::cluster_addr(tc::smem_addr(bar), to));
    };

    // Sample smp into column `col` of S.rows[buf], asynchronously (zeros if !valid).
    auto copy_row = [&](int buf, int col, const float* Xs, const float* Ys, long long n_total, long long smp, bool valid) {
        const float* x = valid ? Xs + smp : Xs;
        for (int k = 0; k < d_in; ++k, x += valid ? n_total : 0) tc::copy4(tc::smem_addr(&S.rows[buf][k][col]), x, valid);
        tc::copy4(tc::smem_addr(&S.rows[buf][kMaxIn][col]), valid ? Ys + smp : Ys, valid);
    };
    // this worker's 16 words of a per-unit array
    auto units16 = [&](const float* first, float (&v)[16]) {
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const float4 a = *reinterpret_cast<const float4*>(
                reinterpret_cast<const unsigned char*>(first) + (2 * cb + (g >> 1)) * kWStride + 16 * (g & 1));
            v[4 * g] = a.x;
            v[4 * g + 1] = a.y;
            v[4 * g + 2] = a.z;
            v[4 * g + 3] = a.w;
        }
    };
    // v = 0 for the units that are off, by the signs of their activations, two times eight at h0 and h1
    auto zero_where_off = [&](const void* h0, const void* h1, float (&v)[16]) {
        const uint4 p = *static_cast<const uint4*>(h0), q = *static_cast<const uint4*>(h1);
        const uint32_t w[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
            v[j] = (w[j / 2] & 0x8000u) ? 0.0f : v[j];
            v[j + 1] = (w[j / 2] & 0x80000000u) ? 0.0f : v[j + 1];
        }
    };
    auto store16 = [&](float (*tile)[kRowF], const float (&v)[16]) {
#pragma unroll
        for (int g = 0; g < 4; ++g)
            *reinterpret_cast<float4*>(&tile[m][c0 + 4 * g]) =
                make_float4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
    };
    auto store16_bf = [&](unsigned char* operand, const float (&v)[16]) {
        *reinterpret_cast<uint4*>(operand + tc::core_offset(m, c0, H)) = pack_bf16x8(v);
        *reinterpret_cast<uint4*>(operand + tc::core_offset(m, c0 + 8, H)) = pack_bf16x8(v + 8);
    };

    // Forward pass of the tile in S.rows[buf] (not the fetching warps).  Leaves X~,
    // H1~ and H2~ rows in shared memory (their signs are the ReLU masks); returns the output of row m without b3 (workers).
    auto forward_tile = [&](int buf) -> float {
        if (worker) {
            const float x0 = 2 * cb < d_in ? S.rows[buf][2 * cb][m] : 0.0f;
            const float x1 = 2 * cb + 1 < d_in ? S.rows[buf][2 * cb + 1][m] : 0.0f;
            *reinterpret_cast<__nv_bfloat162*>(S.a1 + tc::core_offset(m, 2 * cb, 16)) = __floats2bfloat162_rn(x0, x1);
        }
        settle();
        sync_for_mma_tile();
        if (issuer && __all_sync(0xFFFFFFFFu, ok)) {
            tc::mma_bf16(tm, tc::smem_desc(tc::smem_addr(S.a1), 128, 256),
                         tc::smem_desc(tc::smem_addr(S.w[0].w1), 128, kWStride), kIdesc, false);
            tc::mma_commit(&S.bar);
        }
        if (worker) {
            wait_mma();
            // layer 1 epilogue: h1 = relu(z1 + b1) on columns c0 .. c0 + 15
            float z[16], b[16];
            units16(S.w[0].b1, b);
            tc::tmem_ld16(tm + lane_base + c0, z);
#pragma unroll
            for (int j = 0; j < 16; ++j) z[j] = relu_signed(z[j] + b[j]);
            store16_bf(S.a2, z);
        }
        sync_for_mma_tile();
        if (issuer && __all_sync(0xFFFFFFFFu, ok)) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                tc::mma_bf16(tm + 64, tc::smem_desc(tc::smem_addr(S.a2) + 256 * ks, 128, 1024),
                             tc::smem_desc(tc::smem_addr(S.w[0].w2) + 256 * ks, 128, kWStride), kIdesc, ks > 0);
            tc::mma_commit(&S.bar);
        }
        if (worker) {
            float z[16], b[16], yp = 0.0f;
            units16(S.w[0].b2, b);
            wait_mma();
            // layer 2 epilogue: h2 and this block's share of the output
            tc::tmem_ld16(tm + lane_base + 64 + c0, z);
#pragma unroll
            for (int j = 0; j < 16; ++j) z[j] = relu_signed(z[j] + b[j]);
            units16(S.w[0].w3, b);
            const uint4 packed[2] = {pack_bf16x8(z), pack_bf16x8(z + 8)};
            const uint32_t* word = &packed[0].x;
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
                yp = fmaf(__uint_as_float(word[j / 2] << 16), b[j], yp);
                yp = fmaf(__uint_as_float(word[j / 2] & 0xFFFF0000u), b[j + 1], yp);
            }
            *reinterpret_cast<uint4*>(&S.h2t[m][c0]) = packed[0];
            *reinterpret_cast<uint4*>(&S.h2t[m][c0 + 8]) = packed[1];
            S.ypart[cb][m] = yp;
            tc::sync_threads(1, kTcWorkers);
        }
        return worker ? ((S.ypart[0][m] + S.ypart[1][m]) + S.ypart[2][m]) + S.ypart[3][m] : 0.0f;
    };
    // sum += values[first .. first + 64) in order
    auto add64 = [&](const float* values, int first, float& sum) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float4 v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = *reinterpret_cast<const float4*>(values + first + 32 * h + 4 * q);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                sum += v[q].x;
                sum += v[q].y;
                sum += v[q].z;
                sum += v[q].w;
            }
        }
    };

    // x mod n by a 64-bit reciprocal
    const unsigned long long n_mod = static_cast<unsigned long long>(ta.n_tr);
    const unsigned long long n_inv = ~0ull / n_mod;
    auto mod_n = [&](unsigned long long x) {
        unsigned long long r = x - __umul64hi(x, n_inv) * n_mod;
        if (r >= n_mod) r -= n_mod;  // (the quotient is at most 2 too small)
        if (r >= n_mod) r -= n_mod;
        return static_cast<long long>(r);
    };
    // positions lo .. hi - 1 of the minibatch of nb samples at `off` are this CTA's
    auto split = [&](long long nb, long long& lo, long long& hi) {
        const long long chunk = (nb + kTcCluster - 1) / kTcCluster;
        lo = min(nb, rank * chunk);
        hi = min(nb, lo + chunk);
    };
    long long full_lo, full_hi;
    split(ta.B, full_lo, full_hi);
    auto share = [&](long long off, long long& nb, long long& lo, long long& hi) {
        if (off + ta.B <= ta.n_tr) {
            nb = ta.B;
            lo = full_lo;
            hi = full_hi;
        } else {
            nb = ta.n_tr - off;
            split(nb, lo, hi);
        }
    };
    // the tile at position p0 of the minibatch at `off` into S.rows[buf], by the two fetching warps
    auto fetch = [&](int buf, unsigned long long a, unsigned long long b, long long off, long long p0, long long hi) {
        for (int col = t - (kTcThreads - 64); col < kTcRows; col += 64) {
            bool valid = p0 + col < hi;
            const long long smp = mod_n(a * static_cast<unsigned long long>(off + p0 + col) + b);
            if (valid && !MRIP_CHECK(smp >= 0 && smp < ta.n_tr, 401, smp)) valid = false;
            copy_row(buf, col, ta.X, ta.Y, ta.n_tr, smp, valid);
        }
    };
    auto fetch_bc = [&](long long of) {
        const int i = t - (kTcThreads - 64);
        if (i < 2) tc::copy4(tc::smem_addr(&S.bc[of & 1][i]), ta.bc + 2 * of + i, true);
    };
    auto fetch_val = [&](int buf, long long p0, long long hi) {
        for (int col = t - (kTcThreads - 64); col < kTcRows; col += 64)
            copy_row(buf, col, ta.Xv, ta.Yv, ta.n_val, p0 + col, p0 + col < hi);
    };

    long long step = 0;
    bool stop = false;
    float best = ta.best0;
    int bad = ta.bad0, best_epoch = 0, epochs_run = 0;
    unsigned long long oa = 0, ob = 0;  // this epoch's order (fetching warps)
    if (fetcher) {
        oa = ta.ab[0];
        ob = ta.ab[1];
    }
    int buf = 0;  // of the next tile's samples
    long long nb, lo, hi;
    share(0, nb, lo, hi);
    if (fetcher) {
        fetch(buf, oa, ob, 0, lo, hi);
        fetch_bc(0);
        tc::copy_wait();
    }
    __syncthreads();
    for (int ep = 0; ep < ta.epochs && !stop; ++ep) {
        const bool more = ep + 1 < ta.epochs;
        unsigned long long na = 0, nb_ = 0;
        if (fetcher && more) {
            na = ta.ab[2 * ep + 2];
            nb_ = ta.ab[2 * ep + 3];
        }
        for (long long off = 0; off < ta.n_tr; off += ta.B, ++step) {
            if (ta.max_steps > 0 && step >= ta.max_steps) {  // uniform across the cluster
                stop = true;
                break;
            }
            share(off, nb, lo, hi);
            // the tile after position p0's: this step's or the next one's
            auto fetch_ahead = [&](long long p0) {
                if (p0 + kTcRows < hi) {
                    fetch(buf, oa, ob, off, p0 + kTcRows, hi);
                } else if (off + ta.B < ta.n_tr || more) {
                    const bool same = off + ta.B < ta.n_tr;
                    const long long xoff = same ? off + ta.B : 0;
                    long long xnb, xlo, xhi;
                    share(xoff, xnb, xlo, xhi);
                    fetch(buf, same ? oa : na, same ? ob : nb_, xoff, xlo, xhi);
                    if (ta.max_steps <= 0 || step + 1 < ta.max_steps) fetch_bc(step + 1);
                }
            };
            // the blocks of this step, from the 7 other CTAs (after settle())
            auto expect = [&]() {
                if (t == kTcWorkers) {
                    tc::mbar_expect(&S.bar_grad, (kTcCluster - 1) * kGradWords * 4);
                    tc::mbar_expect(&S.bar_weights, (kTcCluster - 1) * kWStride);
                }
            };
            if (lo >= hi) {  // no sample of a small minibatch is this CTA's
                settle();
                expect();
                for (int i = t; i < kTcCluster * kGradWords; i += kTcThreads) (&S.part[0][0])[i] = 0.0f;
                if (fetcher) {
                    fetch_ahead(lo);
                    tc::copy_wait();
                }
            }

            for (long long p0 = lo; p0 < hi; p0 += kTcRows) {
                const bool first = p0 == lo;
                // (adds to a tile's predecessor; the first tile starts from zero)
                auto put = [&](float& dst, float v) {
                    if (first)
                        dst = 0.0f + v;
                    else
                        dst += v;
                };
                buf ^= 1;
                if (fetcher) {
                    settle();  // (then, behind the first product)
                    fetch_ahead(p0);
                    tc::copy_wait();
                } else {
                    const float yhat = forward_tile(buf ^ 1);
                    if (first) expect();
                    if (worker) {
                        const bool valid = p0 + m < hi;
                        const float r = valid ? (yhat + S.w[0].b3) - S.rows[buf ^ 1][kMaxIn][m] : 0.0f;
                        const float dyv = valid ? 2.0f * r / static_cast<float>(nb) : 0.0f;
                        if (cb == 0) {
                            S.dy[m] = dyv;
                            S.r2[m] = r * r;
                        }
                        float d[16];
                        units16(S.w[0].w3, d);
#pragma unroll
                        for (int j = 0; j < 16; ++j) d[j] = dyv * d[j];
                        zero_where_off(&S.h2t[m][c0], &S.h2t[m][c0 + 8], d);
                        store16_bf(S.a3, d);
                    }
                    sync_for_mma_tile();
                    if (issuer && __all_sync(0xFFFFFFFFu, ok)) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks)  // dH1 = dZ2~ W2~
                            tc::mma_bf16(tm, tc::smem_desc(tc::smem_addr(S.a3) + 256 * ks, 128, 1024),
                                         tc::smem_desc(tc::smem_addr(S.w[0].w2) + 2 * kWStride * ks, kWStride, 128),
                                         kIdescH1, ks > 0);
                        tc::mma_commit(&S.bar);
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)  // dW2 = dZ2~^T H1~
                            tc::mma_bf16(tm + 128, tc::smem_desc(tc::smem_addr(S.a3) + 2048 * ks, 1024, 128),
                                         tc::smem_desc(tc::smem_addr(S.a2) + 2048 * ks, 1024, 128), kIdescW2, ks > 0);
                        tc::mma_commit(&S.bar_w2);
                    }
                    if (worker) {
                        // meanwhile: column sums of dZ2 (b2: dy w3 where the unit is on) and, by
                        // the odd column blocks' warps, of dy h2~ (W3); a chunk of 16 rows per
                        // warp, two columns per lane
                        const int chunk = 4 * (cb >> 1) + quarter, q0 = 16 * chunk;
                        float2 a = make_float2(0.0f, 0.0f);
                        float dy[16];
                        uint32_t h[16];
#pragma unroll
                        for (int q = 0; q < 16; q += 4) {
                            const float4 d = *reinterpret_cast<const float4*>(&S.dy[q0 + q]);
                            dy[q] = d.x;
                            dy[q + 1] = d.y;
                            dy[q + 2] = d.z;
                            dy[q + 3] = d.w;
                        }
#pragma unroll
                        for (int q = 0; q < 16; ++q) h[q] = *reinterpret_cast<const uint32_t*>(&S.h2t[q0 + q][2 * lane]);
                        if ((cb & 1) == 0) {
                            const float2 w3 = *reinterpret_cast<const float2*>(&S.w[lane / 4].w3[2 * (lane % 4)]);
#pragma unroll
                            for (int q = 0; q < 16; ++q) {  // (no fma: dZ2 is rounded)
                                a.x = __fadd_rn(a.x, (h[q] & 0x8000u) ? 0.0f : __fmul_rn(dy[q], w3.x));
                                a.y = __fadd_rn(a.y, (h[q] & 0x80000000u) ? 0.0f : __fmul_rn(dy[q], w3.y));
                            }
                        } else {
#pragma unroll
                            for (int q = 0; q < 16; ++q) {
                                a.x = fmaf(dy[q], __uint_as_float(h[q] << 16), a.x);
                                a.y = fmaf(dy[q], __uint_as_float(h[q] & 0xFFFF0000u), a.y);
                            }
                        }
                        *reinterpret_cast<float2*>(&S.colpart[cb & 1][chunk][2 * lane]) = a;
                        wait_mma();
                        // dZ1 = dH1 [z1 > 0] (FP32 for b1, BF16 for dW1)
                        float z[16];
                        tc::tmem_ld16(tm + lane_base + c0, z);
                        zero_where_off(S.a2 + tc::core_offset(m, c0, H), S.a2 + tc::core_offset(m, c0 + 8, H), z);
                        store16_bf(S.a4, z);
                        store16(S.dz1, z);
                    } else if (summer) {
                        float sum = 0.0f;
                        add64(lane == 0 ? S.dy : S.r2, 0, sum);
                        add64(lane == 0 ? S.dy : S.r2, 64, sum);
                        put(S.part[0][lane == 0 ? grad_b3(d_in) : grad_loss(d_in)], sum);
                    }
                }
                sync_for_mma();
                if (issuer && __all_sync(0xFFFFFFFFu, ok)) {
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks)  // dW1 = dZ1~^T X~
                        tc::mma_bf16(tm + 192, tc::smem_desc(tc::smem_addr(S.a4) + 2048 * ks, 1024, 128),
                                     tc::smem_desc(tc::smem_addr(S.a1) + 512 * ks, 256, 128), kIdescW1, ks > 0);
                    tc::mma_commit(&S.bar);
                }
                if (worker) {
                    const int chunk = 2 * cb + (quarter & 1), q0 = 16 * chunk;
                    // meanwhile: rows 0..63 (TMEM lanes 0..63) of dW2 and, by the
                    // warps whose TMEM lanes hold no gradient, the column sums of dZ1 (b1)
                    if (quarter < 2) {
                        wait_on(&S.bar_w2, phase_w2);
                        tc::fence_after_sync();
                        float z[16];
                        tc::tmem_ld16(tm + lane_base + 128 + c0, z);
                        float* block = S.part[m / kTcUnits] + (m % kTcUnits) * (H + 1) + c0;
                        if (first) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) block[j] = 0.0f + z[j];
                        } else {
#pragma unroll
                            for (int j = 0; j < 16; ++j) block[j] += z[j];
                        }
                    } else {
                        float2 a = make_float2(0.0f, 0.0f);
#pragma unroll
                        for (int q = 0; q < 16; ++q) {
                            const float2 d = *reinterpret_cast<const float2*>(&S.dz1[q0 + q][2 * lane]);
                            a.x += d.x;
                            a.y += d.y;
                        }
                        *reinterpret_cast<float2*>(&S.colpart[2][chunk][2 * lane]) = a;
                    }
                    tc::sync_threads(1, kTcWorkers);
                    if (quarter >= 2) {  // the chunks of all three
                        const int i = 32 * chunk + lane;
                        if (i < 3 * H) {
                            const int which = i / H, col = i & (H - 1);
                            float s = 0.0f;
#pragma unroll
                            for (int c = 0; c < kTcChunks; ++c) s += S.colpart[which][c][col];
                            const int order = which == 0 ? 1 : which == 1 ? 2 : 0;  // b2, W3, b1 -> b1, b2, W3
                            put(S.part[col / kTcUnits][grad_b1(d_in) + kTcUnits * order + col % kTcUnits], s);
                        }
                    }
                    wait_mma();
                    if (quarter < 2 && 4 * cb < d_in) {  // rows 0..63 of dW1
                        float z[4];
                        tc::tmem_ld4(tm + lane_base + 192 + 4 * cb, z);
                        float* block = S.part[m / kTcUnits] + grad_w1() + (m % kTcUnits) * (d_in + 1) + 4 * cb;
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (4 * cb + k < d_in) put(block[k], z[k]);
                    }
                }
            }
            sync_for_mma();  // the gradient is complete
            if (sends) send(S.part[warp], kGradWords * 4, S.recv[rank], &S.bar_grad, warp);
            wait_on(&S.bar_grad, phase_grad);
            float g = 0.0f;  // this thread's word, of all CTAs (word grad_loss: the squared residuals)
#pragma unroll
            for (int rr = 0; rr < kTcCluster; ++rr) g += rr == rank ? S.part[rr][t] : S.recv[rr][t];
            if (par >= 0) {
                if (ta.grad) ta.grad[par] = g;
                mom = ta.beta1 * mom + (1.0f - ta.beta1) * g;
                vel = ta.beta2 * vel + (1.0f - ta.beta2) * g * g;
                th = th - ta.lr * (mom / S.bc[step & 1][0]) / (sqrtf(vel / S.bc[step & 1][1]) + ta.eps);
                put_weight(S.w[rank], at, use, th);
            }
            sync_for_mma();  // the owner's new weights are written, its receive buffers read
            if (sends) send(&S.w[rank], kWStride, &S.w[rank], &S.bar_weights, warp);
            if (rank == 0 && t == grad_loss(d_in) && ta.losses) ta.losses[step] = g / static_cast<float>(nb);
            pending = true;
        }
        if (stop) break;
        ++epochs_run;
        oa = na;
        ob = nb_;
        if (ta.n_val > 0) {
            // validation loss of this epoch's parameters (each CTA a slice of
            // the validation samples, in order; the CTAs' sums added in rank
            // order, so every CTA computes the same value and takes the same
            // early-stopping decision)
            const long long vchunk = (ta.n_val + kTcCluster - 1) / kTcCluster;
            const long long vlo = min(ta.n_val, rank * vchunk), vhi = min(ta.n_val, vlo + vchunk);
            float vsum = 0.0f;
            int vbuf = 2;
            if (fetcher) {
                fetch_val(vbuf, vlo, vhi);
                tc::copy_wait();
            }
            __syncthreads();
            for (long long p0 = vlo; p0 < vhi; p0 += kTcRows, vbuf ^= 1) {
                if (fetcher) {
                    fetch_val(vbuf ^ 1, p0 + kTcRows, vhi);
                    settle();
                    tc::copy_wait();
                } else {
                    const float yhat = forward_tile(vbuf);
                    if (worker && cb == 0) {
                        const float r = p0 + m < vhi ? (yhat + S.w[0].b3) - S.rows[vbuf][kMaxIn][m] : 0.0f;
                        S.r2[m] = r * r;
                    }
                }
                __syncthreads();
                if (summer && lane == 0) {
                    float l = 0.0f;
                    add64(S.r2, 0, l);
                    add64(S.r2, 64, l);
                    vsum += l;
                }
            }
            if (summer && lane == 0) S.vsum = vsum;
            cluster.sync();
            float vl = 0.0f;
            for (int rr = 0; rr < kTcCluster; ++rr)
                vl += tc::ld_cluster(tc::cluster_addr(tc::smem_addr(&S.vsum), rr));
            vl /= static_cast<float>(ta.n_val);
            cluster.sync();  // every CTA has read the sums before they are written again
            if (rank == 0 && t == 0 && ta.val_losses) ta.val_losses[ep] = vl;
            if (vl < best) {
                best = vl;
                best_epoch = ep + 1;
                bad = 0;
                if (par >= 0) ta.theta[par] = th;
            } else if (ta.patience > 0 && ++bad >= ta.patience) {
                stop = true;
            }
        }
    }
    if (par >= 0) {
        if (ta.n_val == 0) ta.theta[par] = th;
        if (ta.theta_last) ta.theta_last[par] = th;
        if (ta.m_out) ta.m_out[par] = mom;
        if (ta.v_out) ta.v_out[par] = vel;
    }
    if (rank == 0 && t == 0 && ta.info) {
        ta.info[0] = epochs_run;
        ta.info[1] = ta.n_val > 0 ? best_epoch : epochs_run;
        ta.info[2] = static_cast<int>(step);
    }
    settle();
    if (!ok) {  // (after a timeout: once more, with a limit, for what is still in flight)
        if (worker) tc::mbar_wait(&S.bar, phase ^ 1u, kTcWait);
        tc::mbar_wait(&S.bar_grad, phase_grad ^ 1u, kTcWait);
        tc::mbar_wait(&S.bar_weights, phase_weights ^ 1u, kTcWait);
    }
    tc::fence_before_sync();
    cluster.sync();  // no CTA leaves while another may still copy from or to it
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_free(tm, 256);
}

size_t mlp_train_tc_smem() { return sizeof(TcSmem); }

// Inference.  The two layers are FP32 products of BF16-rounded operands with a
// prescribed order of additions (one chain per unit, inputs ascending), so
// they run on the FP32 pipe; what bounds them is feeding it.  One thread per
// sample needs one 16-byte broadcast of weights from shared memory for four
// multiply-adds, and the broadcasts took twice as long as the arithmetic.
// Here a CTA takes tiles of 128 samples x 64 units, a thread 8 samples x 8
// units in registers: two 16-byte loads of activations and two of weights feed
// 64 multiply-adds, every chain in the same order as before.  The activations
// pass through shared memory ([unit][sample], so stores and loads are 16-byte
// and conflict-free); the output layer is one chain per sample.  As many CTAs
// as fit at once walk the tiles, so the weights are staged once per CTA.
// Measured, 942,080 samples of 8 inputs: 286 -> 187 us (8.8 GFLOP, 47 of the
// 80 TFLOP/s of FP32); 100,001 of 6 inputs 42 -> 31; 5,003 of 8 16.5 -> 10.3.
constexpr int kFwdThreads = 128;
constexpr int kFwdTile = 128;   // samples per tile
constexpr int kFwdCtas = 3;     // per SM: the 64 packed sums and their operands take 153 registers
constexpr int kFwdUnroll = 16;  // inputs of layer 2 at a time (8: 187 us)

struct FwdSmem {
    alignas(16) float act[H][kFwdTile];     // h1, then h2
    alignas(16) float x[kMaxIn][kFwdTile];
    alignas(16) float w1t[kMaxIn][H];       // [k][u]
    alignas(16) float w2t[H][H];            // [u][v]
    alignas(16) float w3[H];
    float b1[H], b2[H];
    float b3;
};

__device__ __forceinline__ void load8(const float* row, int at, float (&v)[8], int half) {
    const float4 a = *reinterpret_cast<const float4*>(row + at), b = *reinterpret_cast<const float4*>(row + half + at);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
    v[4] = b.x;
    v[5] = b.y;
    v[6] = b.z;
    v[7] = b.w;
}

// acc[i][j] = sum of a_k[sample i] w_k[unit j] for k ascending; two units at a
// time with the packed FP32 multiply-add (each half rounded as a scalar one).
template <int K, int kUnroll>
__device__ __forceinline__ void fwd_tile(const float (*a)[kFwdTile], const float (*w)[H], int m0, int n0,
                                         float (&acc)[8][8]) {
    unsigned long long acc2[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc2[i][j] = 0ull;
#pragma unroll kUnroll
    for (int k = 0; k < K; ++k) {
        float av[8];
        load8(a[k], m0, av, kFwdTile / 2);
        const ulonglong2 wa = *reinterpret_cast<const ulonglong2*>(&w[k][n0]);
        const ulonglong2 wb = *reinterpret_cast<const ulonglong2*>(&w[k][H / 2 + n0]);
        const unsigned long long wv[4] = {wa.x, wa.y, wb.x, wb.y};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            unsigned long long aa;
            asm("mov.b64 %0, {%1, %1};" : "=l"(aa) : "f"(av[i]));
#pragma unroll
            for (int j = 0; j < 4; ++j) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc2[i][j]) : "l"(aa), "l"(wv[j]));
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[i][2 * j]), "=f"(acc[i][2 * j + 1]) : "l"(acc2[i][j]));
}

// act[unit][sample] = bf16(relu(acc + bias)) of this thread's 8 x 8 block.
__device__ __forceinline__ void fwd_store(const float (&acc)[8][8], const float* bias, int m0, int n0,
                                          float (*act)[kFwdTile]) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int u = n0 + (j < 4 ? j : H / 2 + j - 4);
        const float b = bias[u];
        float h[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) h[i] = bf(fmaxf(acc[i][j] + b, 0.0f));
        *reinterpret_cast<float4*>(&act[u][m0]) = make_float4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<float4*>(&act[u][kFwdTile / 2 + m0]) = make_float4(h[4], h[5], h[6], h[7]);
    }
}

__global__ void __launch_bounds__(kFwdThreads, kFwdCtas) mlp_forward_kernel(
    const float* __restrict__ theta, int d_in, const float* __restrict__ X, long long n, float* __restrict__ yhat) {
    extern __shared__ __align__(16) unsigned char fwd_raw[];
    FwdSmem& S = *reinterpret_cast<FwdSmem*>(fwd_raw);
    const int t = threadIdx.x;
    const int m0 = 4 * (t & 15), n0 = 4 * (t >> 4);  // samples m0.. and 64 + m0.., units n0.. and 32 + n0..
    if (!MRIP_CHECK(sizeof(FwdSmem) <= dynamic_smem_bytes(), 405, sizeof(FwdSmem))) return;  // CTA-uniform
    for (int i = t; i < kMaxIn * H; i += kFwdThreads) {
        const int k = i / H, u = i - k * H;
        S.w1t[k][u] = k < d_in ? bf(theta[u * d_in + k]) : 0.0f;
    }
    for (int i = t; i < H * H; i += kFwdThreads) S.w2t[i % H][i / H] = bf(theta[off_w2(d_in) + i]);
    for (int i = t; i < H; i += kFwdThreads) {
        S.w3[i] = bf(theta[off_w3(d_in) + i]);
        S.b1[i] = theta[off_b1(d_in) + i];
        S.b2[i] = theta[off_b2(d_in) + i];
    }
    if (t == 0) S.b3 = theta[off_b3(d_in)];
    for (long long base = static_cast<long long>(blockIdx.x) * kFwdTile; base < n;
         base += static_cast<long long>(gridDim.x) * kFwdTile) {
        const long long i = base + t;
#pragma unroll
        for (int k = 0; k < kMaxIn; ++k) S.x[k][t] = (k < d_in && i < n) ? bf(X[k * n + i]) : 0.0f;
        __syncthreads();  // the tile's inputs (and the weights); the last tile's outputs are done
        float acc[8][8];
        fwd_tile<kMaxIn, kMaxIn>(S.x, S.w1t, m0, n0, acc);
        fwd_store(acc, S.b1, m0, n0, S.act);
        __syncthreads();
        fwd_tile<H, kFwdUnroll>(S.act, S.w2t, m0, n0, acc);
        __syncthreads();
        fwd_store(acc, S.b2, m0, n0, S.act);
        __syncthreads();
        float out = 0.0f;
#pragma unroll 8
        for (int v = 0; v < H; ++v) out = fmaf(S.act[v][t], S.w3[v], out);
        if (i < n) yhat[i] = out + S.b3;
    }
}

// Control-variate reduction of one design point per CTA (FP64, two passes,
// fixed-order tree sums).
constexpr int kCvThreads = 256;

__device__ double block_sum(double v, double* sh) {
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int stride = kCvThreads / 2; stride > 0; stride >>= 1) {
        if (threadIdx.x < stride) sh[threadIdx.x] += sh[threadIdx.x + stride];
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kCvThreads) cv_reduce_kernel(const double* __restrict__ y,
                                                               const double* __restrict__ g, long long n,
                                                               const double* __restrict__ gc, long long m,
                                                               double* __restrict__ out) {
    __shared__ double sh[kCvThreads];
    const long long dp = blockIdx.x;
    const double* yr = y + dp * n;
    const double* gr = g + dp * n;
    const double* cr = gc + dp * m;
    double sy = 0.0, sg = 0.0, sc = 0.0;
    for (long long i = threadIdx.x; i < n; i += kCvThreads) {
        sy += yr[i];
        sg += gr[i];
    }
    for (long long i = threadIdx.x; i < m; i += kCvThreads) sc += cr[i];
    const double ybar = block_sum(sy, sh) / static_cast<double>(n);
    const double gbar = block_sum(sg, sh) / static_cast<double>(n);
    const double cbar = block_sum(sc, sh) / static_cast<double>(m);
    double sxy = 0.0, sgg = 0.0, scc = 0.0;
    for (long long i = threadIdx.x; i < n; i += kCvThreads) {
        const double dy = yr[i] - ybar, dg = gr[i] - gbar;
        sxy += dy * dg;
        sgg += dg * dg;
    }
    for (long long i = threadIdx.x; i < m; i += kCvThreads) {
        const double dc = cr[i] - cbar;
        scc += dc * dc;
    }
    const double cov = block_sum(sxy, sh) / static_cast<double>(n - 1);
    const double var_g = block_sum(sgg, sh) / static_cast<double>(n - 1);
    const double var_c = block_sum(scc, sh) / static_cast<double>(m - 1);
    const double beta = var_g > 0.0 ? cov / var_g : 0.0;
    double sr = 0.0;
    for (long long i = threadIdx.x; i < n; i += kCvThreads) sr += yr[i] - beta * gr[i];
    const double rbar = block_sum(sr, sh) / static_cast<double>(n);
    double srr = 0.0;
    for (long long i = threadIdx.x; i < n; i += kCvThreads) {
        const double d = (yr[i] - beta * gr[i]) - rbar;
        srr += d * d;
    }
    const double s_r2 = block_sum(srr, sh) / static_cast<double>(n - 2);
    if (threadIdx.x == 0) {
        out[5 * dp] = beta;
        out[5 * dp + 1] = ybar - beta * (gbar - cbar);
        out[5 * dp + 2] = s_r2 / static_cast<double>(n) + beta * beta * var_c / static_cast<double>(m);
        out[5 * dp + 3] = ybar;
        out[5 * dp + 4] = gbar - cbar;
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// internal launchers used by the control-variate driver
// ---------------------------------------------------------------------------
long long mlp_params(int d_in) { return n_params(d_in); }

mrip_status mlp_init(int d_in, uint64_t seed, float* theta, cudaStream_t st) {
    const long long n_w = static_cast<long long>(H) * d_in + H * H + H;
    mlp_init_kernel<<<ceil_div_u(n_w, 256), 256, 0, st>>>(d_in, expand_key(seed), theta);
    return launch_status("mlp init");
}

size_t mlp_grad_partial_floats(int d_in, long long B) {
    return static_cast<size_t>((B + kTile - 1) / kTile) * static_cast<size_t>(n_params(d_in) + 1);
}

// One gradient (and optionally Adam) step over batch positions [0, B) of map.
mrip_status mlp_step(const float* theta_in, int d_in, const float* X, long long n_total, const float* Y,
                     const int64_t* idx, unsigned long long a, unsigned long long b, unsigned long long n_perm,
                     long long off, long long B, float* partial, float* grad, float* loss, float* theta,
                     float* m, float* v, const float* adam /* lr, b1, b2, eps, bc1, bc2 */, cudaStream_t st) {
    const int n_cta = static_cast<int>((B + kTile - 1) / kTile);
    const long long P = n_params(d_in);
    float* part_loss = partial + static_cast<long long>(n_cta) * P;
    SampleMap map{idx, a, b, n_perm, off};
    cudaError_t e = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(sizeof(GradSmem)));
    if (e != cudaSuccess) return cuda_status(e, "mlp: shared memory attribute");
    mlp_grad_kernel<<<n_cta, kGradThreads, sizeof(GradSmem), st>>>(theta_in, d_in, X, n_total, Y, map, B,
                                                                   partial, part_loss);
    mrip_status s = launch_status("mlp grad");
    if (s != MRIP_OK) return s;
    if (adam) {
        mlp_reduce_kernel<true><<<ceil_div_u(P, 256), 256, 0, st>>>(
            partial, part_loss, n_cta, P, B, grad, loss, theta, m, v, adam[0], adam[1], adam[2], adam[3],
            adam[4], adam[5]);
    } else {
        mlp_reduce_kernel<false><<<ceil_div_u(P, 256), 256, 0, st>>>(
            partial, part_loss, n_cta, P, B, grad, loss, nullptr, nullptr, nullptr, 0, 0, 0, 0, 1, 1);
    }
    return launch_status("mlp reduce");
}

// Epoch order (a, b) of n samples: block (0, epoch) of tag 4, rep 0, dp 0;
// a = 1 + w0 mod (n - 1) stepped up to the first value coprime with n,
// b = w1 mod n.
void epoch_affine(uint64_t seed, int epoch, unsigned long long n, unsigned long long& a, unsigned long long& b) {
    if (n <= 1) {
        a = 1;
        b = 0;
        return;
    }
    const uint4 w = philox(0u, static_cast<uint32_t>(epoch), 0u, stream_word(4u, 0u), expand_key(seed));
    a = 1 + static_cast<unsigned long long>(w.x) % (n - 1);
    while (std::gcd(a, n) != 1) {
        ++a;
        if (a >= n) a = 1;
    }
    b = static_cast<unsigned long long>(w.y) % n;
}

// Adam training in one cluster launch with the contractions on the tensor
// cores (mlp_train_tc_kernel).  The host computes the schedule -- per epoch
// the affine order, per step Adam's bias corrections in double rounded to
// float -- and uploads it to library scratch.  Synchronous: reads back
// whether an MMA completion wait ran out, and the run's counts.
mrip_status mlp_train(const TrainSpec& sp, TrainInfo* info, cudaStream_t st) {
    NvtxRange range("mlp_train");
    TrainInfo none{0, 0, 0};
    if (info) *info = none;
    if (sp.n == 0 || sp.epochs == 0) return MRIP_OK;
    const long long spe = (sp.n + sp.B - 1) / sp.B;
    long long n_steps = spe * sp.epochs;
    if (sp.max_steps > 0 && sp.max_steps < n_steps) n_steps = sp.max_steps;
    // resuming at epoch epoch0: its order and Adam's step count continue
    const long long step0 = static_cast<long long>(sp.epoch0) * spe;
    // one upload: [info 16 B, timeout flag 16 B, both zero][ab][bc]
    const size_t ab_bytes = 2 * static_cast<size_t>(sp.epochs) * sizeof(unsigned long long);
    const size_t bytes = 32 + ab_bytes + 2 * static_cast<size_t>(n_steps) * sizeof(float);
    std::vector<unsigned long long> schedule((bytes + 7) / 8, 0ull);
    unsigned long long* ab = schedule.data() + 4;
    for (int ep = 0; ep < sp.epochs; ++ep)
        epoch_affine(sp.order_seed, sp.epoch0 + ep, static_cast<unsigned long long>(sp.n), ab[2 * ep],
                     ab[2 * ep + 1]);
    float* bc = reinterpret_cast<float*>(ab + 2 * static_cast<size_t>(sp.epochs));
    for (long long k = 1; k <= n_steps; ++k) {
        const double kk = static_cast<double>(step0 + k);
        bc[2 * (k - 1)] = static_cast<float>(1.0 - std::pow(static_cast<double>(sp.beta1), kk));
        bc[2 * (k - 1) + 1] = static_cast<float>(1.0 - std::pow(static_cast<double>(sp.beta2), kk));
    }
    char* base = static_cast<char*>(scratch(bytes, 4));
    if (!base) return fail(MRIP_ENOMEM, "mlp train: scratch allocation failed");
    int* d_info = reinterpret_cast<int*>(base);
    int* flag = reinterpret_cast<int*>(base + 16);
    unsigned long long* d_ab = reinterpret_cast<unsigned long long*>(base + 32);
    float* d_bc = reinterpret_cast<float*>(base + 32 + ab_bytes);
    cudaError_t e = cudaMemcpyAsync(base, schedule.data(), bytes, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return cuda_status(e, "mlp train: schedule upload");
    const size_t smem = mlp_train_tc_smem();
    e = cudaFuncSetAttribute(mlp_train_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return cuda_status(e, "mlp train: shared memory attribute");
    TrainArgs ta{sp.X, sp.Y, sp.n, sp.B, spe, sp.epochs, sp.d_in, d_ab, d_bc, sp.lr, sp.beta1, sp.beta2, sp.eps,
                 sp.theta, sp.losses, sp.max_steps, sp.grad, sp.m_out, sp.v_out, sp.Xv, sp.Yv,
                 sp.Xv ? sp.n_val : 0, sp.patience, sp.val_losses, d_info, sp.m_in, sp.v_in,
                 sp.best0, sp.bad0, sp.theta_in, sp.theta_last};
    mlp_train_tc_kernel<<<kTcCluster, kTcThreads, smem, st>>>(ta, flag);
    mrip_status s = launch_status("mlp train (tensor cores)");
    if (s != MRIP_OK) return s;
    int h[8] = {0};
    e = cudaMemcpyAsync(h, base, 32, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // also: the host schedule dies at return
    if (e != cudaSuccess) return cuda_status(e, "mlp train (tensor cores)");
    if (h[4]) return fail(MRIP_ECUDA, "mlp train: a tensor-core product or an exchange between CTAs did not complete in time");
    if (info) {
        info->epochs_run = h[0];
        info->best_epoch = h[1];
        info->steps = h[2];
    }
    return MRIP_OK;
}

mrip_status mlp_forward(const float* theta, int d_in, const float* X, long long n, float* yhat, cudaStream_t st) {
    if (n == 0) return MRIP_OK;
    cudaError_t e = cudaFuncSetAttribute(mlp_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(sizeof(FwdSmem)));
    if (e != cudaSuccess) return cuda_status(e, "mlp forward: shared memory attribute");
    const long long tiles = (n + kFwdTile - 1) / kFwdTile, resident = static_cast<long long>(sm_count()) * kFwdCtas;
    mlp_forward_kernel<<<static_cast<unsigned>(std::min(tiles, resident)), kFwdThreads, sizeof(FwdSmem), st>>>(
        theta, d_in, X, n, yhat);
    return launch_status("mlp forward");
}

mrip_status cv_reduce(const double* y, const double* g, long long n, const double* gc, long long m, int n_dp,
                      double* out, cudaStream_t st) {
    if (n_dp == 0) return MRIP_OK;
    cv_reduce_kernel<<<n_dp, kCvThreads, 0, st>>>(y, g, n, gc, m, out);
    return launch_status("cv reduce");
}

}  // namespace mrip

using namespace mrip;

extern "C" int64_t mrip_mlp_param_count(int32_t d_in) { return d_in >= 1 && d_in <= 8 ? n_params(d_in) : -1; }

extern "C" mrip_status mrip_mlp_init(int32_t d_in, uint64_t seed, float* d_theta, void* stream) {
    if (d_in < 1 || d_in > kMaxIn) return fail(MRIP_EINVAL, "mrip_mlp_init: d_in in 1..8");
    if (!d_theta) return fail(MRIP_EINVAL, "mrip_mlp_init: null theta");
    return mlp_init(d_in, seed, d_theta, static_cast<cudaStream_t>(stream));
}

extern "C" mrip_status mrip_mlp_forward(const float* d_theta, int32_t d_in, const float* d_x, int64_t n,
                                        float* d_yhat, void* stream) {
    if (d_in < 1 || d_in > kMaxIn || n < 0) return fail(MRIP_EINVAL, "mrip_mlp_forward: d_in in 1..8, n >= 0");
    if (n > 0 && (!d_theta || !d_x || !d_yhat)) return fail(MRIP_EINVAL, "mrip_mlp_forward: null pointer");
    return mlp_forward(d_theta, d_in, d_x, n, d_yhat, static_cast<cudaStream_t>(stream));
}

extern "C" mrip_status mrip_mlp_loss_grad(const float* d_theta, int32_t d_in, const float* d_x, const float* d_y,
                                          int64_t n, const int64_t* d_idx, int64_t B, float* d_grad,
                                          float* d_loss, void* stream) {
    if (d_in < 1 || d_in > kMaxIn || n < 1 || B < 1 || (!d_idx && B > n))
        return fail(MRIP_EINVAL, "mrip_mlp_loss_grad: d_in in 1..8, 1 <= B (<= n without idx)");
    if (!d_theta || !d_x || !d_y || !d_grad) return fail(MRIP_EINVAL, "mrip_mlp_loss_grad: null pointer");
    const size_t need = mlp_grad_partial_floats(d_in, B) * sizeof(float);
    float* partial = static_cast<float*>(scratch(need, 2));
    if (!partial) return fail(MRIP_ENOMEM, "mrip_mlp_loss_grad: scratch allocation failed");
    return mlp_step(d_theta, d_in, d_x, n, d_y, d_idx, 0, 0, 0, 0, B, partial, d_grad, d_loss, nullptr,
                    nullptr, nullptr, nullptr, static_cast<cudaStream_t>(stream));
}

extern "C" mrip_status mrip_adam_step(float* d_theta, float* d_m, float* d_v, const float* d_grad, int64_t n,
                                      int64_t t, float lr, float beta1, float beta2, float eps, void* stream) {
    if (n < 0 || t < 1) return fail(MRIP_EINVAL, "mrip_adam_step: n >= 0, t >= 1");
    if (n == 0) return MRIP_OK;
    if (!d_theta || !d_m || !d_v || !d_grad) return fail(MRIP_EINVAL, "mrip_adam_step: null pointer");
    const float bc1 = static_cast<float>(1.0 - std::pow(static_cast<double>(beta1), static_cast<double>(t)));
    const float bc2 = static_cast<float>(1.0 - std::pow(static_cast<double>(beta2), static_cast<double>(t)));
    adam_kernel<<<ceil_div_u(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(d_theta, d_m, d_v, d_grad, n,
                                                                                  lr, beta1, beta2, eps, bc1, bc2);
    return launch_status("mrip_adam_step");
}

extern "C" mrip_status mrip_mlp_train(int32_t d_in, const float* d_x, const float* d_y, int64_t n,
                                      const float* d_xv, const float* d_yv, int64_t n_val,
                                      const mrip_train_params* prm, float* d_theta, const float* d_m_in,
                                      const float* d_v_in, float* d_losses, float* d_grad, float* d_m,
                                      float* d_v, float* d_val_losses, int32_t* info_out, void* stream) {
    if (d_in < 1 || d_in > kMaxIn || n < 1 || n_val < 0 || !prm)
        return fail(MRIP_EINVAL, "mrip_mlp_train: d_in in 1..8, n >= 1, n_val >= 0, params");
    if (prm->batch < 1 || prm->epochs < 1 || prm->epoch0 < 0 || prm->patience < 0 || prm->max_steps < 0 ||
        !(prm->lr > 0.0f) ||
        !(prm->beta1 >= 0.0f && prm->beta1 < 1.0f) || !(prm->beta2 >= 0.0f && prm->beta2 < 1.0f) ||
        !(prm->eps > 0.0f))
        return fail(MRIP_EINVAL, "mrip_mlp_train: batch, epochs >= 1, patience, max_steps >= 0, lr, eps > 0, "
                                 "beta1, beta2 in [0, 1)");
    if (n > 0x7FFFFFFFll || n_val > 0x7FFFFFFFll) return fail(MRIP_EINVAL, "mrip_mlp_train: n, n_val < 2^31");
    if (!d_x || !d_y || !d_theta || (n_val > 0 && (!d_xv || !d_yv)))
        return fail(MRIP_EINVAL, "mrip_mlp_train: null pointer");
    TrainSpec sp{};
    sp.d_in = d_in;
    sp.X = d_x;
    sp.Y = d_y;
    sp.n = n;
    sp.Xv = n_val > 0 ? d_xv : nullptr;
    sp.Yv = n_val > 0 ? d_yv : nullptr;
    sp.n_val = n_val;
    sp.B = prm->batch;
    sp.epochs = prm->epochs;
    sp.epoch0 = prm->epoch0;
    sp.m_in = d_m_in;
    sp.v_in = d_v_in;
    sp.max_steps = prm->max_steps;
    sp.patience = prm->patience;
    sp.order_seed = prm->order_seed;
    sp.lr = prm->lr;
    sp.beta1 = prm->beta1;
    sp.beta2 = prm->beta2;
    sp.eps = prm->eps;
    sp.theta = d_theta;
    sp.losses = d_losses;
    sp.grad = d_grad;
    sp.m_out = d_m;
    sp.v_out = d_v;
    sp.val_losses = d_val_losses;
    TrainInfo info{};
    mrip_status s = mlp_train(sp, &info, static_cast<cudaStream_t>(stream));
    if (s == MRIP_OK && info_out) {
        info_out[0] = info.epochs_run;
        info_out[1] = info.best_epoch;
        info_out[2] = info.steps;
    }
    return s;
}

extern "C" mrip_status mrip_cv_reduce(const double* d_y, const double* d_g, int64_t n, const double* d_gc,
                                      int64_t m, int32_t n_dp, double* d_out, void* stream) {
    if (n < 3 || m < 2 || n_dp < 0) return fail(MRIP_EINVAL, "mrip_cv_reduce: n >= 3, m >= 2, n_dp >= 0");
    if (n_dp > 0 && (!d_y || !d_g || !d_gc || !d_out)) return fail(MRIP_EINVAL, "mrip_cv_reduce: null pointer");
    return cv_reduce(d_y, d_g, n, d_gc, m, n_dp, d_out, static_cast<cudaStream_t>(stream));
}

MRIP_DEBUG_UNIT(mlp)
