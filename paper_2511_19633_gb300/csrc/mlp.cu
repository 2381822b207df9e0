// Training of the learned-proposal network on the GPU with the library's own
// kernels: FP32 forward and backward passes of the 4 -> 64 -> 64 -> 1 ReLU
// network, the asymmetric squared (expectile) loss that biases the fit to
// lie above its targets, and Adam updates. Inference in the shower uses the
// BF16 tensor-core tile of mlp_infer.cuh; gaps_mlp_forward exposes both
// numerics for calibration and tests.
#include <cooperative_groups.h>

#include "common.cuh"
#include "mlp_infer.cuh"

namespace gaps {
namespace {

struct Layers {
  const float *W1, *b1, *W2, *b2, *W3;
  float b3;
};

__device__ __forceinline__ Layers layers_of(const float* P) {
  Layers L;
  L.W1 = P;
  L.b1 = L.W1 + kMlpH * kMlpIn;
  L.W2 = L.b1 + kMlpH;
  L.b2 = L.W2 + kMlpH * kMlpH;
  L.W3 = L.b2 + kMlpH;
  L.b3 = L.W3[kMlpH];
  return L;
}

__device__ float forward_one(const Layers& L, const float* x, float* h1, float* h2) {
  for (int i = 0; i < kMlpH; ++i) {
    float a = L.b1[i];
#pragma unroll
    for (int k = 0; k < kMlpIn; ++k) a = fmaf(L.W1[i * kMlpIn + k], x[k], a);
    h1[i] = fmaxf(a, 0.0f);
  }
  for (int i = 0; i < kMlpH; ++i) {
    float a = L.b2[i];
    for (int k = 0; k < kMlpH; ++k) a = fmaf(L.W2[i * kMlpH + k], h1[k], a);
    h2[i] = fmaxf(a, 0.0f);
  }
  float y = L.b3;
  for (int k = 0; k < kMlpH; ++k) y = fmaf(L.W3[k], h2[k], y);
  return y;
}

// per-sample gradient accumulated into a block-shared buffer, then global
__global__ void k_loss_grad(const float* P, const float* X, const float* T, uint64_t n, float tau,
                            float* grad, float* loss) {
  extern __shared__ float sg[];  // kMlpParams + 1 (loss)
  for (int q = threadIdx.x; q <= kMlpParams; q += blockDim.x) sg[q] = 0.0f;
  __syncthreads();
  const Layers L = layers_of(P);
  uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s < n) {
    float h1[kMlpH], h2[kMlpH], d2[kMlpH];
    const float* x = X + 4 * s;
    float y = forward_one(L, x, h1, h2);
    float r = y - T[s];
    float w = r < 0.0f ? tau : 1.0f - tau;
    atomicAdd(&sg[kMlpParams], w * r * r / (float)n);
    float dy = 2.0f * w * r / (float)n;
    float* gW1 = sg;
    float* gb1 = gW1 + kMlpH * kMlpIn;
    float* gW2 = gb1 + kMlpH;
    float* gb2 = gW2 + kMlpH * kMlpH;
    float* gW3 = gb2 + kMlpH;
    atomicAdd(&gW3[kMlpH], dy);
    for (int k = 0; k < kMlpH; ++k) {
      atomicAdd(&gW3[k], dy * h2[k]);
      d2[k] = h2[k] > 0.0f ? dy * L.W3[k] : 0.0f;
    }
    for (int i = 0; i < kMlpH; ++i) {
      if (d2[i] == 0.0f) continue;
      atomicAdd(&gb2[i], d2[i]);
      for (int k = 0; k < kMlpH; ++k)
        if (h1[k] != 0.0f) atomicAdd(&gW2[i * kMlpH + k], d2[i] * h1[k]);
    }
    for (int k = 0; k < kMlpH; ++k) {
      if (h1[k] <= 0.0f) continue;
      float a = 0.0f;
      for (int i = 0; i < kMlpH; ++i) a = fmaf(L.W2[i * kMlpH + k], d2[i], a);
      atomicAdd(&gb1[k], a);
      for (int j = 0; j < kMlpIn; ++j) atomicAdd(&gW1[k * kMlpIn + j], a * x[j]);
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < kMlpParams; q += blockDim.x)
    if (sg[q] != 0.0f) atomicAdd(&grad[q], sg[q]);
  if (threadIdx.x == 0) atomicAdd(loss, sg[kMlpParams]);
}

__global__ void k_forward_f32(const float* P, const float* X, uint64_t n, float* out) {
  uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  float h1[kMlpH], h2[kMlpH];
  out[s] = forward_one(layers_of(P), X + 4 * s, h1, h2);
}

// BF16 tensor-core forward, the numerics of the shower's inference
__global__ void k_forward_bf16(const float* P, const float* X, uint64_t n, float* out) {
  __shared__ MlpSmem S;
  __shared__ float feat[8][16][4];
  __shared__ float res[8][16];
  mlp_load_smem(S, P);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint64_t tiles = (n + 15) / 16;
  for (uint64_t tile = (uint64_t)blockIdx.x * 8 + warp; tile < tiles; tile += (uint64_t)gridDim.x * 8) {
    for (int q = lane; q < 64; q += 32) {
      uint64_t row = tile * 16 + q / 4;
      feat[warp][q / 4][q % 4] = row < n ? X[4 * row + q % 4] : 0.0f;
    }
    __syncwarp();
    mlp_tile(S, feat[warp], res[warp]);
    if (lane < 16 && tile * 16 + lane < n) out[tile * 16 + lane] = res[warp][lane];
    __syncwarp();
  }
}

// The network's BF16 image in global memory for the shower's inference
__global__ void k_mlp_image(const float* P, MlpSmem* out) { mlp_load_smem(*out, P); }

// Minibatch Adam training: one cluster of eight blocks loops over minibatches
// of 256 rows drawn with replacement (Philox counter = step).
//
// A step is a chain of small matrix products (0.9 MFLOP forward, twice that
// backward) that no other step can overlap, so its latency is what counts: one
// block took 200 us a step, its gradient loops reading shared memory twice per
// product. Block r of the cluster takes rows 32 r .. 32 r + 31 of the batch
// through the network, and owns the units 8 r .. 8 r + 7 of both hidden layers:
// it forms their weights' gradients over the whole batch and updates them. The
// layer-2 activations and layer-1 deltas that an owner needs, and the updated
// weights, are written into the other blocks' shared memory; three cluster
// barriers a step order them. The optimiser's moments stay in the owners'
// registers. What bounds it now: shared-memory reads (5700 of 18 000 clocks a
// step form W2's gradient, 2800 each the two products with W2). Every sum
// runs over the same terms in the same order as in one block (FP32 FMA chains
// over inputs or over rows 0 .. 255), so the parameters are the same bits; only
// the reported loss is summed in another order.
// 300 steps: 59.7 ms with one block, 3.06 ms now.
constexpr int kB = 256;                // rows of a batch
constexpr int kTrainBlocks = 8;        // the portable cluster size
constexpr int kTR = kB / kTrainBlocks; // rows a block takes through the network
constexpr int kTU = kMlpH / kTrainBlocks;  // units a block owns in each hidden layer
constexpr int kRS = kMlpH + 4;         // row stride of row-major activations (16-byte rows, spread banks)
constexpr int kBS = kB + 4;            // row stride of unit-major ones
constexpr int kWS = kMlpH + 1;         // row stride of W2: rows and columns both read without bank conflicts
static_assert(kTR == 32 && kTU == 8, "the thread mappings below");
struct TrainSmem {
  float h1t[kMlpH][kBS];  // layer-1 activations of the whole batch, unit-major
  float h2t[kTU][kBS];    // owned layer-2 units: activations
  float d2t[kTU][kBS];    // ... and deltas
  float d1t[kTU][kBS];    // owned layer-1 units: deltas
  float x[kB][kMlpIn], xt[kMlpIn][kBS];  // inputs of the batch, row- and input-major
  float h1[kTR][kRS];     // own rows: activations
  float h2[kTR][kRS];     // own rows: activations, then deltas
  float dy[kB];
  float W1[kMlpH][kMlpIn];
  float W2[kMlpH][kWS];
  float b1[kMlpH], b2[kMlpH], W3[kMlpH];
  float b3, loss[kTrainBlocks];
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// one parameter's Adam state, held by the thread that owns it
struct Adam {
  float m, v;
};
__device__ __forceinline__ float adam_step(Adam& s, float p, float gq, float lr, float b1t, float b2t) {
  const float b1c = 0.9f, b2c = 0.999f, eps = 1e-8f;
  // (the contraction of the two sums is fixed here, so that the moments do not
  // depend on how the compiler pairs the products)
  const float a = fmaf(1.0f - b1c, gq, b1c * s.m);
  const float v = fmaf((1.0f - b2c) * gq, gq, b2c * s.v);
  s.m = a;
  s.v = v;
  p -= lr * (a / (1.0f - b1t)) / (sqrtf(v / (1.0f - b2t)) + eps);
  return p;
}

// out[j] = b + sum over 64 inputs of w(input) * in[row r0 + j][input], j = 0..7:
// the weights are read once for eight rows, the rows as broadcast float4
template <class Wf>
__device__ __forceinline__ void dense8(const float (*in)[kRS], int r0, float b, Wf w, float out[8]) {
#pragma unroll
  for (int j = 0; j < 8; ++j) out[j] = b;
#pragma unroll
  for (int k = 0; k < kMlpH; k += 4) {
    const float w0 = w(k), w1 = w(k + 1), w2 = w(k + 2), w3 = w(k + 3);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float4 v = *reinterpret_cast<const float4*>(&in[r0 + j][k]);
      out[j] = fmaf(w3, v.w, fmaf(w2, v.z, fmaf(w1, v.y, fmaf(w0, v.x, out[j]))));
    }
  }
}

// sum over the 256 rows, in row order, of a c
__device__ __forceinline__ float over_rows(const float* a, const float* c) {
  float s = 0.0f;
#pragma unroll 8
  for (int b = 0; b < kB; b += 4) {
    const float4 v = *reinterpret_cast<const float4*>(a + b), w = *reinterpret_cast<const float4*>(c + b);
    s = fmaf(v.w, w.w, fmaf(v.z, w.z, fmaf(v.y, w.y, fmaf(v.x, w.x, s))));
  }
  return s;
}
__device__ __forceinline__ float sum_rows(const float* a) {
  float s = 0.0f;
#pragma unroll 8
  for (int b = 0; b < kB; b += 4) {
    const float4 v = *reinterpret_cast<const float4*>(a + b);
    s += v.x;
    s += v.y;
    s += v.z;
    s += v.w;
  }
  return s;
}

__global__ void __cluster_dims__(kTrainBlocks) __launch_bounds__(kB)
    k_train(float* P, float* m1, float* m2, const float* X, const float* T, uint64_t n, uint64_t steps, float lr,
            float tau, uint64_t seed, float* loss_hist, int hist_every) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(smem_raw);
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x;
  // block r's view of this block's layout
  auto peer = [&](int r) -> TrainSmem& { return *cl.map_shared_rank(&S, r); };
  constexpr int oB1 = kMlpH * kMlpIn, oW2 = oB1 + kMlpH, oB2 = oW2 + kMlpH * kMlpH, oW3 = oB2 + kMlpH, oB3 = oW3 + kMlpH;
  for (int q = tid; q < kMlpH * kMlpIn; q += kB) S.W1[q / kMlpIn][q % kMlpIn] = P[q];
  for (int q = tid; q < kMlpH * kMlpH; q += kB) S.W2[q / kMlpH][q % kMlpH] = P[oW2 + q];
  if (tid < kMlpH) { S.b1[tid] = P[oB1 + tid]; S.b2[tid] = P[oB2 + tid]; S.W3[tid] = P[oW3 + tid]; }
  if (tid == 0) S.b3 = P[oB3];
  // Owned parameters. Threads 0..127: four W2 entries, rows 8 rank + 4 (tid /
  // 64) .. + 3 of column tid % 64. Threads 128..: one entry (b2, W3, b3) after
  // the second barrier's arrival, one (W1, b1) after its wait.
  const int u0 = kTU * rank;
  const bool tile = tid < 128;
  const int ti = tile ? 4 * (tid >> 6) : 0, tk = tid & 63;
  const int s = tid - 128;
  int qa = -1, qb = -1;  // parameter indices of the single entries
  if (!tile) {
    if (s < kTU) qa = oW3 + u0 + s;
    else if (s >= 32 && s < 32 + kTU) qa = oB2 + u0 + s - 32;
    else if (s == 64 && rank == 0) qa = oB3;
    if (s < 4 * kTU) qb = (u0 + s / 4) * kMlpIn + s % 4;
    else if (s >= 32 && s < 32 + kTU) qb = oB1 + u0 + s - 32;
  }
  Adam A[4], Aa{0.0f, 0.0f}, Ab{0.0f, 0.0f};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int q = oW2 + (u0 + ti + j) * kMlpH + tk;
    A[j] = tile ? Adam{m1[q], m2[q]} : Adam{0.0f, 0.0f};
  }
  if (qa >= 0) Aa = Adam{m1[qa], m2[qa]};
  if (qb >= 0) Ab = Adam{m1[qb], m2[qb]};
  float b1t = 1.0f, b2t = 1.0f;
  // batch row tid of the step, loaded a step ahead
  float xr[kMlpIn], tr;
  const uint64_t inv = ~0ull / n;  // x / n is at most two more than the high word of x inv
  auto load_row = [&](uint64_t step) {
    uint32_t rnd[4];
    philox((uint32_t)step, (uint32_t)(step >> 32), (uint32_t)tid, 0x5eedu, (uint32_t)seed, (uint32_t)(seed >> 32), rnd);
    const uint64_t u = ((uint64_t)rnd[1] << 32) | rnd[0];
    uint64_t row = u - __umul64hi(u, inv) * n;  // u mod n
    while (row >= n) row -= n;
#pragma unroll
    for (int k = 0; k < kMlpIn; ++k) xr[k] = X[4 * row + k];
    tr = T[row];
  };
  if (steps > 0) load_row(0);
  cluster_arrive();  // every block of the cluster runs before its memory is written
  cluster_wait();
  __syncthreads();
  const int unit = tid & 63, r0 = 8 * (tid >> 6);  // a unit and eight of the block's rows
  for (uint64_t step = 0; step < steps; ++step) {
    // --- forward pass of the block's rows
    *reinterpret_cast<float4*>(S.x[tid]) = make_float4(xr[0], xr[1], xr[2], xr[3]);
#pragma unroll
    for (int k = 0; k < kMlpIn; ++k) S.xt[k][tid] = xr[k];
    const float t_row = tr;  // row tid's target
    __syncthreads();
    if (step + 1 < steps) load_row(step + 1);
    {
      const float4 w = *reinterpret_cast<const float4*>(S.W1[unit]);
      const float b = S.b1[unit];
      float h[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 v = *reinterpret_cast<const float4*>(S.x[kTR * rank + r0 + j]);
        h[j] = fmaxf(fmaf(w.w, v.w, fmaf(w.z, v.z, fmaf(w.y, v.y, fmaf(w.x, v.x, b)))), 0.0f);
        S.h1[r0 + j][unit] = h[j];
      }
    }
    __syncthreads();
    {
      float h[8];
      dense8(S.h1, r0, S.b2[unit], [&](int k) { return S.W2[unit][k]; }, h);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        h[j] = fmaxf(h[j], 0.0f);
        S.h2[r0 + j][unit] = h[j];
      }
      float4* to = reinterpret_cast<float4*>(&peer(unit / kTU).h2t[unit % kTU][kTR * rank + r0]);
      to[0] = make_float4(h[0], h[1], h[2], h[3]);
      to[1] = make_float4(h[4], h[5], h[6], h[7]);
    }
    __syncthreads();
    // the warp that loaded the block's rows' targets: output, loss and its slope
    if (tid >> 5 == rank) {
      const int r = tid & 31;
      float y = S.b3;
#pragma unroll 4
      for (int k = 0; k < kMlpH; k += 4) {
        const float4 v = *reinterpret_cast<const float4*>(&S.h2[r][k]);
        y = fmaf(S.W3[k], v.x, y);
        y = fmaf(S.W3[k + 1], v.y, y);
        y = fmaf(S.W3[k + 2], v.z, y);
        y = fmaf(S.W3[k + 3], v.w, y);
      }
      const float res = y - t_row;
      const float w = res < 0.0f ? tau : 1.0f - tau;
      const float dy = 2.0f * w * res / (float)kB;
#pragma unroll
      for (int q = 0; q < kTrainBlocks; ++q) peer(q).dy[kTR * rank + r] = dy;
      float l = w * res * res / (float)kB;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if (r == 0) peer(0).loss[rank] = l;
      __syncwarp();
    }
    cluster_arrive();
    // layer 1 of the whole batch, for the owned weights' gradients: 64 rows of
    // one unit a thread (cheaper than 64 KB from the other blocks), while the
    // barrier completes
    {
      const float4 w = *reinterpret_cast<const float4*>(S.W1[unit]);
      const float b = S.b1[unit];
      const int q0 = 64 * (tid >> 6);
#pragma unroll 4
      for (int q = q0; q < q0 + 64; q += 4) {
        float h[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 v = *reinterpret_cast<const float4*>(S.x[q + j]);
          h[j] = fmaxf(fmaf(w.w, v.w, fmaf(w.z, v.z, fmaf(w.y, v.y, fmaf(w.x, v.x, b)))), 0.0f);
        }
        *reinterpret_cast<float4*>(&S.h1t[unit][q]) = make_float4(h[0], h[1], h[2], h[3]);
      }
    }
    cluster_wait();
    // --- delta of layer 2: of the block's rows (in place) ...
    {
      const float w3 = S.W3[unit];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        float& v = S.h2[r0 + j][unit];
        v = v > 0.0f ? S.dy[kTR * rank + r0 + j] * w3 : 0.0f;
      }
    }
    // ... and of the owned units over the batch
    {
      const float dy = S.dy[tid];
#pragma unroll
      for (int i = 0; i < kTU; ++i) S.d2t[i][tid] = S.h2t[i][tid] > 0.0f ? dy * S.W3[u0 + i] : 0.0f;
    }
    __syncthreads();
    // delta of layer 1 of the block's rows, to the units' owners
    {
      float d[8];
      dense8(S.h2, r0, 0.0f, [&](int i) { return S.W2[i][unit]; }, d);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (!(S.h1[r0 + j][unit] > 0.0f)) d[j] = 0.0f;
      float4* to = reinterpret_cast<float4*>(&peer(unit / kTU).d1t[unit % kTU][kTR * rank + r0]);
      to[0] = make_float4(d[0], d[1], d[2], d[3]);
      to[1] = make_float4(d[4], d[5], d[6], d[7]);
    }
    cluster_arrive();
    // --- gradients of the owned weights, and their updates
    b1t *= 0.9f;
    b2t *= 0.999f;
    float pn[4] = {0.0f, 0.0f, 0.0f, 0.0f}, pa = 0.0f, pb = 0.0f;
    if (tile) {
      float g[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      // eight rows at a time, the next eight loaded before this ones' products
      float4 h[2], d[2][4];
      auto load = [&](int b) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          h[u] = *reinterpret_cast<const float4*>(&S.h1t[tk][b + 4 * u]);
#pragma unroll
          for (int j = 0; j < 4; ++j) d[u][j] = *reinterpret_cast<const float4*>(&S.d2t[ti + j][b + 4 * u]);
        }
      };
      load(0);
#pragma unroll 4
      for (int b = 0; b < kB; b += 8) {
        float4 hc[2], dc[2][4];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          hc[u] = h[u];
#pragma unroll
          for (int j = 0; j < 4; ++j) dc[u][j] = d[u][j];
        }
        if (b + 8 < kB) load(b + 8);
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            g[j] = fmaf(dc[u][j].w, hc[u].w,
                        fmaf(dc[u][j].z, hc[u].z, fmaf(dc[u][j].y, hc[u].y, fmaf(dc[u][j].x, hc[u].x, g[j]))));
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) pn[j] = adam_step(A[j], S.W2[u0 + ti + j][tk], g[j], lr, b1t, b2t);
    } else {
      float ga = 0.0f;
      if (s < kTU) ga = over_rows(S.dy, S.h2t[s]);
      else if (s >= 32 && s < 32 + kTU) ga = sum_rows(S.d2t[s - 32]);
      else if (qa == oB3) ga = sum_rows(S.dy);
      if (qa >= 0)
        pa = adam_step(Aa, s < kTU ? S.W3[u0 + s] : qa == oB3 ? S.b3 : S.b2[u0 + s - 32], ga, lr, b1t, b2t);
    }
    cluster_wait();
    if (!tile && qb >= 0) {
      float gb;
      if (s < 4 * kTU) {
        const int k = s % 4;
        gb = over_rows(S.d1t[s / 4], S.xt[k]);
        pb = adam_step(Ab, S.W1[u0 + s / 4][k], gb, lr, b1t, b2t);
      } else {
        gb = sum_rows(S.d1t[s - 32]);
        pb = adam_step(Ab, S.b1[u0 + s - 32], gb, lr, b1t, b2t);
      }
    }
    if (rank == 0 && tid == 255 && loss_hist && hist_every > 0 && step % hist_every == 0) {
      float l = 0.0f;
      for (int r = 0; r < kTrainBlocks; ++r) l += S.loss[r];
      loss_hist[step / hist_every] = l;
    }
    // --- the updated weights to every block (all have read the old ones: the
    // second barrier's arrival follows the last use of another block's units)
#pragma unroll
    for (int r = 0; r < kTrainBlocks; ++r) {
      TrainSmem& D = peer(r);
      if (tile) {
#pragma unroll
        for (int j = 0; j < 4; ++j) D.W2[u0 + ti + j][tk] = pn[j];
      } else {
        if (qa >= 0) {
          if (s < kTU) D.W3[u0 + s] = pa;
          else if (qa == oB3) D.b3 = pa;
          else D.b2[u0 + s - 32] = pa;
        }
        if (qb >= 0) {
          if (s < 4 * kTU) D.W1[u0 + s / 4][s % 4] = pb;
          else D.b1[u0 + s - 32] = pb;
        }
      }
    }
    cluster_arrive();
    cluster_wait();
  }
  // the owners' results
  if (tile) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int q = oW2 + (u0 + ti + j) * kMlpH + tk;
      P[q] = S.W2[u0 + ti + j][tk];
      m1[q] = A[j].m;
      m2[q] = A[j].v;
    }
  } else {
    if (qa >= 0) {
      P[qa] = s < kTU ? S.W3[u0 + s] : qa == oB3 ? S.b3 : S.b2[u0 + s - 32];
      m1[qa] = Aa.m;
      m2[qa] = Aa.v;
    }
    if (qb >= 0) {
      P[qb] = s < 4 * kTU ? S.W1[u0 + s / 4][s % 4] : S.b1[u0 + s - 32];
      m1[qb] = Ab.m;
      m2[qb] = Ab.v;
    }
  }
}

}  // namespace

cudaError_t launch_mlp_image(const float* params, void* image, cudaStream_t stream) {
  k_mlp_image<<<1, 256, 0, stream>>>(params, reinterpret_cast<MlpSmem*>(image));
  return cudaGetLastError();
}
size_t mlp_image_bytes() { return kMlpSmemBytes; }

}  // namespace gaps

using namespace gaps;

extern "C" {

int gaps_mlp_loss_grad(const float* params, const float* features, const float* targets, uint64_t n, float tau,
                       float* grad, float* loss, void* stream) {
  if (!params || !features || !targets || !grad || !loss || n == 0 || !(tau > 0.0f && tau < 1.0f))
    return GAPS_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemsetAsync(grad, 0, kMlpParams * sizeof(float), st) != cudaSuccess) return GAPS_ERR_CUDA;
  if (cudaMemsetAsync(loss, 0, sizeof(float), st) != cudaSuccess) return GAPS_ERR_CUDA;
  const int bs = 128;
  k_loss_grad<<<(unsigned)((n + bs - 1) / bs), bs, (kMlpParams + 1) * sizeof(float), st>>>(
      params, features, targets, n, tau, grad, loss);
  return cudaGetLastError() == cudaSuccess ? GAPS_OK : GAPS_ERR_CUDA;
}

int gaps_mlp_forward(const float* params, const float* features, uint64_t n, int bf16, float* out,
                     void* stream) {
  if (!params || !features || !out) return GAPS_ERR_INVALID_ARG;
  if (n == 0) return GAPS_OK;
  cudaStream_t st = (cudaStream_t)stream;
  if (bf16) {
    uint64_t tiles = (n + 15) / 16;
    unsigned blocks = (unsigned)((tiles + 7) / 8);
    if (blocks > 4096) blocks = 4096;
    k_forward_bf16<<<blocks, 256, 0, st>>>(params, features, n, out);
  } else {
    k_forward_f32<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(params, features, n, out);
  }
  return cudaGetLastError() == cudaSuccess ? GAPS_OK : GAPS_ERR_CUDA;
}

int gaps_mlp_train(float* params, float* adam_m, float* adam_v, const float* features, const float* targets,
                   uint64_t n, uint64_t steps, float lr, float tau, uint64_t seed, float* loss_history,
                   int history_every, void* stream) {
  if (!params || !adam_m || !adam_v || !features || !targets || n == 0) return GAPS_ERR_INVALID_ARG;
  if (!(lr > 0.0f) || !(tau > 0.0f && tau < 1.0f)) return GAPS_ERR_INVALID_ARG;
  const size_t smem = sizeof(TrainSmem);
  if (cudaFuncSetAttribute(k_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return GAPS_ERR_CUDA;
  k_train<<<kTrainBlocks, kB, smem, (cudaStream_t)stream>>>(params, adam_m, adam_v, features, targets, n, steps, lr, tau,
                                                 seed, loss_history, history_every);
  return cudaGetLastError() == cudaSuccess ? GAPS_OK : GAPS_ERR_CUDA;
}

}  // extern "C"
