// Learned trimer screen kernels (include/rimp2_mlp.h): features, forward/backward,
// Adam, inference for the 9-64-64-64-1 SiLU network.  The forward pass uses BF16-rounded
// weights with FP32 accumulation.
//
// The gradient kernel works on tiles of samples whose activations stay in shared memory: every
// layer is a (samples x 64) x (64 x 64) product in FP32 registers, a thread owning four units
// of a sample and reading weights and activations as 16-byte rows; the latency of a tile's
// layer chain bounds a minibatch.  (One warp per sample with the weights as W[unit][k] rows,
// 32-way bank conflicts and five shuffles per weight row, took 1362 us for the gradient of a
// 512-sample minibatch, the tiles 15 us; a whole training step fell from 1370 to 20.6 us.)
// Prediction and features: see k_mlp_predict and log10_pos.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "rimp2_internal.cuh"
#include "rimp2_mlp.h"

namespace {

namespace cg = cooperative_groups;

constexpr int IN = RIMP2_MLP_IN, H = RIMP2_MLP_HIDDEN, P = RIMP2_MLP_PARAMS;
constexpr int OW1 = 0, OB1 = OW1 + H * IN, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H,
              OB3 = OW3 + H * H, OW4 = OB3 + H, OB4 = OW4 + H;
static_assert(OB4 + 1 == P, "parameter layout");
static_assert(H == 64 && OW2 % 4 == 0 && OW3 % 4 == 0, "16-byte weight rows");

constexpr int kSMs = 152;       // streaming multiprocessors of a GB300
constexpr int NT = 256;         // threads of the gradient kernel: 16 unit groups (of 4) x 16 samples
constexpr int LDH = H + 4;      // activation row stride: the rows of a warp's two samples start
                                // 4 banks apart
constexpr int LDX = 12;         // standardised input row stride

__device__ __forceinline__ float bf16_round(float x) {
  return __bfloat162float(__float2bfloat16_rn(x));
}
__device__ __forceinline__ float sigm(float z) { return 1.f / (1.f + expf(-z)); }

// BF16-rounded parameters in shared memory; Wt: [k][unit] for the forward products
struct Weights {
  float w1t[IN * H], b1[H], b2[H], b3[H], w4[H], b4, pad[3];
  float w2t[H * H], w3t[H * H];
};

// The thread's four values of unit u, inputs k..k+3, of a 64 x 64 weight matrix
__device__ __forceinline__ float4 load_w4(const float* __restrict__ w, int u, int k, bool al) {
  const float* p = w + u * H + k;
  float4 v;
  if (al) v = *(const float4*)p;
  else v = make_float4(p[0], p[1], p[2], p[3]);
  return make_float4(bf16_round(v.x), bf16_round(v.y), bf16_round(v.z), bf16_round(v.w));
}

__device__ __forceinline__ void load_weights(Weights& W, const float* __restrict__ m, bool al) {
  const int t = threadIdx.x;
  // lanes hold consecutive units, so the transposed rows are written without conflicts
  const int u = t & 63;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int k = ((t >> 6) + 4 * r) * 4;
    const float4 a = load_w4(m + OW2, u, k, al), b = load_w4(m + OW3, u, k, al);
    W.w2t[(k + 0) * H + u] = a.x; W.w2t[(k + 1) * H + u] = a.y;
    W.w2t[(k + 2) * H + u] = a.z; W.w2t[(k + 3) * H + u] = a.w;
    W.w3t[(k + 0) * H + u] = b.x; W.w3t[(k + 1) * H + u] = b.y;
    W.w3t[(k + 2) * H + u] = b.z; W.w3t[(k + 3) * H + u] = b.w;
  }
  for (int e = t; e < IN * H; e += NT) W.w1t[e] = bf16_round(m[OW1 + (e & 63) * IN + (e >> 6)]);
  if (t < H) {
    W.b1[t] = bf16_round(m[OB1 + t]);
    W.b2[t] = bf16_round(m[OB2 + t]);
    W.b3[t] = bf16_round(m[OB3 + t]);
    W.w4[t] = bf16_round(m[OW4 + t]);
    if (t == 0) W.b4 = bf16_round(m[OB4]);
  }
}

// acc[c] += sum_k in[k] w[k][4 tx + c], in: the thread's sample.  Four chains (k mod 4) added at
// the end, which round less than one and wait less for one another
__device__ __forceinline__ void product(const float* __restrict__ in, const float* __restrict__ w,
                                        int tx, float (&acc)[4]) {
  float a[4][4] = {};
#pragma unroll 4
  for (int k = 0; k < H; k += 4) {
    const float4 h = *(const float4*)(in + k);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const float4 wv = *(const float4*)(w + (k + kk) * H + 4 * tx);
      const float x = kk == 0 ? h.x : kk == 1 ? h.y : kk == 2 ? h.z : h.w;
      a[kk][0] = fmaf(wv.x, x, a[kk][0]);
      a[kk][1] = fmaf(wv.y, x, a[kk][1]);
      a[kk][2] = fmaf(wv.z, x, a[kk][2]);
      a[kk][3] = fmaf(wv.w, x, a[kk][3]);
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) acc[c] += (a[0][c] + a[1][c]) + (a[2][c] + a[3][c]);
}

__device__ __forceinline__ void set_bias(const float* b, int tx, float (&z)[4]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) z[c] = b[4 * tx + c];
}

// h = SiLU(z) and d = SiLU'(z) = s (1 + z (1 - s)) to shared memory
__device__ __forceinline__ void activate(const float (&z)[4], float* h, float* d) {
  float hv[4], dv[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float s = sigm(z[c]);
    hv[c] = z[c] * s;
    dv[c] = s * (1.f + z[c] * (1.f - s));
  }
  *(float4*)h = make_float4(hv[0], hv[1], hv[2], hv[3]);
  *(float4*)d = make_float4(dv[0], dv[1], dv[2], dv[3]);
}

// k_mlp_grad starts beside it and waits for it before its first addition
__global__ void k_zero_grad(float* g, float* loss) {
  rimp2::pdl_trigger();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < P) g[i] = 0.f;
  if (i == 0 && loss) *loss = 0.f;
}

// CTAs of a cluster of the gradient kernel, and how many of them run with an SM each: clusters
// lie within one GPC, and those past 36 share SMs (a step of 20,000 samples: with 152 CTAs 134 us,
// with 144 90)
constexpr int kCluster = 4, kGradCtas = 144;
constexpr int GS = 16;   // samples per tile of the gradient kernel: a 512-sample minibatch
                         // then spreads over 32 CTAs

struct GradSmem {
  Weights W;
  float w2n[H * H], w3n[H * H];   // [unit][k]: dh = W^T dz reads rows of k
  float xs[GS * LDX], dy[GS], rs[GS];
  float h1[GS * LDH], h2[GS * LDH], h3[GS * LDH], d1[GS * LDH], d2[GS * LDH], d3[GS * LDH];
};

// acc[a][c] += sum_s dz[s][4 ty + a] h[s][4 tx + c] over the tile's ns samples
__device__ __forceinline__ void outer(const float* dz, const float* h, int ns, int tx, int ty,
                                      float (&acc)[4][4]) {
#pragma unroll 4
  for (int s = 0; s < ns; ++s) {
    const float4 a = *(const float4*)(dz + s * LDH + 4 * ty);
    const float4 b = *(const float4*)(h + s * LDH + 4 * tx);
    const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      acc[r][0] = fmaf(av[r], b.x, acc[r][0]);
      acc[r][1] = fmaf(av[r], b.y, acc[r][1]);
      acc[r][2] = fmaf(av[r], b.z, acc[r][2]);
      acc[r][3] = fmaf(av[r], b.w, acc[r][3]);
    }
  }
}

// Sums of the CTAs of a cluster: each adds its share of the parameters over the cluster, in a
// fixed order, and adds the result to grad and loss.  img: this CTA's gradient [P], then its loss.
__device__ __forceinline__ void add_cluster(float* img, float* grad, float* loss) {
  const cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  rimp2::pdl_wait();   // k_zero_grad
  const bool al = ((uintptr_t)grad & 15) == 0;
  for (int e = 4 * ((int)cl.block_rank() * NT + (int)threadIdx.x); e < P + 1; e += 4 * kCluster * NT) {
    float4 v[kCluster];
#pragma unroll
    for (int c = 0; c < kCluster; ++c) v[c] = *(const float4*)(cl.map_shared_rank(img, c) + e);
#pragma unroll
    for (int w = kCluster / 2; w > 0; w >>= 1)
#pragma unroll
      for (int c = 0; c < w; ++c) {
        v[c].x += v[c + w].x; v[c].y += v[c + w].y;
        v[c].z += v[c + w].z; v[c].w += v[c + w].w;
      }
    if (al && e + 4 <= P) {
      asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(grad + e),
                   "f"(v[0].x), "f"(v[0].y), "f"(v[0].z), "f"(v[0].w)
                   : "memory");
    } else {
      const float x[4] = {v[0].x, v[0].y, v[0].z, v[0].w};
      for (int k = 0; k < 4; ++k)
        if (e + k < P) atomicAdd(grad + e + k, x[k]);
        else if (e + k == P && loss) atomicAdd(loss, x[k]);
    }
  }
  cl.sync();   // the others have read img
}

// Standardised inputs of the tile's first ns samples (rows idx[s0 + s] of feats, or s0 + s)
__device__ __forceinline__ void load_inputs(const float* __restrict__ feats,
                                            const int* __restrict__ idx, long long s0, int ns,
                                            const float* __restrict__ mean,
                                            const float* __restrict__ stdv, float* xs) {
  for (int e = threadIdx.x; e < GS * IN; e += NT) {
    const int s = e / IN, i = e - s * IN;
    float v = 0.f;
    if (s < ns) {
      const long long row = idx ? (long long)idx[s0 + s] : s0 + s;
      v = (feats[row * IN + i] - mean[i]) / stdv[i];
    }
    xs[s * LDX + i] = v;
  }
}

// Hidden layers 1..3 of the tile (z -> h, and SiLU' for the backward pass): units 4 tx .. + 3 of
// sample ty
__device__ __forceinline__ void hidden_layers(GradSmem& S, int tx, int ty) {
  const int row = ty * LDH, at = row + 4 * tx;
  float z[4];
  set_bias(S.W.b1, tx, z);
#pragma unroll
  for (int i = 0; i < IN; ++i) {
    const float4 wv = *(const float4*)(S.W.w1t + i * H + 4 * tx);
    const float x = S.xs[ty * LDX + i];
    z[0] = fmaf(wv.x, x, z[0]);
    z[1] = fmaf(wv.y, x, z[1]);
    z[2] = fmaf(wv.z, x, z[2]);
    z[3] = fmaf(wv.w, x, z[3]);
  }
  activate(z, S.h1 + at, S.d1 + at);
  __syncthreads();
  set_bias(S.W.b2, tx, z);
  product(S.h1 + row, S.W.w2t, tx, z);
  activate(z, S.h2 + at, S.d2 + at);
  __syncthreads();
  set_bias(S.W.b3, tx, z);
  product(S.h2 + row, S.W.w3t, tx, z);
  activate(z, S.h3 + at, S.d3 + at);
  __syncthreads();
}

// Output layer: the 16 threads of a sample sum their units
__device__ __forceinline__ float output_layer(const GradSmem& S, int tx, int ty) {
  const float4 h = *(const float4*)(S.h3 + ty * LDH + 4 * tx);
  const float* w = S.W.w4 + 4 * tx;
  float s = w[0] * h.x + w[1] * h.y + w[2] * h.z + w[3] * h.w;
#pragma unroll
  for (int off = 8; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  return s + S.W.b4;
}

// Gradient of the minibatch loss.  A CTA takes tiles blockIdx.x, blockIdx.x + gridDim.x, ...
// of GS samples and keeps its sums over them in registers (the 64 x 64 weight gradients as
// 4 x 4 blocks a thread), then the CTAs of a cluster add theirs up through distributed shared
// memory, and each parameter takes one global addition per cluster: those arrive in any order,
// and a long chain of them bounds the gradient's accuracy.  Error in norm against 64 bits,
// additions per CTA -> per cluster (and product's four chains): 32 samples 1.1e-7 -> 0.9e-7,
// 512 0.89e-7 -> 0.54e-7, 2048 1.7e-7 -> 0.86e-7, 20,000 1.8e-7 -> 0.87e-7.  It starts beside
// k_zero_grad, which pays for the cluster's barriers (a training step 21.0 -> 20.6 us).
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(NT)
k_mlp_grad(const float* __restrict__ master, const float* __restrict__ feats,
           const float* __restrict__ y, const int* __restrict__ idx, int n,
           const float* __restrict__ mean, const float* __restrict__ stdv, float* grad,
           float* loss) {
  extern __shared__ __align__(16) unsigned char smem_mlp[];
  GradSmem& S = *(GradSmem*)smem_mlp;
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const bool al_m = ((uintptr_t)master & 15) == 0;
  load_weights(S.W, master, al_m);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int e = 4 * (t + NT * r);
    *(float4*)(S.w2n + e) = load_w4(master + OW2, e / H, e % H, al_m);
    *(float4*)(S.w3n + e) = load_w4(master + OW3, e / H, e % H, al_m);
  }
  float g2[4][4] = {}, g3[4][4] = {};
  float g1[3] = {0.f, 0.f, 0.f};   // dW1 elements t, t + 256, t + 512
  float gb = 0.f, gw4 = 0.f;       // threads 0..191: a bias of layers 1..3; 192..255: dW4
  float gb4 = 0.f, lsum = 0.f;     // thread 0
  const int tiles = n / GS + (n % GS != 0);
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int s0 = tile * GS, ns = min(GS, n - s0);
    __syncthreads();   // weights loaded; the previous tile is no longer read
    load_inputs(feats, idx, s0, ns, mean, stdv, S.xs);
    __syncthreads();
    hidden_layers(S, tx, ty);
    const float yv = output_layer(S, tx, ty);
    float dy = 0.f;
    if (ty < ns) {
      const int row = idx ? idx[s0 + ty] : s0 + ty;
      const float r = yv - y[row];
      dy = 2.f * r / (float)n;
      if (tx == 0) { S.rs[ty] = r * r; S.dy[ty] = dy; }
    }
    // dz3 = dy W4 SiLU'(z3), then dz2 = (W3^T dz3) SiLU'(z2), dz1 = (W2^T dz2) SiLU'(z1), each
    // in place of its SiLU'
    float4* p3 = (float4*)(S.d3 + ty * LDH + 4 * tx);
    float4 v = *p3;
    *p3 = make_float4(dy * S.W.w4[4 * tx] * v.x, dy * S.W.w4[4 * tx + 1] * v.y,
                      dy * S.W.w4[4 * tx + 2] * v.z, dy * S.W.w4[4 * tx + 3] * v.w);
    __syncthreads();
    outer(S.d3, S.h2, ns, tx, ty, g3);
    {
      float dh[4] = {};
      product(S.d3 + ty * LDH, S.w3n, tx, dh);
      float4* p = (float4*)(S.d2 + ty * LDH + 4 * tx);
      v = *p;
      *p = make_float4(dh[0] * v.x, dh[1] * v.y, dh[2] * v.z, dh[3] * v.w);
    }
    __syncthreads();
    outer(S.d2, S.h1, ns, tx, ty, g2);
    {
      float dh[4] = {};
      product(S.d2 + ty * LDH, S.w2n, tx, dh);
      float4* p = (float4*)(S.d1 + ty * LDH + 4 * tx);
      v = *p;
      *p = make_float4(dh[0] * v.x, dh[1] * v.y, dh[2] * v.z, dh[3] * v.w);
    }
    __syncthreads();
    if (t < 192) {
      const float* d = t < 64 ? S.d1 : t < 128 ? S.d2 : S.d3;
      for (int s = 0; s < ns; ++s) gb += d[s * LDH + (t & 63)];
    } else {
      for (int s = 0; s < ns; ++s) gw4 = fmaf(S.dy[s], S.h3[s * LDH + (t & 63)], gw4);
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int e = t + NT * r;
      if (e < IN * H) {
        const int j = e / IN, i = e - j * IN;
        for (int s = 0; s < ns; ++s) g1[r] = fmaf(S.d1[s * LDH + j], S.xs[s * LDX + i], g1[r]);
      }
    }
    if (t == 0)
      for (int s = 0; s < ns; ++s) { gb4 += S.dy[s]; lsum += S.rs[s]; }
  }
  // the weights' place takes the CTA's sums
  static_assert(sizeof(Weights) >= (P + 1 + 3) / 4 * 16, "gradient and loss in 16-byte units");
  __syncthreads();
  float* img = (float*)&S.W;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int e = (4 * ty + r) * H + 4 * tx;
    *(float4*)(img + OW2 + e) = make_float4(g2[r][0], g2[r][1], g2[r][2], g2[r][3]);
    *(float4*)(img + OW3 + e) = make_float4(g3[r][0], g3[r][1], g3[r][2], g3[r][3]);
  }
#pragma unroll
  for (int r = 0; r < 3; ++r)
    if (t + NT * r < IN * H) img[OW1 + t + NT * r] = g1[r];
  if (t < 192) img[(t < 64 ? OB1 : t < 128 ? OB2 : OB3) + (t & 63)] = gb;
  else img[OW4 + (t & 63)] = gw4;
  if (t == 0) {
    img[OB4] = gb4;
    img[P] = lsum / (float)n;
  }
  add_cluster(img, grad, loss);
}

__global__ void k_mlp_adam(float* w, const float* g, float* m, float* v, float c1, float c2,
                           float lr) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P) return;
  const float gi = g[i];
  const float mi = 0.9f * m[i] + 0.1f * gi;
  const float vi = 0.999f * v[i] + 0.001f * gi * gi;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
}

// ---------------------------------------------------------------- prediction
//
// A warp takes 8 samples through all layers: weights (16 units x 16 inputs) times activations
// (16 inputs x 8 samples), m16n8k16.  A layer's results become the next one's operand by
// transposing 8 x 8 blocks between the lanes, so nothing passes through shared memory but the
// weights, and warps never wait for one another.  FP32 activations times BF16 weights stay
// what they were: an activation is cut (by truncation, without error) into three BF16 numbers
// of 8 bits each, and every product of two BF16 numbers is exact in FP32.  The leading parts
// have accumulators of their own, so the rounding of the sums is that of four additions.
// Warp-level products, because 22,018 samples are 145 an SM: a 128-row tcgen05 tile an SM
// would go through TMEM and back in every layer with most tensor cores idle in between.
// The chain of dependent instructions of a warp bounds it (SiLU: an exponential and a division
// each), so tiles are as small as the instruction allows.  22,018 predictions: 23 us with
// FP32 FMAs on tiles of 64 samples in shared memory, 18 with 16 samples a warp as the 16 rows,
// 14 now (all with the launch, in a row of calls).
constexpr int PW = 12;           // warps of a CTA, two CTAs an SM

// A operands in the order in which the lanes read them: [k step][16-unit tile][lane]
struct PredSmem {
  uint4 w1[1][4][32], w2[4][4][32], w3[4][4][32];
  float b[3][H], w4[H];
};

__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) |
         (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi)) << 16;
}
__device__ __forceinline__ bool bf16_pair_bad(uint32_t v) {
  return (v & 0x7f80u) == 0x7f80u || (v & 0x7f800000u) == 0x7f800000u;
}

// Lane's A operand of units 16 mt .. 16 mt + 15 and inputs 16 j .. 16 j + 15 of w [H][n] (n =
// IN or H; inputs from n on are zero); al: rows are 8-byte aligned; bad: a weight is not finite
__device__ __forceinline__ uint4 weight_operand(const float* __restrict__ w, int n, int j, int mt, int lane,
                                                bool al, bool& bad) {
  const int u = 16 * mt + (lane >> 2), k = 16 * j + 2 * (lane & 3);
  auto pair = [&](int uu, int kk) {
    const float* p = w + uu * n + kk;
    if (al) {
      const float2 v = *(const float2*)p;
      return bf16_pair(v.x, v.y);
    }
    return bf16_pair(kk < n ? p[0] : 0.f, kk + 1 < n ? p[1] : 0.f);
  };
  const uint4 v = make_uint4(pair(u, k), pair(u + 8, k), pair(u, k + 8), pair(u + 8, k + 8));
  bad |= bf16_pair_bad(v.x) || bf16_pair_bad(v.y) || bf16_pair_bad(v.z) || bf16_pair_bad(v.w);
  return v;
}

__device__ __forceinline__ void mma16(float (&c)[4], const uint4& a, const uint32_t (&b)[2]) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b[0]), "r"(b[1]));
}

// Transposes an 8 x 8 matrix of 16-bit elements, two of row lane / 4 in every lane
__device__ __forceinline__ uint32_t transpose8(uint32_t x) {
  uint32_t y;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

// (x, y) as three packed BF16 pairs whose sum they are (8 bits each; a trailing part below
// the smallest subnormal is lost); an infinite x or y is its own leading part
__device__ __forceinline__ void split3(float x, float y, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
  const uint32_t ux = __float_as_uint(x), uy = __float_as_uint(y);
  p0 = __byte_perm(ux, uy, 0x7632);
  const float rx = isinf(x) ? 0.f : x - __uint_as_float(ux & 0xffff0000u);
  const float ry = isinf(y) ? 0.f : y - __uint_as_float(uy & 0xffff0000u);
  p1 = __byte_perm(__float_as_uint(rx), __float_as_uint(ry), 0x7632);
  const float sx = rx - __uint_as_float(__float_as_uint(rx) & 0xffff0000u);
  const float sy = ry - __uint_as_float(__float_as_uint(ry) & 0xffff0000u);
  p2 = __byte_perm(__float_as_uint(sx), __float_as_uint(sy), 0x7632);
}

// One layer of the warp's 8 samples: h[mt][0 / 1] = SiLU(W x + b) of unit 16 mt + lane / 4 and
// samples 2 (lane % 4), + 1; h[mt][2 / 3] of that unit + 8.  KS: k steps; x[p][j]: part p of
// the activations, step j.
template <int KS>
__device__ __forceinline__ void pred_layer(const uint32_t (&x)[3][KS][2], const uint4 (*w)[4][32],
                                           const float* bias, int lane, float (&h)[4][4]) {
  float hi[4][4] = {}, lo[4][4] = {};
#pragma unroll
  for (int j = 0; j < KS; ++j)
#pragma unroll
    for (int mt = 0; mt < 4; ++mt) {
      const uint4 a = w[j][mt][lane];
      mma16(hi[mt], a, x[0][j]);
      mma16(lo[mt], a, x[2][j]);
      mma16(lo[mt], a, x[1][j]);
    }
#pragma unroll
  for (int mt = 0; mt < 4; ++mt) {
    const float b0 = bias[16 * mt + (lane >> 2)], b1 = bias[16 * mt + 8 + (lane >> 2)];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float z = hi[mt][c] + (lo[mt][c] + (c < 2 ? b0 : b1));
      h[mt][c] = z * sigm(z);
    }
  }
}

__device__ __forceinline__ void next_operand(const float (&h)[4][4], uint32_t (&x)[3][4][2]) {
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      uint32_t p[3];
      split3(h[j][2 * r], h[j][2 * r + 1], p[0], p[1], p[2]);
#pragma unroll
      for (int q = 0; q < 3; ++q) x[q][j][r] = transpose8(p[q]);
    }
}

// One sample with FP32 FMAs.  For weights that are not finite: an infinite weight times an
// activation's zero part would be NaN instead of nothing.
__device__ __noinline__ float predict_one(const float* __restrict__ m, const float* __restrict__ x,
                                          const float* __restrict__ mean, const float* __restrict__ stdv) {
  float in[H], h[H];
  for (int i = 0; i < IN; ++i) in[i] = (x[i] - mean[i]) / stdv[i];
  for (int l = 0; l < 3; ++l) {
    const float* w = m + (l == 0 ? OW1 : l == 1 ? OW2 : OW3);
    const float* b = m + (l == 0 ? OB1 : l == 1 ? OB2 : OB3);
    const int n = l == 0 ? IN : H;
    for (int u = 0; u < H; ++u) {
      float z = bf16_round(b[u]);
      for (int k = 0; k < n; ++k) z = fmaf(bf16_round(w[u * n + k]), in[k], z);
      h[u] = z * sigm(z);
    }
    for (int u = 0; u < H; ++u) in[u] = h[u];
  }
  float y = 0.f;
  for (int u = 0; u < H; ++u) y = fmaf(bf16_round(m[OW4 + u]), in[u], y);
  return y + bf16_round(m[OB4]);
}

__global__ void __launch_bounds__(32 * PW, 2)
k_mlp_predict(const float* __restrict__ master, const float* __restrict__ feats, long long n,
              const float* __restrict__ mean, const float* __restrict__ stdv,
              float* __restrict__ out) {
  __shared__ PredSmem S;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  bool bad = false;
  const bool al = ((uintptr_t)master & 7) == 0;
#pragma unroll
  for (int e = t; e < 4 * 4 * 32; e += 32 * PW) {
    const int j = e >> 7, mt = (e >> 5) & 3;
    S.w2[j][mt][lane] = weight_operand(master + OW2, H, j, mt, lane, al, bad);
    S.w3[j][mt][lane] = weight_operand(master + OW3, H, j, mt, lane, al, bad);
  }
  if (warp >= PW - 4) S.w1[0][warp - (PW - 4)][lane] = weight_operand(master + OW1, IN, 0, warp - (PW - 4), lane, false, bad);
  if (t < H) {
    S.b[0][t] = bf16_round(master[OB1 + t]);
    S.b[1][t] = bf16_round(master[OB2 + t]);
    S.b[2][t] = bf16_round(master[OB3 + t]);
    S.w4[t] = bf16_round(master[OW4 + t]);
  }
  const float b4 = bf16_round(master[OB4]);
  bad = __syncthreads_or(bad);
  const long long tiles = n / 8 + (n % 8 != 0);
  // neighbouring tiles go to different SMs, so a few thousand samples reach all of them; the
  // second CTA of an SM starts with other warps (schedulers) than the first
  const int slot = (warp + (blockIdx.x / kSMs) * 2) % PW;
  for (long long tile = (long long)slot * gridDim.x + blockIdx.x; tile < tiles;
       tile += (long long)PW * gridDim.x) {
    const long long s0 = tile * 8;
    if (bad) {
      if (lane < 8 && s0 + lane < n) out[s0 + lane] = predict_one(master, feats + (s0 + lane) * IN, mean, stdv);
      continue;
    }
    const int g = lane >> 2, k = 2 * (lane & 3);
    auto input = [&](int i) {
      return s0 + g < n && i < IN ? (feats[(s0 + g) * IN + i] - mean[i]) / stdv[i] : 0.f;
    };
    uint32_t x1[3][1][2], x[3][4][2];
#pragma unroll
    for (int r = 0; r < 2; ++r)
      split3(input(k + 8 * r), input(k + 8 * r + 1), x1[0][0][r], x1[1][0][r], x1[2][0][r]);
    float h[4][4];
    pred_layer<1>(x1, S.w1, S.b[0], lane, h);
    next_operand(h, x);
    pred_layer<4>(x, S.w2, S.b[1], lane, h);
    next_operand(h, x);
    pred_layer<4>(x, S.w3, S.b[2], lane, h);
    // output layer: each lane's 8 units of two samples, then the eight lanes of a sample
    float y0 = 0.f, y1 = 0.f;
#pragma unroll
    for (int mt = 0; mt < 4; ++mt) {
      const float w0 = S.w4[16 * mt + g], w1 = S.w4[16 * mt + 8 + g];
      y0 = fmaf(w1, h[mt][2], fmaf(w0, h[mt][0], y0));
      y1 = fmaf(w1, h[mt][3], fmaf(w0, h[mt][1], y1));
    }
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) {
      y0 += __shfl_xor_sync(0xffffffffu, y0, off);
      y1 += __shfl_xor_sync(0xffffffffu, y1, off);
    }
    if (g == 0) {
      if (s0 + k < n) out[s0 + k] = y0 + b4;
      if (s0 + k + 1 < n) out[s0 + k + 1] = y1 + b4;
    }
  }
}

__device__ __forceinline__ void sort3(float& a, float& b, float& c) {
  float t;
  if (a > b) { t = a; a = b; b = t; }
  if (b > c) { t = b; b = c; c = t; }
  if (a > b) { t = a; a = b; b = t; }
}

// log10 of x >= 1e-16 (or inf, NaN) in FP64: x = 2^e m with m in [0.71, 1.42); with c near 1/m
// from a table of 1/128 steps, log10(x) = e log10(2) - log10(c) + log10(1 + r), r = m c - 1
// (|r| < 2^-7), by the Taylor series of log(1 + r) to r^8.  Around x = 1 both e and log10(c)
// vanish, so nothing cancels: at most 1.6 units in the last place of the FP64 result anywhere
// (emulated with exact rationals; the CUDA library states 2), in 13 FP64 instructions.
constexpr double kLog10Of2 = 0.30102999566398119521;
constexpr double kLog10OfE = 0.43429448190325182765, kLog10OfELow = 1.0983196502167650e-17;
constexpr int kLogUpper = 53;   // first step of m in [1, 2) that is taken as 2^(e + 1) m / 2

// a b = p + the returned remainder, exactly (Dekker)
constexpr double product_rest(double a, double b, double p) {
  const double ta = 134217729.0 * a, ah = ta - (ta - a), al = a - ah;
  const double tb = 134217729.0 * b, bh = tb - (tb - b), bl = b - bh;
  return ((ah * bh - p) + ah * bl + al * bh) + al * bl;
}

// -log10(c), 0.7 < c < 1.42, to an ulp: -2 atanh(z) / log(10), z = (c - 1) / (c + 1), with the
// rounding errors of z and of the last product carried along
constexpr double minus_log10(double c) {
  const double n = c - 1.0, d = c + 1.0, dl = c < 1.0 ? 1.0 - (d - c) : c - (d - 1.0);
  const double z = n / d, zd = z * d, zl = ((n - zd) - product_rest(z, d, zd) - z * dl) / d, z2 = z * z;
  double q = 0.0;
  for (int k = 45; k > 1; k -= 2) q = q * z2 + 1.0 / k;
  const double t = zl + z * (z2 * q), p = z * kLog10OfE;
  return -2.0 * (p + (product_rest(z, kLog10OfE, p) + kLog10OfE * t + kLog10OfELow * z));
}

struct LogTable { double2 e[128]; };   // (c, -log10(c), or -log10(2 c) from kLogUpper on)
constexpr LogTable log_table() {
  LogTable t{};
  for (int i = 0; i < 128; ++i) {
    const double c = i == 0 ? 1.0 : i == 127 ? 0.5 : 1.0 / (1.0 + (i + 0.5) / 128.0);
    t.e[i].x = c;
    t.e[i].y = i == 0 || i == 127 ? 0.0 : minus_log10(i < kLogUpper ? c : 2.0 * c);
  }
  return t;
}
__device__ const LogTable g_log_table = log_table();

__device__ __forceinline__ float log10_pos(double x) {
  const long long u = __double_as_longlong(x);
  const int ef = (int)(u >> 52) & 0x7ff, i = (int)(u >> 45) & 127;
  if (ef == 0x7ff) return (float)fabs(x);
  const double m = __longlong_as_double((u & 0x000fffffffffffffll) | 0x3ff0000000000000ll);
  const double2 t = g_log_table.e[i];
  const double r = fma(m, t.x, -1.0);
  double p = -kLog10OfE / 8.0;
  p = fma(p, r, kLog10OfE / 7.0);
  p = fma(p, r, -kLog10OfE / 6.0);
  p = fma(p, r, kLog10OfE / 5.0);
  p = fma(p, r, -kLog10OfE / 4.0);
  p = fma(p, r, kLog10OfE / 3.0);
  p = fma(p, r, -kLog10OfE / 2.0);
  p = fma(p, r, kLog10OfE);
  return (float)fma(p, r, fma((double)(ef - 1023 + (i >= kLogUpper)), kLog10Of2, t.y));
}

// FP64 instructions bound it (a warp's takes the SM's pipe for 16 clocks): log10_pos needs a
// quarter of the library logarithm's, 22,018 trimers take 9.9 us instead of 13.9 (calls in a row).
__global__ void k_screen_features(const double* __restrict__ cen, const int* __restrict__ nocc,
                                  int n, const int* __restrict__ tri, long long nt,
                                  const double* __restrict__ dde, float* __restrict__ f) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nt) return;
  const int I = tri[3 * t], J = tri[3 * t + 1], K = tri[3 * t + 2];
  auto d = [&](int a, int b) {
    const double dx = cen[3 * a] - cen[3 * b], dy = cen[3 * a + 1] - cen[3 * b + 1],
                 dz = cen[3 * a + 2] - cen[3 * b + 2];
    return (float)sqrt(dx * dx + dy * dy + dz * dz);
  };
  auto lg = [&](int a, int b) { return log10_pos(fabs(dde[(long long)a * n + b]) + 1e-16); };
  float e0 = lg(I, J), e1 = lg(I, K), e2 = lg(J, K);
  sort3(e0, e1, e2);
  float d0 = d(I, J), d1 = d(I, K), d2 = d(J, K);
  sort3(d0, d1, d2);
  float n0 = (float)nocc[I], n1 = (float)nocc[J], n2 = (float)nocc[K];
  sort3(n0, n1, n2);
  float* o = f + t * IN;
  o[0] = d0; o[1] = d1; o[2] = d2;
  o[3] = n0; o[4] = n1; o[5] = n2;
  o[6] = e0; o[7] = e1; o[8] = e2;
}

int check(cudaError_t e) {
  if (e != cudaSuccess) { cudaGetLastError(); return RIMP2_ERR_CUDA; }
  return RIMP2_OK;
}

}  // namespace

extern "C" int rimp2_screen_features(const double* centroids, const int32_t* nocc, int32_t n,
                                     const int32_t* trimers, int64_t nt, const double* dimer_de,
                                     float* feats, void* stream) {
  if (n < 0 || nt < 0 || (nt > 0 && (!centroids || !nocc || !trimers || !dimer_de || !feats)))
    return RIMP2_ERR_BAD_ARG;
  if (nt == 0) return RIMP2_OK;
  // 64-thread blocks: 20,000 trimers should reach every SM's FP64 unit
  k_screen_features<<<(unsigned)((nt + 63) / 64), 64, 0, (cudaStream_t)stream>>>(
      centroids, nocc, n, trimers, nt, dimer_de, feats);
  return check(cudaGetLastError());
}

extern "C" int rimp2_mlp_grad(const float* master, const float* feats, const float* y,
                              const int32_t* idx, int32_t n, const float* mean, const float* stdv,
                              float* grad, float* loss, void* stream) {
  if (n <= 0 || !master || !feats || !y || !mean || !stdv || !grad) return RIMP2_ERR_BAD_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const int smem = (int)sizeof(GradSmem);
  if (cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
      cudaSuccess)
    return check(cudaGetLastError());
  k_zero_grad<<<(P + 255) / 256, 256, 0, s>>>(grad, loss);
  // one CTA per tile, rounded up to whole clusters; more tiles are looped over
  const int tiles = n / GS + (n % GS != 0);
  const int ctas = tiles < kGradCtas ? (tiles + kCluster - 1) / kCluster * kCluster : kGradCtas;
  return check(rimp2::launch_pdl(k_mlp_grad, (unsigned)ctas, NT, smem, s, true, master, feats, y, idx, n, mean,
                                 stdv, grad, loss));
}

extern "C" int rimp2_mlp_adam(float* master, const float* grad, float* m, float* v, int32_t t,
                              float lr, void* stream) {
  if (!master || !grad || !m || !v || t < 1) return RIMP2_ERR_BAD_ARG;
  const float c1 = 1.f - powf(0.9f, (float)t), c2 = 1.f - powf(0.999f, (float)t);
  k_mlp_adam<<<(P + 255) / 256, 256, 0, (cudaStream_t)stream>>>(master, grad, m, v, c1, c2, lr);
  return check(cudaGetLastError());
}

extern "C" int rimp2_mlp_predict(const float* master, const float* feats, int64_t n,
                                 const float* mean, const float* stdv, float* out, void* stream) {
  if (n < 0 || (n > 0 && (!master || !feats || !mean || !stdv || !out))) return RIMP2_ERR_BAD_ARG;
  if (n == 0) return RIMP2_OK;
  // two CTAs an SM: up to 29,184 samples each tile of 8 has a warp of its own
  const long long tiles = n / 8 + (n % 8 != 0);
  const long long blocks = tiles < 2 * kSMs ? tiles : 2 * kSMs;
  k_mlp_predict<<<(unsigned)blocks, 32 * PW, 0, (cudaStream_t)stream>>>(master, feats, n, mean, stdv, out);
  return check(cudaGetLastError());
}
