// Force surrogate network: 4 -> 64 -> 64 -> 64 -> 6 multilayer perceptron with tanh hidden units and
// a linear output, bfloat16 weights, FP32 accumulation, FP32 master weights for Adam.
//
// The network is small (9,030 parameters) and the batches are at most a few ten thousand samples, so
// the kernels are latency-shaped: tiles of 32 samples per block with weights, activations and deltas in
// shared memory and small register tiles, and for the roll-out of the bodies one cluster of 8 blocks.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/cbl.h"

namespace {

constexpr int IN = 4, H = 64, OUT = 6, NL = 4;  // NL weight layers
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + H * IN, OFF_W2 = OFF_B1 + H, OFF_B2 = OFF_W2 + H * H,
              OFF_W3 = OFF_B2 + H, OFF_B3 = OFF_W3 + H * H, OFF_W4 = OFF_B3 + H, OFF_B4 = OFF_W4 + OUT * H,
              NPARAM = OFF_B4 + OUT;
__device__ __forceinline__ float wv(const __nv_bfloat16* w, int k) { return __bfloat162float(w[k]); }

__device__ __forceinline__ void load_weights(const __nv_bfloat16* __restrict__ g, __nv_bfloat16* s) {
  for (int k = threadIdx.x; k < NPARAM; k += blockDim.x) s[k] = g[k];
  __syncthreads();
}

// forward of one sample by one thread, with the weights in shared memory
__device__ __forceinline__ void fwd_one(const __nv_bfloat16* w, const float x[IN], float y[OUT]) {
  float h1[H], h2[H];
#pragma unroll 4
  for (int o = 0; o < H; ++o) {
    float z = wv(w, OFF_B1 + o);
#pragma unroll
    for (int i = 0; i < IN; ++i) z = fmaf(wv(w, OFF_W1 + o * IN + i), x[i], z);
    h1[o] = tanhf(z);
  }
#pragma unroll 4
  for (int o = 0; o < H; ++o) {
    float z = wv(w, OFF_B2 + o);
#pragma unroll 16
    for (int i = 0; i < H; ++i) z = fmaf(wv(w, OFF_W2 + o * H + i), h1[i], z);
    h2[o] = tanhf(z);
  }
  // layer 3 overwrites h1 (no longer needed)
#pragma unroll 4
  for (int o = 0; o < H; ++o) {
    float z = wv(w, OFF_B3 + o);
#pragma unroll 16
    for (int i = 0; i < H; ++i) z = fmaf(wv(w, OFF_W3 + o * H + i), h2[i], z);
    h1[o] = tanhf(z);
  }
#pragma unroll
  for (int o = 0; o < OUT; ++o) {
    float z = wv(w, OFF_B4 + o);
#pragma unroll 16
    for (int i = 0; i < H; ++i) z = fmaf(wv(w, OFF_W4 + o * H + i), h1[i], z);
    y[o] = z;
  }
}

// Forward pass, FT samples per block: each layer is a small product out[o][s] = sum_k W[o][k] h[k][s] on
// CUDA cores (the activations stay FP32 beside bfloat16 weights, which the matrix units' operands
// cannot be), 4 outputs x 4 samples per thread from shared memory: two 16-byte loads for 16
// multiply-adds. Sums run over k in order from the bias, as one thread per sample had them (same
// bits). That form kept its activations in local memory and ran 9,030 dependent multiply-adds:
// 10,000 samples 149 us per call against 40 here (the kernel 16 of them).
constexpr int FT = 32, FST = FT + 4;  // samples per block; row stride of the [k][sample] buffers
constexpr int FWD_NT = 128;
constexpr int HW = H + 4;  // row stride of transposed weights: 16-byte loads, and stores 4 banks apart

// weights as floats, transposed to [k][o] (o contiguous)
__device__ __forceinline__ void load_transposed(const __nv_bfloat16* __restrict__ w, int no, int ni, float* __restrict__ wt,
                                                int stride) {
  for (int e = threadIdx.x; e < no * ni; e += blockDim.x) wt[(e % ni) * stride + e / ni] = __bfloat162float(w[e]);
}

// the same for a 64 x 64 layer (16-byte aligned), 8 weights per load: a warp takes 8 of 32 rows, so its
// stores fall in 32 banks
template <int NT>
__device__ __forceinline__ void load_hidden(const __nv_bfloat16* __restrict__ w, float* __restrict__ wt) {
  constexpr int N = H * H / 8 / NT;
  uint4 v[N];
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int e = threadIdx.x + q * NT;
    v[q] = *reinterpret_cast<const uint4*>(w + (e % H) * H + (e / H) * 8);
  }
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int e = threadIdx.x + q * NT, o = e % H, k0 = (e / H) * 8;
    const unsigned u[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {  // a bfloat16 is the upper half of a float
      wt[(k0 + 2 * j) * HW + o] = __uint_as_float(u[j] << 16);
      wt[(k0 + 2 * j + 1) * HW + o] = __uint_as_float(u[j] & 0xffff0000u);
    }
  }
}

// one hidden layer: out[o][s] = tanh(b[o] + sum_k wt[k][o] in[k][s]); TS samples x 4 outputs per thread
template <int NI, int TS, int NT>
__device__ __forceinline__ void hidden_layer(const float* __restrict__ wt, const __nv_bfloat16* __restrict__ bias,
                                             const float (*in)[FST], float (*out)[FST]) {
  static_assert(NT * TS * 4 == FT * H, "one tile per thread");
  const int s0 = (threadIdx.x % (FT / TS)) * TS, o0 = (threadIdx.x / (FT / TS)) * 4;
  float z[4][TS];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int j = 0; j < TS; ++j) z[q][j] = __bfloat162float(bias[o0 + q]);
#pragma unroll 8
  for (int k = 0; k < NI; ++k) {
    const float4 w = *reinterpret_cast<const float4*>(wt + k * HW + o0);
    float h[TS];
    if constexpr (TS == 4) *reinterpret_cast<float4*>(h) = *reinterpret_cast<const float4*>(&in[k][s0]);
    else *reinterpret_cast<float2*>(h) = *reinterpret_cast<const float2*>(&in[k][s0]);
#pragma unroll
    for (int j = 0; j < TS; ++j) {
      z[0][j] = fmaf(w.x, h[j], z[0][j]);
      z[1][j] = fmaf(w.y, h[j], z[1][j]);
      z[2][j] = fmaf(w.z, h[j], z[2][j]);
      z[3][j] = fmaf(w.w, h[j], z[3][j]);
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int j = 0; j < TS; ++j) out[o0 + q][s0 + j] = tanhf(z[q][j]);
}

struct FwdSmem {
  float w1[IN * HW], w2[H * HW], w3[H * HW], w4[H * OUT];  // [k][o]
  float x[IN][FST], a[H][FST], b[H][FST];
};

__global__ void __launch_bounds__(FWD_NT) k_mlp_fwd(const __nv_bfloat16* __restrict__ wg, const float* __restrict__ x,
                                                    float* __restrict__ y, int n) {
  extern __shared__ __align__(16) unsigned char raw[];
  FwdSmem& S = *reinterpret_cast<FwdSmem*>(raw);
  load_hidden<FWD_NT>(wg + OFF_W2, S.w2);
  load_hidden<FWD_NT>(wg + OFF_W3, S.w3);
  load_transposed(wg + OFF_W1, H, IN, S.w1, HW);
  load_transposed(wg + OFF_W4, OUT, H, S.w4, OUT);
  const int s0 = blockIdx.x * FT;
  for (int e = threadIdx.x; e < FT * IN; e += FWD_NT) {
    const size_t g = (size_t)s0 * IN + e;
    S.x[e % IN][e / IN] = g < (size_t)n * IN ? x[g] : 0.f;
  }
  __syncthreads();
  hidden_layer<IN, 4, FWD_NT>(S.w1, wg + OFF_B1, S.x, S.a);
  __syncthreads();
  hidden_layer<H, 4, FWD_NT>(S.w2, wg + OFF_B2, S.a, S.b);
  __syncthreads();
  hidden_layer<H, 4, FWD_NT>(S.w3, wg + OFF_B3, S.b, S.a);
  __syncthreads();
  for (int e = threadIdx.x; e < FT * OUT; e += FWD_NT) {
    const int s = e / OUT, o = e % OUT;
    if (s0 + s >= n) break;
    float z = __bfloat162float(wg[OFF_B4 + o]);
#pragma unroll 16
    for (int k = 0; k < H; ++k) z = fmaf(S.w4[k * OUT + o], S.a[k][s], z);
    y[(size_t)(s0 + s) * OUT + o] = z;
  }
}

// Training: a block takes tiles of FT samples, keeps their activations and back-propagated deltas in
// shared memory as [unit][sample], and sums its weight gradients over its tiles in registers
// (dW = sum_s delta_s h_s^T, 4 x 4 weights per thread); a cluster of four adds its blocks' through
// distributed shared memory before one atomic per weight. One thread per sample and one atomic per
// weight and 64 samples took 167 us for 3,704 samples per call with the read-back, this 60 (the kernel
// 20); its error against FP64 is 1.0e-7 against 1.3e-7 (fewer roundings of the running sums).
constexpr int TR_NT = 256, TR_CL = 4;  // threads; blocks of a cluster
struct TrainSmem {
  float wt1[IN * HW], wt2[H * HW], wt3[H * HW];  // [k][o], for the forward pass
  float w2[H * H], w3[H * H], w4[OUT * H];    // [o][k], for the backward pass
  float x[IN][FST], h1[H][FST], h2[H][FST], h3[H][FST];
  float d4[OUT][FST], da[H][FST], db[H][FST];
  float loss[TR_NT / 32];
};

// acc[p][q] += sum_s d[l + 16 p][s] a[m + 16 q][s]: rows of a warp's lanes are 36 words apart, so their
// 16-byte loads fall in different banks
__device__ __forceinline__ void outer_tile(float acc[4][4], const float (*d)[FST], const float (*a)[FST]) {
  const int l = threadIdx.x & 15, m = threadIdx.x >> 4;
#pragma unroll 2
  for (int s = 0; s < FT; s += 4) {
    float4 dv[4], av[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      dv[p] = *reinterpret_cast<const float4*>(&d[l + 16 * p][s]);
      av[p] = *reinterpret_cast<const float4*>(&a[m + 16 * p][s]);
    }
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float t = acc[p][q];
        t = fmaf(dv[p].x, av[q].x, t);
        t = fmaf(dv[p].y, av[q].y, t);
        t = fmaf(dv[p].z, av[q].z, t);
        acc[p][q] = fmaf(dv[p].w, av[q].w, t);
      }
  }
}

// sum_s d[r][s] a[s] and sum_s d[r][s] of one row pair
__device__ __forceinline__ float row_dot(const float* __restrict__ d, const float* __restrict__ a, float t) {
#pragma unroll
  for (int s = 0; s < FT; ++s) t = fmaf(d[s], a[s], t);
  return t;
}
__device__ __forceinline__ float row_sum(const float* __restrict__ d, float t) {
#pragma unroll
  for (int s = 0; s < FT; ++s) t += d[s];
  return t;
}

// out[k][s] = (sum_j w[j][k] d[j][s]) (1 - h[k][s]^2), 2 samples x 4 units per thread
template <int NO>
__device__ __forceinline__ void back_layer(const float* __restrict__ w, const float (*d)[FST], const float (*h)[FST],
                                           float (*out)[FST]) {
  const int s0 = (threadIdx.x % (FT / 2)) * 2, k0 = (threadIdx.x / (FT / 2)) * 4;
  float z[4][2] = {};
#pragma unroll 8
  for (int j = 0; j < NO; ++j) {
    const float4 wv4 = *reinterpret_cast<const float4*>(w + j * H + k0);
    const float2 dv = *reinterpret_cast<const float2*>(&d[j][s0]);
    z[0][0] = fmaf(wv4.x, dv.x, z[0][0]);
    z[0][1] = fmaf(wv4.x, dv.y, z[0][1]);
    z[1][0] = fmaf(wv4.y, dv.x, z[1][0]);
    z[1][1] = fmaf(wv4.y, dv.y, z[1][1]);
    z[2][0] = fmaf(wv4.z, dv.x, z[2][0]);
    z[2][1] = fmaf(wv4.z, dv.y, z[2][1]);
    z[3][0] = fmaf(wv4.w, dv.x, z[3][0]);
    z[3][1] = fmaf(wv4.w, dv.y, z[3][1]);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float hv = h[k0 + q][s0 + j];
      out[k0 + q][s0 + j] = z[q][j] * (1.f - hv * hv);
    }
}

// A block's gradient in shared memory, for its cluster: the parameters in order, but the rows of W2 and W3
// ST_W words apart (the threads of a warp store to rows of their own)
constexpr int ST_W = H + 1, ST_W2 = OFF_W2, ST_B2 = ST_W2 + H * ST_W, ST_W3 = ST_B2 + H, ST_B3 = ST_W3 + H * ST_W,
              ST_REST = ST_B3 + H, ST_N = ST_REST + OUT * H + OUT;
__device__ __forceinline__ int stage_of(int k) {  // where parameter k lies
  if (k < OFF_W2) return k;
  if (k < OFF_B2) return ST_W2 + (k - OFF_W2) / H * ST_W + (k - OFF_W2) % H;
  if (k < OFF_W3) return ST_B2 + k - OFF_B2;
  if (k < OFF_B3) return ST_W3 + (k - OFF_W3) / H * ST_W + (k - OFF_W3) % H;
  return ST_B3 + k - OFF_B3;
}
__device__ __forceinline__ void stage_tile(const float acc[4][4], float* __restrict__ st) {
  const int l = threadIdx.x & 15, m = threadIdx.x >> 4;
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) st[(l + 16 * p) * ST_W + m + 16 * q] = acc[p][q];
}

// Mean-squared-error gradient of a batch (added to grad) and the loss (added to *loss).
__global__ void __cluster_dims__(TR_CL, 1, 1) __launch_bounds__(TR_NT) k_mlp_grad(const __nv_bfloat16* __restrict__ wg, const float* __restrict__ x,
                                                    const float* __restrict__ t, int n, float* __restrict__ grad,
                                                    double* __restrict__ loss) {
  extern __shared__ __align__(16) unsigned char raw[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(raw);
  const int tid = threadIdx.x;
  load_hidden<TR_NT>(wg + OFF_W2, S.wt2);
  load_hidden<TR_NT>(wg + OFF_W3, S.wt3);
  load_transposed(wg + OFF_W1, H, IN, S.wt1, HW);
#pragma unroll 4
  for (int e = tid; e < H * H / 2; e += TR_NT) {  // two weights per load
    const unsigned u2 = reinterpret_cast<const unsigned*>(wg + OFF_W2)[e], u3 = reinterpret_cast<const unsigned*>(wg + OFF_W3)[e];
    reinterpret_cast<float2*>(S.w2)[e] = make_float2(__uint_as_float(u2 << 16), __uint_as_float(u2 & 0xffff0000u));
    reinterpret_cast<float2*>(S.w3)[e] = make_float2(__uint_as_float(u3 << 16), __uint_as_float(u3 & 0xffff0000u));
  }
  for (int e = tid; e < OUT * H; e += TR_NT) S.w4[e] = __bfloat162float(wg[OFF_W4 + e]);
  const float inv = 1.0f / ((float)n * OUT);
  float a2[4][4] = {}, a3[4][4] = {}, a1 = 0.f, a4[2] = {0.f, 0.f}, ab = 0.f, ab4 = 0.f, lsum = 0.f;
  const int tiles = (n + FT - 1) / FT;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int s0 = tile * FT;
    __syncthreads();  // the last tile's readers; the weights of the first
    for (int e = tid; e < FT * IN; e += TR_NT) {
      const size_t g = (size_t)s0 * IN + e;
      S.x[e % IN][e / IN] = g < (size_t)n * IN ? x[g] : 0.f;
    }
    __syncthreads();
    hidden_layer<IN, 2, TR_NT>(S.wt1, wg + OFF_B1, S.x, S.h1);
    __syncthreads();
    hidden_layer<H, 2, TR_NT>(S.wt2, wg + OFF_B2, S.h1, S.h2);
    __syncthreads();
    hidden_layer<H, 2, TR_NT>(S.wt3, wg + OFF_B3, S.h2, S.h3);
    __syncthreads();
    if (tid < FT * OUT) {
      const int s = tid % FT, o = tid / FT;
      float r = 0.f;
      if (s0 + s < n) {
        float z = __bfloat162float(wg[OFF_B4 + o]);
#pragma unroll 16
        for (int k = 0; k < H; ++k) z = fmaf(S.w4[o * H + k], S.h3[k][s], z);
        r = z - t[(size_t)(s0 + s) * OUT + o];
      }
      S.d4[o][s] = 2.f * r * inv;
      lsum += r * r * inv;
    }
    __syncthreads();
    // output layer: 6 x 64 weights, 6 biases; delta of layer 3: (W4^T d4) (1 - h3^2)
    a4[0] = row_dot(S.d4[tid / H], S.h3[tid % H], a4[0]);
    if (tid + TR_NT < OUT * H) a4[1] = row_dot(S.d4[(tid + TR_NT) / H], S.h3[(tid + TR_NT) % H], a4[1]);
    if (tid < OUT) ab4 = row_sum(S.d4[tid], ab4);
    back_layer<OUT>(S.w4, S.d4, S.h3, S.da);
    __syncthreads();
    outer_tile(a3, S.da, S.h2);
    if (tid < H) ab = row_sum(S.da[tid], ab);  // b3: threads 0..63, b2: 64..127, b1: 128..191
    back_layer<H>(S.w3, S.da, S.h2, S.db);
    __syncthreads();
    outer_tile(a2, S.db, S.h1);
    if (tid >= H && tid < 2 * H) ab = row_sum(S.db[tid - H], ab);
    back_layer<H>(S.w2, S.db, S.h1, S.da);
    __syncthreads();
    a1 = row_dot(S.da[tid / IN], S.x[tid % IN], a1);
    if (tid >= 2 * H && tid < 3 * H) ab = row_sum(S.da[tid - 2 * H], ab);
  }
  // the cluster's gradients are added pairwise, then to the FP32 gradient: a quarter of the atomics, and of
  // the roundings of a long running sum
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __syncthreads();  // the weights' last readers: the staging takes their place
  float* const st = S.wt1;
  static_assert(sizeof(float) * ST_N <= offsetof(TrainSmem, x), "staging within the weights");
  stage_tile(a3, st + ST_W3);
  stage_tile(a2, st + ST_W2);
  st[OFF_W1 + tid] = a1;
  st[ST_REST + tid] = a4[0];
  if (tid + TR_NT < OUT * H) st[ST_REST + tid + TR_NT] = a4[1];
  if (tid < 3 * H) st[tid < H ? ST_B3 + tid : (tid < 2 * H ? ST_B2 + tid - H : OFF_B1 + tid - 2 * H)] = ab;
  if (tid < OUT) st[ST_REST + OUT * H + tid] = ab4;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if ((tid & 31) == 0) S.loss[tid >> 5] = lsum;
  cluster.sync();
  const float* peer[TR_CL];
#pragma unroll
  for (int c = 0; c < TR_CL; ++c) peer[c] = cluster.map_shared_rank(st, c);
  for (int k = (int)cluster.block_rank() * TR_NT + tid; k < NPARAM; k += TR_CL * TR_NT) {
    const int q = stage_of(k);
    atomicAdd(grad + k, (peer[0][q] + peer[1][q]) + (peer[2][q] + peer[3][q]));
  }
  if (tid == 0) {
    double l = 0.0;
    for (int w = 0; w < TR_NT / 32; ++w) l += (double)S.loss[w];
    atomicAdd(loss, l);
  }
  cluster.sync();  // no block's shared memory goes before its peers have read it
}

__global__ void k_adam(float* __restrict__ w, __nv_bfloat16* __restrict__ wb, float* __restrict__ g,
                       float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= NPARAM) return;
  const float gk = g[k];
  const float mk = b1 * m[k] + (1.f - b1) * gk;
  const float vk = b2 * v[k] + (1.f - b2) * gk * gk;
  m[k] = mk;
  v[k] = vk;
  const float wk = w[k] - lr * (mk / c1) / (sqrtf(vk / c2) + eps);
  w[k] = wk;
  wb[k] = __float2bfloat16_rn(wk);
  g[k] = 0.f;
}

__global__ void k_round_bf16(const float* __restrict__ w, __nv_bfloat16* __restrict__ wb) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < NPARAM) wb[k] = __float2bfloat16_rn(w[k]);
}

}  // namespace

// ---- bodies advanced by the network's pair forces (the surrogate window, on the device) ----------
// The general form, for more bodies and pairs than k_mlp_window holds.
// One block runs `steps` semi-implicit Euler steps of nb rigid spheres under the network's forces and
// torques of the bridged pairs plus a fixed per-body bias force, with the fluid frozen. Per step,
// one thread per (pair, side) forms the pair's features in its frame (e_z from the body to its
// partner, minimum image), standardises them (clipped to the training range), runs the network with
// the weights in shared memory, and adds the de-standardised force and torque, turned back to the
// lattice frame, to its body; then one thread per free body updates V, X (periodic) and omega.
// Features and targets are those of the host-side surrogate: gap s sqrt(R*/V_L), cos(theta),
// R_i/R_j, V_L/R*^3; force over 2 pi R* sigma and torque over 2 pi R*^2 sigma, R* = 2 R_i R_j/(R_i+R_j).
struct AdvNorm {
  float xm[IN], xs[IN], xlo[IN], xhi[IN], ym[OUT], ys[OUT];
};

__device__ __forceinline__ double mimg_adv(double d, double n) { return d - n * rint(d / n); }

__global__ void __launch_bounds__(256) k_mlp_advance(const __nv_bfloat16* __restrict__ wg, double* __restrict__ X,
                                                     double* __restrict__ V, double* __restrict__ Wang,
                                                     const double* __restrict__ M, const double* __restrict__ Iinv,
                                                     const double* __restrict__ R, const int* __restrict__ fixed,
                                                     const double* __restrict__ bias, const int* __restrict__ pairs,
                                                     const double* __restrict__ VL, int nb, int npairs, int steps,
                                                     int nx, int ny, int nz, double cth, AdvNorm nm, double sigma) {
  extern __shared__ __align__(16) unsigned char raw[];
  __nv_bfloat16* w = reinterpret_cast<__nv_bfloat16*>(raw);
  double* F = reinterpret_cast<double*>(raw + ((NPARAM * sizeof(__nv_bfloat16) + 15) / 16) * 16);
  double* T = F + 3 * nb;
  load_weights(wg, w);
  const double dims[3] = {(double)nx, (double)ny, (double)nz};
  for (int it = 0; it < steps; ++it) {
    for (int k = threadIdx.x; k < 3 * nb; k += blockDim.x) F[k] = T[k] = 0.0;
    __syncthreads();
    for (int k = threadIdx.x; k < 2 * npairs; k += blockDim.x) {
      const int p = k >> 1, a = pairs[2 * p + (k & 1)], b = pairs[2 * p + 1 - (k & 1)];
      double d[3], r = 0.0;
      for (int c = 0; c < 3; ++c) {
        d[c] = mimg_adv(X[3 * b + c] - X[3 * a + c], dims[c]);
        r += d[c] * d[c];
      }
      r = sqrt(r);
      double ez[3] = {d[0] / r, d[1] / r, d[2] / r};
      const double ref[3] = {fabs(ez[0]) < 0.9 ? 1.0 : 0.0, fabs(ez[0]) < 0.9 ? 0.0 : 1.0, 0.0};
      double ex[3] = {ref[1] * ez[2] - ref[2] * ez[1], ref[2] * ez[0] - ref[0] * ez[2], ref[0] * ez[1] - ref[1] * ez[0]};
      const double en = sqrt(ex[0] * ex[0] + ex[1] * ex[1] + ex[2] * ex[2]);
      for (int c = 0; c < 3; ++c) ex[c] /= en;
      const double ey[3] = {ez[1] * ex[2] - ez[2] * ex[1], ez[2] * ex[0] - ez[0] * ex[2], ez[0] * ex[1] - ez[1] * ex[0]};
      const double Ra = R[a], Rb = R[b], Rs = 2.0 * Ra * Rb / (Ra + Rb), vl = VL[p];
      const double feat[IN] = {(r - Ra - Rb) * sqrt(Rs / vl), cth, Ra / Rb, vl / (Rs * Rs * Rs)};
      float xi[IN], yo[OUT];
      for (int i = 0; i < IN; ++i) {
        const float v = fminf(fmaxf((float)feat[i], nm.xlo[i]), nm.xhi[i]);
        xi[i] = (v - nm.xm[i]) / nm.xs[i];
      }
      fwd_one(w, xi, yo);
      const double sc = 2.0 * 3.14159265358979323846 * Rs * sigma;
      double fl[3], tl[3];
      for (int c = 0; c < 3; ++c) {
        fl[c] = (double)(yo[c] * nm.ys[c] + nm.ym[c]) * sc;
        tl[c] = (double)(yo[3 + c] * nm.ys[3 + c] + nm.ym[3 + c]) * sc * Rs;
      }
      for (int c = 0; c < 3; ++c) {  // frame rows ex, ey, ez: world = frame^T local
        atomicAdd(&F[3 * a + c], ex[c] * fl[0] + ey[c] * fl[1] + ez[c] * fl[2]);
        atomicAdd(&T[3 * a + c], ex[c] * tl[0] + ey[c] * tl[1] + ez[c] * tl[2]);
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
      if (fixed[i]) continue;
      for (int c = 0; c < 3; ++c) {
        V[3 * i + c] += (F[3 * i + c] + bias[3 * i + c]) / M[i];
        double x = X[3 * i + c] + V[3 * i + c];
        x -= dims[c] * floor(x / dims[c]);
        X[3 * i + c] = x;
        Wang[3 * i + c] += T[3 * i + c] * Iinv[i];
      }
    }
    __syncthreads();
  }
}

// The same window on a cluster of WIN_CTAS blocks, for as many bodies and pairs as its shared memory
// holds. Rows (a pair seen from one of its bodies) and bodies are shared out over the blocks; every block
// keeps all centres. Per step a block forms the features of its rows (one thread per row), runs the
// network on 16 rows at a time with one output unit's weights in each thread's registers, sends each
// row's force and torque to the block of its body, and after a cluster barrier moves its bodies and
// sends their centres to all blocks (second barrier). What does not change within the window (radii,
// scales, three of the four features) is computed once: FP64 runs at 1/64 rate here and bounds the
// geometry. The network's sums run in the order of the one-block form; a body's rows are added in
// row order instead of by atomics. 200 bodies, 60 pairs, 200 steps: 1,158 us against 12,320 (5.7 us per
// step: the network's three dependent layers about half, FP64 geometry and the two barriers the rest).
constexpr int WIN_CTAS = 8, WIN_NT = 256, WIN_ROWS = 64;  // rows per pass of a block
constexpr int ADV_SMEM_MAX = 200 * 1024;

struct WinRow {
  double gap0, scale, fs, ts;  // Ra + Rb; sqrt(R* / V_L); 2 pi R* sigma, times R*
  int a, b;
  float x[IN];  // standardised features; x[0] follows the gap
};
struct WinBody {  // one component of a body's motion
  double v, w, bias, im, ii;  // velocity, angular velocity, bias force, 1 / M, inverse inertia
  long long held;
};
struct WinSmem {
  float w1[IN * H], b1[H], b2[H], b3[H], w4[OUT][H + 4], b4[OUT + 2];
  float x[WIN_ROWS][IN], h[2][16][H + 4], y[WIN_ROWS][8];
};

__host__ __device__ inline int win_share(int n) { return (n + WIN_CTAS - 1) / WIN_CTAS; }
static size_t win_smem(int nb, int npairs) {
  const size_t rows = 2 * (size_t)npairs, own = win_share((int)std::min<size_t>(rows, 1u << 20));
  return sizeof(WinSmem) + sizeof(double) * (3 * (size_t)nb + 6 * rows) + sizeof(WinBody) * 3 * win_share(nb) +
         sizeof(WinRow) * own + sizeof(int) * (rows + win_share(nb) + 1) + 64;
}

__global__ void __cluster_dims__(WIN_CTAS, 1, 1) __launch_bounds__(WIN_NT)
    k_mlp_window(const __nv_bfloat16* __restrict__ wg, double* __restrict__ X, double* __restrict__ V,
                 double* __restrict__ Wang, const double* __restrict__ M, const double* __restrict__ Iinv,
                 const double* __restrict__ R, const int* __restrict__ fixed, const double* __restrict__ bias,
                 const int* __restrict__ pairs, const double* __restrict__ VL, int nb, int npairs, int steps, int nx,
                 int ny, int nz, double cth, AdvNorm nm, double sigma) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), tid = threadIdx.x;
  extern __shared__ __align__(16) unsigned char raw[];
  const int rows = 2 * npairs, rshare = win_share(rows), bshare = win_share(nb);
  const int r0 = min(rank * rshare, rows), nr = min(rows, r0 + rshare) - r0;
  const int b0 = min(rank * bshare, nb), nbo = min(nb, b0 + bshare) - b0;
  WinSmem& S = *reinterpret_cast<WinSmem*>(raw);
  double* const sX = reinterpret_cast<double*>(raw + (sizeof(WinSmem) + 15) / 16 * 16);
  double* const sF = sX + 3 * nb;                       // [row][6]: the rows of this block's bodies
  WinBody* const body = reinterpret_cast<WinBody*>(sF + 6 * rows);
  WinRow* const row = reinterpret_cast<WinRow*>(body + 3 * bshare);
  int* const list = reinterpret_cast<int*>(row + rshare);  // rows by body of this block
  int* const first = list + rows;
  const double dims[3] = {(double)nx, (double)ny, (double)nz}, inv[3] = {1.0 / nx, 1.0 / ny, 1.0 / nz};
  // weights: layers 2 and 3 in registers (output unit o), the rest in shared memory
  const int o = tid & (H - 1), grp = tid >> 6;
  float w2[H], w3[H];
#pragma unroll
  for (int k = 0; k < H; ++k) {
    w2[k] = __bfloat162float(wg[OFF_W2 + o * H + k]);
    w3[k] = __bfloat162float(wg[OFF_W3 + o * H + k]);
  }
  for (int e = tid; e < IN * H; e += WIN_NT) S.w1[e] = __bfloat162float(wg[OFF_W1 + e]);
  for (int e = tid; e < OUT * H; e += WIN_NT) S.w4[e / H][e % H] = __bfloat162float(wg[OFF_W4 + e]);
  if (tid < H) {
    S.b1[tid] = __bfloat162float(wg[OFF_B1 + tid]);
    S.b2[tid] = __bfloat162float(wg[OFF_B2 + tid]);
    S.b3[tid] = __bfloat162float(wg[OFF_B3 + tid]);
  }
  if (tid < OUT) S.b4[tid] = __bfloat162float(wg[OFF_B4 + tid]);
  for (int k = tid; k < 3 * nb; k += WIN_NT) sX[k] = X[k];
  for (int e = tid; e < 3 * nbo; e += WIN_NT) {
    const int i = b0 + e / 3, g = 3 * b0 + e;
    body[e] = WinBody{V[g], Wang[g], bias[g], 1.0 / M[i], Iinv[i], fixed[i]};
  }
  auto standard = [&](double f, int i) {
    const float v = fminf(fmaxf((float)f, nm.xlo[i]), nm.xhi[i]);
    return (v - nm.xm[i]) / nm.xs[i];
  };
  for (int k = tid; k < nr; k += WIN_NT) {
    const int r = r0 + k, p = r >> 1;
    WinRow w;
    w.a = pairs[2 * p + (r & 1)];
    w.b = pairs[2 * p + 1 - (r & 1)];
    const double Ra = R[w.a], Rb = R[w.b], Rs = 2.0 * Ra * Rb / (Ra + Rb), vl = VL[p];
    w.gap0 = Ra + Rb;
    w.scale = sqrt(Rs / vl);
    w.fs = 2.0 * 3.14159265358979323846 * Rs * sigma;
    w.ts = w.fs * Rs;
    w.x[0] = 0.f;
    w.x[1] = standard(cth, 1);
    w.x[2] = standard(Ra / Rb, 2);
    w.x[3] = standard(vl / (Rs * Rs * Rs), 3);
    row[k] = w;
  }
  if (tid == 0) {
    for (int k = 0; k <= nbo; ++k) first[k] = 0;
    for (int r = 0; r < rows; ++r) {
      const int a = pairs[2 * (r >> 1) + (r & 1)] - b0;
      if (a >= 0 && a < nbo) ++first[a + 1];
    }
    for (int k = 0; k < nbo; ++k) first[k + 1] += first[k];
  }
  __syncthreads();
  for (int k = tid; k < nbo; k += WIN_NT) {
    int c = first[k];
    for (int r = 0; r < rows; ++r)
      if (pairs[2 * (r >> 1) + (r & 1)] == b0 + k) list[c++] = r;
  }
  cluster.sync();
  for (int it = 0; it < steps; ++it) {
    for (int p0 = 0; p0 < nr; p0 += WIN_ROWS) {
      const int np = min(WIN_ROWS, nr - p0);
      // geometry, four lanes per row, lane c with component c (FP64 issues 16 cycles a warp whatever its
      // lanes, so the components go side by side): unit vectors ez to the partner, ex = ref x ez normalised
      // (ref the x axis, or the y axis where ez lies near x), ey = ez x ex
      const int rl = tid >> 2, c = tid & 3;
      double ezc = 0.0, exc = 0.0, eyc = 0.0;
      const bool live = rl < np;
      if (__any_sync(0xffffffffu, live)) {
        const WinRow& w = row[p0 + (live ? rl : 0)];
        const int cc = c < 3 ? c : 0;
        double d = sX[3 * w.b + cc] - sX[3 * w.a + cc];
        d -= dims[cc] * rint(d * inv[cc]);
        const int q0 = (tid & 31) & ~3;
        const double d0 = __shfl_sync(0xffffffffu, d, q0), d1 = __shfl_sync(0xffffffffu, d, q0 + 1),
                     d2 = __shfl_sync(0xffffffffu, d, q0 + 2);
        const double r2 = d0 * d0 + d1 * d1 + d2 * d2;
        const bool onx = d0 * d0 < 0.81 * r2;
        const double u = onx ? d1 : d0, s2 = u * u + d2 * d2;
        // lane 3 takes the inverse length of ex, the others that of the distance
        const double ir0 = rsqrt(c == 3 ? s2 : r2);
        const double ir = __shfl_sync(0xffffffffu, ir0, q0), ie = __shfl_sync(0xffffffffu, ir0, q0 + 3);
        ezc = d * ir;
        // ref x ez: (0, -ez2, ez1) or (ez2, 0, -ez0)
        const double e = onx ? (c == 0 ? 0.0 : (c == 1 ? -d2 : d1)) : (c == 0 ? d2 : (c == 1 ? 0.0 : -d0));
        exc = e * ie;
        // ey_c = ez_(c+1) ex_(c+2) - ez_(c+2) ex_(c+1)
        const int n1 = q0 + (c + 1) % 3, n2 = q0 + (c + 2) % 3;
        eyc = __shfl_sync(0xffffffffu, ezc, n1) * __shfl_sync(0xffffffffu, exc, n2) -
              __shfl_sync(0xffffffffu, ezc, n2) * __shfl_sync(0xffffffffu, exc, n1);
        if (live) S.x[rl][c] = c == 0 ? standard((r2 * ir - w.gap0) * w.scale, 0) : w.x[c];
      }
      __syncthreads();
      // network, 16 rows at a time: unit o of rows 4 grp .. 4 grp + 3
      for (int q0 = 0; q0 < np; q0 += 16) {
        float z[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          z[j] = S.b1[o];
          const float* xi = S.x[min(q0 + 4 * grp + j, WIN_ROWS - 1)];
#pragma unroll
          for (int i = 0; i < IN; ++i) z[j] = fmaf(S.w1[o * IN + i], xi[i], z[j]);
          S.h[0][4 * grp + j][o] = tanhf(z[j]);
        }
        __syncthreads();
        auto layer = [&](const float (&w)[H], const float* bias_, int src) {
#pragma unroll
          for (int j = 0; j < 4; ++j) z[j] = bias_[o];
#pragma unroll
          for (int k = 0; k < H; k += 4)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float4 v = *reinterpret_cast<const float4*>(&S.h[src][4 * grp + j][k]);
              z[j] = fmaf(w[k], v.x, z[j]);
              z[j] = fmaf(w[k + 1], v.y, z[j]);
              z[j] = fmaf(w[k + 2], v.z, z[j]);
              z[j] = fmaf(w[k + 3], v.w, z[j]);
            }
#pragma unroll
          for (int j = 0; j < 4; ++j) S.h[src ^ 1][4 * grp + j][o] = tanhf(z[j]);
          __syncthreads();
        };
        layer(w2, S.b2, 0);
        layer(w3, S.b3, 1);
        if (tid < 16 * OUT) {
          const int s = tid / OUT, k6 = tid % OUT;
          float v = S.b4[k6];
#pragma unroll
          for (int k = 0; k < H; k += 4) {
            const float4 a = *reinterpret_cast<const float4*>(&S.w4[k6][k]), h = *reinterpret_cast<const float4*>(&S.h[0][s][k]);
            v = fmaf(a.x, h.x, v);
            v = fmaf(a.y, h.y, v);
            v = fmaf(a.z, h.z, v);
            v = fmaf(a.w, h.w, v);
          }
          if (q0 + s < np) S.y[q0 + s][k6] = v;
        }
        __syncthreads();
      }
      // force and torque in the lattice frame, to the block that moves body a: lane c scales component c of
      // both, then forms component c in the frame's axes
      if (__any_sync(0xffffffffu, live)) {
        const WinRow& w = row[p0 + (live ? rl : 0)];
        const int cc = c < 3 ? c : 0, q0 = (tid & 31) & ~3, yr = live ? rl : 0;
        const double f = (double)(S.y[yr][cc] * nm.ys[cc] + nm.ym[cc]) * w.fs,
                     t = (double)(S.y[yr][3 + cc] * nm.ys[3 + cc] + nm.ym[3 + cc]) * w.ts;
        double fo = exc * __shfl_sync(0xffffffffu, f, q0), to = exc * __shfl_sync(0xffffffffu, t, q0);
        fo += eyc * __shfl_sync(0xffffffffu, f, q0 + 1);
        to += eyc * __shfl_sync(0xffffffffu, t, q0 + 1);
        fo += ezc * __shfl_sync(0xffffffffu, f, q0 + 2);
        to += ezc * __shfl_sync(0xffffffffu, t, q0 + 2);
        if (live && c < 3) {
          double* dst = cluster.map_shared_rank(sF, w.a / bshare) + 6 * (r0 + p0 + rl);
          dst[c] = fo;
          dst[3 + c] = to;
        }
      }
    }
    cluster.sync();
    for (int e = tid; e < 3 * nbo; e += WIN_NT) {
      const int k = e / 3, c = e - 3 * k;
      WinBody& m = body[e];
      if (m.held) continue;
      double f = m.bias, t = 0.0;
      for (int q = first[k]; q < first[k + 1]; ++q) {
        f += sF[6 * list[q] + c];
        t += sF[6 * list[q] + 3 + c];
      }
      m.v += f * m.im;
      m.w += t * m.ii;
      double x = sX[3 * b0 + e] + m.v;
      x -= dims[c] * floor(x * inv[c]);
      if (x >= dims[c]) x -= dims[c];
      if (x < 0.0) x += dims[c];
#pragma unroll
      for (int r = 0; r < WIN_CTAS; ++r) cluster.map_shared_rank(sX, r)[3 * b0 + e] = x;
    }
    cluster.sync();
  }
  for (int e = tid; e < 3 * nbo; e += WIN_NT) {
    if (body[e].held) continue;
    V[3 * b0 + e] = body[e].v;
    Wang[3 * b0 + e] = body[e].w;
    X[3 * b0 + e] = sX[3 * b0 + e];
  }
}

struct cbl_mlp {
  cudaStream_t s = nullptr;
  bool own = false;
  float* w = nullptr;  // FP32 master
  __nv_bfloat16* wb = nullptr;
  float *g = nullptr, *m = nullptr, *v = nullptr;
  double* loss = nullptr;
  int t = 0;
  int sms = 1;
};

extern "C" {

cbl_status cbl_mlp_create(int n_in, int hidden, int n_hidden_layers, int n_out, void* stream, cbl_mlp** out) {
  if (!out) return CBL_ERR_ARG;
  if (n_in != IN || hidden != H || n_hidden_layers != NL - 1 || n_out != OUT) return CBL_ERR_UNSUPPORTED;
  cbl_mlp* m = new cbl_mlp();
  if (stream) {
    m->s = (cudaStream_t)stream;
  } else {
    if (cudaStreamCreateWithFlags(&m->s, cudaStreamNonBlocking) != cudaSuccess) {
      delete m;
      return CBL_ERR_CUDA;
    }
    m->own = true;
  }
  bool ok = cudaMalloc(&m->w, NPARAM * 4) == cudaSuccess && cudaMalloc(&m->wb, NPARAM * 2) == cudaSuccess &&
            cudaMalloc(&m->g, NPARAM * 4) == cudaSuccess && cudaMalloc(&m->m, NPARAM * 4) == cudaSuccess &&
            cudaMalloc(&m->v, NPARAM * 4) == cudaSuccess && cudaMalloc(&m->loss, sizeof(double)) == cudaSuccess;
  if (!ok) {
    cbl_mlp_destroy(m);
    return CBL_ERR_OOM;
  }
  cudaMemsetAsync(m->w, 0, NPARAM * 4, m->s);
  cudaMemsetAsync(m->g, 0, NPARAM * 4, m->s);
  cudaMemsetAsync(m->m, 0, NPARAM * 4, m->s);
  cudaMemsetAsync(m->v, 0, NPARAM * 4, m->s);
  cudaMemsetAsync(m->wb, 0, NPARAM * 2, m->s);
  // (per device, and cheap: set for every network)
  cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
  cudaFuncSetAttribute(k_mlp_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FwdSmem));
  cudaFuncSetAttribute(k_mlp_advance, cudaFuncAttributeMaxDynamicSharedMemorySize, ADV_SMEM_MAX);
  cudaFuncSetAttribute(k_mlp_window, cudaFuncAttributeMaxDynamicSharedMemorySize, ADV_SMEM_MAX);
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&m->sms, cudaDevAttrMultiProcessorCount, dev);
  *out = m;
  return cudaGetLastError() == cudaSuccess ? CBL_OK : CBL_ERR_CUDA;
}

int64_t cbl_mlp_num_params(const cbl_mlp* m) { return m ? NPARAM : 0; }

cbl_status cbl_mlp_set_params(cbl_mlp* m, const float* host) {
  if (!m || !host) return CBL_ERR_ARG;
  if (cudaMemcpyAsync(m->w, host, NPARAM * 4, cudaMemcpyHostToDevice, m->s) != cudaSuccess) return CBL_ERR_CUDA;
  k_round_bf16<<<(NPARAM + 255) / 256, 256, 0, m->s>>>(m->w, m->wb);
  cudaMemsetAsync(m->m, 0, NPARAM * 4, m->s);
  cudaMemsetAsync(m->v, 0, NPARAM * 4, m->s);
  m->t = 0;
  return cudaStreamSynchronize(m->s) == cudaSuccess ? CBL_OK : CBL_ERR_CUDA;
}

cbl_status cbl_mlp_get_params(cbl_mlp* m, float* host) {
  if (!m || !host) return CBL_ERR_ARG;
  if (cudaMemcpyAsync(host, m->w, NPARAM * 4, cudaMemcpyDeviceToHost, m->s) != cudaSuccess) return CBL_ERR_CUDA;
  return cudaStreamSynchronize(m->s) == cudaSuccess ? CBL_OK : CBL_ERR_CUDA;
}

cbl_status cbl_mlp_forward(cbl_mlp* m, const float* x, float* y, int n) {
  if (!m || !x || !y || n < 0) return CBL_ERR_ARG;
  if (n == 0) return CBL_OK;
  k_mlp_fwd<<<(n + FT - 1) / FT, FWD_NT, sizeof(FwdSmem), m->s>>>(m->wb, x, y, n);
  return cudaGetLastError() == cudaSuccess ? CBL_OK : CBL_ERR_CUDA;
}

cbl_status cbl_mlp_advance(cbl_mlp* m, double* X, double* V, double* Wang, const double* M, const double* Iinv,
                           const double* R, const int* fixed, const double* bias, const int* pairs, const double* VL,
                           int nb, int npairs, int steps, const int* dims, double cos_theta, const float* norm,
                           double sigma) {
  if (!m || !X || !V || !Wang || !M || !Iinv || !R || !fixed || !bias || !dims || !norm) return CBL_ERR_ARG;
  if (nb <= 0 || nb > 2048 || npairs < 0 || (npairs && (!pairs || !VL)) || steps < 0) return CBL_ERR_ARG;
  if (dims[0] < 1 || dims[1] < 1 || dims[2] < 1 || !(sigma > 0)) return CBL_ERR_ARG;
  for (int k = 0; k < 4 * IN + 2 * OUT; ++k)
    if (!std::isfinite(norm[k])) return CBL_ERR_ARG;
  for (int k = 0; k < IN; ++k)
    if (!(norm[IN + k] > 0) || norm[2 * IN + k] > norm[3 * IN + k]) return CBL_ERR_ARG;
  if (steps == 0) return CBL_OK;
  AdvNorm nm;
  std::memcpy(&nm, norm, sizeof(nm));
  const size_t smem = ((NPARAM * sizeof(__nv_bfloat16) + 15) / 16) * 16 + sizeof(double) * 6 * (size_t)nb;
  const size_t wsm = win_smem(nb, npairs);
  if (wsm <= (size_t)ADV_SMEM_MAX) {
    k_mlp_window<<<WIN_CTAS, WIN_NT, wsm, m->s>>>(m->wb, X, V, Wang, M, Iinv, R, fixed, bias, pairs, VL, nb, npairs,
                                                  steps, dims[0], dims[1], dims[2], cos_theta, nm, sigma);
    return cudaGetLastError() == cudaSuccess ? CBL_OK : CBL_ERR_CUDA;
  }
  k_mlp_advance<<<1, 256, smem, m->s>>>(m->wb, X, V, Wang, M, Iinv, R, fixed, bias, pairs, VL, nb, npairs, steps,
                                        dims[0], dims[1], dims[2], cos_theta, nm, sigma);
  return cudaGetLastError() == cudaSuccess ? CBL_OK : CBL_ERR_CUDA;
}

cbl_status cbl_mlp_grad(cbl_mlp* m, const float* x, const float* t, int n, float* loss_host) {
  if (!m || !x || !t || n <= 0) return CBL_ERR_ARG;
  cudaMemsetAsync(m->loss, 0, sizeof(double), m->s);
  // whole clusters, one block per SM at most
  const int clusters = std::max(1, std::min(((n + FT - 1) / FT + TR_CL - 1) / TR_CL, m->sms / TR_CL));
  k_mlp_grad<<<clusters * TR_CL, TR_NT, sizeof(TrainSmem), m->s>>>(m->wb, x, t, n, m->g, m->loss);
  if (cudaGetLastError() != cudaSuccess) return CBL_ERR_CUDA;
  if (loss_host) {
    double loss = 0.0;
    if (cudaMemcpyAsync(&loss, m->loss, sizeof(loss), cudaMemcpyDeviceToHost, m->s) != cudaSuccess) return CBL_ERR_CUDA;
    if (cudaStreamSynchronize(m->s) != cudaSuccess) return CBL_ERR_CUDA;
    *loss_host = (float)loss;
  }
  return CBL_OK;
}

cbl_status cbl_mlp_read_grad(cbl_mlp* m, float* host) {
  if (!m || !host) return CBL_ERR_ARG;
  if (cudaMemcpyAsync(host, m->g, NPARAM * 4, cudaMemcpyDeviceToHost, m->s) != cudaSuccess) return CBL_ERR_CUDA;
  return cudaStreamSynchronize(m->s) == cudaSuccess ? CBL_OK : CBL_ERR_CUDA;
}

cbl_status cbl_mlp_zero_grad(cbl_mlp* m) {
  if (!m) return CBL_ERR_ARG;
  return cudaMemsetAsync(m->g, 0, NPARAM * 4, m->s) == cudaSuccess ? CBL_OK : CBL_ERR_CUDA;
}

cbl_status cbl_mlp_adam_step(cbl_mlp* m, float lr, float beta1, float beta2, float eps) {
  if (!m || !(lr > 0) || !(beta1 >= 0 && beta1 < 1) || !(beta2 >= 0 && beta2 < 1)) return CBL_ERR_ARG;
  m->t += 1;
  const float c1 = 1.f - powf(beta1, (float)m->t), c2 = 1.f - powf(beta2, (float)m->t);
  k_adam<<<(NPARAM + 255) / 256, 256, 0, m->s>>>(m->w, m->wb, m->g, m->m, m->v, lr, beta1, beta2, eps, c1, c2);
  return cudaGetLastError() == cudaSuccess ? CBL_OK : CBL_ERR_CUDA;
}

cbl_status cbl_mlp_sync(cbl_mlp* m) {
  if (!m) return CBL_ERR_ARG;
  return cudaStreamSynchronize(m->s) == cudaSuccess ? CBL_OK : CBL_ERR_CUDA;
}

cbl_status cbl_mlp_destroy(cbl_mlp* m) {
  if (!m) return CBL_OK;
  if (m->s) cudaStreamSynchronize(m->s);
  cudaFree(m->w);
  cudaFree(m->wb);
  cudaFree(m->g);
  cudaFree(m->m);
  cudaFree(m->v);
  cudaFree(m->loss);
  if (m->own) cudaStreamDestroy(m->s);
  delete m;
  return CBL_OK;
}

}  // extern "C"
