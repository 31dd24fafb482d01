// CUDA-core kernels of the warm-start network around its convolutions (net_conv.cu): the backward
// of FiLM + SiLU with the per-channel reductions, the epilogue of the K-split convolutions, the
// conditioning MLP, the loss, Adam, the output's denormalisation and small helpers.
// FP32 activations and gradients are channel-major, x[c][b * H * W + y * W + x].
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "net_internal.h"
#include "net_tc.cuh"

namespace mcl {
namespace net {
namespace {

__device__ __forceinline__ float silu_f(float z) { return z / (1.f + expf(-z)); }
__device__ __forceinline__ float dsilu_f(float z) {
  const float s = 1.f / (1.f + expf(-z));
  return s * (1.f + z * (1.f - s));
}

int grid_for(int64_t n, int block, int cap) {
  int64_t g = (n + block - 1) / block;
  return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

// Block sum of NV doubles per thread (blockDim.x == 256), result in thread 0.
template <int NV>
__device__ __forceinline__ void block_sum(double* v, double (*sh)[NV]) {
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] += __shfl_down_sync(0xffffffffu, v[k], off);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < NV; ++k) sh[warp][k] = v[k];
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double s = 0.0;
      for (int w = 0; w < 8; ++w) s += sh[w][k];
      v[k] = s;
    }
  }
  __syncthreads();
}

__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  uint32_t u;
  memcpy(&u, &v, 4);
  return u;
}

// A sum of FP32 terms with the exact errors of its additions beside it (Knuth's two-sum).
struct Sum {
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = __fadd_rn(s, x), z = __fsub_rn(t, s);
    e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z)));
    s = t;
  }
};

// The lane-0 sums of a warp's N compensated sums: FP32 pairs in a fixed order (FP64 runs at 1/64
// of the FP32 rate).
template <int N>
__device__ __forceinline__ void warp_sums(Sum (&v)[N], double* out) {
#pragma unroll
  for (int k = 0; k < N; ++k) {
    for (int off = 16; off > 0; off >>= 1) {
      const float s = __shfl_down_sync(0xffffffffu, v[k].s, off);
      const float e = __shfl_down_sync(0xffffffffu, v[k].e, off);
      v[k].add(s);
      v[k].e = __fadd_rn(v[k].e, e);
    }
    if ((threadIdx.x & 31) == 0) out[k] = (double)v[k].s + (double)v[k].e;
  }
}
// Sums over each half (four warps) of a 256-thread block, FP64 across the warps: out[n] by the
// half's thread n. half_sums' out is the half's own.
template <int N>
__device__ __forceinline__ void half_sums(Sum (&v)[N], double* out) {
  __shared__ double sh[8][N];
  const int warp = threadIdx.x >> 5, t = threadIdx.x & 127;
  warp_sums<N>(v, sh[warp]);
  __syncthreads();
  if (t < N) {
    double s = 0.0;
    for (int w = warp & 4; w < (warp & 4) + 4; ++w) s += sh[w][t];
    out[t] = s;
  }
}
// Sums over the block, out[n] from thread n.
template <int N>
__device__ __forceinline__ void block_sums(Sum (&v)[N], double* out) {
  __shared__ double sh[8][N];
  warp_sums<N>(v, sh[threadIdx.x >> 5]);
  __syncthreads();
  if (threadIdx.x < N) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += sh[w][threadIdx.x];
    out[threadIdx.x] = s;
  }
}

// ---- backward of act(film(pre)) ---------------------------------------------------------------
// Block = (eight channels, a chunk of a sample's pixels): its lower half takes the first four
// channels of every pixel, the upper half the others, so that a thread's sums and loads fit 64
// registers (four blocks per SM). A thread reads four planar values of pre and dy each (coalesced
// over the threads) and writes 8 bytes of the pixel's group. Bound by memory (10 B per value) and
// the arithmetic of SiLU's derivative together; with one block per (channel, sample) the
// 16-channel layers of 256 x 256 ran 256 blocks of scalar loads (161 us at batch 16, where their
// 168 MB take 25 us), now 39 us.
template <bool FILM>
__global__ void __launch_bounds__(256, 4) act_backward_kernel(const ActBwdArgs a) {
  pdl_wait();
  const int groups = a.C / 8;
  const int g = blockIdx.x % groups, chunk = blockIdx.x / groups, b = blockIdx.y;
  const int half = threadIdx.x >> 7, t = threadIdx.x & 127;
  const int64_t P = (int64_t)a.batch * a.hw;
  const int per = (a.hw + a.chunks - 1) / a.chunks;
  const int i1 = min(a.hw, (chunk + 1) * per);
  const int c0 = g * 8 + half * 4;
  float gm[4], bt[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    gm[j] = 1.f;
    bt[j] = 0.f;
    if (FILM) {
      const float* f = a.film + (int64_t)b * a.film_stride + a.film_off;
      gm[j] = 1.f + f[c0 + j];
      bt[j] = f[a.C + c0 + j];
    }
  }
  // sums of dz and, with FiLM, of dz pre; that of dpre is gamma times that of dz
  constexpr int NS = FILM ? 8 : 4;
  Sum acc[NS];
  const float* pre_p = a.pre + (int64_t)c0 * P + (int64_t)b * a.hw;
  const float* dy_p = a.dy + (int64_t)c0 * P + (int64_t)b * a.hw;
  uint2* dst = reinterpret_cast<uint2*>(a.dpre) + ((int64_t)g * P + (int64_t)b * a.hw) * 2 + half;
  for (int i = chunk * per + t; i < i1; i += 128) {
    float pre[4], dy[4], out[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      pre[j] = __ldg(pre_p + j * P + i);
      dy[j] = __ldg(dy_p + j * P + i);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float z = FILM ? gm[j] * pre[j] + bt[j] : pre[j];
      const float dz = dy[j] * dsilu_f(z);
      out[j] = FILM ? dz * gm[j] : dz;
      acc[j].add(dz);
      if constexpr (FILM) acc[4 + j].add(dz * pre[j]);
    }
    dst[2 * (int64_t)i] = make_uint2(pack2(out[0], out[1]), pack2(out[2], out[3]));
  }
  __shared__ double total[2][NS];
  half_sums<NS>(acc, total[half]);
  __syncthreads();
  if (t < 4) {
    double* o = a.sums + (((int64_t)(c0 + t) * a.batch + b) * a.chunks + chunk) * 3;
    const double dz = total[half][t];
    o[0] = FILM ? (double)(t == 0 ? gm[0] : t == 1 ? gm[1] : t == 2 ? gm[2] : gm[3]) * dz : dz;
    o[1] = FILM ? total[half][4 % NS + t] : 0.0;
    o[2] = FILM ? dz : 0.0;
  }
}

// A warp takes four pixels of eight channels, so that every thread has one value: its (at most
// eight) partial products are loaded at once, and the eight channels of a pixel are stored as
// neighbouring 2-byte pieces. Bound by latency: a thread with all eight channels of a pixel chained
// 64 loads (12 to 17 us per layer at batch 1, where a layer's partial sums are 1 to 4 MB).
constexpr int kMaxSplits = 8;
__global__ void __launch_bounds__(256) conv_epilogue_splitk_kernel(
    const float* __restrict__ part, int splits, int batch, int Ho, int Wo, int N,
    const ConvEpilogue e) {
  pdl_wait();
  const int hw = Ho * Wo;
  const int64_t P = (int64_t)batch * hw;
  const int64_t n = (int64_t)((N + 7) / 8) * P * 8;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(t & 7);
    const int64_t r = t >> 3;
    const int g = (int)(r / P);
    const int64_t p = r - g * P;
    const int o = g * 8 + j;
    if (o >= N) continue;
    const int b = (int)(p / hw), i = (int)(p - (int64_t)b * hw);
    float v[kMaxSplits];
#pragma unroll
    for (int z = 0; z < kMaxSplits; ++z)
      if (z < splits) v[z] = part[((int64_t)z * N + o) * P + p];
    const float* f = e.film ? e.film + (int64_t)b * e.film_stride + e.film_off : nullptr;
    const float bias = __ldg(e.bias + o);
    const float gm = f ? __ldg(f + o) : 0.f, bt = f ? __ldg(f + N + o) : 0.f;
    float s = 0.f;
#pragma unroll
    for (int z = 0; z < kMaxSplits; ++z)
      if (z < splits) s += v[z];
    const float pre = s + bias;
    float zz = pre;
    if (f) zz = (1.f + gm) * pre + bt;
    if (e.pre) e.pre[(int64_t)o * P + p] = pre;
    if (!e.y) continue;
    const __nv_bfloat16 y = __float2bfloat16_rn(e.act ? zz / (1.f + expf(-zz)) : zz);
    const int yy = i / Wo, xx = i - yy * Wo;
    __nv_bfloat16* dst = e.y + (int64_t)g * e.y_group * 8 + j;
    if (!e.up) {
      dst[p * 8] = y;
    } else {
      dst += (((int64_t)b * 2 * Ho + 2 * yy) * (2 * Wo) + 2 * xx) * 8;
      dst[0] = y;
      dst[8] = y;
      dst[16 * Wo] = y;
      dst[16 * Wo + 8] = y;
    }
  }
}

// ---- conditioning MLP (sizes are tiny: batch x 3 -> H -> F) -------------------------------------
// Forward over a grid: every block rebuilds the normalised conditions c and the hidden layer
// h = SiLU(W1 c + b1) in shared memory (batch x (3 + H) values) and computes its slice of the
// batch x F outputs r = W2 h + b2; block 0 also stores c and the pre-activations a1.
__global__ void mlp_forward_kernel(const MlpArgs a) {
  extern __shared__ float sm[];
  float* c = sm;                    // [batch][3]
  float* h = sm + 3 * a.batch;      // [batch][H]
  for (int t = threadIdx.x; t < a.batch; t += blockDim.x) {
    const float Ra = a.cond_raw[3 * t], phi = a.cond_raw[3 * t + 1], dp = a.cond_raw[3 * t + 2];
    c[3 * t] = (log10f(Ra) - 4.5f) / 1.5f;
    c[3 * t + 1] = (phi - 0.025f) / 0.025f;
    c[3 * t + 2] = (dp * 1e9f - 55.f) / 45.f;
  }
  __syncthreads();
  if (blockIdx.x == 0)
    for (int t = threadIdx.x; t < a.batch * 3; t += blockDim.x) a.c[t] = c[t];
  for (int t = threadIdx.x; t < a.batch * a.H; t += blockDim.x) {
    const int b = t / a.H, j = t % a.H;
    const float s = a.b1[j] + a.W1[3 * j] * c[3 * b] + a.W1[3 * j + 1] * c[3 * b + 1] +
                    a.W1[3 * j + 2] * c[3 * b + 2];
    if (blockIdx.x == 0) a.a1[t] = s;
    h[t] = silu_f(s);
  }
  __syncthreads();
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < a.batch * a.F;
       t += gridDim.x * blockDim.x) {
    const int b = t / a.F, f = t % a.F;
    // the row's loads in blocks of 16 before their sums (in order): one at a time, each waited
    // for the cache (13 us for 64 of them)
    const float* w = a.W2 + (int64_t)f * a.H;
    float s = a.b2[f];
    int j = 0;
    for (; j + 16 <= a.H; j += 16) {
      float v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = __ldg(w + j + k);
#pragma unroll
      for (int k = 0; k < 16; ++k) s += v[k] * h[b * a.H + j + k];
    }
    for (; j < a.H; ++j) s += w[j] * h[b * a.H + j];
    a.r[t] = s;
  }
}

// Backward, second layer: gW2[f][j] = sum_b dr[b][f] h[b][j], gb2[f] = sum_b dr[b][f] (grid over
// the F x H + F outputs, sums in batch order).
__global__ void mlp_backward_w2_kernel(const MlpArgs a, const float* dr, float* gW2, float* gb2) {
  const int n = a.F * a.H;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n + a.F;
       t += gridDim.x * blockDim.x) {
    if (t < n) {
      const int f = t / a.H, j = t % a.H;
      float s = 0.f;
      for (int b = 0; b < a.batch; ++b)
        s += dr[(int64_t)b * a.F + f] * silu_f(a.a1[b * a.H + j]);
      gW2[t] = s;
    } else {
      const int f = t - n;
      float s = 0.f;
      for (int b = 0; b < a.batch; ++b) s += dr[(int64_t)b * a.F + f];
      gb2[f] = s;
    }
  }
}

// Backward, first layer: block j computes da1[b][j] = (sum_f W2[f][j] dr[b][f]) SiLU'(a1[b][j])
// for every b (warp w < batch: its lanes take every 32nd f, then a fixed shuffle tree), then
// gW1[j][i] = sum_b da1[b][j] c[b][i] and gb1[j] = sum_b da1[b][j] (in batch order).
__global__ void mlp_backward_w1_kernel(const MlpArgs a, const float* dr, float* gW1, float* gb1) {
  extern __shared__ float da1[];  // [batch]
  const int j = blockIdx.x, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int b = threadIdx.x >> 5; b < a.batch; b += nw) {
    float s = 0.f;
    int f = lane;
    for (; f + 7 * 32 < a.F; f += 8 * 32) {  // eight loads of each in flight, sums in order
      float w[8], d[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        w[k] = __ldg(a.W2 + (int64_t)(f + 32 * k) * a.H + j);
        d[k] = __ldg(dr + (int64_t)b * a.F + f + 32 * k);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) s += w[k] * d[k];
    }
    for (; f < a.F; f += 32) s += a.W2[(int64_t)f * a.H + j] * dr[(int64_t)b * a.F + f];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if (lane == 0) da1[b] = s * dsilu_f(a.a1[b * a.H + j]);
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    const int i = threadIdx.x;
    float s = 0.f;
    for (int b = 0; b < a.batch; ++b) s += i < 3 ? da1[b] * a.c[3 * b + i] : da1[b];
    if (i < 3) gW1[3 * j + i] = s;
    else gb1[j] = s;
  }
}

// ---- loss -----------------------------------------------------------------------------------
// Rest value of channel ch for a sample of volume fraction phi0 (phi and rho^w are learned as
// deviations from phi_0 and 1 - phi_0).
__device__ __forceinline__ float base_of(int ch, float phi0) {
  return ch == 3 ? phi0 : (ch == 4 ? 1.f - phi0 : 0.f);
}

// One thread per pixel, all five channels: the gradient goes straight to the output layer's dpre.
__global__ void __launch_bounds__(256) loss_kernel(const LossArgs a) {
  __shared__ double sh[8][1];
  const int chunk = blockIdx.x, b = blockIdx.y;
  const int64_t P = (int64_t)a.batch * a.hw;
  const int64_t n = kFields * P;
  const float inv_n2 = (float)(2.0 / (double)n);
  const int per = (a.hw + a.chunks - 1) / a.chunks;
  const int i1 = min(a.hw, (chunk + 1) * per);
  const float phi0 = a.cond[3 * b + 1];
  double acc[1] = {0.0};
  Sum grad[kFields];
  uint4* dst = reinterpret_cast<uint4*>(a.dpre) + (int64_t)b * a.hw;
  for (int i = chunk * per + threadIdx.x; i < i1; i += blockDim.x) {
    float o[kFields];
#pragma unroll
    for (int ch = 0; ch < kFields; ++ch) {
      const float F = a.target[((int64_t)b * kFields + ch) * a.hw + i];
      const float tgt = (F - base_of(ch, phi0) - a.norm[ch]) / a.norm[kFields + ch];
      const float d = a.out[ch * P + (int64_t)b * a.hw + i] - tgt;
      o[ch] = inv_n2 * d;
      acc[0] += (double)d * (double)d;
      grad[ch].add(o[ch]);
    }
    dst[i] = make_uint4(pack2(o[0], o[1]), pack2(o[2], o[3]), pack2(o[4], 0.f), 0u);
  }
  block_sum<1>(acc, sh);
  if (threadIdx.x == 0) a.partial[(int64_t)b * a.chunks + chunk] = acc[0] / (double)n;
  __shared__ double total[kFields];
  block_sums<kFields>(grad, total);
  __syncthreads();
  if (threadIdx.x < kFields) {
    double* s = a.sums + (((int64_t)threadIdx.x * a.batch + b) * a.chunks + chunk) * 3;
    s[0] = total[threadIdx.x];
    s[1] = s[2] = 0.0;
  }
}

__global__ void sum_partials_kernel(const double* partial, int n, double* out) {
  __shared__ double sh[8][1];
  double acc[1] = {0.0};
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc[0] += partial[i];
  block_sum<1>(acc, sh);
  if (threadIdx.x == 0) out[0] = acc[0];
}

__global__ void adam_kernel(float* p, const float* g, float* m, float* v, int64_t n, float lr,
                            float b1, float b2, float eps, float c1, float c2) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const float gt = g[t];
    const float mt = b1 * m[t] + (1.f - b1) * gt;
    const float vt = b2 * v[t] + (1.f - b2) * gt * gt;
    m[t] = mt;
    v[t] = vt;
    p[t] -= lr * (mt * c1) / (sqrtf(vt * c2) + eps);
  }
}

__global__ void geometry_kernel(uint4* X, int ny, int nx) {
  const int hw = ny * nx;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < hw; i += gridDim.x * blockDim.x) {
    const int x = i % nx, y = i / nx;
    const float xi = ((float)x + 0.5f) / (float)nx - 0.5f;
    const float eta = ((float)y + 0.5f) / (float)ny - 0.5f;
    X[i] = make_uint4(pack2(1.f, xi), pack2(eta, 4.f * xi * eta), 0u, 0u);
  }
}

// fields[b][ch][i] = base + mean[ch] + scale[ch] * out[ch][b*hw + i], then phi and rho^w shifted
// by a constant each so that their cavity means are phi_0 = cond[b][1] and 1 - phi_0: the warm
// start carries the cold start's component masses. Two launches over (chunks of a sample, sample):
// a chunk's FP64 sums of the two deviations, then the fields, every block adding its sample's
// partial sums in the same fixed order. Bound by memory (40 B read and written per node); one
// block per sample walked a sample's 5 x 65536 values with 256 threads on one SM.
// 256 x 256, batch 1: one block took 603 us; with the two launches a whole forward pass went from
// 697 us to 367 us (batch 16 ran 16 blocks).
__global__ void shift_sums_kernel(const float* out, const float* norm, int batch, int hw,
                                  double* partial) {
  __shared__ double sh[8][2];
  const int b = blockIdx.y;
  const int64_t P = (int64_t)batch * hw;
  double acc[2] = {0.0, 0.0};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < hw; i += gridDim.x * blockDim.x) {
    acc[0] += (double)(norm[3] + norm[kFields + 3] * out[3 * P + (int64_t)b * hw + i]);
    acc[1] += (double)(norm[4] + norm[kFields + 4] * out[4 * P + (int64_t)b * hw + i]);
  }
  block_sum<2>(acc, sh);
  if (threadIdx.x == 0) {
    double* o = partial + ((int64_t)b * gridDim.x + blockIdx.x) * 2;
    o[0] = acc[0];
    o[1] = acc[1];
  }
}

__global__ void denormalize_kernel(const float* out, const float* norm, const float* cond,
                                   int batch, int hw, const double* partial, float* fields) {
  __shared__ double sh[8][2];
  __shared__ float s_shift[2];
  const int b = blockIdx.y;
  const int64_t P = (int64_t)batch * hw;
  const float phi0 = cond[3 * b + 1];
  double acc[2] = {0.0, 0.0};
  for (int k = threadIdx.x; k < (int)gridDim.x; k += blockDim.x) {
    acc[0] += partial[((int64_t)b * gridDim.x + k) * 2];
    acc[1] += partial[((int64_t)b * gridDim.x + k) * 2 + 1];
  }
  block_sum<2>(acc, sh);
  if (threadIdx.x == 0) {
    // the deviations' means become zero: the fields' means are the rest values
    s_shift[0] = (float)(-acc[0] / (double)hw);
    s_shift[1] = (float)(-acc[1] / (double)hw);
  }
  __syncthreads();
#pragma unroll
  for (int ch = 0; ch < kFields; ++ch) {
    const float add = ch == 3 ? s_shift[0] : (ch == 4 ? s_shift[1] : 0.f);
    const float base = base_of(ch, phi0);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < hw; i += gridDim.x * blockDim.x)
      fields[((int64_t)b * kFields + ch) * hw + i] =
          base + ((norm[ch] + norm[kFields + ch] * out[ch * P + (int64_t)b * hw + i]) + add);
  }
}

// grid (blocks, 5): per channel, block-strided FP64 sums of x - base and (x - base)^2.
__global__ void field_moments_kernel(const float* fields, const float* cond, int n, int hw,
                                     double* partial) {
  __shared__ double sh[8][2];
  const int ch = blockIdx.y;
  const int64_t total = (int64_t)n * hw;
  double acc[2] = {0.0, 0.0};
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = t / hw, i = t % hw;
    const double x = (double)fields[(s * kFields + ch) * hw + i] -
                     (double)base_of(ch, cond[3 * s + 1]);
    acc[0] += x;
    acc[1] += x * x;
  }
  block_sum<2>(acc, sh);
  if (threadIdx.x == 0) {
    double* o = partial + ((int64_t)ch * gridDim.x + blockIdx.x) * 2;
    o[0] = acc[0];
    o[1] = acc[1];
  }
}

// p[i] = scale * u, u uniform in [-1, 1) from splitmix64 of (seed, stream, i).
__global__ void uniform_fill_kernel(float* p, int64_t n, float scale, uint64_t seed,
                                    uint32_t stream) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    uint64_t z = ((seed << 40) ^ ((uint64_t)stream << 32)) + (uint64_t)t;
    z = (z + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    const double u = (double)(z >> 11) * (1.0 / 9007199254740992.0);
    p[t] = scale * (float)(2.0 * u - 1.0);
  }
}

}  // namespace

cudaError_t launch_uniform_fill(float* p, int64_t n, float scale, uint64_t seed, uint32_t stream,
                                cudaStream_t st) {
  uniform_fill_kernel<<<grid_for(n, 256, 1024), 256, 0, st>>>(p, n, scale, seed, stream);
  return cudaGetLastError();
}

int act_chunks(int C, int batch, int hw) {
  const int groups = std::max(1, C / 8);
  return std::max(1, std::min((hw + 1023) / 1024, 608 / (groups * batch)));
}

namespace {
template <class K, class... A>
cudaError_t launch_pdl(K kernel, dim3 grid, cudaStream_t st, const A&... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}
}  // namespace

cudaError_t launch_act_backward(const ActBwdArgs& a, cudaStream_t st) {
  const dim3 grid(a.C / 8 * a.chunks, a.batch);
  return a.film ? launch_pdl(act_backward_kernel<true>, grid, st, a)
                : launch_pdl(act_backward_kernel<false>, grid, st, a);
}

cudaError_t launch_conv_epilogue_splitk(const float* part, int splits, int batch, int Ho, int Wo,
                                        int N, const ConvEpilogue& e, cudaStream_t st) {
  const int64_t n = (int64_t)((N + 7) / 8) * batch * Ho * Wo * 8;
  return launch_pdl(conv_epilogue_splitk_kernel, dim3(grid_for(n, 256, 2048)), st, part, splits,
                    batch, Ho, Wo, N, e);
}

cudaError_t launch_mlp_forward(const MlpArgs& a, cudaStream_t st) {
  const size_t sm = sizeof(float) * (size_t)a.batch * (3 + a.H);
  mlp_forward_kernel<<<grid_for((int64_t)a.batch * a.F, 256, 152), 256, sm, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_mlp_backward(const MlpArgs& a, const float* dr, float* gW1, float* gb1,
                                float* gW2, float* gb2, cudaStream_t st) {
  mlp_backward_w2_kernel<<<grid_for((int64_t)a.F * a.H + a.F, 256, 304), 256, 0, st>>>(a, dr,
                                                                                        gW2, gb2);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  mlp_backward_w1_kernel<<<a.H, 512, sizeof(float) * (size_t)a.batch, st>>>(a, dr, gW1, gb1);
  return cudaGetLastError();
}

cudaError_t launch_loss(const LossArgs& a, cudaStream_t st) {
  loss_kernel<<<dim3(a.chunks, a.batch), 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_sum_partials(const double* partial, int n, double* out, cudaStream_t st) {
  sum_partials_kernel<<<1, 256, 0, st>>>(partial, n, out);
  return cudaGetLastError();
}

cudaError_t launch_adam(float* p, const float* g, float* m, float* v, int64_t n, float lr,
                        float b1, float b2, float eps, float c1, float c2, cudaStream_t st) {
  adam_kernel<<<grid_for(n, 256, 1024), 256, 0, st>>>(p, g, m, v, n, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

cudaError_t launch_geometry(__nv_bfloat16* X, int ny, int nx, cudaStream_t st) {
  geometry_kernel<<<grid_for((int64_t)ny * nx, 256, 2048), 256, 0, st>>>(
      reinterpret_cast<uint4*>(X), ny, nx);
  return cudaGetLastError();
}

// Chunks per sample: one pass of the block over each (256 nodes) as long as the partial sums of
// the batch fit kShiftPartials and a block's own sum over them stays short (256).
cudaError_t launch_denormalize(const float* out, const float* norm, const float* cond, int batch,
                               int hw, double* partial, float* fields, cudaStream_t st) {
  const int chunks = grid_for(hw, 256, std::min(256, kShiftPartials / (2 * batch)));
  shift_sums_kernel<<<dim3(chunks, batch), 256, 0, st>>>(out, norm, batch, hw, partial);
  denormalize_kernel<<<dim3(chunks, batch), 256, 0, st>>>(out, norm, cond, batch, hw, partial,
                                                          fields);
  return cudaGetLastError();
}

cudaError_t launch_field_moments(const float* fields, const float* cond, int n, int hw,
                                 double* partial, int blocks, cudaStream_t st) {
  field_moments_kernel<<<dim3(blocks, kFields), 256, 0, st>>>(fields, cond, n, hw, partial);
  return cudaGetLastError();
}

}  // namespace net
}  // namespace mcl
