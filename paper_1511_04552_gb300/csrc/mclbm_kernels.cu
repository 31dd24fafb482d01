// Non-step kernels of libmclbm (initial fill, streaming-only test hook, fields, reductions,
// state copies), templated on the storage element type, and the host-side dispatch by
// storage type. The step kernels are in mclbm_device.cuh / mclbm_step_*.cu.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <cfloat>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "mclbm_device.cuh"

namespace mcl {

// ---- streaming only (test hook) -------------------------------------------------------------
template <class T>
__global__ void stream_only_kernel(const T* __restrict__ src, T* __restrict__ dst, const Layout L,
                                   float s) {
  const int64_t n = (int64_t)L.nx * L.ny;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % L.nx), j = (int)(t / L.nx);
    float fw[kQ], fp[kQ], g[kQ];
    pull_node<T, true>(src, L, i, j, fw, fp, g, s);
    const size_t o = (size_t)j * L.pitch + i;
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
      dst[(size_t)q * L.plane + o] = Elem<T>::put(fw[q]);
      dst[(size_t)(kQ + q) * L.plane + o] = Elem<T>::put(fp[q]);
      dst[(size_t)(2 * kQ + q) * L.plane + o] = Elem<T>::put(g[q]);
    }
    if (L.np == kPlanes2) {  // g^p
      pull_thermal<T>(src, L, i, j, 3 * kQ, g, s);
#pragma unroll
      for (int q = 0; q < kQ; ++q) dst[(size_t)(3 * kQ + q) * L.plane + o] = Elem<T>::put(g[q]);
    }
  }
}

// a + b = s + e exactly (Knuth's two-sum; no operation below can be contracted)
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
  return s;
}

// ---- initial equilibrium (Eqs 26-27) ---------------------------------------------------------
// One node in FP64 from the caller's fields, so that the stored values are correctly rounded.
template <class T>
__device__ __noinline__ void init_node_fp64(T* __restrict__ dst, const Layout& L,
                                            const StepConsts& k, const float* __restrict__ warm,
                                            int warm_rho, int i, int j) {
  const size_t n = (size_t)L.nx * L.ny, t = (size_t)j * L.nx + i;
  const double ux = warm[t], uy = warm[n + t], th = warm[2 * n + t], phi = warm[3 * n + t];
  // rho^w = 1 - phi (or the caller's rho^w field), rho^p = phi rho_f / rho_p, as deviations from
  // the initial values
  const double drw = (warm_rho ? (double)warm[4 * n + t] : 1.0 - phi) - k.rho_w0_d;
  const double drp = phi / k.fr_d - k.rho_p0_d;
  const double dth = th - (0.5 - ((double)i + 0.5) / (double)L.nx);
  const double rw = k.rho_w0_d + drw, rp = k.rho_p0_d + drp;
  const double usq = 1.5 * (ux * ux + uy * uy);
  const size_t o = (size_t)j * L.pitch + i;
#pragma unroll
  for (int q = 0; q < kQ; ++q) {
    const double eu = (double)ex(q) * ux + (double)ey(q) * uy;
    const double P = eu * (3.0 + 4.5 * eu) - usq;
    const double W = q == 0 ? 4.0 / 9.0 : (q <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
    dst[(size_t)q * L.plane + o] = Elem<T>::put((float)(W * (drw + rw * P)));
    dst[(size_t)(kQ + q) * L.plane + o] = Elem<T>::put((float)(W * (drp + rp * P)));
    const T g = Elem<T>::put((float)(W * (dth + th * P)));
    dst[(size_t)(2 * kQ + q) * L.plane + o] = g;
    if (L.np == kPlanes2) dst[(size_t)(3 * kQ + q) * L.plane + o] = g;
  }
}

// Unevaluated sums h + l of two FP32 numbers (Dekker; products by fma): about 2^-46 relative to
// the largest term.
struct Two {
  float h, l;
};
__device__ __forceinline__ Two fast_two(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ Two two_of(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ Two operator+(Two a, Two b) {
  float e;
  const float s = two_sum(a.h, b.h, e);
  return fast_two(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ Two operator-(Two a) { return {-a.h, -a.l}; }
__device__ __forceinline__ Two operator*(Two a, Two b) {
  const float p = __fmul_rn(a.h, b.h);
  return fast_two(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ Two times(Two a, float b) {
  const float p = __fmul_rn(a.h, b);
  return fast_two(p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p)));
}
__device__ __forceinline__ Two product(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}

// a / b from inv = 1 / b rounded to nearest: the product corrected by its remainder, which rounds
// like the division itself (Markstein, IBM J. Res. Dev. 34, 1990).
__device__ __forceinline__ double quotient(double a, double b, double inv) {
  const double q = a * inv;
  return __fma_rn(__fma_rn(-q, b, a), inv, q);
}

// The equilibria of the caller's fields, W_q (d + r P_q) with d the deviation and r the absolute
// value of rho^w, rho^p and theta. GB300 does 2 FP64 operations per clock and SM against 128 in
// FP32, and the 27 polynomials in FP64 (about 160 operations per node) were all that the fill
// waited for: 276 us on 1024 x 1024, where its 130 MB take 19 us. So only the cancelling
// subtractions stay in FP64; the polynomials run in pairs of FP32 numbers, and a value whose
// rounding to FP32 their error could decide (Ziv's test: adding and subtracting a bound of the
// error does not round to the same number) sends its node to init_node_fp64. The stored values
// are therefore those of the FP64 evaluation; about one node in 2000 takes the second way.
// 1024 x 1024: 276 us before, 105 us now, still bound by the conversions and subtractions that
// stay in FP64 (its pipe 81 % active).
template <class T>
__global__ void __launch_bounds__(256)
    init_kernel(T* __restrict__ dst, const Layout L, const StepConsts k,
                const float* __restrict__ warm, int warm_rho) {
  const uint32_t n = (uint32_t)L.nx * (uint32_t)L.ny;
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const int j = (int)(t / (uint32_t)L.nx), i = (int)(t - (uint32_t)j * (uint32_t)L.nx);
    const size_t o = (size_t)j * L.pitch + i;
    if (!warm) {  // at rest on the conduction profile every deviation is zero
      for (int p = 0; p < L.np; ++p) dst[(size_t)p * L.plane + o] = Elem<T>::put(0.0f);
      continue;
    }
    const float ux = warm[t], uy = warm[(size_t)n + t], thf = warm[2 * (size_t)n + t];
    const float phi = warm[3 * (size_t)n + t];
    const float rwf = warm_rho ? warm[4 * (size_t)n + t] : 0.0f;
    const double phid = phi;
    const double dw = (warm_rho ? (double)rwf : 1.0 - phid) - k.rho_w0_d;
    const double dp = quotient(phid, k.fr_d, k.inv_fr_d) - k.rho_p0_d;
    const double dt =
        (double)thf - (0.5 - quotient((double)i + 0.5, (double)L.nx, k.inv_nx_d));
    Two d[3] = {two_of(dw), two_of(dp), two_of(dt)};
    Two r[3];
    r[0].h = warm_rho ? rwf : two_sum(1.0f, -phi, r[0].l);
    if (warm_rho) r[0].l = 0.0f;
    r[1] = times({k.inv_fr_h, k.inv_fr_l}, phi);
    r[2] = {thf, 0.0f};
    // P_q = 3 e.u + 4.5 (e.u)^2 - 1.5 u.u: the even part of each axis and diagonal, the odd part
    const Two A = product(ux, ux), B = product(uy, uy), C = times(product(ux, uy), 9.0f);
    const Two AB3 = times(A + B, 3.0f);
    const Two even[5] = {times(A + B, -1.5f), times(A, 3.0f) + times(B, -1.5f),
                         times(B, 3.0f) + times(A, -1.5f), AB3 + C, AB3 + -C};
    float el, fl;
    const float e1 = two_sum(ux, uy, el), e2 = two_sum(uy, -ux, fl);
    const Two odd[5] = {{0.0f, 0.0f}, product(3.0f, ux), product(3.0f, uy),
                        times({e1, el}, 3.0f), times({e2, fl}, 3.0f)};
    // The terms of set s weigh at most |d| + |r| (odd and even parts of P); the pairs above err by
    // at most about 2^-43 of that. Terms so small that FP32 underflow could spoil the low parts
    // are in doubt from the start (all zero is exact); so is NaN, which fails every comparison.
    const float pm = 3.0f * (fabsf(ux) + fabsf(uy)) + 7.5f * (A.h + B.h);
    bool doubt = false;
    float err[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      const float weight = fabsf(d[s].h) + fabsf(r[s].h) * pm;
      err[s] = 0x1p-42f * weight;
      doubt = doubt || !(weight >= 0x1p-80f || weight == 0.0f);
    }
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
      // q of (q, -q): 0, 1, 2, 5, 6 (e_6 = (-1, 1)); the odd part of -q is negated
      const int pr = q == 0 ? 0 : (q == 1 || q == 3 ? 1 : (q == 2 || q == 4 ? 2 :
                                                            (q == 5 || q == 7 ? 3 : 4)));
      const bool minus = q == 3 || q == 4 || q == 7 || q == 8;
      const Two P = q == 0 ? even[0] : even[pr] + (minus ? -odd[pr] : odd[pr]);
      const double Wd = q == 0 ? 4.0 / 9.0 : (q <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
      const Two W = {(float)Wd, (float)(Wd - (double)(float)Wd)};
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const Two v = W * (d[s] + r[s] * P);
        const float e = W.h * err[s];
        doubt = doubt || !(__fadd_rn(v.h, __fadd_rn(v.l, e)) == v.h &&
                           __fadd_rn(v.h, __fsub_rn(v.l, e)) == v.h);
        const T out = Elem<T>::put(v.h);
        dst[(size_t)(s * kQ + q) * L.plane + o] = out;
        if (s == 2 && L.np == kPlanes2) dst[(size_t)(3 * kQ + q) * L.plane + o] = out;
      }
    }
    if (doubt) init_node_fp64<T>(dst, L, k, warm, warm_rho, i, j);
  }
}

// ---- macroscopic fields of the post-stream state ----------------------------------------------
// thp: the particles' thermal set's deviation (= m.th with one set); v[kFields].
__device__ __forceinline__ void node_fields(const StepConsts& k, const Moments& m, float thp,
                                            int i, float* v) {
  const float rw = k.rho_w0 + m.rw, rp = k.rho_p0 + m.rp;
  const float rho = rw + rp;
  const float tc = theta_c(k, i);
  v[0] = (m.mwx + m.mpx) / rho;
  v[1] = (m.mwy + m.mpy) / rho;
  v[2] = tc + (k.two_sets ? mixture_dev(k, rw, rp, m.th, thp) : m.th);
  v[8] = tc + m.th;
  v[9] = tc + thp;
  v[3] = rp * k.phi_per_rho_p;
  v[4] = rw;
  v[5] = rp;
  const bool has_p = k.has_p && rp > 1e-30f;
  v[6] = has_p ? m.mpx / rp : m.mwx / rw;
  v[7] = has_p ? m.mpy / rp : m.mwy / rw;
}

template <class T>
__global__ void fields_kernel(const T* __restrict__ src, const Layout L, const StepConsts k,
                              uint32_t which, float* __restrict__ out) {
  const int64_t n = (int64_t)L.nx * L.ny;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % L.nx), j = (int)(t / L.nx);
    float fw[kQ], fp[kQ], g[kQ];
    pull_node<T, true>(src, L, i, j, fw, fp, g, k.inv_nx);
    const Moments m = moments_of(fw, fp, g);
    float thp = m.th;
    if (k.two_sets) {
      pull_thermal<T>(src, L, i, j, 3 * kQ, g, k.inv_nx);
      thp = sum9(g);
    }
    float v[kFields];
    node_fields(k, m, thp, i, v);
    int slot = 0;
#pragma unroll
    for (int b = 0; b < kFields; ++b)
      if (which & (1u << b)) out[(int64_t)(slot++) * n + t] = v[b];
  }
}

// ---- deterministic FP64 block reduction -------------------------------------------------------
template <int N>
__device__ __forceinline__ void block_reduce_store(double (&acc)[N], double* out) {
  __shared__ double s[32][N];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < N; ++c)
    for (int off = 16; off > 0; off >>= 1) acc[c] += __shfl_down_sync(0xffffffffu, acc[c], off);
  if (lane == 0)
#pragma unroll
    for (int c = 0; c < N; ++c) s[warp][c] = acc[c];
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
#pragma unroll
    for (int c = 0; c < N; ++c) {
      double v = lane < nw ? s[lane][c] : 0.0;
      for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
      if (lane == 0) out[c] = v;
    }
  }
}

// Sums `count` partial rows of kRedWidth doubles in a fixed order into red[0..kRedWidth).
__global__ void final_reduce_kernel(const double* __restrict__ partials, int count,
                                    double* __restrict__ red) {
  double acc[kRedWidth];
#pragma unroll
  for (int c = 0; c < kRedWidth; ++c) acc[c] = 0.0;
  for (int r = threadIdx.x; r < count; r += blockDim.x)
#pragma unroll
    for (int c = 0; c < kRedWidth; ++c) acc[c] += partials[(size_t)r * kRedWidth + c];
  block_reduce_store<kRedWidth>(acc, red);
}

// Wall sums of rows blockIdx.x kWallRows, + gridDim.x kWallRows, ... into out + blockIdx.x stride.
// Latency-bound (4 nodes per row): with one block of 256 threads and four pulls per thread a
// 1024-row cavity took 60 us; eight blocks take 13 us and their final sum 8 us.
template <class T>
__global__ void __launch_bounds__(kWallThreads)
    nusselt_kernel(const T* __restrict__ src, const Layout L, const StepConsts k,
                   double* __restrict__ out) {
  double acc[kRedWidth];
#pragma unroll
  for (int c = 0; c < kRedWidth; ++c) acc[c] = 0.0;
  double wall[2] = {0.0, 0.0};
  wall_gradients<T>(src, L, k, (int)blockIdx.x * kWallRows, (int)gridDim.x * kWallRows, wall);
  acc[0] = wall[0];
  acc[1] = wall[1];
  block_reduce_store<kRedWidth>(acc, out + (size_t)blockIdx.x * kRedWidth);
}

// Adds nine stored populations of a node to an FP64 sum. GB300 does 2 FP64 operations per clock
// and SM against 128 in FP32, and nine conversions with nine additions per node and component
// were what the mass reduction waited for; so the nine are first summed in FP32 with the exact
// errors of the additions kept beside the sum, those errors likewise with theirs, and the three
// parts go to the FP64 sum: s + es + fs is the sum of the nine to 2^-60 of their largest, where nine
// FP64 additions round nine times by 2^-53 of the total. A node whose parts overflow or are not
// finite is added in FP64. 1024 x 1024: 78 us in FP64, 30 us with the errors summed in plain FP32 (which
// loses bits that FP64 holds), 34 us now.
__device__ __forceinline__ void add_nine(const float (&v)[kQ], double& acc) {
  float e[8], f[7];
  const float a = two_sum(v[0], v[1], e[0]), b = two_sum(v[2], v[3], e[1]);
  const float c = two_sum(v[4], v[5], e[2]), d = two_sum(v[6], v[7], e[3]);
  const float ab = two_sum(a, b, e[4]), cd = two_sum(c, d, e[5]);
  const float abcd = two_sum(ab, cd, e[6]);
  const float s = two_sum(abcd, v[8], e[7]);
  const float e01 = two_sum(e[0], e[1], f[0]), e23 = two_sum(e[2], e[3], f[1]);
  const float e45 = two_sum(e[4], e[5], f[2]), e67 = two_sum(e[6], e[7], f[3]);
  const float e03 = two_sum(e01, e23, f[4]), e47 = two_sum(e45, e67, f[5]);
  const float es = two_sum(e03, e47, f[6]);
  const float fs = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + f[6]);
  if (fabsf(s) + fabsf(es) + fabsf(fs) <= FLT_MAX) {
    acc += (double)s;
    acc += (double)es + (double)fs;
  } else {
    for (int q = 0; q < kQ; ++q) acc += (double)v[q];
  }
}

template <class T>
__global__ void mass_kernel(const T* __restrict__ src, const Layout L,
                            double* __restrict__ partials) {
  double acc[kRedWidth];
#pragma unroll
  for (int c = 0; c < kRedWidth; ++c) acc[c] = 0.0;
  const int64_t n = (int64_t)L.nx * L.ny;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % L.nx), j = (int)(t / L.nx);
    const size_t o = (size_t)j * L.pitch + i;
    float fw[kQ], fp[kQ];
#pragma unroll
    for (int q = 0; q < kQ; ++q) {
      fw[q] = Elem<T>::ldg(src + (size_t)q * L.plane + o);
      fp[q] = Elem<T>::ldg(src + (size_t)(kQ + q) * L.plane + o);
    }
    add_nine(fw, acc[0]);
    add_nine(fp, acc[1]);
  }
  block_reduce_store<kRedWidth>(acc, partials + (size_t)blockIdx.x * kRedWidth);
}

template <class T>
__global__ void residual_kernel(const T* __restrict__ src, const Layout L, const StepConsts k,
                                float* __restrict__ snap, int sums,
                                double* __restrict__ partials) {
  double acc[kRedWidth];
#pragma unroll
  for (int c = 0; c < kRedWidth; ++c) acc[c] = 0.0;
  const int64_t n = (int64_t)L.nx * L.ny;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % L.nx), j = (int)(t / L.nx);
    float fw[kQ], fp[kQ], g[kQ];
    pull_node<T, true>(src, L, i, j, fw, fp, g, k.inv_nx);
    const Moments m = moments_of(fw, fp, g);
    float thp = m.th;
    if (k.two_sets) {
      pull_thermal<T>(src, L, i, j, 3 * kQ, g, k.inv_nx);
      thp = sum9(g);
    }
    float v[kFields];
    node_fields(k, m, thp, i, v);
    if (sums) {
      const double now[4] = {v[0], v[1], v[2], v[3]};
      double d[4];
#pragma unroll
      for (int f = 0; f < 4; ++f) d[f] = now[f] - (double)snap[f * n + t];
      acc[0] += d[0] * d[0] + d[1] * d[1];
      acc[1] += now[0] * now[0] + now[1] * now[1];
      acc[2] += d[2] * d[2];
      acc[3] += now[2] * now[2];
      acc[4] += d[3] * d[3];
      acc[5] += now[3] * now[3];
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) snap[f * n + t] = v[f];
  }
  if (sums) block_reduce_store<kRedWidth>(acc, partials + (size_t)blockIdx.x * kRedWidth);
}

// One row of one plane per block: no division per element, and rows whose packed start is 16-byte
// aligned (nx a multiple of 4) move four elements per thread. Bound by memory (read and write
// once). 1024 x 1024 FP32, 226 MB: 88 us with a flat index and 64-bit divisions, now 38 us.
template <class T, int V>
__global__ void state_copy_kernel(const void* __restrict__ src_v, void* __restrict__ dst_v,
                                  const Layout L, int to_packed) {
  const int64_t n = (int64_t)L.nx * L.ny;
  const int64_t rows = (int64_t)L.np * L.ny;
  const int per_row = blockDim.x, sub = threadIdx.y;  // blockDim.y rows side by side
  for (int64_t r = blockIdx.x * (int64_t)blockDim.y + sub; r < rows;
       r += (int64_t)gridDim.x * blockDim.y) {
    const int p = (int)(r / L.ny), j = (int)(r % L.ny);
    const size_t stored = (size_t)p * L.plane + (size_t)j * L.pitch;
    const size_t packed = (size_t)p * n + (size_t)j * L.nx;
    for (int i = threadIdx.x * V; i < L.nx; i += per_row * V) {
      if constexpr (V == 1) {
        if (to_packed)
          static_cast<float*>(dst_v)[packed + i] =
              Elem<T>::get(static_cast<const T*>(src_v)[stored + i]);
        else
          static_cast<T*>(dst_v)[stored + i] =
              Elem<T>::put(static_cast<const float*>(src_v)[packed + i]);
      } else {
        struct alignas(4 * sizeof(T)) Quad { T v[4]; };
        if (to_packed) {
          const Quad q = *reinterpret_cast<const Quad*>(static_cast<const T*>(src_v) + stored + i);
          *reinterpret_cast<float4*>(static_cast<float*>(dst_v) + packed + i) =
              make_float4(Elem<T>::get(q.v[0]), Elem<T>::get(q.v[1]), Elem<T>::get(q.v[2]),
                          Elem<T>::get(q.v[3]));
        } else {
          const float4 f = *reinterpret_cast<const float4*>(
              static_cast<const float*>(src_v) + packed + i);
          Quad q;
          q.v[0] = Elem<T>::put(f.x);
          q.v[1] = Elem<T>::put(f.y);
          q.v[2] = Elem<T>::put(f.z);
          q.v[3] = Elem<T>::put(f.w);
          *reinterpret_cast<Quad*>(static_cast<T*>(dst_v) + stored + i) = q;
        }
      }
    }
  }
}

__global__ void epoch_advance_kernel(uint32_t* epoch) {
  if (threadIdx.x == 0 && blockIdx.x == 0) *epoch += 1u;
}

// ---- launchers ------------------------------------------------------------------------------
namespace {
int grid_for(int64_t n, int block, int cap) {
  int64_t g = (n + block - 1) / block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}
}  // namespace

// Calls f.template operator()<T>() with T the element type of the storage.
template <class F>
cudaError_t by_storage(int storage, F&& f) {
  switch (storage) {
    case MCLBM_STORE_F32:
      return f((float*)nullptr);
    case MCLBM_STORE_F16:
      return f((__half*)nullptr);
    case MCLBM_STORE_BF16:
      return f((__nv_bfloat16*)nullptr);
    default:
      return cudaErrorInvalidValue;
  }
}

StepConfig choose_step_config(int nx, int ny, int np) {
  StepConfig c;
  // default: TMA-staged tiles for lattices with a few tiles per SM, the plain tile kernel below.
  // MCLBM_STEP_VARIANT = tile | tma overrides (diagnostics and comparisons).
  c.variant = (nx >= 64 && ny >= 32) ? 2 : 0;
  const char* v = std::getenv("MCLBM_STEP_VARIANT");
  if (v && std::strcmp(v, "tile") == 0) c.variant = 0;
  if (v && (std::strcmp(v, "tma") == 0 || std::strcmp(v, "two") == 0)) c.variant = 2;
  c.grid = 0;
  c.sr = true;
  c.two = false;
  c.grid2 = 0;
  c.cl_ctas = c.cl_run = c.cl_threads = 0;
  c.re_ctas = c.re_gx = c.re_gy = c.re_threads = 0;
  // MCLBM_STEP_VEC = 1 | 2 forces the nodes per thread (comparisons; default by lattice size)
  const char* vv = std::getenv("MCLBM_STEP_VEC");
  c.vec = (vv && (vv[0] == '1' || vv[0] == '2') && vv[1] == 0) ? vv[0] - '0' : 0;
  // MCLBM_STEP_TILE_H = 8 | 7 forces the TMA kernel's tile height with one node per thread
  // (comparisons; default: 7 where 32 x 8 tiles would leave some SMs with a second tile and
  // 32 x 7 tiles fit two per SM)
  const char* th = std::getenv("MCLBM_STEP_TILE_H");
  c.th = th && std::strcmp(th, "8") == 0 ? 8 : (th && std::strcmp(th, "7") == 0 ? 7 : 0);
  if (np != kPlanes) {  // two thermal sets: the plain tile kernel, one node per thread
    c.variant = 0;
    c.vec = 1;
  }
  return c;
}

cudaError_t prepare_step(StepConfig* c, const Layout& L) {
  if (c->variant != 2) return cudaSuccess;
  switch (L.storage) {
    case MCLBM_STORE_F32:
      return prepare_tma_f32(c, L);
    case MCLBM_STORE_F16:
      return prepare_tma_f16(c, L);
    case MCLBM_STORE_BF16:
      return prepare_tma_bf16(c, L);
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_step(const StepArgs& a, const StepConfig& c, const CUtensorMap* map,
                        cudaStream_t st) {
  switch (a.L.storage) {
    case MCLBM_STORE_F32:
      return launch_step_f32(a, c, map, st);
    case MCLBM_STORE_F16:
      return launch_step_f16(a, c, map, st);
    case MCLBM_STORE_BF16:
      return launch_step_bf16(a, c, map, st);
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t prepare_cluster(StepConfig* c, const Layout& L, bool all, bool two, cudaStream_t st) {
  switch (L.storage) {
    case MCLBM_STORE_F32:
      return prepare_cluster_f32(c, L, all, two, st);
    case MCLBM_STORE_F16:
      return prepare_cluster_f16(c, L, all, two, st);
    case MCLBM_STORE_BF16:
      return prepare_cluster_bf16(c, L, all, two, st);
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_cluster(const StepArgs& a, const StepConfig& c, int n, uint32_t steps0,
                           uint32_t* epoch, cudaStream_t st) {
  switch (a.L.storage) {
    case MCLBM_STORE_F32:
      return launch_cluster_f32(a, c, n, steps0, epoch, st);
    case MCLBM_STORE_F16:
      return launch_cluster_f16(a, c, n, steps0, epoch, st);
    case MCLBM_STORE_BF16:
      return launch_cluster_bf16(a, c, n, steps0, epoch, st);
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t prepare_resident(StepConfig* c, const Layout& L, bool all, bool two) {
  switch (L.storage) {
    case MCLBM_STORE_F32:
      return prepare_resident_f32(c, L, all, two);
    case MCLBM_STORE_F16:
      return prepare_resident_f16(c, L, all, two);
    case MCLBM_STORE_BF16:
      return prepare_resident_bf16(c, L, all, two);
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_resident(const StepArgs& a, const StepConfig& c, int n, void* scratch,
                            uint32_t* epoch, cudaStream_t st) {
  switch (a.L.storage) {
    case MCLBM_STORE_F32:
      return launch_resident_f32(a, c, n, scratch, epoch, st);
    case MCLBM_STORE_F16:
      return launch_resident_f16(a, c, n, scratch, epoch, st);
    case MCLBM_STORE_BF16:
      return launch_resident_bf16(a, c, n, scratch, epoch, st);
    default:
      return cudaErrorInvalidValue;
  }
}

int step_tile_width(const StepConfig&) { return 32; }

// maps[0]: window loads (box = window); maps[1]: output tile stores (box = tile).
cudaError_t make_state_tensor_map(CUtensorMap* maps, void* state0, const Layout& L, int tile_w,
                                  int tile_h) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                     cudaEnableDefault, &q);
    if (e != cudaSuccess) return e;
    if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  CUtensorMapDataType dt;
  switch (L.storage) {
    case MCLBM_STORE_F32:
      dt = CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
      break;
    case MCLBM_STORE_F16:
      dt = CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
      break;
    case MCLBM_STORE_BF16:
      dt = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
      break;
    default:
      return cudaErrorInvalidValue;
  }
  if ((tile_w != 32 && tile_w != 64) || (tile_h != 8 && tile_h != 7)) return cudaErrorInvalidValue;
  const int wx = tile_w + 2 * (16 / L.elem);  // 16 bytes of halo columns on each side
  const cuuint64_t dims[3] = {(cuuint64_t)L.nx, (cuuint64_t)L.ny, (cuuint64_t)(2 * kPlanes)};
  const cuuint64_t strides[2] = {(cuuint64_t)L.pitch * L.elem, (cuuint64_t)L.plane * L.elem};
  const cuuint32_t box[3] = {(cuuint32_t)wx, (cuuint32_t)(tile_h + 4), (cuuint32_t)kPlanes};
  const cuuint32_t tile[3] = {(cuuint32_t)tile_w, (cuuint32_t)tile_h, (cuuint32_t)kPlanes};
  const cuuint32_t elem[3] = {1, 1, 1};
  CUresult r = encode(&maps[0], dt, 3, state0, dims, strides, box, elem,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  r = encode(&maps[1], dt, 3, state0, dims, strides, tile, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t make_two_step_tensor_map(CUtensorMap* map, void* state0, const Layout& L) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                     cudaEnableDefault, &q);
    if (e != cudaSuccess) return e;
    if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  if (L.storage != MCLBM_STORE_F32 || L.np != kPlanes) return cudaErrorInvalidValue;
  const cuuint64_t dims[3] = {(cuuint64_t)L.nx, (cuuint64_t)L.ny, (cuuint64_t)(2 * kPlanes)};
  const cuuint64_t strides[2] = {(cuuint64_t)L.pitch * 4, (cuuint64_t)L.plane * 4};
  const cuuint32_t box[3] = {32 + 2 * 4, 16 + 2 * 4, (cuuint32_t)kPlanes};
  const cuuint32_t elem[3] = {1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, state0, dims, strides, box,
                            elem, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t launch_epoch_advance(uint32_t* epoch, cudaStream_t st) {
  epoch_advance_kernel<<<1, 32, 0, st>>>(epoch);
  return cudaGetLastError();
}

cudaError_t launch_stream_only(const void* src, void* dst, const Layout& L, const StepConsts& k,
                               cudaStream_t st) {
  const int64_t n = (int64_t)L.nx * L.ny;
  return by_storage(L.storage, [&](auto* tag) {
    using T = std::remove_pointer_t<decltype(tag)>;
    stream_only_kernel<T><<<grid_for(n, 256, 4096), 256, 0, st>>>(
        static_cast<const T*>(src), static_cast<T*>(dst), L, k.inv_nx);
    return cudaGetLastError();
  });
}

cudaError_t launch_init(void* dst, const Layout& L, const StepConsts& k, const float* warm,
                        int warm_rho, cudaStream_t st) {
  const int64_t n = (int64_t)L.nx * L.ny;
  return by_storage(L.storage, [&](auto* tag) {
    using T = std::remove_pointer_t<decltype(tag)>;
    init_kernel<T><<<grid_for(n, 256, 4096), 256, 0, st>>>(static_cast<T*>(dst), L, k, warm,
                                                            warm_rho);
    return cudaGetLastError();
  });
}

cudaError_t launch_fields(const void* src, const Layout& L, const StepConsts& k, uint32_t which,
                          float* out, cudaStream_t st) {
  const int64_t n = (int64_t)L.nx * L.ny;
  return by_storage(L.storage, [&](auto* tag) {
    using T = std::remove_pointer_t<decltype(tag)>;
    fields_kernel<T><<<grid_for(n, 256, 4096), 256, 0, st>>>(static_cast<const T*>(src), L, k,
                                                              which, out);
    return cudaGetLastError();
  });
}

// Up to 2 kWallRows rows one block walks them and writes the result itself (a second launch
// costs as much as a second trip); beyond, kWallRows rows per block and a final sum.
cudaError_t launch_nusselt(const void* src, const Layout& L, const StepConsts& k,
                           double* partials, double* red, cudaStream_t st) {
  const int g = L.ny <= 2 * kWallRows ? 1 : grid_for(L.ny, kWallRows, kMaxRedBlocks);
  return by_storage(L.storage, [&](auto* tag) {
    using T = std::remove_pointer_t<decltype(tag)>;
    nusselt_kernel<T><<<g, kWallThreads, 0, st>>>(static_cast<const T*>(src), L, k,
                                                  g == 1 ? red : partials);
    if (g > 1) final_reduce_kernel<<<1, 256, 0, st>>>(partials, g, red);
    return cudaGetLastError();
  });
}

cudaError_t launch_mass(const void* src, const Layout& L, double* partials, double* red,
                        cudaStream_t st) {
  const int64_t n = (int64_t)L.nx * L.ny;
  const int g = grid_for(n, 256, kMaxRedBlocks);
  return by_storage(L.storage, [&](auto* tag) {
    using T = std::remove_pointer_t<decltype(tag)>;
    mass_kernel<T><<<g, 256, 0, st>>>(static_cast<const T*>(src), L, partials);
    final_reduce_kernel<<<1, 256, 0, st>>>(partials, g, red);
    return cudaGetLastError();
  });
}

cudaError_t launch_residual(const void* src, const Layout& L, const StepConsts& k, float* snap,
                            bool sums, double* partials, double* red, cudaStream_t st) {
  const int64_t n = (int64_t)L.nx * L.ny;
  // the sums want few blocks (their FP64 block reductions), a snapshot alone as many as it can
  // get (1024 x 1024: 47 us with 304 blocks, 33 us with 4096)
  const int g = grid_for(n, 256, sums ? kMaxRedBlocks : 4096);
  return by_storage(L.storage, [&](auto* tag) {
    using T = std::remove_pointer_t<decltype(tag)>;
    residual_kernel<T><<<g, 256, 0, st>>>(static_cast<const T*>(src), L, k, snap, sums ? 1 : 0,
                                           partials);
    if (sums) final_reduce_kernel<<<1, 256, 0, st>>>(partials, g, red);
    return cudaGetLastError();
  });
}

// Four elements per thread where both sides of a row allow it: stored rows start on 128 bytes,
// packed ones on nx floats, and the caller's array may start anywhere.
cudaError_t launch_state_copy(const void* src, void* dst, const Layout& L, bool to_packed,
                              cudaStream_t st) {
  const void* packed = to_packed ? dst : src;
  const bool quads = L.nx % 4 == 0 && (reinterpret_cast<uintptr_t>(packed) & 15u) == 0;
  const int per_row = quads ? L.nx / 4 : L.nx;
  const int bx = per_row <= 32 ? 32 : (per_row <= 64 ? 64 : (per_row <= 128 ? 128 : 256));
  const dim3 block(bx, 256 / bx);
  const int64_t rows = (int64_t)L.np * L.ny;
  const int grid = grid_for(rows, (int)block.y, 1 << 16);
  return by_storage(L.storage, [&](auto* tag) {
    using T = std::remove_pointer_t<decltype(tag)>;
    if (quads)
      state_copy_kernel<T, 4><<<grid, block, 0, st>>>(src, dst, L, to_packed ? 1 : 0);
    else
      state_copy_kernel<T, 1><<<grid, block, 0, st>>>(src, dst, L, to_packed ? 1 : 0);
    return cudaGetLastError();
  });
}

}  // namespace mcl
