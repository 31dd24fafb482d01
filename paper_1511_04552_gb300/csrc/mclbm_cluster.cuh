// Cluster-resident form of the fused MCLBM step for small lattices: one thread-block cluster holds
// the whole cavity in shared memory and advances it many steps in one launch.
//
// A launch per step leaves a small cavity waiting: 32 x 32 took 4.4 us per step, of which the
// arithmetic of its 1024 nodes is a few hundred nanoseconds on the chip; the rest is the launch, the
// loads from L2, the stores and their completion. Here each CTA of a cluster (up to 16) owns a
// run of nodes, keeps two buffers of its populations in shared memory, pulls its halo from the
// other CTAs' buffers (distributed shared memory) and meets the others at one cluster
// barrier per step; global memory is touched at the start and the end of a launch. Per node the
// pulls, moments and collision are those of the other step kernels, and the stochastic-rounding
// streams follow the same blocks of 2^k steps, so the states are the same bits.
//
// Nodes are numbered along the lattice's shorter side (u = j nx + i, or i ny + j where nx > ny) and
// cut into equal runs, so that the CTAs are balanced whatever the sizes, and a run's ring - the nodes
// within one line of it, whose theta' and rho'^p its gradients need - is as short as it can be. One
// thread per node (the step is latency-bound here) and, as far as threads go, one per ring node.
#pragma once

#include "mclbm_pair.cuh"

namespace mcl {
namespace cluster {

constexpr int kThreadsMax = 640;  // 96 registers each
constexpr int kThreadsFew = 512;  // 128: no spills, 32 x 32 1.23 us per step against 1.51 with 80
constexpr int kCtasMax = 16;      // beyond 8: opt-in (non-portable) cluster size

// A stored population as FP32 from a shared-memory address of the cluster (this CTA's or another's).
template <class T>
__device__ __forceinline__ float load_at(uint32_t addr);
template <>
__device__ __forceinline__ float load_at<float>(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ uint16_t load16_at(uint32_t addr) {
  uint16_t v;
  asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(v) : "r"(addr));
  return v;
}
template <>
__device__ __forceinline__ float load_at<__half>(uint32_t addr) {
  return __half2float(__ushort_as_half(load16_at(addr)));
}
template <>
__device__ __forceinline__ float load_at<__nv_bfloat16>(uint32_t addr) {
  return __uint_as_float((uint32_t)load16_at(addr) << 16);
}

// Where a node's nine pulled directions come from, walls included (the rules of pull_node): a thread
// keeps its node for the whole launch, so that the wall tests are made once and a pull is an add and
// a load. f: address in the f^w planes (f^p: nine planes on), g: in the g planes (g^p: nine planes
// on), both for buffer 0; bit q of neg: the isothermal wall's negative sign.
struct Sources {
  uint32_t f[kQ], g[kQ], neg;
};
// How nodes are numbered and cut into runs.
struct Runs {
  int nx, ny, line, run;  // line: nodes per line of the numbering; run: nodes per CTA
  bool by_column;         // u = i ny + j
  __device__ __forceinline__ Runs(const Layout& L, int r)
      : nx(L.nx), ny(L.ny), line(min(L.nx, L.ny)), run(r), by_column(L.nx > L.ny) {}
  __device__ __forceinline__ int number(int i, int j) const {
    return by_column ? i * ny + j : j * nx + i;
  }
  __device__ __forceinline__ void node(int u, int& i, int& j) const {
    const int a = u / line, b = u - a * line;
    i = by_column ? a : b;
    j = by_column ? b : a;
  }
};
template <class T>
__device__ __forceinline__ Sources sources_of(const T* buf, const Runs& R, int i, int j) {
  const uint32_t base = tma::smem_u32(buf);
  auto at = [&](int p, int ci, int cj) {  // plane p, node (ci, cj) in its owner's buffer 0
    const int u = R.number(ci, cj), r = u / R.run;
    uint32_t owner;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(owner) : "r"(base), "r"(r));
    return owner + (uint32_t)(p * R.run + u - r * R.run) * (uint32_t)sizeof(T);
  };
  Sources s;
  s.neg = 0;
#pragma unroll
  for (int q = 0; q < kQ; ++q) {
    const int si = i - ex(q), sj = j - ey(q);
    const bool inx = (unsigned)si < (unsigned)R.nx, iny = (unsigned)sj < (unsigned)R.ny;
    if (inx && iny) {
      s.f[q] = at(q, si, sj);
      s.g[q] = s.f[q] + (uint32_t)(2 * kQ * R.run) * (uint32_t)sizeof(T);
    } else {
      s.f[q] = at(opp(q), i, j);
      s.g[q] = inx ? at(2 * kQ + mir(q), si, j) : at(2 * kQ + opp(q), i, j);
      if (!inx) s.neg |= 1u << q;
    }
  }
  return s;
}
// from: byte offset of the buffer read; set: byte offset of nine planes
template <class T, bool FULL, bool TWO>
__device__ __forceinline__ void pull_from(const Sources& s, uint32_t from, uint32_t set, float* fw,
                                          float* fp, float* g, float* gp) {
#pragma unroll
  for (int q = 0; q < kQ; ++q) {
    if (FULL) fw[q] = load_at<T>(s.f[q] + from);
    fp[q] = load_at<T>(s.f[q] + from + set);
    const uint32_t sign = (s.neg << (31 - q)) & 0x80000000u;
    g[q] = __uint_as_float(__float_as_uint(load_at<T>(s.g[q] + from)) ^ sign);
    if (TWO) gp[q] = __uint_as_float(__float_as_uint(load_at<T>(s.g[q] + from + set)) ^ sign);
  }
}

template <class T, bool SR>
struct SharedSink {
  T* base;
  int plane;
  uint32_t seed;
  __device__ __forceinline__ void operator()(int p, float v) const {
    pair::St<T>::template st1<SR>(base + p * plane, v, SR ? pair::rbits(seed, p) : 0u);
  }
};

__device__ __forceinline__ void barrier() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// n steps from a.src (level read) to a.dst (level written; may be the same). steps0: steps done
// before this launch.
template <class T, bool SR, bool ALLF, bool TWO, int MAXT>
__global__ void __launch_bounds__(MAXT, 1)
    step_cluster_kernel(const StepArgs a, int run, int n, uint32_t steps0, uint32_t* epoch) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int NP = TWO ? kPlanes2 : kPlanes;
  const Layout& L = a.L;
  const StepConsts& k = a.k;
  const Runs R(L, run);
  uint32_t rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int u0 = (int)rank * run, u1 = min(L.nx * L.ny, u0 + run), own = u1 - u0;
  T* buf = reinterpret_cast<T*>(smem_raw);
  // moments of the nodes u0 - line .. u1 + line
  float* mth = reinterpret_cast<float*>(smem_raw + ((size_t)2 * NP * run * sizeof(T) + 15) / 16 * 16);
  float* mrp = mth + run + 2 * R.line;
  Sources* table = reinterpret_cast<Sources*>(mrp + run + 2 * R.line);
  const int t = threadIdx.x;

  // ring nodes: up to a line before the run, then up to a line after it. As far as the threads
  // beyond the run's nodes go they have one each; the rest are done by the run's threads before
  // their own, with their sources in shared memory.
  const int ring_lo = min(R.line, u0), ring = ring_lo + min(R.line, L.nx * L.ny - u1);
  auto ring_node = [&](int q) { return q < ring_lo ? u0 - ring_lo + q : u1 + q - ring_lo; };
  const bool mine = t < own;
  const int spare = (int)blockDim.x - own;
  const bool ringer = !mine && t - own < ring;
  const int shared_ring = ring > spare ? ring - spare : 0;  // ring nodes q = spare + ...
  const int u = mine ? u0 + t : (ringer ? ring_node(t - own) : u0);
  int i, j;
  R.node(u, i, j);
  const size_t o = (size_t)j * L.pitch + i;
  // The run's populations between global memory and a buffer, in row-major order over the lines it
  // touches (a run by columns is a few columns wide: its rows are short but contiguous).
  const int c0 = R.by_column ? u0 / R.line : 0, r0 = R.by_column ? 0 : u0 / R.line;
  const int lines = (u1 - 1) / R.line - u0 / R.line + 1;
  const int width = R.by_column ? lines : L.nx, box = lines * R.line;
  auto each_node = [&](auto&& f) {
    for (int e = t; e < box; e += blockDim.x) {
      const int rr = e / width, ci = c0 + e - rr * width, cj = r0 + rr;
      const int v = R.number(ci, cj) - u0;
      if (v >= 0 && v < own) f(v, (size_t)cj * L.pitch + ci);
    }
  };
  each_node([&](int v, size_t at) {
    const T* p0 = static_cast<const T*>(a.src) + at;
    T x[NP];  // all loads before the first store
#pragma unroll
    for (int p = 0; p < NP; ++p) x[p] = p0[(size_t)p * L.plane];
#pragma unroll
    for (int p = 0; p < NP; ++p) buf[p * run + v] = x[p];
  });
  const Sources src = sources_of(buf, R, i, j);
  for (int q = t; q < shared_ring; q += blockDim.x) {
    int ri, rj;
    R.node(ring_node(spare + q), ri, rj);
    table[q] = sources_of(buf, R, ri, rj);
  }
  const uint32_t set = (uint32_t)(kQ * run) * (uint32_t)sizeof(T);

  const uint32_t ep0 = *(volatile const uint32_t*)epoch;
  uint32_t ep = ep0;
  int block_left = 0;
  uint32_t seed = 0, sh = 0;
  barrier();
  for (int s = 0; s < n; ++s) {
    if (SR) {
      // the blocks of 2^k steps a launch sequence of captured graphs would run, each with the next
      // epoch and the seeds 0, 1, ...; an odd last step has a seed of its own
      if (block_left == 0 && n - s >= 2) {
        block_left = 1 << min(31 - __clz(n - s), kGraphLogMax);
        seed = 0;
      }
      if (block_left > 0) {
        sh = mix32(seed++ ^ mix32(ep + 0x632BE5ABu));
        if (--block_left == 0) ++ep;
      } else {
        sh = mix32((0x80000000u ^ (steps0 + (uint32_t)s)) ^ mix32(ep + 0x632BE5ABu));
      }
    }
    const int to = ((s + 1) & 1) * NP * run;
    const uint32_t from = (uint32_t)((s & 1) * NP * run) * (uint32_t)sizeof(T);
    float fw[kQ], fp[kQ], g[kQ], gp[TWO ? kQ : 1];
    // theta' and rho'^p of node v to the moments
    auto moments = [&](int v) {
      const int m = v - u0 + R.line;
      if constexpr (TWO)
        mth[m] = pair::mixture_s<T>(k, pair::sum9(fw), pair::sum9(fp), pair::sum9(g),
                                    pair::sum9(gp));
      else
        mth[m] = pair::sum9(g);
      mrp[m] = pair::sum9(fp);
    };
    for (int q = t; q < shared_ring; q += blockDim.x) {
      const Sources rs = table[q];
      pull_from<T, TWO, TWO>(rs, from, set, fw, fp, g, gp);
      moments(ring_node(spare + q));
    }
    if (mine || ringer) {
      pull_from<T, true, TWO>(src, from, set, fw, fp, g, gp);
      moments(u);
    }
    __syncthreads();
    if (mine) {
      const int m = t + R.line;
      const int dx = R.by_column ? R.line : 1, dy = R.by_column ? 1 : R.line;
      const float th = mth[m], rp = mrp[m];
      // wall ghosts as in the tile kernels: -theta' at the isothermal walls, the node's own value at
      // the others
      const float thN = j + 1 < L.ny ? mth[m + dy] : th, thS = j > 0 ? mth[m - dy] : th;
      const float rpN = j + 1 < L.ny ? mrp[m + dy] : rp, rpS = j > 0 ? mrp[m - dy] : rp;
      const float thE = i + 1 < L.nx ? mth[m + dx] : -th, thW = i > 0 ? mth[m - dx] : -th;
      const float rpE = i + 1 < L.nx ? mrp[m + dx] : rp, rpW = i > 0 ? mrp[m - dx] : rp;
      SharedSink<T, SR> out{buf + to + t, run, SR ? mix32((uint32_t)o ^ sh) : 0u};
      pair::collide<1, ALLF, T, TWO>(k, L, out, i, j, fw, fp, g, gp, thE, thW, thN, thS, rpE, rpW,
                                     rpN, rpS);
    }
    barrier();  // the step's populations are written, and nobody reads the other buffer any more
  }
  each_node([&](int v, size_t at) {
    T* p0 = static_cast<T*>(a.dst) + at;
    const T* res = buf + (n & 1) * NP * run + v;
#pragma unroll
    for (int p = 0; p < NP; ++p) p0[(size_t)p * L.plane] = res[p * run];
  });
  // one epoch per block of 2^k steps: the same count whether or not the rounding uses it
  if (rank == 0 && t == 0)
    *epoch = ep0 + (uint32_t)((n >> kGraphLogMax) + __popc((n & ((1 << kGraphLogMax) - 1)) >> 1));
}

// ---- host side ---------------------------------------------------------------------------------
// Two buffers of the run's populations, its and its ring's moments, the sources of the ring nodes
// that no thread has for itself.
inline size_t smem_bytes(const Layout& L, int run, int threads) {
  const size_t state = ((size_t)2 * L.np * run * L.elem + 15) / 16 * 16;
  const int line = std::min(L.nx, L.ny);
  // the last run may be shorter, with more threads to spare: never more of the table
  const int shared_ring = std::max(0, run + 2 * line - threads);
  return state + (size_t)2 * (run + 2 * line) * sizeof(float) +
         (size_t)shared_ring * sizeof(Sources);
}

template <class T, int MAXT>
const void* kernel_of(bool sr, bool all, bool two) {
  if (two)
    return sr ? (const void*)step_cluster_kernel<T, sizeof(T) == 2, false, true, MAXT>
              : (const void*)step_cluster_kernel<T, false, false, true, MAXT>;
  if (sr)
    return all ? (const void*)step_cluster_kernel<T, sizeof(T) == 2, true, false, MAXT>
               : (const void*)step_cluster_kernel<T, sizeof(T) == 2, false, false, MAXT>;
  return all ? (const void*)step_cluster_kernel<T, false, true, false, MAXT>
             : (const void*)step_cluster_kernel<T, false, false, false, MAXT>;
}
template <class T>
const void* kernel_of(int threads, bool sr, bool all, bool two) {
  return threads <= kThreadsFew ? kernel_of<T, kThreadsFew>(sr, all, two)
                                : kernel_of<T, kThreadsMax>(sr, all, two);
}

inline void fill_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr, const StepConfig& c,
                        const Layout& L, cudaStream_t st) {
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = c.cl_ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg->gridDim = dim3(c.cl_ctas);
  cfg->blockDim = dim3(c.cl_threads);
  cfg->dynamicSmemBytes = smem_bytes(L, c.cl_run, c.cl_threads);
  cfg->stream = st;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
}

// Sets c.cl_* where the kernel is to run (CTAs 0: it is not): a run's nodes fit the threads, its
// populations shared memory, and the SMs that the stream may use can hold the cluster.
template <class T>
cudaError_t prepare(StepConfig* c, const Layout& L, bool all, bool two, cudaStream_t st) {
  c->cl_ctas = 0;
  const int64_t nodes = (int64_t)L.nx * L.ny;
  const int line = std::min(L.nx, L.ny);
  if (nodes > (int64_t)kCtasMax * kThreadsMax) return cudaSuccess;
  for (int most = kCtasMax; most >= 8; most /= 2) {
    // no run shorter than two lines: its ring would reach beyond the neighbouring runs
    const int run = std::max((int)((nodes + most - 1) / most), std::min((int)nodes, 2 * line));
    const int ctas = (int)((nodes + run - 1) / run);
    if (run > kThreadsMax) return cudaSuccess;
    StepConfig t = *c;
    t.cl_run = run;
    t.cl_ctas = ctas;
    t.cl_threads = std::min(kThreadsMax, (run + 2 * line + 31) / 32 * 32);
    if (smem_bytes(L, run, t.cl_threads) > 227 * 1024) return cudaSuccess;
    const void* fn = kernel_of<T>(t.cl_threads, c->sr && sizeof(T) == 2, all, two);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
    if (ctas > 8 &&
        (e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) !=
            cudaSuccess)
      return e;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = {};
    fill_config(&cfg, attr, t, L, st);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) == cudaSuccess && n >= 1) {
      *c = t;
      return cudaSuccess;
    }
    cudaGetLastError();
  }
  return cudaSuccess;
}

template <class T>
cudaError_t launch(const StepArgs& a, const StepConfig& c, int n, uint32_t steps0, uint32_t* epoch,
                   cudaStream_t st) {
  cudaLaunchAttribute attr[1];
  cudaLaunchConfig_t cfg = {};
  fill_config(&cfg, attr, c, a.L, st);
  int run = c.cl_run;
  StepArgs args = a;
  void* params[] = {&args, &run, &n, &steps0, &epoch};
  const bool all = a.k.mask == MCLBM_F_ALL && !a.k.two_sets;
  return cudaLaunchKernelExC(&cfg, kernel_of<T>(c.cl_threads, c.sr && sizeof(T) == 2, all, a.k.two_sets), params);
}

}  // namespace cluster
}  // namespace mcl
