// Convolutions of the warm-start network as implicit GEMMs on the 5th-generation tensor cores:
// forward and stride-1 input gradient (conv_kernel), stride-2 input gradient (dx_stride2_kernel)
// and weight gradient (wgrad_kernel), and the packing of the weights into their operand layouts.
//
// Activations and pre-activation gradients are BF16 in channel groups, x[c / 8][pixel][c % 8]: a
// pixel's eight channels are one 16-byte row of a tcgen05 core matrix (8 rows x 16 bytes, no
// swizzle), so that a shift by one pixel is a shift of the matrix start address by 16 bytes and
// the taps of a convolution read one staged patch at different start addresses.
//
// Before, every convolution materialised its im2col rows (9 x the input, 2.2 GB written and read
// twice per training step of batch 16 at 256 x 256); these kernels expand the taps in shared
// memory only. Every product is accumulated over K in the order, and in the groups of 16, of the
// im2col GEMM (k = c 9 + tap forward, k = o 9 + tap in the stride-1 input gradient, k = o in the
// stride-2 one): a BF16 rounding that flips in one layer would travel through all that follow.
// Only the weight gradient, whose sums feed no further layer, adds its pixels in another order.
//
// Loss and gradient of the 256 x 256 network at batch 16: 6.33 ms with im2col rows, their GEMMs and
// col2im, 1.58 ms with these kernels (ten forward convolutions 0.47 ms, ten weight gradients
// 0.41 ms, nine input gradients 0.33 ms; the rest is element-wise). Forward at batch 1: 367 us (the
// launches of 10 GEMMs with a tensor map and an occupancy query each) to 120 us.
//
// Every mbarrier wait is bounded (2 s); a role that gives up sets the abort word, the copies and
// MMAs in flight are drained (bounded), tensor memory is freed and the error bit is set.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "net_internal.h"
#include "net_tc.cuh"

namespace mcl {
namespace net {
namespace {

constexpr int kRows = 128;                   // pixels of a tile: 8 rows of 16
constexpr int kTileH = 8, kTileW = 16;
constexpr int kSliceChunks = 18;             // 16-byte K chunks of a slice: 2 groups x 9
constexpr int kSliceSteps = 9;               // MMAs of K = 16 per slice
constexpr int kABytes = kSliceChunks * kRows * 16;

__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes,
                                          uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1,
                                            int c2, int c3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, int c0, int c1,
                                            int c2, int c3, int c4, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
      : "memory");
}
// 8 consecutive accumulator columns of this thread's lane, not waited for
__device__ __forceinline__ void tmem_ld8_async(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  uint32_t u;
  memcpy(&u, &v, 4);
  return u;
}

// ---- forward and stride-1 input gradient ----------------------------------------------------
// A persistent grid (one CTA per SM) walks (pixel tile, output-channel tile, K split); the K
// slices of 16 channels (144 k) of all its items form one stream through a ring of stages.
//   warps 8-23 (producers, two sets of 256 threads on alternate slices, so that two slices'
//     loads are in flight): thread = (pixel of the tile, channel group); nine 16-byte loads, one
//     per tap, of the group's channels, repacked from tap-major to k = c 9 + tap by byte permutes
//     and stored as nine 16-byte rows of the K-major A slice [chunk][pixel][16 B];
//   warp 24 lane 0: the slice's weights, packed in the operand layout, as one bulk copy;
//   warp 25 lane 0: the MMAs, into one of two accumulators in tensor memory;
//   warps 0-7: the epilogue of a finished tile while the next one's MMAs run; warps w and w + 4
//     share the pixels of tensor-memory lanes 32 w.. and take alternate groups of 8 channels. Per
//     group every operand is loaded before the first store: a load behind a store of the group
//     waits for it, and with 16 channels in turn that chain made the epilogue the bottleneck (3 us
//     per tile and 16 channels).
// What bounds it is instruction issue where a tile has few slices (d0 of the 256 x 256 network at
// batch 16, 3 slices: 107 us, 66 % of the issue slots; its 906 MB of im2col rows took 0.6 ms to
// write and 175 us to multiply), and beside it the shared-memory pipe: a slice is written (36 KiB),
// read by the tensor core (36 KiB) and its loads (36 KiB, two thirds of them L1 hits) go through
// that pipe too.
constexpr int kProducerSets = 2;
constexpr int kEpilogueThreads = 256;
constexpr int kLoadWarp = 8 + 8 * kProducerSets, kMmaWarp = kLoadWarp + 1;
constexpr int kConvThreads = 32 * (kMmaWarp + 1);

struct Item {
  int z, n, b, y0, x0;  // K split, channel tile, image, tile origin
};
__device__ __forceinline__ Item item_at(const ConvArgs& a, int i) {
  Item it;
  const int r = a.by_tiles.div(i);
  int t = i - r * (int)a.by_tiles.d;
  it.z = a.by_n.div(r);
  it.n = r - it.z * a.n_tiles;
  it.b = a.by_image.div(t);
  t -= it.b * (int)a.by_image.d;
  const int ty = a.by_row.div(t);
  it.y0 = ty * kTileH;
  it.x0 = (t - ty * a.tiles_x) * kTileW;
  return it;
}
// The MMA steps and the slices of an item's K split.
struct Range {
  int step0, step1, s0, s1;
};
__device__ __forceinline__ Range range_of(const ConvArgs& a, int i) {
  Range r;
  const int z = a.split_steps < a.steps ? a.by_n.div(a.by_tiles.div(i)) : 0;
  r.step0 = z * a.split_steps;
  r.step1 = min(r.step0 + a.split_steps, a.steps);
  r.s0 = r.step0 / kSliceSteps;
  r.s1 = r.step1 > r.step0 ? (r.step1 + kSliceSteps - 1) / kSliceSteps : r.s0;
  return r;
}

// Word m of the 36 words of a pixel's 72 values in k order (k = c 9 + tap) from the nine taps'
// words (two channels each).
template <int M>
__device__ __forceinline__ uint32_t k_word(const uint4 (&t)[9]) {
  constexpr int f0 = 2 * M, f1 = 2 * M + 1;
  constexpr int c0 = f0 / 9, t0 = f0 % 9, c1 = f1 / 9, t1 = f1 % 9;
  constexpr uint32_t sel = ((c0 & 1) ? 0x32u : 0x10u) | ((c1 & 1) ? 0x7600u : 0x5400u);
  const uint4 &a = t[t0], &b = t[t1];
  const uint32_t wa = (c0 >> 1) == 0 ? a.x : ((c0 >> 1) == 1 ? a.y : ((c0 >> 1) == 2 ? a.z : a.w));
  const uint32_t wb = (c1 >> 1) == 0 ? b.x : ((c1 >> 1) == 1 ? b.y : ((c1 >> 1) == 2 ? b.z : b.w));
  return __byte_perm(wa, wb, sel);
}
template <int J>
__device__ __forceinline__ void store_chunks(uint8_t* dst, const uint4 (&t)[9]) {
  if constexpr (J < 9) {
    *reinterpret_cast<uint4*>(dst + J * kRows * 16) = make_uint4(
        k_word<4 * J>(t), k_word<4 * J + 1>(t), k_word<4 * J + 2>(t), k_word<4 * J + 3>(t));
    store_chunks<J + 1>(dst, t);
  }
}

template <int MODE>
__global__ void __launch_bounds__(kConvThreads, 1) conv_kernel(const ConvArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ int s_abort;
  __shared__ uint64_t full_a[kConvMaxStages], full_b[kConvMaxStages], empty[kConvMaxStages];
  __shared__ uint64_t acc_full[2], acc_empty[2];
  __shared__ uint32_t tslot;
  const int b_bytes = kSliceChunks * a.nt * 16;
  const int stride = kABytes + b_bytes;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  volatile int* abort = &s_abort;

  if (warp == kMmaWarp) tmem_alloc(smem_addr(&tslot), a.tmem_cols);
  if (tid == 0) {
    for (int s = 0; s < a.stages; ++s) {
      bar_init(smem_addr(&full_a[s]), 256);
      bar_init(smem_addr(&full_b[s]), 1);
      bar_init(smem_addr(&empty[s]), 1);
    }
    for (int k = 0; k < 2; ++k) {
      bar_init(smem_addr(&acc_full[k]), 1);
      bar_init(smem_addr(&acc_empty[k]), kEpilogueThreads);
    }
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tslot;
  pdl_wait();

  // a role's place in the ring: stage, and how often the ring has come round (its parity)
  struct Ring {
    int st = 0;
    uint32_t round = 0;
    __device__ __forceinline__ void step(int by, int stages) {
      st += by;
      if (st >= stages) {
        st -= stages;
        ++round;
      }
    }
  };
  int produced = 0, mma_done = 0;  // slices whose copies / MMAs were issued
  if (warp >= 8 && warp < kLoadWarp) {
    const int pt = tid - kEpilogueThreads;
    const int set = pt >> 8, h = (pt >> 7) & 1, r = pt & 127;
    const int dy = r >> 4, dx = r & 15;
    // cursor: item, slice; and for the item `opened`, the pixel's first tap and its valid taps
    int i = blockIdx.x, s = 0, s_end = 0, opened = -1;
    const uint4* base = nullptr;
    uint32_t mask = 0;
    // moves on by n slices of the stream; false at its end
    auto advance = [&](int n) -> bool {
      s += n;
      while (s >= s_end) {
        const int over = s - s_end;
        i += gridDim.x;
        if (i >= a.items) return false;
        const Range r = range_of(a, i);
        s = r.s0 + over;
        s_end = r.s1;
      }
      return true;
    };
    uint4 t[9];
    auto load = [&]() {
      if (i != opened) {
        opened = i;
        const Item it = item_at(a, i);
        const int y = it.y0 + dy, x = it.x0 + dx;
        const int yi = a.stride * y - 1, xi = a.stride * x - 1;
        const bool in = y < a.Ho && x < a.Wo;
        uint32_t my = 0, mx = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if (in && (unsigned)(yi + k) < (unsigned)a.H) my |= 7u << (3 * k);
          if ((unsigned)(xi + k) < (unsigned)a.W) mx |= 0x49u << k;
        }
        mask = my & mx;
        base = reinterpret_cast<const uint4*>(a.src) + (int64_t)it.b * a.src_image +
               (int64_t)yi * a.W + xi;
      }
      const int g = 2 * s + h;
      if (g >= a.groups) return;  // the same for the whole warp
      const uint4* p0 = base + (int64_t)g * a.src_group;
      const uint4 *p1 = p0 + a.W, *p2 = p1 + a.W;
      if (__all_sync(0xffffffffu, mask == 0x1FFu)) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          t[k] = __ldg(p0 + k);
          t[3 + k] = __ldg(p1 + k);
          t[6 + k] = __ldg(p2 + k);
        }
      } else {
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          t[k] = make_uint4(0u, 0u, 0u, 0u);
          if ((mask >> k) & 1u) t[k] = __ldg((k < 3 ? p0 : (k < 6 ? p1 : p2)) + k % 3);
        }
      }
    };
    // this set takes the slices set, set + kProducerSets, ... of the stream
    Ring ring;
    ring.step(set, a.stages);
    bool live = i < a.items;
    if (live) {
      const Range r = range_of(a, i);
      s = r.s0;
      s_end = r.s1;
      live = advance(set);
    }
    if (live) load();
    while (live) {
      // the warp stays or goes as one: load() votes over all its lanes
      const bool ok = ring.round == 0 ||
                      role_wait(smem_addr(&empty[ring.st]), (ring.round - 1) & 1u, abort);
      if (!__all_sync(0xffffffffu, ok)) {
        *abort = 1;
        break;
      }
      uint8_t* dst = smem + ring.st * stride + (h * 9 * kRows + r) * 16;
      if (2 * s + h < a.groups)
        store_chunks<0>(dst, t);
      else  // an odd group count: the last MMA reads one chunk beyond
        *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bar_arrive(smem_addr(&full_a[ring.st]));
      ring.step(kProducerSets, a.stages);
      live = advance(kProducerSets);
      if (live) load();
    }
  } else if (warp == kLoadWarp) {
    // weights of every slice of the stream
    const bool leader = elect_one();
    Ring ring;
    for (int i = blockIdx.x; i < a.items && !*abort; i += gridDim.x) {
      const Range r = range_of(a, i);
      const int n = item_at(a, i).n;
      for (int s = r.s0; s < r.s1; ++s) {
        if (ring.round > 0 &&
            !role_wait(smem_addr(&empty[ring.st]), (ring.round - 1) & 1u, abort)) {
          *abort = 1;
          break;
        }
        if (leader) {
          const uint32_t fb = smem_addr(&full_b[ring.st]);
          bar_expect_tx(fb, (uint32_t)b_bytes);
          bulk_load(smem_addr(smem + ring.st * stride + kABytes),
                    a.w + (int64_t)(n * a.slices + s) * (b_bytes / 2), (uint32_t)b_bytes, fb);
        }
        ++produced;
        ring.step(1, a.stages);
      }
    }
  } else if (warp == kMmaWarp) {
    const bool leader = elect_one();
    Ring ring;
    int k = 0;
    const uint32_t idesc = instr_desc(kRows, a.nt, false, false);
    // K = 16 is two chunks: core matrices along K one chunk apart, along M or N 128 B apart
    const uint32_t hi = desc_hi(128);
    const uint32_t a_lo0 = desc_lo(smem_addr(smem), kRows * 16);
    const uint32_t b_lo0 = desc_lo(smem_addr(smem + kABytes), (uint32_t)a.nt * 16);
    for (int i = blockIdx.x; i < a.items && !*abort; i += gridDim.x, ++k) {
      const Range r = range_of(a, i);
      const int acc = k & 1;
      const uint32_t d = tmem + (uint32_t)(acc * a.nt);
      if (k >= 2 && !role_wait(smem_addr(&acc_empty[acc]), (uint32_t)(((k >> 1) - 1) & 1), abort)) {
        *abort = 1;
        break;
      }
      tc_fence_after();
      uint32_t accumulate = 0;
      for (int s = r.s0; s < r.s1; ++s) {
        const uint32_t parity = ring.round & 1u;
        if (!role_wait(smem_addr(&full_a[ring.st]), parity, abort) ||
            !role_wait(smem_addr(&full_b[ring.st]), parity, abort)) {
          *abort = 1;
          break;
        }
        tc_fence_after();
        const uint32_t at = (uint32_t)(ring.st * stride) >> 4;
        const int j0 = max(r.step0 - s * kSliceSteps, 0);
        const int j1 = min(r.step1 - s * kSliceSteps, kSliceSteps);
        const uint32_t a_lo = a_lo0 + at, b_lo = b_lo0 + at, b_step = 2 * (uint32_t)a.nt;
#pragma unroll
        for (int j = 0; j < kSliceSteps; ++j) {
          const bool mine = j >= j0 && j < j1;
          mma_bf16_words(leader && mine, d, a_lo + (uint32_t)(j * 2 * kRows), hi,
                         b_lo + (uint32_t)j * b_step, hi, idesc, accumulate);
          accumulate = mine ? 1u : accumulate;
        }
        if (leader) mma_commit(smem_addr(&empty[ring.st]));
        ++mma_done;
        ring.step(1, a.stages);
      }
      if (*abort) break;
      if (leader) mma_commit(smem_addr(&acc_full[acc]));
    }
  } else if (warp < 8) {
    const int r = (warp & 3) * 32 + lane;
    const int dy = r >> 4, dx = r & 15;
    const int hw = a.Ho * a.Wo;
    const int64_t P = (int64_t)a.batch * hw;
    int k = 0;
    for (int i = blockIdx.x; i < a.items; i += gridDim.x, ++k) {
      const Item it = item_at(a, i);
      const int acc = k & 1;
      const bool ok = role_wait(smem_addr(&acc_full[acc]), (uint32_t)((k >> 1) & 1), abort);
      if (!__all_sync(0xffffffffu, ok)) {  // tcgen05.ld is warp-collective
        *abort = 1;
        break;
      }
      tc_fence_after();
      const int y = it.y0 + dy, x = it.x0 + dx;
      const bool in = y < a.Ho && x < a.Wo;
      const int64_t p = (int64_t)it.b * hw + y * a.Wo + x;
      const uint32_t lane_addr =
          tmem + (uint32_t)(acc * a.nt) + ((uint32_t)((warp & 3) * 32) << 16);
      const bool none = MODE == kConvPartial && it.z * a.split_steps >= a.steps;  // beyond K
#pragma unroll 1
      for (int c0 = (warp >> 2) * 8; c0 < a.nt; c0 += 16) {
        __syncwarp();  // lanes beyond the edge have skipped the stores of the group before
        uint32_t u[8];
        tmem_ld8_async(lane_addr + (uint32_t)c0, u);
        const int o0 = it.n * a.nt + c0;
        if constexpr (MODE == kConvForward) {
          const ConvEpilogue& e = a.ep;
          const float* f = e.film ? e.film + (int64_t)it.b * e.film_stride + e.film_off : nullptr;
          float bias[8], g[8], beta[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const bool has = o0 + j < a.N;
            bias[j] = has ? __ldg(e.bias + o0 + j) : 0.f;
            g[j] = has && f ? __ldg(f + o0 + j) : 0.f;
            beta[j] = has && f ? __ldg(f + a.N + o0 + j) : 0.f;
          }
          tmem_ld_wait();
          if (in) {
            float out[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float pre = __uint_as_float(u[j]) + bias[j];
              float zz = pre;
              if (f) zz = (1.f + g[j]) * pre + beta[j];
              u[j] = __float_as_uint(pre);
              out[j] = e.act ? zz / (1.f + expf(-zz)) : zz;
            }
            if (e.pre) {
              float* dst = e.pre + (int64_t)o0 * P + p;
#pragma unroll
              for (int j = 0; j < 8; ++j, dst += P)
                if (o0 + j < a.N) *dst = __uint_as_float(u[j]);
            }
            if (e.y && o0 < a.N)
              store_group(e, o0 / 8, it.b, y, x, a.Ho, a.Wo,
                          make_uint4(pack2(out[0], out[1]), pack2(out[2], out[3]),
                                     pack2(out[4], out[5]), pack2(out[6], out[7])));
          }
        } else if constexpr (MODE == kConvPartial) {
          tmem_ld_wait();
          if (in) {  // one branch: with a test of `in` per store a small forward pass took 3 % longer
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (o0 + j < a.N)
                a.part[((int64_t)it.z * a.N + o0 + j) * P + p] = none ? 0.f : __uint_as_float(u[j]);
          }
        } else {
          // channels [0, cu) to their source (2 x 2 sums, in row order, when it was upsampled),
          // the others to the skip source: cu is a multiple of 8, so a group goes to one of them.
          // Rows are 16 lanes apart, pixels of a row one lane apart.
          const RouteArgs& q = a.route;
          const bool first = o0 < q.cu;
          const bool up = first && q.up;
          tmem_ld_wait();
          float v[8], old[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float own = __uint_as_float(u[j]);
            v[j] = own;
            if (up) {
              v[j] += __shfl_down_sync(0xffffffffu, own, 1);
              v[j] += __shfl_down_sync(0xffffffffu, own, 16);
              v[j] += __shfl_down_sync(0xffffffffu, own, 17);
            }
          }
          if (in && o0 < a.N && !(up && (lane >= 16 || (lane & 1)))) {
            const int64_t step = up ? P / 4 : P;
            float* dst =
                first ? q.dsrc1 + (int64_t)o0 * step : q.dsrc2 + (int64_t)(o0 - q.cu) * step;
            dst += up ? (int64_t)it.b * (hw / 4) + (y / 2) * (a.Wo / 2) + x / 2 : p;
            if (first ? q.acc1 : q.acc2) {
#pragma unroll
              for (int j = 0; j < 8; ++j) old[j] = dst[j * step];
#pragma unroll
              for (int j = 0; j < 8; ++j) v[j] = old[j] + v[j];
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) dst[j * step] = v[j];
          }
        }
      }
      tc_fence_before();
      bar_arrive(smem_addr(&acc_empty[acc]));
    }
  }
  __syncthreads();
  if (*abort) {
    if (warp == kLoadWarp)
      for (int gs = max(0, produced - a.stages); gs < produced; ++gs)
        bar_wait(smem_addr(&full_b[gs % a.stages]), (uint32_t)((gs / a.stages) & 1));
    if (warp == kMmaWarp && mma_done > 0)
      bar_wait(smem_addr(&empty[(mma_done - 1) % a.stages]),
               (uint32_t)(((mma_done - 1) / a.stages) & 1));
    if (tid == 0) atomicOr(a.err, 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) tmem_dealloc(tmem, a.tmem_cols);
}

// ---- stride-2 input gradient ----------------------------------------------------------------
// dX at the four input pixels (2Y + a, 2X + b) takes the taps whose output pixel is (Y, X) or its
// right or lower neighbour. A tile of 16 rows x 8 columns of (Y, X) stages the output gradient's
// 17 x 9 patch by TMA (zero beyond the edge); each tap is one product over the output channels
// with the patch shifted by 0 or 1 pixel, accumulated in tensor-memory columns of its own (16
// input channels x 9 taps), and the epilogue adds a pixel's taps in the order of the taps. Six
// warps, two CTAs per SM (256 tensor-memory columns each); bound by the FP32 gradient it writes
// (and reads where it accumulates). The four layers at batch 16 and 256 x 256: 102 us, where the
// GEMM into the column gradient and col2im's gather took 1.2 ms.
constexpr int kS2Threads = 192, kS2Ch = 16;
constexpr int kS2Px = 9, kS2Rows = 17;

__global__ void __launch_bounds__(kS2Threads) dx_stride2_kernel(
    const __grid_constant__ CUtensorMap map, const DxStride2Args a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ int s_abort;
  __shared__ uint64_t full[kDxStages], empty[kDxStages], acc_full, acc_empty;
  __shared__ uint32_t tslot;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const uint32_t row = (uint32_t)a.kg * kS2Px * 16;  // bytes of a patch row
  volatile int* abort = &s_abort;
  if (warp == 5) tmem_alloc(smem_addr(&tslot), 256);
  if (tid == 0) {
    for (int s = 0; s < kDxStages; ++s) {
      bar_init(smem_addr(&full[s]), 1);
      bar_init(smem_addr(&empty[s]), 1);
    }
    bar_init(smem_addr(&acc_full), 1);
    bar_init(smem_addr(&acc_empty), 128);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tslot;
  pdl_wait();
  const int per = a.tiles_x * a.tiles_y;
  const int tiles = per * a.batch;
  const int items = tiles * a.chunks;
  int produced = 0, mma_done = 0;
  if (warp == 4) {
    const bool leader = elect_one();
    for (int i = blockIdx.x; i < items && !*abort; i += gridDim.x) {
      const int ch = i / tiles, t = i - ch * tiles;
      const int b = t / per, u = t - b * per;
      const int y0 = (u / a.tiles_x) * 16, x0 = (u % a.tiles_x) * 8;
      for (int kc = 0; kc < a.kchunks; ++kc, ++produced) {
        const int st = produced % kDxStages;
        if (produced >= kDxStages &&
            !role_wait(smem_addr(&empty[st]), (uint32_t)((produced / kDxStages - 1) & 1), abort)) {
          *abort = 1;
          break;
        }
        if (leader) {
          const uint32_t fb = smem_addr(&full[st]), sa = smem_addr(smem + st * a.stage_bytes);
          bar_expect_tx(fb, (uint32_t)(kS2Rows * row + a.w_bytes));
          tma_load_4d(sa, &map, x0 * 8, kc * a.kg, y0, b, fb);
          bulk_load(sa + a.a_bytes, a.w + (int64_t)(ch * a.kchunks + kc) * (a.w_bytes / 2),
                    (uint32_t)a.w_bytes, fb);
        }
      }
    }
  } else if (warp == 5) {
    const bool leader = elect_one();
    int k = 0;
    const uint32_t idesc = instr_desc(kRows, kS2Ch, false, false);
    const uint32_t hi_a = desc_hi(row), hi_b = desc_hi(128);
    for (int i = blockIdx.x; i < items && !*abort; i += gridDim.x, ++k) {
      if (k >= 1 && !role_wait(smem_addr(&acc_empty), (uint32_t)((k - 1) & 1), abort)) {
        *abort = 1;
        break;
      }
      tc_fence_after();
      for (int kc = 0; kc < a.kchunks; ++kc, ++mma_done) {
        const int st = mma_done % kDxStages;
        if (!role_wait(smem_addr(&full[st]), (uint32_t)((mma_done / kDxStages) & 1), abort)) {
          *abort = 1;
          break;
        }
        tc_fence_after();
        const uint32_t sa = smem_addr(smem + st * a.stage_bytes), sb = sa + a.a_bytes;
        const uint32_t a_lo0 = desc_lo(sa, kS2Px * 16);
        uint32_t b_lo = desc_lo(sb, kS2Ch * 16);
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          // ky, kx = 0 read the lower / right neighbour's gradient
          uint32_t a_lo = a_lo0 + (tap / 3 == 0 ? row >> 4 : 0u) + (tap % 3 == 0 ? 1u : 0u);
          for (int kk = 0; kk < a.kg / 2; ++kk) {
            mma_bf16_words(leader, tmem + (uint32_t)(tap * kS2Ch), a_lo, hi_a, b_lo, hi_b, idesc,
                           (kc > 0 || kk > 0) ? 1u : 0u);
            a_lo += 2 * kS2Px;
            b_lo += 2 * kS2Ch;
          }
        }
        if (leader) mma_commit(smem_addr(&empty[st]));
      }
      if (*abort) break;
      if (leader) mma_commit(smem_addr(&acc_full));
    }
  } else if (warp < 4) {
    const int r = warp * 32 + lane;
    const int H = 2 * a.Ho, W = 2 * a.Wo;
    int k = 0;
    for (int i = blockIdx.x; i < items; i += gridDim.x, ++k) {
      const bool ok = role_wait(smem_addr(&acc_full), (uint32_t)(k & 1), abort);
      if (!__all_sync(0xffffffffu, ok)) {
        *abort = 1;
        break;
      }
      tc_fence_after();
      const int ch = i / tiles, t = i - ch * tiles;
      const int b = t / per, u = t - b * per;
      const int Y = (u / a.tiles_x) * 16 + (r >> 3), X = (u % a.tiles_x) * 8 + (r & 7);
      const bool in = Y < a.Ho && X < a.Wo;
      const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
      for (int half = 0; half < kS2Ch / 8; ++half) {
        __syncwarp();  // as in conv_kernel
        uint32_t d[9][8];
#pragma unroll
        for (int tap = 0; tap < 9; ++tap)
          tmem_ld8_async(lane_addr + (uint32_t)(tap * kS2Ch + half * 8), d[tap]);
        tmem_ld_wait();
        auto D = [&](int tap, int j) { return __uint_as_float(d[tap][j]); };
        const int c = ch * kS2Ch + half * 8;
        if (in && c < a.C) {  // C is a multiple of 8
          const int64_t plane = (int64_t)a.batch * H * W;
          float* dst = a.dsrc + (int64_t)c * plane + ((int64_t)b * H + 2 * Y) * W + 2 * X;
          float2 top[8], bot[8];
          if (a.accumulate) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              top[j] = *reinterpret_cast<const float2*>(dst + j * plane);
              bot[j] = *reinterpret_cast<const float2*>(dst + j * plane + W);
            }
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float ee = D(4, j), eo = D(3, j) + D(5, j), oe = D(1, j) + D(7, j);
            const float oo = ((D(0, j) + D(2, j)) + D(6, j)) + D(8, j);
            top[j] = a.accumulate ? make_float2(top[j].x + ee, top[j].y + eo) : make_float2(ee, eo);
            bot[j] = a.accumulate ? make_float2(bot[j].x + oe, bot[j].y + oo) : make_float2(oe, oo);
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            *reinterpret_cast<float2*>(dst + j * plane) = top[j];
            *reinterpret_cast<float2*>(dst + j * plane + W) = bot[j];
          }
        }
      }
      tc_fence_before();
      bar_arrive(smem_addr(&acc_empty));
    }
  }
  __syncthreads();
  if (*abort) {
    if (warp == 4)
      for (int gs = max(0, produced - kDxStages); gs < produced; ++gs)
        bar_wait(smem_addr(&full[gs % kDxStages]), (uint32_t)((gs / kDxStages) & 1));
    if (warp == 5 && mma_done > 0)
      bar_wait(smem_addr(&empty[(mma_done - 1) % kDxStages]),
               (uint32_t)(((mma_done - 1) / kDxStages) & 1));
    if (tid == 0) atomicOr(a.err, 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 5) tmem_dealloc(tmem, 256);
}

// ---- weight gradient ------------------------------------------------------------------------
// dW[o][c][tap] = sum over pixels of dpre[o][pixel] x[c][pixel + tap]: M = o, K = pixels, N =
// (tap, channel). A stage holds one tile of 8 rows x 16 pixels of dpre and the patch of x its taps
// read, both by TMA in the MN-major core-matrix layout (8 pixels x 16 bytes; a K step is one row of
// 16 pixels), rows of a patch ordered [y][group][x]: the groups of one row and those of the next follow each other at one
// stride, so that one MMA takes the three vertical taps of all groups (N = 24 groups' columns) and
// a horizontal tap is a start address 16 bytes on. The stride-2 layers read x as four parity
// patches (TMA with a pixel stride of 2). One CTA per (split of the pixel tiles, channel chunk,
// horizontal taps) with its accumulators in tensor memory throughout; partial sums per split are
// added in order by finish_kernel. Rows of M beyond the layer's channels and columns beyond its
// groups read other staged data and are not stored. The ten layers at batch 16 and 256 x 256:
// 0.41 ms; the GEMMs over the im2col rows took 0.8 ms.
constexpr int kWgThreads = 192;

__global__ void __launch_bounds__(kWgThreads) wgrad_kernel(
    const __grid_constant__ WgradMaps maps, const WgradArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ int s_abort;
  __shared__ uint64_t full[kWgMaxStages], empty[kWgMaxStages], acc_full;
  __shared__ uint32_t tslot;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  volatile int* abort = &s_abort;
  if (warp == 5) tmem_alloc(smem_addr(&tslot), a.tmem_cols);
  if (tid == 0) {
    for (int s = 0; s < a.stages; ++s) {
      bar_init(smem_addr(&full[s]), 1);
      bar_init(smem_addr(&empty[s]), 1);
    }
    bar_init(smem_addr(&acc_full), 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tslot;
  pdl_wait();
  // item: o chunk, channel chunk, part of the entries (horizontal taps), split of the tiles
  int u0 = blockIdx.x;
  const int oc = u0 % a.ochunks;
  u0 /= a.ochunks;
  const int ch = u0 % a.chunks;
  u0 /= a.chunks;
  const int e0 = u0 % a.parts * a.entries;
  const int z = u0 / a.parts;
  const int per = a.tiles_x * a.tiles_y;
  const int t0 = z * a.split_tiles, t1 = min(t0 + a.split_tiles, per * a.batch);
  int produced = 0, mma_done = 0;
  if (warp == 4) {
    const bool leader = elect_one();
    int b = t0 / per, u = t0 - b * per;
    int ty = u / a.tiles_x, tx = u - ty * a.tiles_x;
    int st = 0;
    uint32_t round = 0;
    for (int t = t0; t < t1 && !*abort; ++t, ++produced) {
      if (round > 0 && !role_wait(smem_addr(&empty[st]), (round - 1) & 1u, abort)) {
        *abort = 1;
        break;
      }
      if (leader) {
        const int y0 = ty * kTileH, x0 = tx * kTileW;
        const uint32_t fb = smem_addr(&full[st]), sa = smem_addr(smem + st * a.stage_bytes);
        bar_expect_tx(fb, (uint32_t)a.tx_bytes);
        tma_load_4d(sa, &maps.a, x0 * 8, oc * a.go, y0, b, fb);
        const int xb = a.src_images ? b : 0;
        if (!a.s2) {
          tma_load_4d(sa + a.a_bytes, &maps.b[0], x0 * 8 - 8, ch * a.gc, y0 - 1, xb, fb);
        } else {
          for (int p = 0; p < 4; ++p)
            tma_load_5d(sa + a.a_bytes + p * a.patch_bytes, &maps.b[p], 0, x0 - (p & 1),
                        ch * a.gc, y0 - (p >> 1), xb, fb);
        }
      }
      if (++st == a.stages) {
        st = 0;
        ++round;
      }
      if (++tx == a.tiles_x) {
        tx = 0;
        if (++ty == a.tiles_y) {
          ty = 0;
          ++b;
        }
      }
    }
  } else if (warp == 5) {
    const bool leader = elect_one();
    uint32_t d_col[6], e_off[6], e_desc[6], accumulate = 0;
#pragma unroll
    for (int e = 0; e < 6; ++e) {
      const WgradEntry& w = a.e[min(e0 + e, 5)];
      d_col[e] = tmem + (uint32_t)(w.col - a.e[e0].col);
      e_off[e] = (uint32_t)w.off >> 4;
      e_desc[e] = instr_desc(kRows, w.n, true, true);
    }
    const uint32_t a_row = (uint32_t)a.go * kTileW, b_row = (uint32_t)a.b_row >> 4;  // 16 bytes
    const uint32_t hi_a = desc_hi(kTileW * 16), hi_b = desc_hi((uint32_t)a.b_group);
    int st = 0;
    uint32_t round = 0;
    for (int t = t0; t < t1 && !*abort; ++t, ++mma_done) {
      if (!role_wait(smem_addr(&full[st]), round & 1u, abort)) {
        *abort = 1;
        break;
      }
      tc_fence_after();
      const uint32_t sa = smem_addr(smem + st * a.stage_bytes);
      const uint32_t a_lo = desc_lo(sa, 128), b_lo = desc_lo(sa + a.a_bytes, 128);
#pragma unroll
      for (int e = 0; e < 6; ++e) {
        if (e >= a.entries) break;
#pragma unroll
        for (uint32_t ks = 0; ks < kTileH; ++ks)
          mma_bf16_words(leader, d_col[e], a_lo + ks * a_row, hi_a, b_lo + e_off[e] + ks * b_row,
                         hi_b, e_desc[e], ks > 0 ? 1u : accumulate);
      }
      accumulate = 1;
      if (leader) mma_commit(smem_addr(&empty[st]));
      if (++st == a.stages) {
        st = 0;
        ++round;
      }
    }
    if (!*abort && leader) mma_commit(smem_addr(&acc_full));
  } else if (warp < 4) {
    const bool ok = role_wait(smem_addr(&acc_full), 0u, abort);
    if (!__all_sync(0xffffffffu, ok)) {
      *abort = 1;
    } else if (warp * 32 < a.mrows) {
      tc_fence_after();
      const int o = warp * 32 + lane;
      const int col0 = a.e[e0].col;
      const int cols = a.e[e0 + a.entries - 1].col + a.e[e0 + a.entries - 1].n - col0;
      float* part = a.part + (((int64_t)z * a.chunks + ch) * a.ochunks + oc) * a.cols * a.mrows +
                    (int64_t)col0 * a.mrows + o;
      for (int c0 = 0; c0 < cols; c0 += 16) {
        float v[16];
        if (t1 > t0) {
          tmem_ld16(tmem + (uint32_t)c0 + ((uint32_t)(warp * 32) << 16), v);
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = 0.f;
        }
        if (o < a.mrows)
#pragma unroll
          for (int j = 0; j < 16; ++j) part[(int64_t)(c0 + j) * a.mrows] = v[j];
      }
      tc_fence_before();
    }
  }
  __syncthreads();
  if (*abort) {
    if (warp == 4)
      for (int k = max(0, produced - a.stages); k < produced; ++k)
        bar_wait(smem_addr(&full[k % a.stages]), (uint32_t)((k / a.stages) & 1));
    if (warp == 5 && mma_done > 0)
      bar_wait(smem_addr(&empty[(mma_done - 1) % a.stages]),
               (uint32_t)(((mma_done - 1) / a.stages) & 1));
    if (tid == 0) atomicOr(a.err, 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 5) tmem_dealloc(tmem, a.tmem_cols);
}

// ---- weights into the operand layouts -------------------------------------------------------
// BF16, round to nearest, zero beyond the layer's channels: one launch for all layers.
__global__ void pack_weights_kernel(const PackArgs a) {
  pdl_wait();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < a.total;
       t += (int64_t)gridDim.x * blockDim.x) {
    int s = 0;
    while (s + 1 < a.count && t >= a.seg[s + 1].start) ++s;
    const PackSeg& g = a.seg[s];
    const int64_t i = t - g.start;
    const int e = (int)(i % 8);
    int64_t r = i / 8;
    const float* w = a.params + g.w_off;
    float v = 0.f;
    if (g.kind == kPackStride2) {  // [chunk][kchunk][tap][group][16 c][8 o]
      const int c16 = (int)(r % kS2Ch);
      r /= kS2Ch;
      const int gr = (int)(r % g.kg);
      r /= g.kg;
      const int tap = (int)(r % 9);
      r /= 9;
      const int o = ((int)(r % g.slices) * g.kg + gr) * 8 + e;
      const int c = (int)(r / g.slices) * kS2Ch + c16;
      if (o < g.cout && c < g.cin) v = w[(int64_t)o * 9 * g.cin + c * 9 + tap];
    } else {  // [n tile][slice][18][nt][8]: n the output channel, or the input channel of dX
      const int n = (int)(r % g.nt);
      r /= g.nt;
      const int kc = (int)(r % kSliceChunks);
      r /= kSliceChunks;
      const int k = ((int)(r % g.slices) * kSliceChunks + kc) * 8 + e;
      const int nn = (int)(r / g.slices) * g.nt + n;
      const int q = k / 9, tap = k - 9 * q;
      if (g.kind == kPackForward) {
        if (nn < g.cout && q < g.cin) v = w[(int64_t)nn * 9 * g.cin + k];
      } else {
        if (nn < g.cin && q < g.cout) v = w[(int64_t)q * 9 * g.cin + nn * 9 + 8 - tap];
      }
    }
    g.out[i] = __float2bfloat16_rn(v);
  }
}

// ---- the end of the backward pass: partial sums to gradients --------------------------------
// Blocks [0, w_blocks): every weight, its splits added in order (o fastest: the partial sums are
// read coalesced). The rest: one block per (layer, output channel) adds the pixel chunks of each
// sample in order (FiLM's gradients) and the samples in order (the bias).
__global__ void __launch_bounds__(256) finish_kernel(const FinishArgs a) {
  __shared__ double sh[256];
  pdl_wait();
  if ((int)blockIdx.x < a.w_blocks) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < a.total;
         t += (int64_t)a.w_blocks * blockDim.x) {
      int s = 0;
      while (s + 1 < a.count && t >= a.seg[s + 1].start) ++s;
      const FinishSeg& g = a.seg[s];
      const int64_t i = t - g.start;
      const int o = (int)(i % g.cout);
      const int k = (int)(i / g.cout);
      const int c = k / 9, tap = k - 9 * c;
      const int ky = tap / 3, kx = tap - 3 * ky;
      const int gr = c >> 3, ch = gr / g.gc, gl = gr - ch * g.gc;
      int col;
      if (!g.s2)
        col = g.col[kx] + (ky * g.gc + gl) * 8 + (c & 7);
      else if (ky == 1)
        col = g.col[3 + kx] + gl * 8 + (c & 7);
      else
        col = g.col[kx] + ((ky >> 1) * g.gc + gl) * 8 + (c & 7);
      const int oc = o / kRows, ol = o - oc * kRows;
      const int64_t step = (int64_t)g.chunks * g.ochunks * g.cols * g.mrows;
      const float* p = g.part + ((int64_t)(ch * g.ochunks + oc) * g.cols + col) * g.mrows + ol;
      float sum = 0.f;
      for (int z = 0; z < g.splits; ++z) sum += p[z * step];
      g.grad[(int64_t)o * g.kin + k] = sum;
    }
    return;
  }
  int u = (int)blockIdx.x - a.w_blocks, s = 0;
  while (u >= a.seg[s].cout) u -= a.seg[s++].cout;
  const FinishSeg& g = a.seg[s];
  const int o = u;
  for (int b = threadIdx.x; b < a.batch; b += blockDim.x) {
    double v[3] = {0.0, 0.0, 0.0};
    const double* p = g.sums + ((int64_t)o * a.batch + b) * g.sum_chunks * 3;
    for (int k = 0; k < g.sum_chunks; ++k)
      for (int j = 0; j < 3; ++j) v[j] += p[3 * k + j];
    if (g.film_off >= 0) {
      a.dfilm[(int64_t)b * a.film_stride + g.film_off + o] = (float)v[1];
      a.dfilm[(int64_t)b * a.film_stride + g.film_off + g.cout + o] = (float)v[2];
    }
    sh[b] = v[0];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int b = 0; b < a.batch; ++b) v += sh[b];
    g.dbias[o] = (float)v;
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }();
  return fn;
}

bool encode(CUtensorMap* map, int rank, const void* base, const cuuint64_t* dims,
            const cuuint64_t* strides, const cuuint32_t* box) {
  const cuuint32_t elem[5] = {1, 1, 1, 1, 1};
  return encoder() &&
         encoder()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(base), dims,
                   strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <class K, class... A>
cudaError_t launch_pdl(K kernel, int grid, int block, int smem, cudaStream_t st, const A&... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

constexpr int kSmemMax = 227 * 1024 - 1024;  // what a CTA may take, less the static part

int conv_smem(const ConvArgs& a) { return a.stages * (kABytes + kSliceChunks * a.nt * 16); }

}  // namespace

// x [groups][images][H][W][8] as {W x 8, groups, H, images}: a box is [y][group][x][8].
bool encode_groups(CUtensorMap* map, const __nv_bfloat16* x, int groups, int64_t group_pixels,
                   int images, int H, int W, int box_px, int box_groups, int box_rows) {
  const cuuint64_t dims[4] = {(cuuint64_t)W * 8, (cuuint64_t)groups, (cuuint64_t)H,
                              (cuuint64_t)images};
  const cuuint64_t strides[3] = {(cuuint64_t)group_pixels * 16, (cuuint64_t)W * 16,
                                 (cuuint64_t)H * W * 16};
  const cuuint32_t box[4] = {(cuuint32_t)box_px * 8, (cuuint32_t)box_groups, (cuuint32_t)box_rows,
                             1};
  return encode(map, 4, x, dims, strides, box);
}

// The pixels of one parity (py, px) of x as {8, W / 2, groups, H / 2, images}.
bool encode_parity(CUtensorMap* map, const __nv_bfloat16* x, int py, int px, int groups,
                   int64_t group_pixels, int images, int H, int W, int box_px, int box_groups,
                   int box_rows) {
  const cuuint64_t dims[5] = {8, (cuuint64_t)W / 2, (cuuint64_t)groups, (cuuint64_t)H / 2,
                              (cuuint64_t)images};
  const cuuint64_t strides[4] = {32, (cuuint64_t)group_pixels * 16, (cuuint64_t)W * 32,
                                 (cuuint64_t)H * W * 16};
  const cuuint32_t box[5] = {8, (cuuint32_t)box_px, (cuuint32_t)box_groups, (cuuint32_t)box_rows,
                             1};
  return encode(map, 5, x + ((int64_t)py * W + px) * 8, dims, strides, box);
}

int conv_n_tile(int n) { return n >= kRows ? kRows : (n + 15) & ~15; }
int conv_slices(int groups) { return (groups + 1) / 2; }

void plan_conv(ConvArgs* a, int splits, int split_k) {
  a->nt = conv_n_tile(a->N);
  a->n_tiles = (a->N + a->nt - 1) / a->nt;
  a->slices = conv_slices(a->groups);
  a->steps = (72 * a->groups + 15) / 16;
  a->split_steps = splits > 1 ? split_k / 16 : a->steps;
  a->tiles_x = (a->Wo + kTileW - 1) / kTileW;
  a->tiles_y = (a->Ho + kTileH - 1) / kTileH;
  a->items = a->tiles_x * a->tiles_y * a->batch * a->n_tiles * splits;
  a->by_tiles = FastDiv(a->tiles_x * a->tiles_y * a->batch);
  a->by_image = FastDiv(a->tiles_x * a->tiles_y);
  a->by_row = FastDiv(a->tiles_x);
  a->by_n = FastDiv(a->n_tiles);
  a->tmem_cols = a->nt <= 16 ? 32 : (a->nt <= 32 ? 64 : (a->nt <= 64 ? 128 : 256));
  const int stage = kABytes + kSliceChunks * a->nt * 16;
  a->stages = std::min(kConvMaxStages, kSmemMax / stage);
}

cudaError_t launch_conv(const ConvArgs& a, int mode, int sms, cudaStream_t st) {
  const int grid = std::min(a.items, sms), smem = conv_smem(a);
  switch (mode) {
    case kConvForward:
      return launch_pdl(conv_kernel<kConvForward>, grid, kConvThreads, smem, st, a);
    case kConvPartial:
      return launch_pdl(conv_kernel<kConvPartial>, grid, kConvThreads, smem, st, a);
    default:
      return launch_pdl(conv_kernel<kConvRoute>, grid, kConvThreads, smem, st, a);
  }
}

// Output-channel groups per K chunk, and the chunks of 16 input channels.
int dx_stride2_kg(int cout) { return std::min(16, cout / 8); }
void plan_dx_stride2(DxStride2Args* a, int cout) {
  a->kg = dx_stride2_kg(cout);
  a->kchunks = (cout / 8 + a->kg - 1) / a->kg;
  a->chunks = (a->C + kS2Ch - 1) / kS2Ch;
  a->tiles_x = (a->Wo + 7) / 8;
  a->tiles_y = (a->Ho + 15) / 16;
  a->a_bytes = (kS2Rows * kS2Px * 16 * a->kg + 127) / 128 * 128;
  a->w_bytes = 9 * a->kg * kS2Ch * 16;
  a->stage_bytes = (a->a_bytes + a->w_bytes + 127) / 128 * 128;
}

cudaError_t launch_dx_stride2(const CUtensorMap& map, const DxStride2Args& a, int sms,
                              cudaStream_t st) {
  const int smem = kDxStages * a.stage_bytes;
  const int per_sm = 2 * smem <= kSmemMax ? 2 : 1;
  const int items = a.tiles_x * a.tiles_y * a.batch * a.chunks;
  return launch_pdl(dx_stride2_kernel, std::min(items, per_sm * sms), kS2Threads, smem, st, map, a);
}

namespace {

// The part of a plan that depends on the channel groups per chunk.
void wgrad_chunk(WgradArgs* a, int cin_groups, int chunks) {
  auto r16 = [](int n) { return (n + 15) / 16 * 16; };
  a->chunks = chunks;
  a->gc = (cin_groups + chunks - 1) / chunks;
  const int px = a->s2 ? kTileW + 1 : kTileW + 2, rows = a->s2 ? kTileH + 1 : kTileH + 2;
  const int patches = a->s2 ? 4 : 1;
  a->b_group = px * 16;
  a->b_row = a->gc * a->b_group;
  a->patch_bytes = (rows * a->b_row + 127) / 128 * 128;
  a->tx_bytes = a->a_bytes + patches * rows * a->b_row;
  a->stage_bytes = a->a_bytes + patches * a->patch_bytes;
  if (!a->s2) {
    const int n = r16(24 * a->gc);
    for (int dx = 0; dx < 3; ++dx) a->e[dx] = {dx * 16, n, dx * n};
    a->cols = 3 * n;
  } else {
    // kx = 0 and 2 read the odd columns (x - 1 and x of their patch), kx = 1 the even ones; ky
    // likewise: odd rows hold ky = 0 and, one row on, ky = 2
    const int n2 = r16(16 * a->gc), n1 = r16(8 * a->gc);
    for (int kx = 0; kx < 3; ++kx) {
      const int px = kx != 1, shift = kx == 2 ? 16 : 0;
      a->e[kx] = {(2 + px) * a->patch_bytes + shift, n2, kx * n2};
      a->e[3 + kx] = {px * a->patch_bytes + shift, n1, 3 * n2 + kx * n1};
    }
    a->cols = 3 * (n1 + n2);
  }
}

// Channel groups per chunk at most: the columns of all taps in 512 of tensor memory.
int wgrad_most(int s2) { return s2 ? 4 : 6; }

// Splits of the pixels: each is one FP32 accumulation in the tensor core, whose rounding grows
// with its length, and the sums of the splits are added in FP32.
int wgrad_splits(int cout, int kin) {
  const int tiles = ((cout + 127) / 128) * ((((kin + 7) & ~7) + 127) / 128);
  return std::max(1, std::min(64, 152 / tiles));
}

void wgrad_rows(WgradArgs* a, int cout, int stride) {
  const int og = (cout + 7) / 8;
  a->s2 = stride == 2;
  a->go = std::min(16, og);
  a->ochunks = (og + 15) / 16;
  a->mrows = std::min(kRows, og * 8);
  a->a_bytes = kTileH * a->go * kTileW * 16;
}

}  // namespace

// Splits x channel chunks x parts (the horizontal taps apart, or together) CTAs: the splits are
// fixed by the accuracy, the rest is chosen for the least estimated time. An MMA of N columns
// takes max(45, N / 2) cycles (measured), a tile is also bound by its bytes, and CTAs beyond one
// per SM share it.
void plan_wgrad(WgradArgs* a, int cin_groups, int cout, int kin, int Ho, int Wo, int batch,
                int stride, int sms) {
  wgrad_rows(a, cout, stride);
  a->tiles_x = (Wo + kTileW - 1) / kTileW;
  a->tiles_y = (Ho + kTileH - 1) / kTileH;
  a->batch = batch;
  const int tiles = a->tiles_x * a->tiles_y * batch;
  a->split_tiles = (tiles + wgrad_splits(cout, kin) - 1) / wgrad_splits(cout, kin);
  a->splits = (tiles + a->split_tiles - 1) / a->split_tiles;
  const int taps = a->s2 ? 6 : 3;
  double best = 1e30;
  int best_chunks = 1, best_parts = 1;
  for (int gc = std::min(wgrad_most(a->s2), cin_groups); gc >= 1; --gc) {
    wgrad_chunk(a, cin_groups, (cin_groups + gc - 1) / gc);
    for (int parts = 1; parts <= taps; parts *= 3) {
      double mma = 0.0;
      for (int e = 0; e < taps / parts; ++e) mma += std::max(45, a->e[e].n / 2);
      const double tile = std::max(8.0 * mma, a->tx_bytes / 40.0);
      const double ctas = (double)a->splits * a->chunks * a->ochunks * parts;
      const double t = tile * a->split_tiles * std::max(1.0, ctas / sms);
      if (t < 0.97 * best) {
        best = t;
        best_chunks = a->chunks;
        best_parts = parts;
      }
    }
  }
  wgrad_chunk(a, cin_groups, best_chunks);
  a->parts = best_parts;
  a->entries = taps / best_parts;
  int cols = 0;
  for (int e = 0; e < a->entries; ++e) cols += a->e[e].n;  // the first part is the widest
  a->tmem_cols = 32;
  while (a->tmem_cols < cols) a->tmem_cols *= 2;
  // CTAs that share an SM share its memory: room for two where there are more than SMs
  const bool share = a->splits * a->chunks * a->ochunks * a->parts > sms && a->tmem_cols <= 256;
  const int room = (share ? kSmemMax / 2 - 1024 : kSmemMax) - 4096;
  a->stages = std::min(kWgMaxStages, std::max(room / a->stage_bytes, 1));
  if (a->stages < 2) a->stages = std::min(2, (kSmemMax - 4096) / a->stage_bytes);
}

// Floats of partial sums that plan_wgrad may ask for, whatever the batch and the device.
size_t wgrad_part_bound(int cin_groups, int cout, int kin, int stride) {
  WgradArgs a = {};
  wgrad_rows(&a, cout, stride);
  size_t most = 0;
  for (int gc = std::min(wgrad_most(a.s2), cin_groups); gc >= 1; --gc) {
    wgrad_chunk(&a, cin_groups, (cin_groups + gc - 1) / gc);
    most = std::max(most, (size_t)a.chunks * a.cols);
  }
  return most * wgrad_splits(cout, kin) * a.ochunks * a.mrows;
}

// The ring, and 4 KiB that the unused rows and columns of the last stage's operands may touch.
cudaError_t launch_wgrad(const WgradMaps& maps, const WgradArgs& a, cudaStream_t st) {
  const int smem = a.stages * a.stage_bytes + 4096;
  return launch_pdl(wgrad_kernel, a.splits * a.parts * a.chunks * a.ochunks, kWgThreads, smem, st,
                    maps, a);
}

cudaError_t launch_pack_weights(const PackArgs& a, cudaStream_t st) {
  const int grid = (int)std::min<int64_t>((a.total + 255) / 256, 152 * 8);
  return launch_pdl(pack_weights_kernel, grid, 256, 0, st, a);
}

cudaError_t launch_finish(FinishArgs a, cudaStream_t st) {
  int channels = 0;
  for (int s = 0; s < a.count; ++s) channels += a.seg[s].cout;
  a.w_blocks = (int)std::min<int64_t>((a.total + 255) / 256, 152 * 8);
  return launch_pdl(finish_kernel, a.w_blocks + channels, 256, 0, st, a);
}

cudaError_t prepare_conv_kernels() {
  const void* fns[5] = {(const void*)conv_kernel<kConvForward>,
                        (const void*)conv_kernel<kConvPartial>, (const void*)conv_kernel<kConvRoute>,
                        (const void*)dx_stride2_kernel, (const void*)wgrad_kernel};
  for (const void* fn : fns) {
    const cudaError_t e =
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace net
}  // namespace mcl
