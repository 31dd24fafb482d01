// Grid-resident form of the fused MCLBM step for middling lattices: a cooperative grid of at most one
// CTA per SM holds the whole cavity in shared memory, a tile each, and advances it many steps in one
// launch; neighbouring CTAs exchange their edges through L2.
//
// Each CTA keeps its tile with two nodes around it (the window): a node pulls from its neighbours, and
// its gradients need theta' and rho'^p of the nodes next to it (the ring), which are recomputed here
// and pull from one node further. Between two steps a CTA sends every neighbour the populations
// that the neighbour's tile and ring pull from this tile, and nothing else: six directions of its outermost
// line and three of the next. Three values travel as one word together with the step's mark; a word
// is written and read whole (128 bits, 64 with 16-bit storage), so that its mark tells the
// receiver that the values have arrived: there is no flag, no fence and no grid barrier. Two
// slots per word, used in turn, are enough: a CTA writes a slot again only after it has its
// neighbours' words of the step between, which they sent after they had read the slot.
//
// What bounds it: latency. A step is a chain of pulls (27 shared-memory loads), moments, collision
// (about 250 dependent instructions) and the way of the words to L2 and back, of which the last is about
// 1 us and the rest grows with the nodes per SM. Per step, against one launch of the TMA kernel: 100 x
// 100 1.77 us against 4.18 (cluster kernel 2.83), 128 x 128 1.98 against 4.19, with two thermal sets
// 2.64 against 5.47, 256 x 256 2.85 against 4.36, FP16 3.12 against 4.70, 276 x 276 3.3 against 5.74.
// Two sets took 3.42 us with words of one node and direction (two words for their four values): the
// inbox then allowed 56 tiles of 18 x 16 only. Warps of their own for the edge, so that the inner nodes
// are done while the words are under way, took longer (128 x 128 2.75 us): the edge's own chain is the
// step. The waits of a thread are for one word after the other, both read ahead once: what polls more
// loads the way of the words.
//
// What it gives up is other cavities beside it: the latency leaves issue slots that a second grid could
// use, but at 128 registers only small CTAs share an SM. Several cavities stepped at once, each on a
// stream of its own, per step and cavity with 1, 4 and 8 of them, against the TMA or tile kernel: 100 x
// 100 1.77, 0.69, 0.69 against 4.09, 1.04, 0.58; 128 x 128 1.98, 1.09, 1.10 against 4.16, 1.07, 0.72;
// with two sets 2.64, 2.58, 2.57 against 5.38, 1.45, 1.00; 180 x 180 2.14, 2.13, 2.13 against 4.45,
// 1.54, 1.54; 256 x 256 gains at any number. Bounds of two CTAs of 352 threads per SM (88 registers,
// spills) give 0.55, 0.78, 1.44 and 1.48 with eight, but take 11 to 17 % longer for one: the launch
// bounds keep to one cavity; who steps many of these sizes at once batches them (mclbm_batch_step) or
// asks for the other kernels (MCLBM_STEP_VARIANT).
//
// Per node the pulls, moments and collision are those of the other step kernels, and the
// stochastic-rounding streams follow the same blocks of 2^k steps, so the states are the same bits.
#pragma once

#include <type_traits>

#include "mclbm_cluster.cuh"

namespace mcl {
namespace resident {

constexpr int kThreadsMax = 640;  // 96 registers each, as from 17 warps on
constexpr int kThreadsFew = 512;  // 128: no spills
constexpr int kMinTile = 4;       // a tile's sides: an edge's two lines belong to one CTA
constexpr int kMostAcross = 32;   // CTAs along a side: a launch has at least as many steps
constexpr int kValues = 3;        // values of a word
constexpr int kWordsPerThread = 2;
constexpr int kPollLimit = 1 << 21;  // polls of a word before it is given up: a third of a second at least

__device__ __forceinline__ void store16(void* p, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile(
      "{\n\t.reg .b128 w;\n\t.reg .b64 lo, hi;\n\tmov.b64 lo, {%1, %2};\n\tmov.b64 hi, {%3, %4};\n\t"
      "mov.b128 w, {lo, hi};\n\tst.relaxed.gpu.global.b128 [%0], w;\n\t}" ::"l"(p),
      "r"(a), "r"(b), "r"(c), "r"(d)
      : "memory");
}
__device__ __forceinline__ uint4 load16(const void* p) {
  uint4 v;
  asm volatile(
      "{\n\t.reg .b128 w;\n\t.reg .b64 lo, hi;\n\tld.relaxed.gpu.global.b128 w, [%4];\n\t"
      "mov.b128 {lo, hi}, w;\n\tmov.b64 {%0, %1}, lo;\n\tmov.b64 {%2, %3}, hi;\n\t}"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p)
      : "memory");
  return v;
}
__device__ __forceinline__ void store8(void* p, uint32_t a, uint32_t b) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"((uint64_t)a | (uint64_t)b << 32)
               : "memory");
}
__device__ __forceinline__ uint2 load8(const void* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return make_uint2((uint32_t)v, (uint32_t)(v >> 32));
}

// The stored bits of a value.
__device__ __forceinline__ uint32_t bits(const float* p) { return __float_as_uint(*p); }
template <class T>
__device__ __forceinline__ uint32_t bits(const T* p) {
  return *reinterpret_cast<const uint16_t*>(p);
}
__device__ __forceinline__ void put(float* p, uint32_t v) { *p = __uint_as_float(v); }
template <class T>
__device__ __forceinline__ void put(T* p, uint32_t v) {
  *reinterpret_cast<uint16_t*>(p) = (uint16_t)v;
}

// A word: three stored values and their exclusive or with the step's mark, 128 bits with FP32 storage, 64
// with 16-bit. The poll's test takes every lane of the word: a relaxed 128-bit load proved whole only where
// all its lanes are used. Words of one value, with a number in the last lane and two lanes that nobody read, of
// which the poll tested the number and the value was used after it, came with the new number and the old value
// (FP32, two thermal sets: every run of 16 steps was off); with those two lanes tested as well, none did.
template <class T>
struct Word {
  static constexpr int kBytes = sizeof(T) == 4 ? 16 : 8;
  using Bits = typename std::conditional<sizeof(T) == 4, uint4, uint2>::type;
  // The mark of step number 1 .. 2^14: not 0, as in the inbox before the first step, and its neighbours
  // differ in many bits, so that old and new values a few bits apart don't make up for it.
  __device__ __forceinline__ static uint32_t mark(uint32_t number) {
    return sizeof(T) == 4 ? number * 0x9E3779B1u : number * 0x9E37u & 0xFFFFu;
  }
  __device__ __forceinline__ static void send(char* w, uint32_t a, uint32_t b, uint32_t c,
                                              uint32_t mark) {
    const uint32_t d = a ^ b ^ c ^ mark;
    if constexpr (sizeof(T) == 4)
      store16(w, a, b, c, d);
    else
      store8(w, a | b << 16, c | d << 16);
  }
  __device__ __forceinline__ static Bits load(const char* w) {
    if constexpr (sizeof(T) == 4)
      return load16(w);
    else
      return load8(w);
  }
  __device__ __forceinline__ static bool is(const Bits& x, uint32_t mark) {
    if constexpr (sizeof(T) == 4) {
      return (x.x ^ x.y ^ x.z ^ x.w) == mark;
    } else {
      const uint32_t both = x.x ^ x.y;
      return ((both ^ both >> 16) & 0xFFFFu) == mark;
    }
  }
  __device__ __forceinline__ static uint32_t value(const Bits& x, int k) {
    if constexpr (sizeof(T) == 4)
      return k == 0 ? x.x : (k == 1 ? x.y : x.z);
    else
      return (k == 0 ? x.x : (k == 1 ? x.x >> 16 : x.y)) & 0xFFFFu;
  }
};
// What a thread does with one of its words: the places of the values it sends and receives (-1: none),
// where it sends them and where it finds them (bytes in the inbox; in < 0: no such word).
struct Entry {
  int from[kValues], out, to[kValues], in;
};

// How the lattice is cut: gx x gy tiles of at most bw x bh nodes, of `sets` sets of populations. A CTA's
// words come from eight neighbours (m = 0 .. 3: left, right, below, above; 4 .. 7: the diagonal ones),
// each at a fixed place: per node of an edge nine directions, one more for its first and its last
// node; five from a corner.
struct Cut {
  int gx, gy, bw, bh, sets;
  __host__ __device__ int per_node() const { return 9 * sets / kValues; }
  __host__ __device__ int per_end() const { return (sets + kValues - 1) / kValues; }
  __host__ __device__ int per_corner() const { return (5 * sets + kValues - 1) / kValues; }
  __host__ __device__ int from(int m) const {
    const int ex = per_node() * bh + 2 * per_end(), ey = per_node() * bw + 2 * per_end();
    return m < 2 ? m * ex : (m < 4 ? 2 * ex + (m - 2) * ey : 2 * (ex + ey) + (m - 4) * per_corner());
  }
  __host__ __device__ int words() const { return from(8); }
  __host__ __device__ int x0(int cx, int nx) const { return (int)((int64_t)cx * nx / gx); }
  __host__ __device__ int y0(int cy, int ny) const { return (int)((int64_t)cy * ny / gy); }
};
// Direction (sx, sy) of neighbour m, and the message this CTA is to that neighbour.
__host__ __device__ inline void neighbour(int m, int& sx, int& sy) {
  sx = m < 2 ? 2 * m - 1 : (m < 4 ? 0 : ((m & 1) ? 1 : -1));
  sy = m < 2 ? 0 : (m < 4 ? 2 * m - 5 : ((m & 2) ? 1 : -1));
}
__host__ __device__ inline int opposite(int m) { return m < 4 ? m ^ 1 : 7 - (m - 4); }
__host__ __device__ inline int direction(int dx, int dy) {
  if (dy == 0) return dx == 0 ? 0 : (dx > 0 ? 1 : 3);
  if (dx == 0) return dy > 0 ? 2 : 4;
  return dy > 0 ? (dx > 0 ? 5 : 6) : (dx > 0 ? 8 : 7);
}
// Item r of the message from the neighbour at (sx, sy), whose edge is len nodes long: the node's lines
// beyond the edge (lx, ly: 1 or 2; 0 along the edge, where its place is `along`) and its direction.
// From the side: per node of the edge the three directions that come in and the three along it from line
// 1, the three that come in from line 2; and for the ring nodes at a wall, the first and the last, the
// direction that bounces back there. From a corner: the five that reach the tile or its ring.
__host__ __device__ inline bool item(int sx, int sy, int len, int r, int& lx, int& ly, int& along,
                                     int& q) {
  along = 0;
  if (sx != 0 && sy != 0) {
    lx = r == 3 ? 2 : 1;
    ly = r == 4 ? 2 : 1;
    q = direction(r == 1 ? 0 : -sx, r == 2 ? 0 : -sy);
    return r < 5;
  }
  const int side = sx + sy;  // in along the edge's normal, `along` the other way
  int line, in, by;
  if (r < 9 * len) {
    along = r / 9;
    const int k = r - 9 * along;
    line = k < 6 ? 1 : 2;
    in = k >= 3 && k < 6 ? 0 : -side;
    by = k % 3 - 1;
  } else {
    const int end = r - 9 * len;
    if (end > 1) return false;
    along = end ? len - 1 : 0;
    line = 1;
    in = side;
    by = end ? 1 : -1;
  }
  lx = sx ? line : 0;
  ly = sy ? line : 0;
  q = sx ? direction(in, by) : direction(by, in);
  return true;
}

// Value k of word r of that message: its item and set, false where there is none.
__host__ __device__ inline bool value_of(const Cut& c, bool corner, int len, int r, int k, int& it,
                                         int& set) {
  int v = r * kValues + k, limit = 5 * c.sets;
  it = 0;
  if (!corner) {
    const int group = r < c.per_node() * len ? r / c.per_node() : -1;
    if (group >= 0) {
      v -= group * c.per_node() * kValues;
      limit = 9 * c.sets;
      it = 9 * group;
    } else {
      const int end = (r - c.per_node() * len) / c.per_end();
      v -= (c.per_node() * len + end * c.per_end()) * kValues;
      limit = c.sets;
      it = 9 * len + end;
    }
  }
  it += v / c.sets;
  set = v % c.sets;
  return v < limit;
}
// Word w of CTA (cx, cy), whose tile has bw x bh nodes, of planes of `plane` places and rows of WX;
// a word has `bytes` bytes.
__host__ __device__ inline Entry entry_of(const Cut& c, int cx, int cy, int bw, int bh, int WX, int plane,
                                          int bytes, int w) {
  Entry e;
  for (int k = 0; k < kValues; ++k) e.from[k] = e.to[k] = -1;
  e.out = e.in = -1;
  int m = 0;
  while (m < 7 && w >= c.from(m + 1)) ++m;
  const int r = w - c.from(m);
  int sx, sy;
  neighbour(m, sx, sy);
  const int ox = cx + sx, oy = cy + sy;
  if ((unsigned)ox >= (unsigned)c.gx || (unsigned)oy >= (unsigned)c.gy) return e;
  const int len = sx ? bh : bw;  // the neighbour's edge is as long
  for (int k = 0; k < kValues; ++k) {
    int it, set, lx, ly, along, q;
    if (!value_of(c, m >= 4, len, r, k, it, set)) continue;
    if (!item(sx, sy, len, it, lx, ly, along, q)) continue;
    const int ti = sx < 0 ? -lx : (sx > 0 ? bw - 1 + lx : along);
    const int tj = sy < 0 ? -ly : (sy > 0 ? bh - 1 + ly : along);
    e.to[k] = (set * kQ + q) * plane + (tj + 2) * WX + ti + 2;
    // the same word of the message to that neighbour, for which this CTA is at (-sx, -sy)
    item(-sx, -sy, len, it, lx, ly, along, q);
    const int fi = sx < 0 ? lx - 1 : (sx > 0 ? bw - lx : along);
    const int fj = sy < 0 ? ly - 1 : (sy > 0 ? bh - ly : along);
    e.from[k] = (set * kQ + q) * plane + (fj + 2) * WX + fi + 2;
    e.in = ((cy * c.gx + cx) * c.words() + w) * bytes;
    e.out = ((oy * c.gx + ox) * c.words() + c.from(opposite(m)) + r) * bytes;
  }
  return e;
}

// Where a node's nine pulled directions come from (cluster::Sources, here places in the window).
__device__ __forceinline__ cluster::Sources sources_of(int nx, int ny, int WX, int plane, int i, int j,
                                                       int at) {
  cluster::Sources s;
  s.neg = 0;
#pragma unroll
  for (int q = 0; q < kQ; ++q) {
    const int si = i - ex(q), sj = j - ey(q);
    const bool inx = (unsigned)si < (unsigned)nx, iny = (unsigned)sj < (unsigned)ny;
    if (inx && iny) {
      s.f[q] = (uint32_t)(q * plane + at - ey(q) * WX - ex(q));
      s.g[q] = s.f[q] + (uint32_t)(2 * kQ * plane);
    } else {
      s.f[q] = (uint32_t)(opp(q) * plane + at);
      s.g[q] = (uint32_t)(inx ? (2 * kQ + mir(q)) * plane + at - ex(q) : (2 * kQ + opp(q)) * plane + at);
      if (!inx) s.neg |= 1u << q;
    }
  }
  return s;
}

// n steps (even) from a.src to a.dst, the same level. inbox: two slots for every word of every CTA, zero
// at the start.
template <class T, bool SR, bool ALLF, bool TWO, int MAXT>
__global__ void __launch_bounds__(MAXT, 1)
    step_resident_kernel(const StepArgs a, const Cut cut, int n, char* inbox, uint32_t* epoch) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int NP = TWO ? kPlanes2 : kPlanes;
  using W = Word<T>;
  const Layout& L = a.L;
  const StepConsts& k = a.k;
  const int cx = (int)blockIdx.x % cut.gx, cy = (int)blockIdx.x / cut.gx;
  const int x0 = cut.x0(cx, L.nx), y0 = cut.y0(cy, L.ny);
  const int bw = cut.x0(cx + 1, L.nx) - x0, bh = cut.y0(cy + 1, L.ny) - y0;
  const int WX = cut.bw + 4, plane = WX * (cut.bh + 4);
  const int MX = cut.bw + 2;
  T* buf = reinterpret_cast<T*>(smem_raw);
  float* mth = reinterpret_cast<float*>(smem_raw + ((size_t)NP * plane * sizeof(T) + 15) / 16 * 16);
  float* mrp = mth + MX * (cut.bh + 2);
  __shared__ int lost;  // a wait has run out: nothing is waited for any more
  const int t = threadIdx.x;
  if (t == 0) lost = 0;

  // a thread per node of the tile, then one per ring node: its left and right columns, its rows below
  // and above; a ring node beyond a wall is not there
  const int own = bw * bh;
  int wi, wj;  // place in the tile
  if (t < own) {
    wj = t / bw;
    wi = t - wj * bw;
  } else if (t < own + 2 * bh) {
    const int e = t - own;
    wi = e < bh ? -1 : bw;
    wj = e < bh ? e : e - bh;
  } else {
    const int e = t - own - 2 * bh;
    wj = e < bw ? -1 : bh;
    wi = e < bw ? e : e - bw;
  }
  const bool mine = t < own;
  const int i = x0 + wi, j = y0 + wj;
  const bool there = t < own + 2 * (bw + bh) && (unsigned)i < (unsigned)L.nx &&
                     (unsigned)j < (unsigned)L.ny;
  const size_t o = (size_t)j * L.pitch + i;
  const int at = (wj + 2) * WX + wi + 2;
  const cluster::Sources src = sources_of(L.nx, L.ny, WX, plane, i, j, there ? at : 0);

  // the words this thread sends and receives. With one thermal set the values of a word are those of
  // one node and direction, nine planes apart.
  const int words = cut.words();
  const size_t turn = (size_t)gridDim.x * words * W::kBytes;
  Entry e[kWordsPerThread];
#pragma unroll
  for (int x = 0; x < kWordsPerThread; ++x) {
    const int w = t + x * (int)blockDim.x;
    e[x].in = -1;
    if (w < words) e[x] = entry_of(cut, cx, cy, bw, bh, WX, plane, W::kBytes, w);
  }
  auto place = [&](const int* at3, int k) { return TWO ? at3[k] : at3[0] + k * kQ * plane; };

  // the window's populations: the tile and what lies around it, as far as the lattice goes
  for (int e = t; e < plane; e += blockDim.x) {
    const int rr = e / WX, ci = x0 + e - rr * WX - 2, cj = y0 + rr - 2;
    if ((unsigned)ci < (unsigned)L.nx && (unsigned)cj < (unsigned)L.ny) {
      const T* p0 = static_cast<const T*>(a.src) + (size_t)cj * L.pitch + ci;
      T x[NP];  // all loads before the first store
#pragma unroll
      for (int p = 0; p < NP; ++p) x[p] = p0[(size_t)p * L.plane];
#pragma unroll
      for (int p = 0; p < NP; ++p) buf[p * plane + e] = x[p];
    }
  }
  const uint32_t ep0 = *(volatile const uint32_t*)epoch;
  uint32_t ep = ep0;
  int block_left = 0;
  uint32_t seed = 0, sh = 0;
  __syncthreads();
  for (int s = 0; s < n; ++s) {
    if (SR) {  // the blocks of 2^k steps of a launch sequence of captured graphs
      if (block_left == 0) {
        block_left = 1 << min(31 - __clz(n - s), kGraphLogMax);
        seed = 0;
      }
      sh = mix32(seed++ ^ mix32(ep + 0x632BE5ABu));
      if (--block_left == 0) ++ep;
    }
    float fw[kQ], fp[kQ], g[kQ], gp[TWO ? kQ : 1];
    const int m = (wj + 1) * MX + wi + 1;
    if (there) {
#pragma unroll
      for (int q = 0; q < kQ; ++q) {
        using S = pair::St<T>;
        const uint32_t sign = (src.neg << (31 - q)) & 0x80000000u;
        fw[q] = S::ld1(buf + src.f[q]);
        fp[q] = S::ld1(buf + src.f[q] + kQ * plane);
        g[q] = __uint_as_float(__float_as_uint(S::ld1(buf + src.g[q])) ^ sign);
        if (TWO) gp[q] = __uint_as_float(__float_as_uint(S::ld1(buf + src.g[q] + kQ * plane)) ^ sign);
      }
      if constexpr (TWO)
        mth[m] = pair::mixture_s<T>(k, pair::sum9(fw), pair::sum9(fp), pair::sum9(g),
                                    pair::sum9(gp));
      else
        mth[m] = pair::sum9(g);
      mrp[m] = pair::sum9(fp);
    }
    __syncthreads();  // every population is in registers: the window may be written
    if (mine) {
      const float th = mth[m], rp = mrp[m];
      const float thN = j + 1 < L.ny ? mth[m + MX] : th, thS = j > 0 ? mth[m - MX] : th;
      const float rpN = j + 1 < L.ny ? mrp[m + MX] : rp, rpS = j > 0 ? mrp[m - MX] : rp;
      const float thE = i + 1 < L.nx ? mth[m + 1] : -th, thW = i > 0 ? mth[m - 1] : -th;
      const float rpE = i + 1 < L.nx ? mrp[m + 1] : rp, rpW = i > 0 ? mrp[m - 1] : rp;
      cluster::SharedSink<T, SR> sink{buf + at, plane, SR ? mix32((uint32_t)o ^ sh) : 0u};
      pair::collide<1, ALLF, T, TWO>(k, L, sink, i, j, fw, fp, g, gp, thE, thW, thN, thS, rpE, rpW,
                                     rpN, rpS);
    }
    __syncthreads();
    if (s + 1 < n) {
      const uint32_t mark = W::mark((uint32_t)(s + 1));
      char* box = inbox + (size_t)(s & 1) * turn;
#pragma unroll
      for (int x = 0; x < kWordsPerThread; ++x) {
        if (e[x].in < 0) continue;
        uint32_t v[kValues];
#pragma unroll
        for (int y = 0; y < kValues; ++y) {
          const int p = place(e[x].from, y);
          v[y] = !TWO || p >= 0 ? bits(buf + p) : 0u;
        }
        W::send(box + e[x].out, v[0], v[1], v[2], mark);
      }
      // all words are asked for at once, then waited for one by one (without a word: the first is read)
      typename W::Bits got[kWordsPerThread];
#pragma unroll
      for (int x = 0; x < kWordsPerThread; ++x) got[x] = W::load(box + max(e[x].in, 0));
#pragma unroll
      for (int x = 0; x < kWordsPerThread; ++x) {
        if (e[x].in < 0) continue;
        for (int polls = 1; !W::is(got[x], mark); ++polls) {
          if ((polls & 255) == 0 && (polls >= kPollLimit || *(volatile int*)&lost)) {
            *(volatile int*)&lost = 1;
            atomicOr(a.err, 1);
            break;
          }
          got[x] = W::load(box + e[x].in);
        }
#pragma unroll
        for (int y = 0; y < kValues; ++y) {
          const int p = place(e[x].to, y);
          if (!TWO || p >= 0) put(buf + p, W::value(got[x], y));
        }
      }
      __syncthreads();
    }
  }
  for (int u = t; u < own; u += blockDim.x) {
    const int rr = u / bw, cc = u - rr * bw;
    T* p0 = static_cast<T*>(a.dst) + (size_t)(y0 + rr) * L.pitch + x0 + cc;
    const T* res = buf + (rr + 2) * WX + cc + 2;
#pragma unroll
    for (int p = 0; p < NP; ++p) p0[(size_t)p * L.plane] = res[p * plane];
  }
  // one epoch per block of 2^k steps: the same count whether or not the rounding uses it. Every
  // CTA has read the old one: it takes n steps for the last of them to let this CTA get here.
  if (blockIdx.x == 0 && t == 0)
    *epoch = ep0 + (uint32_t)((n >> kGraphLogMax) + __popc((n & ((1 << kGraphLogMax) - 1)) >> 1));
}

// ---- host side ---------------------------------------------------------------------------------
inline size_t smem_bytes(const Layout& L, const Cut& c) {
  return ((size_t)L.np * (c.bw + 4) * (c.bh + 4) * L.elem + 15) / 16 * 16 +
         (size_t)2 * (c.bw + 2) * (c.bh + 2) * sizeof(float);
}
inline size_t inbox_bytes(const Layout& L, const Cut& c) {
  return (size_t)2 * c.gx * c.gy * c.words() * (L.elem == 2 ? 8 : 16);
}
inline int threads_of(const Cut& c) {
  const int nodes = c.bw * c.bh + 2 * (c.bw + c.bh);
  const int words = (c.words() + kWordsPerThread - 1) / kWordsPerThread;
  return (std::max(nodes, words) + 31) / 32 * 32;
}

template <class T, int MAXT>
const void* kernel_of(bool sr, bool all, bool two) {
  constexpr bool kSr = sizeof(T) == 2;
  if (two)
    return sr ? (const void*)step_resident_kernel<T, kSr, false, true, MAXT>
              : (const void*)step_resident_kernel<T, false, false, true, MAXT>;
  if (sr)
    return all ? (const void*)step_resident_kernel<T, kSr, true, false, MAXT>
               : (const void*)step_resident_kernel<T, kSr, false, false, MAXT>;
  return all ? (const void*)step_resident_kernel<T, false, true, false, MAXT>
             : (const void*)step_resident_kernel<T, false, false, false, MAXT>;
}
template <class T>
const void* kernel_of(int threads, bool sr, bool all, bool two) {
  return threads <= kThreadsFew ? kernel_of<T, kThreadsFew>(sr, all, two)
                                : kernel_of<T, kThreadsMax>(sr, all, two);
}

// Sets c.re_* where the kernel can run (re_ctas 0: it cannot): the tiles of the cut with the fewest
// threads per CTA fit the threads and shared memory, the inbox fits the state level that is not read, and
// the device takes the grid at once.
template <class T>
cudaError_t prepare(StepConfig* c, const Layout& L, bool all, bool two) {
  c->re_ctas = 0;
  int dev = 0, sms = 0, coop = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev)) != cudaSuccess)
    return e;
  if (!coop || (int64_t)L.nx * L.ny > (int64_t)sms * kThreadsMax) return cudaSuccess;
  Cut best{};
  int fewest = kThreadsMax + 1;
  for (int gx = 1; gx <= kMostAcross && gx * kMinTile <= L.nx; ++gx) {
    for (int gy = 1; gy <= kMostAcross && gx * gy <= sms && gy * kMinTile <= L.ny; ++gy) {
      const Cut t{gx, gy, (L.nx + gx - 1) / gx, (L.ny + gy - 1) / gy, L.np / kQ};
      if (t.bw * t.bh >= fewest) continue;  // most cuts: too few CTAs
      const int threads = threads_of(t);
      if (threads < fewest && smem_bytes(L, t) <= 226 * 1024 &&
          inbox_bytes(L, t) <= (size_t)L.np * L.plane * L.elem) {
        fewest = threads;
        best = t;
      }
    }
  }
  if (fewest > kThreadsMax) return cudaSuccess;
  const void* fn = kernel_of<T>(fewest, c->sr && sizeof(T) == 2, all, two);
  if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024)) !=
      cudaSuccess)
    return e;
  int per_sm = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, fewest, smem_bytes(L, best))) !=
      cudaSuccess)
    return e;
  if ((int64_t)per_sm * sms < (int64_t)best.gx * best.gy) return cudaSuccess;
  c->re_gx = best.gx;
  c->re_gy = best.gy;
  c->re_ctas = best.gx * best.gy;
  c->re_threads = fewest;
  return cudaSuccess;
}

// scratch: the state level that is not read.
template <class T>
cudaError_t launch(const StepArgs& a, const StepConfig& c, int n, void* scratch, uint32_t* epoch,
                   cudaStream_t st) {
  const Cut cut{c.re_gx, c.re_gy, (a.L.nx + c.re_gx - 1) / c.re_gx,
                (a.L.ny + c.re_gy - 1) / c.re_gy, a.L.np / kQ};
  cudaError_t e = cudaMemsetAsync(scratch, 0, inbox_bytes(a.L, cut), st);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c.re_ctas);
  cfg.blockDim = dim3(c.re_threads);
  cfg.dynamicSmemBytes = smem_bytes(a.L, cut);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  StepArgs args = a;
  Cut cut_arg = cut;
  char* inbox = static_cast<char*>(scratch);
  void* params[] = {&args, &cut_arg, &n, &inbox, &epoch};
  const bool all = a.k.mask == MCLBM_F_ALL && !a.k.two_sets;
  return cudaLaunchKernelExC(
      &cfg, kernel_of<T>(c.re_threads, c.sr && sizeof(T) == 2, all, a.k.two_sets), params);
}

}  // namespace resident
}  // namespace mcl
