// C ABI of the warm-start network (include/mclbm_net.h): workspace planning, the forward and
// backward sequences of launches, Adam, and the exposed tensor-core GEMM. Host code only; the
// kernels are in net_conv.cu, net_kernels.cu and net_gemm.cu.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <vector>

#include "../../include/mclbm.h"
#include "../../include/mclbm_net.h"
#include "net_internal.h"
#include "nvtx_range.h"

using namespace mcl::net;

namespace {

constexpr int kNumLayers = 10;
constexpr int kLossChunks = 64;  // most pixel chunks per sample of the loss
constexpr int kStatBlocks = 256;
static_assert(kFields * kStatBlocks * 2 >= kShiftPartials,
              "the warm start's mean shifts reuse the field statistics' scratch");

struct Layer {
  // definition
  int cu, cs, cout, stride, film, act;
  int src1, src2;  // producing layer of each input source (-1: the geometry input X)
  int up;          // src1 is upsampled by 2
  // shapes
  int H, W, Ho, Wo, kin;
  int groups;      // channel groups of 8 of the input
  int og;          // channel groups of the output
  int fsplits, fsplit_k;  // forward split over K (layers with few output tiles): count, k each
  int64_t w_off, b_off;
  int film_off;  // offset of this layer's (gamma, beta) slice in r, or -1
  // the layer that reads y, the channel group it is written at there, upsampled or not
  int dst, dst_group, dst_up;
  size_t wf_elems, wd_elems;  // packed weights: forward, input gradient
  size_t sums_elems;
  // device buffers
  float *pre, *dy;
  __nv_bfloat16 *in, *wf, *wd, *dpre;  // in: null for the stride-2 layers (they read a skip source)
  float* part;
  double* sums;
};

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

struct mclbm_net {
  mclbm_net_config cfg;
  Layer L[kNumLayers];
  int F = 0;
  int64_t n_params = 0, mlp_off = 0;
  size_t ws_bytes = 0;
  size_t wpart_elems = 0;  // partial sums of the weight gradients
  size_t fpart_elems = 0;  // partial sums of the K-split forward layers
  int sms = 152;           // multiprocessors, set by bind
  // bound memory
  char* ws = nullptr;
  cudaStream_t stream = nullptr;
  float *params = nullptr, *grads = nullptr, *adam_m = nullptr, *adam_v = nullptr;
  float* norm = nullptr;  // mean[5], scale[5] of the fields' deviations from their rest values
  float *wpart = nullptr, *fpart = nullptr;
  float *cond_c = nullptr, *a1 = nullptr, *r = nullptr, *dr = nullptr;
  double *loss_part = nullptr, *loss = nullptr, *stat_part = nullptr;
  // tensor maps and plans of the backward pass, laid out for one batch size
  int plan_batch = 0;
  WgradMaps wg_maps[kNumLayers];
  WgradArgs wg[kNumLayers];
  CUtensorMap dx_map[kNumLayers];
  int* err = nullptr;
  int adam_t = 0;
  bool bound = false;
  char errmsg[512] = {0};
};

namespace {

int fail(mclbm_net* n, int code, const char* fmt, ...) {
  if (n) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(n->errmsg, sizeof(n->errmsg), fmt, ap);
    va_end(ap);
  }
  return code;
}

int cuda_fail(mclbm_net* n, cudaError_t e, const char* what) {
  return fail(n, MCLBM_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

bool config_valid(const mclbm_net_config* c) {
  return c && c->ny >= 16 && c->nx >= 16 && c->ny <= 4096 && c->nx <= 4096 && c->ny % 16 == 0 &&
         c->nx % 16 == 0 && c->c0 >= 8 && c->c0 <= 64 && c->c0 % 8 == 0 && c->hidden >= 1 &&
         c->hidden <= 256 && c->max_batch >= 1 && c->max_batch <= 256 &&
         (int64_t)c->max_batch * c->ny * c->nx <= (int64_t)1 << 26 &&
         c->max_batch * c->hidden <= 4096;  // the MLP kernels keep [batch][hidden] in shared memory
}

// Elements of a packed weight operand with n columns and K groups of 8 channels (see PackSeg).
size_t packed_elems(int n, int groups) {
  const int nt = conv_n_tile(n);
  return (size_t)((n + nt - 1) / nt) * conv_slices(groups) * 18 * nt * 8;
}

// Elements of the layer's own input buffer: one image of the geometry, or the sources of a batch.
size_t in_elems(const mclbm_net* n, int l) {
  const Layer& y = n->L[l];
  return (size_t)y.groups * 8 * y.H * y.W * (l == 0 ? 1 : n->cfg.max_batch);
}

// Layer table, parameter offsets and workspace size (no device work).
void plan(mclbm_net* n) {
  const mclbm_net_config& c = n->cfg;
  const int C0 = c.c0, C1 = 2 * C0, C2 = 4 * C0, C3 = 8 * C0, C4 = 8 * C0;
  // cu, cs, cout, stride, film, act, src1, src2, up
  const int def[kNumLayers][9] = {
      {4, 0, C0, 1, 0, 1, -1, -1, 0},  // e0
      {C0, 0, C1, 2, 0, 1, 0, -1, 0},  // e1
      {C1, 0, C2, 2, 0, 1, 1, -1, 0},  // e2
      {C2, 0, C3, 2, 0, 1, 2, -1, 0},  // e3
      {C3, 0, C4, 2, 1, 1, 3, -1, 0},  // e4
      {C4, C3, C3, 1, 1, 1, 4, 3, 1},  // d3
      {C3, C2, C2, 1, 1, 1, 5, 2, 1},  // d2
      {C2, C1, C1, 1, 1, 1, 6, 1, 1},  // d1
      {C1, C0, C0, 1, 1, 1, 7, 0, 1},  // d0
      {C0, 0, kFields, 1, 0, 0, 8, -1, 0},  // out
  };
  int64_t off = 0;
  int film_off = 0;
  for (int l = 0; l < kNumLayers; ++l) {
    Layer& y = n->L[l];
    std::memset(&y, 0, sizeof(y));
    y.cu = def[l][0];
    y.cs = def[l][1];
    y.cout = def[l][2];
    y.stride = def[l][3];
    y.film = def[l][4];
    y.act = def[l][5];
    y.src1 = def[l][6];
    y.src2 = def[l][7];
    y.up = def[l][8];
    if (y.src1 < 0) {
      y.H = c.ny;
      y.W = c.nx;
    } else {
      const Layer& s = n->L[y.src1];
      y.H = y.up ? 2 * s.Ho : s.Ho;
      y.W = y.up ? 2 * s.Wo : s.Wo;
    }
    y.Ho = y.H / y.stride;
    y.Wo = y.W / y.stride;
    y.kin = 9 * (y.cu + y.cs);
    y.groups = (y.cu + y.cs + 7) / 8;
    y.og = (y.cout + 7) / 8;
    y.dst = -1;
    y.w_off = off;
    off += (int64_t)y.cout * y.kin;
    y.b_off = off;
    off += y.cout;
    y.film_off = -1;
    if (y.film) {
      y.film_off = film_off;
      film_off += 2 * y.cout;
    }
    // forward products with fewer output tiles than half a wave (128 pixels x 128 channels each)
    // are split over K in multiples of 64, partial sums added in order by the epilogue kernel
    const int64_t tiles_f = (((int64_t)c.max_batch * y.Ho * y.Wo + 127) / 128) *
                            ((y.cout + 127) / 128);
    const int nks = (((y.kin + 7) & ~7) + 63) / 64;
    y.fsplits = tiles_f >= 76 ? 1 : (int)std::max<int64_t>(
                                        1, std::min<int64_t>({152 / tiles_f, 8, (int64_t)nks}));
    y.fsplit_k = (nks + y.fsplits - 1) / y.fsplits * 64;
  }
  // where each layer's output goes: a decoder input (upsampled source first, then the skip
  // source) or the output layer's; the stride-2 layers read the skip source where it lies
  for (int l = 0; l < kNumLayers; ++l) {
    const Layer& y = n->L[l];
    if (y.stride == 2) continue;
    if (y.src1 >= 0) {
      n->L[y.src1].dst = l;
      n->L[y.src1].dst_group = 0;
      n->L[y.src1].dst_up = y.up;
    }
    if (y.src2 >= 0) {
      n->L[y.src2].dst = l;
      n->L[y.src2].dst_group = y.cu / 8;
      n->L[y.src2].dst_up = 0;
    }
  }
  n->F = film_off;
  n->mlp_off = off;
  off += (int64_t)c.hidden * 3 + c.hidden + (int64_t)n->F * c.hidden + n->F;
  n->n_params = off;

  // workspace
  const int64_t B = c.max_batch;
  size_t bytes = 0;
  const size_t np = (size_t)n->n_params;
  bytes += 4 * align256(np * 4);  // params, grads, adam m, v
  bytes += align256(2 * kFields * 4);  // normaliser
  n->wpart_elems = 0;
  n->fpart_elems = 0;
  for (int l = 0; l < kNumLayers; ++l) {
    Layer& y = n->L[l];
    const size_t P = (size_t)B * y.Ho * y.Wo;
    const int cin = y.cu + y.cs;
    y.wf_elems = packed_elems(y.cout, y.groups);
    y.wd_elems = l == 0 ? 0
                 : y.stride == 1
                     ? packed_elems(cin, y.og)
                     : (size_t)((cin + 15) / 16) * ((y.og + dx_stride2_kg(y.cout) - 1) /
                                                    dx_stride2_kg(y.cout)) *
                           9 * dx_stride2_kg(y.cout) * 16 * 8;
    // act_chunks is at most 608 / groups per batch, or 1 per sample
    y.sums_elems = (size_t)y.cout * (std::max<size_t>(B, 608) + B * kLossChunks * (l == 9)) * 3;
    bytes += align256((size_t)y.cout * P * 4);               // pre
    bytes += align256((size_t)y.cout * P * 4);               // dy
    if (y.stride == 1) bytes += align256(in_elems(n, l) * 2);  // in
    bytes += align256(y.wf_elems * 2) + align256(y.wd_elems * 2);
    bytes += align256((size_t)y.og * 8 * P * 2);             // dpre
    bytes += align256(y.sums_elems * 8);
    n->wpart_elems += wgrad_part_bound(y.groups, y.cout, y.kin, y.stride);
    if (y.fsplits > 1)
      n->fpart_elems = std::max(n->fpart_elems, (size_t)y.fsplits * y.cout * P);
  }
  bytes += align256(n->wpart_elems * 4);
  bytes += align256(n->fpart_elems * 4);
  bytes += align256((size_t)B * 3 * 4) + align256((size_t)B * c.hidden * 4) +
           2 * align256((size_t)B * n->F * 4);
  bytes += align256((size_t)B * kLossChunks * 8) + align256(8) +
           align256(kFields * kStatBlocks * 2 * 8);
  bytes += align256(4);
  n->ws_bytes = bytes;
}

template <typename T>
T* carve(char*& p, size_t count) {
  T* out = reinterpret_cast<T*>(p);
  p += align256(count * sizeof(T));
  return out;
}

void assign(mclbm_net* n) {
  const mclbm_net_config& c = n->cfg;
  const int64_t B = c.max_batch;
  char* p = n->ws;
  const size_t np = (size_t)n->n_params;
  n->params = carve<float>(p, np);
  n->grads = carve<float>(p, np);
  n->adam_m = carve<float>(p, np);
  n->adam_v = carve<float>(p, np);
  n->norm = carve<float>(p, 2 * kFields);
  for (int l = 0; l < kNumLayers; ++l) {
    Layer& y = n->L[l];
    const size_t P = (size_t)B * y.Ho * y.Wo;
    y.pre = carve<float>(p, (size_t)y.cout * P);
    y.dy = carve<float>(p, (size_t)y.cout * P);
    y.in = y.stride == 1 ? carve<__nv_bfloat16>(p, in_elems(n, l)) : nullptr;
    y.wf = carve<__nv_bfloat16>(p, y.wf_elems);
    y.wd = carve<__nv_bfloat16>(p, y.wd_elems);
    y.dpre = carve<__nv_bfloat16>(p, (size_t)y.og * 8 * P);
    y.sums = carve<double>(p, y.sums_elems);
  }
  n->wpart = carve<float>(p, n->wpart_elems);
  n->fpart = carve<float>(p, n->fpart_elems);
  n->cond_c = carve<float>(p, (size_t)B * 3);
  n->a1 = carve<float>(p, (size_t)B * c.hidden);
  n->r = carve<float>(p, (size_t)B * n->F);
  n->dr = carve<float>(p, (size_t)B * n->F);
  n->loss_part = carve<double>(p, (size_t)B * kLossChunks);
  n->loss = carve<double>(p, 1);
  n->stat_part = carve<double>(p, kFields * kStatBlocks * 2);
  n->err = carve<int>(p, 1);
  float* part = n->wpart;
  for (int l = 0; l < kNumLayers; ++l) {
    n->L[l].part = part;
    part += wgrad_part_bound(n->L[l].groups, n->L[l].cout, n->L[l].kin, n->L[l].stride);
  }
  n->plan_batch = 0;
}

MlpArgs mlp_args(mclbm_net* n, int batch, const float* cond) {
  MlpArgs a;
  const int64_t o = n->mlp_off;
  const int H = n->cfg.hidden;
  a.cond_raw = cond;
  a.W1 = n->params + o;
  a.b1 = a.W1 + 3 * H;
  a.W2 = a.b1 + H;
  a.b2 = a.W2 + (int64_t)n->F * H;
  a.batch = batch;
  a.H = H;
  a.F = n->F;
  a.c = n->cond_c;
  a.a1 = n->a1;
  a.r = n->r;
  return a;
}

// BF16 weights in the operand layouts, from the FP32 parameters.
cudaError_t refresh_bf16_weights(mclbm_net* n) {
  PackArgs a;
  std::memset(&a, 0, sizeof(a));
  a.params = n->params;
  for (int l = 0; l < kNumLayers; ++l) {
    const Layer& y = n->L[l];
    for (int d = 0; d < (l == 0 ? 1 : 2); ++d) {
      PackSeg& g = a.seg[a.count++];
      g.kind = d == 0 ? kPackForward : (y.stride == 1 ? kPackTransposed : kPackStride2);
      g.cout = y.cout;
      g.cin = y.cu + y.cs;
      g.nt = conv_n_tile(d == 0 ? y.cout : g.cin);
      g.kg = dx_stride2_kg(y.cout);
      g.slices = g.kind == kPackStride2 ? (y.og + g.kg - 1) / g.kg
                                        : conv_slices(d == 0 ? y.groups : y.og);
      g.w_off = y.w_off;
      g.start = a.total;
      g.out = d == 0 ? y.wf : y.wd;
      a.total += (int64_t)(d == 0 ? y.wf_elems : y.wd_elems);
    }
  }
  return launch_pack_weights(a, n->stream);
}

// A layer's input: its own buffer, or the skip source inside a decoder's input.
struct Input {
  const __nv_bfloat16* x;
  int64_t group, image;  // pixels between groups and images
};
Input input_of(const mclbm_net* n, int l, int batch) {
  const Layer& y = n->L[l];
  const int64_t hw = (int64_t)y.H * y.W;
  if (l == 0) return {y.in, hw, 0};
  if (y.stride == 1) return {y.in, batch * hw, hw};
  const Layer& s = n->L[y.src1];
  return {n->L[s.dst].in + s.dst_group * batch * hw * 8, batch * hw, hw};
}

cudaError_t forward(mclbm_net* n, int batch, const float* cond, bool keep_pre) {
  cudaStream_t st = n->stream;
  cudaError_t e = launch_mlp_forward(mlp_args(n, batch, cond), st);
  if (e != cudaSuccess) return e;
  for (int l = 0; l < kNumLayers; ++l) {
    Layer& y = n->L[l];
    const Input in = input_of(n, l, batch);
    ConvArgs a;
    std::memset(&a, 0, sizeof(a));
    a.src = in.x;
    a.src_group = in.group;
    a.src_image = in.image;
    a.groups = y.groups;
    a.batch = batch;
    a.H = y.H;
    a.W = y.W;
    a.stride = y.stride;
    a.Ho = y.Ho;
    a.Wo = y.Wo;
    a.N = y.cout;
    a.w = y.wf;
    a.err = n->err;
    ConvEpilogue& ep = a.ep;
    ep.bias = n->params + y.b_off;
    ep.film = y.film ? n->r : nullptr;
    ep.film_stride = n->F;
    ep.film_off = y.film_off;
    // the pre-activations are what the backward pass reads (and the output layer's the result)
    ep.pre = keep_pre || l == kNumLayers - 1 ? y.pre : nullptr;
    ep.act = y.act;
    if (y.dst >= 0) {
      const Layer& d = n->L[y.dst];
      ep.y_group = (int64_t)batch * d.H * d.W;
      ep.y = d.in + y.dst_group * ep.y_group * 8;
      ep.up = y.dst_up;
    }
    plan_conv(&a, y.fsplits, y.fsplit_k);
    if (y.fsplits > 1) {
      a.part = n->fpart;
      if ((e = launch_conv(a, kConvPartial, n->sms, st)) != cudaSuccess) return e;
      e = launch_conv_epilogue_splitk(n->fpart, y.fsplits, batch, y.Ho, y.Wo, y.cout, ep, st);
    } else {
      e = launch_conv(a, kConvForward, n->sms, st);
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Tensor maps and plans of the backward pass for a batch size (kept until another is asked for).
bool plan_backward(mclbm_net* n, int batch) {
  if (n->plan_batch == batch) return true;
  n->plan_batch = 0;
  for (int l = 0; l < kNumLayers; ++l) {
    const Layer& y = n->L[l];
    const int64_t P = (int64_t)batch * y.Ho * y.Wo;
    WgradArgs& a = n->wg[l];
    std::memset(&a, 0, sizeof(a));
    plan_wgrad(&a, y.groups, y.cout, y.kin, y.Ho, y.Wo, batch, y.stride, n->sms);
    a.src_images = l > 0;
    a.part = y.part;
    a.err = n->err;
    WgradMaps& m = n->wg_maps[l];
    if (!encode_groups(&m.a, y.dpre, y.og, P, batch, y.Ho, y.Wo, 16, a.go, 8)) return false;
    const Input in = input_of(n, l, batch);
    const int images = l == 0 ? 1 : batch;
    if (y.stride == 1) {
      if (!encode_groups(&m.b[0], in.x, y.groups, in.group, images, y.H, y.W, 18, a.gc, 10))
        return false;
    } else {
      for (int p = 0; p < 4; ++p)
        if (!encode_parity(&m.b[p], in.x, p >> 1, p & 1, y.groups, in.group, images, y.H, y.W, 17,
                           a.gc, 9))
          return false;
      if (!encode_groups(&n->dx_map[l], y.dpre, y.og, P, batch, y.Ho, y.Wo, 9,
                         dx_stride2_kg(y.cout), 17))
        return false;
    }
  }
  n->plan_batch = batch;
  return true;
}

// Loss and gradients into n->grads (loss into n->loss on the device).
cudaError_t loss_backward(mclbm_net* n, int batch, const float* cond, const float* target) {
  cudaStream_t st = n->stream;
  if (!plan_backward(n, batch)) return cudaErrorNotSupported;
  const int hw = n->cfg.ny * n->cfg.nx;
  Layer& out = n->L[kNumLayers - 1];
  int sum_chunks[kNumLayers];
  LossArgs la;
  la.out = out.pre;
  la.target = target;
  la.cond = cond;
  la.norm = n->norm;
  la.batch = batch;
  la.hw = hw;
  la.chunks = std::min(kLossChunks, act_chunks(8, batch, hw));
  la.dpre = out.dpre;
  la.sums = out.sums;
  la.partial = n->loss_part;
  sum_chunks[kNumLayers - 1] = la.chunks;
  cudaError_t e = launch_loss(la, st);
  if (e != cudaSuccess) return e;
  if ((e = launch_sum_partials(n->loss_part, batch * la.chunks, n->loss, st)) != cudaSuccess)
    return e;

  bool written[kNumLayers] = {false};
  for (int l = kNumLayers - 1; l >= 0; --l) {
    Layer& y = n->L[l];
    if (l < kNumLayers - 1) {
      ActBwdArgs aa;
      aa.dy = y.dy;
      aa.pre = y.pre;
      aa.film = y.film ? n->r : nullptr;
      aa.film_stride = n->F;
      aa.film_off = y.film_off;
      aa.C = y.cout;
      aa.batch = batch;
      aa.hw = y.Ho * y.Wo;
      aa.chunks = act_chunks(y.cout, batch, aa.hw);
      aa.dpre = y.dpre;
      aa.sums = y.sums;
      sum_chunks[l] = aa.chunks;
      if ((e = launch_act_backward(aa, st)) != cudaSuccess) return e;
    }
    if ((e = launch_wgrad(n->wg_maps[l], n->wg[l], st)) != cudaSuccess) return e;
    if (l == 0) break;
    if (y.stride == 2) {
      DxStride2Args d;
      std::memset(&d, 0, sizeof(d));
      d.batch = batch;
      d.Ho = y.Ho;
      d.Wo = y.Wo;
      d.C = y.cu;
      d.w = y.wd;
      d.dsrc = n->L[y.src1].dy;
      d.accumulate = written[y.src1] ? 1 : 0;
      written[y.src1] = true;
      d.err = n->err;
      plan_dx_stride2(&d, y.cout);
      if ((e = launch_dx_stride2(n->dx_map[l], d, n->sms, st)) != cudaSuccess) return e;
      continue;
    }
    // the convolution of the pre-activation gradient with the flipped, transposed kernel
    ConvArgs a;
    std::memset(&a, 0, sizeof(a));
    a.src = y.dpre;
    a.src_image = (int64_t)y.Ho * y.Wo;
    a.src_group = batch * a.src_image;
    a.groups = y.og;
    a.batch = batch;
    a.H = a.Ho = y.Ho;
    a.W = a.Wo = y.Wo;
    a.stride = 1;
    a.N = y.cu + y.cs;
    a.w = y.wd;
    a.err = n->err;
    RouteArgs& ra = a.route;
    ra.cu = y.cu;
    ra.up = y.up;
    ra.dsrc1 = n->L[y.src1].dy;
    ra.acc1 = written[y.src1] ? 1 : 0;
    written[y.src1] = true;
    if (y.src2 >= 0) {
      ra.dsrc2 = n->L[y.src2].dy;
      ra.acc2 = written[y.src2] ? 1 : 0;
      written[y.src2] = true;
    }
    plan_conv(&a, 1, 0);
    if ((e = launch_conv(a, kConvRoute, n->sms, st)) != cudaSuccess) return e;
  }

  FinishArgs f;
  std::memset(&f, 0, sizeof(f));
  f.count = kNumLayers;
  f.batch = batch;
  f.film_stride = n->F;
  f.dfilm = n->dr;
  for (int l = 0; l < kNumLayers; ++l) {
    const Layer& y = n->L[l];
    const WgradArgs& a = n->wg[l];
    FinishSeg& g = f.seg[l];
    g.cout = y.cout;
    g.kin = y.kin;
    g.gc = a.gc;
    g.s2 = a.s2;
    g.chunks = a.chunks;
    g.ochunks = a.ochunks;
    g.cols = a.cols;
    g.mrows = a.mrows;
    g.splits = a.splits;
    g.sum_chunks = sum_chunks[l];
    g.film_off = y.film_off;
    for (int k = 0; k < 6; ++k) g.col[k] = a.e[k].col;
    g.start = f.total;
    f.total += (int64_t)y.cout * y.kin;
    g.part = y.part;
    g.sums = y.sums;
    g.grad = n->grads + y.w_off;
    g.dbias = n->grads + y.b_off;
  }
  if ((e = launch_finish(f, st)) != cudaSuccess) return e;
  const MlpArgs ma = mlp_args(n, batch, nullptr);
  float* gW1 = n->grads + n->mlp_off;
  float* gb1 = gW1 + 3 * n->cfg.hidden;
  float* gW2 = gb1 + n->cfg.hidden;
  float* gb2 = gW2 + (int64_t)n->F * n->cfg.hidden;
  return launch_mlp_backward(ma, n->dr, gW1, gb1, gW2, gb2, st);
}

int check_call(mclbm_net* n, int batch) {
  if (!n) return MCLBM_EINVAL;
  if (!n->bound) return fail(n, MCLBM_ESTATE, "mclbm_net: not bound");
  if (batch < 1 || batch > n->cfg.max_batch)
    return fail(n, MCLBM_EINVAL, "batch %d outside 1..%d", batch, n->cfg.max_batch);
  return MCLBM_OK;
}

// Syncs the stream and reads the error word and the loss.
int finish(mclbm_net* n, double* loss) {
  int err = 0;
  cudaError_t e = cudaMemcpyAsync(&err, n->err, sizeof(int), cudaMemcpyDeviceToHost, n->stream);
  double l = 0.0;
  if (e == cudaSuccess && loss)
    e = cudaMemcpyAsync(&l, n->loss, sizeof(double), cudaMemcpyDeviceToHost, n->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
  if (e != cudaSuccess) return cuda_fail(n, e, "mclbm_net sync");
  if (err) return fail(n, MCLBM_ETIMEOUT, "a tensor-core kernel gave up a bounded wait");
  if (loss) {
    *loss = l;
    if (!std::isfinite(l)) return fail(n, MCLBM_EDIVERGED, "loss is not finite");
  }
  return MCLBM_OK;
}

}  // namespace

extern "C" {

void mclbm_net_config_default(mclbm_net_config* cfg) {
  if (!cfg) return;
  cfg->ny = 256;
  cfg->nx = 256;
  cfg->c0 = 16;
  cfg->hidden = 64;
  cfg->max_batch = 16;
}

int64_t mclbm_net_param_count(const mclbm_net_config* cfg) {
  if (!config_valid(cfg)) return 0;
  mclbm_net n;
  n.cfg = *cfg;
  plan(&n);
  return n.n_params;
}

size_t mclbm_net_workspace_bytes(const mclbm_net_config* cfg) {
  if (!config_valid(cfg)) return 0;
  mclbm_net n;
  n.cfg = *cfg;
  plan(&n);
  return n.ws_bytes;
}

int mclbm_net_create(const mclbm_net_config* cfg, mclbm_net_t** out) {
  if (!out) return MCLBM_EINVAL;
  *out = nullptr;
  if (!config_valid(cfg)) return MCLBM_EINVAL;
  mclbm_net* n = new mclbm_net();
  n->cfg = *cfg;
  plan(n);
  *out = n;
  return MCLBM_OK;
}

void mclbm_net_destroy(mclbm_net_t* net) { delete net; }

const char* mclbm_net_last_error(const mclbm_net_t* net) { return net ? net->errmsg : ""; }

int mclbm_net_bind(mclbm_net_t* n, void* ws, size_t bytes, void* stream) {
  if (!n) return MCLBM_EINVAL;
  if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u))
    return fail(n, MCLBM_EINVAL, "workspace must be 256-byte aligned");
  if (bytes < n->ws_bytes)
    return fail(n, MCLBM_EINVAL, "workspace of %zu bytes, %zu needed", bytes, n->ws_bytes);
  n->ws = static_cast<char*>(ws);
  n->stream = static_cast<cudaStream_t>(stream);
  assign(n);
  cudaStream_t st = n->stream;
  const size_t np = (size_t)n->n_params * 4;
  cudaError_t e = cudaMemsetAsync(n->params, 0, np, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(n->adam_m, 0, np, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(n->adam_v, 0, np, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(n->err, 0, sizeof(int), st);
  float norm[2 * kFields];
  for (int c = 0; c < kFields; ++c) {
    norm[c] = 0.f;
    norm[kFields + c] = 1.f;
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(n->norm, norm, sizeof(norm), cudaMemcpyHostToDevice, st);
  // the geometry input stays as it is for the handle's life
  int dev = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&n->sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = prepare_conv_kernels();
  if (e == cudaSuccess) e = launch_geometry(n->L[0].in, n->cfg.ny, n->cfg.nx, st);
  if (e == cudaSuccess) e = refresh_bf16_weights(n);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(n, e, "mclbm_net_bind");
  n->adam_t = 0;
  n->bound = true;
  return MCLBM_OK;
}

int mclbm_net_set_params(mclbm_net_t* n, const float* p) {
  if (!n || !p) return MCLBM_EINVAL;
  if (!n->bound) return fail(n, MCLBM_ESTATE, "mclbm_net: not bound");
  const size_t np = (size_t)n->n_params * 4;
  cudaError_t e = cudaMemcpyAsync(n->params, p, np, cudaMemcpyDeviceToDevice, n->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(n->adam_m, 0, np, n->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(n->adam_v, 0, np, n->stream);
  if (e == cudaSuccess) e = refresh_bf16_weights(n);
  if (e != cudaSuccess) return cuda_fail(n, e, "mclbm_net_set_params");
  n->adam_t = 0;
  return MCLBM_OK;
}

int mclbm_net_init_params(mclbm_net_t* n, uint64_t seed) {
  if (!n) return MCLBM_EINVAL;
  if (!n->bound) return fail(n, MCLBM_ESTATE, "mclbm_net: not bound");
  cudaStream_t st = n->stream;
  cudaError_t e = cudaMemsetAsync(n->params, 0, (size_t)n->n_params * 4, st);
  uint32_t stream_id = 0;
  for (int l = 0; l < kNumLayers && e == cudaSuccess; ++l) {
    const Layer& y = n->L[l];
    e = launch_uniform_fill(n->params + y.w_off, (int64_t)y.cout * y.kin,
                            (float)std::sqrt(6.0 / y.kin), seed, stream_id++, st);
  }
  const int H = n->cfg.hidden;
  float* W1 = n->params + n->mlp_off;
  float* W2 = W1 + 3 * H + H;
  if (e == cudaSuccess)
    e = launch_uniform_fill(W1, 3 * H, (float)std::sqrt(6.0 / 3.0), seed, stream_id++, st);
  if (e == cudaSuccess)
    e = launch_uniform_fill(W2, (int64_t)n->F * H, (float)(0.1 * std::sqrt(6.0 / H)), seed,
                            stream_id++, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(n->adam_m, 0, (size_t)n->n_params * 4, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(n->adam_v, 0, (size_t)n->n_params * 4, st);
  if (e == cudaSuccess) e = refresh_bf16_weights(n);
  if (e != cudaSuccess) return cuda_fail(n, e, "mclbm_net_init_params");
  n->adam_t = 0;
  return MCLBM_OK;
}

int mclbm_net_get_params(mclbm_net_t* n, float* p) {
  if (!n || !p) return MCLBM_EINVAL;
  if (!n->bound) return fail(n, MCLBM_ESTATE, "mclbm_net: not bound");
  cudaError_t e = cudaMemcpyAsync(p, n->params, (size_t)n->n_params * 4, cudaMemcpyDeviceToDevice,
                                  n->stream);
  return e == cudaSuccess ? MCLBM_OK : cuda_fail(n, e, "mclbm_net_get_params");
}

int mclbm_net_set_normalizer(mclbm_net_t* n, const double* mean, const double* scale) {
  if (!n || !mean || !scale) return MCLBM_EINVAL;
  if (!n->bound) return fail(n, MCLBM_ESTATE, "mclbm_net: not bound");
  float v[2 * kFields];
  for (int c = 0; c < kFields; ++c) {
    if (!(scale[c] > 0.0) || !std::isfinite(mean[c]) || !std::isfinite(scale[c]))
      return fail(n, MCLBM_EINVAL, "normaliser channel %d: mean %g scale %g", c, mean[c], scale[c]);
    v[c] = (float)mean[c];
    v[kFields + c] = (float)scale[c];
  }
  // the host array must outlive the copy: synchronous on the stream
  cudaError_t e = cudaMemcpyAsync(n->norm, v, sizeof(v), cudaMemcpyHostToDevice, n->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
  return e == cudaSuccess ? MCLBM_OK : cuda_fail(n, e, "mclbm_net_set_normalizer");
}

int mclbm_net_field_stats(mclbm_net_t* n, int count, const float* cond, const float* fields,
                          double* mean, double* scale) {
  if (!n || !cond || !fields || !mean || !scale || count < 1) return MCLBM_EINVAL;
  if (!n->bound) return fail(n, MCLBM_ESTATE, "mclbm_net: not bound");
  const int hw = n->cfg.ny * n->cfg.nx;
  cudaError_t e =
      launch_field_moments(fields, cond, count, hw, n->stat_part, kStatBlocks, n->stream);
  std::vector<double> part(kFields * kStatBlocks * 2);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(part.data(), n->stat_part, part.size() * 8, cudaMemcpyDeviceToHost,
                        n->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
  if (e != cudaSuccess) return cuda_fail(n, e, "mclbm_net_field_stats");
  const double N = (double)count * hw;
  for (int c = 0; c < kFields; ++c) {
    double s = 0.0, s2 = 0.0;
    for (int b = 0; b < kStatBlocks; ++b) {
      s += part[(c * kStatBlocks + b) * 2];
      s2 += part[(c * kStatBlocks + b) * 2 + 1];
    }
    const double m = s / N;
    const double var = std::max(0.0, s2 / N - m * m);
    mean[c] = m;
    scale[c] = var > 0.0 ? std::sqrt(var) : 1.0;
  }
  return MCLBM_OK;
}

int mclbm_net_forward(mclbm_net_t* n, int batch, const float* cond, float* fields) {
  mcl::NvtxRange range("mclbm_net_forward");
  int rc = check_call(n, batch);
  if (rc != MCLBM_OK) return rc;
  if (!cond || !fields) return fail(n, MCLBM_EINVAL, "null pointer");
  cudaError_t e = forward(n, batch, cond, false);
  if (e == cudaSuccess)
    e = launch_denormalize(n->L[kNumLayers - 1].pre, n->norm, cond, batch,
                           n->cfg.ny * n->cfg.nx, n->stat_part, fields, n->stream);
  return e == cudaSuccess ? MCLBM_OK : cuda_fail(n, e, "mclbm_net_forward");
}

int mclbm_net_loss_grad(mclbm_net_t* n, int batch, const float* cond, const float* target,
                        float* grad, double* loss) {
  mcl::NvtxRange range("mclbm_net_loss_grad");
  int rc = check_call(n, batch);
  if (rc != MCLBM_OK) return rc;
  if (!cond || !target || !grad || !loss) return fail(n, MCLBM_EINVAL, "null pointer");
  cudaError_t e = forward(n, batch, cond, true);
  if (e == cudaSuccess) e = loss_backward(n, batch, cond, target);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(grad, n->grads, (size_t)n->n_params * 4, cudaMemcpyDeviceToDevice,
                        n->stream);
  if (e != cudaSuccess) return cuda_fail(n, e, "mclbm_net_loss_grad");
  return finish(n, loss);
}

int mclbm_net_train_step(mclbm_net_t* n, int batch, const float* cond, const float* target,
                         float lr, double* loss) {
  mcl::NvtxRange range("mclbm_net_train_step");
  int rc = check_call(n, batch);
  if (rc != MCLBM_OK) return rc;
  if (!cond || !target || !(lr > 0.f)) return fail(n, MCLBM_EINVAL, "bad argument");
  cudaError_t e = forward(n, batch, cond, true);
  if (e == cudaSuccess) e = loss_backward(n, batch, cond, target);
  if (e == cudaSuccess) {
    n->adam_t += 1;
    const double b1 = 0.9, b2 = 0.999;
    const float c1 = (float)(1.0 / (1.0 - std::pow(b1, n->adam_t)));
    const float c2 = (float)(1.0 / (1.0 - std::pow(b2, n->adam_t)));
    e = launch_adam(n->params, n->grads, n->adam_m, n->adam_v, n->n_params, lr, (float)b1,
                    (float)b2, 1e-8f, c1, c2, n->stream);
  }
  if (e == cudaSuccess) e = refresh_bf16_weights(n);
  if (e != cudaSuccess) return cuda_fail(n, e, "mclbm_net_train_step");
  return loss ? finish(n, loss) : MCLBM_OK;
}

int mclbm_gemm_bf16(int M, int N, int K, const void* a, int64_t lda, int a_kmajor, const void* b,
                    int64_t ldb, int b_kmajor, float* d, int64_t ldd, int splits,
                    int64_t k_per_split, int64_t split_stride, void* stream) {
  GemmArgs g;
  std::memset(&g, 0, sizeof(g));
  g.a = static_cast<const __nv_bfloat16*>(a);
  g.lda = lda;
  g.a_kmajor = a_kmajor ? 1 : 0;
  g.b = static_cast<const __nv_bfloat16*>(b);
  g.ldb = ldb;
  g.b_kmajor = b_kmajor ? 1 : 0;
  g.M = M;
  g.N = N;
  g.K = K;
  g.k_per_split = k_per_split;
  g.d = d;
  g.ldd = ldd;
  g.split_stride = split_stride;
  g.err = nullptr;
  if (!gemm_args_valid(g, splits)) return MCLBM_EINVAL;
  return launch_gemm(g, splits, static_cast<cudaStream_t>(stream)) == cudaSuccess ? MCLBM_OK
                                                                                   : MCLBM_ECUDA;
}

}  // extern "C"
