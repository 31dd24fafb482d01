// Internal interfaces of the warm-start network (include/mclbm_net.h): its convolutions
// (net_conv.cu), the CUDA-core kernels around them (net_kernels.cu) and the exposed tensor-core
// GEMM (net_gemm.cu). Host code in net_abi.cu.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace mcl {
namespace net {

// Predicted fields: u_x, u_y, theta, phi, rho^w. Channels 3 and 4 are learned as deviations from
// the sample's rest values phi_0 and 1 - phi_0 (base_fields).
constexpr int kFields = 5;

struct GemmArgs {
  const __nv_bfloat16* a;
  int64_t lda;
  int a_kmajor;
  int a_vec;  // set by launch_gemm: 16-byte loads of A
  const __nv_bfloat16* b;
  int64_t ldb;
  int b_kmajor;
  int b_vec;
  int M, N, K;
  int64_t k_per_split;  // multiple of 64
  float* d;
  int64_t ldd, split_stride;
  int d_vec;  // set by launch_gemm: 16-byte stores of D
  int* err;  // bit 0 set when a bounded wait gave up (may be null)
  int splits;  // set by launch_gemm: K splits (tiles of D are m x n x split)
};

// Checks the operand requirements and launches a persistent grid over the tiles of D and the K
// splits: 256 x 256 tiles by pairs of CTAs where that pays (pair_pays), else 128 x 128.
cudaError_t launch_gemm(const GemmArgs& g, int splits, cudaStream_t st);
// True if the arguments satisfy the alignment and extent rules of launch_gemm.
bool gemm_args_valid(const GemmArgs& g, int splits);

// ---- convolutions (net_conv.cu) -------------------------------------------------------------
// Activations and pre-activation gradients: BF16 [groups of 8 channels][batch * H * W][8], zero in
// the channels that pad the last group. A decoder layer's input holds the upsampled source's
// groups, then the skip source's, written there by the layers that produce them. Pixel counts
// (src_group, y_group, ...) are in units of such 16-byte pixels.

// Forward epilogue: pre[o][p] = D(p, o) + bias[o] (pre may be null);
// z = film ? (1 + film[b][foff + o]) pre + film[b][foff + C + o] : pre;
// y = act ? silu(z) : z, rounded to BF16 into the consumer's input (y may be null), each pixel
// four times with up (nearest upsampling by 2).
struct ConvEpilogue {
  const float* bias;
  const float* film;  // [batch][film_stride] or null
  int film_stride, film_off;
  float* pre;
  __nv_bfloat16* y;
  int64_t y_group;
  int up, act;
};

// Gradient of a convolution's input, channel c of N: channels [0, cu) to dsrc1 [cu][batch * Hs *
// Ws] (summed over each 2 x 2 block, in row order, when that source was upsampled by 2), the rest
// to dsrc2 [N - cu][batch * H * W]; each written (acc = 0) or added to (acc = 1).
struct RouteArgs {
  int cu, up;
  float* dsrc1;
  float* dsrc2;
  int acc1, acc2;
};

enum ConvMode : int { kConvForward, kConvPartial, kConvRoute };
constexpr int kConvMaxStages = 5;

// n / d by a multiplication, for n < 2^31 (Granlund and Montgomery, PLDI 1994).
struct FastDiv {
  uint32_t d = 1, mul = 1, shift = 0;
  FastDiv() = default;
  explicit FastDiv(int div) : d((uint32_t)div) {
    while ((1ull << shift) < d) ++shift;
    mul = (uint32_t)(((1ull << 32) * ((1ull << shift) - d)) / d + 1);
  }
#ifdef __CUDACC__
  __device__ __forceinline__ int div(int n) const {
    return (int)((__umulhi((uint32_t)n, mul) + (uint32_t)n) >> shift);
  }
#endif
};

// A 3 x 3 convolution with zero padding of src (its K order is channel, then tap), D [pixels][N].
struct ConvArgs {
  const __nv_bfloat16* src;
  int64_t src_group, src_image;  // pixels between groups and between images
  int groups, batch, H, W, stride, Ho, Wo, N;
  const __nv_bfloat16* w;  // packed (PackSeg)
  ConvEpilogue ep;         // kConvForward
  float* part;             // kConvPartial: [split][N][batch * Ho * Wo]
  RouteArgs route;         // kConvRoute
  int* err;
  // set by plan_conv
  int nt, n_tiles, slices, steps, split_steps, tiles_x, tiles_y, items, tmem_cols, stages;
  FastDiv by_tiles, by_image, by_row, by_n;  // item -> K split, channel tile, image, tile row
};
int conv_n_tile(int n);       // output channels per tile, padded to 16
int conv_slices(int groups);  // K slices of 16 channels
// splits > 1: K cut into ranges of split_k (a multiple of 16).
void plan_conv(ConvArgs* a, int splits, int split_k);
cudaError_t launch_conv(const ConvArgs& a, int mode, int sms, cudaStream_t st);

// Input gradient of a stride-2 convolution, dsrc [C][batch * 2 Ho * 2 Wo] FP32 (written or added
// to), from the tensor map of its dpre (encode_groups with boxes of 9 pixels x kg groups x 17 rows).
constexpr int kDxStages = 2;
struct DxStride2Args {
  int batch, Ho, Wo, C;
  const __nv_bfloat16* w;
  float* dsrc;
  int accumulate;
  int* err;
  // set by plan_dx_stride2
  int kg, kchunks, chunks, tiles_x, tiles_y, a_bytes, w_bytes, stage_bytes;
};
int dx_stride2_kg(int cout);
void plan_dx_stride2(DxStride2Args* a, int cout);
cudaError_t launch_dx_stride2(const CUtensorMap& map, const DxStride2Args& a, int sms,
                              cudaStream_t st);

// Weight gradient: partial sums part [split][chunk][o chunk][cols][mrows] of the products of dpre
// (maps.a) and the layer's input (maps.b[0], or its four parity maps for stride 2).
constexpr int kWgMaxStages = 8;
struct WgradMaps {
  CUtensorMap a, b[4];
};
struct WgradEntry {
  int off, n, col;  // byte offset in the staged patch, columns of the MMA, first column
};
struct WgradArgs {
  int src_images;  // 0: one image for every sample
  float* part;
  int* err;
  // set by plan_wgrad
  int s2, go, ochunks, mrows, gc, chunks, cols, tiles_x, tiles_y, batch, splits, split_tiles;
  int a_bytes, b_group, b_row, patch_bytes, tx_bytes, stage_bytes, stages, tmem_cols;
  int parts, entries;  // CTAs per (split, chunks), entries of each
  WgradEntry e[6];
};
void plan_wgrad(WgradArgs* a, int cin_groups, int cout, int kin, int Ho, int Wo, int batch,
                int stride, int sms);
size_t wgrad_part_bound(int cin_groups, int cout, int kin, int stride);
cudaError_t launch_wgrad(const WgradMaps& maps, const WgradArgs& a, cudaStream_t st);

// Tensor maps over a grouped tensor (false if the driver refuses).
bool encode_groups(CUtensorMap* map, const __nv_bfloat16* x, int groups, int64_t group_pixels,
                   int images, int H, int W, int box_px, int box_groups, int box_rows);
bool encode_parity(CUtensorMap* map, const __nv_bfloat16* x, int py, int px, int groups,
                   int64_t group_pixels, int images, int H, int W, int box_px, int box_groups,
                   int box_rows);

// The layers' FP32 weights W [cout][cin][3][3] as BF16 operands: forward (n = o, k = c 9 + tap),
// transposed (n = c, k = o 9 + tap of the flipped kernel) and stride 2 (n = c, k = o per tap).
constexpr int kMaxSegs = 24;
enum PackKind : int { kPackForward, kPackTransposed, kPackStride2 };
struct PackSeg {
  int kind, cout, cin, nt, slices, kg;
  int64_t w_off, start;
  __nv_bfloat16* out;
};
struct PackArgs {
  const float* params;
  int count;
  int64_t total;
  PackSeg seg[kMaxSegs];
};
cudaError_t launch_pack_weights(const PackArgs& a, cudaStream_t st);

// Every layer's partial sums to its gradients: weights (WgradArgs::part), biases and FiLM (sums
// [cout][batch][sum_chunks][3] of launch_act_backward and launch_loss).
struct FinishSeg {
  int cout, kin, gc, s2, chunks, ochunks, cols, mrows, splits, sum_chunks, film_off;
  int col[6];
  int64_t start;
  const float* part;
  const double* sums;
  float *grad, *dbias;
};
struct FinishArgs {
  int count, batch, film_stride, w_blocks;
  int64_t total;
  float* dfilm;
  FinishSeg seg[10];
};
cudaError_t launch_finish(FinishArgs a, cudaStream_t st);

// Shared-memory limits of the kernels above on the current device.
cudaError_t prepare_conv_kernels();

// ---- CUDA-core kernels (net_kernels.cu) ---------------------------------------------------
// Backward of act(film(pre)) for one layer: dpre (BF16 groups) and, per (o, b) and pixel chunk,
// the sums {sum dpre, sum dz pre, sum dz} (compensated FP32 per block, FP64 across its warps).
struct ActBwdArgs {
  const float* dy;    // [C][P]
  const float* pre;   // [C][P]
  const float* film;  // [batch][film_stride] or null
  int film_stride, film_off;
  int C, batch, hw, chunks;
  __nv_bfloat16* dpre;
  double* sums;  // [C][batch][chunks][3]
};
// Pixel chunks of a layer with C channels: enough blocks for the device, a thousand pixels each.
int act_chunks(int C, int batch, int hw);
cudaError_t launch_act_backward(const ActBwdArgs& a, cudaStream_t st);

// The convolution epilogue after a K-split forward convolution: part [splits][N][P] summed over
// the splits in order, then as ConvEpilogue.
cudaError_t launch_conv_epilogue_splitk(const float* part, int splits, int batch, int Ho, int Wo,
                                        int N, const ConvEpilogue& e, cudaStream_t st);

// Conditioning MLP. cond_raw [batch][3] (Ra, phi, d_p) -> c [batch][3], a1 [batch][H],
// r [batch][F].
struct MlpArgs {
  const float* cond_raw;
  const float* W1;
  const float* b1;
  const float* W2;
  const float* b2;
  int batch, H, F;
  float* c;
  float* a1;
  float* r;
};
cudaError_t launch_mlp_forward(const MlpArgs& a, cudaStream_t st);
// Given dr [batch][F]: gradients of W1, b1, W2, b2 (written, not accumulated).
cudaError_t launch_mlp_backward(const MlpArgs& a, const float* dr, float* gW1, float* gb1,
                                float* gW2, float* gb2, cudaStream_t st);

// Loss against target fields [batch][5][hw]: dpre [batch * hw][8] = BF16 of 2 (out - t) / n,
// t = (F - base - mean) / scale (the output layer has no activation), its sums per (channel,
// sample, chunk) as launch_act_backward leaves them, and per-block FP64 sums of (out - t)^2 / n in
// partial [batch * chunks].
struct LossArgs {
  const float* out;     // [5][batch * hw]
  const float* target;  // [batch][5][hw]
  const float* cond;    // [batch][3] raw (Ra, phi, d_p): the base of channels 3 and 4
  const float* norm;    // mean[5], scale[5]
  int batch, hw, chunks;
  __nv_bfloat16* dpre;
  double* sums;
  double* partial;
};
cudaError_t launch_loss(const LossArgs& a, cudaStream_t st);
// out[0] = sum of partial[0..n) in a fixed order.
cudaError_t launch_sum_partials(const double* partial, int n, double* out, cudaStream_t st);

// Adam over n parameters; c1 = 1/(1 - b1^t), c2 = 1/(1 - b2^t).
cudaError_t launch_adam(float* p, const float* g, float* m, float* v, int64_t n, float lr,
                        float b1, float b2, float eps, float c1, float c2, cudaStream_t st);

// p[i] = scale * u_i, u_i uniform in [-1, 1) (splitmix64 of seed, stream and i).
cudaError_t launch_uniform_fill(float* p, int64_t n, float scale, uint64_t seed, uint32_t stream,
                                cudaStream_t st);
// Geometry input, one image [ny * nx][8] BF16 (channels 4 to 7 zero).
cudaError_t launch_geometry(__nv_bfloat16* X, int ny, int nx, cudaStream_t st);
// fields[b][ch][i] = base[b][ch] + mean[ch] + scale[ch] * out[ch][b*hw + i]; phi (ch 3) and
// rho^w (ch 4) are then shifted so that their means are phi_0 = cond[b][1] and 1 - phi_0.
// partial: kShiftPartials doubles of scratch (batch <= 256: at least five chunks per sample).
constexpr int kShiftPartials = 2560;
cudaError_t launch_denormalize(const float* out, const float* norm, const float* cond, int batch,
                               int hw, double* partial, float* fields, cudaStream_t st);
// Per-channel FP64 sum and sum of squares of fields - base, fields [n][5][hw], cond [n][3], into
// partial[5][blocks][2].
cudaError_t launch_field_moments(const float* fields, const float* cond, int n, int hw,
                                 double* partial, int blocks, cudaStream_t st);

}  // namespace net
}  // namespace mcl
