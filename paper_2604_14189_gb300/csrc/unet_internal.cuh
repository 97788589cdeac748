// Internal interfaces of the learned gradient preconditioner (a U-Net run
// in BF16 with FP32 accumulation): the tcgen05 convolution kernels
// (unet_conv.cu), the element-wise and reduction kernels (unet_ops.cu) and
// the network driver (unet_api.cu).
//
// Tensors are NHWC BF16: element (b, y, x, c) of a view with pixel stride
// ps (channels of the underlying buffer; a view may start at a channel
// offset, e.g. one half of a concatenation buffer) sits at
// base[((b H + y) W + x) ps + c].
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace sweep {

typedef __nv_bfloat16 bf16;

// One 3 x 3 convolution as an implicit GEMM on the tensor cores:
//   out[p][n] = op( sum_{tap, k} in[p + off(tap)][k] * w[n][tap][k] + bias[n] )
// over tiles of 16 x 8 ns pixels (M = 128 pixels each, N = n output channels,
// K = 9 taps x input channels in chunks of kc).  The data gradient of a
// convolution is the same operation on the output gradient with the
// weights transposed and mirrored (w'[ci][8 - tap][co] = w[co][tap][ci]).
enum ConvOp { kOpNone = 0, kOpRelu = 1, kOpMask = 2 };
struct ConvArgs {
  CUtensorMap tin;   // input view {cin, W, H, B}, box {kc, 8 ns + 2, 18, 1}
  CUtensorMap tw;    // weights {cin, 9, cout}, box {kc, 1, n}
  int B, H, W;
  int cin, cout, kc;  // kc = 64 (128-byte swizzle of the weights) or 32 (64-byte)
  int n, ns;          // a CTA's output channels and 8-pixel column groups
  int stages;         // of the ring
  int stays;          // the input tile is staged once (else once per tap)
  int late;           // reads and overwrites nothing of the kernel launched before: runs
                      // beside it, and only its end waits for it
  const float* bias;  // [cout] or NULL
  int op;             // ConvOp
  const bf16* in;
  int in_ps;
  const bf16* mask;   // kOpMask: out *= (mask > 0), same pixel/channel
  int mask_ps;
  bf16* out;
  int out_ps;
  bf16* pool;         // [B][H/2][W/2][cout] 2 x 2 averages of the output, or NULL
  bf16* up;           // [B][2H][2W][cout] its nearest upsampling, or NULL
  const float* head;  // cout = 32: weights and bias of the 1 x 1 head, or NULL
  float* head_out;    // [B][H][W]
  int* status;        // latched on a wait that gives up
  // what the launcher makes the maps from once it has chosen n and ns
  const bf16* w;
  bool (*make_maps)(ConvArgs&);
};

// Weight gradient of one 3 x 3 convolution on the tensor cores:
//   D[(tap, ci)][co] = sum over pixels p of in[p + off(tap)][ci] dy[p][co]
// (both operands MN-major, K = 16 pixels of a row per MMA).  The pixels are
// taken in raster order, in strips of 64, and split into equal ranges; a range
// is one accumulation, and the ranges' sums are added in a fixed order, so the
// split is part of the result.  Within a split the work is cut by taps: a unit
// is one accumulator of 128 rows made of 128 / kc runs of kc channels, of up to
// cpb = 128 / kc channel chunks (a block):
//   several chunks (9 units): unit = tap, run j = chunk j;
//   one chunk of 64 (5 units): two taps: a pixel apart (kx = 0, 1) or a row
//   apart (kx = 2);
//   one chunk of 32 (3 units): unit = ky, runs a pixel apart (kx = 0, 1, 2).
// A CTA does one unit of one split.  (Several units that share a staged row load
// less but leave SMs idle: 8 x 256 x 256, 32 -> 32 channels 43 us for 33, 64 -> 32
// 103 for 56; other layers within 10 %.)
constexpr int kWgPix = 64;  // pixels of a strip
struct WgradPlan {
  int kc, nchunks, cpb, blocks;  // input channels
  int kb;                        // output channels per staged box
  int pw, ph, q;                 // columns and rows of a strip, strips of a stage
  int units, splits;             // units of all blocks
  int ring;      // bytes of a CTA's stages
  size_t smem;
};
__host__ __device__ inline int wgrad_chunks(const WgradPlan& P, int block) {
  const int n = P.nchunks - block * P.cpb;
  return n < P.cpb ? n : P.cpb;
}
__host__ __device__ inline int wgrad_units(const WgradPlan& P, int block) {
  return wgrad_chunks(P, block) > 1 ? 9 : P.kc == 64 ? 5 : 3;
}
// Block of unit i of all, whose number in it is *u.
__host__ __device__ inline int wgrad_block(const WgradPlan& P, int i, int* u) {
  const int f = wgrad_units(P, 0);  // every block but the last has as many as the first
  const int block = i / f < P.blocks - 1 ? i / f : P.blocks - 1;
  *u = i - block * f;
  return block;
}
// Tap of a unit's run 0, and whether run 1 is the tap a row below (else it is
// the next pixel's or, with several chunks, the next chunk's).
struct WgradUnit {
  int ky, kx, down;
};
__host__ __device__ inline WgradUnit wgrad_unit(const WgradPlan& P, int chunks, int u) {
  if (chunks > 1) return {u / 3, u % 3, 0};
  if (P.kc == 32) return {u, 0, 0};
  return {u < 2 ? 0 : u == 2 ? 1 : 2, u == 1 || u == 4 ? 2 : 0, u == 1};
}
// Row m of a unit: its tap and input channel; false: unused.
__host__ __device__ inline bool wgrad_row(const WgradPlan& P, int block, int u, int m, int* tap,
                                          int* ci) {
  const int chunks = wgrad_chunks(P, block), j = m / P.kc;
  const WgradUnit n = wgrad_unit(P, chunks, u);
  *ci = block * P.cpb * P.kc + m % P.kc;
  *tap = 3 * n.ky + n.kx;
  if (chunks > 1) {
    *ci += j * P.kc;
    return j < chunks;
  }
  *tap += n.down ? 3 * j : j;
  return n.down ? j < 2 : n.kx + j < 3 && (P.kc == 32 || j < 2);
}
struct WgradArgs {
  CUtensorMap tin;   // input view {cin, W, H, B}, box {kc, q pw + 2, ph, 1}
  CUtensorMap tdy;   // output-gradient view {cout, W, H, B}, box {kb, q pw, ph, 1}
  WgradPlan plan;
  int B, H, W;
  int cin, cout;
  float* partial;    // [split][unit][cout][128]
  int* status;
};

int launch_conv(ConvArgs a, cudaStream_t st);  // chooses n, ns, stages; SWEEP_OK or an error
WgradPlan wgrad_plan(int B, int H, int W, int cin, int cout, size_t* partial);
void launch_wgrad(const WgradArgs& a, cudaStream_t st);

// ---- element-wise and reduction kernels (unet_ops.cu)
struct WeightPrep {  // one 3 x 3 layer of the flat parameter vector
  long long off;     // W[cout][3][3][cin] in the flat FP32 vector
  int cin, cout;
  bf16* w;           // out [cout][9][cin]
  bf16* wt;          // out [cin][9][cout], taps mirrored (data gradient), or NULL
};
constexpr int kUnetLayers = 17;
struct WeightPrepAll {
  WeightPrep l[kUnetLayers];
};
void launch_prep_weights(const float* theta, const WeightPrepAll& p, long long total_w,
                         cudaStream_t st);
void launch_pack_input(const float* in, int in_ch, bf16* x0, long long npix, cudaStream_t st);
// d[p][c] = bf16( (sum over the 2 x 2 children of p of g[child][c]) * (x[p][c] > 0) )
void launch_up_backward_mask(const bf16* g, int g_ps, const bf16* x, bf16* d, int B, int h,
                             int w, int C, cudaStream_t st);
// d[p][c] = bf16( 0.25 gp[parent(p)][c] * (s[p][c] > 0) + gskip[p][c] )
void launch_pool_backward_combine(const bf16* gp, const bf16* s, int s_ps, const bf16* gskip,
                                  int gskip_ps, bf16* d, int B, int H, int W, int C,
                                  cudaStream_t st);
// loss = mean (out - t)^2 (FP64); dout = 2 (out - t) / N;
// dpre[p][c] = bf16(dout[p] wh[c] (x[p][c] > 0)); head gradients
void launch_head_backward(const bf16* x, const float* theta_head, const float* out,
                          const float* target, long long npix, bf16* dpre, double* partial,
                          int nblocks, double* loss, float* grad_head, cudaStream_t st);
// partial[block][co] = sum over the block's pixels of dy[p][co]
void launch_bias_grad(const bf16* dy, int dy_ps, int cout, long long npix, float* partial,
                      int nblocks, cudaStream_t st);
// dW[co][tap][ci] from a.partial and db[co] (or NULL) from the nb partials bpart
void launch_wgrad_reduce(const WgradArgs& a, float* dW, const float* bpart, int nb, float* db,
                         cudaStream_t st);
void launch_adam(float* theta, const float* grad, float* m, float* v, long long n, int step,
                 float lr, float b1, float b2, float eps, cudaStream_t st);

}  // namespace sweep
