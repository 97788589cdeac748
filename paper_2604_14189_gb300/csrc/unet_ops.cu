// Element-wise and reduction kernels of the U-Net preconditioner: weight
// conversion to BF16 (and the mirrored transpose the data gradient uses), input
// packing, the backward passes of the 2 x 2 average pooling, of the nearest 2x
// upsampling (both with the ReLU masks) and of the 1 x 1 head with the MSE loss
// (forward, these three are part of the convolution before them,
// unet_conv.cu), bias and weight-gradient reductions, and the Adam update.
//
// BF16 tensors are NHWC with channel counts that are multiples of 8, so a
// thread moves 8 channels (16 bytes) at a time.  Reductions are FP32 (FP64
// for the loss) with partial sums in a fixed order: the same inputs give the
// same bits.
//
// Every kernel of the network is launched as a dependent of the one before it
// (grid_dep_wait, sweep_internal.cuh): its launch, set-up and, in a
// convolution, first weights overlap that kernel's tail.  Inference of 1 x 256 x
// 256 takes 162 us and a training step of 8 x 256 x 256 1.32 ms; with plain
// launches, a kernel of its own for each pooling, upsampling and head and one
// shifted tile per tap of a convolution (unet_conv.cu) 370 us and 3.19 ms.
#include "sweep_internal.cuh"
#include "unet_internal.cuh"

namespace sweep {
namespace {

constexpr int kT = 256;

__device__ __forceinline__ void unpack8(const uint4& u, float* f) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 t = __bfloat1622float2(h[i]);
    f[2 * i] = t.x;
    f[2 * i + 1] = t.y;
  }
}

__device__ __forceinline__ uint4 pack8(const float* f) {
  uint4 u;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
  return u;
}

__device__ __forceinline__ uint4 ld8(const bf16* p) { return *reinterpret_cast<const uint4*>(p); }
__device__ __forceinline__ void st8(bf16* p, uint4 v) { *reinterpret_cast<uint4*>(p) = v; }

int blocks_for(long long n, int per_block = kT) {
  long long b = (n + per_block - 1) / per_block;
  return (int)(b < 1 ? 1 : (b > 1048576 ? 1048576 : b));
}

// Block: one (tap, 32 output x 32 input channels) tile of a layer, transposed
// through shared memory so that both copies are written along their rows.  (A
// thread per weight with scattered 2-byte stores took 48 us for the 2.1 M
// weights; now 9.)
__global__ void __launch_bounds__(256) prep_weights_kernel(const float* __restrict__ theta,
                                                           const __grid_constant__ WeightPrepAll p) {
  __shared__ bf16 t[32][33];
  grid_dep_wait();
  grid_dep_trigger();
  int k = blockIdx.x, l = 0;
  while (l < kUnetLayers - 1 && k >= p.l[l].cout / 32 * (p.l[l].cin / 32) * 9) {
    k -= p.l[l].cout / 32 * (p.l[l].cin / 32) * 9;
    ++l;
  }
  const WeightPrep& L = p.l[l];
  const int tap = k % 9, nci = L.cin / 32;
  const int ci0 = k / 9 % nci * 32, co0 = k / 9 / nci * 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int co = 8 * i + w;
    const long long j = ((long long)(co0 + co) * 9 + tap) * L.cin + ci0 + lane;
    const bf16 h = __float2bfloat16_rn(theta[L.off + j]);
    L.w[j] = h;
    t[co][lane] = h;
  }
  if (!L.wt) return;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int ci = 8 * i + w;
    L.wt[((long long)(ci0 + ci) * 9 + (8 - tap)) * L.cout + co0 + lane] = t[lane][ci];
  }
}

__global__ void pack_input_kernel(const float* __restrict__ in, int in_ch, bf16* __restrict__ x0,
                                  long long npix) {
  // runs next to the weight preparation launched before it, of which it needs
  // nothing; only its end waits
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < npix;
       p += (long long)gridDim.x * blockDim.x) {
    float f[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) f[c] = c < in_ch ? in[p * in_ch + c] : 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) st8(x0 + p * 32 + 8 * q, pack8(f + 8 * q));
  }
  grid_dep_wait();
  grid_dep_trigger();
}

template <typename I>
__global__ void up_backward_mask_kernel(const bf16* __restrict__ g, int g_ps,
                                        const bf16* __restrict__ x, bf16* __restrict__ d, int B,
                                        int h, int w, int C) {
  grid_dep_wait();
  grid_dep_trigger();
  const int H = 2 * h, W = 2 * w;
  const I ng = C / 8, n = (I)B * h * w * ng;
  for (I i = (I)blockIdx.x * kT + threadIdx.x; i < n; i += (I)gridDim.x * kT) {
    const int c = (int)(i % ng) * 8;
    I p = i / ng;
    const int xx = (int)(p % w);
    p /= w;
    const int y = (int)(p % h);
    const int b = (int)(p / h);
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int dy = 0; dy < 2; ++dy)
#pragma unroll
      for (int dx = 0; dx < 2; ++dx) {
        float f[8];
        unpack8(ld8(g + (((long long)b * H + 2 * y + dy) * W + 2 * xx + dx) * g_ps + c), f);
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[k] += f[k];
      }
    const long long o = (((long long)b * h + y) * w + xx) * C + c;
    float m[8];
    unpack8(ld8(x + o), m);
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (!(m[k] > 0.f)) acc[k] = 0.f;
    st8(d + o, pack8(acc));
  }
}

template <typename I>
__global__ void pool_backward_combine_kernel(const bf16* __restrict__ gp,
                                             const bf16* __restrict__ s, int s_ps,
                                             const bf16* __restrict__ gskip, int gskip_ps,
                                             bf16* __restrict__ d, int B, int H, int W, int C) {
  grid_dep_wait();
  grid_dep_trigger();
  const I ng = C / 8, n = (I)B * H * W * ng;
  for (I i = (I)blockIdx.x * kT + threadIdx.x; i < n; i += (I)gridDim.x * kT) {
    const int c = (int)(i % ng) * 8;
    const I row = i / ng / W;
    const long long p = (long long)(i / ng);
    const int x = (int)(i / ng - row * W);
    const int y = (int)(row % H);
    const int b = (int)(row / H);
    float a[8], m[8], k2[8];
    unpack8(ld8(gp + (((long long)b * (H / 2) + y / 2) * (W / 2) + x / 2) * C + c), a);
    unpack8(ld8(s + p * s_ps + c), m);
    unpack8(ld8(gskip + p * gskip_ps + c), k2);
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] = (m[k] > 0.f ? 0.25f * a[k] : 0.f) + k2[k];
    st8(d + p * C + c, pack8(a));
  }
}

// Per block: FP64 loss partial, FP32 partials of the 33 head gradients.
__global__ void __launch_bounds__(kT) head_backward_kernel(
    const bf16* __restrict__ x, const float* __restrict__ th, const float* __restrict__ out,
    const float* __restrict__ tgt, long long npix, bf16* __restrict__ dpre,
    double* __restrict__ lpart, float* __restrict__ hpart) {
  __shared__ double sl[kT / 32];
  __shared__ float sh[kT / 32][33];
  grid_dep_wait();
  grid_dep_trigger();
  const float scale = 2.0f / (float)npix;
  double l = 0.0;
  float gw[33];
#pragma unroll
  for (int k = 0; k < 33; ++k) gw[k] = 0.f;
#pragma unroll 2
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < npix;
       p += (long long)gridDim.x * blockDim.x) {
    const float r = out[p] - tgt[p];
    l += (double)r * (double)r;
    const float dout = scale * r;
    gw[32] += dout;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float f[8], o[8];
      unpack8(ld8(x + p * 32 + 8 * q), f);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        gw[8 * q + k] = fmaf(dout, f[k], gw[8 * q + k]);
        o[k] = f[k] > 0.f ? dout * th[8 * q + k] : 0.f;
      }
      st8(dpre + p * 32 + 8 * q, pack8(o));
    }
  }
  // block sums in a fixed order
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 33; ++k) {
    float v = gw[k];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) sh[warp][k] = v;
  }
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if (lane == 0) sl[warp] = l;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < kT / 32; ++i) t += sl[i];
    lpart[blockIdx.x] = t;
  }
  if (threadIdx.x < 33) {
    float t = 0.f;
    for (int w = 0; w < kT / 32; ++w) t += sh[w][threadIdx.x];
    hpart[(long long)blockIdx.x * 33 + threadIdx.x] = t;
  }
}

// The sums of the blocks' partials: the loss by a warp's tree, a head gradient
// in block order, from shared memory (straight from global: 24 us, now 6).
__global__ void __launch_bounds__(kT) head_backward_total_kernel(const double* lpart,
                                                                 const float* hpart, int nb,
                                                                 long long npix, double* loss,
                                                                 float* grad_head) {
  extern __shared__ float sp[];  // [nb][33]
  grid_dep_wait();
  grid_dep_trigger();
  for (int i = threadIdx.x; i < nb * 33; i += kT) sp[i] = hpart[i];
  if (threadIdx.x >= kT - 32 && loss) {
    double t = 0.0;
    for (int i = threadIdx.x & 31; i < nb; i += 32) t += lpart[i];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == kT - 32) *loss = t / (double)npix;
  }
  __syncthreads();
  if (threadIdx.x < 33) {
    float t = 0.f;
#pragma unroll 8
    for (int i = 0; i < nb; ++i) t += sp[i * 33 + threadIdx.x];
    grad_head[threadIdx.x] = t;
  }
}

// partial[block][co] = sum over the block's pixels of dy[p][co]: a thread
// owns 4 channels and every (256 / (cout / 8))-th pixel of the block's range;
// the block then adds its rows in a fixed order.  dy is older than the kernel
// launched before this one (the weight gradient, which leaves room for a block
// per SM), so the two run together; only the end waits for it.
__global__ void __launch_bounds__(512) bias_grad_kernel(const bf16* __restrict__ dy, int ps,
                                                        int cout, long long npix,
                                                        float* __restrict__ partial) {
  __shared__ float red[512][5];
  grid_dep_trigger();
  const int groups = cout / 4;                  // 8 .. 64
  const int rows = 256 / (cout / 8);            // pixels in flight per block
  const int g = threadIdx.x % groups, r = threadIdx.x / groups;
  const long long per = (npix + gridDim.x - 1) / gridDim.x;
  const long long p0 = blockIdx.x * per;
  const long long p1 = p0 + per < npix ? p0 + per : npix;
  float acc[4] = {0, 0, 0, 0};
  if (r < rows)
#pragma unroll 8
    for (long long p = p0 + r; p < p1; p += rows) {
      const uint2 u = *reinterpret_cast<const uint2*>(dy + p * ps + 4 * g);
      const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
      const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
      acc[0] += a.x;
      acc[1] += a.y;
      acc[2] += b.x;
      acc[3] += b.y;
    }
#pragma unroll
  for (int k = 0; k < 4; ++k) red[threadIdx.x][k] = acc[k];
  __syncthreads();
  if ((int)threadIdx.x < cout) {
    const int gg = threadIdx.x / 4, k = threadIdx.x % 4;
    float t = 0.f;
    for (int rr = 0; rr < rows; ++rr) t += red[rr * groups + gg][k];
    grid_dep_wait();
    partial[(long long)blockIdx.x * cout + threadIdx.x] = t;
  }
}

// dW[co][tap][ci] = sum_s of its partial sums.  A column (unit, co) has 128
// rows, four per lane.  The order is fixed: eight sums of the splits s = w,
// w + 8, ... (each as its even and odd terms), added in turn; a warp does all
// eight (G = 1) or, of many splits, one (G = 8).  The blocks past those sum the
// bias gradient's partials the same way, 32 channels each.
__device__ __forceinline__ void add4(float4& t, const float4& x) {
  t.x += x.x;
  t.y += x.y;
  t.z += x.z;
  t.w += x.w;
}
template <int G>
__global__ void __launch_bounds__(256) wgrad_reduce_kernel(const __grid_constant__ WgradArgs a,
                                                           const float* __restrict__ bpart,
                                                           int nb, float* __restrict__ dW,
                                                           float* __restrict__ db) {
  __shared__ float4 red[8][32];
  grid_dep_wait();
  grid_dep_trigger();
  const WgradPlan& P = a.plan;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int blocks = P.units * a.cout * G / 8;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  if ((int)blockIdx.x >= blocks) {
    const int c = ((int)blockIdx.x - blocks) * 32 + lane;
    float t0 = 0.f, t1 = 0.f;
    int j = w;
#pragma unroll 8
    for (; j + 8 < nb; j += 16) {
      t0 += bpart[(long long)j * a.cout + c];
      t1 += bpart[(long long)(j + 8) * a.cout + c];
    }
    if (j < nb) t0 += bpart[(long long)j * a.cout + c];
    red[w][lane].x = t0 + t1;
    __syncthreads();
    if (w == 0) {
      float t = 0.f;
      for (int k = 0; k < 8; ++k) t += red[k][lane].x;
      db[c] = t;
    }
    return;
  }
  const int col = G == 8 ? blockIdx.x : blockIdx.x * 8 + w;
  const int n = col % a.cout;
  int u;
  const int block = wgrad_block(P, col / a.cout, &u);
  const size_t stride = (size_t)P.units * a.cout * 32;
  const float4* p = reinterpret_cast<const float4*>(a.partial) + (size_t)col * 32 + lane;
  auto sum = [&](int first) {
    float4 t0 = zero, t1 = zero;
    int s = first;
#pragma unroll 4
    for (; s + 8 < P.splits; s += 16) {
      add4(t0, p[s * stride]);
      add4(t1, p[(s + 8) * stride]);
    }
    if (s < P.splits) add4(t0, p[s * stride]);
    add4(t0, t1);
    return t0;
  };
  float4 t = zero;
  if (G == 8) {
    red[w][lane] = sum(w);
    __syncthreads();
    if (w) return;
    for (int k = 0; k < 8; ++k) add4(t, red[k][lane]);
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) add4(t, sum(k));
  }
  int tap, ci;  // (four rows lie in one run)
  if (!wgrad_row(P, block, u, 4 * lane, &tap, &ci)) return;
  float* o = dW + ((size_t)n * 9 + tap) * a.cin + ci;
  if ((reinterpret_cast<uintptr_t>(o) & 15) == 0) {
    *reinterpret_cast<float4*>(o) = t;
  } else {
    o[0] = t.x;
    o[1] = t.y;
    o[2] = t.z;
    o[3] = t.w;
  }
}

__global__ void adam_kernel(float* __restrict__ th, const float* __restrict__ g,
                            float* __restrict__ m, float* __restrict__ v, long long n, float lr,
                            float b1, float b2, float eps, float c1, float c2) {
  grid_dep_wait();
  grid_dep_trigger();
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    th[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

}  // namespace

// Launches kernel<int> or, past 2^31 elements, kernel<long long>.
#define LAUNCH_INDEXED(kernel, n, ...)                                                     \
  do {                                                                                     \
    const long long n_ = (n);                                                              \
    const dim3 grid_(blocks_for(n_)), block_(kT);                                          \
    if (n_ < (1LL << 31) - 1048576LL * kT)                                                 \
      launch_dependent(kernel<int>, grid_, block_, 0, st, __VA_ARGS__);                    \
    else                                                                                   \
      launch_dependent(kernel<long long>, grid_, block_, 0, st, __VA_ARGS__);              \
    note_launches(1);                                                                      \
  } while (0)

void launch_prep_weights(const float* theta, const WeightPrepAll& p, long long total_w,
                         cudaStream_t st) {
  launch_dependent(prep_weights_kernel, dim3((unsigned)(total_w / (32 * 32))), dim3(256), 0, st,
                   theta, p);
  note_launches(1);
}

void launch_pack_input(const float* in, int in_ch, bf16* x0, long long npix, cudaStream_t st) {
  launch_dependent(pack_input_kernel, dim3(blocks_for(npix)), dim3(kT), 0, st, in, in_ch, x0,
                   npix);
  note_launches(1);
}

void launch_up_backward_mask(const bf16* g, int g_ps, const bf16* x, bf16* d, int B, int h,
                             int w, int C, cudaStream_t st) {
  LAUNCH_INDEXED(up_backward_mask_kernel, (long long)B * h * w * (C / 8), g, g_ps, x, d, B, h, w,
                 C);
}

void launch_pool_backward_combine(const bf16* gp, const bf16* s, int s_ps, const bf16* gskip,
                                  int gskip_ps, bf16* d, int B, int H, int W, int C,
                                  cudaStream_t st) {
  LAUNCH_INDEXED(pool_backward_combine_kernel, (long long)B * H * W * (C / 8), gp, s, s_ps, gskip,
                 gskip_ps, d, B, H, W, C);
}

void launch_head_backward(const bf16* x, const float* theta_head, const float* out,
                          const float* target, long long npix, bf16* dpre, double* partial,
                          int nblocks, double* loss, float* grad_head, cudaStream_t st) {
  // float partials of the head gradients follow the FP64 loss partials
  float* hpart = reinterpret_cast<float*>(partial + nblocks);
  launch_dependent(head_backward_kernel, dim3(nblocks), dim3(kT), 0, st, x, theta_head, out,
                   target, npix, dpre, partial, hpart);
  launch_dependent(head_backward_total_kernel, dim3(1), dim3(kT), nblocks * 33 * sizeof(float), st,
                   partial, hpart, nblocks, npix, loss, grad_head);
  note_launches(2);
}

void launch_bias_grad(const bf16* dy, int dy_ps, int cout, long long npix, float* partial,
                      int nblocks, cudaStream_t st) {
  launch_dependent(bias_grad_kernel, dim3(nblocks), dim3(512), 0, st, dy, dy_ps, cout, npix,
                   partial);
  note_launches(1);
}

void launch_wgrad_reduce(const WgradArgs& a, float* dW, const float* bpart, int nb, float* db,
                         cudaStream_t st) {
  const int cols = a.plan.units * a.cout, bias = db ? a.cout / 32 : 0;
  if (a.plan.splits > 32)
    launch_dependent(wgrad_reduce_kernel<8>, dim3(cols + bias), dim3(256), 0, st, a, bpart, nb, dW,
                     db);
  else
    launch_dependent(wgrad_reduce_kernel<1>, dim3(cols / 8 + bias), dim3(256), 0, st, a, bpart, nb,
                     dW, db);
  note_launches(1);
}

void launch_adam(float* theta, const float* grad, float* m, float* v, long long n, int step,
                 float lr, float b1, float b2, float eps, cudaStream_t st) {
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  launch_dependent(adam_kernel, dim3(blocks_for(n)), dim3(kT), 0, st, theta, grad, m, v, n, lr, b1,
                   b2, eps, c1, c2);
  note_launches(1);
}

}  // namespace sweep
