// 3 x 3 convolutions of the U-Net preconditioner on the 5th-generation
// tensor cores (tcgen05, BF16 operands, FP32 accumulator in tensor memory).
//
// conv_kernel: an implicit GEMM with M = 128 pixels per accumulator, N output
// channels, and K = 9 taps x cin in (tap, channel chunk) order.  A CTA takes a
// tile of 16 rows x 8, 16 or 32 columns (1, 2 or 4 accumulators) and all or
// part of the output channels.  The input tile is staged once, with a
// one-pixel halo (TMA boxes of the NHWC tensor; the zero padding is the box's
// out-of-bounds fill), and a tap is an offset into it; the weights' (tap,
// chunk) slices go through a ring.  What bounds it: MMAs into one accumulator
// follow one another at about 146 cycles and an MMA of N <= 64 takes 44
// cycles, whatever its N; a CTA's set-up, first loads and epilogue take about
// 3 us.  So the launcher's cost model looks for several accumulators in
// flight on an SM (of one CTA, or of several) before large tiles.  Staging a
// shifted tile per tap with one accumulator per CTA read the input nine times
// through L2: 8 x 256 x 256 pixels, 32 -> 32 channels, 40 us, now 23 (10 us
// are the bytes at the copy rate); 8 x 64 x 64, 256 -> 128: 76 us, now 22;
// 8 x 32 x 32, 256 -> 256: 25 us, now 15 (11 us are the chain of MMAs).
// The epilogue also writes what the next layer reads instead of the output: its
// 2 x 2 average, its upsampling or the 1 x 1 head's value, from the same
// registers, which saves an inference seven of 26 kernels.
//
// wgrad_kernel: the weight gradient, a split-K GEMM over the pixels (see
// WgradPlan in unet_internal.cuh).  Both operands are staged pixel-major by TMA,
// i.e. MN-major for the MMA; the input with a pixel more on either side, so that
// the taps of a row are offsets into one staged box, and 128 pixels a stage
// where the rows are that long.  Each CTA writes its FP32 partial sums; a
// reduction kernel adds the splits in a fixed order.  Bound by the chain of
// dependent MMAs of a split (146 cycles each: without any loads 8 x 256 x 256,
// 32 -> 32 channels takes 31 us) and, close behind, by the lines that TMA
// fetches.  Four boxes per 64 pixels and 128 (tap, ci) rows took 104 us there,
// now 33; 64 -> 32 channels 142, now 56; 8 x 128 x 128, 128 -> 64: 69, now 33.
//
// Every mbarrier wait is bounded (tma.cuh); a wait that gives up latches
// SWEEP_ETIMEOUT, the CTA skips its stores, waits for its own copies in
// flight and frees its tensor memory before it exits.
#include <algorithm>
#include <mutex>

#include "sweep_internal.cuh"
#include "tcgen05.cuh"
#include "unet_internal.cuh"

namespace sweep {
namespace {

constexpr int kConvMaxStages = 24;
constexpr size_t kSmemPerSm = 228 * 1024;  // per SM, of which 1 KB per CTA is reserved
// dynamic shared memory a kernel may ask for (below the 227 KB opt-in limit,
// which also counts the static barriers)
constexpr int kConvMaxSmem = 225 * 1024;
constexpr int kWgMaxSmem = 225 * 1024;
constexpr int kWgHalf = 104 * 1024;  // two per SM leave room for a block of the bias gradient
constexpr int kWgMaxCtas = 512;

__host__ __device__ inline uint32_t tmem_cols(int n) {
  uint32_t c = 32;
  while (c < (uint32_t)n) c <<= 1;
  return c;
}

// whole-warp bounded wait (lane 0's outcome is the warp's)
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity) {
  bool got = mbar_wait(bar, parity);
  return __shfl_sync(0xffffffffu, got ? 1 : 0, 0) != 0;
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

// The values of w whose mask is positive, 0 for the others (8 BF16 each).
__device__ __forceinline__ uint4 mask8(uint4 w, const uint4& m) {
  __nv_bfloat16* v = reinterpret_cast<__nv_bfloat16*>(&w);
  const __nv_bfloat16* k = reinterpret_cast<const __nv_bfloat16*>(&m);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (!(__bfloat162float(k[i]) > 0.f)) v[i] = __float2bfloat16_rn(0.f);
  return w;
}

__device__ __forceinline__ uint4 shfl_xor4(const uint4& v, int m) {
  return make_uint4(
      __shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m),
      __shfl_xor_sync(0xffffffffu, v.z, m), __shfl_xor_sync(0xffffffffu, v.w, m));
}

// Averages of 8 BF16 values each, summed in this order.
__device__ __forceinline__ uint32_t average4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  auto f = [](const uint32_t& u) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u));
  };
  const float2 x = f(a), y = f(b), z = f(c), w = f(d);
  return pack2((((x.x + y.x) + z.x) + w.x) * 0.25f, (((x.y + y.y) + z.y) + w.y) * 0.25f);
}
__device__ __forceinline__ uint4 average4(const uint4& a, const uint4& b, const uint4& c,
                                          const uint4& d) {
  return make_uint4(average4(a.x, b.x, c.x, d.x), average4(a.y, b.y, c.y, d.y),
                    average4(a.z, b.z, c.z, d.z), average4(a.w, b.w, c.w, d.w));
}

// Convolution tile: 16 rows x 8 ns columns of pixels.  An accumulator takes
// 128 of them (16 rows x 8 columns): the 8 pixels of a row are one 8-row core
// matrix of the A operand, and SBO is the row pitch of the staged tile.
constexpr int kConvRows = 16;
constexpr int kConvThreads = 192;  // warps 0-3: epilogue, 4: TMA, 5: MMA
constexpr int kMaxChunks = 8;      // input channel chunks

// Bytes of a staged chunk of kc channels: a line of 2 kc bytes per pixel,
// padded to whole swizzle atoms.
__host__ __device__ inline uint32_t chunk_bytes(int ns, int kc) {
  return (uint32_t)((8 * ns + 2) * (kConvRows + 2) * 2 * kc + 1023) / 1024 * 1024;
}

template <int KC, int NS>
__global__ void __launch_bounds__(kConvThreads)
    conv_kernel(const __grid_constant__ ConvArgs a) {
  __shared__ __align__(8) uint64_t full[kConvMaxStages];
  __shared__ __align__(8) uint64_t empty[kConvMaxStages];
  __shared__ __align__(8) uint64_t inbar[kMaxChunks];
  __shared__ __align__(8) uint64_t done;
  __shared__ uint32_t tmem_holder;
  __shared__ int failed;
  __shared__ __align__(16) float bias[256];
  __shared__ float head[33];
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_u = smem_u32(smem_raw);
  const uint32_t base_u = (raw_u + 1023u) & ~1023u;
  uint8_t* base = smem_raw + (base_u - raw_u);
  const int S = a.stages;
  const int PW = 8 * NS + 2;                              // staged pixels per row
  const uint32_t CS = chunk_bytes(NS, KC);
  const int nch = a.cin / KC, kiters = 9 * nch;
  // the staged input, then the ring: weights and, when the input does not
  // stay, a chunk of it behind them
  const uint32_t wbytes = (uint32_t)(a.n * KC * 2), stage_bytes = wbytes + (a.stays ? 0 : CS);
  const int kept = a.stays ? nch : 0;
  const uint32_t in_u = base_u, ring_u = base_u + (uint32_t)kept * CS;
  uint8_t* in = base;
  base += (size_t)kept * CS;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t ncols = tmem_cols(a.n * NS);

  const int nblk = a.cout / a.n;
  int t = blockIdx.x / nblk;
  const int n0 = (blockIdx.x - t * nblk) * a.n;
  const int ntx = a.W / (8 * NS), nty = (a.H + kConvRows - 1) / kConvRows;
  const int b = t / (ntx * nty);
  t -= b * ntx * nty;
  const int y0 = (t / ntx) * kConvRows, x0 = (t % ntx) * 8 * NS;

  if (warp == 5) {
    tmem_alloc(&tmem_holder, ncols);
    tmem_relinquish();
  }
  if (threadIdx.x == 128) {
    for (int i = 0; i < S; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < kept; ++i) mbar_init(&inbar[i], 1);
    mbar_init(&done, 1);
    failed = 0;
    fence_barrier_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_holder;
  if (warp != 4) {  // (the TMA warp waits on its own)
    if (!a.late) grid_dep_wait();
    grid_dep_trigger();
  }

  if (warp == 4) {  // TMA producer
    if (lane == 0) {
      // The weights are older than the kernel launched before this one: the
      // ring's first pass goes out ahead of the wait for that kernel.
      const uint32_t tx =
          wbytes + (a.stays ? 0 : (uint32_t)(PW * (kConvRows + 2) * 2 * KC));
      auto weights = [&](int k, int s) {
        mbar_arrive_expect_tx(&full[s], tx);
        tma_load_3d(base + (size_t)s * stage_bytes, &a.tw, &full[s], k % nch * KC, k / nch, n0);
      };
      const int first = min(S, kiters);
      for (int k = 0; k < first; ++k) weights(k, k);
      if (!a.late) grid_dep_wait();
      for (int k = 0; k < kept; ++k) {  // the input tile, chunk by chunk (zero off the image)
        mbar_arrive_expect_tx(&inbar[k], (uint32_t)(PW * (kConvRows + 2) * 2 * KC));
        tma_load_4d(in + (size_t)k * CS, &a.tin, &inbar[k], k * KC, x0 - 1, y0 - 1, b);
      }
      int k = 0, s = 0, ph = 1;
      for (; k < kiters; ++k) {
        if (k >= S) {
          if (!mbar_wait(&empty[s], ph)) {
            latch(a.status, SWEEP_ETIMEOUT);
            failed = 1;
            break;
          }
          weights(k, s);
        }
        if (!a.stays)
          tma_load_4d(base + (size_t)s * stage_bytes + wbytes, &a.tin, &full[s], k % nch * KC,
                      x0 - 1, y0 - 1, b);
        if (++s == S) {
          s = 0;
          ph ^= 1;
        }
      }
      // every copy has landed before the CTA may exit
      for (int j = k > S ? k - S : 0; j < k; ++j) mbar_wait(&full[j % S], (j / S) & 1);
      for (int j = 0; j < kept; ++j) mbar_wait(&inbar[j], 0);
    }
    __syncwarp();
  } else if (warp == 5) {  // MMA issuer (the whole warp, one lane issuing)
    const uint32_t e = elect_one();
    const uint32_t idesc = idesc_bf16_f32(128, a.n, 0, 0);
    const uint32_t swz = KC == 64 ? kSwizzle128 : kSwizzle64;
    const uint32_t line = 2u * KC;  // bytes of a staged pixel
    const uint64_t adesc = smem_desc(in_u, 16u, (uint32_t)PW * line, swz);
    const uint64_t bdesc = smem_desc(ring_u, 16u, 8u * KC * 2u, swz);
    int s = 0, ph = 0;
    bool ok = true;
    for (int tap = 0; tap < 9 && ok; ++tap) {
      // (addresses are the descriptors' low bits, in 16 bytes)
      const uint64_t shift = (uint64_t)((uint32_t)(tap / 3 * PW + tap % 3) * (line >> 4));
      uint64_t at = adesc + shift;
      for (int ch = 0; ch < nch; ++ch) {
        ok = mbar_wait(&full[s], ph) && (tap > 0 || !a.stays || mbar_wait(&inbar[ch], 0));
        if (!__all_sync(0xffffffffu, ok)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint64_t bd = bdesc + (uint64_t)((uint32_t)s * stage_bytes >> 4);
        if (!a.stays) at = adesc + shift + (uint64_t)(((uint32_t)s * stage_bytes + wbytes) >> 4);
#pragma unroll
        for (int j = 0; j < KC / 16; ++j)
#pragma unroll
          for (int q = 0; q < NS; ++q)
            mma_bf16_warp(e, tmem + (uint32_t)(q * a.n), at + 2 * j + (line >> 1) * q, bd + 2 * j,
                          idesc, (tap | ch | j) != 0);
        mma_commit_warp(e, &empty[s]);  // the stage is free once these MMAs have read it
        at += CS >> 4;
        if (++s == S) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    if (!ok && lane == 0) {
      latch(a.status, SWEEP_ETIMEOUT);
      failed = 1;
    }
    mma_commit_warp(e, &done);  // every MMA issued has completed
    __syncwarp();
  }

  // The epilogue.  A lane holds 32 channels of pixel (row 4 warp + lane / 8,
  // column lane % 8) of its accumulator; through shared memory (the staged
  // input's, free by then) four lanes take the 64 bytes of a pixel, so that a
  // store covers whole sectors.  The bias and the first step's mask are read
  // while the MMAs run, a step's mask while the step before it is stored.
  const int px = lane >> 2, cu = lane & 3, steps = NS * (a.n / 32);
  const long long row0 = (long long)b * a.H + y0 + 4 * warp;
  const long long pix0 = row0 * a.W + x0 + px;
  uint4 mk[4];
  auto load_mask = [&](int q, int c0) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (y0 + 4 * warp + i < a.H)
        mk[i] = *reinterpret_cast<const uint4*>(
            a.mask + (pix0 + 8 * q + (long long)i * a.W) * a.mask_ps + n0 + c0 + 8 * cu);
  };
  if (warp < 4) {
    if (a.bias)
      for (int i = threadIdx.x; i < a.n; i += 128) bias[i] = a.bias[n0 + i];
    if (a.head && threadIdx.x < 33) head[threadIdx.x] = a.head[threadIdx.x];
    if (a.op == kOpMask) load_mask(0, 0);
  }
  const bool got = mbar_wait(&done, 0);
  const bool bad = __syncthreads_or(!got) || failed;
  tc_fence_after();
  if (!bad && warp < 4) {
    uint8_t* xch = in + warp * 2048;
    int q = 0, c0 = 0;
    for (int k = 0; k < steps; ++k) {
      float v[32];
      tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(q * a.n + c0), v);
      if (a.bias) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 f = *reinterpret_cast<const float4*>(bias + c0 + 4 * i);
          v[4 * i] += f.x;
          v[4 * i + 1] += f.y;
          v[4 * i + 2] += f.z;
          v[4 * i + 3] += f.w;
        }
      }
      if (a.op == kOpRelu) {
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = fmaxf(v[i], 0.f);
      }
      if (a.head) {  // the 1 x 1 head (cout = 32) of the lane's own pixel
        const int hr = 4 * warp + (lane >> 3);
        float t = 0.f;
#pragma unroll
        for (int i = 0; i < 32; ++i)
          t = fmaf(__bfloat162float(__float2bfloat16_rn(v[i])), head[i], t);
        if (y0 + hr < a.H)
          a.head_out[((long long)b * a.H + y0 + hr) * a.W + x0 + 8 * q + (lane & 7)] = t + head[32];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        uint4 w;
        w.x = pack2(v[8 * u + 0], v[8 * u + 1]);
        w.y = pack2(v[8 * u + 2], v[8 * u + 3]);
        w.z = pack2(v[8 * u + 4], v[8 * u + 5]);
        w.w = pack2(v[8 * u + 6], v[8 * u + 7]);
        *reinterpret_cast<uint4*>(xch + lane * 64 + ((u ^ (lane >> 1)) & 3) * 16) = w;
      }
      __syncwarp();
      const int ch = n0 + c0 + 8 * cu, col = x0 + 8 * q + px;  // the lane's when it stores
      bf16* o = a.out + (pix0 + 8 * q) * a.out_ps + ch;
      uint4 w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int p = 8 * i + px;
        w[i] = *reinterpret_cast<const uint4*>(xch + p * 64 + ((cu ^ (p >> 1)) & 3) * 16);
        if (a.op == kOpMask) w[i] = mask8(w[i], mk[i]);
      }
      if ((c0 += 32) == a.n) {
        c0 = 0;
        ++q;
      }
      if (a.op == kOpMask && k + 1 < steps) load_mask(q, c0);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (y0 + 4 * warp + i < a.H)
          *reinterpret_cast<uint4*>(o + (long long)i * a.W * a.out_ps) = w[i];
      if (a.up) {  // the nearest upsampling: four copies
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (y0 + 4 * warp + i < a.H) {
            bf16* d = a.up + (4 * (row0 + i) * a.W + 2 * col) * a.cout + ch;
            const long long pitch = 2LL * a.W * a.cout;
            *reinterpret_cast<uint4*>(d) = w[i];
            *reinterpret_cast<uint4*>(d + a.cout) = w[i];
            *reinterpret_cast<uint4*>(d + pitch) = w[i];
            *reinterpret_cast<uint4*>(d + pitch + a.cout) = w[i];
          }
      }
      if (a.pool) {  // the 2 x 2 average (even H, W): the odd columns' lanes hand theirs over
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
          const uint4 r0 = shfl_xor4(w[i], 4), r1 = shfl_xor4(w[i + 1], 4);
          if (!(px & 1) && y0 + 4 * warp + i < a.H)
            *reinterpret_cast<uint4*>(
                a.pool + ((row0 + i) / 2 * (a.W / 2) + col / 2) * a.cout + ch) =
                average4(w[i], r0, w[i + 1], r1);
        }
      }
      __syncwarp();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 5) {
    tc_fence_after();
    tmem_dealloc(tmem, ncols);
  }
  if (a.late) grid_dep_wait();
}

constexpr int kWgMaxStages = 16;

// Bytes of a staged chunk of kc channels: ph rows of q pw + 2 pixels, in whole
// swizzle atoms (a unit's unused runs read past it, into what lies behind).
__host__ __device__ inline uint32_t wg_chunk_bytes(const WgradPlan& P) {
  return (uint32_t)(P.ph * (P.q * P.pw + 2) * 2 * P.kc + 1023) / 1024 * 1024;
}
__global__ void __launch_bounds__(kConvThreads, 2)
    wgrad_kernel(const __grid_constant__ WgradArgs a) {
  __shared__ __align__(8) uint64_t full[kWgMaxStages];
  __shared__ __align__(8) uint64_t empty[kWgMaxStages];
  __shared__ __align__(8) uint64_t done;
  __shared__ uint32_t tmem_holder;
  __shared__ int failed;
  extern __shared__ uint8_t smem_raw[];
  const WgradPlan& P = a.plan;
  const uint32_t raw_u = smem_u32(smem_raw);
  const uint32_t base_u = (raw_u + 1023u) & ~1023u;
  uint8_t* base = smem_raw + (base_u - raw_u);
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t ncols = tmem_cols(a.cout);

  // this CTA's unit (of an input channel block) and its strips
  const int split = blockIdx.x / P.units;
  int u;
  const int block = wgrad_block(P, blockIdx.x - split * P.units, &u);
  const int chunks = wgrad_chunks(P, block);
  const WgradUnit unit = wgrad_unit(P, chunks, u);
  const int rows = 1 + unit.down;  // of strips
  const uint32_t CS = wg_chunk_bytes(P), DS = (uint32_t)(P.q * kWgPix * 2 * P.kb);
  const uint32_t in_bytes = (uint32_t)(rows * chunks) * CS;
  const uint32_t dy_bytes = (uint32_t)(P.q * kWgPix * 2 * a.cout);
  const uint32_t stage_bytes = in_bytes + dy_bytes;
  const int S = min(kWgMaxStages, P.ring / (int)stage_bytes);
  const int ntx = a.W / P.pw, nty = a.H / P.ph;
  const long long T = (long long)a.B * ntx * nty;
  const long long t0 = T * split / P.splits;
  const int strips = (int)(T * (split + 1) / P.splits - t0);

  if (warp == 5) {
    tmem_alloc(&tmem_holder, ncols);
    tmem_relinquish();
  }
  if (threadIdx.x == 128) {
    for (int i = 0; i < S; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    mbar_init(&done, 1);
    failed = 0;
    fence_barrier_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_holder;
  grid_dep_wait();
  grid_dep_trigger();

  if (warp == 4) {  // TMA producer
    if (lane == 0) {
      const uint32_t bytes =
          (uint32_t)(rows * chunks * P.ph * (P.q * P.pw + 2) * 2 * P.kc) + dy_bytes;
      int k = 0, s = 0, ph = 1;
      int tx = (int)(t0 % ntx), ty = (int)(t0 / ntx % nty), b = (int)(t0 / ntx / nty);
      for (int left = strips; left > 0; ++k) {
        if (k >= S && !mbar_wait(&empty[s], ph)) {
          latch(a.status, SWEEP_ETIMEOUT);
          failed = 1;
          break;
        }
        uint8_t* st = base + (size_t)s * stage_bytes;
        mbar_arrive_expect_tx(&full[s], bytes);
        for (int r = 0; r < rows; ++r)
          for (int c = 0; c < chunks; ++c)
            tma_load_4d(st + (size_t)(r * chunks + c) * CS, &a.tin, &full[s],
                        (block * P.cpb + c) * P.kc, P.pw * tx - 1, P.ph * ty + unit.ky + r - 1, b);
        for (int q = 0; q < a.cout / P.kb; ++q)
          tma_load_4d(st + in_bytes + (size_t)q * DS, &a.tdy, &full[s], q * P.kb, P.pw * tx,
                      P.ph * ty, b);
        if (++s == S) {
          s = 0;
          ph ^= 1;
        }
        const int n = min(min(P.q, ntx - tx), left);  // strips of this stage, of one row
        left -= n;
        if ((tx += n) == ntx) {
          tx = 0;
          if (++ty == nty) {
            ty = 0;
            ++b;
          }
        }
      }
      for (int j = k > S ? k - S : 0; j < k; ++j) mbar_wait(&full[j % S], (j / S) & 1);
    }
    __syncwarp();
  } else if (warp == 5) {  // MMA issuer: both operands MN-major, 16 pixels of a row per MMA
    const uint32_t e = elect_one();
    const uint32_t idesc = idesc_bf16_f32(128, a.cout, 1, 1);
    const uint32_t la = 2u * P.kc, lb = 2u * P.kb;  // bytes of a staged pixel
    const uint64_t b0 = smem_desc(base_u + in_bytes, DS, 8u * lb,
                                  P.kb == 64 ? kSwizzle128 : kSwizzle64);
    const uint64_t a0 = smem_desc(base_u + (uint32_t)unit.kx * la,
                                  chunks > 1 || unit.down ? CS : la, 8u * la,
                                  P.kc == 64 ? kSwizzle128 : kSwizzle64);
    int s = 0, ph = 0, tx = (int)(t0 % ntx);
    uint32_t acc = 0;
    bool ok = true;
    for (int left = strips; left > 0;) {
      ok = mbar_wait(&full[s], ph);
      if (!__all_sync(0xffffffffu, ok)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint64_t so = (uint64_t)((uint32_t)s * stage_bytes >> 4);
      const int n = min(min(P.q, ntx - tx), left);
      left -= n;
      tx = tx + n == ntx ? 0 : tx + n;
      for (int h = 0; h < n; ++h) {
#pragma unroll
        for (int j = 0; j < kWgPix / 16; ++j) {
          // (a strip of several rows is a stage of its own: h = 0)
          const uint32_t px = (uint32_t)(kWgPix * h + 16 * j + 2 * (16 * j / P.pw));
          mma_bf16_warp(e, tmem, a0 + so + (uint64_t)(px * la >> 4),
                        b0 + so + (uint64_t)((uint32_t)(kWgPix * h + 16 * j) * lb >> 4), idesc,
                        acc);
          acc = 1;
        }
      }
      mma_commit_warp(e, &empty[s]);
      if (++s == S) {
        s = 0;
        ph ^= 1;
      }
    }
    if (!ok && lane == 0) {
      latch(a.status, SWEEP_ETIMEOUT);
      failed = 1;
    }
    mma_commit_warp(e, &done);
    __syncwarp();
  }

  const bool got = mbar_wait(&done, 0);
  const bool bad = __syncthreads_or(!got) || failed;
  tc_fence_after();
  if (!bad && warp < 4) {
    // a warp stores 32 rows of a column
    float* out = a.partial + (size_t)blockIdx.x * a.cout * 128 + warp * 32 + lane;
    for (int c0 = 0; c0 < a.cout; c0 += 32) {
      float v[32];
      tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
      for (int i = 0; i < 32; ++i) out[(size_t)(c0 + i) * 128] = v[i];
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 5) {
    tc_fence_after();
    tmem_dealloc(tmem, ncols);
  }
}

}  // namespace

// A convolution launch with tile width 8 ns and n output channels per CTA:
// its weight stages, shared memory and estimated cycles (0: does not fit).
// As many CTAs per SM as leave each a few stages (they hide one another's
// set-up and epilogue), then as many stages as fit (small ones need many: a
// stage takes a microsecond to arrive).  The estimate of a wave: its K steps
// at the larger of the latency of dependent MMAs and the SM's tensor work,
// plus set-up and epilogue.  Against a sweep of every (ns, n, CTAs per SM) on
// 32 layers from 1 x 16 x 16 to 8 x 256 x 256 it picks the fastest or one
// within 12 %; a fixed ns = 1, n = cout takes 1.3 to 2.2 times as long from
// 8 x 64 x 64 up, a fixed ns = 4 1.2 to 1.6 times below.  stays: false stages
// the input again for every tap, for inputs whose tile does not fit.
struct ConvFit {
  int ns, n;
  bool stays;
  int stages, ctas;
  size_t smem;
  double cycles;
};
constexpr double kConvChain = 146;   // cycles between MMAs into one accumulator
constexpr double kConvFixed = 6000;  // set-up, first loads, drain
constexpr double kConvOut = 16;      // epilogue, per output channel of an accumulator
ConvFit conv_fit(const ConvArgs& a, int ns, int n, bool stays) {
  ConvFit f{ns, n, stays, 0, 0, 0, 0.0};
  const int chunks = a.cin / a.kc, kiters = 9 * chunks;
  const size_t chunk = chunk_bytes(ns, a.kc), in = 1024 + (stays ? chunk * chunks : 0);
  const size_t stage = (size_t)n * a.kc * 2 + (stays ? 0 : chunk);
  const int cols = (int)tmem_cols(n * ns);
  if (cols > 512 || (stays && chunks > kMaxChunks)) return f;
  f.ctas = a.B * ((a.H + kConvRows - 1) / kConvRows) * (a.W / (8 * ns)) * (a.cout / n);
  const int sms = device_sms(), per_sm = (f.ctas + sms - 1) / sms;
  for (int res = std::max(1, std::min({512 / cols, per_sm, 4})); res >= 1; --res) {
    const size_t budget = std::min<size_t>(kSmemPerSm / res - 3072, kConvMaxSmem);
    if (budget < in + 2 * stage) continue;
    const int s = (int)std::min<size_t>(kConvMaxStages, (budget - in) / stage);
    if (res > 1 && s < std::min(3, kiters)) continue;
    f.stages = std::min(s, kiters);
    // no more CTAs on an SM than have tensor memory
    f.smem = std::max(in + f.stages * stage, kSmemPerSm / (512 / cols + 1) + 1);
    const double k = kiters * (a.kc / 16);
    const double mma = std::max(40.0, 0.6 * n);
    const int waves = (per_sm + res - 1) / res, last = per_sm - (waves - 1) * res;
    const double step = std::max(kConvChain, ns * res * mma);
    f.cycles = (waves - 1) * (k * step + kConvFixed) +
               k * std::max(kConvChain, ns * last * mma) + kConvFixed + ns * n * kConvOut * waves;
    return f;
  }
  return f;
}

void (*const kConvKernels[])(const ConvArgs) = {conv_kernel<32, 1>, conv_kernel<32, 2>,
                                                conv_kernel<32, 4>, conv_kernel<64, 1>,
                                                conv_kernel<64, 2>, conv_kernel<64, 4>};

int launch_conv(ConvArgs a, cudaStream_t st) {
  static std::once_flag once;
  std::call_once(once, [] {
    for (auto* f : kConvKernels)
      cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kConvMaxSmem);
  });
  ConvFit best{};
  for (const bool stays : {true, false}) {  // (false when nothing else fits)
    for (int ns = 1; ns <= 4 && 8 * ns <= a.W; ns *= 2)
      for (int n = 32; n <= std::min(a.cout, 256); n += 32) {
        if (a.cout % n) continue;
        const ConvFit f = conv_fit(a, ns, n, stays);
        if (f.cycles > 0 && (best.cycles == 0 || f.cycles < best.cycles)) best = f;
      }
    if (best.cycles > 0) break;
  }
  if (best.cycles == 0) return SWEEP_EUNSUPPORTED;
  a.ns = best.ns;
  a.n = best.n;
  a.stays = best.stays;
  a.stages = best.stages;
  if (!a.make_maps(a)) return SWEEP_ECUDA;
  auto* kernel = kConvKernels[(a.kc == 64 ? 3 : 0) + (a.ns == 4 ? 2 : a.ns - 1)];
  launch_dependent(kernel, dim3(best.ctas), dim3(kConvThreads), best.smem, st, a);
  note_launches(1);
  return SWEEP_OK;
}

// The cut of a weight gradient.  Splits: as many as give 2 CTAs per SM with 128
// rows of (tap, ci) each (at most kWgMaxCtas CTAs).  partial: floats of the
// partial sums.
WgradPlan wgrad_plan(int B, int H, int W, int cin, int cout, size_t* partial) {
  WgradPlan P{};
  P.kc = cin % 64 == 0 ? 64 : 32;
  P.kb = cout % 64 == 0 ? 64 : 32;
  P.nchunks = cin / P.kc;
  P.cpb = 128 / P.kc;
  P.blocks = (P.nchunks + P.cpb - 1) / P.cpb;
  P.pw = std::min(W, kWgPix);
  P.ph = kWgPix / P.pw;
  P.q = W >= 2 * kWgPix ? 2 : 1;  // (1 for all: 46 us for 33, 88 for 56, as above)
  P.units = (P.blocks - 1) * wgrad_units(P, 0) + wgrad_units(P, P.blocks - 1);
  const long long T = (long long)B * (H / P.ph) * (W / P.pw);
  const int mtiles = (9 * cin + 127) / 128;
  P.splits = std::max(1, std::min(2 * device_sms(), kWgMaxCtas) / mtiles);
  P.splits = (int)std::max(1LL, std::min<long long>(P.splits, T));
  size_t staged = 0;  // most of a unit's
  for (int i = 0; i < P.units; ++i) {
    int u;
    const int chunks = wgrad_chunks(P, wgrad_block(P, i, &u));
    staged = std::max(staged, (size_t)(1 + wgrad_unit(P, chunks, u).down) * chunks *
                                  wg_chunk_bytes(P));
  }
  const size_t stage = staged + (size_t)P.q * kWgPix * 2 * cout;
  // (the unused runs of a short block's units read past the last stage)
  const int last = wgrad_chunks(P, P.blocks - 1);
  const size_t slack = 1024 + (last > 1 ? (size_t)(P.cpb - last) * wg_chunk_bytes(P) : 0);
  const int cols = (int)tmem_cols(cout);
  const int res = cols <= 256 && slack + 2 * stage <= kWgHalf ? 2 : 1;
  const size_t most = res == 2 ? kWgHalf : kWgMaxSmem;
  P.ring = (int)std::min(most - slack, kWgMaxStages * stage);
  P.smem = std::max(slack + P.ring, kSmemPerSm / (512 / cols + 1) + 1);
  if (partial) *partial = (size_t)P.splits * P.units * cout * 128;
  return P;
}

void launch_wgrad(const WgradArgs& a, cudaStream_t st) {
  static std::once_flag once;
  std::call_once(once, [] {
    cudaFuncSetAttribute(wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgMaxSmem);
  });
  const WgradPlan& P = a.plan;
  launch_dependent(wgrad_kernel, dim3(P.splits * P.units), dim3(kConvThreads), P.smem, st, a);
  note_launches(1);
}

}  // namespace sweep
