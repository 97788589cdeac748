// Device code of the fused acoustic kernels (acoustic_fused.cu): one launch
// advances a tile by several time steps, every part of a step (stencil, CPML
// of both axes, source, receivers, boundary ring, and backward the imaging
// condition) in the one kernel.
//
// Why: on small grids a time step is bound by the fixed cost of its two
// launches (stencil, then CPML: 2.2 us each on GB300 however small the
// grid), not by its bytes.  A CTA takes its tile with a halo of 4 T cells per
// side (4 cells is the reach of one step, of the stencil and of the CPML
// memory variables alike), T steps on a region that shrinks by 4 cells a
// step, and writes the tile.  Neighbouring tiles recompute each other's
// halos, so no CTA waits for another and a launch needs no co-residency.
//
// A step of such a tile is a few hundred cycles of work, so what bounds it is
// the latency of a thread's own chain of instructions.  Hence a thread owns
// the same 4 cells of a row through all T steps and keeps everything that
// only they need in registers (the older wave field, K, the memory variables
// that no neighbour reads, the image), with its addresses and masks; shared
// memory holds what neighbours read (the wave field, psi or its adjoint's
// terms), double-buffered, with one barrier per step.  (Versions that dealt
// a step's cells out anew and kept the whole state in shared memory took
// 2.1 us per forward step on a 200 x 200 + 40 grid.)
//
// Layout: the extended tile has EZ x EX cells, cell (0, 0) at grid
// (z0 - 4 T, x0 - 4 T); shared arrays hold it with pitch EP, zero off the
// grid (the Dirichlet condition).  Its outermost 4 cells are only read.
#pragma once

#include "acoustic_common.cuh"
#include "tma.cuh"

namespace sweep {
namespace {

template <int T_, int BZ_, int BX_, int V_>
struct FusedTile {
  static constexpr int T = T_, BZ = BZ_, BX = BX_, V = V_;
  static constexpr int H = 4 * T;
  static constexpr int EZ = BZ + 2 * H, EX = BX + 2 * H;
  // pitch of the shared arrays: a warp that covers several rows of owned
  // cells (EX - 8 wide) reads them as if they were one line, without conflicts
  static constexpr int EP = (EX - 8 + 31) / 32 * 32 == EX - 8 ? EX : EX + 24, E = EZ * EP;
  // owned cells: all but the outermost 4, a thread per V of a row
  static constexpr int NG = (EX - 8) / V, NW = (EZ - 8) * NG;
  static constexpr int NT = (NW + 31) / 32 * 32;
  // the outermost 4: 4-cell groups
  static constexpr int EG = EX / 4, NR = 8 * EG + 2 * (EZ - 8);
  static_assert(V == 2 || V == 4, "cells of a thread");
  static_assert(BX % 4 == 0, "16-byte groups");
  static_assert(NT <= 1024, "threads");
  // group i of the outermost cells
  __device__ __forceinline__ static void rim(int i, int* r, int* c) {
    if (i < 8 * EG) {
      const int k = i / EG;
      *r = k < 4 ? k : EZ - 8 + k;
      *c = 4 * (i - k * EG);
    } else {
      const int k = i - 8 * EG;
      *r = 4 + k / 2;
      *c = k & 1 ? EX - 4 : 0;
    }
  }
};

// V cells as pairs: the packed FP32 instructions take two a time (a thread's
// chain of instructions is what a step waits for).
template <int V>
struct Vec {
  float2 v[V / 2];
  __device__ __forceinline__ float& operator[](int c) {
    return c & 1 ? v[c / 2].y : v[c / 2].x;
  }
};
__device__ __forceinline__ float2 two(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float a, float2 b, float2 c) {
  return __ffma2_rn(two(a), b, c);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(two(-1.f), b, a); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
// a + b as an atomic addition gives it: subnormal operands and sums are zero.
__device__ __forceinline__ float add_red(float a, float b) {
  float r;
  asm("add.rn.ftz.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 add_red(float2 a, float2 b) {
  return make_float2(add_red(a.x, b.x), add_red(a.y, b.y));
}
// a x + b y, the second product rounded on its own
__device__ __forceinline__ float2 lin2(float2 a, float2 x, float2 b, float2 y) {
  return __ffma2_rn(a, x, mul2(b, y));
}
template <int V>
__device__ __forceinline__ Vec<V> zerov() {
  Vec<V> r;
#pragma unroll
  for (int i = 0; i < V / 2; ++i) r.v[i] = two(0.f);
  return r;
}
template <int V>
__device__ __forceinline__ Vec<V> ldv(const float* p) {
  Vec<V> r;
  if constexpr (V == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    r.v[0] = make_float2(t.x, t.y);
    r.v[1] = make_float2(t.z, t.w);
  } else {
    r.v[0] = *reinterpret_cast<const float2*>(p);
  }
  return r;
}
template <int V>
__device__ __forceinline__ void stv(float* p, const Vec<V>& a) {
  if constexpr (V == 4)
    *reinterpret_cast<float4*>(p) = make_float4(a.v[0].x, a.v[0].y, a.v[1].x, a.v[1].y);
  else
    *reinterpret_cast<float2*>(p) = a.v[0];
}
__device__ __forceinline__ float4 ld16(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st16(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

__device__ __forceinline__ constexpr float c1w(int k) {  // weight of offset k > 0 in d1
  return k == 1 ? kD1 : k == 2 ? kD2 : k == 3 ? kD3 : kD4;
}
__device__ __forceinline__ constexpr float c2w(int k) {  // weight of offset +-k in d2
  return k == 0 ? kC0 : k == 1 ? kC1 : k == 2 ? kC2 : k == 3 ? kC3 : kC4;
}

// Sums of d2 and d1 (acoustic_common.cuh) term by term, k = 1 .. 4, with the
// roundings that those have in the per-step kernels.
__device__ __forceinline__ void acc_d2(float2& s, int k, float2 c, float2 sum) {
  s = fma2(c2w(k), sum, k == 1 ? mul2(two(kC0), c) : s);
}
__device__ __forceinline__ void acc_d1(float2& s, int k, float2 diff) {
  s = k == 1 ? diff : k == 2 ? fma2(c1w(1), s, mul2(two(c1w(2)), diff)) : fma2(c1w(k), diff, s);
}

// V cells of a row with 4 more on each side: pairs at even offsets as they
// lie in memory, and at odd ones
template <int V>
struct Row {
  float2 e[V / 2 + 4], o[V / 2 + 3];
  __device__ __forceinline__ void load(const float* p, const Vec<V>& own) {  // p: the first own cell
    if constexpr (V == 4) {
      const float4 l = ld16(p - 4), r = ld16(p + 4);
      e[0] = make_float2(l.x, l.y);
      e[1] = make_float2(l.z, l.w);
      e[4] = make_float2(r.x, r.y);
      e[5] = make_float2(r.z, r.w);
    } else {
      e[0] = ldv<2>(p - 4).v[0];
      e[1] = ldv<2>(p - 2).v[0];
      e[3] = ldv<2>(p + 2).v[0];
      e[4] = ldv<2>(p + 4).v[0];
    }
#pragma unroll
    for (int i = 0; i < V / 2; ++i) e[2 + i] = own.v[i];
    odd();
  }
  __device__ __forceinline__ void odd() {
#pragma unroll
    for (int i = 0; i < V / 2 + 3; ++i) o[i] = make_float2(e[i].y, e[i + 1].x);
  }
  __device__ __forceinline__ float2 at(int s) const { return s & 1 ? o[s / 2] : e[s / 2]; }
  __device__ __forceinline__ float2 d2(int i) const {  // of own pair i
    float2 s = two(0.f);
#pragma unroll
    for (int k = 1; k <= 4; ++k)
      acc_d2(s, k, at(4 + 2 * i), add2(at(4 + 2 * i + k), at(4 + 2 * i - k)));
    return s;
  }
  __device__ __forceinline__ float2 d1(int i) const {
    float2 s = two(0.f);
#pragma unroll
    for (int k = 1; k <= 4; ++k) acc_d1(s, k, sub2(at(4 + 2 * i + k), at(4 + 2 * i - k)));
    return s;
  }
};

// Index of ring cell (zi, xi) (interior coordinates; the order of
// ring_cell, acoustic_cpml.cuh), -1 off the ring.
__device__ __forceinline__ int ring_index(const Geom& g, int zi, int xi) {
  const int w = g.ringw, W = g.nx + 2 * w;
  if (zi < -w || zi >= g.nz + w || xi < -w || xi >= g.nx + w) return -1;
  if (zi < 0) return (zi + w) * W + xi + w;
  if (zi >= g.nz) return (w + zi - g.nz) * W + xi + w;
  if (xi < 0) return 2 * w * W + zi * w + xi + w;
  if (xi >= g.nx) return 2 * w * W + g.nz * w + zi * w + (xi - g.nx);
  return -1;
}

// The receivers of this shot in rows [r0, r1) x columns [c0, c1) of the
// extended tile: (cell offset, receiver) pairs, any order.
template <class C>
__device__ __forceinline__ void list_receivers(const Geom& g, const int32_t* rec, int s, int oz,
                                               int ox, int r0, int r1, int c0, int c1,
                                               int2* list, int* count) {
  for (int i = threadIdx.x; i < g.nrec; i += C::NT) {
    const long long k = 2 * ((long long)s * g.nrec + i);
    const int r = rec[k] + g.P - oz, c = rec[k + 1] + g.P - ox;
    if (r >= r0 && r < r1 && c >= c0 && c < c1)
      list[atomicAdd(count, 1)] = make_int2(r * C::EP + c, i);
  }
}

__device__ __forceinline__ void copy_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_async_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// The columns a launch reads and writes: the grid's, to a whole 4-cell group.
// (Those beyond, up to the row pitch, belong to no tile.)
__device__ __forceinline__ int grid_end(const Geom& g) { return (g.NX + 3) & ~3; }

// Computes an address before the wait for the previous launch, not after it.
__device__ __forceinline__ const float* pin(const float* p) {
  asm volatile("" : "+l"(p));
  return p;
}

// What a thread owns: V cells of row r from column col of the extended tile.
template <class C>
struct FusedCells {
  int r, col, o;     // row, column, offset in the shared arrays
  int gz, gx;        // grid position
  bool in, own;      // on the grid; in the CTA's own tile
  int last;          // last step of the launch that still needs these cells
  long long go;      // offset in the shot's fields
  __device__ __forceinline__ FusedCells(const Geom& g, int s, int oz, int ox, int steps) {
    const int b = threadIdx.x / C::NG;
    r = 4 + b;
    col = 4 + C::V * (threadIdx.x - b * C::NG);
    o = r * C::EP + col;
    gz = oz + r;
    gx = ox + col;
    const bool w = C::NW == C::NT || (int)threadIdx.x < C::NW;
    in = w && gz >= 0 && gz < g.NZ && gx >= 0 && gx < grid_end(g);
    const int dz = max(C::H - r, r - (C::H + C::BZ - 1));
    const int dx = max(C::H - col, col - (C::H + C::BX - C::V));  // 4-cell steps count

    const int d = max(max(dz, dx), 0);
    own = in && d == 0;
    last = in ? steps - 1 - (d + 3) / 4 : -1;
    go = (long long)s * g.fstride + (long long)gz * g.NXp + gx;
  }
};

// ------------------------------------------------------------------ forward
template <class C>
struct alignas(16) FusedFwdSmem {  // (the receiver list follows it)
  float u[2][C::E], pz[2][C::E], px[2][C::E];
  float fn[C::T];
  int nrec;
};

template <class C>
__device__ __forceinline__ void fused_fwd_body(const AcFusedArgs& a, FusedFwdSmem<C>& m,
                                               int2* list) {
  constexpr int V = C::V, VP = V / 2;
  typedef Vec<V> vec;
  const Geom& g = a.g;
  const int tid = threadIdx.x, s = blockIdx.z;
  const int x0 = blockIdx.x * C::BX, z0 = blockIdx.y * C::BZ;
  const int ox = x0 - C::H, oz = z0 - C::H;
  // do the owned cells meet a strip?
  const bool zb = g.P > 0 && (oz + 4 < g.P || oz + C::EZ - 4 > g.P + g.nz);
  const bool xb = g.P > 0 && (ox + 4 < g.P || ox + C::EX - 4 > g.P + g.nx);
  // prologue: only the call's inputs, so it overlaps the previous launch
  if (tid == 0) m.nrec = 0;
  __syncthreads();
  grid_dep_trigger();
  if (a.data)
    list_receivers<C>(g, a.rec, s, oz, ox, C::H, C::H + C::BZ, C::H, C::H + C::BX, list, &m.nrec);
  if (tid < a.steps) m.fn[tid] = a.wavelet[(long long)s * g.nt + a.n + tid];
  const FusedCells<C> q(g, s, oz, ox, a.steps);
  const bool zs = zb && q.in && z_border(g, q.gz);
  const bool xs = xb && q.in && (q.gx < g.P || q.gx + V - 1 >= g.P + g.nx);
  const int srow = a.src[2 * s] + g.P - oz, scol = a.src[2 * s + 1] + g.P - ox;
  const int sc = srow == q.r && scol >= q.col && scol < q.col + V ? scol - q.col : -1;
  int ri[V];
  bool ring = false;
  unsigned xm = 0;  // cells of an x strip
#pragma unroll
  for (int c = 0; c < V; ++c) {
    ri[c] = a.save && q.own ? ring_index(g, q.gz - g.P, q.gx + c - g.P) : -1;
    ring = ring || ri[c] >= 0;
    xm |= (x_border(g, q.gx + c) ? 1u : 0u) << c;
  }
  const float *pu = pin(a.ui + q.go), *pup = pin(a.upi + q.go),
              *pk = pin(a.K + (long long)q.gz * g.NXp + q.gx), *ppz = pin(a.pzi + q.go),
              *pzz = pin(a.zzi + q.go), *ppx = pin(a.pxi + q.go), *pzx = pin(a.zxi + q.go);
  grid_dep_wait();
  const int status = *a.status;
  // All loads of a launch are issued before the first use: the owned cells'
  // state to registers (u^n and psi go on to shared memory), u^n and psi of
  // the outermost cells to shared memory.
  const vec zv = zerov<V>();
  vec uc = zv, up = zv, kk = zv, pz = zv, zz = zv, px = zv, zx = zv, A = zv, B = zv;
  float Az = 0.f, Bz = 0.f;
  if (q.in) {
    uc = ldv<V>(pu);
    up = ldv<V>(pup);
    kk = ldv<V>(pk);
  }
  if (zs) {
    pz = ldv<V>(ppz);
    zz = ldv<V>(pzz);
    Az = a.az[q.gz];
    Bz = a.bz[q.gz];
  }
  if (xs) {
    px = ldv<V>(ppx);
    zx = ldv<V>(pzx);
    A = ldv<V>(a.ax + q.gx);
    B = ldv<V>(a.bx + q.gx);
  }
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int i = tid; i < C::NR; i += C::NT) {
    int r, c;
    C::rim(i, &r, &c);
    const int z = oz + r, x = ox + c, o = r * C::EP + c;
    const bool in = z >= 0 && z < g.NZ && x >= 0 && x < grid_end(g);
    const long long k = (long long)s * g.fstride + (long long)z * g.NXp + x;
    const float4 u = in ? ld16(a.ui + k) : z4;
    const float4 p = zb && in && z_border(g, z) ? ld16(a.pzi + k) : z4;
    const float4 w = xb && in && (x < g.P || x + 3 >= g.P + g.nx) ? ld16(a.pxi + k) : z4;
    st16(m.u[0] + o, u);
    if (zb) st16(m.pz[0] + o, p);
    if (xb) st16(m.px[0] + o, w);
  }
  if (C::NW == C::NT || tid < C::NW) {  // (off the grid, and psi off the strips: zero for good)
    stv<V>(m.u[0] + q.o, uc);
    if (!q.in) stv<V>(m.u[1] + q.o, zv);
    if (zb) {
      stv<V>(m.pz[0] + q.o, pz);
      if (!zs) stv<V>(m.pz[1] + q.o, zv);
    }
    if (xb) {
      stv<V>(m.px[0] + q.o, px);
      if (!xs) stv<V>(m.px[1] + q.o, zv);
    }
  }
  if (__syncthreads_or(status != 0)) return;  // the call has failed already
  const int nl = a.data ? m.nrec : 0;
  int cur = 0;
#pragma unroll 1
  for (int j = 0; j < a.steps; ++j) {
    const int n = a.n + j;
    if (ring) {  // the ring cells of u^n into their slot
      float* sv = a.save + ((long long)n * g.nshot + s) * g.nring;
#pragma unroll
      for (int c = 0; c < V; ++c)
        if (ri[c] >= 0) sv[ri[c]] = uc[c];
    }
    if (j <= q.last) {
      const float* U = m.u[cur] + q.o;
      Row<V> e;
      e.load(U, uc);
      // the plain update, then each axis' CPML term added, as the stencil and
      // CPML kernels do it: the same roundings.  (In a corner those add the two
      // terms in either order, but nearly always x first: an x thread has one
      // addition for its 4 cells, a z thread one per row.)
      float2 L[VP], tz[VP], tx[VP];
#pragma unroll
      for (int i = 0; i < VP; ++i) {
        L[i] = tz[i] = tx[i] = two(0.f);
      }
      if (zs) {
        float2 d1u[VP], dp[VP];
        const float* Q = m.pz[cur] + q.o;
#pragma unroll
        for (int i = 0; i < VP; ++i) d1u[i] = dp[i] = two(0.f);
#pragma unroll
        for (int k = 1; k <= 4; ++k) {
          const vec lo = ldv<V>(U - k * C::EP), hi = ldv<V>(U + k * C::EP);
          const vec pl = ldv<V>(Q - k * C::EP), ph = ldv<V>(Q + k * C::EP);
#pragma unroll
          for (int i = 0; i < VP; ++i) {
            acc_d2(L[i], k, uc.v[i], add2(hi.v[i], lo.v[i]));
            acc_d1(d1u[i], k, sub2(hi.v[i], lo.v[i]));
            acc_d1(dp[i], k, sub2(ph.v[i], pl.v[i]));
          }
        }
#pragma unroll
        for (int i = 0; i < VP; ++i) {
          zz.v[i] = lin2(two(Az), zz.v[i], two(Bz), add2(L[i], dp[i]));
          pz.v[i] = lin2(two(Bz), d1u[i], two(Az), pz.v[i]);
          tz[i] = mul2(kk.v[i], add2(dp[i], zz.v[i]));
        }
        stv<V>(m.pz[cur ^ 1] + q.o, pz);
      } else {
#pragma unroll
        for (int k = 1; k <= 4; ++k) {
          const vec lo = ldv<V>(U - k * C::EP), hi = ldv<V>(U + k * C::EP);
#pragma unroll
          for (int i = 0; i < VP; ++i) acc_d2(L[i], k, uc.v[i], add2(hi.v[i], lo.v[i]));
        }
      }
      if (xs) {
        Row<V> p;
        p.load(m.px[cur] + q.o, px);
#pragma unroll
        for (int i = 0; i < VP; ++i) {
          const float2 d2u = e.d2(i), dp = p.d1(i);
          // zero off the strip (a = b = 0)
          zx.v[i] = lin2(A.v[i], zx.v[i], B.v[i], add2(d2u, dp));
          px.v[i] = lin2(A.v[i], px.v[i], B.v[i], e.d1(i));
          tx[i] = mul2(kk.v[i], add2(dp, zx.v[i]));
          if (!((xm >> (2 * i)) & 1u)) tx[i].x = 0.f;
          if (!((xm >> (2 * i + 1)) & 1u)) tx[i].y = 0.f;
          L[i] = add2(L[i], d2u);
        }
        stv<V>(m.px[cur ^ 1] + q.o, px);
      } else {
#pragma unroll
        for (int i = 0; i < VP; ++i) L[i] = add2(L[i], e.d2(i));
      }
      vec out;
#pragma unroll
      for (int i = 0; i < VP; ++i)
        out.v[i] = fma2(kk.v[i], L[i], sub2(add2(uc.v[i], uc.v[i]), up.v[i]));
      if (sc >= 0) {
        const float fn = m.fn[j];
#pragma unroll
        for (int c = 0; c < V; ++c)
          if (c == sc) out[c] += kk[c] * fn;
      }
#pragma unroll
      for (int i = 0; i < VP; ++i) {
        if (xs) out.v[i] = add_red(out.v[i], tx[i]);
        if (zs) out.v[i] = add_red(out.v[i], tz[i]);
      }
      stv<V>(m.u[cur ^ 1] + q.o, out);
      up = uc;
      uc = out;
    }
    __syncthreads();
    // traces of u^{n+1} (the next step writes the other buffer)
    for (int i = tid; i < nl; i += C::NT)
      a.data[((long long)s * g.nrec + list[i].y) * g.nt + n] = m.u[cur ^ 1][list[i].x];
    cur ^= 1;
  }
  // the tile's state: u^{n+steps}, u^{n+steps-1}, and the strips' memory variables
  if (q.own) {
    stv<V>(a.uo + q.go, uc);
    stv<V>(a.upo + q.go, up);
    if (zs) {
      stv<V>(a.pzo + q.go, pz);
      stv<V>(a.zzo + q.go, zz);
    }
    if (xs) {
      stv<V>(a.pxo + q.go, px);
      stv<V>(a.zxo + q.go, zx);
    }
  }
}

// ----------------------------------------------------------------- backward
// Per axis C = b (mu^{n+1} + zetabar^n) and D = b psibar^n in the strips
// (zero elsewhere): what a cell's neighbours need of its memory variables.
template <class C>
struct alignas(16) FusedBwdSmem {
  float mu[2][C::E], u[2][C::E];
  float cz[2][C::E], dz[2][C::E], cx[2][C::E], dx[2][C::E];
  float inj[2][C::E];             // residual to inject, per step parity
  float ring[C::T][C::NW * C::V];  // u^{n-1} of the owned ring cells, per step
  float fn[C::T];
  int nrec;
};

template <class C>
__device__ __forceinline__ void fused_bwd_body(const AcFusedArgs& a, FusedBwdSmem<C>& m,
                                               int2* list, float* rres) {
  constexpr int V = C::V, VP = V / 2;
  typedef Vec<V> vec;
  const Geom& g = a.g;
  const int tid = threadIdx.x, s = blockIdx.z;
  const int x0 = blockIdx.x * C::BX, z0 = blockIdx.y * C::BZ;
  const int ox = x0 - C::H, oz = z0 - C::H;
  // does the extended tile meet a strip (its memory variables reach the 4
  // cells next to it), or the interior (u needed; a tile whose own cells hold
  // only ring cells restores them for its neighbours)?
  const bool zb = g.P > 0 && (oz < g.P || oz + C::EZ > g.P + g.nz);
  const bool xb = g.P > 0 && (ox < g.P || ox + C::EX > g.P + g.nx);
  const bool ub = a.imaging && oz + C::EZ > g.P && oz < g.P + g.nz && ox + C::EX > g.P &&
                  ox < g.P + g.nx;
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  if (tid == 0) m.nrec = 0;
  __syncthreads();
  grid_dep_trigger();
  if (a.res) {  // injected by every tile that owns or recomputes the receiver's cell
    list_receivers<C>(g, a.rec, s, oz, ox, 4, C::EZ - 4, 4, C::EX - 4, list, &m.nrec);
    for (int i = 4 * tid; i < C::E; i += 4 * C::NT) {
      st16(m.inj[0] + i, z4);
      st16(m.inj[1] + i, z4);
    }
  }
  if (tid < a.steps) {
    const int n = a.n - tid;
    m.fn[tid] = a.imaging && n < g.nt ? a.wavelet[(long long)s * g.nt + n] : 0.f;
  }
  const FusedCells<C> q(g, s, oz, ox, a.steps);
  const bool zs = zb && q.in && z_border(g, q.gz);
  const bool zn = zb && q.in && (q.gz < g.P + 4 || q.gz >= g.P + g.nz - 4);  // zs or next to it
  const bool xn = xb && q.in && ((q.gx & ~3) < g.P + 4 || (q.gx | 3) >= g.P + g.nx - 4);
  unsigned zm = 0, xm = 0, im = 0, rm = 0;  // strip rows / columns of the windows, interior, ring
  if (zn)
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const int z = q.gz - 4 + k;
      zm |= (z >= 0 && z < g.NZ && z_border(g, z) ? 1u : 0u) << k;
    }
  if (xn)
#pragma unroll
    for (int k = 0; k < V + 8; ++k) {
      const int x = q.gx - 4 + k;
      xm |= (x >= 0 && x < g.NX && x_border(g, x) ? 1u : 0u) << k;
    }
  const bool xs = (xm >> 4) & ((1u << V) - 1);
  int ri[V];
#pragma unroll
  for (int c = 0; c < V; ++c) {
    if (ub && q.in && interior(g, q.gz, q.gx + c)) im |= 1u << c;
    ri[c] = ub && q.in ? ring_index(g, q.gz - g.P, q.gx + c - g.P) : -1;
    rm |= (ri[c] >= 0 ? 1u : 0u) << c;
  }
  const int srow = a.src[2 * s] + g.P - oz, scol = a.src[2 * s + 1] + g.P - ox;
  const int sc = srow == q.r && scol >= q.col && scol < q.col + V ? scol - q.col : -1;
  const float *pm = pin(a.mi + q.go), *pmp = pin(a.mpi + q.go),
              *pk = pin(a.K + (long long)q.gz * g.NXp + q.gx), *pu = pin(a.ui + q.go),
              *pup = pin(a.upi + q.go), *pgr = pin(a.graw + q.go), *ppz = pin(a.pzi + q.go),
              *pzz = pin(a.zzi + q.go), *ppx = pin(a.pxi + q.go), *pzx = pin(a.zxi + q.go);
  grid_dep_wait();
  const int status = *a.status;
  // all loads before the first use, as in the forward kernel
  const vec zv = zerov<V>();
  vec mc = zv, mp = zv, kk = zv, uc = zv, up = zv, gr = zv, il = zv, pz = zv, zz = zv, px = zv,
      zx = zv, A = zv, B = zv;
  float Az = 0.f, Bz = 0.f;
  if (q.in) {
    mc = ldv<V>(pm);
    mp = ldv<V>(pmp);
    kk = ldv<V>(pk);
    if (ub) {
      uc = ldv<V>(pu);
      up = ldv<V>(pup);
      if (q.own) {
        gr = ldv<V>(pgr);
        if (a.illum) il = ldv<V>(a.illum + q.go);
      }
    }
  }
  if (zs) {
    pz = ldv<V>(ppz);
    zz = ldv<V>(pzz);
    Az = a.az[q.gz];
    Bz = a.bz[q.gz];
  }
  if (xs) {
    px = ldv<V>(ppx);
    zx = ldv<V>(pzx);
    A = ldv<V>(a.ax + q.gx);
    B = ldv<V>(a.bx + q.gx);
  }
  if (rm)
    for (int j = 0; j < a.steps; ++j) {  // u^{n-1} of the ring, from the forward's save
      const int n = a.n - j;
      if (n >= 1 && n <= g.nt - 1) {
#pragma unroll
        for (int c = 0; c < V; ++c)
          if (ri[c] >= 0)
            copy_async4(&m.ring[j][V * tid + c],
                        a.save + ((long long)(n - 1) * g.nshot + s) * g.nring + ri[c]);
      }
    }
  __syncthreads();  // the receiver list is complete
  const int nl = a.res ? m.nrec : 0;
  for (int i = tid; i < nl * C::T; i += C::NT) {  // the residual samples r^{n-1}
    const int k = i / C::T, j = i - k * C::T, n = a.n - j;
    if (j < a.steps && n >= 1)
      copy_async4(rres + i, a.res + ((long long)s * g.nrec + list[k].y) * g.nt + n - 1);
  }
  for (int i = tid; i < C::NR; i += C::NT) {
    int r, c;
    C::rim(i, &r, &c);
    const int z = oz + r, x = ox + c, o = r * C::EP + c;
    const bool in = z >= 0 && z < g.NZ && x >= 0 && x < grid_end(g);
    const long long k = (long long)s * g.fstride + (long long)z * g.NXp + x;
    const bool zr = zb && in && z_border(g, z);
    const bool xr = xb && in && (x < g.P || x + 3 >= g.P + g.nx);
    const float4 mu = in ? ld16(a.mi + k) : z4;
    const float4 u = ub && in ? ld16(a.ui + k) : z4;
    const float4 e = zr ? ld16(a.zzi + k) : z4, f = zr ? ld16(a.pzi + k) : z4;
    const float bz = zr ? a.bz[z] : 0.f;
    const float4 v = xr ? ld16(a.zxi + k) : z4, w = xr ? ld16(a.pxi + k) : z4;
    const float4 b = xr ? ld16(a.bx + x) : z4;
    st16(m.mu[0] + o, mu);
    if (ub) st16(m.u[0] + o, u);
    if (zb) {
      st16(m.cz[0] + o, make_float4(bz * (mu.x + e.x), bz * (mu.y + e.y), bz * (mu.z + e.z),
                                    bz * (mu.w + e.w)));
      st16(m.dz[0] + o, make_float4(bz * f.x, bz * f.y, bz * f.z, bz * f.w));
    }
    if (xb) {
      st16(m.cx[0] + o, make_float4(b.x * (mu.x + v.x), b.y * (mu.y + v.y), b.z * (mu.z + v.z),
                                    b.w * (mu.w + v.w)));
      st16(m.dx[0] + o, make_float4(b.x * w.x, b.y * w.y, b.z * w.z, b.w * w.w));
    }
  }
  // C and D of the owned cells (zero off the strips) from the memory variables
  auto put_z = [&](int buf) {
    vec cv, dv;
#pragma unroll
    for (int i = 0; i < VP; ++i) {
      cv.v[i] = mul2(two(Bz), add2(mc.v[i], zz.v[i]));
      dv.v[i] = mul2(two(Bz), pz.v[i]);
    }
    stv<V>(m.cz[buf] + q.o, cv);
    stv<V>(m.dz[buf] + q.o, dv);
  };
  auto put_x = [&](int buf) {
    vec cv, dv;
#pragma unroll
    for (int i = 0; i < VP; ++i) {
      cv.v[i] = mul2(B.v[i], add2(mc.v[i], zx.v[i]));
      dv.v[i] = mul2(B.v[i], px.v[i]);
    }
    stv<V>(m.cx[buf] + q.o, cv);
    stv<V>(m.dx[buf] + q.o, dv);
  };
  if (C::NW == C::NT || tid < C::NW) {
    stv<V>(m.mu[0] + q.o, mc);
    if (ub) stv<V>(m.u[0] + q.o, uc);
    if (!q.in) stv<V>(m.mu[1] + q.o, zv);  // off the grid: zero for good
    if (!(im | rm)) stv<V>(m.u[1] + q.o, zv);
    if (zb) {
      put_z(0);
      if (!zs) put_z(1);
    }
    if (xb) {
      put_x(0);
      if (!xs) put_x(1);
    }
  }
  copy_async_wait();
  if (__syncthreads_or(status != 0)) return;  // the call has failed already
  if (nl > 0) {  // the first step's residual
    for (int i = tid; i < nl; i += C::NT)
      if (a.n >= 1) atomicAdd(&m.inj[0][list[i].x], rres[i * C::T]);
    __syncthreads();
  }
  int cur = 0, ucur = 0;
#pragma unroll 1
  for (int j = 0; j < a.steps; ++j) {
    const int n = a.n - j;
    const bool adj = n >= 1, img = ub && n <= g.nt - 1, rec = img && adj;
    const bool need = j <= q.last;
    if (nl > 0 && j + 1 < a.steps && n - 1 >= 1)  // the next step's residual
      for (int i = tid; i < nl; i += C::NT)
        atomicAdd(&m.inj[(j + 1) & 1][list[i].x], rres[i * C::T + j + 1]);
    if (a.wgrad && sc >= 0 && q.own && n < g.nt) {  // f-bar^n = mu^{n+1}(s)
      float v = mc[0];
#pragma unroll
      for (int c = 1; c < V; ++c) v = c == sc ? mc[c] : v;
      a.wgrad[(long long)s * g.nt + n] = v;
    }
    if (img && need && (im | rm)) {
      // u^{n-1}: the interior runs backwards, the ring comes from the save
      vec out = zv;
      if (im) {
        const float* U = m.u[ucur] + q.o;
        Row<V> e;
        e.load(U, uc);
        vec lap;
#pragma unroll
        for (int i = 0; i < VP; ++i) lap.v[i] = two(0.f);
#pragma unroll
        for (int k = 1; k <= 4; ++k) {
          const vec lo = ldv<V>(U - k * C::EP), hi = ldv<V>(U + k * C::EP);
#pragma unroll
          for (int i = 0; i < VP; ++i) acc_d2(lap.v[i], k, uc.v[i], add2(hi.v[i], lo.v[i]));
        }
#pragma unroll
        for (int i = 0; i < VP; ++i) lap.v[i] = add2(lap.v[i], e.d2(i));
        if (sc >= 0) {
          const float fn = m.fn[j];
#pragma unroll
          for (int c = 0; c < V; ++c)
            if (c == sc) lap[c] += fn;
        }
#pragma unroll
        for (int c = 0; c < V; ++c) {
          if ((im >> c) & 1u) {
            gr[c] += mc[c] * lap[c];  // written for own cells only
            il[c] += uc[c] * uc[c];
            out[c] = 2.f * uc[c] - up[c] + kk[c] * lap[c];
          }
        }
      }
      if (rec) {
        if (rm) {
#pragma unroll
          for (int c = 0; c < V; ++c)
            if ((rm >> c) & 1u) out[c] = m.ring[j][V * tid + c];
        }
        stv<V>(m.u[ucur ^ 1] + q.o, out);
        up = uc;
        uc = out;
      }
    }
    if (adj && need) {
      const float* M = m.mu[cur] + q.o;
      Row<V> e;
      e.load(M, mc);
      // the plain update, then each axis' CPML terms added, then the residual:
      // the roundings of the per-step kernels
      float2 L[VP], tz[VP], tx[VP];
#pragma unroll
      for (int i = 0; i < VP; ++i) L[i] = tz[i] = tx[i] = two(0.f);
      if (zn) {
        const float *Q = m.cz[cur] + q.o, *D = m.dz[cur] + q.o;
        float2 sC[VP], sD[VP], sG[VP];  // d2 C, d1 D, -d1 (m G)
#pragma unroll
        for (int i = 0; i < VP; ++i) sC[i] = sD[i] = sG[i] = two(0.f);
#pragma unroll
        for (int k = 1; k <= 4; ++k) {
          const vec lo = ldv<V>(M - k * C::EP), hi = ldv<V>(M + k * C::EP);
          const vec cl = ldv<V>(Q - k * C::EP), ch = ldv<V>(Q + k * C::EP);
          const vec dl = ldv<V>(D - k * C::EP), dh = ldv<V>(D + k * C::EP);
          const bool ml = (zm >> (4 - k)) & 1u, mh = (zm >> (4 + k)) & 1u;
#pragma unroll
          for (int i = 0; i < VP; ++i) {
            acc_d2(L[i], k, mc.v[i], add2(hi.v[i], lo.v[i]));
            acc_d2(sC[i], k, mul2(two(Bz), add2(mc.v[i], zz.v[i])), add2(ch.v[i], cl.v[i]));
            acc_d1(sD[i], k, sub2(dh.v[i], dl.v[i]));
            const float2 gh = add2(hi.v[i], ch.v[i]), gl = add2(lo.v[i], cl.v[i]);
            acc_d1(sG[i], k, sub2(ml ? gl : two(0.f), mh ? gh : two(0.f)));
          }
        }
#pragma unroll
        for (int i = 0; i < VP; ++i) {
          tz[i] = mul2(kk.v[i], sub2(sC[i], sD[i]));
          if (zs) {
            pz.v[i] = fma2(Az, pz.v[i], sG[i]);
            zz.v[i] = mul2(two(Az), add2(mc.v[i], zz.v[i]));
          }
        }
      } else {
#pragma unroll
        for (int k = 1; k <= 4; ++k) {
          const vec lo = ldv<V>(M - k * C::EP), hi = ldv<V>(M + k * C::EP);
#pragma unroll
          for (int i = 0; i < VP; ++i) acc_d2(L[i], k, mc.v[i], add2(hi.v[i], lo.v[i]));
        }
      }
#pragma unroll
      for (int i = 0; i < VP; ++i) L[i] = add2(L[i], e.d2(i));
      if (xn) {
        vec own;
        Row<V> c, d;
#pragma unroll
        for (int i = 0; i < VP; ++i) own.v[i] = mul2(B.v[i], px.v[i]);
        d.load(m.dx[cur] + q.o, own);
#pragma unroll
        for (int i = 0; i < VP; ++i) own.v[i] = mul2(B.v[i], add2(mc.v[i], zx.v[i]));
        c.load(m.cx[cur] + q.o, own);
#pragma unroll
        for (int i = 0; i < VP; ++i) tx[i] = mul2(kk.v[i], sub2(c.d2(i), d.d1(i)));
        if (xs) {
#pragma unroll
          for (int k = 0; k < VP + 4; ++k) {  // -m (mu + C)
            c.e[k] = mul2(two(-1.f), add2(c.e[k], e.e[k]));
            if (!((xm >> (2 * k)) & 1u)) c.e[k].x = 0.f;
            if (!((xm >> (2 * k + 1)) & 1u)) c.e[k].y = 0.f;
          }
          c.odd();
#pragma unroll
          for (int i = 0; i < VP; ++i) {
            const float2 p = fma2(A.v[i], px.v[i], c.d1(i));
            const float2 t = mul2(A.v[i], add2(mc.v[i], zx.v[i]));
            const bool mx = (xm >> (4 + 2 * i)) & 1u, my = (xm >> (5 + 2 * i)) & 1u;
            px.v[i] = make_float2(mx ? p.x : 0.f, my ? p.y : 0.f);
            zx.v[i] = make_float2(mx ? t.x : 0.f, my ? t.y : 0.f);
          }
        }
      }
      vec out;
#pragma unroll
      for (int i = 0; i < VP; ++i)
        out.v[i] = fma2(kk.v[i], L[i], sub2(add2(mc.v[i], mc.v[i]), mp.v[i]));
#pragma unroll
      for (int i = 0; i < VP; ++i) {
        if (xn) out.v[i] = add_red(out.v[i], tx[i]);
        if (zn) out.v[i] = add_red(out.v[i], tz[i]);
      }
      if (nl > 0) {  // mu^n(r) += K(r) r^{n-1}
        float* I = m.inj[j & 1] + q.o;
        vec v = ldv<V>(I);
        bool any = false;
#pragma unroll
        for (int c = 0; c < V; ++c) any = any || v[c] != 0.f;
        if (any) {
#pragma unroll
          for (int c = 0; c < V; ++c)
            if (v[c] != 0.f) out[c] = add_red(out[c], __fmul_rn(kk[c], v[c]));
          stv<V>(I, zv);
        }
      }
      stv<V>(m.mu[cur ^ 1] + q.o, out);
      mp = mc;
      mc = out;
      if (zs) put_z(cur ^ 1);
      if (xs) put_x(cur ^ 1);
    }
    __syncthreads();
    if (adj) cur ^= 1;
    if (adj && a.imaging && n <= g.nt - 1) ucur ^= 1;
  }
  if (q.own) {
    stv<V>(a.mo + q.go, mc);
    stv<V>(a.mpo + q.go, mp);
    if (ub) {
      stv<V>(a.uo + q.go, uc);
      stv<V>(a.upo + q.go, up);
      stv<V>(a.graw + q.go, gr);
      if (a.illum) stv<V>(a.illum + q.go, il);
    }
    if (zs) {
      stv<V>(a.pzo + q.go, pz);
      stv<V>(a.zzo + q.go, zz);
    }
    if (xs) {
      stv<V>(a.pxo + q.go, px);
      stv<V>(a.zxo + q.go, zx);
    }
  }
}

}  // namespace
}  // namespace sweep
