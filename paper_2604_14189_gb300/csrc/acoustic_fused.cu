// Fused acoustic kernels (see acoustic_fused.cuh): the launch variants and
// the rule that chooses one of them, or the per-step stencil + CPML kernels,
// for a problem.
#include <algorithm>
#include <climits>

#include "acoustic_fused.cuh"

namespace sweep {
namespace {

template <class C, int RES>
__global__ void __launch_bounds__(C::NT, RES)
    ac_fused_fwd_kernel(const __grid_constant__ AcFusedArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  FusedFwdSmem<C>& m = *reinterpret_cast<FusedFwdSmem<C>*>(smem_raw);
  fused_fwd_body<C>(a, m, reinterpret_cast<int2*>(&m + 1));
}

template <class C, int RES>
__global__ void __launch_bounds__(C::NT, RES)
    ac_fused_bwd_kernel(const __grid_constant__ AcFusedArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  FusedBwdSmem<C>& m = *reinterpret_cast<FusedBwdSmem<C>*>(smem_raw);
  int2* list = reinterpret_cast<int2*>(&m + 1);
  fused_bwd_body<C>(a, m, list, reinterpret_cast<float*>(list + (a.res ? a.g.nrec : 0)));
}

struct Variant {
  FusedShape s;
  int res;                 // CTAs per SM
  int waves;               // most waves it is used for in a gradient (else one)
  int alone;               // most tiles of a shot outside of a gradient
  int threads;
  size_t smem, rec_bytes;  // fixed shared memory, and more per receiver
  void (*kernel)(const AcFusedArgs);
};

template <int T, int BZ, int BX, int V, int RES, int WAVES>
Variant fwd_variant() {
  using C = FusedTile<T, BZ, BX, V>;
  return {{T, BZ, BX}, RES, WAVES, INT_MAX, C::NT, sizeof(FusedFwdSmem<C>), sizeof(int2),
          ac_fused_fwd_kernel<C, RES>};
}
template <int T, int BZ, int BX, int V, int RES, int ALONE = INT_MAX>
Variant bwd_variant() {
  using C = FusedTile<T, BZ, BX, V>;
  return {{T, BZ, BX}, RES, 1, ALONE, C::NT, sizeof(FusedBwdSmem<C>), sizeof(int2) + 4 * T,
          ac_fused_bwd_kernel<C, RES>};
}

// Fastest first.  A launch costs about the same however few of its CTAs'
// slots are used, so the variant with the most steps per launch whose CTAs
// still run at once is the fastest: us per step on GB300 (200 x 200 + 40
// grids of 1, 2, 3, 4, 6, 8 shots; the 141 x 187 + 23 grid of 3 for the second
// variants) against the stencil + CPML kernels' 4.4, 4.5, 4.6, 5.1, 6.3, 7.1
// forward and 8.7, 8.6, 8.7, 9.0, 9.7, 13.0 backward (with illumination):
//   forward   3 steps, 24 x 24, one CTA per SM: 1.9 | 3.4 | 4.7 | 6.0 | 8.5
//             2 steps, 32 x 32, one: 2.3 (141 x 187)
//             2 steps, 24 x 24, two: 2.5 | 2.5 | 3.7 | 4.2 | 5.9
//             2 steps, 24 x 24, three: 3.1 | 3.1 | 3.2 | 4.5 | 5.3 | 6.8
//   backward  2 steps, 24 x 24, one: 4.0 | 6.5 | 8.7
//             2 steps, 32 x 32, one: 5.0 (141 x 187)
//             1 step, 16 x 32, three: 5.8 | 5.7 | 8.6 | 9.3
//             1 step, 32 x 32, two: 6.6 | 6.8 | 6.6 | 9.6
// (The register limits that let these CTAs share an SM cost spills: forward, three
// CTAs of 24 x 24, 136 bytes at 80 registers, the others 12 to 24 at 128; backward,
// 32 x 32, 44 and 32 bytes at 128, the other two none.)
// Past one wave the per-step kernels, which pipeline their loads, are as fast
// or faster: 301 x 901 + 40 with 20 shots takes them 26.6 us forward against
// 61.  A second wave of the last forward variant pays where the forward saves
// its ring (the per-step kernels do that at a cost, these at none): gradients
// on 36 random grids of 457 to 912 CTAs take 1.0 to 1.3 times as long without
// it; forward runs alone 0.92 to 1.4 times (352 x 401 + 29, 2 shots: 4.8 us a
// step against 5.1), so they don't take it.  The last backward variant, without
// the imaging that it takes along in a gradient, is faster than the per-step
// kernels only on shots of a few tiles, whose cells are mostly border.  An adjoint
// of 300 steps with 30 and 1000 receivers a shot takes, fused against per step, of
// 4 tiles (72 shots) 1.70 against 2.11 and 2.15 against 2.72 ms, of 9 (32 shots)
// 1.65 : 1.90 and 1.94 : 2.07, of 70 (4 shots) 1.45 : 1.51 and 1.67 : 1.52, of 255
// 1.44 : 1.32 and 1.55 : 1.36.  Whole calls: 200 x 200 + 40 forward, 1000
// steps, 4.40 -> 1.91 ms; 141 x 187 + 23 gradient, 3 shots, 900 steps, 10.8 ->
// 6.0 ms.
const Variant* variants(int dir, int* n) {
  static const Variant f[] = {fwd_variant<3, 24, 24, 4, 1, 1>(), fwd_variant<2, 32, 32, 4, 1, 1>(),
                              fwd_variant<2, 24, 24, 4, 2, 1>(), fwd_variant<2, 24, 24, 4, 3, 2>()};
  static const Variant b[] = {bwd_variant<2, 24, 24, 2, 1>(), bwd_variant<2, 32, 32, 4, 1>(),
                              bwd_variant<1, 16, 32, 4, 3>(), bwd_variant<1, 32, 32, 4, 2, 16>()};
  *n = dir ? (int)(sizeof(b) / sizeof(b[0])) : (int)(sizeof(f) / sizeof(f[0]));
  return dir ? b : f;
}

constexpr size_t kMaxSmem = 227 * 1024;    // of a CTA
constexpr size_t kSmemPerSm = 228 * 1024;  // of which each CTA takes 1 KB more than it asks for

// Can `ctas` CTAs that list nrec receivers run in `waves` waves?
bool runs(const Variant& v, int nrec, long long ctas, int waves) {
  const size_t need = v.smem + v.rec_bytes * nrec;
  const long long slots = (long long)device_sms() * waves, res = (ctas + slots - 1) / slots;
  return res <= v.res && need <= kMaxSmem && res * (need + 1024) <= kSmemPerSm;
}

}  // namespace

int fused_variant(const Geom& g, int dir, bool gradient) {
  if (g.nrec > kFusedMaxRec || g.nshot < 1) return -1;
  int n;
  const Variant* v = variants(dir, &n);
  for (int i = 0; i < n; ++i) {
    const long long tiles = (long long)((g.NX + v[i].s.bx - 1) / v[i].s.bx) *
                            ((g.NZ + v[i].s.bz - 1) / v[i].s.bz);
    if (!gradient && tiles > v[i].alone) continue;
    if (runs(v[i], g.nrec, tiles * g.nshot, gradient ? v[i].waves : 1)) return i;
  }
  return -1;
}

FusedShape fused_shape(int dir, int v) {
  int n;
  return variants(dir, &n)[v].s;
}

void launch_ac_fused(int dir, int v, const AcFusedArgs& a, cudaStream_t st) {
  int n;
  const Variant& V = variants(dir, &n)[v];
  static const bool attr = [] {  // thread-safe one-time initialisation
    for (int d = 0; d < 2; ++d) {
      int k;
      const Variant* all = variants(d, &k);
      for (int i = 0; i < k; ++i)
        cudaFuncSetAttribute(all[i].kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)std::min(all[i].smem + all[i].rec_bytes * kFusedMaxRec, kMaxSmem));
    }
    return true;
  }();
  (void)attr;
  const Geom& g = a.g;
  const bool rec = dir ? a.res != nullptr : a.data != nullptr;
  const dim3 grid((g.NX + V.s.bx - 1) / V.s.bx, (g.NZ + V.s.bz - 1) / V.s.bz, g.nshot);
  launch_dependent(V.kernel, grid, dim3(V.threads), V.smem + (rec ? V.rec_bytes * g.nrec : 0),
                   st, a);
  note_launches(1);
}

}  // namespace sweep
