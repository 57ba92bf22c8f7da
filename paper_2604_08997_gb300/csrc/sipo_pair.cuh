// sipo_pair.cuh -- single-precision projector, two bins a warp.
//
// k_project loads a voxel column's z segment once for every ray that it reaches
// and is bound by that delivery (L1: 8 wavefronts a tap at 8 z values a lane).
// Here a warp sums two neighbouring bins of one view: a column that reaches either
// is loaded once (3.4 a line for 4.5 taps), with a weight for each bin, one of
// them zero for the outer columns.  Taps keep the order of the per-ray walk, and
// a zero weight leaves a sum of finite values unchanged, so the sums are those of
// k_project bit for bit.  An infinite or NaN voxel would reach the other bin as
// 0 * inf: the plain operator sums a pair that came out NaN again, one bin at a
// time (fp2_again).  (Four bins a warp, without zero weights through 13 line shapes, moved even
// less but was slower: 16 to 24 warps an SM could not cover a line's chain of
// table, jump, loads and multiply-adds.)
//
// Bound: latency times concurrency of the column loads; 32 warps an SM with four
// columns each in flight beat 24 or 16 warps with more.  256^3 x 360, ms, k_project
// / here: solver step 0.359 / 0.344, another target 0.606 / 0.560, all columns in
// the vial 1.064 / 0.913; 96^3 x 391 0.0591 / 0.0529 and 0.126 / 0.105.  With 24 warps
// 0.352, 0.574, 1.001; three columns in flight 0.365, 0.592, 0.969; eight with 16
// warps 0.447, 0.725, 1.091.
#pragma once

#include "sipo_ops.cuh"

namespace sipo {

constexpr int kPairVox = 5;                  // u in (j - 1, j + 2): at most 3 sqrt 2 wide
constexpr int kPairList = 32 * kPairVox;
constexpr int kPairBatch = 4;                 // columns in flight a warp

struct PairList {
  alignas(16) int col[kPairList];
  float2 w[kPairList];  // weights in bins j and j + 1
};

// What the lines of one view and bin pair share.
struct PairRay {
  float c, s, inv_a, h;  // h: half the candidate window with its margin
  int k, j;
  bool spread;           // per-bin line ranges apply (flags outside the vial)
  int2 ra, rb;           // line ranges of bins j and j + 1
};

template <bool ROWS, bool FAST>
__device__ __forceinline__ int fp2_line_taps(const Geo<float>& g, const NeedBits& nb, bool use_bits,
                                             const PairRay& ray, int line, int (&col)[kPairVox],
                                             float2 (&wt)[kPairVox]) {
  const float ja = float(ray.j), jb = float(ray.j + 1);
  float cf, inner = 0.0f, xf = 0.0f;
  int i0;
  if constexpr (ROWS) {
    inner = geo_inner(float(line) - g.cy, ray.s, g.off);
    ceil_split((ja + 0.5f - inner) * ray.inv_a + g.cx - ray.h, cf, i0);
  } else {
    xf = float(line) - g.cx;
    ceil_split((ja + 0.5f - g.off - xf * ray.c) * ray.inv_a + g.cy - ray.h, cf, i0);
  }
  unsigned okm;
  if (use_bits) {
    okm = nb.window<31u>(ROWS ? nb.rows : nb.cols, line, i0);
  } else {
    const int2 sp = ROWS ? g.xspan[line] : g.yspan[line];
    okm = 0u;
#pragma unroll
    for (int m = 0; m < kPairVox; ++m) okm |= unsigned(i0 + m >= sp.x && i0 + m <= sp.y) << m;
  }
  if (okm == 0u) return 0;
  const float f0 = ROWS ? cf - g.cx : cf - g.cy;
  float eline = 1.0f;
  if (g.ex) eline = ROWS ? g.ey[(size_t)ray.k * g.ny + line] : g.ex[(size_t)ray.k * g.nx + line];
  const bool in_a = !ray.spread || (line >= ray.ra.x && line <= ray.ra.y);
  const bool in_b = !ray.spread || (line >= ray.rb.x && line <= ray.rb.y);
  int nt = 0;
#pragma unroll
  for (int m = 0; m < kPairVox; ++m) {
    const float u = ROWS ? geo_outer(f0 + float(m), ray.c, inner)
                         : geo_outer(xf, ray.c, geo_inner(f0 + float(m), ray.s, g.off));
    float ta = tap_weight<FAST>(u, ja, ja - 1.0f), tb = tap_weight<FAST>(u, jb, ja);
    const bool ok = (okm >> m) & 1u;
    ta = ok && in_a ? ta : 0.0f;
    tb = ok && in_b ? tb : 0.0f;
    const int ix = ROWS ? i0 + m : line, iy = ROWS ? line : i0 + m;
    if (g.ex && (ta != 0.0f || tb != 0.0f)) {
      const float e = ROWS ? g.ex[(size_t)ray.k * g.nx + ix] * eline : eline * g.ey[(size_t)ray.k * g.ny + iy];
      ta = ta != 0.0f ? ta * e : 0.0f;  // (e may be infinite: a bin out of reach stays at zero)
      tb = tb != 0.0f ? tb * e : 0.0f;
    }
    col[m] = iy * g.nx + ix;
    wt[m] = make_float2(ta, tb);
    // counted by the weights that fp2_walk lists: a strong attenuation may have
    // brought both to zero, and a place reserved for them would stay unwritten
    nt += ta != 0.0f || tb != 0.0f;
  }
  return nt;
}

template <bool ROWS, bool FAST, typename Z, typename SI>
__device__ __forceinline__ void fp2_walk(const Geo<float>& g, const SI* vz, const NeedBits& nb, bool use_bits,
                                         const PairRay& ray, int lo, int hi, const ZSpan<Z>& zs, PairList& tl,
                                         float (&acc)[2][Z::ZL]) {
  constexpr int ZL = Z::ZL;
  const int lane = threadIdx.x & 31;
  const size_t nz = g.nz;
  for (int r0 = lo; r0 <= hi; r0 += 32) {
    int col[kPairVox];
    float2 wt[kPairVox];
    int nt = 0;
#pragma unroll
    for (int m = 0; m < kPairVox; ++m) { col[m] = 0; wt[m] = make_float2(0.0f, 0.0f); }
    if (r0 + lane <= hi) nt = fp2_line_taps<ROWS, FAST>(g, nb, use_bits, ray, r0 + lane, col, wt);
    // exclusive prefix of the tap counts over the lanes = list positions
    int incl = nt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    if (total == 0) continue;
    int pos = incl - nt;
#pragma unroll
    for (int m = 0; m < kPairVox; ++m) {
      if (nt != 0 && (wt[m].x != 0.0f || wt[m].y != 0.0f)) {
        tl.col[pos] = col[m];
        tl.w[pos] = wt[m];
        ++pos;
      }
    }
    SIPO_DCHECK(pos == incl, 0);
    __syncwarp();
#ifdef SIPO_CHECKED
    for (int q = lane; q < total; q += 32) SIPO_DCHECK((unsigned(tl.col[q]) < unsigned(g.nx * g.ny)), 0);
#endif
    int t = 0;
    for (; t + kPairBatch <= total; t += kPairBatch) {
      float v[kPairBatch][ZL];
#pragma unroll
      for (int u = 0; u < kPairBatch; ++u) load_zf<Z>(vz + (size_t)tl.col[t + u] * nz, zs, v[u]);
#pragma unroll
      for (int u = 0; u < kPairBatch; ++u) {
        const float2 w = tl.w[t + u];
        fma_z<float, ZL>(acc[0], w.x, v[u]);
        fma_z<float, ZL>(acc[1], w.y, v[u]);
      }
    }
    for (; t < total; ++t) {
      float v[ZL];
      load_zf<Z>(vz + (size_t)tl.col[t] * nz, zs, v);
      const float2 w = tl.w[t];
      fma_z<float, ZL>(acc[0], w.x, v);
      fma_z<float, ZL>(acc[1], w.y, v);
    }
    __syncwarp();
  }
}

// The plain operator's bins j0 and j0 + 1 of view k one after the other, by the
// per-ray walk, written to out.  Out of line, as it runs only where a sum is NaN:
// 96 x 90 x 96, 391 views took 87.8 us so, 90.5 us with the pair's own loop run again,
// 97 us with these walks inside the kernel (86.5 us without the check); 128^2 x 130, 360
// views 224 us, 247 us with the loop run again.
template <typename SI, typename Z, typename O>
__device__ __noinline__ void fp2_again(const Geo<float>* gp, const SI* vol, O* out, int k, int j0, int tz,
                                       PairList* list) {
  static_assert(sizeof(TapList<float>) <= sizeof(PairList), "list of a ray");
  const Geo<float>& g = *gp;
  TapList<float>& tl = *reinterpret_cast<TapList<float>*>(list);
  const float c = g.cs[2 * k], s = g.cs[2 * k + 1];
  const bool rows = fabsf(c) >= fabsf(s);
  ZSpan<Z> zs;
  zs.init(g.nz, tz);
  const SI* vz = vol + zs.z0;
  for (int j = j0; j < min(j0 + 2, g.nd); ++j) {
    const size_t at = (size_t)k * g.nd + j;
    const float es = g.es ? g.es[at] : 1.0f;
    float acc[Z::ZL];
#pragma unroll
    for (int i = 0; i < Z::ZL; ++i) acc[i] = 0.0f;
    if (es != 0.0f) {
      int lo = 0, hi = (rows ? g.ny : g.nx) - 1;
      fp_ray_span<float>(g, float(j) - g.off, c, s, rows, lo, hi);
      if (rows) fp_walk<true, false, Z, SI, float>(g, vz, NeedBits{}, false, k, float(j), c, s, lo, hi, zs, tl, acc);
      else fp_walk<false, false, Z, SI, float>(g, vz, NeedBits{}, false, k, float(j), c, s, lo, hi, zs, tl, acc);
#pragma unroll
      for (int i = 0; i < Z::ZL; ++i) acc[i] *= es;
    }
    if (!Z::kRagged || zs.fresh != 0u) store_owned<Z>(out + at * g.nz + zs.z0, zs, acc);
  }
}

// Tile: aw consecutive views x 8 / aw consecutive bin pairs, one z tile; a warp
// sums one pair of one view.  Other arguments as k_project.
template <typename SI, typename S, typename Z, int MODE, typename O>
__global__ void __launch_bounds__(kThreads, 4)
k_project_pair(const Geo<float> g, const SI* __restrict__ vol, const Bufs<S, float> b, O* __restrict__ out,
               const uint8_t* __restrict__ act_col, const NeedBits nb, const int2* __restrict__ rspan, int aw) {
  static_assert(MODE == kFpStore || MODE == kFpPrimal, "modes without reductions");
  const bool use_bits = nb.rows != nullptr;
  if (MODE != kFpStore && b.st->done) return;
  constexpr int ZL = Z::ZL;
  const int warp = threadIdx.x >> 5;
  const int nzc = (g.nz + Z::T - 1) / Z::T;
  const int bw = kWarps / aw;
  const int np = (g.nd + 1) / 2, njb = (np + bw - 1) / bw, nka = (g.na + aw - 1) / aw;
  const long long ntiles = (long long)nka * njb * nzc;
  double red[1] = {};
  StepScalars<float> sc{};
  if (MODE == kFpPrimal) sc = read_scalars<float>(b.st);
  __shared__ PairList taps[kWarps];
  for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int k = int(t % nka) * aw + warp % aw;
    const long long t1 = t / nka;
    const int tz = int(t1 % nzc);
    const int j0 = (int(t1 / nzc) * bw + warp / aw) * 2;
    if (aw > 1) __syncthreads();  // keeps the rays of a tile abreast, so that they meet in L1
    if (j0 >= g.nd || k >= g.na) continue;
    PairRay ray;
    ray.c = g.cs[2 * k];
    ray.s = g.cs[2 * k + 1];
    const bool rows = fabsf(ray.c) >= fabsf(ray.s);
    const float a = rows ? ray.c : ray.s;
    ray.inv_a = 1.0f / a;
    ray.h = 1.5f / fabsf(a) + kCandEps;
    ray.k = k;
    ray.j = j0;
    ray.spread = use_bits && nb.spread && g.r2i >= 0;
    int2 range[2];
    unsigned live = 0u;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int j = j0 + q;
      range[q] = make_int2(0x3fffffff, -1);
      if (j >= g.nd) continue;
      const size_t at = (size_t)k * g.nd + j;
      if (MODE != kFpStore && act_col != nullptr && !act_col[at]) continue;
      live |= 1u << q;
      if (g.es && g.es[at] == 0.0f) continue;
      int l = 0, h = (rows ? g.ny : g.nx) - 1;
      fp_ray_span<float>(g, float(j) - g.off, ray.c, ray.s, rows, l, h);
      if (rspan) {
        const int2 r = rspan[at];
        l = max(l, r.x);
        h = min(h, r.y);
      }
      if (l <= h) range[q] = make_int2(l, h);
    }
    if (live == 0u) continue;
    ray.ra = range[0];
    ray.rb = range[1];
    const int lo = min(range[0].x, range[1].x), hi = max(range[0].y, range[1].y);
    ZSpan<Z> zs;
    zs.init(g.nz, tz);
    const SI* vz = vol + zs.z0;
    PairList& tl = taps[warp];
    float acc[2][ZL];
#pragma unroll
    for (int i = 0; i < ZL; ++i) acc[0][i] = acc[1][i] = 0.0f;
    if (rows) {
      if (j0 >= 2) fp2_walk<true, true, Z, SI>(g, vz, nb, use_bits, ray, lo, hi, zs, tl, acc);
      else fp2_walk<true, false, Z, SI>(g, vz, nb, use_bits, ray, lo, hi, zs, tl, acc);
    } else {
      if (j0 >= 2) fp2_walk<false, true, Z, SI>(g, vz, nb, use_bits, ray, lo, hi, zs, tl, acc);
      else fp2_walk<false, false, Z, SI>(g, vz, nb, use_bits, ray, lo, hi, zs, tl, acc);
    }
    if constexpr (MODE == kFpStore) {
      bool nan = false;
#pragma unroll
      for (int i = 0; i < ZL; ++i) nan = nan || acc[0][i] != acc[0][i] || acc[1][i] != acc[1][i];
      if (__any_sync(0xffffffffu, nan)) {
        const Geo<float> gl = g;  // (the address of g itself, as a grid constant: solver step 0.559 -> 0.588 ms)
        fp2_again<SI, Z, O>(&gl, vol, out, k, j0, tz, &tl);
        continue;
      }
    }
    if (Z::kRagged && zs.fresh == 0u) continue;
    SIPO_DCHECK(zs.z0 + zs.at(Z::NG - 1) + Z::G - 1 < g.nz, 0);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (!((live >> q) & 1u)) continue;
      const size_t at = (size_t)k * g.nd + j0 + q;
      const float es = g.es ? g.es[at] : 1.0f;
#pragma unroll
      for (int i = 0; i < ZL; ++i) acc[q][i] = es != 0.0f ? acc[q][i] * es : 0.0f;
      fp_finish<S, float, Z, MODE, O>(b, sc, out, at * g.nz + zs.z0, zs, acc[q], red, nullptr);
    }
  }
}

}  // namespace sipo
