// sipo_flat.cuh -- the projector pair for flat volumes (few z values).
//
// k_project and k_backproject give the lanes of a warp the z values of one
// column, so that one weight serves 32 or more of them.  A 2-D slice has one z
// value: 31 lanes idle there, and the work per weight is one multiply-add.
// Here the lanes hold 32 neighbouring bins of a view (projector) or 32
// neighbouring voxels of a row (backprojector) of one z slice instead, each
// lane computing its own weights.  The weights are those of the z-lane kernels
// bit for bit (same u, same rounding).
//
// Single precision: every warp has a tile of its own and adds its terms in the
// order of the z-lane kernels, so the sums are theirs bit for bit too (a solve
// amplifies a change of order: up to 2e-5 in the duals of Case 2 after 64
// iterations).  Double precision: the eight warps of a block share a tile, each
// summing every eighth chunk of lines (or every eighth view), and the first warp
// adds the eight partial sums in order.
//
// Bound: instruction issue on the weights (about 55 per bin and line, 20 per
// voxel and view), not bytes: a 512 x 512 slice and its 360 x 512 sinogram stay
// in L2.  512 x 512, 360 views, single precision: 0.34 ms for a projection and a
// backprojection, where the z-lane kernels took 5.4 ms; 64 x 64, 96 views, double
// precision: 0.06 ms for the pair (0.25 ms), bound by FP64 issue.
#pragma once

#include "sipo_ops.cuh"

namespace sipo {

// Lines per chunk of a warp, so that a block's staged columns stay below 48 KB
// in both compute types.
template <typename C> constexpr int flat_chunk() { return sizeof(C) == 8 ? 8 : 16; }
// Voxel rows that 32 bins reach over a chunk of columns: 32 / |sin| <= 45.3
// across the bins, chunk - 1 along it (slope <= 1), and the rounding of both
// ends.
template <typename C> constexpr int flat_rows() { return 50 + flat_chunk<C>(); }
// Margin of the candidate window, computed in single precision for both
// compute types: the voxels of a line with floor(u) = j lie in an interval of
// length 1/|a| <= sqrt 2, so the window with both margins is shorter than 2 and
// holds two integers at most; the margin covers the rounding of the window
// start.  With M the largest of the two sides and the detector, the intercept is
// below 2 M and the start follows from it with an error of 6 M 2^-24 (intercept
// and margin, slope and sum, each rounded once); single precision adds 9 M 2^-24
// of the intercept's own terms and 3 M 2^-24 of u: together 0.0176 at M =
// kFlatSide.  (FP64 on 524288 voxels a side: 1% of the taps lost on the last lines.)
constexpr float kFlatEps = 0.02f;
constexpr int kFlatBins = 31;  // bins per tile (lane 0 holds the bin below the first)

// i - half (half = (n - 1) / 2) in the compute type, from i as a float and an int.
__device__ __forceinline__ float flat_coord(float cf, int, float half) { return cf - half; }
__device__ __forceinline__ double flat_coord(float, int i, double half) {
  // 2^51 + i without a conversion: a word of spacing 1/2, low word 2 i
  // (i in -2^29 .. 2^29 keeps the high word by the offset 2^30)
  const double t = __hiloint2double(0x43200000, int(2u * unsigned(i + (1 << 29))));
  return t - (2251799813685248.0 + 536870912.0 + half);
}

// Whether floor(u) = j for w = u - j (0 <= w < 1).  Exact for j >= 0, where
// u - j is exact near the interval; bin -1 compares the floor itself.
__device__ __forceinline__ bool flat_hit(float w) { return __float_as_uint(w) < 0x3f800000u; }
__device__ __forceinline__ bool flat_hit(double w) { return unsigned(__double2hiint(w)) < 0x3ff00000u; }

// w == 0 without an FP64 comparison.
__device__ __forceinline__ bool flat_zero(float w) { return w == 0.0f; }
__device__ __forceinline__ bool flat_zero(double w) {
  return ((unsigned(__double2hiint(w)) << 1) | unsigned(__double2loint(w))) == 0u;
}

// Sums of one lane's bin j over the warp's chunks of lines: each voxel with
// floor(u) = j gives (1 - w) v to bin j and w v to bin j + 1, the
// backprojector's two taps, so that a voxel is read and weighed once for both
// bins.  Single precision: `own` takes this lane's voxels and those of the lane
// below (by shuffles), in increasing index along the line, like the per-ray walk;
// double precision: `next` collects w v and moves up at the end.  ROWS: the ray is walked along y (lines are rows, read from global
// memory: the lanes' voxels are neighbours along x); otherwise along x, the
// chunk's columns staged in shared memory with reads along x.  EDGE: any tile
// (bin -1 among its bins, any z stride, inputs that reach outside the vial);
// otherwise one z value.  ATT: attenuation.  wide: the input vanishes where it
// should not count except outside the vial, where each ray counts it on its own
// lines [mine.x, mine.y] (a solver's blurred duals; as k_project with NeedBits).
// STRICT: a voxel that a weight of zero meets is left out, whatever it holds (0 *
// inf would make the bin NaN).
template <bool ROWS, bool EDGE, bool ATT, bool STRICT, typename SI, typename C>
__device__ __forceinline__ void flat_walk(const Geo<C>& g, const SI* vz, int k, C jf, C c, C s, int lo, int hi,
                                          bool wide, int2 mine, C (*stage)[flat_chunk<C>() + 1], C& own, C& next) {
  constexpr int kCh = flat_chunk<C>(), kRows = flat_rows<C>();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nz = EDGE ? g.nz : 1;
  const int2 above = make_int2(__shfl_down_sync(0xffffffffu, mine.x, 1), __shfl_down_sync(0xffffffffu, mine.y, 1));
  const C a = ROWS ? c : s;
  const C inv_a = C(1) / a;
  // first candidate on a line: ceil(base + slope line)
  const float slope = float(-(ROWS ? s : c) * inv_a);
  const float base = float((jf - g.off + (ROWS ? g.cy * s : g.cx * c)) * inv_a + (ROWS ? g.cx : g.cy) +
                           (inv_a < C(0) ? inv_a : C(0))) - kFlatEps;
  constexpr bool kShare = sizeof(C) == 8;
  const bool up = a > C(0);
  for (int r0 = lo + (kShare ? warp * kCh : 0); r0 <= hi; r0 += (kShare ? kWarps : 1) * kCh) {
    const int n = min(kCh, hi - r0 + 1);
    int ylo = 0;
    if constexpr (!ROWS) {
      // rows of the volume from the lowest to the highest candidate
      float f0, f1;
      int i0, i1;
      ceil_split(fmaf(float(r0), slope, base), f0, i0);
      ceil_split(fmaf(float(r0 + n - 1), slope, base), f1, i1);
      ylo = max(0, __reduce_min_sync(0xffffffffu, min(i0, i1)));
      const int yhi = min(g.ny - 1, __reduce_max_sync(0xffffffffu, max(i0, i1) + 1));
      const int x = lane & (kCh - 1);
      const int nrow = min(kRows, yhi - ylo + 1);
      SIPO_DCHECK(yhi - ylo + 1 <= kRows, 0);
      const SI* p = vz + ((size_t)(ylo + lane / kCh) * g.nx + r0 + x) * nz;
      const size_t step = (size_t)(32 / kCh) * g.nx * nz;
      __syncwarp();  // the previous chunk is read
#pragma unroll 4
      for (int yy = lane / kCh; yy < nrow; yy += 32 / kCh, p += step) stage[yy][x] = x < n ? to_c(*p) : C(0);
      __syncwarp();
    }
    // the part of u that the lanes share, one line per lane
    C shared_u = C(0);
    if constexpr (sizeof(C) == 8)
      shared_u = ROWS ? geo_inner(C(r0 + lane) - g.cy, s, g.off) : __dmul_rn(C(r0 + lane) - g.cx, c);
    float lf = float(r0);
#pragma unroll 4
    for (int r = 0; r < n; ++r, lf += 1.0f) {
      const int line = r0 + r;
      float cf;
      int i0;
      ceil_split(fmaf(lf, slope, base), cf, i0);
      int2 sp = ROWS ? g.xspan[line] : g.yspan[line];
      if (EDGE && wide) sp = make_int2(0, (ROWS ? g.nx : g.ny) - 1);
      const unsigned len = unsigned(sp.y - sp.x + 1) & ~unsigned((sp.y - sp.x) >> 31);  // 0: empty span
      const C f0 = flat_coord(cf, i0, ROWS ? g.cx : g.cy);
      C sh;
      if constexpr (sizeof(C) == 8) sh = __shfl_sync(0xffffffffu, shared_u, r);
      else sh = ROWS ? geo_inner(C(lf) - g.cy, s, g.off) : C(lf) - g.cx;
      C el = C(1);
      if constexpr (ATT) el = ROWS ? g.ey[(size_t)k * g.ny + line] : g.ex[(size_t)k * g.nx + line];
      const SI* vl = vz + (size_t)line * g.nx * nz;
      C va[2], vb[2], wa[2], wb[2];  // values for bins j and j + 1 and their weights, of the two candidates
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const int i = i0 + m;
        const C f = m == 0 ? f0 : f0 + C(1);
        C u;
        if constexpr (ROWS) u = geo_outer(f, c, sh);
        else if constexpr (sizeof(C) == 8) u = __dadd_rn(sh, geo_inner(f, s, g.off));
        else u = geo_outer(sh, c, geo_inner(f, s, g.off));
        C w = u - jf;
        bool hit;
        if constexpr (EDGE) {
          C flo;
          int fi;
          floor_split(u, flo, fi);
          hit = flo == jf;
        } else {
          hit = flat_hit(w);
        }
        hit = hit && unsigned(i - sp.x) < len;
        // a hit lies inside the staged rows (the window start is monotone along
        // the chunk); a miss adds w * 0
        C v = C(0), w0 = C(1) - w;
        if (hit) {
          if constexpr (ROWS) v = to_c(vl[i * nz]);
          else v = stage[i - ylo][r];
          if constexpr (ATT) {
            // the tap weight times (Ex Ey), in the backprojector's order
            const C e = ROWS ? g.ex[(size_t)k * g.nx + i] * el : el * g.ey[(size_t)k * g.ny + i];
            w0 *= e;
            w *= e;
          }
        }
        if (EDGE && wide) {
          if (line < mine.x || line > mine.y) w0 = C(0);
          if (line < above.x || line > above.y) w = C(0);
        }
        va[m] = STRICT && ATT && w0 == C(0) ? C(0) : v;  // (1 - w is above zero)
        vb[m] = STRICT && flat_zero(w) ? C(0) : v;
        wa[m] = w0;
        wb[m] = w;
      }
      if constexpr (kShare) {
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          own = fma(wa[m], va[m], own);
          next = fma(wb[m], vb[m], next);
        }
      } else {
        C vp[2], wp[2];  // those of the bin below, which reach this bin with w
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          vp[m] = __shfl_up_sync(0xffffffffu, vb[m], 1);
          wp[m] = __shfl_up_sync(0xffffffffu, wb[m], 1);
        }
        if (up) {  // u grows with the index: the bin below comes first
          own = fma(wp[1], vp[1], fma(wp[0], vp[0], own));
          own = fma(wa[1], va[1], fma(wa[0], va[0], own));
        } else {
          own = fma(wa[1], va[1], fma(wa[0], va[0], own));
          own = fma(wp[1], vp[1], fma(wp[0], vp[0], own));
        }
      }
    }
  }
}

template <typename SI, typename S, typename C, int MODE, typename O>
__global__ void __launch_bounds__(kThreads, 4)
k_project_flat(const Geo<C> g, const SI* __restrict__ vol, const Bufs<S, C> b, O* __restrict__ out,
               const uint8_t* __restrict__ act_col, const int2* __restrict__ rspan, bool wide) {
  if (MODE != kFpStore && b.st->done) return;
  constexpr int NR = fp_reductions(MODE);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int njb = (g.nd + kFlatBins - 1) / kFlatBins;
  const long long ntiles = (long long)g.na * njb * g.nz;
  double red[NR > 0 ? NR : 1] = {};
  StepScalars<C> sc{};
  if (MODE == kFpPrimal || MODE == kFpPrimalCheck) sc = read_scalars<C>(b.st);
  __shared__ C stage[kWarps][flat_rows<C>()][flat_chunk<C>() + 1];
  __shared__ C psum[sizeof(C) == 8 ? kWarps : 1][32];
  extern __shared__ __align__(16) unsigned long long kz_block[];
  if constexpr (MODE == kFpCertZ) {
    for (int z = threadIdx.x; z < g.nz; z += blockDim.x) kz_block[z] = 0ull;
    __syncthreads();
  }
  constexpr bool kShare = sizeof(C) == 8;
  for (long long t = kShare ? blockIdx.x : blockIdx.x * kWarps + warp; t < ntiles;
       t += (kShare ? 1 : kWarps) * gridDim.x) {
    const int k = int(t % g.na);
    const long long t1 = t / g.na;
    const int z = int(t1 % g.nz);
    const int jb = int(t1 / g.nz);
    const int j = jb * kFlatBins - 1 + lane;
    const bool live = lane > 0 && j < g.nd &&
                      (MODE == kFpStore || act_col == nullptr || act_col[(size_t)k * g.nd + j]);
    const C esj = live ? (g.es ? g.es[(size_t)k * g.nd + j] : C(1)) : C(0);
    const C c = g.cs[2 * k], s = g.cs[2 * k + 1];
    const bool rows = fabs(c) >= fabs(s);
    const C jf = C(j);
    int lo = 0x3fffffff, hi = -1;
    if (esj != C(0)) {
      lo = 0;
      hi = (rows ? g.ny : g.nx) - 1;
      fp_ray_span<C>(g, jf - g.off, c, s, rows, lo, hi);
      if (rspan) {
        const int2 r = rspan[(size_t)k * g.nd + j];
        lo = max(lo, r.x);
        hi = min(hi, r.y);
      }
      if (lo > hi) { lo = 0x3fffffff; hi = -1; }
    }
    const int2 mine = make_int2(lo, hi);
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    const SI* vz = vol + z;
    C own = C(0), next = C(0);
    if (lo <= hi) {
      const bool att = g.ex != nullptr;
      // The plain operator leaves out what a zero weight meets: in double precision
      // as it goes (no time: the two integer operations hide behind FP64 issue), in
      // single precision by a second walk where a sum came out NaN (as it goes: 9% of
      // a 512 x 512 slice's projection).
      constexpr bool kStrict = MODE == kFpStore;
#define SIPO_FLAT_WALK(R, E, A, Z) \
  flat_walk<R, E, A, Z, SI, C>(g, vz, k, jf, c, s, lo, hi, wide, mine, stage[warp], own, next)
#define SIPO_FLAT(R, E, A) SIPO_FLAT_WALK(R, E, A, kStrict && kShare)
      if (jb == 0 || g.nz != 1 || wide) {
        if (rows) { if (att) SIPO_FLAT(true, true, true); else SIPO_FLAT(true, true, false); }
        else { if (att) SIPO_FLAT(false, true, true); else SIPO_FLAT(false, true, false); }
      } else if (rows) {
        if (att) SIPO_FLAT(true, false, true); else SIPO_FLAT(true, false, false);
      } else {
        if (att) SIPO_FLAT(false, false, true); else SIPO_FLAT(false, false, false);
      }
      if constexpr (kStrict && !kShare) {
        if (__any_sync(0xffffffffu, own != own)) {
          own = C(0);
          if (rows) { if (att) SIPO_FLAT_WALK(true, true, true, true); else SIPO_FLAT_WALK(true, true, false, true); }
          else { if (att) SIPO_FLAT_WALK(false, true, true, true); else SIPO_FLAT_WALK(false, true, false, true); }
        }
      }
#undef SIPO_FLAT
#undef SIPO_FLAT_WALK
    }
    C tot[1] = {own};
    if constexpr (kShare) {
      next = __shfl_up_sync(0xffffffffu, next, 1);  // what bin j - 1's voxels give to bin j
      __syncthreads();  // the previous tile's sums are read
      psum[warp][lane] = own + next;
      __syncthreads();
      tot[0] = psum[0][lane];
#pragma unroll
      for (int w = 1; w < kWarps; ++w) tot[0] += psum[w][lane];
    }
    if ((!kShare || warp == 0) && live) {
      tot[0] = esj != C(0) ? tot[0] * esj : C(0);
      ZSpan<ZForm<1, 1, false>> zs;
      zs.z0 = z;
      fp_finish<S, C, ZForm<1, 1, false>, MODE, O>(b, sc, out, ((size_t)k * g.nd + j) * g.nz + z, zs, tot, red,
                                                   kz_block);
    }
  }
  fp_reduce<MODE, kShare ? 1 : kWarps>(g, b, red, kz_block, blockIdx.x * (kShare ? 1LL : kWarps) < ntiles);
}

// Views k = first, first + kWarps, ... (double precision) or all views of one voxel.  Z1: one z value; ES: vial
// factors (and ATT: attenuation).
template <bool ES, bool ATT, bool Z1, typename SI, typename C>
__device__ __forceinline__ C flat_gather(const Geo<C>& g, const SI* sz, int first, C xf, C yf, int ix, int iy,
                                         bool in) {
  const int nz = Z1 ? 1 : g.nz;
  C acc = C(0);
  const SI* row = sz + (size_t)first * g.nd * nz;
  constexpr int kStep = sizeof(C) == 8 ? kWarps : 1;
  const size_t step = (size_t)kStep * g.nd * nz;
  const int lane = threadIdx.x & 31;
  C shared_inner = C(0);
  int left = 0;  // views whose inner part the lanes still hold
#pragma unroll 4
  for (int k = first; k < g.na; k += kStep, row += step) {
    C inner;
    if constexpr (sizeof(C) == 8) {
      // the row's part of u, one view per lane: FP64 arithmetic is the scarce
      // resource (2 lanes a clock and SM), shuffles are not
      if (left == 0) {
        const int kl = min(k + lane * kStep, g.na - 1);
        shared_inner = geo_inner(yf, g.cs[2 * kl + 1], g.off);
        left = 32;
      }
      inner = __shfl_sync(0xffffffffu, shared_inner, 32 - left);
      --left;
    } else {
      inner = geo_inner(yf, g.cs[2 * k + 1], g.off);
    }
    const C u = geo_outer(xf, g.cs[2 * k], inner);
    C flo;
    int i0;
    floor_split(u, flo, i0);
    C w1 = u - flo;
    C w0 = C(1) - w1;
    const bool ok0 = in && unsigned(i0) < unsigned(g.nd), ok1 = in && unsigned(i0 + 1) < unsigned(g.nd);
    if constexpr (ATT) {
      const C e = g.ex[(size_t)k * g.nx + ix] * g.ey[(size_t)k * g.ny + iy];
      w0 *= e;
      w1 *= e;
    }
    if constexpr (ES) {
      const C* esk = g.es + (size_t)k * g.nd + i0;
      w0 *= ok0 ? esk[0] : C(0);
      w1 *= ok1 ? esk[1] : C(0);
    }
    const SI* p = row + i0 * nz;
    const C v0 = ok0 ? to_c(p[0]) : C(0), v1 = ok1 ? to_c(p[nz]) : C(0);
    acc = fma(w1, v1, fma(w0, v0, acc));
  }
  return acc;
}

// Tile: 32 voxels along x of one row, one z.
template <typename SI, typename S, typename C, int MODE, typename O>
__global__ void __launch_bounds__(kThreads, sizeof(C) == 8 ? 3 : 4)
k_backproject_flat(const Geo<C> g, const SI* __restrict__ sino, const Bufs<S, C> b, O* __restrict__ out,
                   const uint8_t* __restrict__ need) {
  if (MODE != kBpStore && b.st->done) return;
  constexpr int NR = MODE == kBpDual ? 2 : 0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ntx = (g.nx + 31) / 32;
  const long long ntiles = (long long)ntx * g.ny * g.nz;
  double red[NR > 0 ? NR : 1] = {};
  StepScalars<C> sc{};
  if (MODE != kBpStore) sc = read_scalars<C>(b.st);
  constexpr bool kShare = sizeof(C) == 8;
  __shared__ C psum[kShare ? kWarps : 1][32];
  const int first = kShare ? warp : 0;
  for (long long t = kShare ? blockIdx.x : blockIdx.x * kWarps + warp; t < ntiles;
       t += (kShare ? 1 : kWarps) * gridDim.x) {
    const int z = int(t % g.nz);
    const long long t1 = t / g.nz;
    const int ix = int(t1 % ntx) * 32 + lane;
    const int iy = int(t1 / ntx);
    const int2 sp = g.xspan[iy];
    const bool in = ix < g.nx && ix >= sp.x && ix <= sp.y && (need == nullptr || need[(size_t)iy * g.nx + ix]);
    const unsigned any = __ballot_sync(0xffffffffu, in);
    C acc = C(0);
    if (any != 0u) {  // (the same for every warp that shares the tile)
      const C xf = C(ix) - g.cx, yf = C(iy) - g.cy;
      const SI* sz = sino + z;
      const int cx = min(ix, g.nx - 1);
      if (g.nz != 1) {
        acc = g.ex ? flat_gather<true, true, false>(g, sz, first, xf, yf, cx, iy, in)
                   : (g.es ? flat_gather<true, false, false>(g, sz, first, xf, yf, cx, iy, in)
                           : flat_gather<false, false, false>(g, sz, first, xf, yf, cx, iy, in));
      } else {
        acc = g.ex ? flat_gather<true, true, true>(g, sz, first, xf, yf, cx, iy, in)
                   : (g.es ? flat_gather<true, false, true>(g, sz, first, xf, yf, cx, iy, in)
                           : flat_gather<false, false, true>(g, sz, first, xf, yf, cx, iy, in));
      }
    }
    C tot[1] = {acc};
    if constexpr (kShare) {
      __syncthreads();
      psum[warp][lane] = acc;
      __syncthreads();
      tot[0] = psum[0][lane];
#pragma unroll
      for (int w = 1; w < kWarps; ++w) tot[0] += psum[w][lane];
    }
    if ((!kShare || warp == 0) && ix < g.nx) {
      const size_t base = ((size_t)iy * g.nx + ix) * g.nz + z;
      if constexpr (MODE == kBpStore) {
        if (need == nullptr || in) store_z<O, C, 1>(out + base, tot);
      } else if (in) {
        dual_update<S, C, 1, false>(b, sc, base, tot, red);
      }
    }
  }
  if constexpr (MODE == kBpDual) block_reduce_store<2, 0u, kShare ? 1 : kWarps>(red, b.part, kSlSBand, blockIdx.x * (kShare ? 1LL : kWarps) < ntiles);
}

}  // namespace sipo
