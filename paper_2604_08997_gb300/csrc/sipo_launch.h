// sipo_launch.h -- host launchers of the operator kernels (one translation
// unit per operator so that the builds compile in parallel).
#pragma once

#include <cuda_runtime.h>

#include "sipo_solver.cuh"
#include "sipo_ops.cuh"

namespace sipo {

// nb: packed per-column flags of voxels whose input may be non-zero (rows ==
// nullptr: every in-vial voxel); rspan: per-ray walked-axis span holding such
// columns (nullptr: whole ray).
template <typename SI, typename S, typename C, int MODE, typename O>
void launch_project(const Geo<C>& g, const SI* vol, const Bufs<S, C>& b, O* out,
                    const uint8_t* act_col, cudaStream_t stream,
                    const NeedBits& nb = NeedBits{}, const int2* rspan = nullptr);

// Packs need[y][x] into the row-major and column-major bit arrays of NeedBits.
void launch_need_bits(const uint8_t* need, uint32_t* rows, uint32_t* cols, int nx, int ny, int wr, int wc,
                      cudaStream_t stream);

// Per-ray span of the projector walk that meets flagged columns (k_ray_spans).
template <typename C>
void launch_ray_spans(const Geo<C>& g, const uint8_t* need, int2* out, cudaStream_t stream);

// tile: entry of the backprojector tile table.  FP64: 0 = 8 columns per warp, 2
// blocks/SM; 1 = 4 columns, 2 blocks/SM; 2-6 = 4 columns, 3 blocks/SM.  Single
// precision: the row-pattern kernel at 2 (0, 1, 3) or 3 (2, 4) blocks/SM; 5, 6 =
// its form with rows staged by tensor-memory copies where bp_staged allows it,
// else as 4.
constexpr int kBpTiles = 7;

// Runs the bounded mbarrier wait (sipo_wait.cuh) on its own: one
// block of `threads` threads waits `budget` cycles on a barrier that receives
// its one arrival only if `arrive`; *timed_out = threads whose wait gave up.
// 0 on success, -1 on a CUDA error.  Synchronous.
int wait_selftest(long long budget, int arrive, int threads, unsigned int* timed_out);

// Checked builds (-DSIPO_CHECKED): the check bits recorded by the kernels of
// each translation unit, read and cleared; 0 in plain builds.
unsigned int check_flags_project();
unsigned int check_flags_backproject();
template <typename SI, typename S, typename C, int MODE, typename O>
void launch_backproject(const Geo<C>& g, const SI* sino, const Bufs<S, C>& b, O* out,
                        const uint8_t* need, cudaStream_t stream, const BpTiles& tiles, int tile = 0);

// Volumes that take the kernels of sipo_flat.cuh (lanes over bins or voxels): at few z
// values the z lanes of the other kernels idle more than the flat ones repeat
// weights.  Single precision, 200 x 200, 300 views, us, z lanes / flat: projector 274 / 115
// at nz = 4, 277 / 246 at 8, 279 / 349 at 12 (fp_plan chooses below that); backprojector
// 317 / 149 at 8, 317 / 209 at 12, 319 / 411 at 16.
// Double precision (z lanes: single values, the same at every nz below 32), 180 views,
// us, z lanes / flat.  Projector: 200 x 200 1427 / 1109 at 3, 1445 at 4; 64 x 64 161 / 165 at
// 3, 220 at 4; a detector twice the grid, whose outer rays end at once in z lanes, 200 x
// 200, 60 views 569 / 475 at 2, 690 at 3.  Backprojector: 200 x 200 1190 / 935 at 6, 1248 at 8;
// 128 x 128 430 / 370 at 6, 454 at 8; 64 x 64, where z lanes of four columns leave warps free,
// 268 / 138 at 9.
// The flat projector's candidate window holds up to sides (and detectors) of kFlatSide.
constexpr int kFlatSide = 16384;
template <typename C> inline bool fp_flat(const Geo<C>& g) {
  const int side = g.nx > g.ny ? g.nx : g.ny;
  const int most = sizeof(C) == 4 ? 8 : (g.nd > side + side / 2 ? 2 : 3);
  return g.nz <= most && side <= kFlatSide && g.nd <= kFlatSide;
}
template <typename C> inline bool bp_flat(int nx, int ny, int nz) {
  if (sizeof(C) == 4) return nz <= 12;
  return nz <= ((nx + 3LL) / 4 * ny >= 24LL * 152 ? 6 : 9);  // 24 warps an SM of z lanes
}

// Whether the staged backprojector covers sinograms of SI with this z extent: a lane
// takes groups of four values, and a tensor map needs strides of whole 16 bytes
// (bf16: nz a multiple of 8).
template <typename SI> inline bool bp_staged(int nz) { return nz % 4 == 0 && nz * sizeof(SI) % 16 == 0; }

// Group size G of the z layout (elements of C in 16 bytes).
template <typename C> constexpr int z_group() { return 16 / int(sizeof(C)); }

// Largest group of z values (elements of C in at most 16 bytes) that nz and the
// buffers' alignment allow: every z column then starts on a group boundary.
template <typename C, typename A, typename B>
inline int z_group_for(int nz, const A* a, const B* b) {
  int G = z_group<C>();
  const uintptr_t pa = reinterpret_cast<uintptr_t>(a), pb = reinterpret_cast<uintptr_t>(b);
  while (G > 1 && (nz % G != 0 || pa % (G * sizeof(A)) != 0 || pb % (G * sizeof(B)) != 0)) G /= 2;
  return G;
}

// Single-precision z forms and their time per tile: the measured ones of the solver's
// projector and backprojector (mean of both, 240^2 x 512 and 160^2 x 48, 300 views)
// relative to the form {4, 1}; they follow the 16-, 8- or 4-byte loads of a tap plus
// its fixed part.  E.g. 160^2 x 160, projector: {2, 3} 0.098 ms, {4, 2} 0.113, {4, 1} 0.152.
// The last one is {4, 2} where nz is whole tiles of 256.
struct ZCost { int G, NG; double time; };
constexpr int kZForms = 11;
constexpr ZCost kZCosts[kZForms] = {{4, 2, 1.5}, {4, 1, 1.0}, {2, 4, 1.63}, {2, 3, 1.3}, {2, 2, 1.09},
                                    {2, 1, 0.87}, {1, 8, 2.2}, {1, 4, 1.17}, {1, 2, 0.96}, {1, 1, 0.76}, {4, 2, 1.25}};

// Warps that the projector keeps resident on a GB300 (32 an SM).  Below that a
// launch lasts as long as one warp, whatever their number.
constexpr double kFpSlots = 152.0 * 32.0;

// The form (index of kZCosts) with the least time, for groups of at most gmax values
// (widest: of exactly gmax, as the solver's sums are formed group by group).  warps:
// warps per z tile of a launch that may leave slots empty, where a narrower form on
// more warps takes less time; 0: tiles * time per tile.  *cost: its time.
inline int z_form(int nz, int gmax, bool widest, double warps, double* cost) {
  int best = 9;
  *cost = 1e300;
  for (int i = 0; i < kZForms; ++i) {
    const ZCost& f = kZCosts[i];
    if ((widest ? f.G != gmax : f.G > gmax) || (i == 10 && nz % 256 != 0) || (i == 0 && nz % 256 == 0)) continue;
    const int T = 32 * f.G * f.NG;
    const double tiles = (nz + T - 1) / T, t = warps > 0 ? warps * tiles : tiles;
    const double c = (t > kFpSlots || warps <= 0 ? t : kFpSlots) * f.time;
    if (c < *cost) { *cost = c; best = i; }
  }
  return best;
}

// Calls f(ZForm) with the form chosen for extent nz and groups of at most gmax values
// (see z_form).  Double precision keeps two forms of pairs, and single values up to
// nz = 32, where pairs leave half of the lanes idle (200^2 x 16: 2.70 ms, single 1.81).
template <typename C, typename F>
inline void with_z_form(int nz, int gmax, F&& f, bool widest = false, double warps = 0.0) {
  if constexpr (sizeof(C) == 8) {
    if (gmax >= 2 && nz % 128 == 0) f(ZForm<2, 2, false>{});
    else if (gmax >= 2 && nz > 32) f(ZForm<2, 1, true>{});
    else f(ZForm<1, 1, true>{});
  } else {
    double cost;
    if (warps <= 0 && gmax >= 4 && nz % 256 == 0) return f(ZForm<4, 2, false>{});
    switch (z_form(nz, gmax, widest, warps, &cost)) {
      case 0: return f(ZForm<4, 2, true>{});
      case 1: return f(ZForm<4, 1, true>{});
      case 2: return f(ZForm<2, 4, true>{});
      case 3: return f(ZForm<2, 3, true>{});
      case 4: return f(ZForm<2, 2, true>{});
      case 5: return f(ZForm<2, 1, true>{});
      case 6: return f(ZForm<1, 8, true>{});
      case 7: return f(ZForm<1, 4, true>{});
      case 8: return f(ZForm<1, 2, true>{});
      case 9: return f(ZForm<1, 1, true>{});
      default: return f(ZForm<4, 2, false>{});
    }
  }
}

// How a projection without sums (the plain operator, the solver's step) runs in
// single precision; every choice gives the same sums, bit for bit.
struct FpPlan {
  bool flat;     // lanes over bins (nz <= 8)
  bool pair;     // two bins a warp, else one
  double warps;  // per z tile, for with_z_form
};

// Two bins a warp move fewer columns, one bin a warp makes twice the warps, each done
// in 0.65 of the time; the flat form costs 1.75 a warp and is full at 1500 warps.  The
// three figures are fitted to 296 projections (48^2 to 320^2, nz 1 to 384, 4 to 128
// views, every form timed): the choice is 2% behind the best of all on average,
// 26% at worst.  Pairs and the widest form everywhere were 36% behind: 200^2 x 200,
// 8 views, 90 us, now 35; 64^2 x 130, 32 views 24.8 -> 16.6; flat slices of 200^2, 8
// views 31 -> 20.7.
template <typename C>
inline FpPlan fp_plan(const Geo<C>& g, int gmax, bool flat_ok) {
  const double rays = double(g.na) * g.nd, pairs = double(g.na) * ((g.nd + 1) / 2);
  double ray_cost, pair_cost;
  z_form(g.nz, gmax, false, rays, &ray_cost);
  z_form(g.nz, gmax, false, pairs, &pair_cost);
  ray_cost *= 0.65;
  const double z_cost = ray_cost < pair_cost ? ray_cost : pair_cost;
  const double fw = double(g.na) * ((g.nd + 30) / 31) * g.nz;
  FpPlan p;
  p.flat = flat_ok && 1.75 * (fw > 1500.0 ? fw : 1500.0) < z_cost;
  p.pair = pair_cost <= ray_cost;
  p.warps = p.pair ? pairs : rays;
  return p;
}

}  // namespace sipo
