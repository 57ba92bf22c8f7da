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

// z extents that take the kernels of sipo_flat.cuh (lanes over bins or voxels):
// below these the z lanes of the other kernels idle more than the flat ones
// repeat weights.  200 x 200, 300 views, us, z lanes / flat: single precision,
// projector 274 / 115 at nz = 4, 277 / 246 at 8, 279 / 349 at 12; backprojector
// 317 / 149 at 8, 317 / 209 at 12, 319 / 411 at 16; double precision, projector
// 2696 / 1859 at 4, 2696 / 2738 at 6; backprojector 2387 / 1950 at 8, 2480 / 2879 at 12.
// The flat projector's candidate window holds up to sides (and detectors) of kFlatSide.
constexpr int kFlatSide = 16384;
template <typename C> inline bool fp_flat(const Geo<C>& g) {
  return g.nz <= (sizeof(C) == 8 ? 5 : 8) && g.nx <= kFlatSide && g.ny <= kFlatSide && g.nd <= kFlatSide;
}
template <typename C> inline bool bp_flat(int nz) { return nz <= (sizeof(C) == 8 ? 9 : 12); }

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

// Calls f(ZForm) with the z form for extent nz and groups of at most gmax values
// (see ZForm): the form with the least tiles * time per tile.  The times are the
// measured ones of the solver's projector and backprojector (mean of both, 240^2 x
// 512 and 160^2 x 48, 300 views, FP32) relative to the form {4, 1}; they follow
// the 16-, 8- or 4-byte loads of a tap plus its fixed part.  E.g. 160^2 x 160,
// projector: {2, 3} 0.098 ms, {4, 2} 0.113, {4, 1} 0.152.  Double precision
// keeps two forms of pairs, and single values up to nz = 32, where pairs leave
// half of the lanes idle (200^2 x 16: 2.70 ms, single 1.81).  widest: only groups
// of gmax values (the solver's sums are formed group by group).
template <typename C, typename F>
inline void with_z_form(int nz, int gmax, F&& f, bool widest = false) {
  if constexpr (sizeof(C) == 8) {
    if (gmax >= 2 && nz % 128 == 0) f(ZForm<2, 2, false>{});
    else if (gmax >= 2 && nz > 32) f(ZForm<2, 1, true>{});
    else f(ZForm<1, 1, true>{});
  } else {
    if (gmax >= 4 && nz % 256 == 0) return f(ZForm<4, 2, false>{});
    struct Cost { int G, NG; double time; };
    constexpr Cost forms[10] = {{4, 2, 1.5}, {4, 1, 1.0}, {2, 4, 1.63}, {2, 3, 1.3}, {2, 2, 1.09},
                                {2, 1, 0.87}, {1, 8, 2.2}, {1, 4, 1.17}, {1, 2, 0.96}, {1, 1, 0.76}};
    int best = 9;
    double least = 1e300;
    for (int i = 0; i < 10; ++i) {
      const int T = 32 * forms[i].G * forms[i].NG;
      const double cost = ((nz + T - 1) / T) * forms[i].time;
      if ((widest ? forms[i].G == gmax : forms[i].G <= gmax) && cost < least) { least = cost; best = i; }
    }
    switch (best) {
      case 0: return f(ZForm<4, 2, true>{});
      case 1: return f(ZForm<4, 1, true>{});
      case 2: return f(ZForm<2, 4, true>{});
      case 3: return f(ZForm<2, 3, true>{});
      case 4: return f(ZForm<2, 2, true>{});
      case 5: return f(ZForm<2, 1, true>{});
      case 6: return f(ZForm<1, 8, true>{});
      case 7: return f(ZForm<1, 4, true>{});
      case 8: return f(ZForm<1, 2, true>{});
      default: return f(ZForm<1, 1, true>{});
    }
  }
}

}  // namespace sipo
