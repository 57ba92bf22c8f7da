// sipo_bp_tma.cuh -- row-pattern backprojector with the detector rows staged in
// shared memory by the Tensor Memory Accelerator (sm_103a).
//
// The weights, row patterns and sums are those of k_backproject2 (bit for bit
// the same sums).  What changes is where the rows come from.  A block has ROWS
// warps = ROWS voxel rows of 4 columns; for each view it needs the bins that its
// voxels reach: over 4 x 8 voxels floor(u) spans at most ceil(3 |cos| + 7 |sin|) + 1
// <= 9 values, over 4 x 2 (the other tile) at most 5, so a box of 10 or 6 bins from
// the block's smallest floor(u) holds every tap.  One more warp copies the
// boxes ([T z values] x [bins] of one view, cp.async.bulk.tensor; bins off the
// detector and z beyond the column arrive as zeros) into a ring of stages, two
// views a stage, as far ahead as the ring allows; the others read their rows from
// shared memory at constant offsets.  Each stage has a full barrier (the copies'
// bytes) and an empty one (the reading warps): no block-wide barrier inside a
// tile, and the copies of the next tile start while this one is finished.
//
// Bound: on a full chip shared-memory delivery, about 38 wavefronts a warp and
// view (33 for the rows, 5 for the table) and 10 for the copies' writes; on small
// parts the chain of one warp's views.  256^3 x 360, all columns in the vial:
// 0.72 ms (14.6 -> 23 TFLOP/s) where the rows read through L1 took 1.12 ms; solver
// steps 0.326 ms (0.471 through L1) and, on a larger part, 0.493 ms (0.611).
//
// Waits are bounded: one that outlives kWaitCycles sets the context's fault word
// (tiles.fault, read by the host) and the block's abort flag, on which every wait
// ends; the copying warp waits (bounded) for its last copies before it ends.
#pragma once

#include <cuda.h>

#include "sipo_ops.cuh"
#include "sipo_wait.cuh"

namespace sipo {

template <int ROWS> constexpr int bt_bins() { return ROWS == 8 ? 10 : 6; }  // per staged box
constexpr int kBtViews = 2;     // views per stage
constexpr int kBtStages = 4;    // stages of the ring

// One box of the 3-D tensor map (z, bin, view) into shared memory, completing
// on `bar` (its byte count is announced by mbar_expect_tx).
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int z, int bin, int view,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(z), "r"(bin), "r"(view),
      "r"(smem_u32(bar))
      : "memory");
}

// Per view of a warp: the four voxels' weights (w0, w1 each), the first row
// inside the box, the pattern, floor(u) relative to the box (generic body).
struct alignas(16) BtEnt {
  float4 w01, w23;  // (w0, w1) of voxels 0, 1 and of 2, 3
  int row, pat;
  int rel;          // floor(u_v) - box start, one byte per voxel
  int pad;
};

template <typename SI, int NG, int ROWS>
struct BtSmem {
  static constexpr int T = 128 * NG;  // z values per box
  static constexpr int kBoxBytes = bt_bins<ROWS>() * T * int(sizeof(SI));
  static constexpr int kStageBytes = kBtViews * kBoxBytes;
  static constexpr size_t kTableOff = size_t(kBtStages) * kStageBytes;
  static constexpr size_t kBarOff = kTableOff + ROWS * kBp2Chunk * sizeof(BtEnt);
  static constexpr size_t kBytes = kBarOff + 2 * kBtStages * sizeof(uint64_t) + 16 + 128;  // + alignment slack
};

// Wait that also ends when the block aborts.
__device__ __forceinline__ bool bt_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                        volatile unsigned int* fault) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (*abort_flag) return false;
    if (clock64() - t0 > kWaitCycles) {
      fault[0] = 1u;
      *abort_flag = 1;
      return false;
    }
  }
  return true;
}

// The block's first bin of view k over the tile [tx0, tx0 + 4) x [y0, y1]: u is
// monotone in x and in y, so a corner has the smallest floor.
__device__ __forceinline__ int bt_box(const Geo<float>& g, int k, int tx0, int y0, int y1) {
  const float c = g.cs[2 * k], s = g.cs[2 * k + 1];
  const float xf0 = float(tx0) - g.cx;
  const float ia = geo_inner(float(y0) - g.cy, s, g.off), ib = geo_inner(float(y1) - g.cy, s, g.off);
  int lo = 0x7fffffff;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float f;
    int i;
    floor_split(geo_outer(xf0 + ((q & 1) ? 3.0f : 0.0f), c, (q & 2) ? ib : ia), f, i);
    lo = min(lo, i);
  }
  return lo;
}

template <typename SI, int NG>
__device__ __forceinline__ void bt_row(const SI* p, float (&v)[4 * NG]) {
#pragma unroll
  for (int q = 0; q < NG; ++q) {
    if constexpr (sizeof(SI) == 4) {
      const float4 r = *reinterpret_cast<const float4*>(p + q * 128);
      v[q * 4] = r.x; v[q * 4 + 1] = r.y; v[q * 4 + 2] = r.z; v[q * 4 + 3] = r.w;
    } else {
      const uint2 r = *reinterpret_cast<const uint2*>(p + q * 128);
      v[q * 4] = __uint_as_float(r.x << 16);
      v[q * 4 + 1] = __uint_as_float(r.x & 0xffff0000u);
      v[q * 4 + 2] = __uint_as_float(r.y << 16);
      v[q * 4 + 3] = __uint_as_float(r.y & 0xffff0000u);
    }
  }
}

__device__ __forceinline__ float4 bt_weights(const BtEnt& e, int v) {
  const float4 p = v < 2 ? e.w01 : e.w23;
  return (v & 1) ? make_float4(p.z, p.z, p.w, p.w) : make_float4(p.x, p.x, p.y, p.y);
}

template <typename SI, int NG, int PAT>
__device__ __forceinline__ void bt_body(const SI* row, const BtEnt& e, float (&acc)[kBp2NV][4 * NG]) {
  constexpr int NR = bp2_rows(PAT);
  float r[NR][4 * NG];
#pragma unroll
  for (int j = 0; j < NR; ++j) bt_row<SI, NG>(row + j * (128 * NG), r[j]);
#pragma unroll
  for (int v = 0; v < kBp2NV; ++v)
    bp2_fma<4 * NG>(acc[v], bt_weights(e, v), r[bp2_off(PAT, v)], r[bp2_off(PAT, v) + 1]);
}

template <typename SI, int NG>
__device__ __forceinline__ void bt_view(const SI* box, const BtEnt& e, float (&acc)[kBp2NV][4 * NG]) {
  const SI* row = box + e.row * (128 * NG);
  switch (e.pat) {
#define SIPO_BT_CASE(P) \
  case P:               \
    bt_body<SI, NG, P>(row, e, acc); break;
    SIPO_BP2_PATTERNS(SIPO_BT_CASE)
#undef SIPO_BT_CASE
    case kBp2Skip: break;
    default:
#pragma unroll
      for (int v = 0; v < kBp2NV; ++v) {
        float r0[4 * NG], r1[4 * NG];
        const SI* p = box + ((e.rel >> (8 * v)) & 0xff) * (128 * NG);
        bt_row<SI, NG>(p, r0);
        bt_row<SI, NG>(p + 128 * NG, r1);
        bp2_fma<4 * NG>(acc[v], bt_weights(e, v), r0, r1);
      }
  }
}

// NG groups of four z values a lane: tiles of 128 NG (nz % 4 == 0).  ROWS:
// tiles.rows.  need, list and modes as k_backproject2.  Two rows: 6 blocks an SM with
// one group; with two groups of FP32 a block's 52 KB of shared memory leave 4, and the
// bound of 6 only keeps a thread to 112 registers.
template <typename SI, typename S, int NG, int ROWS, int MODE, typename O>
__global__ void __launch_bounds__(32 * (ROWS + 1), ROWS == 8 ? 2 : 6)
k_backproject_tma(const Geo<float> g, const __grid_constant__ CUtensorMap tmap, const Bufs<S, float> b,
                  O* __restrict__ out, const uint8_t* __restrict__ need, const BpTiles tiles) {
  using SM = BtSmem<SI, NG, ROWS>;
  constexpr int NV = kBp2NV, ZL = 4 * NG, T = SM::T;
  if (MODE != kBpStore && b.st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + SM::kBarOff);
  uint64_t* empty = full + kBtStages;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + kBtStages);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kBtStages; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, ROWS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *abort_flag = 0;
  }
  __syncthreads();
  const int ntx = (g.nx + NV - 1) / NV, nty = (g.ny + ROWS - 1) / ROWS;
  const int nzc = (g.nz + T - 1) / T;
  const long long ntiles = (tiles.list ? (long long)tiles.n : (long long)ntx * nty) * nzc;
  constexpr int NR = MODE == kBpDual ? 2 : 0;
  double red[NR > 0 ? NR : 1] = {};

  // a tile without a voxel inside the vial is written (plain operator) but not summed
  auto tile_live = [&](int ty, int tx) {
    for (int y = ty * ROWS; y < min(g.ny, (ty + 1) * ROWS); ++y) {
      const int2 sp = g.xspan[y];
      if (sp.x <= min(g.nx, tx * NV + NV) - 1 && sp.y >= tx * NV) return true;
    }
    return false;
  };

  if (warp == ROWS) {
    // ---- copying warp: lane l finds the boxes of views k0 + l, lane 0 issues
    unsigned seq = 0;
    bool ok = true;
    for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      const int tile = tiles.list ? tiles.list[t / nzc] : int(t / nzc);
      const int tx = tile % ntx, ty = tile / ntx, zt = int(t % nzc) * T;
      if (!tile_live(ty, tx)) continue;
      const int y0 = ty * ROWS, y1 = min(g.ny, y0 + ROWS) - 1;
      for (int k0 = 0; k0 < g.na && ok; k0 += 32) {
        const int box = k0 + lane < g.na ? bt_box(g, k0 + lane, tx * NV, y0, y1) : 0;
        const int kn = min(32, g.na - k0);
        for (int a = 0; a < kn && ok; a += kBtViews, ++seq) {
          const unsigned slot = seq % kBtStages, round = seq / kBtStages;
          const int b0 = __shfl_sync(0xffffffffu, box, a), b1 = __shfl_sync(0xffffffffu, box, min(a + 1, 31));
          int good = 1;
          if (lane == 0) {
            // the slot's readers of the round before are done
            if (round > 0) good = bt_wait(empty + slot, (round - 1) & 1u, abort_flag, tiles.fault);
            if (good) {
              const int n = min(kBtViews, kn - a);
              unsigned char* dst = smem + slot * SM::kStageBytes;
              mbar_expect_tx(full + slot, uint32_t(n * SM::kBoxBytes));
              tma_load_3d(dst, &tmap, zt, b0, k0 + a, full + slot);
              if (n > 1) tma_load_3d(dst + SM::kBoxBytes, &tmap, zt, b1, k0 + a + 1, full + slot);
            }
          }
          ok = __shfl_sync(0xffffffffu, good, 0) != 0;
          if (!ok) break;  // seq counts the stages issued
        }
      }
    }
    if (lane == 0) {
      // copies in flight write this block's shared memory: wait for them (bounded),
      // also where a reading warp gives up after the last one was issued
      for (unsigned s = seq > kBtStages ? seq - kBtStages : 0; s < seq; ++s)
        mbar_wait(full + s % kBtStages, (s / kBtStages) & 1u);
    }
  } else {
    StepScalars<float> sc{};
    if (MODE != kBpStore) sc = read_scalars<float>(b.st);
    BtEnt* tb = reinterpret_cast<BtEnt*>(smem + SM::kTableOff) + warp * kBp2Chunk;
    unsigned seq = 0;
    bool ok = true;
    for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      const int tile = tiles.list ? tiles.list[t / nzc] : int(t / nzc);
      const int tx = tile % ntx, ty = tile / ntx, z0 = int(t % nzc) * T + lane * 4;
      const int iy = ty * ROWS + warp;
      unsigned mask = 0;
      if (iy < g.ny) {
        const int2 sp = g.xspan[iy];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const int ix = tx * NV + v;
          if (ix < g.nx && ix >= sp.x && ix <= sp.y && (need == nullptr || need[(size_t)iy * g.nx + ix]))
            mask |= 1u << v;
        }
      }
      float acc[NV][ZL];
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int i = 0; i < ZL; ++i) acc[v][i] = 0.0f;
      if (tile_live(ty, tx)) {
        const float yf = float(iy) - g.cy, xf0 = float(tx * NV) - g.cx;
        const int y0 = ty * ROWS, y1 = min(g.ny, y0 + ROWS) - 1;
        for (int k0 = 0; k0 < g.na && ok; k0 += kBp2Chunk) {
          const int kn = min(kBp2Chunk, g.na - k0);
          if (mask != 0u && lane < kn) {
            Bp2Ent e;
            bp2_weights(g, k0 + lane, yf, xf0, iy, tx * NV, mask, e);
            const int b0 = bt_box(g, k0 + lane, tx * NV, y0, y1);
            BtEnt o;
            o.w01 = make_float4(e.w[0].x, e.w[0].z, e.w[1].x, e.w[1].z);
            o.w23 = make_float4(e.w[2].x, e.w[2].z, e.w[3].x, e.w[3].z);
            o.row = e.b - b0;
            o.pat = e.pat;
            o.rel = (e.i0.x - b0) | (e.i0.y - b0) << 8 | (e.i0.z - b0) << 16 | (e.i0.w - b0) << 24;
            o.pad = 0;
            // (a span wider than the box, which these tiles cannot have, is not read)
            if (o.row < 0 || max(max(e.i0.x, e.i0.y), max(e.i0.z, e.i0.w)) + 1 - b0 >= bt_bins<ROWS>()) {
              o.pat = kBp2Skip;
              tiles.fault[1] = 1u;
            }
            tb[lane] = o;
          }
          __syncwarp();
          for (int a = 0; a < kn; a += kBtViews, ++seq) {
            const unsigned slot = seq % kBtStages;
            // the entries do not depend on the copies: read ahead of the wait
            const BtEnt e0 = tb[a], e1 = tb[min(a + 1, kBp2Chunk - 1)];
            ok = bt_wait(full + slot, (seq / kBtStages) & 1u, abort_flag, tiles.fault);
            if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
            if (mask != 0u) {
              const SI* box = reinterpret_cast<const SI*>(smem + slot * SM::kStageBytes) + lane * 4;
              bt_view<SI, NG>(box, e0, acc);
              if (a + 1 < kn) bt_view<SI, NG>(box + SM::kBoxBytes / sizeof(SI), e1, acc);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(empty + slot);
          }
          __syncwarp();
        }
        if (!ok) break;
      }
      if (iy < g.ny) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const int ix = tx * NV + v;
          if (ix >= g.nx) continue;
          const size_t base = ((size_t)iy * g.nx + ix) * g.nz + z0;
#pragma unroll
          for (int q = 0; q < NG; ++q) {
            if (z0 + q * 128 >= g.nz) continue;
            const float part[4] = {acc[v][4 * q], acc[v][4 * q + 1], acc[v][4 * q + 2], acc[v][4 * q + 3]};
            if constexpr (MODE == kBpStore) {
              if (need == nullptr || ((mask >> v) & 1u)) store_group<O, float, 4>(out + base + q * 128, part);
            } else if ((mask >> v) & 1u) {
              dual_update<S, float, 4, false>(b, sc, base + q * 128, part, red);
            }
          }
        }
      }
    }
  }
  if constexpr (MODE == kBpDual) block_reduce_store<2, 0u, ROWS>(red, b.part, kSlSBand, blockIdx.x < ntiles);
}

}  // namespace sipo
