// sipo_tiles.h -- block tiles of the single-precision backprojector, chosen from
// the shape alone (host code without CUDA, so that the rule can be run anywhere).
//
// The rows of a tile decide which voxels share a block's FP64 partial sum, and the
// split decides the order of a voxel's sum over views; both enter the results.  So
// the rules count against a fixed number of SMs, those of a GB300, as the grid of
// the reducing kernels does, and not against those of the device at hand.
#pragma once

namespace sipo {

constexpr int kPlanSms = 152;

struct BpPlan {
  int rows, split;  // rows of 4 voxels, and log2 of the warps that share a row's views
};

// Tiles of 8 rows where they cover the SMs one and a half times, else of 2: a tile
// lasts as long as its views, and on a small part more of them, on more SMs, is what
// is left to gain.  Staged rows, solver step, ms with 8 / 4 / 2 rows (tiles of 8):
// 64^3 x 180 (41) 0.060 / 0.057 / 0.054; 112^3 x 333 (134) 0.111 / 0.103 / 0.101; 160^3 x
// 300 (164) 0.136 / 0.125 / 0.126; 192^3 x 300 (286) 0.158 / 0.247 / 0.241; 256^3 x 360
// (490) 0.338 / 0.422 / 0.505.  Rows read in place, 8 / 2 rows: 64^2 x 66 x 180 0.090 /
// 0.088; 128^2 x 130 x 360 0.174 / 0.170; 160^2 x 162 x 300 0.152 / 0.148; BF16 160^2 x 164 x
// 300 0.172 / 0.153.
inline int bp_rows(double tiles_of_8) { return tiles_of_8 < 3 * kPlanSms / 2 ? 2 : 8; }

// The plain operator with rows read in place: the chain of a warp's views is long,
// so it is shared by up to eight warps until there are 1.75 rounds of the 3 resident
// blocks an SM.  128^2 x 130 x 360 (122 tiles of 8 rows), ms by split 0, 1, 2, 3:
// 0.199, 0.116, 0.079, 0.087.  A warp keeps seven views at least: with fewer the shares
// cost more to add than they take off the chain (64^2 x 66, 8 views, eight warps 14.4 us,
// one 10.6).  tiles(rows): tiles with work.
template <typename F>
inline BpPlan bp_split(int views, F&& tiles) {
  BpPlan p{8, 0};
  while (p.split < 3 && (views >> (p.split + 1)) >= 7 && tiles(p.rows) < 1.75 * 3 * kPlanSms) {
    ++p.split;
    p.rows >>= 1;
  }
  return p;
}

}  // namespace sipo
