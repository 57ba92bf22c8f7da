// Instantiations of the projector P_mu (gather form) for every storage type
// and epilogue used by the library.
#include "sipo_launch.h"
#include "sipo_flat.cuh"
#include "sipo_ops.cuh"
#include "sipo_pair.cuh"

#include <algorithm>

namespace sipo {

// Bits recorded by this translation unit's kernels in a checked build (0 in
// plain builds); cleared by the read.
unsigned int check_flags_project() {
#ifdef SIPO_CHECKED
  unsigned int v = 0, zero = 0;
  if (cudaMemcpyFromSymbol(&v, g_sipo_check, sizeof(v)) != cudaSuccess) return 0;
  cudaMemcpyToSymbol(g_sipo_check, &zero, sizeof(zero));
  return v;
#else
  return 0;
#endif
}


// bits[line][word] from flags need[y][x]; by_rows selects line = y (bits over
// x) or line = x (bits over y).
__global__ void k_need_bits(const uint8_t* __restrict__ need, uint32_t* __restrict__ bits, int nx, int ny,
                            int words, int by_rows) {
  const int lines = by_rows ? ny : nx, len = by_rows ? nx : ny;
  const long long n = (long long)lines * words;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int line = int(i / words), w = int(i % words);
    uint32_t v = 0;
    for (int bt = 0; bt < 32; ++bt) {
      const int pos = w * 32 + bt - kNbPad;
      if (pos >= 0 && pos < len) {
        const int x = by_rows ? pos : line, y = by_rows ? line : pos;
        if (need[(size_t)y * nx + x]) v |= 1u << bt;
      }
    }
    bits[i] = v;
  }
}


template <typename SI, typename S, typename C, int MODE, typename O>
void launch_project(const Geo<C>& g, const SI* vol, const Bufs<S, C>& b, O* out,
                    const uint8_t* act_col, cudaStream_t stream, const NeedBits& nb,
                    const int2* rspan) {
  // the slice-mode certificate keeps one 8-byte maximum per z in shared memory
  const size_t dyn = MODE == kFpCertZ ? size_t(g.nz) * sizeof(unsigned long long) : 0;
  const int gmax = z_group_for<C>(g.nz, vol, out);
  // the modes of the check step have sums, whose order follows the form: they keep
  // one rule by extent (they run once a period).  bf16 steps always take pairs: the
  // compiler rounds their Halpern step in another order from kernel to kernel, and
  // bf16 iterates show it (2e-2 after two periods).
  constexpr bool kPairs = sizeof(C) == 4 && (MODE == kFpPrimal || MODE == kFpStore);
  constexpr bool kPlanned = kPairs && (MODE == kFpStore || sizeof(S) == 4);
  bool flat = fp_flat<C>(g);
  FpPlan plan{flat, true, 0.0};
  if constexpr (kPlanned) {
    plan = fp_plan<C>(g, gmax, flat);
    flat = plan.flat;
  }
  if (flat) {
    // a solver's input vanishes outside its flagged columns; those may lie
    // outside the vial where a PSF spreads them
    const bool wide = nb.rows != nullptr && g.r2i >= 0 && nb.spread;
    k_project_flat<SI, S, C, MODE, O><<<kRedBlocks, kThreads, dyn, stream>>>(g, vol, b, out, act_col, rspan, wide);
    return;
  }
  with_z_form<C>(g.nz, gmax, [&](auto form) {
    using Z = decltype(form);
    if constexpr (kPairs) {
      // 4 views a tile: 0.344 / 0.560 ms on two targets at 256^3 x 360, 8 views 0.321 / 0.587;
      // 96^3 x 391 0.0529, 0.0552.  One view a tile on few warps: the same within 4%.
      if (!kPlanned || plan.pair)
        k_project_pair<SI, S, Z, MODE, O><<<kRedBlocks, kThreads, 0, stream>>>(g, vol, b, out, act_col, nb, rspan, 4);
      else if constexpr (kPlanned)
        k_project<SI, S, C, Z, MODE, O><<<kRedBlocks, kThreads, 0, stream>>>(g, vol, b, out, act_col, nb, rspan, 4);
    } else {
      // Views per tile: 4 where every block has several tiles to even out, else 1.
      // 256^3 x 360 (9.5 tiles a block): 0.420 ms with 1, 0.394 with 2, 0.360 with 4,
      // 0.364 with 8 (another target: 0.704, 0.605, 0.616, 0.655); 96^3 x 391 (4
      // tiles a block): 0.067 ms with 1, 0.072 with 4.
      const long long tiles = (long long)g.na * ((g.nd + kWarps - 1) / kWarps) * ((g.nz + Z::T - 1) / Z::T);
      const int aw = tiles >= 8LL * kRedBlocks ? 4 : 1;
      k_project<SI, S, C, Z, MODE, O><<<kRedBlocks, kThreads, dyn, stream>>>(g, vol, b, out, act_col, nb, rspan, aw);
    }
  }, false, plan.warps);
}

void launch_need_bits(const uint8_t* need, uint32_t* rows, uint32_t* cols, int nx, int ny, int wr, int wc,
                      cudaStream_t stream) {
  const int gr = int(std::min<long long>(((long long)ny * wr + kThreads - 1) / kThreads, (long long)device_sms() * 16));
  const int gc = int(std::min<long long>(((long long)nx * wc + kThreads - 1) / kThreads, (long long)device_sms() * 16));
  k_need_bits<<<gr, kThreads, 0, stream>>>(need, rows, nx, ny, wr, 1);
  k_need_bits<<<gc, kThreads, 0, stream>>>(need, cols, nx, ny, wc, 0);
}

template <typename C>
void launch_ray_spans(const Geo<C>& g, const uint8_t* need, int2* out, cudaStream_t stream) {
  const long long n = (long long)g.na * g.nd;
  const int grid = int(std::min<long long>((n + kWarps - 1) / kWarps, (long long)device_sms() * 16));
  k_ray_spans<C><<<grid, kThreads, 0, stream>>>(g, need, out);
}
template void launch_ray_spans<float>(const Geo<float>&, const uint8_t*, int2*, cudaStream_t);
template void launch_ray_spans<double>(const Geo<double>&, const uint8_t*, int2*, cudaStream_t);

#define SIPO_FP(SI, S, C, M, O) \
  template void launch_project<SI, S, C, M, O>(const Geo<C>&, const SI*, const Bufs<S, C>&, O*, \
                                                const uint8_t*, cudaStream_t, const NeedBits&, \
                                                const int2*);
#define SIPO_FP_SOLVER(S, C)          \
  SIPO_FP(S, S, C, kFpPrimal, C)      \
  SIPO_FP(S, S, C, kFpPrimalCheck, C) \
  SIPO_FP(S, S, C, kFpResid, C)

SIPO_FP_SOLVER(float, float)
SIPO_FP_SOLVER(__nv_bfloat16, float)
SIPO_FP_SOLVER(double, double)
// bound-based certificate: the candidate volume is in the compute type
SIPO_FP(float, float, float, kFpCert, float)
SIPO_FP(float, __nv_bfloat16, float, kFpCert, float)
SIPO_FP(double, double, double, kFpCert, double)
SIPO_FP(float, float, float, kFpCertZ, float)
SIPO_FP(float, __nv_bfloat16, float, kFpCertZ, float)
SIPO_FP(double, double, double, kFpCertZ, double)
SIPO_FP(float, float, float, kFpStore, float)
SIPO_FP(double, double, double, kFpStore, double)
SIPO_FP(__nv_bfloat16, __nv_bfloat16, float, kFpStore, float)

}  // namespace sipo
