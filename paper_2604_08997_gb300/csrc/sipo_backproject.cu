// Instantiations of the backprojector P_mu^T for every storage type and
// epilogue used by the library.
#include "sipo_flat.cuh"
#include "sipo_launch.h"
#include "sipo_ops.cuh"
#include "sipo_wait.cuh"

#include <type_traits>

namespace sipo {

// Bits recorded by this translation unit's kernels in a checked build (0 in
// plain builds); cleared by the read.
unsigned int check_flags_backproject() {
#ifdef SIPO_CHECKED
  unsigned int v = 0, zero = 0;
  if (cudaMemcpyFromSymbol(&v, g_sipo_check, sizeof(v)) != cudaSuccess) return 0;
  cudaMemcpyToSymbol(g_sipo_check, &zero, sizeof(zero));
  return v;
#else
  return 0;
#endif
}


int wait_selftest(long long budget, int arrive, int threads, unsigned int* timed_out) {
  unsigned int* d = nullptr;
  if (cudaMalloc(&d, sizeof(unsigned int)) != cudaSuccess) return -1;
  cudaError_t e = cudaMemset(d, 0, sizeof(unsigned int));
  if (e == cudaSuccess) {
    k_wait_selftest<<<1, threads>>>(budget, arrive, d);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpy(timed_out, d, sizeof(unsigned int), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? 0 : -1;
}

template <typename SI, typename S, typename C, int MODE, typename O>
void launch_backproject(const Geo<C>& g, const SI* sino, const Bufs<S, C>& b, O* out,
                        const uint8_t* need, cudaStream_t stream, const BpTiles& tiles, int tile) {
  if (bp_flat<C>(g.nz)) {
    k_backproject_flat<SI, S, C, MODE, O><<<kRedBlocks, kThreads, 0, stream>>>(g, sino, b, out, need);
    return;
  }
  if constexpr (std::is_same<C, float>::value) {
    with_z_form<C>(g.nz, z_group_for<C>(g.nz, sino, out), [&](auto form) {
      using Z = decltype(form);
      if (tile == 0 || tile == 1 || tile == 3)
        k_backproject2<SI, S, Z, 2, MODE, O><<<kRedBlocks, kThreads, 0, stream>>>(g, sino, b, out, need, tiles);
      else
        k_backproject2<SI, S, Z, 3, MODE, O><<<kRedBlocks, kThreads, 0, stream>>>(g, sino, b, out, need, tiles);
    });
  } else {
    auto go = [&](auto zl) {
      constexpr int ZL = decltype(zl)::value;
      if (tile == 0)
        k_backproject<SI, S, C, ZL, 8, 2, MODE, O><<<kRedBlocks, kThreads, 0, stream>>>(g, sino, b, out, need);
      else if (tile == 1)
        k_backproject<SI, S, C, ZL, 4, 2, MODE, O><<<kRedBlocks, kThreads, 0, stream>>>(g, sino, b, out, need);
      else
        k_backproject<SI, S, C, ZL, 4, 3, MODE, O><<<kRedBlocks, kThreads, 0, stream>>>(g, sino, b, out, need);
    };
    const int G = z_group_for<C>(g.nz, sino, out);
    if (G == 2 && g.nz % 128 == 0) go(std::integral_constant<int, 4>{});
    else if (G == 2 && g.nz > 32) go(std::integral_constant<int, 2>{});
    else go(std::integral_constant<int, 1>{});
  }
}

#define SIPO_BP(SI, S, C, M, O) \
  template void launch_backproject<SI, S, C, M, O>(const Geo<C>&, const SI*, const Bufs<S, C>&, \
                                                    O*, const uint8_t*, cudaStream_t, const BpTiles&, int);
#define SIPO_BP_SOLVER(S, C)       \
  SIPO_BP(S, S, C, kBpDual, C)     \
  SIPO_BP(S, S, C, kBpStore, C)

SIPO_BP_SOLVER(float, float)
SIPO_BP_SOLVER(__nv_bfloat16, float)
SIPO_BP_SOLVER(double, double)

}  // namespace sipo
