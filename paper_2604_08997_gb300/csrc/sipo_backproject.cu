// Instantiations of the backprojector P_mu^T for every storage type and
// epilogue used by the library.
#include <cudaTypedefs.h>

#include <mutex>

#include "sipo_bp_tma.cuh"
#include "sipo_flat.cuh"
#include "sipo_launch.h"
#include "sipo_ops.cuh"

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

namespace {

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static std::once_flag once;
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// 3-D tensor map of a sinogram [na][nd][nz] with boxes of T z x `rows` bins
// x 1 view; what lies outside reads as zeros.  False when the map cannot be made
// (no driver entry point, unaligned buffer or stride).
template <typename SI>
bool sino_map(const SI* sino, int nz, int nd, int na, int T, int rows, CUtensorMap* map) {
  const auto fn = encode_fn();
  if (!fn || (reinterpret_cast<uintptr_t>(sino) & 15u) != 0 || (nz * sizeof(SI)) % 16 != 0) return false;
  const cuuint64_t dims[3] = {cuuint64_t(nz), cuuint64_t(nd), cuuint64_t(na)};
  const cuuint64_t strides[2] = {cuuint64_t(nz) * sizeof(SI), cuuint64_t(nz) * nd * sizeof(SI)};
  const cuuint32_t box[3] = {cuuint32_t(T), cuuint32_t(rows), 1u};
  const cuuint32_t estr[3] = {1u, 1u, 1u};
  const CUtensorMapDataType dt = sizeof(SI) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  return fn(map, dt, 3, const_cast<SI*>(sino), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <typename SI, typename S, int NG, int ROWS, int MODE, typename O>
bool launch_bp_tma(const Geo<float>& g, const SI* sino, const Bufs<S, float>& b, O* out, const uint8_t* need,
                   const BpTiles& tiles, cudaStream_t stream) {
  CUtensorMap map;
  if (reinterpret_cast<uintptr_t>(out) % 16 != 0 || 
      !sino_map<SI>(sino, g.nz, g.nd, g.na, 128 * NG, bt_bins<ROWS>(), &map))
    return false;
  constexpr size_t bytes = BtSmem<SI, NG, ROWS>::kBytes;
  // more than the 48 KB default of dynamic shared memory (per device, cheap)
  if (cudaFuncSetAttribute(k_backproject_tma<SI, S, NG, ROWS, MODE, O>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           int(bytes)) != cudaSuccess)
    return false;
  k_backproject_tma<SI, S, NG, ROWS, MODE, O><<<kRedBlocks, 32 * (ROWS + 1), bytes, stream>>>(g, map, b, out, need, tiles);
  return true;
}

}  // namespace

template <typename SI, typename S, typename C, int MODE, typename O>
void launch_backproject(const Geo<C>& g, const SI* sino, const Bufs<S, C>& b, O* out,
                        const uint8_t* need, cudaStream_t stream, const BpTiles& tiles, int tile) {
  if (bp_flat<C>(g.nx, g.ny, g.nz)) {
    k_backproject_flat<SI, S, C, MODE, O><<<kRedBlocks, kThreads, 0, stream>>>(g, sino, b, out, need);
    return;
  }
  if constexpr (std::is_same<C, float>::value) {
    if (tile >= 5 && bp_staged<SI>(g.nz)) {
      auto go = [&](auto ng) {
        constexpr int NG = decltype(ng)::value;
        return tiles.rows == 8 ? launch_bp_tma<SI, S, NG, 8, MODE, O>(g, sino, b, out, need, tiles, stream)
                               : launch_bp_tma<SI, S, NG, 2, MODE, O>(g, sino, b, out, need, tiles, stream);
      };
      // two groups a lane unless they would leave more than a quarter of the lanes idle
      const bool two = (g.nz + 255) / 256 * 3 <= (g.nz + 127) / 128 * 2;
      if (two ? go(std::integral_constant<int, 2>{}) : go(std::integral_constant<int, 1>{}))
        return;  // else no tensor map: the kernel with global loads
    }
    with_z_form<C>(g.nz, z_group_for<C>(g.nz, sino, out), [&](auto form) {
      using Z = decltype(form);
      const int threads = 32 * tiles.rows << tiles.split;
      const size_t bytes = size_t(threads / 32) * bp2_warp_bytes<Z>();
      if (tile == 0 || tile == 1 || tile == 3)
        k_backproject2<SI, S, Z, 2, MODE, O><<<kRedBlocks, threads, bytes, stream>>>(g, sino, b, out, need, tiles);
      else
        k_backproject2<SI, S, Z, 3, MODE, O><<<kRedBlocks, threads, bytes, stream>>>(g, sino, b, out, need, tiles);
    }, MODE == kBpDual && g.nz % 4 == 0);
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
