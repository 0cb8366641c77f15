// Launchers of the symmetric force-gradient pass (sym_vjp.cuh).
#include <algorithm>

#include "nbody_internal.h"
#include "sym_vjp.cuh"

namespace nbody {
namespace {

// MINB resident CTAs per SM (a register bound of 65 536 / (threads x MINB))
template <int W, int R, bool P, int MINB>
__global__ void __launch_bounds__(W * 32, MINB) k_vjp_sym(const SymLaunch L) {
  extern __shared__ __align__(16) unsigned char raw[];
  auto& sm = *reinterpret_cast<symv::Smem<W, R, P>*>(raw);
  pdl_wait();
  symv::items<W, R, P>(L, L.counter, sm);
  pdl_trigger();
  retire_cta(L.counter);
}

template <int W, bool P>
__global__ void __launch_bounds__(W * 32) k_vjp_sym64(const SymLaunch L) {
  extern __shared__ __align__(16) unsigned char raw[];
  auto& sm = *reinterpret_cast<symv::Smem64<W, P>*>(raw);
  pdl_wait();
  symv::items64<W, P>(L, L.counter, sm);
  pdl_trigger();
  retire_cta(L.counter);
}

template <typename K>
int occupancy_of(K kern, int block, size_t smem) {
  int n = 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, block, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

}  // namespace

// Compiled: warps, i-bodies per lane, resident CTAs (mixed); warps (FP64)
#define NBODY_SYM_VJP_TILINGS(X) X(4, 1, 5) X(4, 2, 3) X(8, 2, 1)
#define NBODY_SYM_VJP64_TILINGS(X) X(2) X(4) X(8)

cudaError_t launch_sym_vjp(int precision, const SymLaunch& L, cudaStream_t st) {
  if (L.n_ctas <= 0) return cudaErrorInvalidConfiguration;
  if (precision == 1) {
#define NBODY_X(W, R, MINB)                                                                                           \
  if (L.block == W * 32 && L.ipt == R)                                                                                \
    return L.params                                                                                                   \
               ? launch_pdl_smem(k_vjp_sym<W, R, true, MINB>, L.n_ctas, W * 32, sizeof(symv::Smem<W, R, true>), st, L) \
               : launch_pdl_smem(k_vjp_sym<W, R, false, MINB>, L.n_ctas, W * 32, sizeof(symv::Smem<W, R, false>), st, L);
    NBODY_SYM_VJP_TILINGS(NBODY_X)
#undef NBODY_X
    return cudaErrorInvalidConfiguration;
  }
#define NBODY_X(W)                                                                                                    \
  if (L.block == W * 32 && L.ipt == 1)                                                                                \
    return L.params ? launch_pdl_smem(k_vjp_sym64<W, true>, L.n_ctas, W * 32, sizeof(symv::Smem64<W, true>), st, L)   \
                    : launch_pdl_smem(k_vjp_sym64<W, false>, L.n_ctas, W * 32, sizeof(symv::Smem64<W, false>), st, L);
  NBODY_SYM_VJP64_TILINGS(NBODY_X)
#undef NBODY_X
  return cudaErrorInvalidConfiguration;
}

int sym_vjp_ctas_per_sm(int precision, int block, int ipt) {
  if (precision == 1) {
#define NBODY_X(W, R, MINB)                                                                              \
  if (block == W * 32 && ipt == R)                                                                       \
    return std::min(occupancy_of(k_vjp_sym<W, R, true, MINB>, W * 32, sizeof(symv::Smem<W, R, true>)),   \
                    occupancy_of(k_vjp_sym<W, R, false, MINB>, W * 32, sizeof(symv::Smem<W, R, false>)));
    NBODY_SYM_VJP_TILINGS(NBODY_X)
#undef NBODY_X
    return 0;
  }
#define NBODY_X(W)                                                                               \
  if (block == W * 32 && ipt == 1)                                                               \
    return std::min(occupancy_of(k_vjp_sym64<W, true>, W * 32, sizeof(symv::Smem64<W, true>)),   \
                    occupancy_of(k_vjp_sym64<W, false>, W * 32, sizeof(symv::Smem64<W, false>)));
  NBODY_SYM_VJP64_TILINGS(NBODY_X)
#undef NBODY_X
  return 0;
}

}  // namespace nbody
