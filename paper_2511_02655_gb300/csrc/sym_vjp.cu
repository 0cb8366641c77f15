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

template <int W, bool P, int KS>
__global__ void __launch_bounds__(W * KS * 32) k_vjp_sym64(const SymLaunch L) {
  extern __shared__ __align__(16) unsigned char raw[];
  auto& sm = *reinterpret_cast<symv::Smem64<W * KS, P>*>(raw);
  pdl_wait();
  symv::items64<W, P, KS>(L, L.counter, sm);
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

// Compiled: warps, i-bodies per lane, resident CTAs (mixed); warps and warps to a block of the work (FP64,
// SymLaunch::split)
#define NBODY_SYM_VJP_TILINGS(X) X(4, 1, 5) X(4, 2, 3) X(8, 2, 1)
#define NBODY_SYM_VJP64_TILINGS(X) X(2, 1) X(2, 2) X(2, 4) X(4, 1) X(4, 2) X(4, 4) X(8, 1)

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
#define NBODY_X(W, KS)                                                                                              \
  if (L.block == W * 32 && L.ipt == 1 && (L.split == KS || W == 8))                                                 \
    return L.params ? launch_pdl_smem(k_vjp_sym64<W, true, KS>, L.n_ctas, W * KS * 32,                              \
                                      sizeof(symv::Smem64<W * KS, true>), st, L)                                    \
                    : launch_pdl_smem(k_vjp_sym64<W, false, KS>, L.n_ctas, W * KS * 32,                             \
                                      sizeof(symv::Smem64<W * KS, false>), st, L);
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
  // (of the unsplit kernel; the shared ones are for lists that leave most of the chip free anyway,
  // and asking for them here allows their shared memory as well)
  int n = 0;
#define NBODY_X(W, KS)                                                                                            \
  if (block == W * 32 && ipt == 1) {                                                                              \
    const int k = std::min(occupancy_of(k_vjp_sym64<W, true, KS>, W * KS * 32, sizeof(symv::Smem64<W * KS, true>)),   \
                           occupancy_of(k_vjp_sym64<W, false, KS>, W * KS * 32, sizeof(symv::Smem64<W * KS, false>))); \
    if (k <= 0) return 0;                                                                                         \
    if (KS == 1) n = k;                                                                                           \
  }
  NBODY_SYM_VJP64_TILINGS(NBODY_X)
#undef NBODY_X
  return n;
}

}  // namespace nbody
