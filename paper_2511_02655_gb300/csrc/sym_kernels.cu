// Launchers of the symmetric force pass (sym_common.cuh).
#include <algorithm>
#include <type_traits>

#include "nbody_internal.h"
#include "sym64.cuh"
#include "sym_common.cuh"

namespace nbody {
namespace {

// MINB resident CTAs per SM: 16 warps per SM at R = 4 (<= 128 registers), 24 at R = 2
// (<= 80 registers).
template <int LAW, int W, int R, int PHI, int MINB>
__global__ void __launch_bounds__(W * 32, MINB) k_force_sym(const SymLaunch L) {
  extern __shared__ __align__(16) unsigned char raw[];
  auto& sm = *reinterpret_cast<sym::Smem<W, R, kSymTile>*>(raw);
  pdl_wait();
  ItemSource source{L.counter, &sm.item};
  auto next = [&](SymItem& it) {
    const int n = source.next();
    if (n < L.n_items) it = L.items[n];
    return n < L.n_items;
  };
  sym::items<LAW, W, R, kSymTile, PHI>(L, next, sm);
  pdl_trigger();
  retire_cta(L.counter);
}

// With 4 warps to a block of the work 24 warps per SM are resident at most (short lists): left to
// itself the compiler keeps to 64 registers and spills.
template <int LAW, int W, int R, int PHI, int KS>
__global__ void __launch_bounds__(W * KS * 32, KS < 4 ? 0 : std::max(1, 24 / (W * KS)))
    k_force_sym64(const SymLaunch L) {
  __shared__ sym64::Smem<W * KS> sm;
  pdl_wait();
  sym64::items<LAW, W, R, PHI, KS>(L, L.counter, sm);
  pdl_trigger();
  retire_cta(L.counter);
}

// More than 48 KB of shared memory per CTA has to be asked for, once per kernel and device.
template <typename K>
cudaError_t allow_smem(K kern, size_t bytes) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <typename K>
int occupancy_of(K kern, int block, size_t smem) {
  int n = 0;
  if (allow_smem(kern, smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, block, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

}  // namespace

// Compiled: warps, i-bodies per lane (and resident CTAs).
#define NBODY_SYM_TILINGS(X) X(4, 2, 6) X(4, 4, 4) X(8, 2, 3) X(8, 4, 2)
#define NBODY_SYM64_TILINGS(X) X(2, 1) X(4, 1) X(8, 1) X(4, 2)
// ... of which these also exist with 2 and 4 warps to a block of the work (SymLaunch::split)
#define NBODY_SYM64_SPLITS(X) X(2, 1) X(4, 1)

// f(law, potential) as integral constants
template <typename F>
static auto with_modes(const int law, const int phi, F f) {
  using std::integral_constant;
  auto with_law = [&](auto l) {
    return phi == sym::kPhiBoth     ? f(l, integral_constant<int, sym::kPhiBoth>())
           : phi == sym::kPhiEnergy ? f(l, integral_constant<int, sym::kPhiEnergy>())
                                    : f(l, integral_constant<int, sym::kPhiNone>());
  };
  return law == 0 ? with_law(integral_constant<int, 0>()) : with_law(integral_constant<int, 1>());
}

cudaError_t launch_sym_force(int precision, const SymLaunch& L, cudaStream_t st) {
  if (L.n_ctas <= 0) return cudaErrorInvalidConfiguration;
  return with_modes(L.law, L.phi, [&](auto law, auto phi) -> cudaError_t {
    constexpr int LAW = decltype(law)::value, PHI = decltype(phi)::value;
    if (precision == 0) {
#define NBODY_X(W, R)                                                                                              \
  if (L.block == W * 32 && L.ipt == R && L.split == 4)                                                             \
    return launch_pdl(k_force_sym64<LAW, W, R, PHI, 4>, L.n_ctas, W * 128, st, L);                                 \
  if (L.block == W * 32 && L.ipt == R && L.split == 2)                                                             \
    return launch_pdl(k_force_sym64<LAW, W, R, PHI, 2>, L.n_ctas, W * 64, st, L);
      NBODY_SYM64_SPLITS(NBODY_X)
#undef NBODY_X
#define NBODY_X(W, R) \
  if (L.block == W * 32 && L.ipt == R) return launch_pdl(k_force_sym64<LAW, W, R, PHI, 1>, L.n_ctas, W * 32, st, L);
      NBODY_SYM64_TILINGS(NBODY_X)
#undef NBODY_X
      return cudaErrorInvalidConfiguration;
    }
#define NBODY_X(W, R, MINB)            \
  if (L.block == W * 32 && L.ipt == R) \
    return launch_pdl_smem(k_force_sym<LAW, W, R, PHI, MINB>, L.n_ctas, W * 32, sizeof(sym::Smem<W, R, kSymTile>), st, L);
    NBODY_SYM_TILINGS(NBODY_X)
#undef NBODY_X
    return cudaErrorInvalidConfiguration;
  });
}

// the occupancy that every potential mode of the tiling reaches
int sym_force_ctas_per_sm(int precision, int block, int ipt, int law) {
  int least = 1 << 20;
  for (int mode : {sym::kPhiNone, sym::kPhiBoth, sym::kPhiEnergy})
    least = std::min(least, with_modes(law, mode, [&](auto l, auto phi) -> int {
              constexpr int LAW = decltype(l)::value, PHI = decltype(phi)::value;
              if (precision == 0) {
#define NBODY_X(W, R) \
  if (block == W * 32 && ipt == R) return occupancy_of(k_force_sym64<LAW, W, R, PHI, 1>, W * 32, 0);
                NBODY_SYM64_TILINGS(NBODY_X)
#undef NBODY_X
                return 0;
              }
#define NBODY_X(W, R, MINB)        \
  if (block == W * 32 && ipt == R) \
    return occupancy_of(k_force_sym<LAW, W, R, PHI, MINB>, W * 32, sizeof(sym::Smem<W, R, kSymTile>));
              NBODY_SYM_TILINGS(NBODY_X)
#undef NBODY_X
              return 0;
            }));
  return least;
}

}  // namespace nbody
