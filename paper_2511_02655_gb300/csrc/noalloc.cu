// nbody_forces_noalloc: an entry point that computes the mixed-precision
// all-pairs forces of one system without allocating any memory.
//
// Who needs it: code that cannot call cudaMalloc at the point where it wants
// forces, e.g. a host program that runs under a fixed device-memory budget
// handed out by a surrounding framework, a plugin whose host only passes it
// ready-made device buffers, or a caller that must not trigger the allocator
// (and its implicit synchronisation) in the middle of its own work. The
// regular path needs an nbody_ctx, and creating one allocates the context's
// staging, partial-sum and work-list buffers; this entry point takes no
// context and allocates nothing.
//
// Its scratch lives in one file-scope __device__ array of fixed size, held on
// every GPU that loads the library's module until the process exits: the staging
// parameters and their partial sums, the float32 staging copy of the bodies and the
// float32 remainders the near-pair refinement reads, and in what those leave of
// the array the partial sums of the force passes. Host code cannot use the array's
// name as a device address (on the host it names a host-side stand-in), so
// the device address is looked up with cudaGetSymbolAddress once per device,
// on the first call made with that device current, and passed to the kernels.
//
// The force passes are those of the context path, their work items computed from
// the CTA's index instead of read from a list. The fewer the bodies, the more
// slots of partial sums the array has room for:
//   symmetric pass (sym_common.cuh) up to kMaxSymBodies, packed one-sided pass
//   in j-slices while there is a slot at all (524 288 bodies), writing the results
//   itself above.
// A single CTA per i-tile of scalar arithmetic, as it was, left most of the GPU idle:
// 20 001 bodies took 1.53 ms on 40 CTAs (and the staging origin, one CTA, 49 us);
// now the whole call takes 162 us (2.5e12 interactions/s).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <mutex>

#include "../../include/nbody.h"
#include "force_common.cuh"
#include "nbody_internal.h"
#include "pair_common.cuh"
#include "post_common.cuh"
#include "sym_common.cuh"

namespace nbody {
void set_global_error_text(const char* msg);  // capi.cu
}

namespace {

using namespace nbody;

constexpr int64_t kMaxBodies = NBODY_NOALLOC_MAX_BODIES;
constexpr int kSumCtas = 96;  // CTAs of the staging origin's sums
constexpr int kSumThreads = 256;
constexpr size_t kHeaderBytes = 8192;
constexpr size_t kSumsOffset = 256;  // header: SysParam, then the sums [kSumCtas][kEnergyVals]
constexpr size_t kScratchBytes = kHeaderBytes + 2 * sizeof(float4) * (size_t)kMaxBodies;
static_assert(sizeof(SysParam) <= kSumsOffset && kSumsOffset + kSumCtas * kEnergyVals * sizeof(double) <= kHeaderBytes,
              "header layout");
// Near-pair refinement radius: 4 softening lengths, as in the context path.
constexpr double kNearRadiusEps = 4.0;

// Layout: the header; then for n bodies the float4 staging entries [n], the float4 remainders
// [n] and slots of fpair4 [n] each, as many as fit.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

struct Scratch {
  SysParam* sys;
  double* sums;
  float4* st;
  float4* lo;
  fpair4* part;
};
__host__ __device__ inline Scratch scratch_of(unsigned char* p, const int n) {
  float4* st = reinterpret_cast<float4*>(p + kHeaderBytes);
  return Scratch{reinterpret_cast<SysParam*>(p), reinterpret_cast<double*>(p + kSumsOffset), st, st + n,
                 reinterpret_cast<fpair4*>(st + 2 * (size_t)n)};
}

constexpr int kMaxDevices = 64;
std::mutex g_mu;
void* g_scratch_addr[kMaxDevices] = {};
int g_sm_count[kMaxDevices] = {};  // set with the address

nbody_status fail(nbody_status s, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  nbody::set_global_error_text(buf);
  return s;
}

// Device memory of the current device holding at least `bytes` from p
// (the extent is checked where the driver can report the allocation's range).
nbody_status check_dev_ptr(const void* p, size_t bytes, int dev, const char* name, bool nullable) {
  if (!p) return nullable ? NBODY_OK : fail(NBODY_EINVAL, "nbody_forces_noalloc: %s is NULL", name);
  if (reinterpret_cast<uintptr_t>(p) % 8 != 0)
    return fail(NBODY_EINVAL, "nbody_forces_noalloc: %s is not 8-byte aligned", name);
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return fail(NBODY_EINVAL, "nbody_forces_noalloc: %s is not a CUDA pointer", name);
  }
  if (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged)
    return fail(NBODY_EINVAL, "nbody_forces_noalloc: %s is not device memory", name);
  if (at.type == cudaMemoryTypeDevice && at.device != dev)
    return fail(NBODY_EINVAL, "nbody_forces_noalloc: %s is on device %d, current device is %d", name, at.device, dev);
  size_t avail = 0;
  if (!nbody::allocation_holds(p, bytes, &avail))
    return fail(NBODY_EINVAL, "nbody_forces_noalloc: %s needs %zu bytes, its allocation holds %zu from that address",
                name, bytes, avail);
  return NBODY_OK;
}

// Sums of the staging origin and the extents, per CTA (fixed order: CTA-strided bodies).
__global__ void __launch_bounds__(kSumThreads) k_na_sums(const double* x, const double* m, const int n,
                                                         unsigned char* scratch) {
  constexpr int NW = kSumThreads / 32;
  __shared__ Extent ext[NW];
  pdl_wait();
  const Scratch S = scratch_of(scratch, n);
  double v[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  Extent q{0u, 0u, 1u};
  const double m0 = m[0];
  for (int64_t i = (int64_t)blockIdx.x * kSumThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kSumThreads)
    centre_terms(x[3 * i], x[3 * i + 1], x[3 * i + 2], m[i], x, m0, v, q);
  q.warp_join();
  if (threadIdx.x % 32 == 0) ext[threadIdx.x / 32] = q;
  block_sum<7, kSumThreads>(v);  // its barriers also publish ext
  if (threadIdx.x == 0) {
    for (int w = 1; w < NW; ++w) q.join(ext[w]);
    double* o = S.sums + (int64_t)blockIdx.x * kEnergyVals;
#pragma unroll
    for (int k = 0; k < 7; ++k) o[k] = v[k];
    o[7] = q.pack();
  }
}

// Staging: every CTA adds the n_sums partial sums itself (one warp, fixed order).
__global__ void __launch_bounds__(256) k_na_stage(const double* x, const double* m, const int n, const int n_sums,
                                                  const double eps, unsigned char* scratch) {
  __shared__ SysParam sp;
  pdl_wait();
  const Scratch S = scratch_of(scratch, n);
  if (threadIdx.x < 32) {
    double w[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    Extent e{0u, 0u, 1u};
    for (int k = (int)threadIdx.x; k < n_sums; k += 32) {
      const double* p = S.sums + (int64_t)k * kEnergyVals;
#pragma unroll
      for (int c = 0; c < 7; ++c) w[c] += p[c];
      e.join(Extent::unpack(p[7]));
    }
#pragma unroll
    for (int c = 0; c < 7; ++c) w[c] = warp_sum(w[c]);
    e.warp_join();
    if (threadIdx.x == 0) {
      staging_params(sp, w, e, n, x, m[0], true, eps, kNearRadiusEps);
      if (blockIdx.x == 0) *S.sys = sp;
    }
  }
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256)
    stage_store(1, S.st, (int)i, x[3 * i], x[3 * i + 1], x[3 * i + 2], m[i], sp, S.lo);
}

// ---- symmetric pass: rows of H bodies, row r in pieces of `step` j-bodies from its start on

constexpr int kMaxSymSlots = 96, kMaxRows = 64;

struct SymPlan {
  int n, H, step, rows;
  int first[kMaxRows + 1];  // first item of each row
  __host__ __device__ int pieces(const int r) const { return (n - r * H + step - 1) / step; }
  __host__ __device__ int slots(const int r) const { return r + 1 + pieces(r); }  // slots of a body of row r
};

// Above this size the slots (42 at the line) leave the symmetric pass too few and too large items
// to fill the GPU: whole calls at the line take 278 us with it (24 000 bodies) and 295 us one-sided
// (24 001); at 30 000 bodies its best plan took 591 us, the one-sided pass takes 443 us.
constexpr int kMaxSymBodies = 24000;

// Plan for i-tiles of `itile` bodies and `ctas` CTAs resident at once: pieces of equal pairs, long
// enough that all items run in one wave and the slots suffice, at least one 64-body block.
void plan_sym(const int n, const int itile, const int ctas, const int slots, SymPlan& P) {
  const int max_rows = std::min(kMaxRows, slots / 2 + 16);  // (slots >= 42: a row count of 37 or more is allowed)
  P.n = n;
  P.H = itile * ((n + itile * max_rows - 1) / (itile * max_rows));
  P.rows = (n + P.H - 1) / P.H;
  const double want = 0.5 * (double)n * ((double)n + P.H) / ctas / (double)P.H;
  P.step = 64 * std::max(1, (int)(want / 64.0));
  for (;; P.step += 64) {
    int most = 0;
    P.first[0] = 0;
    for (int r = 0; r < P.rows; ++r) {
      P.first[r + 1] = P.first[r] + P.pieces(r);
      most = std::max(most, P.slots(r));
    }
    if ((P.first[P.rows] <= ctas && most <= slots) || P.step >= n) return;  // (one piece per row: rows + 1 slots)
  }
}

template <int R, bool PHI>
__global__ void __launch_bounds__(128, R == 4 ? 4 : 6) k_na_force_sym(const SymPlan P, unsigned char* scratch) {
  extern __shared__ __align__(16) unsigned char raw[];
  auto& sm = *reinterpret_cast<sym::Smem<4, R, kSymTile>*>(raw);
  pdl_wait();
  pdl_trigger();
  const Scratch S = scratch_of(scratch, P.n);
  SymLaunch L{};
  L.stage_x = S.st, L.stage_lo = S.lo, L.part = reinterpret_cast<double*>(S.part), L.sys = S.sys;
  L.n_total = P.n, L.part_rows = (int64_t)kMaxBodies - P.n;
  bool done = false;
  auto next = [&](SymItem& it) {
    if (done) return false;
    done = true;
    int r = 0;
    while ((int)blockIdx.x >= P.first[r + 1]) ++r;
    const int k = (int)blockIdx.x - P.first[r], i0 = r * P.H;
    it = SymItem{0, i0, min(P.n, i0 + P.H), i0 + k * P.step, min(P.n, i0 + (k + 1) * P.step), r + 1 + k, r, P.n, 0};
    return true;
  };
  sym::items<0, 4, R, kSymTile, PHI>(L, next, sm);
}

// ---- one-sided pass: i-tiles of 256 bodies, `slices` equal j-slices of `len` bodies

constexpr int kOneTile = 512;

template <bool PHI, bool DIRECT>
__global__ void __launch_bounds__(128, 3) k_na_force_one(const int n, const int len, const double G, double* a,
                                                         double* phi, unsigned char* scratch) {
  __shared__ fc::SmemMixed2<kOneTile> sm;
  pdl_wait();
  pdl_trigger();
  const Scratch S = scratch_of(scratch, n);
  PairLaunch L{};
  L.stage_x = S.st, L.stage_lo = S.lo, L.sys = S.sys, L.n_total = n, L.sigma2 = 1.0;
  L.part_slices = 1 << 20, L.block_bodies = 256;
  bool done = false;
  auto next = [&] {
    const int it = done ? -1 : (int)blockIdx.x;
    done = true;
    return it;
  };
  auto item = [&](const int it) {
    const int tiles = (n + 255) / 256, t = it % tiles, s = it / tiles;
    return WorkItem{0, t * 256, min(n, t * 256 + 256), s * len, min(n, (s + 1) * len), s, s + 1};
  };
  auto put = [&](const WorkItem& w, const int i, const fpair4& q) {
    if (!DIRECT) {
      S.part[(int64_t)w.slice * n + i] = q;
      return;
    }
    const double gp = G * (S.sys->scale * S.sys->inv_mscale), ga = gp * S.sys->scale;
    a[3 * (int64_t)i + 0] = ga * ((double)q.xy.x + (double)q.xy.y);
    a[3 * (int64_t)i + 1] = ga * ((double)q.xy.z + (double)q.xy.w);
    a[3 * (int64_t)i + 2] = ga * ((double)q.zp.x + (double)q.zp.y);
    if (PHI) phi[i] = -gp * ((double)q.zp.z + (double)q.zp.w);
  };
  fc::items_mixed2<0, 128, 2, kOneTile, PHI>(L, next, item, put, sm);
}

// a and phi from the slots (row height H > 0: a symmetric plan's, else `slices` for every body):
// four threads per body, as in the O(N) kernels of the context path.
__global__ void __launch_bounds__(256) k_na_combine(const SymPlan P, const int n, const int slices, const double G,
                                                    double* a, double* phi, unsigned char* scratch) {
  constexpr int CB = 64, SG = 4;
  __shared__ SlotSums<CB, SG> red[4];
  pdl_wait();
  pdl_trigger();
  const Scratch S = scratch_of(scratch, n);
  const int b = (int)threadIdx.x % CB, g = (int)threadIdx.x / CB, i = (int)blockIdx.x * CB + b;
  float h[4] = {0.f, 0.f, 0.f, 0.f}, l[4] = {0.f, 0.f, 0.f, 0.f};
  if (i < n) {
    const int ns = P.H > 0 ? P.slots(i / P.H) : slices;
    const fpair4* p = S.part + i;
#pragma unroll 8
    for (int s = g; s < ns; s += SG) add_slot(p[(int64_t)s * n], h, l);
  }
  add_groups(red, g, b, h, l);
  if (g != 0 || i >= n) return;
  const double gp = G * (S.sys->scale * S.sys->inv_mscale), ga = gp * S.sys->scale;
  a[3 * (int64_t)i + 0] = ga * ((double)h[0] + (double)l[0]);
  a[3 * (int64_t)i + 1] = ga * ((double)h[1] + (double)l[1]);
  a[3 * (int64_t)i + 2] = ga * ((double)h[2] + (double)l[2]);
  if (phi) phi[i] = -gp * ((double)h[3] + (double)l[3]);
}

template <int R>
cudaError_t launch_na_sym(const SymPlan& P, bool phi, unsigned char* sp, cudaStream_t st) {
  constexpr size_t smem = sizeof(sym::Smem<4, R, kSymTile>);
  static_assert(smem <= 48 * 1024, "no opt-in needed");
  return phi ? launch_pdl_smem(k_na_force_sym<R, true>, P.first[P.rows], 128, smem, st, P, sp)
             : launch_pdl_smem(k_na_force_sym<R, false>, P.first[P.rows], 128, smem, st, P, sp);
}

cudaError_t enqueue(const double* x, const double* m, const int n, const double G, const double eps, double* a,
                    double* phi, unsigned char* sp, const int n_sms, cudaStream_t st) {
  cudaError_t e;
  const int n_sums = std::min(kSumCtas, (n + kSumThreads - 1) / kSumThreads);
  if ((e = launch_pdl(k_na_sums, n_sums, kSumThreads, st, x, m, n, sp))) return e;
  if ((e = launch_pdl(k_na_stage, std::min((n + 255) / 256, 4096), 256, st, x, m, n, n_sums, eps, sp))) return e;
  const int room = (int)((kMaxBodies - n) / n);  // slots
  SymPlan P{};
  int slices = 0;
  if (n <= kMaxSymBodies) {
    // short i-tiles for small systems: their few tiles would leave SMs idle
    const int R = n <= 2048 ? 1 : n <= 8192 ? 2 : 4;
    plan_sym(n, 128 * R, n_sms * (R == 4 ? 4 : 6), std::min(room, kMaxSymSlots), P);
    e = R == 1   ? launch_na_sym<1>(P, phi != nullptr, sp, st)
        : R == 2 ? launch_na_sym<2>(P, phi != nullptr, sp, st)
                 : launch_na_sym<4>(P, phi != nullptr, sp, st);
  } else {
    P = SymPlan{};
    // about eight items per resident CTA (3 per SM)
    const int tiles = (n + 255) / 256;
    slices = std::max(1, std::min(room, (8 * 3 * n_sms + tiles - 1) / tiles));
    const int len = std::max(4, 4 * (int)(((int64_t)n + 4 * slices - 1) / (4 * slices)));
    slices = (n + len - 1) / len;
    const unsigned grid = (unsigned)tiles * (unsigned)slices;
    if (room < 1) {
      return phi ? launch_pdl(k_na_force_one<true, true>, grid, 128, st, n, len, G, a, phi, sp)
                 : launch_pdl(k_na_force_one<false, true>, grid, 128, st, n, len, G, a, phi, sp);
    }
    e = phi ? launch_pdl(k_na_force_one<true, false>, grid, 128, st, n, len, G, a, phi, sp)
            : launch_pdl(k_na_force_one<false, false>, grid, 128, st, n, len, G, a, phi, sp);
  }
  if (e) return e;
  return launch_pdl(k_na_combine, (n + 63) / 64, 256, st, P, n, slices, G, a, phi, sp);
}

// Loads the code of every kernel of this entry point on the current device: functions are
// loaded on first use otherwise, and a later call of another size would allocate.
cudaError_t load_kernels() {
  cudaFuncAttributes at;
  for (const void* f :
       {(const void*)k_na_sums, (const void*)k_na_stage, (const void*)k_na_combine,
        (const void*)k_na_force_sym<1, true>, (const void*)k_na_force_sym<1, false>,
        (const void*)k_na_force_sym<2, true>, (const void*)k_na_force_sym<2, false>,
        (const void*)k_na_force_sym<4, true>, (const void*)k_na_force_sym<4, false>,
        (const void*)k_na_force_one<true, true>, (const void*)k_na_force_one<true, false>,
        (const void*)k_na_force_one<false, true>, (const void*)k_na_force_one<false, false>})
    if (const cudaError_t e = cudaFuncGetAttributes(&at, f)) return e;
  return cudaSuccess;
}

}  // namespace

extern "C" nbody_status nbody_forces_noalloc(const double* x, const double* m, int64_t n, double G, double eps,
                                             double* a, double* phi, void* cuda_stream) {
  if (n < 0 || n > kMaxBodies)
    return fail(NBODY_EINVAL, "nbody_forces_noalloc: n = %lld is outside [0, %lld] (NBODY_NOALLOC_MAX_BODIES)",
                (long long)n, (long long)kMaxBodies);
  if (!std::isfinite(G) || !std::isfinite(eps) || eps < 0)
    return fail(NBODY_EINVAL, "nbody_forces_noalloc: G must be finite and eps finite and >= 0");
  if (n == 0) return NBODY_OK;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return fail(NBODY_EUNSUPPORTED, "nbody_forces_noalloc: no usable current CUDA device");
  }
  nbody_status s;
  const size_t n3b = (size_t)n * 3 * sizeof(double), n1b = (size_t)n * sizeof(double);
  if ((s = check_dev_ptr(x, n3b, dev, "x", false)) || (s = check_dev_ptr(m, n1b, dev, "m", false)) ||
      (s = check_dev_ptr(a, n3b, dev, "a", false)) || (s = check_dev_ptr(phi, n1b, dev, "phi", true)))
    return s;
  void* scratch = nullptr;
  int n_sms = 0;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_scratch_addr[dev]) {
      void* p = nullptr;
      cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e == cudaSuccess) e = load_kernels();
      if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g_sm_count[dev], cudaDevAttrMultiProcessorCount, dev);
      if (e != cudaSuccess || !p) {
        cudaGetLastError();
        return fail(NBODY_ECUDA, "nbody_forces_noalloc: loading the device code failed on device %d: %s", dev,
                    cudaGetErrorString(e));
      }
      g_scratch_addr[dev] = p;
    }
    scratch = g_scratch_addr[dev];
    n_sms = g_sm_count[dev];
  }
  const cudaError_t e = enqueue(x, m, (int)n, G, eps, a, phi, static_cast<unsigned char*>(scratch),
                                n_sms, static_cast<cudaStream_t>(cuda_stream));
  if (e != cudaSuccess) return fail(NBODY_ECUDA, "nbody_forces_noalloc: launch failed: %s", cudaGetErrorString(e));
  return NBODY_OK;
}
