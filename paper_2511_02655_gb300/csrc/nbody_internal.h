// Internal declarations shared by the CUDA translation units of libnbody.
// Nothing here is part of the C ABI (include/nbody.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "work_lists.h"

namespace nbody {

// One unit of all-pairs work: i-bodies [i_begin, i_end) of one system against
// its j-bodies [j_begin, j_end), partial sums written to slice `slice` of the
// system's n_slices. Indices are global body indices (rows of the caller's
// arrays).
struct WorkItem {
  int32_t sys;
  int32_t i_begin, i_end;
  int32_t j_begin, j_end;
  int32_t slice;
  int32_t n_slices;
};

// Per-system staging of the mixed path. Positions are staged as (x - c) * scale
// and masses as m * mscale, with powers of two as scales for gravity (set from
// the largest coordinate and mass at the start of every call, k_centre): the
// float32 pair arithmetic then has the same range whatever the caller's units are
// and the scaling costs no rounding. Where all masses of a system are equal they
// are staged as 1 (uniform). Lennard-Jones: scale = 1 / sigma, masses unused.
struct __align__(16) SysParam {
  double c[3];
  double scale, mscale, inv_mscale;
  float eps2, r2c;   // staged softening^2 and near-pair radius^2 (0: no refinement)
  uint32_t uniform;  // mixed: 1 if all masses are equal (staged as 1). FP64: the number of the last call that
                     // met unequal masses (checked when a call first stages; PostLaunch::epoch)
  uint32_t pad;
};

constexpr int kEnergyVals = 8;      // K, U, Px, Py, Pz, Lx, Ly, Lz per chunk
constexpr int kAdjVals = 8;         // VJP partial values per body per slice

// Force partial of one body and slice on the mixed path: the four compensated
// float32 sums (hi, lo) of the force kernels (sum m d / s^3 per axis and
// sum m / s), stored as they are: (hx, lx, hy, ly), (hz, lz, hp, lp). The
// O(N) kernel adds the slices as float32 pairs (TwoSum) and converts the total
// once, instead of converting each slice and adding on the FP64 pipe.
struct __align__(32) fpair4 {
  float4 xy;
  float4 zp;
};

// Knuth's TwoSum: hi + lo absorbs t, with the rounding error of hi + t carried
// into lo (Knuth, TAOCP vol. 2, 4.2.2). Six float32 additions, no branches.
__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float t) {
  const float s = hi + t;
  const float bp = s - hi;
  const float err = (hi - (s - bp)) + (t - bp);
  hi = s;
  lo += err;
}

// Programmatic dependent launch (sm_90 and later) between the kernels of a
// step: a kernel launched with launch_pdl may be scheduled while the kernel
// before it on the stream is still finishing; pdl_wait(), its first
// statement, waits (in hardware) until that grid has completed and its memory
// is visible, so data dependences are exactly those of plain stream order and
// only the launch latency overlaps. pdl_trigger() lets the next such kernel be
// scheduled once every CTA of this one has passed it (or exited). The all-pairs
// kernels call it when they run out of items. The O(N) kernels do not: their CTAs
// fill part of the SMs, and the persistent all-pairs grid placed around them is
// uneven for its whole run (FP64, 1024 bodies, 10 steps: 428 us with a trigger at
// the start of k_post, 371 us without; FP64 gradients at 2048 bodies 7.05 and
// 6.49 ms). Both are no-ops for a kernel launched without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_smem(void (*kern)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                                   Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(KArgs...), unsigned grid, unsigned block, cudaStream_t st, Args... args) {
  return launch_pdl_smem(kern, grid, block, 0, st, args...);
}

// Device status word bits (latched, read by nbody_sync).
constexpr unsigned kFlagNonFinite = 1u;
constexpr unsigned kFlagTimeout = 2u;
constexpr unsigned kFlagIndex = 4u;  // NBODY_DEBUG builds: an index check failed, the access was skipped

// Index checks of NBODY_DEBUG builds: nb_debug_ok(cond, status) is true when
// cond holds; otherwise it latches kFlagIndex in *status and returns false, and
// the caller skips the access. Release builds compile it to `true`.
#ifdef NBODY_DEBUG
__device__ __forceinline__ bool nb_debug_ok(const bool cond, unsigned* status) {
  if (!cond && status) atomicOr(status, kFlagIndex);
  return cond;
}
#else
__device__ __forceinline__ constexpr bool nb_debug_ok(const bool, unsigned*) { return true; }
#endif

// Host-side argument check (capi.cu): false when the driver reports that the
// device allocation holding p ends before p + bytes (cuMemGetAddressRange);
// *avail then holds the bytes left from p. True when the driver does not
// expose the query or does not know p.
bool allocation_holds(const void* p, size_t bytes, size_t* avail);

// ---------------------------------------------------------------------------
// all-pairs kernels (force_kernels.cu, adjoint_kernels.cu)

struct PairLaunch {
  const void* stage_x;   // float4 (x-c, m) [mixed] or double4_32a (x, m) [fp64], [N]
  const void* stage_w;   // VJP only: float4 / double4_32a (w, 0), [N]
  const WorkItem* items;
  int32_t n_items;
  unsigned* counter;     // [2]: next item, CTAs done (zero between launches)
  double* part;          // [slices][N] x (force: 1, VJP: 2, or 3 with params) of fpair4 (mixed) or double4_32a (FP64)
  int64_t n_total;
  double eps2;           // FP64 softening^2 (mixed: sys)
  const SysParam* sys;   // mixed: staged softening and near-pair radius of each system
  const float4* stage_lo;  // mixed: float32 remainders (x - c) - hi [N], near-pair refinement
  int variant;           // mixed kernels: 0 scalar float32, 1 packed float32x2
  int law;               // 0 softened gravity, 1 Lennard-Jones
  double sigma2;         // Lennard-Jones sigma^2
  int block, ipt, jtile; // tiling
  int n_ctas;            // persistent grid size
  int params;            // VJP: also the sums for the G and eps gradients (third double4)
  int phi;               // force (mixed packed): accumulate the potential (0: skip it, partial .w = 0)
  int32_t part_slices;   // slices the partial buffer holds (index checks of NBODY_DEBUG builds)
  int32_t block_bodies;  // debug checks: i-bodies a work item may hold (block x ipt)
  unsigned* status;      // device status word (index checks of NBODY_DEBUG builds)
};

// Launch of a symmetric pass (sym_kernels.cu, sym_vjp.cu).
struct SymLaunch {
  const void* stage_x;     // as in PairLaunch
  const void* stage_w;
  const float4* stage_lo;
  const SymItem* items;
  int32_t n_items;
  unsigned* counter;
  double* part;            // fpair4 (mixed) or double4_32a (FP64)
  int64_t part_rows;       // bodies' entries the partial buffer holds (index checks of NBODY_DEBUG builds)
  int64_t n_total;
  const SysParam* sys;
  double eps2, sigma2;     // FP64 path
  int law, block, ipt, n_ctas;
  int split;               // FP64 force: warps that share a block's work (1, 2, 4; where compiled)
  int phi;                 // potential: 0 none, 1 of every body, 2 for an energy record (sym::kPhi*)
  uint32_t epoch;          // FP64: number of the call (SysParam::uniform)
  int params;              // VJP: also the sums for the G and eps gradients
  unsigned* status;
};

#ifdef NBODY_DEBUG
// NBODY_DEBUG check of a work item against the buffers it indexes: its body
// ranges inside the rows, its i-range inside one CTA's tile, its slice inside
// the partial-sum buffer. The kernel skips an item that fails.
__device__ __forceinline__ bool item_ok(const WorkItem& w, const PairLaunch& L) {
  return nb_debug_ok(w.i_begin >= 0 && w.i_begin < w.i_end && w.i_end <= L.n_total && w.j_begin >= 0 &&
                         w.j_begin < w.j_end && w.j_end <= L.n_total && w.i_end - w.i_begin <= L.block_bodies &&
                         w.slice >= 0 && w.slice < w.n_slices && w.n_slices <= L.part_slices,
                     L.status);
}

__device__ __forceinline__ bool sym_item_ok(const SymItem& w, const SymLaunch& L) {
  const bool rows = w.i_begin >= 0 && w.i_begin < w.i_end && w.i_end <= L.n_total && w.j_begin >= w.i_begin &&
                    w.j_begin < w.j_end && w.j_end <= L.n_total && w.slot_i >= 0 && w.slot_j >= 0 && w.stride > 0;
  return nb_debug_ok(rows && w.row0 + w.i_begin >= 0 &&
                         w.row0 + (int64_t)w.slot_i * w.stride + w.i_end <= L.part_rows &&
                         w.row0 + (int64_t)w.slot_j * w.stride + w.j_end <= L.part_rows,
                     L.status);
}

// NBODY_DEBUG check of a chunk of an O(N) kernel: rows, system index and (when
// part_rows > 0) its slots against the entries the partial-sum buffer holds. A
// chunk that fails is processed as an empty one.
__device__ __forceinline__ bool chunk_ok(const Chunk& c, const int64_t n_total, const int n_sys,
                                         const int64_t part_rows, unsigned* status) {
  return nb_debug_ok(c.begin >= 0 && c.begin < c.end && c.end <= n_total && c.end - c.begin <= kChunk && c.sys >= 0 &&
                         c.sys < n_sys &&
                         (part_rows <= 0 || (c.n_slices >= 1 && c.row0 + c.begin >= 0 &&
                                             c.row0 + (int64_t)(c.n_slices - 1) * c.stride + c.end <= part_rows)),
                     status);
}
#else
__device__ __forceinline__ constexpr bool item_ok(const WorkItem&, const PairLaunch&) { return true; }
__device__ __forceinline__ constexpr bool sym_item_ok(const SymItem&, const SymLaunch&) { return true; }
__device__ __forceinline__ constexpr bool chunk_ok(const Chunk&, int64_t, int, int64_t, unsigned*) { return true; }
#endif

// Returns cudaErrorInvalidConfiguration for an unsupported tiling.
cudaError_t launch_force(int precision, const PairLaunch& L, cudaStream_t st);
cudaError_t launch_vjp(int precision, const PairLaunch& L, cudaStream_t st);
// CTAs of the force kernel that fit on one SM for the tiling (0 if unsupported).
int force_ctas_per_sm(int precision, int variant, int block, int ipt, int jtile, int law);
int vjp_ctas_per_sm(int precision, int variant, int block, int ipt, int jtile);

// Symmetric force pass: threads per CTA (block) and i-bodies per lane (ipt) select the
// compiled kernel; cudaErrorInvalidConfiguration / 0 if there is none.
cudaError_t launch_sym_force(int precision, const SymLaunch& L, cudaStream_t st);
int sym_force_ctas_per_sm(int precision, int block, int ipt, int law);
constexpr int kSymTile = 256;   // j-bodies per shared-memory tile of the symmetric kernels, mixed
constexpr int kSymTile64 = 64;  // ... and FP64
cudaError_t launch_sym_vjp(int precision, const SymLaunch& L, cudaStream_t st);
int sym_vjp_ctas_per_sm(int precision, int block, int ipt);
constexpr int kSymVjpTile = 128;  // j-tile of the mixed symmetric VJP (FP64: kSymTile64)

// ---------------------------------------------------------------------------
// O(N) kernels (post_kernels.cu)

enum PostMode : unsigned {
  kCombine = 1u,   // a, phi <- G * sum over slices of the partials
  kKickEnd = 2u,   // v += dt/2 a           (closing half-kick of a step)
  kEnergy = 4u,    // per-chunk partial energies / momenta at (x, v)
  kDrift = 8u,     // v += dt/2 a; x += dt v (opening half-kick + drift of the next step)
  kStage = 16u,    // staging tile entry from x (after the drift, if any)
  kMasses = 64u,   // FP64, with kStage: note unequal masses in SysParam::uniform
  kVirial = 32u,   // per-chunk partial K and Clausius virial W = sum m x.a (not with kEnergy)
};

struct PostLaunch {
  const Chunk* chunks;
  int32_t n_chunks;
  int chunk;               // bodies of a chunk at most (compiled: 16, 32, 64, 128)
  int few_slots;           // at most eight slots per body
  const double* part;      // [slices][N] of fpair4 (mixed) or double4_32a (FP64)
  int64_t n_total;
  double G, half_dt, dt;
  double* x;
  double* v;
  const double* m;
  double* a;
  double* phi;             // nullable
  double* x_copy;          // nullable: copy of x after the drift
  unsigned mode;
  int precision;
  int law;                 // 0 gravity: a = G S, phi = -G S_phi; 1 Lennard-Jones: a = 24 eps S / m, phi = 4 eps S_phi / m
  double lj_eps;
  double stage_scale;      // Lennard-Jones: staged positions are (x - c) * stage_scale (mixed: 1 / sigma)
  double box;              // > 0: reflecting walls of [0, box]^3 applied after the drift
  void* stage;             // float4 / double4_32a [N]
  void* stage_lo;          // mixed: float4 remainders of the staged coordinates [N] (nullable)
  SysParam* sys;           // [n_sys] staging origin and scales
  uint32_t epoch;          // FP64: number of the call
  const int64_t* off;      // [n_sys + 1] first body of each system
  double* epart;           // [n_chunks][kEnergyVals]
  unsigned* status;        // device status word
  double u_weight;         // kEnergy: U = u_weight sum m phi (1/2, or 1 if phi holds each pair once)
  double* eout;            // kEnergy: nullable [n_sys][9] record formed by the last CTA (null: partials only)
  const double* eprev;     // nullable: chunk partials [n_chunks][kEnergyVals] of the previous step's record,
  double* eprev_out;       //   finished into eprev_out [n_sys][9] by one extra CTA (blockIdx.x == n_chunks)
  double* vout;            // kVirial: [n_sys][3] record {K, W, -2K/W} formed by the last CTA
  const int32_t* sys_chunk;  // [n_sys + 1] chunk range of each system
  int n_sys;
  unsigned* done;          // last-CTA ticket (zero between launches)
  int64_t part_rows;       // entries the partial buffer holds (index checks of NBODY_DEBUG builds)
};
cudaError_t launch_post(const PostLaunch& P, cudaStream_t st);

// SysParam::uniform = 0 of every system (FP64, at the start of a captured call).
cudaError_t launch_clear_marks(SysParam* sys, int n_sys, cudaStream_t st);

// Staging parameters of every system (mixed path): the origin c is the
// mass-weighted mean position (plain mean if the mass is 0), and for gravity the
// scales are set from the extent, the softening and the largest mass. Per-chunk sums into cpart
// [n_chunks][kEnergyVals], then per system in a fixed order by the last CTA (of all, or of
// the system; tickets).
struct CentreLaunch {
  const Chunk* chunks;
  int32_t n_chunks;
  const int32_t* sys_chunk;
  const int64_t* off;
  int n_sys;
  const double* x;
  const double* m;
  double* cpart;
  SysParam* sys;
  int law;
  double eps, near_eps;  // gravity: softening length, near-pair radius in softening lengths
  unsigned* done;
  unsigned* sys_done;    // [n_sys] tickets of the systems (more than four; zero between launches)
  int64_t n_total;
  unsigned* status;
};
cudaError_t launch_centre(const CentreLaunch& C, cudaStream_t st);

struct AdjLaunch {
  const Chunk* chunks;
  int32_t n_chunks;
  int chunk;               // as in PostLaunch
  int few_slots;
  const double* part;      // 2 (3 with g_params) x fpair4 (mixed) or double4_32a (FP64) [slices][N]
  int64_t n_total;
  double G, coef, dt;      // lam_x += coef * gx ; g_m += coef * gm ; lam_v += dt lam_x
  const double* m;
  double* lam_x;
  double* lam_v;
  double* g_m;
  int drift_rev;           // apply lam_v += dt lam_x and restage w = lam_v
  const double* x_next;    // nullable: positions to stage for the next VJP
  int precision;
  void* stage_x;
  void* stage_w;
  void* stage_lo;          // mixed: float4 remainders of the staged positions (nullable)
  const SysParam* sys;
  unsigned* status;
  double* g_params;        // nullable [n_sys][2]: += coef (w.da/dG, w.da/deps), formed by the last CTA
  double eps;
  double* cpart;           // [n_chunks][kEnergyVals] chunk partials (g_params only)
  const int32_t* sys_chunk;
  int n_sys;
  unsigned* done;          // last-CTA ticket (zero between launches)
  int64_t part_rows;       // bodies' entries the partial buffer holds (index checks of NBODY_DEBUG builds)
};
cudaError_t launch_adj_update(const AdjLaunch& A, cudaStream_t st);

// dst[k][0 .. n[k]) = src[k][...] for k = 0..3 in one launch (entries with a
// null pointer or n = 0 are skipped); grid at most 8 CTAs per SM.
struct Copy4 {
  const double* src[4];
  double* dst[4];
  int64_t n[4];
};
cudaError_t launch_copy4(const Copy4& C, int n_sms, cudaStream_t st);

// stage w = lam (float4 / double4_32a) or positions x (as_position; with their
// float32 remainders into stage_lo when given) for a VJP without an update
cudaError_t launch_stage_vec(const Chunk* chunks, int n_chunks, int chunk, int precision, const double* vec,
                             const double* m, const SysParam* sys, void* stage, void* stage_lo, int as_position, int64_t n_total,
                             int n_sys, unsigned* status, cudaStream_t st);

}  // namespace nbody
