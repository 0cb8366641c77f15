// O(N) kernels around the all-pairs passes: staging, slice combination, the
// leapfrog kicks and drift (Verlet half-stepping, Sec. II-A), the fixed-order
// float64 reductions of energy and momenta (Sec. VI) and of the virial, the
// reverse-sweep update of the adjoint (with its G and eps sums), and the copy
// kernel of the host-buffer step. One CTA handles one chunk of one system, so chunk
// partials never mix systems and every sum has a fixed order.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "nbody_internal.h"
#include "post_common.cuh"

namespace nbody {
namespace {

// Threads that add a chunk's terms: its bodies', or a whole warp (others hold zeros)
template <int CB>
constexpr unsigned kSumThreads = CB < 32 ? 32 : CB;

// The parameters of a chunk's system for shared memory (used from global memory they would be read again after each
// store that might be to them, a round trip to L2 each time): a word per thread, loaded with the body's own values
// and stored ahead of the barrier that publishes it.
__device__ __forceinline__ uint32_t load_param_word(const SysParam* sys, const Chunk& c) {
  return threadIdx.x < sizeof(SysParam) / 4 && c.begin < c.end
             ? reinterpret_cast<const uint32_t*>(sys + c.sys)[threadIdx.x] : 0u;
}
__device__ __forceinline__ void store_param_word(SysParam& s, const uint32_t word) {
  if (threadIdx.x < sizeof(SysParam) / 4) reinterpret_cast<uint32_t*>(&s)[threadIdx.x] = word;
}

// One CTA per chunk, SG threads per body to add the slices and one to do
// the rest (a CTA of one thread per body when the mode combines nothing). Adding
// the slices is a chain of 32-byte loads from L2, and that latency and the FP64 pipe
// bound the kernel: on the 10 000-body Lennard-Jones gas (40 slices) a step took 89 us
// with one thread per body and 128-body chunks and 84 us with four and 64; with
// 32-body chunks, eight threads and the body's own loads ahead of the slices' it went
// from 70.5 to 69.1 us (on top of a faster force pass); 1024 bodies: 13.7 to 12.2 us, and 11.7 with the chunk
// read ahead of the wait.
// At 65 536 bodies eight threads cost 1% (1024-thread CTAs), so chunks of 128 keep four. After a one-sided
// pass of at most eight slots per body (ensembles of small systems) chunks are of 128 at any size, and above
// 32 768 bodies two threads share a body's slots: a step of 64 systems of 512 bodies 29.4 us in chunks of 64
// with eight threads, 27.2 so; of 64 systems of 2048 152.7 us with four threads, 148.7 with two.
template <int CB, int SG>
__global__ void __launch_bounds__(SG * CB) k_post(const PostLaunch P) {
  __shared__ union {
    SlotSums<CB, SG> f[4];
    double d[4][SG - 1][CB];
  } red;
  __shared__ SysParam sp;
  Chunk c{};  // (the chunk list is as old as the context: read while the kernel before finishes)
  if ((int)blockIdx.x < P.n_chunks) c = P.chunks[blockIdx.x];
  pdl_wait();  // the force kernel before it has finished writing the partials
  if ((int)blockIdx.x == P.n_chunks) {
    // the extra CTA: the previous step's energy record from its chunk partials
    systems_final<kEnergyVals, SG * CB>(P.sys_chunk, P.n_sys, P.eprev, P.n_chunks, P.status,
                                             [&](int sy, const double (&v)[kEnergyVals]) {
                                               emit_energy(P.eprev_out, sy, v);
                                             });
    return;
  }
  if (!chunk_ok(c, P.n_total, P.n_sys, (P.mode & kCombine) ? P.part_rows : 0, P.status))
    c.begin = c.end = 0;  // NBODY_DEBUG builds only: processed as an empty chunk
  double e[kEnergyVals];
#pragma unroll
  for (int k = 0; k < kEnergyVals; ++k) e[k] = 0.0;
  const unsigned mode = P.mode;
  const int b = (int)threadIdx.x % CB, g = (int)threadIdx.x / CB;
  const int i = c.begin + b;
  // (a chunk of 16 has half a warp without bodies in a pass that combines nothing)
  const bool live = i < c.end && g < SG;
  const uint32_t word = load_param_word(P.sys, c);
  BodyIn in;
  if (g == 0 && live) in = load_body(P, mode, i);
  const bool masses = P.precision == 0 && P.law == 0 && P.off;
  const double m0 = masses && (mode & (kCombine | kMasses)) && c.begin < c.end ? P.m[P.off[c.sys]] : 1.0;
  if (masses && (mode & kMasses) && g == 0 && live && __double_as_longlong(in.m) != __double_as_longlong(m0))
    P.sys[c.sys].uniform = P.epoch;

  if (!(mode & kCombine)) {
    store_param_word(sp, word);
    __syncthreads();
  }

  double sx = 0.0, sy = 0.0, sz = 0.0, sphi = 0.0;
  if ((mode & kCombine) && P.precision == 1) {
    const fpair4* fp = reinterpret_cast<const fpair4*>(P.part) + (c.row0 + i);
    float h[4] = {0.f, 0.f, 0.f, 0.f}, l[4] = {0.f, 0.f, 0.f, 0.f};
    if (live) {
#pragma unroll 8
      for (int s = g; s < c.n_slices; s += SG) add_slot(fp[(int64_t)s * c.stride], h, l);
    }
    store_param_word(sp, word);
    add_groups(red.f, g, b, h, l);
    if (g == 0) {
      sx = (double)h[0] + (double)l[0], sy = (double)h[1] + (double)l[1];
      sz = (double)h[2] + (double)l[2], sphi = (double)h[3] + (double)l[3];
    }
  } else if (mode & kCombine) {
    const double4_32a* part = reinterpret_cast<const double4_32a*>(P.part) + (c.row0 + i);
    double s4[4] = {0.0, 0.0, 0.0, 0.0};
    if (live) {
#pragma unroll 8
      for (int s = g; s < c.n_slices; s += SG) {
        const double4_32a q = part[(int64_t)s * c.stride];
        s4[0] += q.x, s4[1] += q.y, s4[2] += q.z, s4[3] += q.w;
      }
    }
    store_param_word(sp, word);
    add_groups(red.d, g, b, s4);
    // FP64 gravity: the mass that a system's bodies share is left out of the sums
    const double m_all = masses && sp.uniform != P.epoch ? m0 : 1.0;
    sx = m_all * s4[0], sy = m_all * s4[1], sz = m_all * s4[2], sphi = m_all * s4[3];
  }
  if (g == 0 && live && post_body(P, mode, i, sp, in, sx, sy, sz, sphi, e)) atomicOr(P.status, kFlagNonFinite);
  if (mode & kVirial) {
    double kw[2] = {e[0], e[1]};
    if (threadIdx.x < kSumThreads<CB>) block_sum<2, kSumThreads<CB>, true>(kw);
    if (threadIdx.x == 0) P.epart[(int64_t)blockIdx.x * kEnergyVals + 0] = kw[0],
                          P.epart[(int64_t)blockIdx.x * kEnergyVals + 1] = kw[1];
    if (last_of(P.done, (unsigned)P.n_chunks)) {
      __threadfence();
      systems_final<2, SG * CB>(P.sys_chunk, P.n_sys, P.epart, P.n_chunks, P.status,
                                     [&](int sy, const double (&v)[2]) {
                                       double* o = P.vout + 3 * (int64_t)sy;
                                       o[0] = v[0];
                                       o[1] = v[1];
                                       o[2] = v[1] != 0.0 ? -2.0 * v[0] / v[1] : 0.0;
                                     });
    }
    return;
  }
  if (mode & kEnergy) {
    if (threadIdx.x < kSumThreads<CB>) block_sum<kEnergyVals, kSumThreads<CB>, true>(e);
    if (threadIdx.x == 0) {
#pragma unroll
      for (int k = 0; k < kEnergyVals; ++k) P.epart[(int64_t)blockIdx.x * kEnergyVals + k] = e[k];
    }
    // the last chunk CTA to finish forms the per-system records (no separate launch); with
    // eout null the partials wait for the next step's k_post
    if (P.eout && last_of(P.done, (unsigned)P.n_chunks)) {
      __threadfence();
      systems_final<kEnergyVals, SG * CB>(P.sys_chunk, P.n_sys, P.epart, P.n_chunks, P.status,
                                               [&](int sy, const double (&v)[kEnergyVals]) {
                                                 emit_energy(P.eout, sy, v);
                                               });
    }
  }
}

__global__ void __launch_bounds__(kChunk) k_centre(const CentreLaunch C) {
  constexpr int CB = kChunk;
  constexpr int NW = CB / 32;
  __shared__ Extent ext[NW];
  const int lane = (int)threadIdx.x & 31, wid = (int)threadIdx.x >> 5;
  pdl_wait();
  Chunk c = C.chunks[blockIdx.x];
  if (!chunk_ok(c, C.n_total, C.n_sys, 0, C.status)) c.begin = c.end = 0;  // NBODY_DEBUG builds only
  double v[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  Extent q{0u, 0u, 1u};
  const int i = c.begin + (int)threadIdx.x;
  if (i < c.end) {
    const int64_t first = C.off[c.sys];
    centre_terms(C.x[3 * i + 0], C.x[3 * i + 1], C.x[3 * i + 2], C.m[i], C.x + 3 * first, C.m[first], v, q);
  }
  q.warp_join();
  if (lane == 0) ext[wid] = q;
  block_sum<7, CB>(v);  // its barriers also publish ext
  if (threadIdx.x == 0) {
    for (int w = 1; w < NW; ++w) q.join(ext[w]);
    double* o = C.cpart + (int64_t)blockIdx.x * kEnergyVals;
#pragma unroll
    for (int k = 0; k < 7; ++k) o[k] = v[k];
    o[7] = q.pack();
  }
  // The last CTA adds up to four systems' chunks; of more, each system's own last CTA does: one CTA for all of
  // them takes 3 us for every four systems (512 systems of 128 bodies: 466 us, 15 us this way; a step of a
  // twenty-step call 52 and 22.5 us).
  const bool own = C.n_sys > 4;
  const int sy0 = own ? c.sys : 0, sy1 = own ? c.sys + 1 : C.n_sys;
  if (own && c.begin >= c.end) return;  // NBODY_DEBUG builds only
  if (!last_of(own ? C.sys_done + c.sys : C.done,
               own ? (unsigned)(C.sys_chunk[sy1] - C.sys_chunk[sy0]) : gridDim.x))
    return;
  __threadfence();
  for (int sy = sy0; sy < sy1; ++sy) {
    Extent e{0u, 0u, 1u};
    for (int k = C.sys_chunk[sy] + (int)threadIdx.x; k < C.sys_chunk[sy + 1]; k += CB)
      e.join(Extent::unpack(__ldcg(C.cpart + (int64_t)k * kEnergyVals + 7)));
    e.warp_join();
    __syncthreads();
    if (lane == 0) ext[wid] = e;
    __syncthreads();
    for (int w = 0; w < NW; ++w) e.join(ext[w]);
    systems_final<7, CB>(C.sys_chunk + sy, 1, C.cpart, gridDim.x, C.status, [&](int, const double (&w)[7]) {
      const int64_t first = C.off[sy], n = C.off[sy + 1] - first;
      staging_params(C.sys[sy], w, e, n, C.x + 3 * first, n > 0 ? C.m[first] : 0.0, C.law == 0, C.eps, C.near_eps);
    });
  }
}

// (64 registers: 1024 threads per SM, so that the 512 CTAs of 16 384 bodies run at once)
template <int CB, int SG>
__global__ void __launch_bounds__(SG * CB, 1024 / (SG * CB)) k_adj_update(const AdjLaunch A) {
  __shared__ union {
    SlotSums<CB, SG> f[10];
    double d[10][SG - 1][CB];
  } red;
  __shared__ SysParam sp;  // (as in k_post)
  Chunk c = A.chunks[blockIdx.x];
  pdl_wait();  // the VJP kernel has finished writing the partials
  if (!chunk_ok(c, A.n_total, A.n_sys, A.part_rows, A.status)) c.begin = c.end = 0;  // NBODY_DEBUG builds only
  const uint32_t word = load_param_word(A.sys, c);
  const int kw = A.g_params ? 3 : 2;  // partials (fpair4 / double4_32a) per body and slice
  double pv[2] = {0.0, 0.0};          // this thread's w.da/dG and sum m (d.w) / s^5
  const int b = (int)threadIdx.x % CB, g = (int)threadIdx.x / CB;
  const int i = c.begin + b;
  const bool live = i < c.end;
  double S[10];  // A1 (3), A2, Gb (3), Gm, Pg, Pe of the body
  if (A.precision == 1) {
    // compensated float32 pairs (fpair4), added as pairs on the FP32 pipe
    const fpair4* fp = reinterpret_cast<const fpair4*>(A.part);
    float h[10], l[10];
#pragma unroll
    for (int q = 0; q < 10; ++q) h[q] = l[q] = 0.f;
    auto add = [&](const int q, const float hv, const float lv) {
      two_sum_acc(h[q], l[q], hv);
      l[q] += lv;
    };
    if (live) {
#pragma unroll 4
      for (int s = g; s < c.n_slices; s += SG) {
        const int64_t k = kw * (c.row0 + (int64_t)s * c.stride + i);
        const fpair4 p = fp[k], q = fp[k + 1];
        add(0, p.xy.x, p.xy.y), add(1, p.xy.z, p.xy.w), add(2, p.zp.x, p.zp.y), add(3, p.zp.z, p.zp.w);
        add(4, q.xy.x, q.xy.y), add(5, q.xy.z, q.xy.w), add(6, q.zp.x, q.zp.y), add(7, q.zp.z, q.zp.w);
        if (A.g_params) {
          const fpair4 r = fp[k + 2];
          add(8, r.xy.x, r.xy.y), add(9, r.xy.z, r.xy.w);
        }
      }
    }
    store_param_word(sp, word);
    add_groups(red.f, g, b, h, l);
#pragma unroll
    for (int q = 0; q < 10; ++q) S[q] = g == 0 ? (double)h[q] + (double)l[q] : 0.0;
  } else {
    const double4_32a* part = reinterpret_cast<const double4_32a*>(A.part);
#pragma unroll
    for (int q = 0; q < 10; ++q) S[q] = 0.0;
    if (live) {
#pragma unroll 4
      for (int s = g; s < c.n_slices; s += SG) {
        const int64_t k = kw * (c.row0 + (int64_t)s * c.stride + i);
        const double4_32a p = part[k], q = part[k + 1];
        S[0] += p.x, S[1] += p.y, S[2] += p.z, S[3] += p.w;
        S[4] += q.x, S[5] += q.y, S[6] += q.z, S[7] += q.w;
        if (A.g_params) {
          const double4_32a r = part[k + 2];
          S[8] += r.x, S[9] += r.y;
        }
      }
    }
    store_param_word(sp, word);
    add_groups(red.d, g, b, S);
  }
  if (g == 0 && live) {
    // the staged sums carry powers of the staging scales, and all but A1 and Gm a staged mass
    const double q = sp.scale, q2 = q * q, q2m = q2 * sp.inv_mscale, K = A.G * (q2m * q);
    if (A.g_params) pv[0] = q2m * S[8], pv[1] = q2 * q2m * S[9];
    const double mi = A.m[i], ms = mi * sp.mscale, gm = q2 * S[7];
    double w0 = A.lam_v[3 * i + 0], w1 = A.lam_v[3 * i + 1], w2 = A.lam_v[3 * i + 2];
    const double gx0 = K * (ms * S[0] - S[3] * w0 - 3.0 * S[4]);
    const double gx1 = K * (ms * S[1] - S[3] * w1 - 3.0 * S[5]);
    const double gx2 = K * (ms * S[2] - S[3] * w2 - 3.0 * S[6]);
    const double gmi = -A.G * gm;
    if (!(isfinite(gx0) && isfinite(gx1) && isfinite(gx2) && isfinite(gmi))) atomicOr(A.status, kFlagNonFinite);
    const double l0 = A.lam_x[3 * i + 0] + A.coef * gx0;
    const double l1 = A.lam_x[3 * i + 1] + A.coef * gx1;
    const double l2 = A.lam_x[3 * i + 2] + A.coef * gx2;
    A.lam_x[3 * i + 0] = l0, A.lam_x[3 * i + 1] = l1, A.lam_x[3 * i + 2] = l2;
    A.g_m[i] += A.coef * gmi;
    if (A.drift_rev) {
      w0 += A.dt * l0, w1 += A.dt * l1, w2 += A.dt * l2;
      A.lam_v[3 * i + 0] = w0, A.lam_v[3 * i + 1] = w1, A.lam_v[3 * i + 2] = w2;
      if (A.precision == 1)
        static_cast<float4*>(A.stage_w)[i] = make_float4((float)w0, (float)w1, (float)w2, 0.f);
      else
        static_cast<double4_32a*>(A.stage_w)[i] = make_double4_32a(w0, w1, w2, 0.0);
    }
    if (A.x_next)
      stage_store(A.precision, A.stage_x, i, A.x_next[3 * i + 0], A.x_next[3 * i + 1], A.x_next[3 * i + 2], mi,
                  sp, A.stage_lo);
  }
  if (!A.g_params) return;
  // dL/dG += coef sum_k w_k . da_k/dG; dL/deps += coef (-3 G eps) sum_k sum_j m_j (d.w_k) / s^5,
  // per system in a fixed order (chunk partials, then the last CTA)
  if (threadIdx.x < kSumThreads<CB>) block_sum<2, kSumThreads<CB>, true>(pv);
  if (threadIdx.x == 0) A.cpart[(int64_t)blockIdx.x * kEnergyVals + 0] = pv[0],
                        A.cpart[(int64_t)blockIdx.x * kEnergyVals + 1] = pv[1];
  if (!last_of(A.done, gridDim.x)) return;
  __threadfence();
  systems_final<2, SG * CB>(A.sys_chunk, A.n_sys, A.cpart, gridDim.x, A.status, [&](int sy, const double (&v)[2]) {
    const double dG = A.coef * v[0], de = A.coef * (-3.0 * A.G * A.eps) * v[1];
    if (!(isfinite(dG) && isfinite(de))) atomicOr(A.status, kFlagNonFinite);
    A.g_params[2 * sy + 0] += dG;
    A.g_params[2 * sy + 1] += de;
  });
}

template <int CB>
__global__ void __launch_bounds__(kSumThreads<CB>) k_stage_vec(const Chunk* chunks, int precision, const double* vec,
                                                  const double* m, const SysParam* sys, void* stage,
                                                            void* stage_lo, int as_position, const int64_t n_total,
                                                            const int n_sys, unsigned* status) {
  pdl_wait();
  Chunk c = chunks[blockIdx.x];
  if (!chunk_ok(c, n_total, n_sys, 0, status)) c.begin = c.end = 0;  // NBODY_DEBUG builds only
  const SysParam& sp = sys[c.sys];
  for (int i = c.begin + (int)threadIdx.x; i < c.end; i += (int)kSumThreads<CB>) {
    const double v0 = vec[3 * i + 0], v1 = vec[3 * i + 1], v2 = vec[3 * i + 2];
    if (as_position) {
      stage_store(precision, stage, i, v0, v1, v2, m[i], sp, stage_lo);
    } else if (precision == 1) {
      static_cast<float4*>(stage)[i] = make_float4((float)v0, (float)v1, (float)v2, 0.f);
    } else {
      static_cast<double4_32a*>(stage)[i] = make_double4_32a(v0, v1, v2, 0.0);
    }
  }
}

__global__ void __launch_bounds__(128) k_clear_marks(SysParam* sys, const int n_sys) {
  pdl_wait();
  const int s = (int)(blockIdx.x * 128 + threadIdx.x);
  if (s < n_sys) sys[s].uniform = 0u;
}

// Up to four plain copies of float64 arrays in one launch (the host-buffer
// step's transfers through mapped pinned host memory).
__global__ void __launch_bounds__(256) k_copy4(const Copy4 C) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double* __restrict__ src = C.src[k];
    double* __restrict__ dst = C.dst[k];
    const int64_t n = (src && dst) ? C.n[k] : 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) dst[i] = src[i];
  }
}

}  // namespace

cudaError_t launch_copy4(const Copy4& C, int n_sms, cudaStream_t st) {
  int64_t most = 0;
  for (int k = 0; k < 4; ++k) most = std::max<int64_t>(most, C.src[k] && C.dst[k] ? C.n[k] : 0);
  if (most == 0) return cudaSuccess;
  const int64_t want = (most + 255) / 256;
  const int grid = (int)std::min<int64_t>(want, (int64_t)std::max(1, n_sms) * 8);
  k_copy4<<<grid, 256, 0, st>>>(C);
  return cudaGetLastError();
}

// f(bodies per chunk, slot groups of k_post, of k_adj_update), as integral constants (the latter has
// ten sums per body to pass through shared memory)
template <typename F>
static cudaError_t with_chunk(const int chunk, F f) {
  using std::integral_constant;
  switch (chunk) {
    case 16: return f(integral_constant<int, 16>(), integral_constant<int, 16>(), integral_constant<int, 16>());
    case 32: return f(integral_constant<int, 32>(), integral_constant<int, 8>(), integral_constant<int, 8>());
    case 64: return f(integral_constant<int, 64>(), integral_constant<int, 8>(), integral_constant<int, 8>());
    default: return f(integral_constant<int, kChunk>(), integral_constant<int, 4>(), integral_constant<int, 4>());
  }
}

// Few slots per body and chunks enough to fill the SMs: two threads a body, of four (or eight) the others would
// find no slot.
static bool two_groups(const int few_slots, const int chunk, const int64_t n_total) {
  return few_slots && chunk == kChunk && n_total > 256 * kChunk;
}

cudaError_t launch_post(const PostLaunch& P, cudaStream_t st) {
  if (P.n_chunks <= 0) return cudaSuccess;
  auto launch = [&](auto cb, auto sg, auto) {
    constexpr int CB = decltype(cb)::value, SG = decltype(sg)::value;
    // a pass that combines nothing needs one thread per body only
    return launch_pdl(k_post<CB, SG>, (unsigned)P.n_chunks + (P.eprev_out ? 1u : 0u),
                      (P.mode & kCombine) ? SG * CB : (int)kSumThreads<CB>, st, P);
  };
  if (two_groups(P.few_slots, P.chunk, P.n_total))
    return launch(std::integral_constant<int, kChunk>(), std::integral_constant<int, 2>(), 0);
  return with_chunk(P.chunk, launch);
}

// (a memset node in its place is no part of the chain of dependent launches: 4.6 us of a captured call)
cudaError_t launch_clear_marks(SysParam* sys, int n_sys, cudaStream_t st) {
  return launch_pdl(k_clear_marks, (unsigned)(n_sys + 127) / 128, 128, st, sys, n_sys);
}

cudaError_t launch_centre(const CentreLaunch& C, cudaStream_t st) {
  if (C.n_sys <= 0 || C.n_chunks <= 0) return cudaSuccess;
  return launch_pdl(k_centre, C.n_chunks, kChunk, st, C);
}

cudaError_t launch_adj_update(const AdjLaunch& A, cudaStream_t st) {
  if (A.n_chunks <= 0) return cudaSuccess;
  auto launch = [&](auto cb, auto, auto sg) {
    constexpr int CB = decltype(cb)::value, SG = decltype(sg)::value;
    return launch_pdl(k_adj_update<CB, SG>, A.n_chunks, SG * CB, st, A);
  };
  if (two_groups(A.few_slots, A.chunk, A.n_total))
    return launch(std::integral_constant<int, kChunk>(), 0, std::integral_constant<int, 2>());
  return with_chunk(A.chunk, launch);
}

cudaError_t launch_stage_vec(const Chunk* chunks, int n_chunks, int chunk, int precision, const double* vec,
                             const double* m, const SysParam* sys, void* stage, void* stage_lo, int as_position, int64_t n_total,
                             int n_sys, unsigned* status, cudaStream_t st) {
  if (n_chunks <= 0) return cudaSuccess;
  return with_chunk(chunk, [&](auto cb, auto, auto) {
    constexpr int CB = decltype(cb)::value;
    return launch_pdl(k_stage_vec<CB>, n_chunks, (int)kSumThreads<CB>, st, chunks, precision, vec, m, sys, stage,
                      stage_lo, as_position, n_total, n_sys, status);
  });
}

}  // namespace nbody
