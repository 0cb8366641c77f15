// Device helpers of the O(N) kernels around the all-pairs passes
// (post_kernels.cu): the per-body combine / kick / drift / staging / energy
// terms of one body, the fixed-order CTA and per-system float64 sums, and the
// last-arrival ticket.
#pragma once

#include <math.h>

#include "nbody_internal.h"

namespace nbody {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Deterministic CTA sum of NV values per thread; result valid in thread 0.
// The sum is transposed so that every thread adds: the CTA's NV x THREADS
// values go to shared memory, then a group of TPV lanes per value adds its
// row in a fixed interleaved order and a TPV-lane xor shuffle finishes it.
// For NV = 8 and 64 threads that is 11 float64 additions per thread instead
// of the 40 of a per-value warp butterfly (float64 adds are GB300's scarce
// resource in these kernels). FIRST: only the CTA's first THREADS threads take
// part (they meet at named barrier 1); otherwise THREADS is the whole CTA.
template <bool FIRST, int THREADS>
__device__ __forceinline__ void sum_barrier() {
  if (FIRST)
    asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
  else
    __syncthreads();
}

template <int NV, int THREADS, bool FIRST = false>
__device__ __forceinline__ void block_sum(double (&v)[NV]) {
  constexpr int NVP = NV <= 1 ? 1 : NV <= 2 ? 2 : NV <= 4 ? 4 : NV <= 8 ? 8 : 16;
  constexpr int TPV0 = THREADS / NVP;
  constexpr int TPV = TPV0 > 32 ? 32 : TPV0;  // lanes per value: one aligned group inside a warp
  constexpr int EPT = THREADS / TPV;          // entries each of those lanes adds
  static_assert(TPV >= 1 && THREADS % 32 == 0 && NV <= 16, "block_sum layout");
  __shared__ double red[NV][THREADS];
  __shared__ double res[NV];
  sum_barrier<FIRST, THREADS>();  // an earlier block_sum of the same shape may still be reading
#pragma unroll
  for (int k = 0; k < NV; ++k) red[k][threadIdx.x] = v[k];
  sum_barrier<FIRST, THREADS>();
  const int k = (int)threadIdx.x / TPV, p = (int)threadIdx.x % TPV;
  double s = 0.0;
  if (k < NV) {
#pragma unroll
    for (int e = 0; e < EPT; ++e) s += red[k][p + e * TPV];
  }
#pragma unroll
  for (int o = TPV / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (k < NV && p == 0) res[k] = s;
  sum_barrier<FIRST, THREADS>();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = res[q];
  }
}

// The slices of one body, added by SG threads (thread group g of the CTA
// takes slices g, g + SG, ...) and then over the groups in order, all of it
// for NC components per slice. Mixed: compensated float32 pairs, added as pairs on
// the FP32 pipe (TwoSum of the hi parts, the lo parts and rounding errors summed
// alongside). Valid in group 0; every thread of the CTA calls it.
template <int CB, int SG>
struct SlotSums {
  float h[SG - 1][CB];
  float l[SG - 1][CB];
};

template <int NC, int CB, int SG>
__device__ __forceinline__ void add_groups(SlotSums<CB, SG> (&red)[NC], const int g, const int b, float (&h)[NC],
                                           float (&l)[NC]) {
  if (g > 0) {
#pragma unroll
    for (int c = 0; c < NC; ++c) red[c].h[g - 1][b] = h[c], red[c].l[g - 1][b] = l[c];
  }
  __syncthreads();
  if (g == 0) {
#pragma unroll
    for (int k = 0; k < SG - 1; ++k)
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        two_sum_acc(h[c], l[c], red[c].h[k][b]);
        l[c] += red[c].l[k][b];
      }
  }
}

template <int NC, int CB, int SG1>
__device__ __forceinline__ void add_groups(double (&red)[NC][SG1][CB], const int g, const int b,
                                           double (&s)[NC]) {
  if (g > 0) {
#pragma unroll
    for (int c = 0; c < NC; ++c) red[c][g - 1][b] = s[c];
  }
  __syncthreads();
  if (g == 0) {
#pragma unroll
    for (int k = 0; k < SG1; ++k)
#pragma unroll
      for (int c = 0; c < NC; ++c) s[c] += red[c][k][b];
  }
}

// One slot of a body's force partials onto its sums.
__device__ __forceinline__ void add_slot(const fpair4 q, float (&h)[4], float (&l)[4]) {
  two_sum_acc(h[0], l[0], q.xy.x), l[0] += q.xy.y;
  two_sum_acc(h[1], l[1], q.xy.z), l[1] += q.xy.w;
  two_sum_acc(h[2], l[2], q.zp.x), l[2] += q.zp.y;
  two_sum_acc(h[3], l[3], q.zp.z), l[3] += q.zp.w;
}

// Largest distance along an axis from the system's first body and largest mass of a chunk by their
// float64 high words (sign bit off: the words order as the magnitudes) and whether its masses all equal its
// system's first, as one 64-bit value that is carried beside the chunk's sums.
struct Extent {
  unsigned x, m, uniform;
  __device__ __forceinline__ void join(const Extent& o) {
    x = max(x, o.x), m = max(m, o.m), uniform &= o.uniform;
  }
  __device__ __forceinline__ void warp_join() {
    x = __reduce_max_sync(0xffffffffu, x);
    m = __reduce_max_sync(0xffffffffu, m);
    uniform = __reduce_and_sync(0xffffffffu, uniform);
  }
  __device__ __forceinline__ double pack() const {
    return __hiloint2double((int)x, (int)(m << 1 | uniform));
  }
  __device__ __forceinline__ static Extent unpack(const double d) {
    const unsigned l = (unsigned)__double2loint(d);
    return Extent{(unsigned)__double2hiint(d), l >> 1, l & 1u};
  }
};

__device__ __forceinline__ unsigned high_word(const double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// Binary exponent of the float64 with high word h, and whether it is one to scale by (not 0, tiny, infinite or NaN).
__device__ __forceinline__ int exponent_of(const unsigned h) { return (int)(h >> 20) - 1023; }
__device__ __forceinline__ bool scalable(const int e) { return e >= -900 && e <= 900; }

// Staged lengths of gravity. The farthest body of a system lies below 2^12 from its origin: the powers of
// distances from there down to 2^-25, s^-5 (the force gradient) included, stay in float32's range. Where that
// would stage the softening below 2^-24, it is lifted to 2^-24 as far as the farthest body stays below 2^22, and
// beyond that as far as the lengths are not staged longer than they are: far from the rest, an escaper loses the
// last bits of its gradient's powers before near pairs' turn infinite. Without softening the nearest distance is
// not known, and a system is not staged smaller than it is up to that size.
constexpr int kFarExp = 10, kFarthestExp = 20, kNearExp = -24;
__device__ __forceinline__ int staging_exponent(const int far, const int eps) {  // (binary exponents)
  const int room = kFarthestExp - far, near = scalable(eps) ? kNearExp - eps : min(0, room);
  return max(kFarExp - far, max(min(near, room), min(near, 0)));
}

// One body's terms of the staging origin's sums (sum m x, sum m, sum x) and its extent about the
// system's first body (position f, mass m0).
__device__ __forceinline__ void centre_terms(const double x0, const double x1, const double x2, const double mi,
                                             const double* f, const double m0, double (&v)[7], Extent& q) {
  v[0] += mi * x0, v[1] += mi * x1, v[2] += mi * x2, v[3] += mi;
  v[4] += x0, v[5] += x1, v[6] += x2;
  q.join(Extent{max(max(high_word(x0 - f[0]), high_word(x1 - f[1])), high_word(x2 - f[2])), high_word(mi),
                __double_as_longlong(mi) == __double_as_longlong(m0) ? 1u : 0u});
}

// Staging parameters of a system of n bodies from those sums: the origin, and for gravity the
// scales (f, m0: its first body).
__device__ __forceinline__ void staging_params(SysParam& o, const double (&w)[7], const Extent& e, const int64_t n,
                                               const double* f, const double m0, const bool gravity, const double eps,
                                               const double near_eps) {
  double c0 = 0.0, c1 = 0.0, c2 = 0.0;
  if (w[3] > 0.0 && isfinite(w[3])) {
    c0 = w[0] / w[3], c1 = w[1] / w[3], c2 = w[2] / w[3];
  } else if (n > 0) {
    c0 = w[4] / (double)n, c1 = w[5] / (double)n, c2 = w[6] / (double)n;
  }
  if (!(isfinite(c0) && isfinite(c1) && isfinite(c2))) c0 = c1 = c2 = 0.0;
  o.c[0] = c0, o.c[1] = c1, o.c[2] = c2;
  if (!gravity || n <= 0) return;
  // no body is farther from the origin than twice the larger of these (the origin's own distance from the
  // first body counts where negative masses put it outside); the softening counts as an extent, so that
  // its staged square stays finite
  const unsigned off = max(max(high_word(c0 - f[0]), high_word(c1 - f[1])), high_word(c2 - f[2]));
  const int far = exponent_of(max(max(e.x, off), high_word(eps)));
  const double s = scalable(far) ? ldexp(1.0, staging_exponent(far, exponent_of(high_word(eps)))) : 1.0;
  const double e2 = eps * s, rc = near_eps * e2;
  const unsigned h0 = high_word(m0);
  const bool uniform = e.uniform && m0 > 0.0 && h0 >= (123u << 20) && h0 <= (1923u << 20);
  const int em = exponent_of(e.m);
  const double ms = scalable(em) ? ldexp(1.0, -em) : 1.0;
  o.scale = s;
  o.mscale = uniform ? 1.0 / m0 : ms;
  o.inv_mscale = uniform ? m0 : 1.0 / ms;
  o.eps2 = (float)(e2 * e2), o.r2c = (float)(rc * rc);
  o.uniform = uniform ? 1u : 0u;
}

// Reflecting walls of [0, box] ("boundary checking"): a coordinate that left
// the box is mirrored back across the wall and its velocity component flips;
// repeated (bounded) for steps that cross the box more than once.
__device__ __forceinline__ void reflect(double& x, double& v, const double box) {
  for (int k = 0; k < 64; ++k) {
    if (x < 0.0) {
      x = -x, v = -v;
    } else if (x > box) {
      x = 2.0 * box - x, v = -v;
    } else {
      return;
    }
  }
}

// Staging entry of body i. Mixed: float4 ((x - c) * scale, m * mscale) rounded to
// float32 and, when lo is given, the float32 remainders of the scaled coordinates
// used by the near-pair refinement (SysParam). FP64: double4 (x, m).
__device__ __forceinline__ void stage_store(int precision, void* stage, int i, double x, double y, double z,
                                            double m, const SysParam& sp, void* lo = nullptr) {
  if (precision == 1) {
    const double X = (x - sp.c[0]) * sp.scale, Y = (y - sp.c[1]) * sp.scale, Z = (z - sp.c[2]) * sp.scale;
    const float hx = (float)X, hy = (float)Y, hz = (float)Z;
    static_cast<float4*>(stage)[i] = make_float4(hx, hy, hz, sp.uniform ? 1.f : (float)(m * sp.mscale));
    if (lo)
      static_cast<float4*>(lo)[i] =
          make_float4((float)(X - (double)hx), (float)(Y - (double)hy), (float)(Z - (double)hz), 0.f);
  } else {
    static_cast<double4_32a*>(stage)[i] = make_double4_32a(x, y, z, m);
  }
}

// Final per-system sums of partials [n_parts][kEnergyVals] (one per chunk of
// an O(N) kernel), in a fixed order whichever CTA runs it. The partials were
// written by other CTAs of the same launch, so they are read from L2
// (ld.global.cg). Up to four systems: the whole CTA adds each system's
// partials (thread t takes partials t, t + THREADS, ...), then block_sum; more
// systems: one warp per system, lanes striding over its range, then a warp
// butterfly. Every thread of the CTA must call it.
template <int NV, int THREADS, typename Emit>
__device__ __forceinline__ void systems_final(const int32_t* sys_part, const int n_sys, const double* part,
                                              const int n_parts, unsigned* status, Emit emit) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (n_sys <= 4) {
    for (int sy = 0; sy < n_sys; ++sy) {
      double v[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) v[k] = 0.0;
      // NBODY_DEBUG builds: the system's range lies inside the partials
      const bool ok = nb_debug_ok(sys_part[sy] >= 0 && sys_part[sy] <= sys_part[sy + 1] &&
                                      sys_part[sy + 1] <= n_parts,
                                  threadIdx.x == 0 ? status : nullptr);
#pragma unroll 4
      for (int c = sys_part[sy] + (int)threadIdx.x; ok && c < sys_part[sy + 1]; c += THREADS) {
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] += __ldcg(part + (int64_t)c * kEnergyVals + k);
      }
      block_sum<NV, THREADS>(v);
      if (threadIdx.x == 0) emit(sy, v);
    }
    return;
  }
  for (int sy = wid; sy < n_sys; sy += THREADS / 32) {
    double v[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = 0.0;
    const bool ok = nb_debug_ok(sys_part[sy] >= 0 && sys_part[sy] <= sys_part[sy + 1] && sys_part[sy + 1] <= n_parts,
                                lane == 0 ? status : nullptr);
    for (int c = sys_part[sy] + lane; ok && c < sys_part[sy + 1]; c += 32) {
#pragma unroll
      for (int k = 0; k < NV; ++k) v[k] += __ldcg(part + (int64_t)c * kEnergyVals + k);
    }
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = warp_sum(v[k]);
    if (lane == 0) emit(sy, v);
  }
}

// True in every thread of the CTA that arrives last of `expected` arrivals at
// the ticket `done` (its results were published with a fence before the
// ticket); that CTA resets the ticket for the next launch. No CTA waits.
__device__ __forceinline__ bool last_of(unsigned* done, const unsigned expected) {
  __shared__ bool s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(done, 1u) == expected - 1u;
    if (s_last) *done = 0u;
  }
  __syncthreads();
  return s_last;
}

__device__ __forceinline__ void emit_energy(double* out, const int sy, const double (&v)[kEnergyVals]) {
  double* o = out + 9 * (int64_t)sy;
  o[0] = v[0] + v[1];
  o[1] = v[0];
  o[2] = v[1];
#pragma unroll
  for (int k = 2; k < kEnergyVals; ++k) o[k + 1] = v[k];
}

// What post_body reads of body i, loaded before the slices are added, so that these
// loads and the slices' are in flight together (x, v, m and a are distinct arrays).
struct BodyIn {
  double x0 = 0.0, x1 = 0.0, x2 = 0.0, v0 = 0.0, v1 = 0.0, v2 = 0.0, m = 0.0, a0 = 0.0, a1 = 0.0, a2 = 0.0;
};
__device__ __forceinline__ BodyIn load_body(const PostLaunch& P, const unsigned mode, const int i) {
  BodyIn b;
  const bool need_x = mode & (kKickEnd | kEnergy | kDrift | kStage | kVirial);
  const bool need_v = mode & (kKickEnd | kEnergy | kDrift | kVirial);
  if (need_x) b.x0 = P.x[3 * i + 0], b.x1 = P.x[3 * i + 1], b.x2 = P.x[3 * i + 2];
  if (need_v) b.v0 = P.v[3 * i + 0], b.v1 = P.v[3 * i + 1], b.v2 = P.v[3 * i + 2];
  if (need_x || (mode & kCombine && P.law != 0)) b.m = P.m[i];
  if (!(mode & kCombine) && (mode & (kKickEnd | kDrift)))
    b.a0 = P.a[3 * i + 0], b.a1 = P.a[3 * i + 1], b.a2 = P.a[3 * i + 2];
  return b;
}

// The O(N) work of one body i in the PostMode bits of `mode`: with kCombine its
// summed partials (sx, sy, sz, sp) become a = G S (or the Lennard-Jones
// scaling) and phi; then the closing half-kick, the energy or virial terms
// (accumulated into e), the opening half-kick and drift of the next step (with
// the walls), and the staging entry of the new position. s holds the system's
// staging origin and scales. Returns true if a combined value is not finite.
__device__ __forceinline__ bool post_body(const PostLaunch& P, const unsigned mode, const int i, const SysParam& s,
                                          const BodyIn& in, const double sx, const double sy, const double sz,
                                          const double sp, double (&e)[kEnergyVals]) {
  bool bad = false;
  double x0 = in.x0, x1 = in.x1, x2 = in.x2, v0 = in.v0, v1 = in.v1, v2 = in.v2;
  const double m = in.m;
  double ax = 0.0, ay = 0.0, az = 0.0, ph = 0.0;
  if (mode & kCombine) {
    if (P.law == 0) {  // softened gravity; the staged sums carry mscale / scale^2 (mscale / scale)
      const double gp = P.G * (s.scale * s.inv_mscale), ga = gp * s.scale;
      ax = ga * sx, ay = ga * sy, az = ga * sz, ph = -gp * sp;
    } else {  // Lennard-Jones: per unit mass of body i (sums over staged coordinates in units of sigma
              // carry one factor sigma: S = sigma * sum (u^3 - 2 u^6) d / r^2, hence the stage_scale)
      const double im = 1.0 / m, ca = 24.0 * P.lj_eps * P.stage_scale * im, cp = 4.0 * P.lj_eps * im;
      ax = ca * sx, ay = ca * sy, az = ca * sz, ph = cp * sp;
    }
    P.a[3 * i + 0] = ax, P.a[3 * i + 1] = ay, P.a[3 * i + 2] = az;
    if (P.phi) P.phi[i] = ph;
    bad = !(isfinite(ax) && isfinite(ay) && isfinite(az) && isfinite(ph));
  } else if (mode & (kKickEnd | kDrift)) {
    ax = in.a0, ay = in.a1, az = in.a2;
  }
  if (mode & kVirial) {
    e[0] += 0.5 * m * (v0 * v0 + v1 * v1 + v2 * v2);
    e[1] += m * (x0 * ax + x1 * ay + x2 * az);
  }
  if (!(mode & (kKickEnd | kEnergy | kDrift | kStage))) return bad;
  if (mode & (kKickEnd | kEnergy | kDrift)) {
    if (mode & kKickEnd) {
      v0 += P.half_dt * ax, v1 += P.half_dt * ay, v2 += P.half_dt * az;
    }
    if (mode & kEnergy) {
      e[0] += 0.5 * m * (v0 * v0 + v1 * v1 + v2 * v2);
      e[1] += P.u_weight * m * ph;
      e[2] += m * v0, e[3] += m * v1, e[4] += m * v2;
      e[5] += m * (x1 * v2 - x2 * v1);
      e[6] += m * (x2 * v0 - x0 * v2);
      e[7] += m * (x0 * v1 - x1 * v0);
    }
    if (mode & kDrift) {
      v0 += P.half_dt * ax, v1 += P.half_dt * ay, v2 += P.half_dt * az;
      x0 += P.dt * v0, x1 += P.dt * v1, x2 += P.dt * v2;
      if (P.box > 0.0) {
        reflect(x0, v0, P.box);
        reflect(x1, v1, P.box);
        reflect(x2, v2, P.box);
      }
      P.x[3 * i + 0] = x0, P.x[3 * i + 1] = x1, P.x[3 * i + 2] = x2;
      if (P.x_copy) P.x_copy[3 * i + 0] = x0, P.x_copy[3 * i + 1] = x1, P.x_copy[3 * i + 2] = x2;
    }
    if (mode & (kKickEnd | kDrift)) P.v[3 * i + 0] = v0, P.v[3 * i + 1] = v1, P.v[3 * i + 2] = v2;
  }
  if (mode & kStage) stage_store(P.precision, P.stage, i, x0, x1, x2, m, s, P.stage_lo);
  return bad;
}

}  // namespace nbody
