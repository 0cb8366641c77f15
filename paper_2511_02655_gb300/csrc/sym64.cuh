// All-pairs force pass of the FP64 path that evaluates every unordered pair once;
// work list, slots and the travelling j-sums are those of sym_common.cuh.
//
// Bound: GB300's FP64 pipe, two lanes per clock and SM against 128 of the FP32 and
// 64 of the integer pipe. Everything that is not a float64 operation is therefore
// free up to dozens of operations, and the pair is written for the fewest float64
// ones: 16 per unordered pair of softened gravity (8 per interaction; 3 more with
// both potentials, 2 fewer where all masses of a system are equal) where the one-sided
// kernel with the library's rsqrt takes about 20 per interaction. N = 12 002 with
// potentials and unequal masses: 4.67 ms with the one-sided kernel, 2.43 ms here (19
// operations a pair take 2.18 ms at the pipe's rate). The error against 64-bit sums is
// no larger (3.3e-16 and 1.6e-16 relative): s^-3 is good to 1.5 ulp, 0.25 ulp on average.
#pragma once

#include <type_traits>

#include "nbody_internal.h"
#include "pair_common.cuh"
#include "sym_common.cuh"

namespace nbody {
namespace sym64 {

// v * 2^-scale as a double, for an integer 0 < v < 2^53 (exact)
__device__ __forceinline__ double int_scaled(const uint64_t v, const int scale) {
  const int top = 63 - __clzll((long long)v);
  const uint64_t m = v << (52 - top);
  return __hiloint2double((int)((uint32_t)(m >> 32) + ((uint32_t)(1022 + top - scale) << 20)), (int)(uint32_t)m);
}

// float32 value of a double below 1 in magnitude (rounded; below 2^-126 it becomes 0), and back (exact; 0 becomes
// 2^-127), in integer operations
__device__ __forceinline__ float small_to_float(const double e) {
  const uint32_t h = (uint32_t)__double2hiint(e), l = (uint32_t)__double2loint(e);
  const uint32_t u = max(h & 0x7fffffffu, 0x38000000u) - 0x38000000u;
  return __uint_as_float((h & 0x80000000u) | (((u << 3) | (l >> 29)) + ((l >> 28) & 1u)));
}
__device__ __forceinline__ double float_to_double(const float t) {  // t >= 0
  const uint32_t b = __float_as_uint(t);
  return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

// s^2 = f 4^q with 1 <= f < 4. The integer steps below need a normal s^2 whose powers
// stay normal too: 2^-600 <= s^2 < 2^600; blocks that hold anything else (0, infinities,
// NaN) are done with the library's functions instead (block32's caller).
constexpr int kExpRange = 600;
__device__ __forceinline__ bool in_range(const double r2) {
  return (uint32_t)(__double2hiint(r2) - ((1023 - kExpRange) << 20)) < (uint32_t)(2 * kExpRange) << 20;
}

// Start values of the roots of s^2: y = M 2^-17 is the hardware's approximate reciprocal
// root of f rounded to 17 bits, so that y^2 (34 bits) and y^3 (51 bits) are exact
// doubles, formed as integers; e = 1 - f y^2 (one rounding of a difference of magnitude
// 2^-16). Newton's correction then is a polynomial in e whose terms from e^2 on
// need float32 only: (1 - e)^(-3/2) = 1 + 3/2 e + e^2 (15/8 + 35/16 e) + O(e^4).
struct Root {
  uint64_t M2, M3;
  int q;
  double e;
  float ef;
};
__device__ __forceinline__ Root root_of(const double r2) {
  Root t;
  const uint32_t h = (uint32_t)__double2hiint(r2), l = (uint32_t)__double2loint(r2);
  const int ex = (int)(h >> 20) - 1023, odd = ex & 1;
  t.q = (ex - odd) >> 1;
  const float y = rsq_approx(__uint_as_float((((h << 3) | (l >> 29)) & 0x7fffffu) + ((127u + (uint32_t)odd) << 23)));
  const uint32_t M = __float_as_uint(y + 64.f) - 0x42800000u;  // the spacing of floats at 64 is 2^-17
  t.M2 = (uint64_t)M * M;
  t.M3 = t.M2 * M;
  const double f = __hiloint2double((int)((h & 0xfffffu) | ((1023u + (uint32_t)odd) << 20)), (int)l);
  t.e = fma(-f, int_scaled(t.M2, 34), 1.0);
  t.ef = small_to_float(t.e);
  return t;
}
// s^-3 from the start values: one float64 operation. y^3 (1 + p), p = e^2 (15/8 + 35/16 e) >= 0 below
// 2^-30, is the double y^3 plus p times its 53-bit mantissa in units of the last place, an integer
// addition (a carry runs into the exponent, as it should); the linear term 3/2 y^3 is exact.
__device__ __forceinline__ double inv3_of(const Root& t) {
  const float p = (t.ef * t.ef) * fmaf(2.1875f, t.ef, 1.875f);
  const uint64_t m = t.M3 << (__clzll((long long)t.M3) - 11);
  const float fm = __uint_as_float(((127u + 52u) << 23) | ((uint32_t)(m >> 29) & 0x7fffffu));
  const long long y3 = __double_as_longlong(int_scaled(t.M3, 51 + 3 * t.q)) + __float2int_rn(p * fm);
  return fma(int_scaled(3u * t.M3, 52 + 3 * t.q), t.e, __longlong_as_double(y3));
}
// s^-2: two float64 operations
__device__ __forceinline__ double inv2_of(const Root& t) {
  const float p = (t.ef * t.ef) * (1.f + t.ef);
  const double c = t.e + float_to_double(p), y2 = int_scaled(t.M2, 34 + 2 * t.q);
  return fma(y2, c, y2);
}
// 1 / s^2 alone: y is the hardware's approximate reciprocal of f' in [1, 2), 24 bits, e = 1 - f' y
// of magnitude 2^-22 and 1 / f' = y (1 + e + e^2) + O(e^3): three float64 operations
__device__ __forceinline__ double rcp_f64(const double r2) {
  const uint32_t h = (uint32_t)__double2hiint(r2), l = (uint32_t)__double2loint(r2);
  const int ex = (int)(h >> 20) - 1023;
  const float y = rcp_approx(__uint_as_float((((h << 3) | (l >> 29)) & 0x7fffffu) + (127u << 23)));
  const double f = __hiloint2double((int)((h & 0xfffffu) | (1023u << 20)), (int)l);
  const double yd = float_to_double(y);
  const double e = fma(-f, yd, 1.0);
  const float ef = small_to_float(e);
  const double c = e + float_to_double(ef * ef);
  const double ys = __hiloint2double(__double2hiint(yd) - (ex << 20), __double2loint(yd));
  return fma(ys, c, ys);
}

// Pair weights: the force on the i-body is wj d, on the j-body -wi d; t is the potential term
// (times the other body's mass for gravity). FAST: s^2 is in range.
template <int LAW, bool FAST, int PHI, bool EQ>
__device__ __forceinline__ void weights(const double r2, const double s2, const double mj, const double mi, double& wj,
                                        double& wi, double& t) {
  if (LAW == 0) {
    if (FAST) {
      const double i3 = inv3_of(root_of(r2));
      wj = EQ ? i3 : mj * i3, wi = EQ ? i3 : mi * i3;
      if (PHI) t = i3 * r2;
    } else {
      const double inv = rsqrt(r2), i2 = inv * inv;
      wj = EQ ? inv * i2 : (mj * inv) * i2, wi = EQ ? wj : (mi * inv) * i2;
      if (PHI) t = inv;
    }
  } else {  // u = sigma^2 / r^2
    const double inv2 = FAST ? rcp_f64(r2) : 1.0 / r2;
    const double u = s2 * inv2, u3 = u * u * u, u6 = u3 * u3;
    wj = wi = fma(-2.0, u6, u3) * inv2;
    if (PHI) t = u6 - u3;
  }
}

constexpr int kTile = kSymTile64;  // j-bodies per shared-memory tile (blocks of 32, one per lane)

template <int W>
struct Smem {
  double q[4][kTile / 32][64];  // x, y, z, m of the tile's blocks; entries 32.. repeat 0..
  double jacc[W][4][kTile];     // each warp's sums for the tile's j-bodies
  int item;
};

// Pairs of a lane in flight together: a pair is a chain of about ten float64 and forty
// integer operations, and small systems have few warps per scheduler to hide it.
constexpr int kUnroll = 4;

// The 32 steps of one block, or the 32 / KS from k0 on of a warp that shares it with KS - 1 others. FAST:
// returns whether the lane met an s^2 out of range, in which case the sums are void and the block is to be
// repeated without FAST (there is no branch per pair, so that the pairs of several steps overlap).
template <int LAW, bool SYM, bool MASK, int PHI, bool EQ, bool FAST, int R, int KS>
__device__ __forceinline__ bool block32(const double (&q)[4][kTile / 32][64], const int b, const int k0, const int jg0,
                                        const int lane,
                                        const int ig0, const double (&xi)[R], const double (&yi)[R],
                                        const double (&zi)[R], const double (&mi)[R], const double eps2,
                                        const double s2, double (&ax)[R], double (&ay)[R], double (&az)[R],
                                        double (&pp)[R], double& jx, double& jy, double& jz, double& jp) {
  const int src = (lane + 1) & 31;
  bool out = false;
#pragma unroll(FAST ? kUnroll / R : 1)
  for (int k = 0; k < 32 / KS; ++k) {
    const int p = lane + k0 + k;
    const double xj = q[0][b][p], yj = q[1][b][p], zj = q[2][b][p], mj = q[3][b][p];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const double dx = xj - xi[r], dy = yj - yi[r], dz = zj - zi[r];
      const double r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2)));
      const bool self = MASK && jg0 + (p & 31) == ig0 + 32 * r;
      if (FAST) out |= !self && !in_range(r2);
      double wj, wi, t = 0.0;
      weights<LAW, FAST, PHI, EQ>(r2, s2, mj, mi[r], wj, wi, t);
      if (self) wj = 0.0, t = 0.0;
      ax[r] = fma(dx, wj, ax[r]);
      ay[r] = fma(dy, wj, ay[r]);
      az[r] = fma(dz, wj, az[r]);
      if (MASK && PHI == sym::kPhiEnergy) t *= 0.5;
      if (PHI) pp[r] = LAW == 0 && !EQ ? fma(mj, t, pp[r]) : pp[r] + t;
      if (SYM) {
        jx = fma(-dx, wi, jx);
        jy = fma(-dy, wi, jy);
        jz = fma(-dz, wi, jz);
        if (PHI == sym::kPhiBoth) jp = LAW == 0 && !EQ ? fma(mi[r], t, jp) : jp + t;
      }
    }
    if (SYM) {
      jx = __shfl_sync(0xffffffffu, jx, src);
      jy = __shfl_sync(0xffffffffu, jy, src);
      jz = __shfl_sync(0xffffffffu, jz, src);
      if (PHI == sym::kPhiBoth) jp = __shfl_sync(0xffffffffu, jp, src);
    }
  }
  return out;
}

// A block with FAST, repeated without it where any lane met an s^2 out of range.
template <int LAW, bool SYM, bool MASK, int PHI, bool EQ, int R, int KS>
__device__ __forceinline__ void block(const double (&q)[4][kTile / 32][64], const int b, const int k0, const int jg0,
                                      const int lane,
                                      const int ig0, const double (&xi)[R], const double (&yi)[R],
                                      const double (&zi)[R], const double (&mi)[R], const double eps2, const double s2,
                                      double (&ax)[R], double (&ay)[R], double (&az)[R], double (&pp)[R], double& jx,
                                      double& jy, double& jz, double& jp) {
  double bx[R], by[R], bz[R], bp[R];
#pragma unroll
  for (int r = 0; r < R; ++r) bx[r] = ax[r], by[r] = ay[r], bz[r] = az[r], bp[r] = pp[r];
  const bool out = block32<LAW, SYM, MASK, PHI, EQ, true, R, KS>(q, b, k0, jg0, lane, ig0, xi, yi, zi, mi, eps2, s2,
                                                                 bx, by, bz, bp, jx, jy, jz, jp);
  if (__any_sync(0xffffffffu, out)) {
    jx = jy = jz = jp = 0.0;
    block32<LAW, SYM, MASK, PHI, EQ, false, R, KS>(q, b, k0, jg0, lane, ig0, xi, yi, zi, mi, eps2, s2, ax, ay, az, pp,
                                                   jx, jy, jz, jp);
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r) ax[r] = bx[r], ay[r] = by[r], az[r] = bz[r], pp[r] = bp[r];
  }
}

// Work items, taken from `counter` until none is left.
// KS warps share the W warps' i-bodies and blocks, each a range of the rotation's steps (short lists,
// SymLaunch::split): the j-sums need nothing new, as the CTA's warps' sums are added anyway, the i-sums
// are added at the end of the i-tile.
template <int LAW, int W, int R, int PHI, int KS>
__device__ __forceinline__ void items(const SymLaunch& L, unsigned* counter, Smem<W * KS>& sm) {
  constexpr int T = W * KS * 32, TI = W * 32 * R, NC = PHI == sym::kPhiBoth ? 4 : 3;  // sums of a j-body
  const int tid = (int)threadIdx.x, lane = tid & 31, w = tid >> 5, wi = w % W, k0 = w / W * (32 / KS);
  const double4_32a* __restrict__ st = static_cast<const double4_32a*>(L.stage_x);
  double4_32a* part = reinterpret_cast<double4_32a*>(L.part);
  const double eps2 = L.eps2, s2 = L.sigma2;

  ItemSource source{counter, &sm.item};
  for (;;) {
    const int n = source.next();
    if (n >= L.n_items) break;
    const SymItem it = L.items[n];
    if (!sym_item_ok(it, L)) continue;  // NBODY_DEBUG builds only
    double4_32a* oi = part + (it.row0 + (int64_t)it.slot_i * it.stride);
    double4_32a* oj = part + (it.row0 + (int64_t)it.slot_j * it.stride);
    // Padding, i and j on opposite sides so that their difference is not 0. Gravity: massless and
    // far beyond the item's bodies, but in range; Lennard-Jones (no masses in the sums): so far
    // that u^3 is exactly 0.
    // Equal masses are left out of the sums: bodies count 1, padding 0, and blocks without padding
    // need no products with them.
    const bool uniform = LAW == 0 && L.sys[it.sys].uniform != L.epoch;
    const double4_32a q0 = st[it.i_begin];
    const double pad = LAW == 0 ? 1.0e30 * (1.0 + fabs(q0.x) + fabs(q0.y) + fabs(q0.z)) : 3.0e89;

    for (int i0 = it.i_begin; i0 < it.i_end; i0 += TI) {
      double xi[R], yi[R], zi[R], mi[R], ax[R], ay[R], az[R], pp[R];
      const int wi0 = i0 + wi * 32 * R, ig0 = wi0 + lane;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int ig = ig0 + 32 * r;
        const double4_32a v = ig < it.i_end ? st[ig] : make_double4_32a(-pad, -pad, -pad, 0.0);
        xi[r] = v.x, yi[r] = v.y, zi[r] = v.z, mi[r] = uniform && ig < it.i_end ? 1.0 : v.w;
        ax[r] = ay[r] = az[r] = pp[r] = 0.0;
      }
      const int js = max(it.j_begin, i0);
      const bool add = i0 > it.i_begin;
      for (int jt = js; jt < it.j_end; jt += kTile) {
        for (int t = tid; t < kTile; t += T) {
          const double4_32a v = jt + t < it.j_end ? st[jt + t] : make_double4_32a(pad, pad, pad, 0.0);
          double* d = &sm.q[0][t >> 5][t & 31];
          constexpr int S = (kTile / 32) * 64;
          d[0] = d[32] = v.x, d[S] = d[S + 32] = v.y, d[2 * S] = d[2 * S + 32] = v.z;
          d[3 * S] = d[3 * S + 32] = uniform && jt + t < it.j_end ? 1.0 : v.w;
        }
        __syncthreads();
        for (int b = 0; b < kTile / 32; ++b) {
          const int jg0 = jt + 32 * b;
          double jx = 0.0, jy = 0.0, jz = 0.0, jp = 0.0;
          if (jg0 < it.j_end && wi0 < it.i_end) {
            const bool both = jg0 >= wi0 + 32 * R;
            auto run = [&](auto eq) {
              constexpr bool EQ = decltype(eq)::value;
              if (both)
                block<LAW, true, false, PHI, EQ, R, KS>(sm.q, b, k0, jg0, lane, ig0, xi, yi, zi, mi, eps2, s2, ax, ay,
                                                        az, pp, jx, jy, jz, jp);
              else if (jg0 + 32 > wi0)
                block<LAW, false, true, PHI, EQ, R, KS>(sm.q, b, k0, jg0, lane, ig0, xi, yi, zi, mi, eps2, s2, ax, ay,
                                                        az, pp, jx, jy, jz, jp);
            };
            if (LAW == 0 && uniform && jg0 + 32 <= it.j_end && wi0 + 32 * R <= it.i_end)
              run(std::integral_constant<bool, LAW == 0>());
            else
              run(std::false_type());
          }
          const int p = 32 * b + ((lane + k0 + 32 / KS) & 31);  // whose sums have travelled here
          sm.jacc[w][0][p] = jx, sm.jacc[w][1][p] = jy, sm.jacc[w][2][p] = jz;
          if (PHI == sym::kPhiBoth) sm.jacc[w][3][p] = jp;
        }
        __syncthreads();
        for (int t = tid; t < kTile; t += T) {
          const int j = jt + t;
          if (j >= it.j_end) continue;
          double s[4] = {0.0, 0.0, 0.0, 0.0};
          if (add) {
            const double4_32a o = oj[j];
            s[0] = o.x, s[1] = o.y, s[2] = o.z, s[3] = o.w;
          }
#pragma unroll
          for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int u = 0; u < W * KS; ++u) s[c] += sm.jacc[u][c][t];
          oj[j] = make_double4_32a(s[0], s[1], s[2], s[3]);
        }
      }
      if (KS > 1) {  // the i-sums of the warps that share the bodies, through the j-sums' space
        static_assert(R <= kTile / 32, "");
        __syncthreads();
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int p = 32 * r + lane;
          sm.jacc[w][0][p] = ax[r], sm.jacc[w][1][p] = ay[r], sm.jacc[w][2][p] = az[r], sm.jacc[w][3][p] = pp[r];
        }
        __syncthreads();
        if (w < W)
#pragma unroll
          for (int u = 1; u < KS; ++u)
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const int p = 32 * r + lane, o = w + u * W;
              ax[r] += sm.jacc[o][0][p], ay[r] += sm.jacc[o][1][p], az[r] += sm.jacc[o][2][p], pp[r] += sm.jacc[o][3][p];
            }
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (w < W && ig0 + 32 * r < it.i_end) oi[ig0 + 32 * r] = make_double4_32a(ax[r], ay[r], az[r], pp[r]);
      __syncthreads();  // the tile and the j-sums are free for the next i-tile
    }
  }
}

}  // namespace sym64
}  // namespace nbody
