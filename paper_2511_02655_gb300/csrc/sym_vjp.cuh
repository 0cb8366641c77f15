// The force gradient (vector-Jacobian product, adjoint_kernels.cu) with every
// unordered pair evaluated once, in packed float32x2 and in FP64 arithmetic. Work
// list, slots, the travelling j-sums and the tiles are those of sym_common.cuh and
// sym64.cuh; the body sums are those of the one-sided kernels,
//   A1 = sum w_j / s^3,  A2 = sum m_j / s^3,  Gm = sum (d.w_j) / s^3,
//   Gb = sum (m_k (d.w_j) - m_j (d.w_k)) d / s^5
// (with P also Pg = sum m_j (d.w_k) / s^3 and Pe = sum m_j (d.w_k) / s^5).
// Seen from the other end d changes its sign and the weights change places, so the
// bracket of Gb stays and the pair feeds both bodies from one set of powers and dot
// products: 34 float32 operations and one MUFU.RSQ for two interactions instead of
// 52 and two (FP64: 36 instead of about 86). Bound: the FP32 (FP64) pipe.
#pragma once

#include "nbody_internal.h"
#include "pair_common.cuh"
#include "sym64.cuh"
#include "sym_common.cuh"

namespace nbody {
namespace symv {

constexpr int kTile = kSymVjpTile;  // j-bodies per shared-memory tile, mixed

// Padding: s^-3 underflows to 0 there, which is all that these sums need of it. (The force pass's distance, at
// which the reciprocal root itself is 0, would let d.w overflow from |w| = 2e18 on: times the padding's mass 0
// a NaN in the sums of every body of a partial tile. Here it takes 1e20, as in the one-sided kernels.)
constexpr float kPad = 1.0e18f;

template <int W, int R, bool P>
struct Smem {
  static constexpr int NC = P ? 10 : 8;
  float4 xy[kTile / 64][64];  // x0 x1 y0 y1 of a pair of j-bodies, as in sym::Smem
  float4 zm[kTile / 64][64];  // z0 z1 m0 m1
  float4 wxy[kTile / 64][64];
  float2 wz[kTile / 64][64];
  float2 jacc[W][NC][kTile / 64][32];
  float2 hl[NC][R][W * 32];
  int item;
};

// The i-bodies of a lane: -x (both lanes of a pair), -m and w
template <int R>
struct Bodies {
  float2 nx[R], ny[R], nz[R], nm[R], wx[R], wy[R], wz[R];
};
// Sums in the order A1 (3), A2, Gb (3), Gm, Pg, Pe; `i` holds Gb negated, `j` Gm
template <int NC>
struct Sums {
  float2 v[NC];
};

template <bool SYM, bool MASK, bool P, int R>
__device__ __forceinline__ void step(const float4 X, const float4 Z, const float4 WXY, const float2 wzj, const int jg,
                                     const int ig0, const Bodies<R>& B, const float2 e2, Sums<P ? 10 : 8> (&si)[R],
                                     Sums<P ? 10 : 8>& sj, float& mn) {
  const float2 xj = make_float2(X.x, X.y), yj = make_float2(X.z, X.w);
  const float2 zj = make_float2(Z.x, Z.y), mj = make_float2(Z.z, Z.w);
  const float2 wxj = make_float2(WXY.x, WXY.y), wyj = make_float2(WXY.z, WXY.w);
  mn = 3.0e38f;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float2 dx = __fadd2_rn(xj, B.nx[r]);
    const float2 dy = __fadd2_rn(yj, B.ny[r]);
    const float2 dz = __fadd2_rn(zj, B.nz[r]);
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
    const bool s0 = MASK && jg == ig0 + 32 * r, s1 = MASK && jg + 1 == ig0 + 32 * r;
    mn = fminf(mn, fminf(s0 ? 3.0e38f : r2.x, s1 ? 3.0e38f : r2.y));
    float2 inv = make_float2(rsq_approx(r2.x), rsq_approx(r2.y));
    if (MASK) inv.x = s0 ? 0.f : inv.x, inv.y = s1 ? 0.f : inv.y;
    const float2 i2 = __fmul2_rn(inv, inv);
    const float2 i3 = __fmul2_rn(i2, inv);
    const float2 i5 = __fmul2_rn(i3, i2);
    const float2 dwj = __ffma2_rn(dx, wxj, __ffma2_rn(dy, wyj, __fmul2_rn(dz, wzj)));
    const float2 dwk = __ffma2_rn(dx, B.wx[r], __ffma2_rn(dy, B.wy[r], __fmul2_rn(dz, B.wz[r])));
    const float2 pk = __fmul2_rn(mj, dwk);  // m_j (d.w_k)
    const float2 du = __ffma2_rn(B.nm[r], dwj, pk);  // the bracket of Gb, negated
    const float2 qk = P ? __fmul2_rn(B.nm[r], dwj) : pk;  // -m_k (d.w_j)
    const float2 t = __fmul2_rn(du, i5);
    auto acc = [](float2& s, const float2 a, const float2 b) { s = __ffma2_rn(a, b, s); };
    Sums<P ? 10 : 8>& s = si[r];
    acc(s.v[0], i3, wxj), acc(s.v[1], i3, wyj), acc(s.v[2], i3, wzj), acc(s.v[3], i3, mj);
    acc(s.v[4], t, dx), acc(s.v[5], t, dy), acc(s.v[6], t, dz), acc(s.v[7], dwj, i3);
    if constexpr (P) acc(s.v[8], pk, i3), acc(s.v[9], pk, i5);
    if (SYM) {
      acc(sj.v[0], i3, B.wx[r]), acc(sj.v[1], i3, B.wy[r]), acc(sj.v[2], i3, B.wz[r]), acc(sj.v[3], i3, B.nm[r]);
      acc(sj.v[4], t, dx), acc(sj.v[5], t, dy), acc(sj.v[6], t, dz), acc(sj.v[7], dwk, i3);
      if constexpr (P) acc(sj.v[8], qk, i3), acc(sj.v[9], qk, i5);
    }
  }
}
// Signs that turn the sums of step() into those of the file's head
__device__ __forceinline__ float sign_i(const int c) { return c >= 4 && c < 7 ? -1.f : 1.f; }
__device__ __forceinline__ float sign_j(const int c) { return c == 3 || c == 7 ? -1.f : 1.f; }

template <bool SYM, bool MASK, bool P, int R>
__device__ __forceinline__ unsigned block64(const float4* bxy, const float4* bzm, const float4* bwxy, const float2* bwz,
                                            const int jg0, const int lane, const int ig0, const Bodies<R>& B,
                                            const float2 e2, const float r2c, Sums<P ? 10 : 8> (&si)[R],
                                            Sums<P ? 10 : 8>& sj) {
  constexpr int NC = P ? 10 : 8;
  const int src = (lane + 1) & 31;
  unsigned near = 0u;
#pragma unroll 2
  for (int k = 0; k < 32; ++k) {
    const int jg = MASK ? jg0 + 2 * ((lane + k) & 31) : 0;
    float mn;
    step<SYM, MASK, P, R>(bxy[lane + k], bzm[lane + k], bwxy[lane + k], bwz[lane + k], jg, ig0, B, e2, si, sj, mn);
    if (mn < r2c) near |= 1u << k;
    if (SYM) {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        sj.v[c].x = __shfl_sync(0xffffffffu, sj.v[c].x, src);
        sj.v[c].y = __shfl_sync(0xffffffffu, sj.v[c].y, src);
      }
    }
  }
  return near;
}

// Terms of one pair with separation d, times sg, added to (ci, cj) in the sums' signs of step()
template <bool SYM, bool P>
__device__ __forceinline__ void pair_terms(const float dx, const float dy, const float dz, const float r2,
                                           const float mj, const float wxj, const float wyj, const float wzj,
                                           const float nm, const float wx, const float wy, const float wz,
                                           const float sg, float (&ci)[P ? 10 : 8], float (&cj)[P ? 10 : 8]) {
  const float inv = rsq_approx(r2), i2 = inv * inv, i3 = i2 * inv, i5 = i3 * i2;
  const float dwj = fmaf(dx, wxj, fmaf(dy, wyj, dz * wzj)), dwk = fmaf(dx, wx, fmaf(dy, wy, dz * wz));
  const float pk = mj * dwk, qk = nm * dwj, du = fmaf(nm, dwj, pk);
  const float t = (du * i5) * sg, a = i3 * sg, f = i5 * sg;
  ci[0] = fmaf(a, wxj, ci[0]), ci[1] = fmaf(a, wyj, ci[1]), ci[2] = fmaf(a, wzj, ci[2]), ci[3] = fmaf(a, mj, ci[3]);
  ci[4] = fmaf(t, dx, ci[4]), ci[5] = fmaf(t, dy, ci[5]), ci[6] = fmaf(t, dz, ci[6]), ci[7] = fmaf(dwj, a, ci[7]);
  if constexpr (P) ci[8] = fmaf(pk, a, ci[8]), ci[9] = fmaf(pk, f, ci[9]);
  if (SYM) {
    cj[0] = fmaf(a, wx, cj[0]), cj[1] = fmaf(a, wy, cj[1]), cj[2] = fmaf(a, wz, cj[2]), cj[3] = fmaf(a, nm, cj[3]);
    cj[4] = fmaf(t, dx, cj[4]), cj[5] = fmaf(t, dy, cj[5]), cj[6] = fmaf(t, dz, cj[6]), cj[7] = fmaf(dwk, a, cj[7]);
    if constexpr (P) cj[8] = fmaf(qk, a, cj[8]), cj[9] = fmaf(qk, f, cj[9]);
  }
}

// Second look at the near pairs of a block (as sym::refine_block)
template <bool SYM, bool P, int W, int R>
__device__ __forceinline__ void refine_block(const unsigned near, unsigned any, Smem<W, R, P>& sm, const int w,
                                             const int b, const int jg0, const int j_end, const int lane, const int ig0,
                                             const int i_end, const Bodies<R>& B, const float eps2, const float r2c,
                                             const float4* __restrict__ lo, Sums<P ? 10 : 8> (&si)[R]) {
  constexpr int NC = P ? 10 : 8;
  while (any) {
    const int k = __ffs(any) - 1;
    any &= any - 1u;
    if (near >> k & 1u) {
      const int p = (lane + k) & 31;
      const float4 X = sm.xy[b][p], Z = sm.zm[b][p], V = sm.wxy[b][p];
      const float2 U = sm.wz[b][p];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int jg = jg0 + 2 * p + h;
        const float qx = h ? X.y : X.x, qy = h ? X.w : X.z, qz = h ? Z.y : Z.x, qm = h ? Z.w : Z.z;
        const float vx = h ? V.y : V.x, vy = h ? V.w : V.z, vz = h ? U.y : U.x;
        float cj[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) cj[c] = 0.f;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int ig = ig0 + 32 * r;
          const float dx = qx + B.nx[r].x, dy = qy + B.ny[r].x, dz = qz + B.nz[r].x;
          const float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps2)));
          if (r2 < r2c && ig < i_end && jg < j_end && ig != jg) {
            float ex, ey, ez, e2, ci[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) ci[c] = 0.f;
            refine_pair(lo, ig, jg, dx, dy, dz, eps2, ex, ey, ez, e2);
            pair_terms<SYM, P>(dx, dy, dz, r2, qm, vx, vy, vz, B.nm[r].x, B.wx[r].x, B.wy[r].x, B.wz[r].x, -1.f, ci,
                               cj);
            pair_terms<SYM, P>(ex, ey, ez, e2, qm, vx, vy, vz, B.nm[r].x, B.wx[r].x, B.wy[r].x, B.wz[r].x, 1.f, ci,
                               cj);
#pragma unroll
            for (int c = 0; c < NC; ++c) si[r].v[c].x += ci[c];
          }
        }
        if (SYM) {
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            float* s = &sm.jacc[w][c][b][p].x + h;
            *s += cj[c];
          }
        }
      }
    }
    __syncwarp();
  }
}

template <int NC>
__device__ __forceinline__ void put_partial(fpair4* o, const float (&h)[NC], const float (&l)[NC]) {
#pragma unroll
  for (int c = 0; c < NC; c += 4) {
    float4 a = make_float4(h[c], l[c], h[c + 1], l[c + 1]), b = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c + 2 < NC) b = make_float4(h[c + 2], l[c + 2], h[c + 3], l[c + 3]);
    __stcg(&o[c / 4].xy, a);
    __stcg(&o[c / 4].zp, b);
  }
}

template <int W, int R, bool P>
__device__ __forceinline__ void items(const SymLaunch& L, unsigned* counter, Smem<W, R, P>& sm) {
  constexpr int T = W * 32, NB = kTile / 64, TI = T * R, LPT = (kTile + T - 1) / T, NC = P ? 10 : 8, KW = P ? 3 : 2;
  const int tid = (int)threadIdx.x, lane = tid & 31, w = tid >> 5;
  const float4* __restrict__ st = static_cast<const float4*>(L.stage_x);
  const float4* __restrict__ sw = static_cast<const float4*>(L.stage_w);
  const float4* __restrict__ lo = L.stage_lo;
  fpair4* part = reinterpret_cast<fpair4*>(L.part);
  const float2 zero = make_float2(0.f, 0.f);

  ItemSource source{counter, &sm.item};
  for (;;) {
    const int n = source.next();
    if (n >= L.n_items) break;
    const SymItem it = L.items[n];
    if (!sym_item_ok(it, L)) continue;  // NBODY_DEBUG builds only
    const float eps2 = L.sys[it.sys].eps2, r2c = lo ? L.sys[it.sys].r2c : 0.f;
    const float2 e2 = make_float2(eps2, eps2);
    fpair4* oi = part + KW * (it.row0 + (int64_t)it.slot_i * it.stride);
    fpair4* oj = part + KW * (it.row0 + (int64_t)it.slot_j * it.stride);

    for (int i0 = it.i_begin; i0 < it.i_end; i0 += TI) {
      Bodies<R> B;
      Sums<NC> si[R];
      const int wi0 = i0 + w * 32 * R, ig0 = wi0 + lane;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int ig = ig0 + 32 * r;
        const bool ok = ig < it.i_end;
        const float4 q = ok ? st[ig] : make_float4(-kPad, -kPad, -kPad, 0.f);
        const float4 u = ok ? sw[ig] : make_float4(0.f, 0.f, 0.f, 0.f);
        B.nx[r] = make_float2(-q.x, -q.x), B.ny[r] = make_float2(-q.y, -q.y), B.nz[r] = make_float2(-q.z, -q.z);
        B.nm[r] = make_float2(-q.w, -q.w);
        B.wx[r] = make_float2(u.x, u.x), B.wy[r] = make_float2(u.y, u.y), B.wz[r] = make_float2(u.z, u.z);
#pragma unroll
        for (int c = 0; c < NC; ++c) sm.hl[c][r][tid] = zero;
      }
      const int js = max(it.j_begin, i0);
      const bool add = i0 > it.i_begin;
      for (int jt = js; jt < it.j_end; jt += kTile) {
#pragma unroll
        for (int k = 0; k < LPT; ++k) {
          const int t = tid + k * T, j = jt + t;
          if (t < kTile) {
            const float4 q = j < it.j_end ? st[j] : make_float4(kPad, kPad, kPad, 0.f);
            const float4 u = j < it.j_end ? sw[j] : make_float4(0.f, 0.f, 0.f, 0.f);
            const int b = t >> 6, p = (t & 63) >> 1, h = t & 1;
            float* a = &sm.xy[b][p].x + h;
            float* c = &sm.zm[b][p].x + h;
            float* d = &sm.wxy[b][p].x + h;
            float* e = &sm.wz[b][p].x + h;
            a[0] = a[128] = q.x, a[2] = a[130] = q.y, c[0] = c[128] = q.z, c[2] = c[130] = q.w;
            d[0] = d[128] = u.x, d[2] = d[130] = u.y, e[0] = e[64] = u.z;
          }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int c = 0; c < NC; ++c) si[r].v[c] = zero;
        for (int b = 0; b < NB; ++b) {
          const int jg0 = jt + 64 * b;
          Sums<NC> sj;
#pragma unroll
          for (int c = 0; c < NC; ++c) sj.v[c] = zero;
          unsigned near = 0u;
          bool both = false;
          if (jg0 < it.j_end && wi0 < it.i_end) {
            both = jg0 >= wi0 + 32 * R;
            if (both)
              near = block64<true, false, P, R>(sm.xy[b], sm.zm[b], sm.wxy[b], sm.wz[b], jg0, lane, ig0, B, e2, r2c, si,
                                                sj);
            else if (jg0 + 64 > wi0)
              near = block64<false, true, P, R>(sm.xy[b], sm.zm[b], sm.wxy[b], sm.wz[b], jg0, lane, ig0, B, e2, r2c, si,
                                                sj);
          }
#pragma unroll
          for (int c = 0; c < NC; ++c) sm.jacc[w][c][b][lane] = sj.v[c];
          const unsigned any = __reduce_or_sync(0xffffffffu, near);
          if (any) {
            __syncwarp();
            if (both)
              refine_block<true, P, W, R>(near, any, sm, w, b, jg0, it.j_end, lane, ig0, it.i_end, B, eps2, r2c, lo, si);
            else
              refine_block<false, P, W, R>(near, any, sm, w, b, jg0, it.j_end, lane, ig0, it.i_end, B, eps2, r2c, lo,
                                           si);
          }
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            float2 s = sm.hl[c][r][tid];
            two_sum_acc(s.x, s.y, sign_i(c) * (si[r].v[c].x + si[r].v[c].y));
            sm.hl[c][r][tid] = s;
          }
        __syncthreads();
        for (int t = tid; t < kTile; t += T) {
          const int j = jt + t;
          if (j >= it.j_end) continue;
          fpair4* o = oj + KW * (int64_t)j;
          float h[NC], l[NC];
#pragma unroll
          for (int c = 0; c < NC; c += 2) {
            float4 old = make_float4(0.f, 0.f, 0.f, 0.f);
            if (add) old = __ldcg(reinterpret_cast<const float4*>(o) + c / 2);
            h[c] = old.x, l[c] = old.y, h[c + 1] = old.z, l[c + 1] = old.w;
          }
#pragma unroll
          for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int u = 0; u < W; ++u)
              two_sum_acc(h[c], l[c], sign_j(c) * (&sm.jacc[u][c][t >> 6][(t & 63) >> 1].x)[t & 1]);
          put_partial<NC>(o, h, l);
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int ig = ig0 + 32 * r;
        if (ig < it.i_end) {
          float h[NC], l[NC];
#pragma unroll
          for (int c = 0; c < NC; ++c) h[c] = sm.hl[c][r][tid].x, l[c] = sm.hl[c][r][tid].y;
          put_partial<NC>(oi + KW * (int64_t)ig, h, l);
        }
      }
      __syncthreads();  // the tile and the j-sums are free for the next i-tile
    }
  }
}

// ---- FP64: one j-body per lane (see sym64.cuh)

template <int W, bool P>
struct Smem64 {
  static constexpr int NC = P ? 10 : 8;
  double q[7][kSymTile64 / 32][64];  // x, y, z, m, w
  double jacc[W][NC][kSymTile64];
  int item;
};

struct Body64 {
  double x, y, z, m, wx, wy, wz;
};

template <bool SYM, bool MASK, bool P, bool FAST, int KS>
__device__ __forceinline__ bool block32(const double (&q)[7][kSymTile64 / 32][64], const int b, const int k0,
                                        const int jg0, const int lane, const int ig, const Body64& B, const double eps2,
                                        double (&si)[P ? 10 : 8], double (&sj)[P ? 10 : 8]) {
  constexpr int NC = P ? 10 : 8;
  const int src = (lane + 1) & 31;
  bool out = false;
#pragma unroll(FAST ? 2 : 1)
  for (int k = 0; k < 32 / KS; ++k) {
    const int p = lane + k0 + k;
    const double dx = q[0][b][p] - B.x, dy = q[1][b][p] - B.y, dz = q[2][b][p] - B.z, mj = q[3][b][p];
    const double wxj = q[4][b][p], wyj = q[5][b][p], wzj = q[6][b][p];
    const double r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2)));
    const bool self = MASK && jg0 + (p & 31) == ig;
    double i2, i3;
    if (FAST) {
      out |= !self && !sym64::in_range(r2);
      const sym64::Root t = sym64::root_of(r2);
      i2 = sym64::inv2_of(t), i3 = sym64::inv3_of(t);
    } else {
      const double inv = rsqrt(r2);
      i2 = inv * inv, i3 = i2 * inv;
    }
    if (self) i2 = i3 = 0.0;
    const double i5 = i3 * i2;
    const double dwj = fma(dx, wxj, fma(dy, wyj, dz * wzj)), dwk = fma(dx, B.wx, fma(dy, B.wy, dz * B.wz));
    const double pk = mj * dwk;
    const double du = fma(B.m, dwj, -pk);     // m_k (d.w_j) - m_j (d.w_k)
    const double qk = P ? B.m * dwj : 0.0;  // m_k (d.w_j)
    const double t = du * i5;
    auto acc = [](double& s, const double x, const double y) { s = fma(x, y, s); };
    acc(si[0], i3, wxj), acc(si[1], i3, wyj), acc(si[2], i3, wzj), acc(si[3], i3, mj);
    acc(si[4], t, dx), acc(si[5], t, dy), acc(si[6], t, dz), acc(si[7], dwj, i3);
    if constexpr (P) acc(si[8], pk, i3), acc(si[9], pk, i5);
    if (SYM) {
      acc(sj[0], i3, B.wx), acc(sj[1], i3, B.wy), acc(sj[2], i3, B.wz), acc(sj[3], i3, B.m);
      acc(sj[4], -t, dx), acc(sj[5], -t, dy), acc(sj[6], -t, dz), acc(sj[7], -dwk, i3);
      if constexpr (P) acc(sj[8], -qk, i3), acc(sj[9], -qk, i5);
#pragma unroll
      for (int c = 0; c < NC; ++c) sj[c] = __shfl_sync(0xffffffffu, sj[c], src);
    }
  }
  return out;
}

template <bool SYM, bool MASK, bool P, int KS>
__device__ __forceinline__ void block(const double (&q)[7][kSymTile64 / 32][64], const int b, const int k0, const int jg0,
                                      const int lane, const int ig, const Body64& B, const double eps2,
                                      double (&si)[P ? 10 : 8], double (&sj)[P ? 10 : 8]) {
  constexpr int NC = P ? 10 : 8;
  double s0[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) s0[c] = si[c], si[c] = 0.0;
  if (__any_sync(0xffffffffu, block32<SYM, MASK, P, true, KS>(q, b, k0, jg0, lane, ig, B, eps2, si, sj))) {
#pragma unroll
    for (int c = 0; c < NC; ++c) si[c] = sj[c] = 0.0;
    block32<SYM, MASK, P, false, KS>(q, b, k0, jg0, lane, ig, B, eps2, si, sj);
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) si[c] += s0[c];
}

template <int W, bool P, int KS>
__device__ __forceinline__ void items64(const SymLaunch& L, unsigned* counter, Smem64<W * KS, P>& sm) {
  constexpr int T = W * KS * 32, TI = W * 32, NC = P ? 10 : 8, KW = P ? 3 : 2, J = kSymTile64;
  const int tid = (int)threadIdx.x, lane = tid & 31, w = tid >> 5, wi = w % W, k0 = w / W * (32 / KS);
  const double4_32a* __restrict__ st = static_cast<const double4_32a*>(L.stage_x);
  const double4_32a* __restrict__ sw = static_cast<const double4_32a*>(L.stage_w);
  double4_32a* part = reinterpret_cast<double4_32a*>(L.part);
  const double eps2 = L.eps2;

  ItemSource source{counter, &sm.item};
  for (;;) {
    const int n = source.next();
    if (n >= L.n_items) break;
    const SymItem it = L.items[n];
    if (!sym_item_ok(it, L)) continue;  // NBODY_DEBUG builds only
    double* oi = reinterpret_cast<double*>(part + KW * (it.row0 + (int64_t)it.slot_i * it.stride));
    double* oj = reinterpret_cast<double*>(part + KW * (it.row0 + (int64_t)it.slot_j * it.stride));
    const double4_32a q0 = st[it.i_begin];
    const double pad = 1.0e30 * (1.0 + fabs(q0.x) + fabs(q0.y) + fabs(q0.z));  // as in sym64::items

    for (int i0 = it.i_begin; i0 < it.i_end; i0 += TI) {
      const int wi0 = i0 + wi * 32, ig = wi0 + lane;
      const bool live = ig < it.i_end;
      Body64 B{-pad, -pad, -pad, 0.0, 0.0, 0.0, 0.0};
      if (live) {
        const double4_32a v = st[ig], u = sw[ig];
        B = Body64{v.x, v.y, v.z, v.w, u.x, u.y, u.z};
      }
      double si[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) si[c] = 0.0;
      const int js = max(it.j_begin, i0);
      const bool add = i0 > it.i_begin;
      for (int jt = js; jt < it.j_end; jt += J) {
        for (int t = tid; t < J; t += T) {
          double4_32a v = make_double4_32a(pad, pad, pad, 0.0), u = make_double4_32a(0.0, 0.0, 0.0, 0.0);
          if (jt + t < it.j_end) v = st[jt + t], u = sw[jt + t];
          double* d = &sm.q[0][t >> 5][t & 31];
          constexpr int S = (J / 32) * 64;
          d[0] = d[32] = v.x, d[S] = d[S + 32] = v.y, d[2 * S] = d[2 * S + 32] = v.z, d[3 * S] = d[3 * S + 32] = v.w;
          d[4 * S] = d[4 * S + 32] = u.x, d[5 * S] = d[5 * S + 32] = u.y, d[6 * S] = d[6 * S + 32] = u.z;
        }
        __syncthreads();
        for (int b = 0; b < J / 32; ++b) {
          const int jg0 = jt + 32 * b;
          double sj[NC];
#pragma unroll
          for (int c = 0; c < NC; ++c) sj[c] = 0.0;
          if (jg0 < it.j_end && wi0 < it.i_end) {
            if (jg0 >= wi0 + 32)
              block<true, false, P, KS>(sm.q, b, k0, jg0, lane, ig, B, eps2, si, sj);
            else if (jg0 + 32 > wi0)
              block<false, true, P, KS>(sm.q, b, k0, jg0, lane, ig, B, eps2, si, sj);
          }
#pragma unroll
          for (int c = 0; c < NC; ++c) sm.jacc[w][c][32 * b + ((lane + k0 + 32 / KS) & 31)] = sj[c];
        }
        __syncthreads();
        for (int t = tid; t < J; t += T) {
          const int j = jt + t;
          if (j >= it.j_end) continue;
          double* o = oj + 4 * KW * (int64_t)j;
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            double s = add ? o[c] : 0.0;
#pragma unroll
            for (int u = 0; u < W * KS; ++u) s += sm.jacc[u][c][t];
            o[c] = s;
          }
        }
      }
      if (KS > 1) {  // as in sym64::items
        __syncthreads();
#pragma unroll
        for (int c = 0; c < NC; ++c) sm.jacc[w][c][lane] = si[c];
        __syncthreads();
        if (w < W)
#pragma unroll
          for (int u = 1; u < KS; ++u)
#pragma unroll
            for (int c = 0; c < NC; ++c) si[c] += sm.jacc[w + u * W][c][lane];
      }
      if (live && w < W) {
        double* o = oi + 4 * KW * (int64_t)ig;
#pragma unroll
        for (int c = 0; c < NC; ++c) o[c] = si[c];
      }
      __syncthreads();  // the tile and the j-sums are free for the next i-tile
    }
  }
}

}  // namespace symv
}  // namespace nbody
