// All-pairs force pass that evaluates every unordered pair once (Newton's third
// law), for softened gravity and the Lennard-Jones law in packed float32x2
// arithmetic.
//
// Why: the one-sided kernels (force_common.cuh) are bound by the FP32 pipe and
// evaluate each pair from both of its ends. Separation, s^2, the reciprocal root
// and its powers are the same from either end, so one evaluation that feeds both
// bodies costs 16 float32 operations (18 with both potentials) and one MUFU.RSQ
// for two interactions instead of 2 x 12 (2 x 13) and two; where all masses of a
// system are equal their two products drop out as well (14).
//
// How: a warp holds 32 R i-bodies in registers (R per lane) and works through
// blocks of 64 j-bodies, two per lane as float32x2 pairs. In step k = 0..31 of a
// block lane l meets j-pair (l + k) mod 32. The pair's coordinates come from a
// shared-memory tile (kept twice in a row, so that l + k needs no wrap), its
// running sums travel: after each step every lane passes them to the lane below
// (SHFL), which meets that pair next, and after 32 steps they are complete
// for the warp's i-bodies. The CTA's W warps share the j-tile; their j-sums go to
// shared memory, are added with TwoSum and written as one compensated partial per
// j-body and row of i-tiles. Nothing is added with atomics and every sum has a
// fixed order.
//
// Work list: the i-range of a system is cut into rows of whole i-tiles; a row
// meets the bodies from its own start to the system's end, in pieces of a few
// i-tile areas each (SymItem). Body slots of partial sums: one per row that meets
// the body as j (slot = row), then one per piece of the body's own row.
// Within a row's own i-tile, warps meet later 64-body blocks symmetrically and
// the blocks overlapping their own i-bodies one-sided, with the self pair masked.
#pragma once

#include "nbody_internal.h"
#include "pair_common.cuh"

namespace nbody {
namespace sym {

// Padding of tiles and i-tiles: so far away that s^2 overflows to infinity and
// its reciprocal (root) is exactly 0; i- and j-padding lie on opposite sides, so
// that their difference is finite too.
constexpr float kPad = 3.0e19f;

template <int W, int R, int J>
struct Smem {
  float4 xy[J / 64][64];  // pair p of a 64-body block (its bodies 2p, 2p+1): x0 x1 y0 y1; entries 32.. repeat 0..
  float4 zm[J / 64][64];  // z0 z1 m0 m1
  float2 jacc[W][4][J / 64][32];  // each warp's sums for the j-pairs of the tile
  float2 hl[4][R][W * 32];        // compensated (hi, lo) sums of the thread's i-bodies
  int item;
};

// Potential: none, of both bodies, or for an energy record, which needs only sum m phi: each pair's
// term counted once, at its i-body (and half in the one-sided blocks, which hold a pair twice), one
// operation and two shuffles less; U is then the whole sum, not half of it.
enum { kPhiNone = 0, kPhiBoth = 1, kPhiEnergy = 2 };

// One step: the lane's j-pair against its R i-bodies. SYM: also the j-pair's sums;
// MASK: the self pair is left out (jg: global index of the pair's first body); EQ: equal
// masses, left out of the sums (staged as 1). mn: the smallest s^2 met.
template <int LAW, bool SYM, bool MASK, int PHI, bool EQ, int R>
__device__ __forceinline__ void step(const float4 X, const float4 Z, const int jg, const int ig0, const float2 (&nx)[R],
                                     const float2 (&ny)[R], const float2 (&nz)[R], const float2 (&mi)[R],
                                     const float2 e2, float2 (&ax)[R], float2 (&ay)[R], float2 (&az)[R],
                                     float2 (&pp)[R], float2& jx, float2& jy, float2& jz, float2& jp, float& mn) {
  const float2 xj = make_float2(X.x, X.y), yj = make_float2(X.z, X.w);
  const float2 zj = make_float2(Z.x, Z.y), mj = make_float2(Z.z, Z.w);
  constexpr bool HALF = MASK && PHI == kPhiEnergy;  // these blocks hold both orders of a pair
  mn = 3.0e38f;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float2 dx = __fadd2_rn(xj, nx[r]);
    const float2 dy = __fadd2_rn(yj, ny[r]);
    const float2 dz = __fadd2_rn(zj, nz[r]);
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
    const bool s0 = MASK && jg == ig0 + 32 * r, s1 = MASK && jg + 1 == ig0 + 32 * r;
    mn = fminf(mn, fminf(s0 ? 3.0e38f : r2.x, s1 ? 3.0e38f : r2.y));
    float2 inv = LAW == 0 ? make_float2(rsq_approx(r2.x), rsq_approx(r2.y))
                          : make_float2(rcp_approx(r2.x), rcp_approx(r2.y));
    if (MASK) inv.x = s0 ? 0.f : inv.x, inv.y = s1 ? 0.f : inv.y;
    if (LAW == 0) {
      const float2 i3 = __fmul2_rn(__fmul2_rn(inv, inv), inv);
      const float2 wj = EQ ? i3 : __fmul2_rn(i3, mj);
      ax[r] = __ffma2_rn(dx, wj, ax[r]);
      ay[r] = __ffma2_rn(dy, wj, ay[r]);
      az[r] = __ffma2_rn(dz, wj, az[r]);
      const float2 one = HALF ? __fmul2_rn(inv, make_float2(0.5f, 0.5f)) : inv;
      if (PHI) pp[r] = EQ ? __fadd2_rn(pp[r], one) : __ffma2_rn(mj, one, pp[r]);
      if (SYM) {
        const float2 wi = EQ ? i3 : __fmul2_rn(i3, mi[r]);
        jx = __ffma2_rn(dx, wi, jx);
        jy = __ffma2_rn(dy, wi, jy);
        jz = __ffma2_rn(dz, wi, jz);
        if (PHI == kPhiBoth) jp = EQ ? __fadd2_rn(jp, inv) : __ffma2_rn(mi[r], inv, jp);
      }
    } else {  // u = sigma^2 / r^2 (positions staged in units of sigma)
      const float2 u3 = __fmul2_rn(inv, __fmul2_rn(inv, inv));
      const float2 u6 = __fmul2_rn(u3, u3);
      const float2 w = __fmul2_rn(__ffma2_rn(u6, make_float2(-2.f, -2.f), u3), inv);
      ax[r] = __ffma2_rn(dx, w, ax[r]);
      ay[r] = __ffma2_rn(dy, w, ay[r]);
      az[r] = __ffma2_rn(dz, w, az[r]);
      if (SYM) {
        jx = __ffma2_rn(dx, w, jx);
        jy = __ffma2_rn(dy, w, jy);
        jz = __ffma2_rn(dz, w, jz);
      }
      if (PHI) {
        const float2 p = __ffma2_rn(u3, make_float2(-1.f, -1.f), u6);
        pp[r] = HALF ? __ffma2_rn(p, make_float2(0.5f, 0.5f), pp[r]) : __fadd2_rn(pp[r], p);
        if (SYM && PHI == kPhiBoth) jp = __fadd2_rn(jp, p);
      }
    }
  }
}

// Unroll depth of the step loop (even: bank-conflict-free code either way; 4 was
// 2-3% faster than 2 and 1 with R = 4 at N = 65 536, 8 no faster).
constexpr int kUnroll = 4;

// The 32 steps of one 64-body block. Returns the lane's bit mask of steps that met
// a near pair (s^2 below r2c).
template <int LAW, bool SYM, bool MASK, int PHI, bool EQ, int R>
__device__ __forceinline__ unsigned block64(const float4* bxy, const float4* bzm, const int jg0, const int lane,
                                            const int ig0, const float2 (&nx)[R], const float2 (&ny)[R],
                                            const float2 (&nz)[R], const float2 (&mi)[R], const float2 e2,
                                            const float r2c, float2 (&ax)[R], float2 (&ay)[R], float2 (&az)[R],
                                            float2 (&pp)[R], float2& jx, float2& jy, float2& jz, float2& jp) {
  unsigned near = 0u;
  const int src = (lane + 1) & 31;
  auto pass = [&](float2& v) {
    v.x = __shfl_sync(0xffffffffu, v.x, src);
    v.y = __shfl_sync(0xffffffffu, v.y, src);
  };
#pragma unroll(kUnroll)
  for (int k = 0; k < 32; ++k) {
    const float4 X = bxy[lane + k], Z = bzm[lane + k];
    const int jg = MASK ? jg0 + 2 * ((lane + k) & 31) : 0;
    float mn;
    step<LAW, SYM, MASK, PHI, EQ, R>(X, Z, jg, ig0, nx, ny, nz, mi, e2, ax, ay, az, pp, jx, jy, jz, jp, mn);
    if (mn < r2c) near |= 1u << k;
    if (SYM) {
      pass(jx), pass(jy), pass(jz);
      if (PHI == kPhiBoth) pass(jp);
    }
  }
  return near;
}

// The refined-minus-unrefined force term f d (and potential term) of one near pair, with the
// first pass's operations for the unrefined part: t = (f d, f's potential) without masses.
template <int LAW>
__device__ __forceinline__ void pair_terms(const float r2, float& f, float& p) {
  if (LAW == 0) {
    p = rsq_approx(r2);
    f = (p * p) * p;
  } else {
    const float u = rcp_approx(r2);
    const float u3 = u * (u * u), u6 = u3 * u3;
    f = fmaf(u6, -2.f, u3) * u;
    p = fmaf(u3, -1.f, u6);
  }
}

// Second look at the near pairs of a block: `near` holds the lane's flagged steps, in which it
// revisits its own j-pair. Lanes walk their own flags, so that a warp takes as many rounds as its
// busiest lane has flagged steps, not as many as the union of all lanes' steps (in a
// Lennard-Jones gas, where a lane flags one or two of the 32 steps but the warp a quarter of
// them, a force pass at 10 000 bodies fell from over 85 us to 65). The i-sums are corrected in registers, the
// j-sums in the warp's shared entries; lanes that meet the same j-pair in a round take
// turns in lane order.
template <int LAW, bool SYM, int PHI, int R, int NB>
__device__ __forceinline__ void refine_block(unsigned near, const float4* bxy, const float4* bzm, const int b,
                                             const int jg0, const int j_end, const int lane, const int ig0,
                                             const int i_end, const float2 (&nx)[R], const float2 (&ny)[R],
                                             const float2 (&nz)[R], const float2 (&mi)[R], const float eps2,
                                             const float r2c, const float4* __restrict__ lo, float2 (&ax)[R],
                                             float2 (&ay)[R], float2 (&az)[R], float2 (&pp)[R],
                                             float2 (&jacc)[4][NB][32]) {
  while (__any_sync(0xffffffffu, near != 0u)) {
    const bool on = near != 0u;
    const int p = on ? (lane + __ffs(near) - 1) & 31 : 0;
    near &= near - 1u;
    float2 cx = make_float2(0.f, 0.f), cy = cx, cz = cx, cp = cx;  // corrections of the pair's two j-bodies
    if (on) {
      const float4 X = bxy[p], Z = bzm[p];
      const int jg = jg0 + 2 * p;
      unsigned sub = 0u;  // the near ones among the 2 R pairs of the step
#pragma unroll
      for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float dx = (h ? X.y : X.x) + nx[r].x, dy = (h ? X.w : X.z) + ny[r].x, dz = (h ? Z.y : Z.x) + nz[r].x;
          const float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps2)));
          const int ig = ig0 + 32 * r;
          if (r2 < r2c && ig < i_end && jg + h < j_end && ig != jg + h) sub |= 1u << (2 * r + h);
        }
      }
      while (sub) {
        const int k = __ffs(sub) - 1, h = k & 1, r = k >> 1;
        sub &= sub - 1u;
        float bx = nx[0].x, by = ny[0].x, bz = nz[0].x, m = mi[0].x;
#pragma unroll
        for (int q = 1; q < R; ++q)
          if (r == q) bx = nx[q].x, by = ny[q].x, bz = nz[q].x, m = mi[q].x;
        const float dx = (h ? X.y : X.x) + bx, dy = (h ? X.w : X.z) + by, dz = (h ? Z.y : Z.x) + bz;
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps2)));
        float ex, ey, ez, e2, fu, pu, fr, pr;
        refine_pair(lo, ig0 + 32 * r, jg + h, dx, dy, dz, eps2, ex, ey, ez, e2);
        pair_terms<LAW>(r2, fu, pu);
        pair_terms<LAW>(e2, fr, pr);
        const float mj = LAW == 0 ? (h ? Z.w : Z.z) : 1.f;
        if (LAW == 1) m = 1.f;
        const float uj = fu * mj, vj = fr * mj;
        const float tx = fmaf(ex, vj, -(dx * uj)), ty = fmaf(ey, vj, -(dy * uj)), tz = fmaf(ez, vj, -(dz * uj));
        const float half = PHI == kPhiEnergy && !SYM ? 0.5f : 1.f;
        const float tp = PHI ? half * fmaf(mj, pr, -(mj * pu)) : 0.f;
#pragma unroll
        for (int q = 0; q < R; ++q)
          if (r == q) {
            ax[q].x += tx, ay[q].x += ty, az[q].x += tz;
            if (PHI) pp[q].x += tp;
          }
        if (SYM) {
          const float ui = fu * m, vi = fr * m;
          const float sx = fmaf(ex, vi, -(dx * ui)), sy = fmaf(ey, vi, -(dy * ui)), sz = fmaf(ez, vi, -(dz * ui));
          const float sp = PHI == kPhiBoth ? fmaf(m, pr, -(m * pu)) : 0.f;
          if (h)
            cx.y += sx, cy.y += sy, cz.y += sz, cp.y += sp;
          else
            cx.x += sx, cy.x += sy, cz.x += sz, cp.x += sp;
        }
      }
    }
    if (SYM) {
      const unsigned same = __match_any_sync(0xffffffffu, on ? p : 32 + lane);
      const int turn = __popc(same & ((1u << lane) - 1u));
      const int turns = __reduce_max_sync(0xffffffffu, turn);
      for (int t = 0; t <= turns; ++t) {
        if (on && turn == t) {
          auto add = [&](float2& s, const float2 c) { s.x += c.x, s.y += c.y; };
          add(jacc[0][b][p], cx), add(jacc[1][b][p], cy), add(jacc[2][b][p], cz);
          if (PHI == kPhiBoth) add(jacc[3][b][p], cp);
        }
        __syncwarp();
      }
    }
  }
}

// Work items, taken from next(SymItem&) until it returns false (called by all threads of the
// CTA, after a barrier of its own if it is called again).
template <int LAW, int W, int R, int J, int PHI, typename Next>
__device__ __forceinline__ void items(const SymLaunch& L, Next next, Smem<W, R, J>& sm) {
  constexpr int T = W * 32, NB = J / 64, TI = T * R, LPT = (J + T - 1) / T;
  constexpr int NC = PHI ? 4 : 3, NCJ = PHI == kPhiBoth ? 4 : 3;  // sums of an i-body, of a j-body
  const int tid = (int)threadIdx.x, lane = tid & 31, w = tid >> 5;
  const float4* __restrict__ st = static_cast<const float4*>(L.stage_x);
  const float4* __restrict__ lo = L.stage_lo;
  fpair4* part = reinterpret_cast<fpair4*>(L.part);

  SymItem it;
  while (next(it)) {
    if (!sym_item_ok(it, L)) continue;  // NBODY_DEBUG builds only
    const float eps2 = L.sys[it.sys].eps2, r2c = lo ? L.sys[it.sys].r2c : 0.f;
    const bool uniform = LAW == 0 && L.sys[it.sys].uniform != 0u;
    const float2 e2 = make_float2(eps2, eps2);
    fpair4* __restrict__ oi = part + (it.row0 + (int64_t)it.slot_i * it.stride);
    fpair4* oj = part + (it.row0 + (int64_t)it.slot_j * it.stride);

    for (int i0 = it.i_begin; i0 < it.i_end; i0 += TI) {
      float2 nx[R], ny[R], nz[R], mi[R], ax[R], ay[R], az[R], pp[R];
      const int wi0 = i0 + w * 32 * R, ig0 = wi0 + lane;  // the lane's bodies: ig0 + 32 r
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int ig = ig0 + 32 * r;
        const float4 q = ig < it.i_end ? st[ig] : make_float4(-kPad, -kPad, -kPad, 0.f);
        nx[r] = make_float2(-q.x, -q.x);
        ny[r] = make_float2(-q.y, -q.y);
        nz[r] = make_float2(-q.z, -q.z);
        mi[r] = make_float2(q.w, q.w);
#pragma unroll
        for (int c = 0; c < NC; ++c) sm.hl[c][r][tid] = make_float2(0.f, 0.f);
      }
      // a row's own bodies are met from the i-tile on; the row's first i-tile meets (and so
      // writes) every j-body of the piece, later ones add to what it wrote
      const int js = max(it.j_begin, i0);
      const bool add = i0 > it.i_begin;
      auto fetch = [&](const int j) {
        return j < it.j_end ? st[j] : make_float4(kPad, kPad, kPad, 0.f);
      };
      float4 pre[LPT];
#pragma unroll
      for (int k = 0; k < LPT; ++k)
        if (tid + k * T < J) pre[k] = fetch(js + tid + k * T);

      for (int jt = js; jt < it.j_end; jt += J) {
#pragma unroll
        for (int k = 0; k < LPT; ++k) {
          const int t = tid + k * T;
          if (t < J) {
            float* a = &sm.xy[t >> 6][(t & 63) >> 1].x + (t & 1);
            float* c = &sm.zm[t >> 6][(t & 63) >> 1].x + (t & 1);
            a[0] = pre[k].x, a[2] = pre[k].y, c[0] = pre[k].z, c[2] = pre[k].w;
            a[128] = pre[k].x, a[130] = pre[k].y, c[128] = pre[k].z, c[130] = pre[k].w;
          }
        }
        __syncthreads();
        if (jt + J < it.j_end) {
#pragma unroll
          for (int k = 0; k < LPT; ++k)
            if (tid + k * T < J) pre[k] = fetch(jt + J + tid + k * T);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) ax[r] = ay[r] = az[r] = pp[r] = make_float2(0.f, 0.f);
        for (int b = 0; b < NB; ++b) {
          const int jg0 = jt + 64 * b;
          float2 jx = make_float2(0.f, 0.f), jy = jx, jz = jx, jp = jx;
          unsigned near = 0u;
          bool both = false;
          if (jg0 < it.j_end && wi0 < it.i_end) {
            both = jg0 >= wi0 + 32 * R;
            if (both) {
              if (uniform)
                near = block64<LAW, true, false, PHI, true, R>(sm.xy[b], sm.zm[b], jg0, lane, ig0, nx, ny, nz, mi, e2,
                                                               r2c, ax, ay, az, pp, jx, jy, jz, jp);
              else
                near = block64<LAW, true, false, PHI, false, R>(sm.xy[b], sm.zm[b], jg0, lane, ig0, nx, ny, nz, mi,
                                                                e2, r2c, ax, ay, az, pp, jx, jy, jz, jp);
            } else if (jg0 + 64 > wi0) {
              near = block64<LAW, false, true, PHI, false, R>(sm.xy[b], sm.zm[b], jg0, lane, ig0, nx, ny, nz, mi, e2,
                                                              r2c, ax, ay, az, pp, jx, jy, jz, jp);
            }
          }
          sm.jacc[w][0][b][lane] = jx, sm.jacc[w][1][b][lane] = jy, sm.jacc[w][2][b][lane] = jz;
          if (PHI == kPhiBoth) sm.jacc[w][3][b][lane] = jp;
          if (__any_sync(0xffffffffu, near != 0u)) {
            __syncwarp();
            if (both)
              refine_block<LAW, true, PHI, R, NB>(near, sm.xy[b], sm.zm[b], b, jg0, it.j_end, lane, ig0, it.i_end,
                                                  nx, ny, nz, mi, eps2, r2c, lo, ax, ay, az, pp, sm.jacc[w]);
            else
              refine_block<LAW, false, PHI, R, NB>(near, sm.xy[b], sm.zm[b], b, jg0, it.j_end, lane, ig0, it.i_end,
                                                   nx, ny, nz, mi, eps2, r2c, lo, ax, ay, az, pp, sm.jacc[w]);
          }
        }
        auto fold = [&](float2& s, const float2 v) { two_sum_acc(s.x, s.y, v.x + v.y); };
#pragma unroll
        for (int r = 0; r < R; ++r) {
          fold(sm.hl[0][r][tid], ax[r]), fold(sm.hl[1][r][tid], ay[r]), fold(sm.hl[2][r][tid], az[r]);
          if (PHI) fold(sm.hl[3][r][tid], pp[r]);
        }
        __syncthreads();
        // the tile's j-sums over the CTA's warps (the pair force on j is minus that on i)
#pragma unroll
        for (int k = 0; k < LPT; ++k) {
          const int t = tid + k * T, j = jt + t;
          if (t < J && j < it.j_end) {
            float4 oxy = make_float4(0.f, 0.f, 0.f, 0.f), ozp = oxy;
            if (add) oxy = __ldcg(&oj[j].xy), ozp = __ldcg(&oj[j].zp);
            float h[4] = {oxy.x, oxy.z, ozp.x, ozp.z}, l[4] = {oxy.y, oxy.w, ozp.y, ozp.w};
#pragma unroll
            for (int c = 0; c < NCJ; ++c)
#pragma unroll
              for (int u = 0; u < W; ++u) {
                const float v = (&sm.jacc[u][c][t >> 6][(t & 63) >> 1].x)[t & 1];
                two_sum_acc(h[c], l[c], c < 3 ? -v : v);
              }
            __stcg(&oj[j].xy, make_float4(h[0], l[0], h[1], l[1]));
            __stcg(&oj[j].zp, make_float4(h[2], l[2], h[3], l[3]));
          }
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int ig = ig0 + 32 * r;
        if (ig < it.i_end) {
          const float2 a = sm.hl[0][r][tid], b = sm.hl[1][r][tid], c = sm.hl[2][r][tid];
          const float2 d = PHI ? sm.hl[NC - 1][r][tid] : make_float2(0.f, 0.f);
          oi[ig] = fpair4{make_float4(a.x, a.y, b.x, b.y), make_float4(c.x, c.y, d.x, d.y)};
        }
      }
      __syncthreads();  // the tile and the j-sums are free for the next i-tile
    }
  }
}

}  // namespace sym
}  // namespace nbody
