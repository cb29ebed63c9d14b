// Mixed force on spatially sorted bodies (device code).
//
// With the j records along a Hilbert curve and the active bodies listed in the
// same order, a warp's 64 bodies and every 32 consecutive j (a subtile) fill
// small boxes. Most pairs of a warp and a subtile are then far apart, and
// far pairs need less work for the same result:
//  - coordinates: x'_j = x_j - c and x'_i = x_i - c, each rounded once to
//    FP32 about the centre c of the block's 256 bodies (far_rule.h; once per
//    staged j), leave one subtraction per component instead of the three of
//    the double-single difference. Where the boxes are further apart than the
//    radius rho of those bodies, |x'_j| + |x'_i| <= 3 |d|, so the rounding of
//    x'_j and x'_i is at most 3/2 units of d's last place, as the two
//    roundings of the double-single difference of far bodies are one. Neither
//    form's distances have a mean error (split_round): one that differs
//    between them would change a pair's force when it crosses over;
//  - the step criterion: q_i is a maximum, so a subtile whose largest possible
//    term, max((v_i + v_j)^2 / s^2, m_j / s^3) at the boxes' distance with the
//    largest speeds and mass in them, is below the q that every body of the
//    warp already has, needs no criterion at all (near boxes in the
//    double-single form included). A body starts from the criterion against
//    its own subtile, whose bodies are its neighbours.
// A far pair then takes 13 FMA-pipe operations and about 31 register reads
// instead of 26 and 57, a near one without the criterion 19 and 41. Of the
// pairs of all of 131072 bodies three quarters are far, of 16384 a quarter.
// All of 131072 bodies: 11.4 ms with both sorts, 14.65 in the unsorted form;
// the start of their era 269 ms, 389 before. Errors against 64 bits (relative
// 2-norms): a 2.7e-8 (3.2e-8 unsorted), phi 7e-9 (9e-9), q 1.1e-7 (1.1e-7).
#pragma once

#include "far_rule.h"
#include "force_device.cuh"

namespace tsbts {

constexpr int kSubJ = 32;                 // j per subtile
constexpr int kFarTileSubs = 16;          // subtiles per shared-memory tile
constexpr int kFarTile = kSubJ * kFarTileSubs;

struct __align__(16) FarTile {
  MixTile<kFarTile> t;
  float cx[kFarTile], cy[kFarTile], cz[kFarTile];  // relative to the centre
};

struct FarSm {
  FarTile tile;
  float box[4][6];  // per warp: the bodies' box
  int before[kThreads], warp_total[4];
};

// the box (lower, upper corner) of the valid points of a warp, to every lane
struct WarpBox {
  float lo[3], hi[3];
};

__device__ __forceinline__ unsigned order_bits(float x) {
  const unsigned u = __float_as_uint(x);
  return u & 0x80000000u ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float from_order(unsigned u) {
  return __uint_as_float(u & 0x80000000u ? u & 0x7fffffffu : ~u);
}

__device__ __forceinline__ WarpBox warp_box(bool valid, float x, float y,
                                            float z) {
  WarpBox b;
  const float p[3] = {x, y, z};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const unsigned u = order_bits(p[c]);
    b.lo[c] = from_order(__reduce_min_sync(kFull, valid ? u : ~0u));
    b.hi[c] = from_order(__reduce_max_sync(kFull, valid ? u : 0u));
  }
  return b;
}

// Summary of one subtile, written by the warp that stores its records: box
// corners, largest speed and largest mass (valid: this lane's j exists).
__device__ __forceinline__ void store_subtile(float4* meta, int sub,
                                              bool valid, float x, float y,
                                              float z, float u, float v,
                                              float w, float m) {
  const WarpBox b = warp_box(valid, x, y, z);
  const float sp = sqrtf(fmaf(u, u, fmaf(v, v, w * w)));
  const unsigned s = __reduce_max_sync(
      kFull, valid ? __float_as_uint(sp) : 0u);
  const unsigned mm = __reduce_max_sync(
      kFull, valid ? __float_as_uint(fabsf(m)) : 0u);
  if ((threadIdx.x & 31) == 0) {
    meta[2 * sub] = make_float4(b.lo[0], b.lo[1], b.lo[2],
                                __uint_as_float(s));
    meta[2 * sub + 1] = make_float4(b.hi[0], b.hi[1], b.hi[2],
                                    __uint_as_float(mm));
  }
}

// a lower bound of the distance of two intervals whose ends were rounded
__device__ __forceinline__ float box_gap(float alo, float ahi, float blo,
                                         float bhi) {
  const float up = (blo - ahi) - 2.4e-7f * (fabsf(blo) + fabsf(ahi));
  const float dn = (alo - bhi) - 2.4e-7f * (fabsf(alo) + fabsf(bhi));
  return fmaxf(0.f, fmaxf(up, dn));
}

// two interactions of a far pair of boxes without the criterion: one
// subtraction per component
template <bool kPhi>
__device__ __forceinline__ void pair_far2(const f2 (&ci)[3], f2 x, f2 y, f2 z,
                                          f2 m, f2 eps2, f2 (&s)[4]) {
  const f2 dx = sub2(x, ci[0]), dy = sub2(y, ci[1]), dz = sub2(z, ci[2]);
  const f2 s2 = fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, eps2)));
  float s0, s1;
  upk(s2, s0, s1);
  const f2 rinv = pk(rsqrt_ftz(s0), rsqrt_ftz(s1));
  const f2 mr = mul2(m, rinv);
  const f2 mr3 = mul2(mr, mul2(rinv, rinv));
  s[0] = fma2(mr3, dx, s[0]);
  s[1] = fma2(mr3, dy, s[1]);
  s[2] = fma2(mr3, dz, s[2]);
  if (kPhi) s[3] = add2(s[3], mr);
}

// Exclusive counts of active slots before each thread's share of the mask
// words, so that rank -> slot takes a search and a short walk.
__device__ __forceinline__ void rank_setup(const ForceArgs& A, FarSm& sm) {
  const int words = (A.n + 31) / 32;
  const int per = (words + kThreads - 1) / kThreads;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  int c = 0;
  for (int w = t * per; w < min(words, (t + 1) * per); ++w)
    c += __popc(A.amask[w]);
  int x = c;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sm.warp_total[wid] = x;
  __syncthreads();
  for (int w = 0; w < wid; ++w) x += sm.warp_total[w];
  sm.before[t] = x - c;
  __syncthreads();
}

// the slot of rank k (below the number of active slots)
__device__ __forceinline__ int rank_slot(const ForceArgs& A, const FarSm& sm,
                                         int k) {
  const int words = (A.n + 31) / 32;
  const int per = (words + kThreads - 1) / kThreads;
  int lo = 0, hi = kThreads - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (sm.before[mid] <= k)
      lo = mid;
    else
      hi = mid - 1;
  }
  int rem = k - sm.before[lo], w = lo * per;
  unsigned m = A.amask[w];
  for (int c = __popc(m); rem >= c && w + 1 < words; c = __popc(m)) {
    rem -= c;
    m = A.amask[++w];
  }
  for (; rem > 0; --rem) m &= m - 1;
  return w * 32 + __ffs(m) - 1;
}

// One item: bodies g * 256 .. of the sorted list against the subtiles
// split, split + S, split + 2 S, ... (strided, so that every item has its
// share of near ones). Warp w holds bodies 64 w + lane and 64 w + 32 + lane of
// the group. eps^2 is a normal float.
template <bool kPhi>
__device__ __forceinline__ void far_item(const ForceArgs& A, int n_act, int g,
                                         int split, int S, FarSm& sm) {
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const float eps2 = A.eps2f;
  const float far = 1e30f;
  int own[2], k[2];
  MixI I[2];
  float q[2] = {0.f, 0.f};
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    k[r] = g * 256 + wid * 64 + r * 32 + lane;
    own[r] = -1;
    float4 h = {}, l = {}, v = {};
    if (k[r] < n_act) {
      own[r] = A.amask ? rank_slot(A, sm, k[r]) : A.idx[k[r]];
      // (the consumer's list follows the ranks)
      if (A.amask && split == 0) A.act[k[r]] = A.order[own[r]];
      h = A.jhi[own[r]];
      l = A.jlo[own[r]];
      v = A.jv[own[r]];
    }
    I[r] = MixI{h.x, h.y, h.z, l.x, l.y, l.z, v.x, v.y, v.z};
  }
  // the criterion against each body's own subtile
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    if (own[r] < 0) continue;
    const int b = own[r] & ~(kSubJ - 1), e = min(kSubJ, A.n - b);
    float ax = 0, ay = 0, az = 0, ph = 0;
    for (int o = 0; o < e; ++o) {
      const int j = b + (own[r] + 1 + o) % kSubJ;
      if (j >= A.n || j == own[r]) continue;
      pair_mixed_g<false>(I[r], A.jhi[j], A.jlo[j], A.jv[j], eps2, ax, ay, az,
                          ph, q[r]);
    }
  }
  // boxes of the warp's bodies and of the block's, largest speed
  WarpBox wb;
  float vmax;
  {
    const WarpBox b0 = warp_box(own[0] >= 0, I[0].xh, I[0].yh, I[0].zh);
    const WarpBox b1 = warp_box(own[1] >= 0, I[1].xh, I[1].yh, I[1].zh);
    const bool any0 = __any_sync(kFull, own[0] >= 0);
    const bool any1 = __any_sync(kFull, own[1] >= 0);
    float s = 0.f;
#pragma unroll
    for (int r = 0; r < 2; ++r)
      s = fmaxf(s, sqrtf(fmaf(I[r].u, I[r].u,
                              fmaf(I[r].v, I[r].v, I[r].w * I[r].w))));
    vmax = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(s)));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      wb.lo[c] = any1 ? fminf(b0.lo[c], b1.lo[c]) : (any0 ? b0.lo[c] : far);
      wb.hi[c] = any1 ? fmaxf(b0.hi[c], b1.hi[c]) : (any0 ? b0.hi[c] : -far);
    }
  }
  __syncthreads();  // the previous item's use of sm is over
  if (lane == 0)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      sm.box[wid][c] = wb.lo[c];
      sm.box[wid][3 + c] = wb.hi[c];
    }
  __syncthreads();
  float cen[3], rho2 = 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float lo = sm.box[0][c], hi = sm.box[0][3 + c];
    for (int w = 1; w < 4; ++w) {
      lo = fminf(lo, sm.box[w][c]);
      hi = fmaxf(hi, sm.box[w][3 + c]);
    }
    cen[c] = 0.5f * (lo + hi);
    rho2 = fmaf(0.25f * (hi - lo), hi - lo, rho2);
  }
  // both bodies' operands of the two forms
  f2 ii[2][9], ci[2][3];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const float x[9] = {I[r].xh, I[r].yh, I[r].zh, I[r].xl, I[r].yl,
                        I[r].zl, I[r].u,  I[r].v,  I[r].w};
#pragma unroll
    for (int c = 0; c < 9; ++c) ii[r][c] = pk(x[c], x[c]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float d = about(x[c], x[3 + c], cen[c]);
      ci[r][c] = pk(d, d);
    }
  }
  const f2 e2 = pk(eps2, eps2);
  DS s[2][4] = {};
  const int subs = (A.n + kSubJ - 1) / kSubJ;
  const int mine = split < subs ? (subs - split + S - 1) / S : 0;
  FarTile& T = sm.tile;
  for (int m0 = 0; m0 < mine; m0 += kFarTileSubs) {
    const int ns = min(kFarTileSubs, mine - m0);
    __syncthreads();
    for (int c = t; c < ns * kSubJ; c += kThreads) {
      const int j = (split + S * (m0 + c / kSubJ)) * kSubJ + (c & (kSubJ - 1));
      float4 h = make_float4(far, far, far, 0.f), l = {}, v = {};
      if (j < A.n) {
        h = A.jhi[j];
        l = A.jlo[j];
        v = A.jv[j];
      }
      T.t.xh[c] = h.x; T.t.yh[c] = h.y; T.t.zh[c] = h.z; T.t.m[c] = h.w;
      T.t.xl[c] = l.x; T.t.yl[c] = l.y; T.t.zl[c] = l.z;
      T.t.u[c] = v.x; T.t.v[c] = v.y; T.t.w[c] = v.z;
      T.cx[c] = about(h.x, l.x, cen[0]);
      T.cy[c] = about(h.y, l.y, cen[1]);
      T.cz[c] = about(h.z, l.z, cen[2]);
    }
    __syncthreads();
    // the tile's subtiles as this warp sees them (lane e: subtile e)
    const unsigned qm = __reduce_min_sync(
        kFull, min(own[0] >= 0 ? __float_as_uint(q[0]) : ~0u,
                   own[1] >= 0 ? __float_as_uint(q[1]) : ~0u));
    bool is_far = false, no_crit = false;
    if (lane < ns) {
      const int sub = split + S * (m0 + lane);
      const float4 lo = A.meta[2 * sub], hi = A.meta[2 * sub + 1];
      const float gx = box_gap(wb.lo[0], wb.hi[0], lo.x, hi.x);
      const float gy = box_gap(wb.lo[1], wb.hi[1], lo.y, hi.y);
      const float gz = box_gap(wb.lo[2], wb.hi[2], lo.z, hi.z);
      const float d2 = 0.9999f * fmaf(gx, gx, fmaf(gy, gy, gz * gz));
      is_far = d2 > rho2;
      // (both comparisons fail where a speed or mass is no number)
      const float r2 = 1.0001f / (d2 + eps2), w = vmax + lo.w;
      const float least = __uint_as_float(qm);
      no_crit = qm != ~0u && w * w * r2 <= least &&
                hi.w * r2 * sqrtf(r2) <= least;
    }
    const unsigned plain = __ballot_sync(kFull, no_crit);
    const unsigned fars = __ballot_sync(kFull, is_far) & plain;
    unsigned selfs = 0;  // subtiles of this tile that hold one of the bodies
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int sub = own[r] >= 0 ? own[r] / kSubJ : -1;
      const int e = sub >= 0 && sub % S == split ? sub / S - m0 : -1;
      selfs |= __reduce_or_sync(kFull, e >= 0 && e < ns ? 1u << e : 0u);
    }
    // FP32 sums over one subtile, then folded: its bodies pull the same way,
    // so that longer sums (256 j as in the unsorted form) would grow with
    // each term and round 1.25 to 1.5 times as far from 64 bits
    for (int e = 0; e < ns; ++e) {
      const f2 z = pk(0.f, 0.f);
      f2 p[2][4] = {{z, z, z, z}, {z, z, z, z}};
      const int c0 = e * kSubJ;
      if (fars >> e & 1) {
#pragma unroll 2
        for (int c = c0; c < c0 + kSubJ; c += 4) {
          const ulonglong2 x = lds4(&T.cx[c]), y = lds4(&T.cy[c]),
                           zz = lds4(&T.cz[c]), m = lds4(&T.t.m[c]);
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            pair_far2<kPhi>(ci[r], x.x, y.x, zz.x, m.x, e2, p[r]);
            pair_far2<kPhi>(ci[r], x.y, y.y, zz.y, m.y, e2, p[r]);
          }
        }
      } else if ((plain & ~selfs) >> e & 1) {
#pragma unroll 2
        for (int c = c0; c < c0 + kSubJ; c += 4) {
          J2 a, b;
          load_j4(T.t, c, a, b);
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            pair_mixed2<kPhi, false, false, false>(ii[r], a, 0, e2, p[r], q[r]);
            pair_mixed2<kPhi, false, false, false>(ii[r], b, 0, e2, p[r], q[r]);
          }
        }
      } else if (selfs >> e & 1) {
        const int base = (split + S * (m0 + e)) * kSubJ - c0;
#pragma unroll 1
        for (int c = c0; c < c0 + kSubJ; c += 4) {
          J2 a, b;
          load_j4(T.t, c, a, b);
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const int self = own[r] - base;
            pair_mixed2<kPhi, true, true>(ii[r], a, c, e2, p[r], q[r], self);
            pair_mixed2<kPhi, true, true>(ii[r], b, c + 2, e2, p[r], q[r],
                                          self);
          }
        }
      } else {
#pragma unroll 2
        for (int c = c0; c < c0 + kSubJ; c += 4) {
          J2 a, b;
          load_j4(T.t, c, a, b);
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            pair_mixed2<kPhi, false, false>(ii[r], a, 0, e2, p[r], q[r]);
            pair_mixed2<kPhi, false, false>(ii[r], b, 0, e2, p[r], q[r]);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < (kPhi ? 4 : 3); ++c) {
          float a0, a1;
          upk(p[r][c], a0, a1);
          ds_add(s[r][c], a0 + a1);
        }
    }
  }
#pragma unroll
  for (int r = 0; r < 2; ++r)
    if (own[r] >= 0)
      write_partial<kPhi>(A, n_act, split, k[r], to_double(s[r][0]),
                          to_double(s[r][1]), to_double(s[r][2]),
                          -to_double(s[r][3]), to_double(q[r]));
}

// Splits of the far items: as many as fit a whole number of waves of the
// grid best (tiled_try's rule for the widest groups), at least
// kFarTileSubs subtiles each.
__host__ __device__ inline int far_splits(int n_act, int n, int grid,
                                          long long part_cap) {
  const int n_g = (n_act + 255) / 256, subs = (n + kSubJ - 1) / kSubJ;
  int smax = subs / kFarTileSubs;
  if (smax > kSplitCap) smax = kSplitCap;
  if ((long long)smax * 5 * n_act > part_cap)
    smax = (int)(part_cap / (5LL * n_act));
  if (smax < 1) smax = 1;
  int best = 1;
  float best_cost = 3e38f;
  for (int w = 1; w <= 8; ++w) {
    int S = grid * w / n_g;
    if (S > smax) S = smax;
    if (S < 1) S = 1;
    const int waves = (n_g * S + grid - 1) / grid;
    const float c = (float)waves * ((float)((subs + S - 1) / S) + 12.f);
    if (c < best_cost) {
      best_cost = c;
      best = S;
    }
  }
  return best;
}

}  // namespace tsbts
