// Device code of the force kernels (Sec. 2 Alg. 2 step 5; Eq. 3; Plummer
// softening of Sec. 3), shared by the single-system kernels (k_force.cu)
// and the ensemble kernels (k_ensemble.cu). One work item is an i-group of
// IG active bodies against one j-chunk; *_item computes one item, *_items
// walks the items of a plan over a persistent grid.
#pragma once

#include "tsbts_internal.cuh"

namespace tsbts {

constexpr int kThreads = 128;   // threads per block
constexpr int kTileF64 = 64;    // j per shared-memory tile, FP64
constexpr int kTileMix = 512;   // j per shared-memory tile, mixed
constexpr int kStrip = 256;     // j per thread between two folds, mixed
constexpr int kLaneMinMix = 16; // fewest j per thread in a split item
constexpr int kLaneMinF64 = 8;
// Most j-splits of a tiled plan: kSplitCap, which bounds what the consumer
// reads of many bodies, and kSplitCapFew for at most kFewBodies active ones,
// whose groups leave SMs idle with 16. Of 131072 bodies, in us with 16 and
// with 64: 64 active 47.4 and 32.0, 128 69.9 and 39.3, 256 64.6 and 53.6, 512
// 94.6 and 82.3 (513, with 16: 98.9); of 20000 128 24.8 and 18.8, 512 27.0
// and 25.7.
constexpr int kSplitCap = 16;
constexpr int kSplitCapFew = 64;
constexpr int kFewBodies = 512;
constexpr int kSplitCapDirect = 128;  // most j-splits of a direct-load plan
constexpr int kDirectBatch = 4;  // j records per lane loaded in one batch
constexpr int kMixMaxGroup = 2 * kThreads;  // bodies of a tiled mixed item
constexpr int kMixMinBlocks = 3;  // register budget of the mixed kernels

// Tiled plan for n_act active bodies: over the group widths 256 .. 8 and
// over w = 1 .. 5 waves of the grid, take the largest split count S whose
// items fit w waves, and rate it by the waves its items take times the time
// of an item, in quads of j per lane. Sharing a tile among fewer bodies
// makes a quad dearer (staging, distinct shared loads: measured at 131072 j
// 1163, 1123, 1057 and 960 G interactions/s with 256, 128, 64 and 32 bodies
// per item: + 1/40 per lane of a body); an item's own cost (loading its
// bodies, combining and writing sums) counts as kItemQuads. On a grid of 456
// blocks this fills more than 95% of the last wave for nearly every count;
// one width and split count per power of two of n_act took 40 groups of 128
// bodies (5000 of 20000) at 59%, 184 us per call instead of 122.
constexpr int kItemQuads = 12;
constexpr int kTiledTries = 6 * 5;  // widths x wave counts, at most 32

__host__ __device__ inline Plan tiled_try(int k, int n_act, int n, int grid,
                                          long long part_cap, float* cost) {
  const int jg = 1 << (k % 6), w = k / 6 + 1;
  const int ig = kMixMaxGroup / jg;
  const unsigned n_g = (unsigned)(n_act + ig - 1) / ig;
  const unsigned quads = (unsigned)(n + 3) / 4;
  unsigned smax = quads / (jg * (kLaneMinMix / 4));
  const unsigned cap = n_act <= kFewBodies ? kSplitCapFew : kSplitCap;
  if (smax > cap) smax = cap;
  if ((long long)smax * 5 * n_act > part_cap)
    smax = (unsigned)(part_cap / (5LL * n_act));
  unsigned S = (unsigned)(grid * w) / n_g;
  if (S > smax) S = smax;
  if (S < 1) S = 1;
  const unsigned waves = (n_g * S + grid - 1) / grid;
  const unsigned lane = (quads + S * jg - 1) / (S * jg);
  *cost = (float)waves * ((float)lane * (1.f + 0.025f * jg) + kItemQuads);
  return Plan{ig, (int)n_g, (int)S, (int)(4 * ((quads + S - 1) / S)), 0};
}

inline Plan tiled_plan(int n_act, int n, int grid, long long part_cap) {
  Plan best{};
  float best_cost = 3e38f;
  for (int k = 0; k < kTiledTries; ++k) {
    float c;
    const Plan p = tiled_try(k, n_act, n, grid, part_cap, &c);
    if (c < best_cost) {
      best_cost = c;
      best = p;
    }
  }
  return best;
}

// the same on the device, lane k rating try k
__device__ __forceinline__ Plan tiled_plan_warp(int n_act, int n, int grid,
                                                long long part_cap) {
  const int lane = threadIdx.x & 31;
  float c;
  Plan p = tiled_try(lane < kTiledTries ? lane : 0, n_act, n, grid, part_cap,
                     &c);
  const unsigned key = (__float_as_uint(c) & ~31u) | (unsigned)lane;
  const int src = (int)(__reduce_min_sync(kFull, key) & 31u);
  p.ig = __shfl_sync(kFull, p.ig, src);
  p.n_g = __shfl_sync(kFull, p.n_g, src);
  p.S = __shfl_sync(kFull, p.S, src);
  p.chunk = __shfl_sync(kFull, p.chunk, src);
  return p;
}

template <bool kPhi = true>
__device__ __forceinline__ void write_partial(const ForceArgs& A, int n_act,
                                              int split, int k, double ax,
                                              double ay, double az, double ph,
                                              double q) {
  // a plan whose partial sums do not fit the buffer writes nothing (every
  // plan the library makes fits; this guards the buffer, not the result)
  if ((long long)(split + 1) * 5 * n_act > A.part_cap) return;
  double* p = A.part + (long long)split * 5 * n_act;
  p[0 * n_act + k] = ax;
  p[1 * n_act + k] = ay;
  p[2 * n_act + k] = az;
  if (kPhi) p[3 * n_act + k] = ph;
  p[4 * n_act + k] = q;
}

// ---------------------------------------------------------------------
// FP64, j-split: sums in any order.
// ---------------------------------------------------------------------
struct __align__(16) F64Tile {
  double x[kTileF64], y[kTileF64], z[kTileF64];
  double u[kTileF64], v[kTileF64], w[kTileF64], m[kTileF64];
};

struct F64Acc {
  double ax, ay, az, ph;
};

// 1/sqrt(x) of a normal x (relative error about 2^-22; a subnormal x, which
// no caller passes, would count as 0)
__device__ __forceinline__ float rsqrt_ftz(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 1/sqrt(s2) in FP64 for the j-split path: the FP32 reciprocal square root y
// (2^-22 relative) and one third-order step for y^-2 = s2 (Householder):
// with e = 1 - s2 y^2, y <- y + y e (1/2 + 3 e / 8), whose error is
// 5 e^3 / 16 < 2^-62. The FP64 pipe of this GPU is narrow (a warp's FP64
// instruction takes 64 cycles) and the integer pipe is idle, so the
// conversions to and from FP32 and the range test are integer operations on
// the exponent fields (the significand is cut, not rounded: another 2^-24 in
// y), which leaves five FP64 operations. s2 outside 2^-119 .. 2^119 (and
// NaN) takes the correctly rounded form.
__device__ __forceinline__ double rsqrt_f64(double s2) {
  const int hi = __double2hiint(s2), lo = __double2loint(s2);
  if ((unsigned)hi - 0x38800000u >= 0x0ee00000u)
    return __ddiv_rn(1.0, __dsqrt_rn(s2));
  const float f = __uint_as_float(
      __funnelshift_l((unsigned)lo, (unsigned)hi - 0x38000000u, 3));
  const unsigned r = __float_as_uint(rsqrt_ftz(f));
  const double y = __hiloint2double((int)((r >> 3) + 0x38000000u),
                                    (int)(r << 29));
  const double e = fma(-(s2 * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// the larger of q and x as bit patterns of doubles, where q >= 0; like
// `if (x > q) q = x`, which a NaN or a negative x leaves alone (integer
// operations: an FP64 comparison would take the FP64 pipe)
__device__ __forceinline__ unsigned long long max_bits(unsigned long long q,
                                                       double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return b <= 0x7ff0000000000000ULL && b > q ? b : q;
}

// One pair term with the reciprocal square root and fused multiply-adds
// (the sums are not in the oracle's order anyway, and each term agrees with
// the rounded definition to ~1e-16): 25 FP64 operations. The maximum of the
// criterion is taken on the bit patterns (q). With the FP64 conversions,
// range test and comparisons and two second-order steps it was 37; 5000 of
// 20000 bodies went from 7.30 to 5.85 ms.
__device__ __forceinline__ void pair_f64_fast(const F64Tile& T, int t,
                                              double xi, double yi, double zi,
                                              double ui, double vi, double wi,
                                              double eps2, F64Acc& s,
                                              unsigned long long& q) {
  const double dx = T.x[t] - xi;
  const double dy = T.y[t] - yi;
  const double dz = T.z[t] - zi;
  const double s2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2)));
  const double rinv = rsqrt_f64(s2);
  const double rinv2 = rinv * rinv;
  const double mr = T.m[t] * rinv;
  const double f = mr * rinv2;
  s.ax = fma(f, dx, s.ax);
  s.ay = fma(f, dy, s.ay);
  s.az = fma(f, dz, s.az);
  s.ph -= mr;
  const double wx = T.u[t] - ui;
  const double wy = T.v[t] - vi;
  const double wz = T.w[t] - wi;
  const double c = fma(wx, wx, fma(wy, wy, wz * wz)) * rinv2;
  q = max_bits(max_bits(q, c), f);
}

template <int IG>
__device__ void f64_item(const ForceArgs& A, int n_act, const Plan& P,
    int g, int split, F64Tile& T, double (*red)[kThreads]) {
  constexpr int JG = kThreads / IG;
  constexpr int TJ = kTileF64;
  const int t = threadIdx.x;
  const int il = t % IG, jl = t / IG;
  const double eps2 = A.eps2;
  {
    const int k = g * IG + il;
    const bool valid = k < n_act;
    const int i = valid ? A.idx[k] : -1;
    double xi = 0, yi = 0, zi = 0, ui = 0, vi = 0, wi = 0;
    if (valid) {
      xi = A.x[0][i];
      yi = A.x[1][i];
      zi = A.x[2][i];
      ui = A.w[0][i];
      vi = A.w[1][i];
      wi = A.w[2][i];
    }
    F64Acc s = {0.0, 0.0, 0.0, 0.0};
    unsigned long long qb = 0;
    const int j0 = split * P.chunk;
    const int j1 = min(A.n, j0 + P.chunk);
    for (int jt = j0; jt < j1; jt += TJ) {
      const int cnt = min(TJ, j1 - jt);
      __syncthreads();
      for (int q = t; q < cnt; q += kThreads) {
        const int j = jt + q;
        T.x[q] = A.x[0][j];
        T.y[q] = A.x[1][j];
        T.z[q] = A.x[2][j];
        T.u[q] = A.w[0][j];
        T.v[q] = A.w[1][j];
        T.w[q] = A.w[2][j];
        T.m[q] = A.m[j];
      }
      __syncthreads();
      for (int q = jl; q < cnt; q += JG) {
        if (jt + q == i) continue;
        pair_f64_fast(T, q, xi, yi, zi, ui, vi, wi, eps2, s, qb);
      }
    }
    double qm = __longlong_as_double((long long)qb);
    if constexpr (JG > 1) {
      red[0][t] = s.ax;
      red[1][t] = s.ay;
      red[2][t] = s.az;
      red[3][t] = s.ph;
      red[4][t] = qm;
      __syncthreads();
      for (int half = JG / 2; half >= 1; half >>= 1) {
        if (jl < half) {
          const int o = t + half * IG;
          for (int c = 0; c < 4; ++c) red[c][t] = __dadd_rn(red[c][t], red[c][o]);
          red[4][t] = fmax(red[4][t], red[4][o]);
        }
        __syncthreads();
      }
      if (jl == 0) {
        s.ax = red[0][t];
        s.ay = red[1][t];
        s.az = red[2][t];
        s.ph = red[3][t];
        qm = red[4][t];
      }
    }
    if (jl == 0 && valid)
      write_partial(A, n_act, split, k, s.ax, s.ay, s.az, s.ph, qm);
  }
}

// ---------------------------------------------------------------------
// FP64 with ascending-j sums (bit-identical to a sequential evaluation): a
// block takes B active bodies. The pair terms of a tile of j are formed in
// parallel and put into shared memory; the sums then add them in ascending
// j, one lane per sum. The self pair and j past the end contribute zeros (a
// sum that starts at +0 is never -0, so adding a zero leaves it unchanged);
// the potential's terms are stored negated (s - t and s + (-t) round
// alike). q is a maximum, exact in any order, and taken on the bit patterns.
//
// What bounds it: each FP64 instruction of a warp occupies its scheduler's
// FP64 pipe for 64 cycles, however many lanes it serves, so the sums of one
// j cost 64 cycles per warp that adds, and a pair term ~50 of them. Hence
//  - kOverlap (few bodies per block): all sums of the block sit in the
//    lanes of warp 0 (lane 4 b + c: body b, component c), while the other
//    three warps, on the three other pipes, form the next tile's terms: with
//    one body the block runs at the latency of the chain of n additions;
//  - otherwise every warp forms terms, then warp c adds component c with
//    one lane per body, so that up to 32 bodies share each addition.
// Measured, 129 of 4099 bodies: 159 us; one thread adding all four sums of
// one body (four instructions per j, on one pipe) took 698 us. Without kOverlap the alternative is a
// thread per body that forms and adds its terms, which does no more pairs
// per FP64 instruction and leaves most of the chip idle at these counts.
// ---------------------------------------------------------------------
constexpr int kExactOverlapBodies = 7;   // bodies per block with kOverlap
constexpr int kExactBodies = 32;         // without
constexpr int kExactTerms = 2 * 4 * kExactOverlapBodies * 97;

struct ExactSm {
  double t[kExactTerms];  // [buffer][component][body][tile j, padded by one]
  double x[6][kExactBodies];
  unsigned long long q[kExactBodies];
  int i[kExactBodies];
};
static_assert(4 * kExactBodies * 33 <= kExactTerms, "term buffer");

struct F64J {
  double x, y, z, u, v, w, m;
};

__device__ __forceinline__ F64J load_f64_j(const ForceArgs& A, int j) {
  F64J J = {};
  if (j < A.n)
    J = F64J{A.x[0][j], A.x[1][j], A.x[2][j], A.w[0][j],
             A.w[1][j], A.w[2][j], A.m[j]};
  return J;
}

// active bodies k0 .. k0 + B - 1 of the list
template <bool kOverlap>
__device__ void f64_exact_group(const ForceArgs& A, int n_act, int k0, int B,
                                ExactSm& sm) {
  constexpr int TJ = kOverlap ? 96 : 32;           // j per tile
  constexpr int TT = kOverlap ? 96 : kThreads;     // threads forming terms
  constexpr int RB = TT / TJ;                      // bodies side by side
  constexpr int NB = kOverlap ? kExactOverlapBodies : kExactBodies / RB;
  constexpr int SB = TJ + 1;                       // stride of a body's terms
  constexpr int SC = (kOverlap ? kExactOverlapBodies : kExactBodies) * SB;
  const int t = threadIdx.x, lane = t & 31;
  const double eps2 = A.eps2;
  __syncthreads();  // the previous group's use of sm is over
  if (t < B) {
    const int i = A.idx[k0 + t];
    sm.i[t] = i;
    for (int c = 0; c < 3; ++c) {
      sm.x[c][t] = A.x[c][i];
      sm.x[3 + c][t] = A.w[c][i];
    }
    sm.q[t] = 0;
  }
  __syncthreads();
  const bool forms = !kOverlap || t >= 32;
  const int tt = kOverlap ? t - 32 : t;
  const int tj = tt % TJ, tb = tt / TJ;
  // this lane's sum: body sb, component sc
  const int sb = kOverlap ? lane >> 2 : lane;
  const int sc = kOverlap ? lane & 3 : t >> 5;
  const bool adds = (!kOverlap || t < 32) && sb < B;
  double sum = 0.0;
  unsigned long long q[NB];
#pragma unroll
  for (int e = 0; e < NB; ++e) q[e] = 0;

  auto form = [&](int j, const F64J& J, double* T) {
#pragma unroll
    for (int e = 0; e < NB; ++e) {
      const int b = tb + e * RB;
      if (b >= B) break;
      double tx = 0.0, ty = 0.0, tz = 0.0, tp = 0.0;
      if (j < A.n && j != sm.i[b]) {
        const double dx = __dsub_rn(J.x, sm.x[0][b]);
        const double dy = __dsub_rn(J.y, sm.x[1][b]);
        const double dz = __dsub_rn(J.z, sm.x[2][b]);
        const double s2 = __dadd_rn(
            __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)),
                      __dmul_rn(dz, dz)),
            eps2);
        const double sq = __dsqrt_rn(s2);
        const double f = __ddiv_rn(J.m, __dmul_rn(s2, sq));
        tx = __dmul_rn(f, dx);
        ty = __dmul_rn(f, dy);
        tz = __dmul_rn(f, dz);
        tp = __ddiv_rn(J.m, sq);
        const double wx = __dsub_rn(J.u, sm.x[3][b]);
        const double wy = __dsub_rn(J.v, sm.x[4][b]);
        const double wz = __dsub_rn(J.w, sm.x[5][b]);
        const double c = __ddiv_rn(
            __dadd_rn(__dadd_rn(__dmul_rn(wx, wx), __dmul_rn(wy, wy)),
                      __dmul_rn(wz, wz)),
            s2);
        q[e] = max_bits(max_bits(q[e], c), f);
      }
      double* p = T + b * SB + tj;
      p[0] = tx;
      p[SC] = ty;
      p[2 * SC] = tz;
      p[3 * SC] = -tp;
    }
  };
  // the sums of a tile: 32 terms are fetched at once (waiting for eight at a
  // time cost 16 cycles an addition), and as many eights added as hold
  // terms; those past the end are zeros
  auto add = [&](const double* T, int cnt) {
    const double* p = T + sc * SC + sb * SB;
#pragma unroll 1
    for (int e = 0; e < cnt; e += 32) {
      double y[32];
#pragma unroll
      for (int w = 0; w < 32; ++w) y[w] = p[e + w];
#pragma unroll
      for (int o = 0; o < 32; o += 8) {
        if (e + o < cnt) {
#pragma unroll
          for (int w = 0; w < 8; ++w) sum = __dadd_rn(sum, y[o + w]);
        }
      }
    }
  };

  const int tiles = (A.n + TJ - 1) / TJ;
  F64J J = {};
  if (forms) J = load_f64_j(A, tj);
  for (int k = 0; k < tiles + (kOverlap ? 1 : 0); ++k) {
    double* T = sm.t + (kOverlap ? (k & 1) * 4 * SC : 0);
    if (forms && k < tiles) {
      // the next tile's j are on their way while this tile's terms form
      const F64J N = load_f64_j(A, (k + 1) * TJ + tj);
      form(k * TJ + tj, J, T);
      J = N;
    }
    if constexpr (kOverlap) {
      if (adds && k > 0)
        add(sm.t + ((k - 1) & 1) * 4 * SC, min(TJ, A.n - (k - 1) * TJ));
      __syncthreads();
    } else {
      __syncthreads();
      if (adds) add(T, min(TJ, A.n - k * TJ));
      __syncthreads();
    }
  }
  if (forms) {
#pragma unroll
    for (int e = 0; e < NB; ++e)
      if (tb + e * RB < B && q[e]) atomicMax(&sm.q[tb + e * RB], q[e]);
  }
  __syncthreads();
  // (a buffer too small for the sums gets none, as in write_partial)
  if (5LL * n_act > A.part_cap) return;
  if (adds) A.part[(long long)sc * n_act + k0 + sb] = sum;
  if (t < B)
    A.part[4LL * n_act + k0 + t] = __longlong_as_double((long long)sm.q[t]);
}

// bodies per block for `bodies` active bodies on a device of `sms` SMs, one
// block per SM (two chains of additions on one SM share a scheduler's FP64
// pipe: 129 blocks of a grid of two per SM took 246 us, of one per SM 170)
__device__ __forceinline__ int exact_bodies(int bodies, int sms) {
  return max(1, min(kExactBodies, (bodies + sms - 1) / sms));
}

template <int IG>
__device__ void f64_items(const ForceArgs& A, int n_act, const Plan& P,
                          F64Tile& T, double (*red)[kThreads]) {
  for (int w = blockIdx.x; w < P.n_g * P.S; w += gridDim.x)
    f64_item<IG>(A, n_act, P, w / P.S, w % P.S, T, red);
}

// ---------------------------------------------------------------------
// Mixed: FP32 pair terms on double-single relative coordinates
// d = (x_hi,j - x_hi,i) + (x_lo,j - x_lo,i); FP32 sums over kStrip j per
// thread folded into hi/lo compensated accumulators; q is an exact FP32 max.
//
// What bounds the pair loop: an interaction is 26 FMA-pipe operations, in
// packed f32x2 instructions of two pipe cycles each, so 26 pipe cycles per
// warp; and those instructions and the two maxima read about 57 registers
// per interaction, of which a scheduler reads two per cycle (packed FMAs of
// three distinct operands, or packed adds beside maxima, measure 2/3 of the
// pipe's rate), so about 28 cycles are the floor of this form.
//  - Each thread holds two bodies: a register that holds a component of j
//    and a 128-bit shared load of four of them serve twice as many
//    interactions.
//  - The reciprocal square root is the form that flushes subnormals, three
//    instructions fewer than rsqrtf: s^2 >= eps^2 is a normal float, and
//    then both give the same bits (kSafe: rsqrtf).
//  - With JG > 1, JG neighbouring lanes share two bodies and take the j
//    quads in turn; their sums are combined by shuffles.
// All 131072 bodies: 14.8 ms (1163 G interactions/s, 34 cycles each), 16.3
// ms before; the same with one body per thread: 16.1 ms.
// ---------------------------------------------------------------------
// structure of arrays: consecutive j pair up for f32x2. The tile is read
// with 16-byte shared loads, so it must start on a 16-byte boundary
// wherever the kernel places it among its other shared variables.
template <int TJ>
struct __align__(16) MixTile {
  float xh[TJ], yh[TJ], zh[TJ], m[TJ];
  float xl[TJ], yl[TJ], zl[TJ];
  float u[TJ], v[TJ], w[TJ];
};

struct MixI {
  float xh, yh, zh, xl, yl, zl, u, v, w;
};

// compensated accumulator: value = hi + lo
struct DS {
  float hi, lo;
};

__device__ __forceinline__ void ds_add(DS& a, float t) {
  const float s = __fadd_rn(a.hi, t);
  const float bb = __fsub_rn(s, a.hi);
  const float err = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)),
                              __fsub_rn(t, bb));
  a.hi = s;
  a.lo = __fadd_rn(a.lo, err);
}

__device__ __forceinline__ void ds_add(DS& a, DS b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float bb = __fsub_rn(s, a.hi);
  const float err = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)),
                              __fsub_rn(b.hi, bb));
  a.hi = s;
  a.lo = __fadd_rn(__fadd_rn(a.lo, b.lo), err);
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// packed pairs of floats (two j per instruction)
typedef unsigned long long f2;

__device__ __forceinline__ f2 pk(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1,%2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void upk(f2 x, float& a, float& b) {
  asm("mov.b64 {%0,%1}, %2;" : "=f"(a), "=f"(b) : "l"(x));
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// the j operands of two interactions, one packed pair per component
struct J2 {
  f2 xh, yh, zh, m, xl, yl, zl, u, v, w;
};

__device__ __forceinline__ ulonglong2 lds4(const float* p) {
  return *reinterpret_cast<const ulonglong2*>(p);
}

// j = t .. t + 3 (t a multiple of 4): one 128-bit shared load per component
template <int TJ>
__device__ __forceinline__ void load_j4(const MixTile<TJ>& T, int t, J2& a,
                                        J2& b) {
  const ulonglong2 xh = *reinterpret_cast<const ulonglong2*>(&T.xh[t]);
  const ulonglong2 yh = *reinterpret_cast<const ulonglong2*>(&T.yh[t]);
  const ulonglong2 zh = *reinterpret_cast<const ulonglong2*>(&T.zh[t]);
  const ulonglong2 m = *reinterpret_cast<const ulonglong2*>(&T.m[t]);
  const ulonglong2 xl = *reinterpret_cast<const ulonglong2*>(&T.xl[t]);
  const ulonglong2 yl = *reinterpret_cast<const ulonglong2*>(&T.yl[t]);
  const ulonglong2 zl = *reinterpret_cast<const ulonglong2*>(&T.zl[t]);
  const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(&T.u[t]);
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&T.v[t]);
  const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&T.w[t]);
  a = J2{xh.x, yh.x, zh.x, m.x, xl.x, yl.x, zl.x, u.x, v.x, w.x};
  b = J2{xh.y, yh.y, zh.y, m.y, xl.y, yl.y, zl.y, u.y, v.y, w.y};
}

template <bool kSafe>
__device__ __forceinline__ float rsqrt_of(float x) {
  return kSafe ? rsqrtf(x) : rsqrt_ftz(x);
}

// two interactions (j = t, t + 1) on one body, all FMA-pipe work packed.
// kSafe: any s^2 >= 0 (rsqrtf). kMask: the pair with tile index `self` is the
// body itself: its 1/s is set to 0, so it adds exact zeros and the sums
// equal those of the loop over the other j.
template <bool kPhi, bool kSafe, bool kMask, bool kCrit = true>
__device__ __forceinline__ void pair_mixed2(const f2 (&ii)[9], const J2& J,
                                            int t, f2 eps2, f2 (&s)[4],
                                            float& q, int self = -1) {
  const f2 dx = add2(sub2(J.xh, ii[0]), sub2(J.xl, ii[3]));
  const f2 dy = add2(sub2(J.yh, ii[1]), sub2(J.yl, ii[4]));
  const f2 dz = add2(sub2(J.zh, ii[2]), sub2(J.zl, ii[5]));
  const f2 s2 = fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, eps2)));
  float s0, s1;
  upk(s2, s0, s1);
  float r0 = rsqrt_of<kSafe>(s0), r1 = rsqrt_of<kSafe>(s1);
  if (kMask) {
    if (t == self) r0 = 0.f;
    if (t + 1 == self) r1 = 0.f;
  }
  const f2 rinv = pk(r0, r1);
  const f2 rinv2 = mul2(rinv, rinv);
  const f2 mr = mul2(J.m, rinv);
  const f2 mr3 = mul2(mr, rinv2);
  s[0] = fma2(mr3, dx, s[0]);
  s[1] = fma2(mr3, dy, s[1]);
  s[2] = fma2(mr3, dz, s[2]);
  if (kPhi) s[3] = add2(s[3], mr);
  if (kCrit) {
    const f2 wx = sub2(J.u, ii[6]);
    const f2 wy = sub2(J.v, ii[7]);
    const f2 wz = sub2(J.w, ii[8]);
    const f2 w2 = fma2(wx, wx, fma2(wy, wy, mul2(wz, wz)));
    const f2 c = mul2(w2, rinv2);
    float c0, c1, m0, m1;
    upk(c, c0, c1);
    upk(mr3, m0, m1);
    q = max3(max3(q, c0, m0), c1, m1);
  }
}

// x as a double, by moving its exponent and significand (the FP64 pipe,
// which a conversion would take, is 64 times narrower than the integer one)
__device__ __forceinline__ double to_double(float x) {
  const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xffu;
  if (e - 1u >= 254u) return (double)x;  // zero, subnormal, inf, NaN
  return __hiloint2double(
      (int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)),
      (int)(u << 29));
}

__device__ __forceinline__ double to_double(DS a) {
  return to_double(a.hi) + to_double(a.lo);
}

// Work item of the tiled plans: ig = 256 / JG active bodies against one
// j-chunk, JG neighbouring lanes per pair of bodies (bodies il and
// il + ig / 2 of the group). Lane jl takes the quads of j jl, jl + JG, ...
// of each tile; a tile is filled up to a whole number of quads per lane with
// massless j at a distance whose square overflows, which add exact zeros.
// A body's own j is masked: while a tile is staged the warp ORs, over its
// bodies, the positions in the lanes' quad order that hold one of them, and
// only those iterations run the masked form. Both forms round alike, so a
// body's sums do not depend on its warp-mates. kSafe: eps^2 is no normal
// float; the other iterations then take rsqrtf too. (With the masked form,
// which is not unrolled, in every iteration instead, all of 65536 bodies at
// eps = 0 took 4.41 ms, 4.14 now.)
template <int JG, bool kPhi, bool kSafe>
__device__ __forceinline__ void mixed_item(const ForceArgs& A, int n_act,
                                           const Plan& P, int g, int split,
                                           MixTile<kTileMix>& T) {
  constexpr int IG = kMixMaxGroup / JG;
  constexpr int U = 2;                  // quads per lane and loop iteration
  constexpr int kRound = 4 * JG * U;    // j of one iteration of the warp
  constexpr int kIter = kStrip / 4;     // quads per lane between two folds
  const int t = threadIdx.x;
  const int il = t / JG, jl = t % JG;
  const float far = 1e30f;
  int own[2];
  f2 ii[2][9];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int k = g * IG + r * (IG / 2) + il;
    own[r] = k < n_act ? A.idx[k] : -1;
    float4 h = {}, l = {}, v = {};
    if (own[r] >= 0) {
      h = A.jhi[own[r]];
      l = A.jlo[own[r]];
      v = A.jv[own[r]];
    }
    ii[r][0] = pk(h.x, h.x); ii[r][1] = pk(h.y, h.y); ii[r][2] = pk(h.z, h.z);
    ii[r][3] = pk(l.x, l.x); ii[r][4] = pk(l.y, l.y); ii[r][5] = pk(l.z, l.z);
    ii[r][6] = pk(v.x, v.x); ii[r][7] = pk(v.y, v.y); ii[r][8] = pk(v.z, v.z);
  }
  DS s[2][4] = {};
  float q[2] = {0.f, 0.f};
  const f2 e2 = pk(A.eps2f, A.eps2f);
  const int j0 = split * P.chunk;
  const int j1 = min(A.n, j0 + P.chunk);
  for (int jt = j0; jt < j1; jt += kTileMix) {
    const int cnt = min(kTileMix, j1 - jt);
    const int cntp = (cnt + kRound - 1) / kRound * kRound;
    __syncthreads();
#pragma unroll 2
    for (int c = t; c < cntp; c += kThreads) {
      float4 h = make_float4(far, far, far, 0.f), l = {}, v = {};
      if (c < cnt) {
        h = A.jhi[jt + c];
        l = A.jlo[jt + c];
        v = A.jv[jt + c];
      }
      T.xh[c] = h.x; T.yh[c] = h.y; T.zh[c] = h.z; T.m[c] = h.w;
      T.xl[c] = l.x; T.yl[c] = l.y; T.zl[c] = l.z;
      T.u[c] = v.x; T.v[c] = v.y; T.w[c] = v.z;
    }
    __syncthreads();
    // this tile's position of each body's own j, and its quad number
    // among this lane's (own_m < 0: not in the tile or another lane's)
    int self[2], own_m[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      self[r] = own[r] >= jt && own[r] < jt + cnt ? own[r] - jt : -1;
      own_m[r] = self[r] < 0 ? -1 : self[r] / (4 * JG);
    }
    const int iters = cntp / (4 * JG);
    for (int m0 = 0; m0 < iters; m0 += kIter) {
      unsigned lo = 0, hi = 0;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const unsigned m = (unsigned)(own_m[r] - m0);
        if (own_m[r] >= 0 && m < 32u) lo |= 1u << m;
        if (own_m[r] >= 0 && m - 32u < 32u) hi |= 1u << (m - 32u);
      }
      lo = __reduce_or_sync(kFull, lo);
      if (kTileMix / (4 * JG) > 32) hi = __reduce_or_sync(kFull, hi);
      unsigned long long mask = ((unsigned long long)hi << 32) | lo;
      const f2 z = pk(0.f, 0.f);
      f2 p[2][4] = {{z, z, z, z}, {z, z, z, z}};
      const int m1 = min(iters - m0, kIter);
      for (int m = 0; m < m1; m += U, mask >>= U) {
        const int c0 = 4 * (jl + JG * (m0 + m));
        if ((mask & ((1ULL << U) - 1)) == 0) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            J2 a, b;
            load_j4(T, c0 + 4 * JG * u, a, b);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              pair_mixed2<kPhi, kSafe, false>(ii[r], a, 0, e2, p[r], q[r]);
              pair_mixed2<kPhi, kSafe, false>(ii[r], b, 0, e2, p[r], q[r]);
            }
          }
        } else {
#pragma unroll 1
          for (int u = 0; u < U; ++u) {
            const int c = c0 + 4 * JG * u;
            J2 a, b;
            load_j4(T, c, a, b);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              pair_mixed2<kPhi, true, true>(ii[r], a, c, e2, p[r], q[r],
                                            self[r]);
              pair_mixed2<kPhi, true, true>(ii[r], b, c + 2, e2, p[r], q[r],
                                            self[r]);
            }
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
  // the JG lanes of a body pair: a butterfly, so every lane holds the sums
#pragma unroll
  for (int o = JG / 2; o >= 1; o >>= 1) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
      for (int c = 0; c < (kPhi ? 4 : 3); ++c)
        ds_add(s[r][c], DS{__shfl_xor_sync(kFull, s[r][c].hi, o),
                           __shfl_xor_sync(kFull, s[r][c].lo, o)});
      q[r] = fmaxf(q[r], __shfl_xor_sync(kFull, q[r], o));
    }
  }
  // lane r of a pair writes body r (one lane writes both when JG = 1)
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const bool second = JG > 1 ? jl == 1 : r == 1;
    if (JG > 1 && (r == 1 || jl > 1)) break;
    if ((second ? own[1] : own[0]) < 0) continue;
    DS x[4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
      x[c] = DS{second ? s[1][c].hi : s[0][c].hi,
                second ? s[1][c].lo : s[0][c].lo};
    write_partial<kPhi>(A, n_act, split, g * IG + (second ? IG / 2 : 0) + il,
                  to_double(x[0]), to_double(x[1]), to_double(x[2]),
                  -to_double(x[3]), to_double(second ? q[1] : q[0]));
  }
}

template <int JG, bool kPhi, bool kSafe>
__device__ void mixed_items(const ForceArgs& A, int n_act, const Plan& P,
                            MixTile<kTileMix>& T) {
  for (int w = blockIdx.x; w < P.n_g * P.S; w += gridDim.x)
    mixed_item<JG, kPhi, kSafe>(A, n_act, P, w / P.S, w % P.S, T);
}

// Reduce the JG j-lane partial sums of each body in a fixed-order tree in
// shared memory and write the item's partial sums.
template <int IG>
__device__ __forceinline__ void finish_mixed_item(const ForceArgs& A,
                                                  int n_act, int split, int k,
                                                  bool valid, DS sx, DS sy,
                                                  DS sz, DS sp, float q,
                                                  float (*red)[kThreads]) {
  constexpr int JG = kThreads / IG;
  const int t = threadIdx.x;
  const int jl = t / IG;
  {
    if constexpr (JG > 1) {
      red[0][t] = sx.hi; red[1][t] = sx.lo;
      red[2][t] = sy.hi; red[3][t] = sy.lo;
      red[4][t] = sz.hi; red[5][t] = sz.lo;
      red[6][t] = sp.hi; red[7][t] = sp.lo;
      red[8][t] = q;
      __syncthreads();
      for (int half = JG / 2; half >= 1; half >>= 1) {
        if (jl < half) {
          const int o = t + half * IG;
          for (int c = 0; c < 8; c += 2) {
            DS a = {red[c][t], red[c + 1][t]};
            ds_add(a, DS{red[c][o], red[c + 1][o]});
            red[c][t] = a.hi;
            red[c + 1][t] = a.lo;
          }
          red[8][t] = fmaxf(red[8][t], red[8][o]);
        }
        __syncthreads();
      }
      if (jl == 0) {
        sx = DS{red[0][t], red[1][t]};
        sy = DS{red[2][t], red[3][t]};
        sz = DS{red[4][t], red[5][t]};
        sp = DS{red[6][t], red[7][t]};
        q = red[8][t];
      }
    }
    if (jl == 0 && valid)
      write_partial(A, n_act, split, k, to_double(sx), to_double(sy),
                    to_double(sz), -to_double(sp), to_double(q));
    __syncthreads();  // red is reused by the next item
  }
}

template <bool kSafe>
__device__ __forceinline__ void pair_mixed_g(const MixI& I, const float4 h,
                                             const float4 l, const float4 vv,
                                             float eps2, float& ax, float& ay,
                                             float& az, float& ph, float& q) {
  const float dx = __fsub_rn(h.x, I.xh) + __fsub_rn(l.x, I.xl);
  const float dy = __fsub_rn(h.y, I.yh) + __fsub_rn(l.y, I.yl);
  const float dz = __fsub_rn(h.z, I.zh) + __fsub_rn(l.z, I.zl);
  const float s2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps2)));
  const float rinv = rsqrt_of<kSafe>(s2);
  const float rinv2 = rinv * rinv;
  const float mr = h.w * rinv;
  const float mr3 = mr * rinv2;
  ax = fmaf(mr3, dx, ax);
  ay = fmaf(mr3, dy, ay);
  az = fmaf(mr3, dz, az);
  ph += mr;
  const float wx = vv.x - I.u;
  const float wy = vv.y - I.v;
  const float wz = vv.z - I.w;
  const float w2 = fmaf(wx, wx, fmaf(wy, wy, wz * wz));
  q = max3(q, w2 * rinv2, mr3);
}

// The j sweep of a direct-load item: j-lane jl of a body reads
// j = j0 + jl, j0 + jl + JG, ... straight from global memory.
template <int JG, int BATCH, bool kSafe>
__device__ __forceinline__ void direct_sweep(const ForceArgs& A,
                                             const MixI& I, int i, int j0,
                                             int jl, int j1, DS (&s)[4],
                                             float& q) {
  const float eps2 = A.eps2f;
  float ax = 0, ay = 0, az = 0, ph = 0;
  auto fold = [&]() {
    ds_add(s[0], ax);
    ds_add(s[1], ay);
    ds_add(s[2], az);
    ds_add(s[3], ph);
    ax = ay = az = ph = 0.f;
  };
  int cnt = 0;
  if constexpr (BATCH == 1) {
#pragma unroll 4
    for (int j = j0 + jl; j < j1; j += JG) {
      const float4 h = A.jhi[j], l = A.jlo[j], vv = A.jv[j];
      if (j != i) pair_mixed_g<kSafe>(I, h, l, vv, eps2, ax, ay, az, ph, q);
      if (++cnt == kStrip) {
        cnt = 0;
        fold();
      }
    }
  } else {
    for (int jb = j0 + jl; jb < j1; jb += JG * BATCH) {
      float4 h[BATCH], l[BATCH], vv[BATCH];
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int j = jb + u * JG;
        if (j < j1) {
          h[u] = __ldg(A.jhi + j);
          l[u] = __ldg(A.jlo + j);
          vv[u] = __ldg(A.jv + j);
        }
      }
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int j = jb + u * JG;
        if (j < j1 && j != i)
          pair_mixed_g<kSafe>(I, h[u], l[u], vv[u], eps2, ax, ay, az, ph, q);
      }
      cnt += BATCH;
      if (cnt >= kStrip) {
        cnt = 0;
        fold();
      }
    }
  }
  fold();
}

// Narrow groups without shared-memory staging (the j records are
// L2-resident), so a small active set costs no block-wide tile loads.
// BATCH j records per lane are loaded in one batch before any is used, so
// a small item waits for a few round trips to L2, not one per j; BATCH = 1
// keeps the register budget of kernels that hold more state (ensembles).
template <int IG, int BATCH = kDirectBatch>
__device__ void mixed_direct_item(const ForceArgs& A, int n_act, const Plan& P,
    int g, int split, float (*red)[kThreads]) {
  constexpr int JG = kThreads / IG;
  const int t = threadIdx.x;
  const int il = t % IG, jl = t / IG;
  const int k = g * IG + il;
  const bool valid = k < n_act;
  const int i = valid ? A.idx[k] : -1;
  MixI I = {};
  if (valid) {
    const float4 h = A.jhi[i], l = A.jlo[i], vv = A.jv[i];
    I.xh = h.x; I.yh = h.y; I.zh = h.z;
    I.xl = l.x; I.yl = l.y; I.zl = l.z;
    I.u = vv.x; I.v = vv.y; I.w = vv.z;
  }
  DS s[4] = {};
  float q = 0.f;
  const int j0 = split * P.chunk;
  const int j1 = min(A.n, j0 + P.chunk);
  if (normal_eps2(A.eps2f))
    direct_sweep<JG, BATCH, false>(A, I, i, j0, jl, j1, s, q);
  else
    direct_sweep<JG, BATCH, true>(A, I, i, j0, jl, j1, s, q);
  finish_mixed_item<IG>(A, n_act, split, k, valid, s[0], s[1], s[2], s[3], q,
                        red);
}

template <int IG>
__device__ void mixed_items_direct(const ForceArgs& A, int n_act,
                                   const Plan& P, float (*red)[kThreads]) {
  for (int w = blockIdx.x; w < P.n_g * P.S; w += gridDim.x)
    mixed_direct_item<IG>(A, n_act, P, w / P.S, w % P.S, red);
}

}  // namespace tsbts
