// Arithmetic of the spatially ordered mixed force (force_far.cuh, k_sort.cu)
// that host code can run too.
#pragma once

#include <cstring>

#ifdef __CUDACC__
#define TSBTS_HD __host__ __device__ __forceinline__
#else
#define TSBTS_HD inline
#endif

namespace tsbts {

// x - c for x = h + l (|l| at most a unit in h's last place), rounded once:
// the remainder of h - c is exact (Knuth's two-sum) and joins l before the
// last addition. Rounded twice, as (h - c) + l, the result can be a whole
// unit off instead of half of one, and where h is cut toward zero it leans: l
// has the sign of x, and it vanishes wherever h - c is on a coarser grid than
// l. The mean error of a far pair's distance was then
// -9.8e-9 of it, and is less than 1e-10 now; the energy of 36864 bodies after
// an era of 1/8 was 5.5e-11 of it off the FP64 path's with the same block
// steps, and 1.0e-11 with one rounding (see split_round for the rest).
TSBTS_HD float about(float h, float l, float c) {
  const float t = h - c;
  const float b = t + c, a = t - b;
  const float e = (h - b) - (c + a);
  return t + (l + e);
}

// The bit pattern of one type as another of its size
template <class To, class From>
TSBTS_HD To bits_as(From x) {
  static_assert(sizeof(To) == sizeof(From), "same size");
  To y;
  memcpy(&y, &x, sizeof y);
  return y;
}

// Double-single split of x with hi rounded to nearest (ties away from zero)
// and lo the exact remainder rounded to float, with integer operations and
// one float product (the FP64 pipe, which the conversions would take, is 64
// times narrower). For |x| in 2^-70 .. 2^100 (the caller's range test);
// hi + lo is x to 2^-49.
//
// Rounded, not cut: the differences of a near pair, (h_j - h_i) + (l_j -
// l_i), round the first part, and where that drops l_j - l_i, parts cut
// toward zero leave the distance too short (3.3e-9 of it on average for
// distant pairs of a Plummer sphere; rounded ones do not lean). Far pairs
// have no such mean, and a pair's force changes by twice that difference
// whenever it crosses between the two forms: the energy of 131072 bodies
// after an era of 1/8 time units was 2.9e-11 of it off the unsorted form's
// with cut parts, 0.4e-11 with rounded ones.
TSBTS_HD void split_round(double x, float& hi, float& lo) {
  const unsigned long long b = bits_as<unsigned long long>(x);
  const int e = (int)((b >> 52) & 0x7ff);
  const unsigned sign = (unsigned)(b >> 63) << 31;
  const unsigned long long m = (b & ((1ULL << 52) - 1)) + (1ULL << 28);
  // (a carry out of the significand goes into the exponent)
  hi = bits_as<float>(sign | (((unsigned)(e - 1023 + 127) << 23) +
                              (unsigned)(m >> 29)));
  const int r = (int)(m & ((1u << 29) - 1)) - (1 << 28);
  const float scale = bits_as<float>((unsigned)(e - 1023 - 52 + 127) << 23);
  lo = bits_as<float>(bits_as<unsigned>((float)r * scale) ^ sign);
}

// Cells of the curve: 10 bits of a coordinate about the bodies' centre, mapped
// to (-1, 1) by x / (|x| + scale). The centre (the median of a sample) and the
// scale (half the mean |x| + |y| + |z| about it) are the bodies' own, so the
// order does not depend on where they are: with cells about the coordinate
// origin, a Plummer sphere of 65536 bodies had 41% far pairs 100 radii away
// from it and none 3000 radii away instead of 60% (all of 131072 bodies 13.0
// and 16.2 ms, 11.5 now, 14.7 in the unsorted form). A median, because a
// mean follows a single escaping body. (Where the origin was the centre, the
// median's own error moves the cells' edges: six spheres 11.33 ms on average
// about the origin, 11.46 about the median; of 92000 bodies 6.13 and 6.10.)
TSBTS_HD unsigned curve_cell(float x, float scale) {
  const float u = x / ((x < 0.f ? -x : x) + scale);
  const int i = (int)((u * 0.5f + 0.5f) * 1024.f);
  return (unsigned)(i < 0 ? 0 : (i > 1023 ? 1023 : i));
}

// Position along the Hilbert curve of a cell (10 bits per axis), by
// J. Skilling's transform ("Programming the Hilbert curve", AIP Conf. Proc.
// 707, 2004): undo the excess work from the top bit down, Gray-encode,
// interleave. Runs of consecutive bodies fill smaller boxes than in Morton
// order, whose jumps leave 47% of the subtiles of 131072 bodies too near for
// the cheap form, against 25%.
TSBTS_HD unsigned hilbert(unsigned x, unsigned y, unsigned z) {
  unsigned X[3] = {x, y, z};
  for (unsigned Q = 512; Q > 1; Q >>= 1) {
    const unsigned P = Q - 1;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      if (X[i] & Q) {
        X[0] ^= P;
      } else {
        const unsigned t = (X[0] ^ X[i]) & P;
        X[0] ^= t;
        X[i] ^= t;
      }
    }
  }
  X[1] ^= X[0];
  X[2] ^= X[1];
  unsigned t = 0;
  for (unsigned Q = 512; Q > 1; Q >>= 1)
    if (X[2] & Q) t ^= Q - 1;
  unsigned h = 0;
#pragma unroll
  for (int b = 9; b >= 0; --b)
#pragma unroll
    for (int i = 0; i < 3; ++i) h = h << 1 | ((X[i] ^ t) >> b & 1u);
  return h;
}

// body of the sample whose median is the centre: one of each of
// kCentreSample runs of bodies, at a place in its run that no regular
// arrangement of the bodies follows
constexpr int kCentreSample = 1024;

TSBTS_HD int centre_sample(int k, int n) {
  const int a = (int)((long long)k * n / kCentreSample);
  const int b = (int)((long long)(k + 1) * n / kCentreSample);
  return a + (b - a > 1 ? (int)(((unsigned)k * 2654435761u >> 8) %
                                (unsigned)(b - a))
                        : 0);
}

}  // namespace tsbts
