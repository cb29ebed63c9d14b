// Arithmetic of the spatially ordered mixed force (force_far.cuh, k_sort.cu)
// that host code can run too.
#pragma once

#ifdef __CUDACC__
#define TSBTS_HD __host__ __device__ __forceinline__
#else
#define TSBTS_HD inline
#endif

namespace tsbts {

// x - c for x = h + l (|l| at most a unit in h's last place), rounded once:
// the remainder of h - c is exact (Knuth's two-sum) and joins l before the
// last addition. Rounded twice, as (h - c) + l, the result can be a whole
// unit off instead of half of one, and it leans: h is cut toward zero in the
// integrator, so that l has the sign of x, and it vanishes wherever h - c is
// on a coarser grid than l. The mean error of a far pair's distance was
// -9.8e-9 of it, and less than 1e-10 now (double-single form: -3.3e-9); the
// energy of 36864 bodies after an era of 1/8 was 5.5e-11 of it off the FP64
// path's with the same block steps, and 1.0e-11 now (unsorted form 0.2e-11,
// the scheme's own error 1.9e-10).
TSBTS_HD float about(float h, float l, float c) {
  const float t = h - c;
  const float b = t + c, a = t - b;
  const float e = (h - b) - (c + a);
  return t + (l + e);
}

}  // namespace tsbts
