// Spatial order of bodies for the mixed force (force_far.cuh): positions along
// a Hilbert curve (far_rule.h) and a bitonic sort of 64-bit keys (curve
// position above, index below, so the order is unique and the same on every
// run). The sort runs once per era (or force call) on at most 2^20 keys; its
// launches, not its work, are its cost (about 30 at 2^17 keys).
#include "far_rule.h"
#include "tsbts_kernels.cuh"

namespace tsbts {

namespace {

constexpr int kSortThreads = 1024;
constexpr int kSortLocal = 2 * kSortThreads;  // keys sorted in shared memory
constexpr int kScaleBlocks = 128;
static_assert(kScaleBlocks + 3 == kSortPart, "partial sums and centre");

__device__ __forceinline__ void exchange(unsigned long long& a,
                                         unsigned long long& b, bool up) {
  if ((a > b) == up) {
    const unsigned long long t = a;
    a = b;
    b = t;
  }
}

// the bodies' centre, into part[kScaleBlocks ..]: block a takes the median of
// coordinate a over a sample, by a bitonic sort of the bit patterns
__global__ void __launch_bounds__(kCentreSample)
    sort_centre_kernel(int n, const double* x, const double* y,
                       const double* z, int stride, double* part) {
  __shared__ unsigned long long s[kCentreSample];
  const double* p = blockIdx.x == 0 ? x : (blockIdx.x == 1 ? y : z);
  const int t = threadIdx.x, m = min(n, kCentreSample);
  unsigned long long u = ~0ULL;
  if (t < m) {
    const int i = n > kCentreSample ? centre_sample(t, n) : t;
    u = (unsigned long long)__double_as_longlong(p[(long long)i * stride]);
    u = u >> 63 ? ~u : u | 1ULL << 63;  // ordered like the doubles
  }
  s[t] = u;
  for (int k = 2; k <= kCentreSample; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      __syncthreads();
      const int o = t ^ j;
      if (o > t) exchange(s[t], s[o], (t & k) == 0);
    }
  __syncthreads();
  if (t == 0) {
    u = s[m / 2];
    const double c =
        __longlong_as_double((long long)(u >> 63 ? u & ~(1ULL << 63) : ~u));
    part[kScaleBlocks + blockIdx.x] = isfinite(c) ? c : 0.0;
  }
}

__global__ void __launch_bounds__(256)
    sort_scale_kernel(int n, const double* x, const double* y,
                      const double* z, int stride, double* part) {
  __shared__ float sm[256];
  const double cx = part[kScaleBlocks], cy = part[kScaleBlocks + 1],
               cz = part[kScaleBlocks + 2];
  float s = 0.f;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += kScaleBlocks * 256) {
    const long long o = (long long)i * stride;
    s += fabsf((float)(x[o] - cx)) + fabsf((float)(y[o] - cy)) +
         fabsf((float)(z[o] - cz));
  }
  sm[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sm[threadIdx.x] += sm[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = (double)sm[0];
}

__global__ void __launch_bounds__(256)
    sort_keys_kernel(int n, int n2, const double* x, const double* y,
                     const double* z, int stride, const double* part,
                     unsigned long long* key) {
  __shared__ float scale;
  if (threadIdx.x == 0) {
    float s = 0.f;
    for (int b = 0; b < kScaleBlocks; ++b) s += (float)part[b];
    // half the mean coordinate sum; any positive finite scale will do
    s = 0.5f * s / (float)n;
    scale = s > 1e-30f && s < 1e30f ? s : 1.f;
  }
  __syncthreads();
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n2) return;
  unsigned long long k = ~0ULL;
  if (i < n) {
    const long long o = (long long)i * stride;
    const double* c = part + kScaleBlocks;
    const unsigned m = hilbert(curve_cell((float)(x[o] - c[0]), scale),
                               curve_cell((float)(y[o] - c[1]), scale),
                               curve_cell((float)(z[o] - c[2]), scale));
    k = (unsigned long long)m << 32 | (unsigned)i;
  }
  key[i] = k;
}

// strides j_first .. 1 of the merge of size k (k0 .. k1), inside blocks of
// kSortLocal keys
__global__ void __launch_bounds__(kSortThreads)
    bitonic_local_kernel(unsigned long long* key, int k0, int k1) {
  __shared__ unsigned long long s[kSortLocal];
  const int base = blockIdx.x * kSortLocal, t = threadIdx.x;
  s[t] = key[base + t];
  s[t + kSortThreads] = key[base + t + kSortThreads];
  for (int k = k0; k <= k1; k <<= 1)
    for (int j = min(k, kSortLocal) >> 1; j > 0; j >>= 1) {
      __syncthreads();
      const int a = 2 * t - (t & (j - 1));
      exchange(s[a], s[a + j], ((base + a) & k) == 0);
    }
  __syncthreads();
  key[base + t] = s[t];
  key[base + t + kSortThreads] = s[t + kSortThreads];
}

__global__ void __launch_bounds__(256)
    bitonic_global_kernel(unsigned long long* key, int n2, int k, int j) {
  const int t = blockIdx.x * 256 + threadIdx.x;
  if (t >= n2 / 2) return;
  const int a = 2 * t - (t & (j - 1));
  unsigned long long x = key[a], y = key[a + j];
  exchange(x, y, (a & k) == 0);
  key[a] = x;
  key[a + j] = y;
}

__global__ void order_kernel(int n, const unsigned long long* key, int* order,
                             int* slot) {
  const int p = blockIdx.x * 256 + threadIdx.x;
  if (p >= n) return;
  const int i = (int)(key[p] & 0xffffffffu);
  order[p] = i;
  if (slot) slot[i] = p;
}

__global__ void list_keys_kernel(int n_act, int n2, const int* idx,
                                 const int* slot, unsigned long long* key) {
  const int k = blockIdx.x * 256 + threadIdx.x;
  if (k >= n2) return;
  key[k] = k < n_act ? (unsigned long long)slot[idx[k]] << 32 | (unsigned)k
                     : ~0ULL;
}

__global__ void list_kernel(int n_act, const unsigned long long* key,
                            int* list, int* pos) {
  const int p = blockIdx.x * 256 + threadIdx.x;
  if (p >= n_act) return;
  list[p] = (int)(key[p] >> 32);
  pos[p] = (int)(key[p] & 0xffffffffu);
}

int blocks(long long n) { return (int)((n + 255) / 256); }

int sort_keys(unsigned long long* key, int n2, cudaStream_t s) {
  int launches = 1;
  const int nb = n2 / kSortLocal;
  bitonic_local_kernel<<<nb, kSortThreads, 0, s>>>(key, 2, kSortLocal);
  for (int k = 2 * kSortLocal; k <= n2; k <<= 1) {
    for (int j = k >> 1; j >= kSortLocal; j >>= 1, ++launches)
      bitonic_global_kernel<<<blocks(n2 / 2), 256, 0, s>>>(key, n2, k, j);
    bitonic_local_kernel<<<nb, kSortThreads, 0, s>>>(key, k, k);
    ++launches;
  }
  return launches;
}

}  // namespace

int sort_capacity(long long n) {
  int n2 = kSortLocal;
  while (n2 < n) n2 <<= 1;
  return n2;
}

int launch_spatial_order(int n, const double* x, const double* y,
                         const double* z, int stride, double* part,
                         unsigned long long* key, int* order, int* slot,
                         cudaStream_t s) {
  const int n2 = sort_capacity(n);
  sort_centre_kernel<<<3, kCentreSample, 0, s>>>(n, x, y, z, stride, part);
  sort_scale_kernel<<<kScaleBlocks, 256, 0, s>>>(n, x, y, z, stride, part);
  sort_keys_kernel<<<blocks(n2), 256, 0, s>>>(n, n2, x, y, z, stride, part,
                                              key);
  const int l = sort_keys(key, n2, s);
  order_kernel<<<blocks(n), 256, 0, s>>>(n, key, order, slot);
  return l + 4;
}

void launch_sorted_list(int n_act, const int* idx, const int* slot,
                        unsigned long long* key, int* list, int* pos,
                        cudaStream_t s) {
  const int n2 = sort_capacity(n_act);
  list_keys_kernel<<<blocks(n2), 256, 0, s>>>(n_act, n2, idx, slot, key);
  sort_keys(key, n2, s);
  list_kernel<<<blocks(n_act), 256, 0, s>>>(n_act, key, list, pos);
}

}  // namespace tsbts
