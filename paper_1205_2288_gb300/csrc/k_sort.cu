// Spatial order of bodies for the mixed force (force_far.cuh): positions along
// a Hilbert curve and a bitonic sort of 64-bit keys (curve position above,
// index below, so the order is unique and the same on every run). The sort runs once per era (or force call) on at most 2^20 keys;
// its launches, not its work, are its cost (about 30 at 2^17 keys).
#include "tsbts_kernels.cuh"

namespace tsbts {

namespace {

constexpr int kSortThreads = 1024;
constexpr int kSortLocal = 2 * kSortThreads;  // keys sorted in shared memory
constexpr int kScaleBlocks = 128;

__global__ void __launch_bounds__(256)
    sort_scale_kernel(int n, const double* x, const double* y,
                      const double* z, int stride, double* part) {
  __shared__ float sm[256];
  float s = 0.f;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += kScaleBlocks * 256) {
    const long long o = (long long)i * stride;
    s += fabsf((float)x[o]) + fabsf((float)y[o]) + fabsf((float)z[o]);
  }
  sm[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sm[threadIdx.x] += sm[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = (double)sm[0];
}

// 10 bits of a coordinate, mapped to (-1, 1) by x / (|x| + scale)
__device__ __forceinline__ unsigned cell(float x, float scale) {
  const float u = x / (fabsf(x) + scale);
  return (unsigned)min(1023, max(0, (int)((u * 0.5f + 0.5f) * 1024.f)));
}

// Position along the Hilbert curve of a cell (10 bits per axis), by
// J. Skilling's transform ("Programming the Hilbert curve", AIP Conf. Proc.
// 707, 2004): undo the excess work from the top bit down, Gray-encode,
// interleave. Runs of consecutive bodies fill smaller boxes than in Morton
// order, whose jumps leave 47% of the subtiles of 131072 bodies too near for
// the cheap form, against 25%.
__device__ __forceinline__ unsigned hilbert(unsigned x, unsigned y,
                                            unsigned z) {
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
    const unsigned m = hilbert(cell((float)x[o], scale),
                               cell((float)y[o], scale),
                               cell((float)z[o], scale));
    k = (unsigned long long)m << 32 | (unsigned)i;
  }
  key[i] = k;
}

__device__ __forceinline__ void exchange(unsigned long long& a,
                                         unsigned long long& b, bool up) {
  if ((a > b) == up) {
    const unsigned long long t = a;
    a = b;
    b = t;
  }
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
  sort_scale_kernel<<<kScaleBlocks, 256, 0, s>>>(n, x, y, z, stride, part);
  sort_keys_kernel<<<blocks(n2), 256, 0, s>>>(n, n2, x, y, z, stride, part,
                                              key);
  const int l = sort_keys(key, n2, s);
  order_kernel<<<blocks(n), 256, 0, s>>>(n, key, order, slot);
  return l + 3;
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
