// Force kernels of the TSBTS library (Sec. 2 Alg. 2 step 5; Eq. 3; Plummer
// softening of Sec. 3): for each active body i and all j != i
//   a_i   = sum m_j d_ij / s^3,   phi_i = -sum m_j / s,
//   q_i   = max max(|v_ij|^2 / s^2, m_j / s^3),   s^2 = |d_ij|^2 + eps^2.
//
// Work decomposition (the GB300 analogue of the paper's Alg. 4 data/work
// partition). A persistent grid walks work items (i-group, j-chunk). The
// launch reads the active count from device memory and takes, on the
// device, the group width and the number of j-chunks:
//  - wide groups: the lanes sweep the j-chunk for their own bodies (data
//    partition); the mixed path holds two bodies per thread and runs two j
//    per packed f32x2 instruction;
//  - narrow groups (fewer active bodies): several lanes share each body's
//    j-chunk and their partial sums are combined in a fixed order inside the
//    block (work partition inside a block).
// The j range is further split across blocks so that the grid stays full;
// split partial sums go to a scratch buffer and are added in split order by
// the consumer. Every order is fixed, so results are deterministic.
//
// j records are staged tile by tile in shared memory with coalesced loads;
// the pair loop is FMA-pipe bound.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <iterator>
#include <map>
#include <mutex>
#include <vector>

#include "force_far.cuh"
#include "step_device.cuh"

namespace tsbts {

// Host choice of the work plan for n_act active bodies: tiled_plan in the
// mixed path; in FP64, over i-group widths 128 .. 1 and split counts,
// minimise the waves of the grid (two blocks per SM) times an item's time,
// plus the consumer's cost of reading S partial sums. Few blocks per SM, each
// with work: the FP64 pipe is saturated by one block, and of a grid of eight
// per SM the blocks with work may share SMs while others idle (1024 of 131072
// bodies ran at 11 G interactions/s, all of them at 22). 5000 of 20000
// bodies: 5.85 ms with S chosen for the waves of eight blocks per SM, 4.61 ms
// now.
Plan plan_force(int precision, int exact, int n_act, int n,
                const ForceLaunch& fl, long long part_cap) {
  Plan best = {kThreads, (n_act + kThreads - 1) / kThreads, 1, n, 0};
  // ascending-j sums have one split and take no plan (force_exact_kernel)
  if (exact || n_act <= 0) return best;
  if (precision) return tiled_plan(n_act, n, fl.grid, part_cap);
  double best_cost = 1e300;
  for (int ig = kThreads; ig >= 1; ig >>= 1) {
    if (ig > 2 * n_act && ig > 1) continue;
    const int jg = kThreads / ig;
    const long long n_g = (n_act + ig - 1) / ig;
    long long smax = n / ((long long)jg * kLaneMinF64);
    smax = std::max<long long>(1, std::min<long long>(smax, 2 * kSplitCap));
    for (int S = 1; S <= smax; ++S) {
      if (S > 1 && (long long)S * 5 * n_act > part_cap) break;
      const long long chunk = (n + S - 1) / S;
      const long long waves = (n_g * S + fl.grid - 1) / fl.grid;
      const double per_item = (double)((chunk + jg - 1) / jg) + 2.0;
      const double cost = 2 * waves * per_item + 0.3 * S;
      if (cost < best_cost) {
        best_cost = cost;
        best = Plan{ig, (int)n_g, S, (int)chunk, 0};
      }
    }
  }
  return best;
}

// The plan of a launch: fixed by the caller or from the bucket table. A
// bucket's plan was made for the bucket's largest count; a smaller count has
// fewer groups, so its split count is chosen again (tiled: tiled_plan;
// direct: as many as keep the grid full). FP64 keeps the bucket's split
// count: where that fills the grid's two blocks per SM, half the groups still
// give every SM one, which fills its FP64 pipe.
__device__ __forceinline__ Plan launch_plan(const ForceArgs& A,
                                            const PlanTable& PT, int n_act,
                                            int precision) {
  if (A.has_plan) return A.plan;
  Plan p = PT.b[plan_bucket(n_act, PT.nb)];
  if (precision && !p.direct)
    return tiled_plan_warp(n_act, A.n, gridDim.x, A.part_cap);
  p.n_g = (n_act + p.ig - 1) / p.ig;
  if (precision) {
    const int jg = kThreads / p.ig;
    int S = min((int)gridDim.x / p.n_g, kSplitCapDirect);
    S = min(S, max(1, A.n / (jg * 2)));
    while (S > p.S && (long long)S * 5 * n_act > A.part_cap) --S;
    if (S > p.S) {
      p.S = S;
      p.chunk = (((A.n + S - 1) / S) + 1) & ~1;
    }
  }
  return p;
}

// Launch prologue shared by both precisions: wait for the prediction
// kernel (programmatic dependent launch), read the active count. Returns
// false when there is nothing to do.
__device__ __forceinline__ bool force_prologue(const ForceArgs& A,
                                               int& n_act) {
  pdl_wait();
  pdl_launch_dependents();
  if (A.done && *A.done) return false;
  n_act = A.n_act_fixed >= 0 ? A.n_act_fixed : *A.n_act_ptr;
  return n_act > 0;
}

__global__ void __launch_bounds__(kThreads)
    force_fp64_kernel(const __grid_constant__ ForceArgs A,
                      const __grid_constant__ PlanTable PT) {
  int n_act = 0;
  if (!force_prologue(A, n_act)) return;
  const Plan P = launch_plan(A, PT, n_act, 0);
  if (blockIdx.x == 0 && threadIdx.x == 0 && A.nsplit_out)
    *A.nsplit_out = P.S;
  __shared__ F64Tile T;
  __shared__ double red[5][kThreads];
  switch (P.ig) {
    case 128: f64_items<128>(A, n_act, P, T, red); break;
    case 64: f64_items<64>(A, n_act, P, T, red); break;
    case 32: f64_items<32>(A, n_act, P, T, red); break;
    case 16: f64_items<16>(A, n_act, P, T, red); break;
    case 8: f64_items<8>(A, n_act, P, T, red); break;
    case 4: f64_items<4>(A, n_act, P, T, red); break;
    case 2: f64_items<2>(A, n_act, P, T, red); break;
    default: f64_items<1>(A, n_act, P, T, red); break;
  }
}

// FP64 with ascending-j sums (f64_exact_group), one block per SM
__global__ void __launch_bounds__(kThreads)
    force_exact_kernel(const __grid_constant__ ForceArgs A) {
  int n_act = 0;
  if (!force_prologue(A, n_act)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0 && A.nsplit_out) *A.nsplit_out = 1;
  __shared__ ExactSm sm;
  const int B = exact_bodies(n_act, gridDim.x);
  for (int k0 = blockIdx.x * B; k0 < n_act; k0 += gridDim.x * B) {
    const int nb = min(B, n_act - k0);
    if (B <= kExactOverlapBodies)
      f64_exact_group<true>(A, n_act, k0, nb, sm);
    else
      f64_exact_group<false>(A, n_act, k0, nb, sm);
  }
}

// kPhi: the potential is summed (26 against 25 FMA-pipe operations; the
// integrator does not read it). kSorted: bodies in spatial order, large
// active sets by far_item. kSafe: eps^2 is no normal float (never with
// kSorted).
template <bool kPhi, bool kSorted, bool kSafe>
__global__ void __launch_bounds__(kThreads, kMixMinBlocks)
    force_mixed_kernel(const __grid_constant__ ForceArgs A,
                       const __grid_constant__ PlanTable PT) {
  union Sm {
    FarSm far;
    MixTile<kTileMix> tile;
    float red[9][kThreads];
  };
  __shared__ __align__(16) unsigned char
      smem[kSorted ? sizeof(Sm)
                   : (sizeof(MixTile<kTileMix>) > sizeof(float[9][kThreads])
                          ? sizeof(MixTile<kTileMix>)
                          : sizeof(float[9][kThreads]))];
  int n_act = 0;
  if (!force_prologue(A, n_act)) return;
  if constexpr (kSorted) {
    if (n_act >= A.far_min) {
      FarSm& far = *reinterpret_cast<FarSm*>(smem);
      const int S = far_splits(n_act, A.n, gridDim.x, A.part_cap);
      if (blockIdx.x == 0 && threadIdx.x == 0 && A.nsplit_out)
        *A.nsplit_out = S;
      const int items = (n_act + 255) / 256 * S;
      if (A.amask && blockIdx.x < items) rank_setup(A, far);
      for (int w = blockIdx.x; w < items; w += gridDim.x)
        far_item<kPhi>(A, n_act, w / S, w % S, S, far);
      return;
    }
  }
  const Plan P = launch_plan(A, PT, n_act, 1);
  if (blockIdx.x == 0 && threadIdx.x == 0 && A.nsplit_out)
    *A.nsplit_out = P.S;
  // (a launch runs one form: staged tiles and the lanes' sums share memory)
  float(*red)[kThreads] = reinterpret_cast<float(*)[kThreads]>(smem);
  if (P.direct && P.ig <= 32) {
    // direct loads serve the narrow groups
    switch (P.ig) {
      case 32: mixed_items_direct<32>(A, n_act, P, red); break;
      case 16: mixed_items_direct<16>(A, n_act, P, red); break;
      case 8: mixed_items_direct<8>(A, n_act, P, red); break;
      case 4: mixed_items_direct<4>(A, n_act, P, red); break;
      case 2: mixed_items_direct<2>(A, n_act, P, red); break;
      default: mixed_items_direct<1>(A, n_act, P, red); break;
    }
    return;
  }
  MixTile<kTileMix>& T = *reinterpret_cast<MixTile<kTileMix>*>(smem);
  switch (P.ig) {
    case 256: mixed_items<1, kPhi, kSafe>(A, n_act, P, T); break;
    case 128: mixed_items<2, kPhi, kSafe>(A, n_act, P, T); break;
    case 64: mixed_items<4, kPhi, kSafe>(A, n_act, P, T); break;
    case 32: mixed_items<8, kPhi, kSafe>(A, n_act, P, T); break;
    case 16: mixed_items<16, kPhi, kSafe>(A, n_act, P, T); break;
    default: mixed_items<32, kPhi, kSafe>(A, n_act, P, T); break;
  }
}

// ---------------------------------------------------------------------
// Consumers of the partial sums, packing, launch shapes.
// ---------------------------------------------------------------------
// Sum of the S split partials of each active body into row-major a, phi, q.
// One thread per body adds its splits in order; for few bodies
// (kFewFinalize) a warp takes a body, lane 8 c + g adding splits g, g + 8,
// ... of component c, and a fixed shuffle tree adds the eight sums: an FP64
// addition takes 64 cycles, so 128 splits of one body in one thread took
// about 40 us (one active body of 131072: 61 us per call, 46 us now).
constexpr int kFewFinalize = 2048;
constexpr int kFinalizeThreads = 64;

__global__ void __launch_bounds__(kFinalizeThreads)
    force_finalize_kernel(const double* part, int S, int n_act,
                          const int* pos, double* a, double* phi, double* q) {
  const int k = blockIdx.x * kFinalizeThreads + threadIdx.x;
  if (k >= n_act) return;
  double s[4];
  for (int c = 0; c < 4; ++c) s[c] = part[(long long)c * n_act + k];
  double qq = part[4LL * n_act + k];
#pragma unroll 4
  for (int sp = 1; sp < S; ++sp) {
    const double* p = part + (long long)sp * 5 * n_act;
    for (int c = 0; c < 4; ++c)
      s[c] = __dadd_rn(s[c], p[(long long)c * n_act + k]);
    qq = fmax(qq, p[4LL * n_act + k]);
  }
  const int o = pos ? pos[k] : k;
  a[3 * (long long)o + 0] = s[0];
  a[3 * (long long)o + 1] = s[1];
  a[3 * (long long)o + 2] = s[2];
  phi[o] = s[3];
  q[o] = qq;
}

__global__ void __launch_bounds__(kFinalizeThreads)
    force_finalize_warp_kernel(const double* part, int S, int n_act,
                               double* a, double* phi, double* q) {
  const int k = (blockIdx.x * kFinalizeThreads + threadIdx.x) >> 5;
  if (k >= n_act) return;
  const int lane = threadIdx.x & 31, c = lane >> 3, g = lane & 7;
  const long long stride = 5LL * n_act;
  double m = 0.0;  // q >= 0
  for (int sp = lane; sp < S; sp += 32)
    m = fmax(m, part[sp * stride + 4LL * n_act + k]);
  const double* p = part + (long long)c * n_act + k;
  double s = g < S ? p[g * stride] : 0.0;
#pragma unroll 4
  for (int sp = g + 8; sp < S; sp += 8) s = __dadd_rn(s, p[sp * stride]);
  for (int o = 4; o >= 1; o >>= 1) s += __shfl_down_sync(kFull, s, o);
  for (int o = 16; o >= 1; o >>= 1)
    m = fmax(m, __shfl_xor_sync(kFull, m, o));
  if (g == 0) {
    if (c < 3)
      a[3 * (long long)k + c] = s;
    else
      phi[k] = s;
  }
  if (lane == 1) q[k] = m;
}

__global__ void pack_aos_kernel(int precision, int n, const double* m,
                                const double* r, const double* v, double* sx,
                                double* sy, double* sz, double* sw0,
                                double* sw1, double* sw2, double* sm,
                                float4* jhi, float4* jlo, float4* jv) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n;
       j += gridDim.x * blockDim.x) {
    const double x = r[3LL * j], y = r[3LL * j + 1], z = r[3LL * j + 2];
    const double u = v[3LL * j], vv = v[3LL * j + 1], w = v[3LL * j + 2];
    if (precision == 0) {
      sx[j] = x; sy[j] = y; sz[j] = z;
      sw0[j] = u; sw1[j] = vv; sw2[j] = w;
      sm[j] = m[j];
    } else {
      const float xh = (float)x, yh = (float)y, zh = (float)z;
      jhi[j] = make_float4(xh, yh, zh, (float)m[j]);
      jlo[j] = make_float4((float)(x - (double)xh), (float)(y - (double)yh),
                           (float)(z - (double)zh), 0.f);
      jv[j] = make_float4((float)u, (float)vv, (float)w, 0.f);
    }
  }
}

ForceLaunch force_launch_shape(int precision, int device) {
  // fixed table per device (this path allocates nothing)
  constexpr int kMaxDevices = 64;
  static std::mutex mu;
  static ForceLaunch cache[2][kMaxDevices];
  std::lock_guard<std::mutex> g(mu);
  ForceLaunch* c = cache[precision ? 1 : 0];
  const bool cached = device >= 0 && device < kMaxDevices;
  if (cached && c[device].grid > 0) return c[device];
  int sms = 0, per_sm = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if (precision)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &per_sm, force_mixed_kernel<true, false, false>, kThreads, 0);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, force_fp64_kernel,
                                                  kThreads, 0);
  if (sms < 1) sms = 1;
  if (per_sm < 1) per_sm = 1;
  ForceLaunch fl;
  fl.grid = precision ? sms * per_sm : 2 * sms;  // (plan_force)
  fl.sms = sms;

  fl.threads = kThreads;
  fl.tile_i = kThreads;
  fl.part_cap = 5LL * sms * per_sm * kThreads;
  if (cached) c[device] = fl;
  return fl;
}

long long force_partial_capacity(const ForceLaunch& fl, long long n) {
  const long long want = std::min<long long>(5LL * 2 * kSplitCap * n,
                                             1LL << 27);
  return std::max<long long>(fl.part_cap, want);
}

cudaError_t launch_force(int precision, const ForceArgs& fa,
                         const ForceLaunch& fl, cudaStream_t s,
                         const PlanTable* pt, bool pdl) {
  const PlanTable none{};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(fl.grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  if (precision) {
    auto* k = fa.no_phi ? force_mixed_kernel<false, false, false>
                        : force_mixed_kernel<true, false, false>;
    if (!normal_eps2(fa.eps2f))
      k = fa.no_phi ? force_mixed_kernel<false, false, true>
                    : force_mixed_kernel<true, false, true>;
    else if (fa.meta)
      k = fa.no_phi ? force_mixed_kernel<false, true, false>
                    : force_mixed_kernel<true, true, false>;
    return cudaLaunchKernelEx(&cfg, k, fa, pt ? *pt : none);
  }
  if (fa.exact) {
    cfg.gridDim = dim3(fl.sms);
    return cudaLaunchKernelEx(&cfg, force_exact_kernel, fa);
  }
  return cudaLaunchKernelEx(&cfg, force_fp64_kernel, fa, pt ? *pt : none);
}

// ---------------------------------------------------------------------
// Autotuner of the mixed force plans.
// ---------------------------------------------------------------------
namespace {

struct TuneKey {
  int device, n, grid;
  bool operator<(const TuneKey& o) const {
    return device != o.device ? device < o.device
           : n != o.n         ? n < o.n
                              : grid < o.grid;
  }
};

std::mutex g_tune_mu;
std::map<TuneKey, std::vector<Plan>> g_tuned;

// candidate plans for b active bodies: the tiled one (tiled_plan; its width
// and split count are chosen again for each count), and direct-load ones of
// the narrower
// groups with split counts {1, 2, 3, 4, 6, 8, ...} up to kSplitCapDirect and
// the one that fills the waves of the grid best, within the per-thread work
// floor and the partial-sum buffer: a small active set spreads over the
// whole grid and each lane waits for one batch of loads.
std::vector<Plan> candidates(int b, int n, int grid, long long part_cap) {
  static const int kS[] = {1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128};
  std::vector<Plan> out;
  out.push_back(tiled_plan(b, n, grid, part_cap));
  for (int ig = 32; ig >= 1; ig >>= 1) {
    if (ig > 2 * b && ig > 1) continue;
    const int jg = kThreads / ig;
    const int n_g = (b + ig - 1) / ig;
    long long smax = n / ((long long)jg * 2);
    smax = std::max<long long>(1, std::min<long long>(smax, kSplitCapDirect));
    std::vector<int> ss(std::begin(kS), std::end(kS));
    int best_s = 1;
    double best_fill = 0;
    for (int S = 1; S <= smax; ++S) {
      const long long items = (long long)n_g * S;
      const double fill =
          (double)items / (double)(((items + grid - 1) / grid) * grid);
      if (fill > best_fill + 1e-9) {
        best_fill = fill;
        best_s = S;
      }
    }
    ss.push_back(best_s);
    std::sort(ss.begin(), ss.end());
    ss.erase(std::unique(ss.begin(), ss.end()), ss.end());
    for (int S : ss) {
      if (S > smax) continue;
      if ((long long)S * 5 * b > part_cap) continue;
      long long chunk = (n + S - 1) / S;
      chunk = (chunk + 1) & ~1LL;
      out.push_back(Plan{ig, n_g, S, (int)chunk, 1});
    }
  }
  return out;
}

}  // namespace

const std::vector<Plan>* tuned_plans(int device, int n, int grid) {
  std::lock_guard<std::mutex> g(g_tune_mu);
  auto it = g_tuned.find(TuneKey{device, n, grid});
  return it == g_tuned.end() ? nullptr : &it->second;
}

// Time the candidate plans of every power-of-two active count up to n on
// the j records in `base` (bodies idx[0..b) active) and keep the fastest;
// an active count between two buckets takes the plan of the larger one.
// The table is cached per (device, n, grid) for the life of the process.
cudaError_t autotune_mixed_plans(int device, const ForceArgs& base,
                                 const ForceLaunch& fl, int* d_nsplit,
                                 cudaStream_t s, std::vector<Plan>* table) {
  const int n = base.n;
  if (const std::vector<Plan>* t = tuned_plans(device, n, fl.grid)) {
    *table = *t;
    return cudaSuccess;
  }
  std::vector<int> buckets;
  for (long long b = 1; b < n; b *= 2) buckets.push_back((int)b);
  buckets.push_back(n);
  // each candidate: one warm-up launch, then kReps batches of kBatch
  // back-to-back launches, each batch bracketed by events (the event clock
  // ticks in microseconds, coarser than a small launch); its time is the
  // median batch over kBatch (robust to a stray slow batch). A candidate
  // whose warm-up is over 4x the best so far is dropped.
  constexpr int kReps = 3;
  constexpr int kBatch = 8;
  cudaEvent_t ev[kReps + 1];
  cudaError_t err = cudaSuccess;
  int made = 0;
  for (; made <= kReps && err == cudaSuccess; ++made)
    err = cudaEventCreate(&ev[made]);
  if (err != cudaSuccess) made -= 1;
  std::vector<Plan> best(buckets.size());
  std::vector<float> best_t(buckets.size(), 0.f);
  for (size_t bi = 0; bi < buckets.size() && err == cudaSuccess; ++bi) {
    const int b = buckets[bi];
    float best_ms = 1e30f;
    for (const Plan& p : candidates(b, n, fl.grid, base.part_cap)) {
      ForceArgs fa = base;
      fa.n_act_fixed = b;
      fa.n_act_ptr = nullptr;
      fa.nsplit_out = d_nsplit;
      fa.done = nullptr;
      fa.plan = p;
      fa.has_plan = 1;
      // the warm-up launch, timed, sets the batch: launches of more than
      // ~0.1 ms are timed one at a time
      cudaEventRecord(ev[0], s);
      launch_force(1, fa, fl, s);
      cudaEventRecord(ev[1], s);
      err = cudaEventSynchronize(ev[1]);
      if (err != cudaSuccess) break;
      float warm = 0;
      cudaEventElapsedTime(&warm, ev[0], ev[1]);
      const int batch = warm > 0.1f ? 1 : kBatch;
      if (warm > 4.0f * best_ms) continue;  // far slower than the best
      for (int r = 0; r < kReps; ++r) {
        cudaEventRecord(ev[r], s);
        for (int q = 0; q < batch; ++q) launch_force(1, fa, fl, s);
      }
      cudaEventRecord(ev[kReps], s);
      err = cudaEventSynchronize(ev[kReps]);
      if (err != cudaSuccess) break;
      float t[kReps];
      for (int r = 0; r < kReps; ++r) cudaEventElapsedTime(&t[r], ev[r], ev[r + 1]);
      std::sort(t, t + kReps);
      const float ms = t[kReps / 2] / batch;
      if (ms < best_ms) {
        best_ms = ms;
        best[bi] = p;
      }
    }
    best_t[bi] = best_ms;
  }
  for (int k = 0; k < made; ++k) cudaEventDestroy(ev[k]);
  if (err == cudaSuccess) err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  if (std::getenv("TSBTS_PRINT_PLANS")) {
    for (size_t bi = 0; bi < buckets.size(); ++bi)
      std::fprintf(stderr,
                   "tsbts plan n=%d n_act<=%d: ig %d S %d chunk %d %s %.2f us\n",
                   n, buckets[bi], best[bi].ig, best[bi].S, best[bi].chunk,
                   best[bi].direct ? "direct" : "tiled", 1e3 * best_t[bi]);
  }
  table->assign(n + 1, Plan{kMixMaxGroup, 0, 1, n, 0});
  size_t bi = 0;
  for (int k = 1; k <= n; ++k) {
    while (buckets[bi] < k) ++bi;
    Plan p = best[bi];
    if (!p.direct) {
      (*table)[k] = tiled_plan(k, n, fl.grid, base.part_cap);
      continue;
    }
    p.n_g = (k + p.ig - 1) / p.ig;
    if ((long long)p.S * 5 * k > base.part_cap) {
      p.S = 1;
      p.chunk = (n + 1) & ~1;
    }
    (*table)[k] = p;
  }
  std::lock_guard<std::mutex> g(g_tune_mu);
  g_tuned[TuneKey{device, n, fl.grid}] = *table;
  return cudaSuccess;
}

cudaError_t launch_force_finalize(const double* part, int S, int n_act,
                                  const int* pos, double* a, double* phi,
                                  double* q, cudaStream_t s) {
  if (n_act <= 0) return cudaSuccess;
  constexpr int T = kFinalizeThreads;
  if (S > 2 && n_act <= kFewFinalize && !pos)
    force_finalize_warp_kernel<<<(32 * n_act + T - 1) / T, T, 0, s>>>(
        part, S, n_act, a, phi, q);
  else
    force_finalize_kernel<<<(unsigned)((n_act + T - 1LL) / T), T, 0, s>>>(
        part, S, n_act, pos, a, phi, q);
  return cudaGetLastError();
}

int far_splits_host(int n_act, int n, int grid, long long part_cap) {
  return far_splits(n_act, n, grid, part_cap);
}

__global__ void __launch_bounds__(256)
    pack_sorted_kernel(int n, const int* order, const double* m,
                       const double* r, const double* v, float4* jhi,
                       float4* jlo, float4* jv, float4* meta) {
  const int p = blockIdx.x * 256 + threadIdx.x;
  float4 h = {}, u = {};
  if (p < n) {
    const long long j = order[p];
    const double x = r[3 * j], y = r[3 * j + 1], z = r[3 * j + 2];
    const float xh = (float)x, yh = (float)y, zh = (float)z;
    h = make_float4(xh, yh, zh, (float)m[j]);
    u = make_float4((float)v[3 * j], (float)v[3 * j + 1],
                    (float)v[3 * j + 2], 0.f);
    jhi[p] = h;
    jlo[p] = make_float4((float)(x - (double)xh), (float)(y - (double)yh),
                         (float)(z - (double)zh), 0.f);
    jv[p] = u;
  }
  if ((p & ~31) < n)
    store_subtile(meta, p / 32, p < n, h.x, h.y, h.z, u.x, u.y, u.z, h.w);
}

cudaError_t launch_pack_sorted(int n, const int* order, const double* m,
                               const double* r, const double* v, float4* jhi,
                               float4* jlo, float4* jv, float4* meta,
                               cudaStream_t s) {
  pack_sorted_kernel<<<(n + 255) / 256, 256, 0, s>>>(n, order, m, r, v, jhi,
                                                     jlo, jv, meta);
  return cudaGetLastError();
}

cudaError_t launch_pack_aos(int precision, int n, const double* m,
                            const double* r, const double* v, double* sx,
                            double* sy, double* sz, double* sw0, double* sw1,
                            double* sw2, double* sm, float4* jhi, float4* jlo,
                            float4* jv, cudaStream_t s) {
  const int threads = 256;
  const int grid = std::min((n + threads - 1) / threads, 8192);
  pack_aos_kernel<<<grid, threads, 0, s>>>(precision, n, m, r, v, sx, sy, sz,
                                           sw0, sw1, sw2, sm, jhi, jlo, jv);
  return cudaGetLastError();
}

}  // namespace tsbts
