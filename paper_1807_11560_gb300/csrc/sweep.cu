// Persistent kernel for one whole band-limited time sweep (the Heun shoot of
// Eq. 51, its tangent of Eq. 30, or the backward adjoint Jacobi sweep of
// Eqs. 53-54): every evaluation of the sweep runs in one cooperative launch, its
// two phases (trig.cuh) separated by grid-wide barriers.  On small product grids
// a phase lasts a few microseconds, so the kernel boundaries between them bound
// the sweep time.
//
// Waits are bounded: a CTA that spins longer than the limit records the failure
// in a flag the host reads (LDDMM_ETIMEOUT) and every CTA leaves at its next
// barrier.  The launch is cooperative, so all CTAs are resident.
#include "trig.cuh"

namespace lddmm {
namespace {

using namespace dev;

constexpr long long kSpinLimit = 1LL << 24;   // polls of an L2 line: well over a second

template <typename T>
struct SweepArgs {
  Plan<T> p;                  // padded product-grid plan
  const T* Lhat;
  T* T1;
  T* P1;
  const EvalDesc<T>* ev;      // device array of nev evaluations
  int nev;
  EvalGeom g;
  unsigned* bar;              // arrival counter
  double* flag;               // set to 1 when a barrier wait gives up
  long long spin_limit;       // polls before a wait gives up
  unsigned stall;             // test hook: arrivals the first barrier waits for beyond the grid
};

__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid-wide barrier on a monotonic arrival counter (zeroed before the launch):
// the k-th barrier of the launch completes when the counter reaches
// k * gridDim.x.  One atomic per CTA, then acquire loads until the target.
__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned& target, double* flag, long long limit,
                                             unsigned extra = 0) {
  __syncthreads();
  target += gridDim.x + extra;
  int ok = 1;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(count, 1u);
    long long it = 0;
    while (load_acquire(count) < target) {
      if (++it > limit) {
        *(volatile double*)flag = 1.0;
        break;
      }
    }
    if (*(volatile double*)flag != 0.0) ok = 0;
  }
  return __syncthreads_and(ok) != 0;
}

// NS: the band phase's accumulators, as its kernel launched by itself has them
template <typename T, int MODE, int PT, int NS>
__global__ void __launch_bounds__(kPhaseThreads, 1)
k_sweep(const __grid_constant__ SweepArgs<T> a) {
  constexpr int NT = kPhaseThreads;
  extern __shared__ __align__(16) unsigned char smraw[];
  // evaluation descriptors in shared memory: the previous (its epilogue), the
  // current and the next one, which is fetched while the current one runs
  __shared__ __align__(16) EvalDesc<T> sev[3];
  static_assert(sizeof(EvalDesc<T>) % sizeof(unsigned long long) == 0, "descriptor size");
  constexpr int kDescWords = (int)(sizeof(EvalDesc<T>) / sizeof(unsigned long long));
  V2<T>* sm = reinterpret_cast<V2<T>*>(smraw);
  auto fetch = [&](int ev) {
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(a.ev + ev);
    unsigned long long* dst = reinterpret_cast<unsigned long long*>(&sev[ev % 3]);
    for (int i = threadIdx.x; i < kDescWords; i += NT) dst[i] = src[i];
  };
  const Plan<T>& p = a.p;
  const int n_band = (p.k.Kq() + (1 << a.g.tqs) - 1) >> a.g.tqs, n_plane = p.g.n1 * a.g.nparts;
  unsigned target = 0;
  fetch(0);
  for (int ev = 0; ev <= a.nev; ++ev) {
    if (ev + 1 < a.nev) fetch(ev + 1);
    __syncthreads();
    const EvalDesc<T>* prev = &sev[(ev + 2) % 3];
    const EvalDesc<T>* cur = &sev[ev % 3];
    const bool more = ev < a.nev;
    const PiEpi<T>* e = ev > 0 && prev->epi.nout > 0 ? &prev->epi : nullptr;
    if (more || e != nullptr) {
      for (int i = blockIdx.x; i < n_band; i += gridDim.x) {
        band_item<T, MODE, NT, PT == 0, NS>(p, a.g.tqs, e, a.g.nparts, a.P1, more ? cur->A : nullptr,
                                             more ? cur->B : nullptr, a.T1, a.Lhat, i, sm);
        __syncthreads();
      }
    }
    if (!more) return;
    // (the test hook makes the very first barrier wait for arrivals that never come)
    if (!grid_barrier(a.bar, target, a.flag, a.spin_limit, ev == 0 ? a.stall : 0u)) return;
    for (int i = blockIdx.x; i < n_plane; i += gridDim.x) {
      if constexpr (PT == 0) plane_item_flat<T, MODE, NT>(p, a.g.ppc, a.g.nparts, a.T1, cur->slot, cur->slot2, a.P1, i, sm);
      else plane_item<T, MODE, NT, PT>(p, a.g.ppc, a.g.nparts, a.T1, cur->slot, cur->slot2, a.P1, i, sm);
      __syncthreads();
    }
    if (!grid_barrier(a.bar, target, a.flag, a.spin_limit)) return;
  }
}

template <typename T, int MODE, int PT, int NS>
cudaError_t launch_ns(const SweepArgs<T>& a, size_t smem, cudaStream_t st, int max_ctas) {
  auto kern = k_sweep<T, MODE, PT, NS>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0, dev_id = 0, sms = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kPhaseThreads, smem)) != cudaSuccess)
    return e;
  if ((e = cudaGetDevice(&dev_id)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev_id)) != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const int grid = std::max(1, std::min(per_sm * sms, max_ctas));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)kPhaseThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

template <typename T, int MODE, int PT>
cudaError_t launch_pt(const SweepArgs<T>& a, size_t smem, cudaStream_t st, int max_ctas) {
  if constexpr (PT != 0 && kSplit<T> != 1)
    if (shared_sms(a.p, a.g.tqs)) return launch_ns<T, MODE, PT, 1>(a, smem, st, max_ctas);
  return launch_ns<T, MODE, PT, kSplit<T>>(a, smem, st, max_ctas);
}

template <typename T, int MODE>
cudaError_t launch(const SweepArgs<T>& a, size_t smem, cudaStream_t st, int max_ctas) {
  if (a.p.flat) return launch_pt<T, MODE, 0>(a, smem, st, max_ctas);   // 2D
  if (a.g.ppc <= 3) return launch_pt<T, MODE, 3>(a, smem, st, max_ctas);
  if (a.g.ppc <= 5) return launch_pt<T, MODE, 5>(a, smem, st, max_ctas);
  return launch_pt<T, MODE, 9>(a, smem, st, max_ctas);
}

}  // namespace

template <typename T>
cudaError_t sweep_launch(const Plan<T>& p, PwMode mode, const EvalDesc<T>* ev, int nev, const T* Lhat, T* T1, T* P1,
                         unsigned* bar, double* flag, cudaStream_t st, int stall) {
  SweepArgs<T> a;
  a.spin_limit = stall > 0 ? (long long)stall : kSpinLimit;
  a.stall = stall > 0 ? 1u : 0u;
  a.p = p;
  a.Lhat = Lhat;
  a.T1 = T1;
  a.P1 = P1;
  a.ev = ev;
  a.nev = nev;
  a.g = p.geom[mode];
  a.bar = bar;
  a.flag = flag;
  const bool flat = p.flat;
  const size_t smem =
      std::max(band_shape(p, 1 << a.g.tqs, fields_out(mode, flat), fields_in(mode, flat)).smem,
               flat ? plane_flat_smem<T>(mode, a.g.ppc)
                    : plane_shape(p, mode_in(mode), mode_out(mode), a.g.ppc, a.g.ppc <= 3 ? 3 : (a.g.ppc <= 5 ? 5 : 9)).smem);
  const int max_ctas = std::max((p.k.Kq() + (1 << a.g.tqs) - 1) >> a.g.tqs, p.g.n1 * a.g.nparts);
  cudaError_t e = cudaMemsetAsync(bar, 0, kSweepBarWords * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  switch (mode) {
    case PW_F: return launch<T, PW_F>(a, smem, st, max_ctas);
    case PW_T: return launch<T, PW_T>(a, smem, st, max_ctas);
    case PW_TC: return launch<T, PW_TC>(a, smem, st, max_ctas);
    case PW_GT: return launch<T, PW_GT>(a, smem, st, max_ctas);
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t sweep_launch<float>(const Plan<float>&, PwMode, const EvalDesc<float>*, int, const float*, float*,
                                         float*, unsigned*, double*, cudaStream_t, int);
template cudaError_t sweep_launch<double>(const Plan<double>&, PwMode, const EvalDesc<double>*, int, const double*,
                                          double*, double*, unsigned*, double*, cudaStream_t, int);

}  // namespace lddmm
