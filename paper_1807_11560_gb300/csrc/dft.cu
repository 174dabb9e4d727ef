// Stand-alone kernels of the truncated transforms (iota and pi of Section 3.1,
// Eq. 46) and of one pseudo-spectral evaluation (Eqs. 4, 48, 49) for sm_103a;
// the bodies and the form of the transforms are in trig.cuh.
//
//   k_band        band phase of an evaluation
//   k_plane       plane phase of an evaluation
//   k_iota_band   k1 -> x1 of scalar band fields (image grid)
//   k_iota_plane  k2 -> x2, k3 -> x3 of one x1 plane of up to three fields
//   k_pi_plane    x3 -> k3, x2 -> k2 of part of one x1 plane of a grid field
//   k_pi_band     x1 -> k1 of projected image-grid planes
//   k_band_load, k_band_store   Hermitian arrays <-> band vectors
#include <atomic>
#include <utility>

#include "trig.cuh"

namespace lddmm {
namespace {

using namespace dev;

constexpr int kImgThreads = 256;
constexpr int kIotaGroup = 3;     // fields per image-plane item (one velocity)
constexpr int kIotaBandGroup = 6; // fields per k1 -> x1 item

// raises a kernel's dynamic shared memory limit once per device
template <auto Kernel>
cudaError_t allow_smem() {
  static std::atomic<unsigned long long> done{0};
  int d = 0;
  cudaError_t e = cudaGetDevice(&d);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (d & 63);
  if (done.load(std::memory_order_relaxed) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
  return e;
}

// Launch with programmatic stream serialisation: the kernel may be scheduled
// while the previous kernel of the stream still runs; its body waits in
// pdl_wait before it reads or writes what other kernels use.
template <typename... KArgs, typename... Args>
cudaError_t launch_chain(void (*kern)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  cfg.attrs = at;
  cfg.numAttrs = chain_attrs(at);
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

template <typename T>
struct BandArgs {
  Plan<T> p;
  PiEpi<T> e;
  const T *P1, *A, *B, *Lhat;
  T* T1;
  int tqs, nparts, prev;
};

// Band phase.  A chain of dependent stages (partial planes from L2, x1 -> k1, the time
// step, k1 -> x1) over a few columns: latency on small bands, shared-memory reads at
// 64^3.  Alone and cold at band 32^3: 8.3 us (tangent), 9.3 (shoot), 12.3 (backward);
// with the plane phase, one evaluation of a sweep takes 9.4 us at band 16^3, 18.7 at
// 32^3 and 161 at 64^3, where three kernels of complex half-spectrum sums took 17,
// 33-36 and 850.  MINB = 2: at most 128 registers, two CTAs per SM.
template <typename T, int MODE, bool FLAT, int MINB>
__global__ void __launch_bounds__(kPhaseThreads, MINB)
k_band(const __grid_constant__ BandArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  // 2D bands of more items than SMs (one to an SM) let the plane phase start as they end:
  // before, its small items would fill the SMs of the first wave and leave the rest idle
  if (!FLAT || gridDim.x <= kSMs) pdl_trigger();
  band_item<T, MODE, kPhaseThreads, FLAT, MINB == 1 ? kSplit<T> : 1>(
      a.p, a.tqs, a.prev ? &a.e : nullptr, a.nparts, a.P1, a.A, a.B, a.T1, a.Lhat, blockIdx.x,
      reinterpret_cast<V2<T>*>(smraw));
}

// Plane phase: bound by packed-FMA issue and shared-memory reads, about one pair read
// per one or two FMAs.  Alone and cold at band 32^3: 11.5 us (tangent), 14.3 (shoot),
// 16.7 (backward).
template <typename T, int MODE, int PT>
__global__ void __launch_bounds__(plane_threads<T>(PT), 1)
k_plane(const __grid_constant__ Plan<T> p, int ppc, int nparts, const T* T1, T* slot, T* slot2, T* P1) {
  extern __shared__ __align__(16) unsigned char smraw[];
  pdl_trigger();
  plane_item<T, MODE, plane_threads<T>(PT), PT>(p, ppc, nparts, T1, slot, slot2, P1, blockIdx.x,
                                              reinterpret_cast<V2<T>*>(smraw));
}

// The plane phase of a 2D problem: latency, and in FP64 the double pipe (a product of
// the 64^2 / 16^2 configuration, 40 evaluations: 0.98 ms; 2.5 ms with complex
// half-spectrum sums).
template <typename T, int MODE>
__global__ void __launch_bounds__(kPhaseThreads)
k_plane_flat(const __grid_constant__ Plan<T> p, int ppc, int nparts, const T* T1, T* slot, T* slot2, T* P1) {
  extern __shared__ __align__(16) unsigned char smraw[];
  pdl_trigger();
  plane_item_flat<T, MODE, kPhaseThreads>(p, ppc, nparts, T1, slot, slot2, P1, blockIdx.x,
                                          reinterpret_cast<V2<T>*>(smraw));
}

// ---- image grid ----------------------------------------------------------------
constexpr int kChunk = 32;        // folded x1 points per twiddle chunk
constexpr int kIotaPT = 8;        // row pairs per thread of k2 -> x2

// k1 -> x1 of up to six fields for 2^tqs quads of columns, kChunk points at a time: bound
// by its writes to L2 (17 us for the 33 fields of 11 velocities, 160 planes, band 32^3).
template <typename T>
__global__ void __launch_bounds__(kImgThreads)
k_iota_band(const __grid_constant__ Plan<T> p, const __grid_constant__ IotaList<T> d, int tqs, T* T1) {
  extern __shared__ __align__(16) unsigned char smraw[];
  V2<T>* sG = reinterpret_cast<V2<T>*>(smraw);             // [NF][H1][PC]
  const int PC = 4 << tqs, H1 = p.k.H1, q0 = blockIdx.x << tqs, nq = min(1 << tqs, p.k.Kq() - q0);
  const int f0 = blockIdx.y * kIotaBandGroup, NF = min(kIotaBandGroup, d.nf - f0), ntp = up8(p.NT1);
  V2<T>* sF = sG + up2(kIotaBandGroup * H1 * PC);          // [H1][kChunk]
  const V2<T>* tab = reinterpret_cast<const V2<T>*>(p.e1f);
  pdl_trigger();
  pdl_wait();
  for (int it = threadIdx.x; it < NF * H1 * PC; it += kImgThreads) {
    const int col = it & (PC - 1), r = it >> (tqs + 2);
    const int f = r / H1, h = r - f * H1;
    if (col < 4 * nq)
      sG[it] = reinterpret_cast<const V2<T>*>(d.src[f0 + f])[((long long)(q0 + (col >> 2)) * H1 + h) * 4 + (col & 3)];
  }
  for (int t0 = 0; t0 < p.NT1; t0 += kChunk) {
    const int nt = min(kChunk, p.NT1 - t0);
    if (t0 > 0) __syncthreads();
    for (int i = threadIdx.x; i < H1 * kChunk; i += kImgThreads) {
      const int h = i / kChunk, t = i - h * kChunk;
      sF[i] = t0 + t < ntp ? tab[(long long)h * ntp + t0 + t] : zero2<T>();
    }
    __syncthreads();
    band_to_planes<T, kImgThreads, false>(p, sG, sF, NF, f0, d.nf, q0, nq, tqs, t0, nt, kChunk, T1);
  }
}

// iota of up to three fields on `ppi` row pairs of one x1 plane (odd G3; even ones take
// k_iota_plane_even).  k3 -> x3 costs K3/2 products per point and dominates: a lane owns TL points t (and their
// partners G3 - t) of RB rows, so a row's coefficients are read once per warp
// (broadcast) and a twiddle once per RB rows.  Packed FMAs and shared reads bind it:
// with k_iota_band 324 us for 33 fields of 160x192x161 at band 32^3 (247 for 160x192x160
// in the even kernel).
template <typename T, int TL, int RB>
__global__ void __launch_bounds__(kImgThreads)
k_iota_plane(const __grid_constant__ Plan<T> p, const __grid_constant__ IotaList<T> d, int ppi, const T* T1) {
  extern __shared__ __align__(16) unsigned char smraw[];
  V2<T>* sm = reinterpret_cast<V2<T>*>(smraw);
  const int f0 = blockIdx.y * kIotaGroup, NF = min(kIotaGroup, d.nf - f0), x1 = blockIdx.z;
  const int t0 = blockIdx.x * ppi, np = min(ppi, p.NT2 - t0);
  const PlaneShape<T> s = plane_shape(p, kIotaGroup, 0, ppi, kIotaPT);
  const int R = s.R, K3e = p.K3e, K3s = s.K3s, NT3 = p.NT3, G2 = p.g.n2, G3 = p.g.n3;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  V2<T>* S1 = sm + s.off_s;
  pdl_trigger();
  plane_tables<T, kImgThreads, kIotaPT>(p, s, t0, np, true, false, sm);
  pdl_wait();
  __syncthreads();
  rows_from_band<T, kImgThreads, kIotaGroup, kIotaPT>(p, T1 + ((long long)x1 * d.nf + f0) * p.k.Kq() * 4, NF, np, s,
                                                      sm + s.off_2f, S1);
  __syncthreads();
  const int ntb = (NT3 + 32 * TL - 1) / (32 * TL), nrb = (2 * np + RB - 1) / RB;
  for (int it = warp; it < NF * nrb * ntb; it += kImgThreads / 32) {
    const int tb = it % ntb, r = it / ntb;
    const int row0 = (r % nrb) * RB, f = r / nrb;
    V2<T> acc[RB][TL];
#pragma unroll
    for (int i = 0; i < RB; ++i)
#pragma unroll
      for (int j = 0; j < TL; ++j) acc[i][j] = zero2<T>();
    int tt[TL], rr[RB];
#pragma unroll
    for (int j = 0; j < TL; ++j) tt[j] = min(tb * 32 * TL + 32 * j + lane, NT3 - 1);
#pragma unroll
    for (int i = 0; i < RB; ++i) rr[i] = (f * R + min(row0 + i, 2 * np - 1)) * K3s;   // past the item: its last row
    const V2<T>* w = sm;
#pragma unroll 2
    for (int b = 0; b < K3e; b += 2, w += 2 * NT3) {
      V2<T> w0[TL], w1[TL];
#pragma unroll
      for (int j = 0; j < TL; ++j) {
        w0[j] = w[tt[j]];
        w1[j] = w[NT3 + tt[j]];
      }
#pragma unroll
      for (int i = 0; i < RB; ++i) {
        V2<T> a0, a1;
        ld2(S1 + rr[i] + b, a0, a1);
#pragma unroll
        for (int j = 0; j < TL; ++j) acc[i][j] = fma2(a1, w1[j], fma2(a0, w0[j], acc[i][j]));
      }
    }
    // rows come in pairs x2 = u, G2 - u (row0 is even): two row pointers that walk
    // towards each other, the points of a lane at fixed distances from them
    static_assert(RB % 2 == 0, "row pairs");
    bool ok[TL], two[TL];
#pragma unroll
    for (int j = 0; j < TL; ++j) {
      const int t = tb * 32 * TL + 32 * j + lane;
      ok[j] = t < NT3;
      two[j] = ok[j] && t > 0 && 2 * t != G3;
    }
    const int u0 = t0 + (row0 >> 1), first = tb * 32 * TL + lane;
    T* ra = d.dst[f0 + f] + ((long long)x1 * G2 + u0) * G3;
    T* rb = d.dst[f0 + f] + ((long long)x1 * G2 + G2 - u0) * G3;
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const int u = u0 + i / 2;
      const bool live = row0 + i < 2 * np && !((i & 1) && (u == 0 || 2 * u == G2));
      T* up = ((i & 1) ? rb : ra) + first;
      T* dn = ((i & 1) ? rb : ra) + (G3 - first);
#pragma unroll
      for (int j = 0; j < TL; ++j) {
        T E, O;
        un2(acc[i][j], E, O);
        if (live && ok[j]) up[32 * j] = E + O;
        if (live && two[j]) dn[-32 * j] = E - O;
      }
      if (i & 1) {
        ra += G3;
        rb -= G3;
      }
    }
  }
}

// The same for even G3: the sums over even and odd k3 kept apart give four points,
// f at G3/2 -+ t from their differences, so t runs to G3/4 and the products halve.
// A half warp takes the rows x2 = u of RB row pairs and the other half their partners
// G2 - u, its 16 lanes TL points each: per two k3 a lane reads RB + TL pairs of
// coefficients and twiddles for 2 RB TL packed FMAs, and stores runs of 64 bytes.
// 128 registers, so that two CTAs share an SM and one's stores and k2 -> x2 overlap
// the other's sums.  33 fields of 160x192x160, band 32^3 (649 MB written): 230 us, 306
// in k_iota_plane, 327 with tiles of 5 pairs and one CTA per SM, 248 with 80 registers
// and three.
template <typename T, int TL, int RB>
__global__ void __launch_bounds__(kImgThreads, sizeof(T) == 4 ? 2 : 1)
k_iota_plane_even(const __grid_constant__ Plan<T> p, const __grid_constant__ IotaList<T> d, int ppi, const T* T1) {
  extern __shared__ __align__(16) unsigned char smraw[];
  V2<T>* sm = reinterpret_cast<V2<T>*>(smraw);
  const int f0 = blockIdx.y * kIotaGroup, NF = min(kIotaGroup, d.nf - f0), x1 = blockIdx.z;
  const int t0 = blockIdx.x * ppi, np = min(ppi, p.NT2 - t0);
  const PlaneShape<T> s = plane_shape(p, kIotaGroup, 0, ppi, kIotaPT);
  const int R = s.R, K3e = p.K3e, K3s = s.K3s, NT3 = p.NT3, G2 = p.g.n2, G3 = p.g.n3, NQ = G3 / 4 + 1;
  const int warp = threadIdx.x >> 5, side = (threadIdx.x >> 4) & 1, lane = threadIdx.x & 15;
  V2<T>* S1 = sm + s.off_s;
  pdl_trigger();
  plane_tables<T, kImgThreads, kIotaPT>(p, s, t0, np, true, false, sm);
  pdl_wait();
  __syncthreads();
  rows_from_band<T, kImgThreads, kIotaGroup, kIotaPT>(p, T1 + ((long long)x1 * d.nf + f0) * p.k.Kq() * 4, NF, np, s,
                                                      sm + s.off_2f, S1);
  __syncthreads();
  const int ntb = (NQ + 16 * TL - 1) / (16 * TL), nrb = (np + RB - 1) / RB;
  for (int it = warp; it < NF * nrb * ntb; it += kImgThreads / 32) {
    const int tb = it % ntb, r = it / ntb;
    const int pr0 = (r % nrb) * RB, f = r / nrb, first = tb * 16 * TL + lane;
    V2<T> ev[RB][TL], od[RB][TL];
    int tt[TL], rr[RB];
#pragma unroll
    for (int j = 0; j < TL; ++j) tt[j] = min(first + 16 * j, NQ - 1);
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      rr[i] = (f * R + 2 * min(pr0 + i, np - 1) + side) * K3s;   // past the item: its last pair
#pragma unroll
      for (int j = 0; j < TL; ++j) ev[i][j] = od[i][j] = zero2<T>();
    }
    const V2<T>* w = sm;
#pragma unroll 2
    for (int b = 0; b < K3e; b += 2, w += 2 * NT3) {
      V2<T> w0[TL], w1[TL];
#pragma unroll
      for (int j = 0; j < TL; ++j) {
        w0[j] = w[tt[j]];
        w1[j] = w[NT3 + tt[j]];
      }
#pragma unroll
      for (int i = 0; i < RB; ++i) {
        V2<T> a0, a1;
        ld2(S1 + rr[i] + b, a0, a1);
#pragma unroll
        for (int j = 0; j < TL; ++j) {
          ev[i][j] = fma2(a0, w0[j], ev[i][j]);
          od[i][j] = fma2(a1, w1[j], od[i][j]);
        }
      }
    }
    const int u0 = t0 + pr0;
    T* row = d.dst[f0 + f] + ((long long)x1 * G2 + (side ? G2 - u0 : u0)) * G3;
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const int u = u0 + i;
      const bool live = pr0 + i < np && !(side && (u == 0 || 2 * u == G2));
#pragma unroll
      for (int j = 0; j < TL; ++j) {
        const int t = first + 16 * j;
        T e0, o0, e1, o1;
        un2(ev[i][j], e0, o0);
        un2(od[i][j], e1, o1);
        const T E = e0 + e1, O = o0 + o1, D = e0 - e1, Q = o1 - o0;
        if (live && t < NQ) {
          row[t] = E + O;
          if (t > 0) row[G3 - t] = E - O;
          if (4 * t != G3) {
            row[G3 / 2 - t] = D + Q;
            if (t > 0) row[G3 / 2 + t] = D - Q;
          }
        }
      }
      row += side ? -G3 : G3;
    }
  }
}

// the projected field (PiKind) at a point, formed as the rows are folded
template <typename T, int KIND>
__device__ __forceinline__ T pi_source(const T* __restrict__ fld, const PiField<T>& s, const Dims& g, int f, int x1,
                                       int x2, int x3) {
  const long long at = ((long long)x1 * g.n2 + x2) * g.n3 + x3;
  if (KIND == PI_FIELD) return fld[at];
  const int n = f == 0 ? g.n1 : (f == 1 ? g.n2 : g.n3), x = f == 0 ? x1 : (f == 1 ? x2 : x3);
  const long long st = f == 0 ? (long long)g.n2 * g.n3 : (f == 1 ? g.n3 : 1);
  const long long up = at + (x + 1 == n ? (1 - n) : 1) * st, dn = at + (x == 0 ? n - 1 : -1) * st;
  const T h = T(0.5) * T(n);
  const T dm = (s.m[up] - s.m[dn]) * h;
  if (KIND == PI_RESIDUAL) return s.c * (s.m[at] - s.y[at]) * dm;
  if (KIND == PI_INCREMENT) return s.c * s.y[at] * dm;
  return s.c * (s.dm[at] * dm + (s.m[at] - s.y[at]) * ((s.dm[up] - s.dm[dn]) * h));
}

// the np row pairs from t0 of plane x1 of field f: folded along x3 into shared memory,
// x3 -> k3, then x2 -> k2 into (add: onto) the partial plane out
template <typename T, int KIND>
__device__ __forceinline__ void pi_plane_part(const Plan<T>& p, const PiField<T>& src, const PlaneShape<T>& s, int ppi,
                                              int f, int x1, int t0, int np, V2<T>* sm, T* out, bool add) {
  const int NT3 = p.NT3, NT3e = p.NT3e, G2 = p.g.n2, G3 = p.g.n3;
  V2<T>*Z = sm + s.off_s, *sP = sm + s.off_p;
  const T* fld = src.f[f];
#pragma unroll 4
  for (int it = threadIdx.x; it < 2 * np * NT3; it += kImgThreads) {
    const int row = fdiv(it, p.dNT3), t = it - row * NT3, u = t0 + (row >> 1);
    const bool live = !((row & 1) && (u == 0 || 2 * u == G2)), two = t > 0 && 2 * t != G3;
    const int x2 = (row & 1) && live ? G2 - u : u;
    const T a = pi_source<T, KIND>(fld, src, p.g, f, x1, x2, t);
    const T b = pi_source<T, KIND>(fld, src, p.g, f, x1, x2, two ? G3 - t : t);
    V2<T>* o = sP + row * NT3e + t;
    *o = two ? mk2(a + b, a - b) : mk2(a, T(0));
    if (t == NT3 - 1 && NT3e > NT3) o[1] = zero2<T>();
  }
  __syncthreads();
  rows_to_k3<T, kImgThreads, 1, 1, kSplit<T>>(p, sP, t0, ppi, np, sm + s.off_3b, Z);
  __syncthreads();
  band_from_rows<T, kImgThreads, 1, 2, kSplit<T>>(p, Z, ppi, np, sm + s.off_2b, out, add);
}

// pi of `ppi` row pairs of one x1 plane of one field.  The row loads (six
// neighbours a point for the terminal fields) and the packed FMAs bind it: 63-79 us for
// three terminal fields of 160x192x160, band 32^3, where a pass that formed the fields
// (25 us) and the transform's plane kernels (95 us) ran before.
template <typename T, int KIND>
__global__ void __launch_bounds__(kImgThreads)
k_pi_plane(const __grid_constant__ Plan<T> p, const __grid_constant__ PiField<T> src, int ppi, T* __restrict__ P1) {
  extern __shared__ __align__(16) unsigned char smraw[];
  V2<T>* sm = reinterpret_cast<V2<T>*>(smraw);
  const int f = blockIdx.y, x1 = blockIdx.z, t0 = blockIdx.x * ppi, np = min(ppi, p.NT2 - t0);
  const PlaneShape<T> s = plane_shape(p, 0, 1, ppi, 1);
  pdl_trigger();
  plane_tables<T, kImgThreads, 1>(p, s, t0, np, false, true, sm);
  pdl_wait();
  T* out = P1 + (((long long)x1 * gridDim.x + blockIdx.x) * gridDim.y + f) * p.k.Kq() * 4;
  pi_plane_part<T, KIND>(p, src, s, ppi, f, x1, t0, np, sm, out, false);
}
// the same for `reps` times ppi row pairs one after another, where a partial plane of each
// would take too much scratch (pi_split)
template <typename T, int KIND>
__global__ void __launch_bounds__(kImgThreads)
k_pi_plane_seq(const __grid_constant__ Plan<T> p, const __grid_constant__ PiField<T> src, int ppi, int reps,
               T* __restrict__ P1) {
  extern __shared__ __align__(16) unsigned char smraw[];
  V2<T>* sm = reinterpret_cast<V2<T>*>(smraw);
  const int f = blockIdx.y, x1 = blockIdx.z, first = blockIdx.x * reps * ppi, end = min(first + reps * ppi, p.NT2);
  const PlaneShape<T> s = plane_shape(p, 0, 1, ppi, 1);
  T* out = P1 + (((long long)x1 * gridDim.x + blockIdx.x) * gridDim.y + f) * p.k.Kq() * 4;
  pdl_trigger();
  pdl_wait();
  for (int t0 = first; t0 < end; t0 += ppi) {
    const int np = min(ppi, end - t0);
    if (t0 > first) __syncthreads();
    plane_tables<T, kImgThreads, 1>(p, s, t0, np, false, true, sm);
    pi_plane_part<T, KIND>(p, src, s, ppi, f, x1, t0, np, sm, out, t0 > first);
  }
}

// the two plane steps of a 2D image: one output per thread.  k_pi_plane_flat takes part of
// one plane and forms its folded points once, in shared memory: a thread that formed them
// for itself was bound by that (FP64 terminal fields of 300 x 4096, band 64^2: 2.2 ms; 0.42).
template <typename T>
__global__ void __launch_bounds__(kImgThreads)
k_iota_plane_flat(const __grid_constant__ Plan<T> p, const __grid_constant__ IotaList<T> d, const T* T1) {
  const int K2h = p.k.K2h, NT2 = p.NT2, G2 = p.g.n2, t = blockIdx.x * kImgThreads + threadIdx.x, f = blockIdx.y,
            x1 = blockIdx.z;
  pdl_trigger();
  pdl_wait();
  if (t >= NT2) return;
  const T* v = T1 + ((long long)x1 * d.nf + f) * K2h * 4;
  const V2<T>* w = reinterpret_cast<const V2<T>*>(p.e2f) + t;
  V2<T> acc = zero2<T>();
#pragma unroll 8
  for (int a = 0; a < K2h; ++a) acc = fma2(ldq(v + 4 * a).c, w[(long long)a * NT2], acc);
  T E, O;
  un2(acc, E, O);
  T* o = d.dst[f] + (long long)x1 * G2;
  o[t] = E + O;
  if (t > 0 && 2 * t != G2) o[G2 - t] = E - O;
}
template <typename T, int KIND>
__global__ void __launch_bounds__(kImgThreads)
k_pi_plane_flat(const __grid_constant__ Plan<T> p, const __grid_constant__ PiField<T> src, int ppi,
                T* __restrict__ P1) {
  const int K2h = p.k.K2h, K2p = up8(K2h), G2 = p.g.n2, f = blockIdx.y, x1 = blockIdx.z;
  const int t0 = blockIdx.x * ppi, t1 = min(t0 + ppi, p.NT2);
  pdl_trigger();
  pdl_wait();
  const T* fld = src.f[f];
  __shared__ V2<T> sZ[kImgThreads];                        // folded points, each formed once
  const int a = threadIdx.x;                               // K_2 <= 512: a frequency per thread
  V2<T> acc = zero2<T>();
  for (int c0 = t0; c0 < t1; c0 += kImgThreads) {
    const int n = min(kImgThreads, t1 - c0), t = c0 + a;
    if (c0 > t0) __syncthreads();
    if (a < n) {
      const bool two = t > 0 && 2 * t != G2;
      const T u = pi_source<T, KIND>(fld, src, p.g, f, x1, t, 0);
      const T v = two ? pi_source<T, KIND>(fld, src, p.g, f, x1, G2 - t, 0) : T(0);
      sZ[a] = two ? mk2(u + v, u - v) : mk2(u, T(0));
    }
    __syncthreads();
    if (a < K2h) {
      const V2<T>* w = reinterpret_cast<const V2<T>*>(p.e2b) + (long long)c0 * K2p + a;
      sum_flat<T>(n, acc, [&](int i) { return sZ[i]; }, [&](int i) { return w[(long long)i * K2p]; });
    }
  }
  if (a < K2h)
    stq(P1 + ((((long long)x1 * gridDim.x + blockIdx.x) * gridDim.y + f) * K2h + a) * 4, Quad<T>{acc, zero2<T>()});
}

// The Hermitian array at the signs neg of the frequencies f from the coefficients
// v(s1, s2, s3): the sum of prod_j w_j v, w = 1 for a zero frequency, else 1/2 (cosine) or
// -i sigma / 2 (sine)
template <typename T, typename V>
__device__ __forceinline__ cplx<T> hermitian_value(const int* f, const bool* neg, V&& v) {
  cplx<T> z{T(0), T(0)};
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const int sn[3] = {m & 1, (m >> 1) & 1, (m >> 2) & 1};
    T w = T(1);
    int turns = 0;                                         // factors -i
    bool skip = false;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if (f[j] == 0) {
        if (sn[j]) skip = true;
        continue;
      }
      w *= T(0.5);
      if (sn[j]) {
        ++turns;
        if (neg[j]) w = -w;
      }
    }
    if (skip) continue;
    const T u = w * v(sn[0], sn[1], sn[2]);
    if (turns == 0) z.x += u;
    else if (turns == 1) z.y -= u;
    else if (turns == 2) z.x -= u;
    else z.y += u;
  }
  return z;
}

// x1 -> k1 of the nf projected planes of image-grid fields and their scaling:
// (13 us for 160 planes of three fields, band 32^3: latency and L2 reads)
// coef * (applyK ? 1/L^ : 1) * the sums (twice per axis of nonzero frequency), as band
// vectors out, or with HERM as the Hermitian arrays herm.  A quad holds every sign of its
// frequencies (the Nyquist slots stand where the negative of a zero would), so an item
// writes them without the launch and the round trip of k_band_store (a call on host
// arrays, 2D 64^2 / 16^2: 60 us with it, 50; on device arrays at 64^3 / 16^3: 40, 36).
template <typename T, bool HERM>
__global__ void __launch_bounds__(kImgThreads)
k_pi_band(const __grid_constant__ Plan<T> p, const T* P1, int nf, int nparts, int tqs, T coef, int applyK,
          const T* __restrict__ Lhat, T* __restrict__ out, cplx<T>* __restrict__ herm) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int PC = 4 << tqs, H1 = p.k.H1, q0 = blockIdx.x << tqs, nq = min(1 << tqs, p.k.Kq() - q0), H1p = up4(H1);
  V2<T>* sW = reinterpret_cast<V2<T>*>(smraw);             // [kChunk][H1p]
  V2<T>* sE = sW + kChunk * H1p;                           // [nf][kChunk][PC]
  V2<T>* sY = sE + 3 * kChunk * PC;                        // [nf][H1][PC]
  pdl_trigger();
  for (int t0 = 0; t0 < p.NT1; t0 += kChunk) {
    const int nt = min(kChunk, p.NT1 - t0);
    if (t0 > 0) __syncthreads();
    copy2<T, kImgThreads>(sW, p.e1b + (long long)t0 * H1p, nt * H1p);
    if (t0 == 0) pdl_wait();
    fold_planes<T, kImgThreads>(p, P1, nf, nparts, q0, nq, tqs, t0, nt, FastDiv{nt > 1 ? 0xffffffffu / nt + 1u : 0u},
                                sE);
    __syncthreads();
    contract_k1<T, kImgThreads, false, sizeof(T) == 4 ? 4 : 1>(p, nf, nt, tqs, H1p, sE, sW, t0 > 0, sY);
  }
  __syncthreads();
  auto scale = [&](int q, int h, int a, int b, int sc) {
    const T l = applyK ? T(1) / Lhat[2 * (((long long)q * H1 + h) * 4 + sc)] : T(1);
    return coef * l * (h ? T(2) : T(1)) * (a ? T(2) : T(1)) * (b ? T(2) : T(1));
  };
  if constexpr (HERM) {
    for (int it = threadIdx.x; it < nf * H1 * PC * 2; it += kImgThreads) {   // (c, h, quad, signs)
      const int m = it & 7, ql = (it >> 3) & ((1 << tqs) - 1), r = it >> (tqs + 3);
      const int c = r / H1, h = r - c * H1, q = q0 + ql;
      if (ql >= nq) continue;
      const int a = fdiv(q, p.dK3h), f[3] = {h, a, q - a * p.k.K3h}, n[3] = {p.b.k1, p.b.k2, p.b.k3};
      const bool neg[3] = {(m & 1) != 0, (m & 2) != 0, (m & 4) != 0};
      if (neg[2] && n[2] == 1) continue;
      int pos[3];
      bool nyq = false;
      for (int j = 0; j < 3; ++j) {
        if (neg[j] && f[j] == 0) nyq = true;
        pos[j] = !neg[j] ? f[j] : (f[j] == 0 ? n[j] / 2 : n[j] - f[j]);
      }
      const V2<T>* y = sY + (c * H1 + h) * PC + 4 * ql;
      const cplx<T> z = hermitian_value<T>(f, neg, [&](int s1, int s2, int s3) {
        const int sc = 2 * s3 + s2;
        T x, u;
        un2(y[sc], x, u);
        return scale(q, h, a, f[2], sc) * (s1 ? u : x);
      });
      herm[(long long)c * p.b.vol() + ((long long)pos[0] * n[1] + pos[1]) * n[2] + pos[2]] = nyq ? cplx<T>{T(0), T(0)} : z;
    }
    return;
  }
  for (int it = threadIdx.x; it < nf * H1 * PC; it += kImgThreads) {
    const int col = it & (PC - 1), r = it >> (tqs + 2);
    const int c = r / H1, h = r - c * H1, q = q0 + (col >> 2), sc = col & 3;
    if (col >= 4 * nq) continue;
    const int a = fdiv(q, p.dK3h), b = q - a * p.k.K3h;
    const bool dead = (a == 0 && (sc & 1)) || (b == 0 && (sc & 2));
    const T f = scale(q, h, a, b, sc);
    T x, y;
    un2(sY[it], x, y);
    reinterpret_cast<V2<T>*>(out)[(long long)c * p.k.Kq() * H1 * 4 + ((long long)q * H1 + h) * 4 + sc] =
        dead ? zero2<T>() : mk2(f * x, h ? f * y : T(0));
  }
}

// ---- Hermitian arrays <-> band vectors -------------------------------------------
// V[s1][s2][s3] = Re sum over the signs of (h, a, b) of prod_j (s_j ? i sigma_j : 1)
// in(sigma k): the real part keeps exactly the Hermitian part of the input.  One
// thread per slot; eight scattered reads each, 8 us at band 32^3.
template <typename T>
__global__ void k_band_load(const cplx<T>* __restrict__ in, T* __restrict__ out, int ncomp, Band bd) {
  const Trig k = trig_of(bd);
  const long long kvol = k.vol();
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= ncomp * kvol) return;
  const int c = (int)(idx / kvol);
  const int r = (int)(idx - c * kvol), s = (r >> 1) & 3, h = (r >> 3) % k.H1, q = (r >> 3) / k.H1;
  const int a = q / k.K3h, b = q - a * k.K3h;
  const int f[3] = {h, a, b}, sn[3] = {r & 1, s & 1, s >> 1}, n[3] = {bd.k1, bd.k2, bd.k3};
  T v = T(0);
  if (!((f[0] == 0 && sn[0]) || (f[1] == 0 && sn[1]) || (f[2] == 0 && sn[2]))) {
    for (int m = 0; m < 8; ++m) {
      int pos[3], turns = 0;                               // product of i sigma: i^ones times the signs
      bool skip = false;
      T sg = T(1);
      for (int j = 0; j < 3; ++j) {
        const bool neg = (m >> j) & 1;
        if (neg && f[j] == 0) skip = true;
        pos[j] = neg ? n[j] - f[j] : f[j];
        if (sn[j]) {
          ++turns;
          if (neg) sg = -sg;
        }
      }
      if (skip) continue;
      const cplx<T> z = in[(long long)c * bd.vol() + ((long long)pos[0] * bd.k2 + pos[1]) * bd.k3 + pos[2]];
      v += sg * (turns == 0 ? z.x : (turns == 1 ? -z.y : (turns == 2 ? -z.x : z.y)));   // Re(i^turns z)
    }
  }
  out[idx] = v;
}

// out(sigma k) = hermitian_value of the slot's quad; Nyquist slots are zero
template <typename T>
__global__ void k_band_store(const T* __restrict__ in, cplx<T>* __restrict__ out, int ncomp, Band bd) {
  const Trig k = trig_of(bd);
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= ncomp * bd.vol()) return;
  const int c = (int)(idx / bd.vol());
  const int r = (int)(idx - c * bd.vol());
  const int pos[3] = {r / (bd.k2 * bd.k3), (r / bd.k3) % bd.k2, r % bd.k3}, n[3] = {bd.k1, bd.k2, bd.k3};
  int f[3];
  bool neg[3], nyq = false;
  for (int j = 0; j < 3; ++j) {
    neg[j] = 2 * pos[j] > n[j];
    f[j] = neg[j] ? n[j] - pos[j] : pos[j];
    if (n[j] > 1 && 2 * pos[j] == n[j]) nyq = true;
  }
  cplx<T> z{T(0), T(0)};
  if (!nyq) {
    const T* v = in + (long long)c * k.vol() + ((long long)(f[1] * k.K3h + f[2]) * k.H1 + f[0]) * 8;
    z = hermitian_value<T>(f, neg, [&](int s1, int s2, int s3) { return v[(2 * s3 + s2) * 2 + s1]; });
  }
  out[idx] = z;
}

// row pairs per thread of k2 -> x2: all of an item's where that fits the registers
int plane_pt(int ppc) { return ppc <= 3 ? 3 : (ppc <= 5 ? 5 : 9); }
template <typename T>
size_t plane_smem(const Plan<T>& p, int mode, int ppc) {
  return plane_shape(p, mode_in(mode), mode_out(mode), ppc, plane_pt(ppc)).smem;
}

// quads per band-phase item (2^tqs <= 4): one item per SM while every (k1, column)
// has a thread and the item fits shared memory
template <typename T>
int band_tqs(const Plan<T>& p, int mode) {
  int s = 0;
  while (s < 2 && (p.k.Kq() >> s) > kSMs && p.k.H1 * (8 << s) <= kPhaseThreads &&
         band_shape(p, 2 << s, mode_out(mode), mode_in(mode)).smem <= (size_t)kMaxSmem)
    ++s;
  return s;
}

// Row pairs per image-plane item: as many as give every thread a k2 -> x2 (or x3 ->
// k3) sum, so that one pass of loads feeds the item, then cut evenly.
inline int even_pairs(int NT2, int most, int step) {
  const int parts = (NT2 + most - 1) / most, pairs = (NT2 + parts - 1) / parts;
  return (pairs + step - 1) / step * step;
}
template <typename T>
int iota_pairs(const Plan<T>& p) {
  int most = std::max(1, kImgThreads / (kIotaGroup * p.k.K3h)) * kIotaPT;
  while (most > kIotaPT && plane_shape(p, kIotaGroup, 0, most, kIotaPT).smem > (size_t)96 * 1024) most -= kIotaPT;
  return even_pairs(p.NT2, most, kIotaPT);
}
// Most elements of the image-grid scratch: what a transform that takes axis 1 last would
// hold of 33 fields, or 2^24; at least one partial plane and one velocity.  The planes of
// the kernels here grow with the first axis, so a long one with a thin band would take
// many times that (19020 x 2965 x 21, band 2 x 416 x 18, one time step: 72 GB for 33 fields
// at once and a partial plane per item, beside 165 GB of the rest; 1.7 GB so).
template <typename T>
long long image_scratch(const Plan<T>& p) {
  return std::max(33LL * p.b.k1 * p.g.n2 * p.g.n3, 1LL << 24);
}
struct PiSplit {
  int ppi, reps, nparts;   // row pairs at once, times one after another, partial planes
};
template <typename T>
PiSplit pi_split(const Plan<T>& p) {
  PiSplit s{p.NT2, 1, 1};
  if (p.flat) {
    // a thread sums the points of an item in turn: parts of 64 row pairs while a wave has
    // room (a pi call of a 64 x 1024 image, band 8 x 512: 88 us whole, 57 in parts)
    const int parts = std::max(1, std::min((p.NT2 + 63) / 64, 4 * kSMs / p.g.n1));
    s.ppi = (p.NT2 + parts - 1) / parts;
  } else {
    int most = std::max(1, 2 * kImgThreads / p.K3e);
    while (most > 1 && plane_shape(p, 0, 1, most, 1).smem > (size_t)96 * 1024) --most;
    s.ppi = even_pairs(p.NT2, most, 1);
    const int parts = (p.NT2 + s.ppi - 1) / s.ppi;
    const long long fit = std::max(1LL, image_scratch(p) / ((long long)p.g.n1 * 3 * p.k.Kq() * 4));
    if (parts > fit) s.reps = (int)((parts + fit - 1) / fit);
  }
  s.nparts = (p.NT2 + s.ppi * s.reps - 1) / (s.ppi * s.reps);
  return s;
}

template <typename T, int MODE, int PT>
cudaError_t launch_plane_pt(const Plan<T>& p, const T* T1, T* slot, T* slot2, T* P1, cudaStream_t st) {
  const EvalGeom g = p.geom[MODE];
  cudaError_t e = allow_smem<k_plane<T, MODE, PT>>();
  if (e != cudaSuccess) return e;
  return launch_chain(k_plane<T, MODE, PT>, dim3((unsigned)(p.g.n1 * g.nparts)), plane_threads<T>(PT),
                      plane_smem(p, MODE, g.ppc), st, p, g.ppc, g.nparts, T1, slot, slot2, P1);
}
template <typename T, int MODE>
cudaError_t launch_plane(const Plan<T>& p, const T* T1, T* slot, T* slot2, T* P1, cudaStream_t st) {
  const EvalGeom g = p.geom[MODE];
  const int pt = plane_pt(g.ppc);
  if (p.flat) {
    cudaError_t e = allow_smem<k_plane_flat<T, MODE>>();
    if (e != cudaSuccess) return e;
    return launch_chain(k_plane_flat<T, MODE>, dim3((unsigned)(p.g.n1 * g.nparts)), kPhaseThreads,
                        plane_flat_smem<T>(MODE, g.ppc), st, p, g.ppc, g.nparts, T1, slot, slot2, P1);
  }
  if (pt == 3) return launch_plane_pt<T, MODE, 3>(p, T1, slot, slot2, P1, st);
  if (pt == 5) return launch_plane_pt<T, MODE, 5>(p, T1, slot, slot2, P1, st);
  return launch_plane_pt<T, MODE, 9>(p, T1, slot, slot2, P1, st);
}

template <typename T, int MODE, bool FLAT, int MINB>
cudaError_t launch_band_as(const Plan<T>& p, const PiEpi<T>* prev, const T* P1, const T* A, const T* B, T* T1,
                           const T* Lhat, cudaStream_t st) {
  BandArgs<T> a{};
  a.p = p;
  a.P1 = P1;
  a.A = A;
  a.B = B;
  a.Lhat = Lhat;
  a.T1 = T1;
  a.tqs = p.geom[MODE].tqs;
  a.nparts = p.geom[MODE].nparts;
  if (prev != nullptr && prev->nout > 0) {
    a.e = *prev;
    a.prev = 1;
  } else if (A == nullptr) {
    return cudaSuccess;
  }
  cudaError_t e = allow_smem<k_band<T, MODE, FLAT, MINB>>();
  if (e != cudaSuccess) return e;
  return launch_chain(k_band<T, MODE, FLAT, MINB>, dim3((unsigned)((p.k.Kq() + (1 << a.tqs) - 1) >> a.tqs)), kPhaseThreads,
                      band_shape(p, 1 << a.tqs, fields_out(MODE, FLAT), fields_in(MODE, FLAT)).smem, st, a);
}
template <typename T, int MODE>
cudaError_t launch_band(const Plan<T>& p, const PiEpi<T>* prev, const T* P1, const T* A, const T* B, T* T1,
                        const T* Lhat, cudaStream_t st) {
  if (p.flat) return launch_band_as<T, MODE, true, 1>(p, prev, P1, A, B, T1, Lhat, st);
  // more items than SMs: two to an SM (band 64^3: 166 us per evaluation against 182
  // with one, band 40^3: 36.4 / 39.6); below that the registers are worth more (32^3:
  // 21.6 / 19.5)
  if (shared_sms(p, p.geom[MODE].tqs))
    return launch_band_as<T, MODE, false, sizeof(T) == 4 ? 2 : 1>(p, prev, P1, A, B, T1, Lhat, st);
  return launch_band_as<T, MODE, false, 1>(p, prev, P1, A, B, T1, Lhat, st);
}

template <typename T, int TL, int RB>
cudaError_t launch_iota_plane(const Plan<T>& p, const IotaList<T>& d, const T* T1, cudaStream_t st) {
  const unsigned groups = (unsigned)((d.nf + kIotaGroup - 1) / kIotaGroup);
  const int ppi = iota_pairs(p);
  cudaError_t e = allow_smem<k_iota_plane<T, TL, RB>>();
  if (e != cudaSuccess) return e;
  return launch_chain(k_iota_plane<T, TL, RB>,
                      dim3((unsigned)((p.NT2 + ppi - 1) / ppi), groups, (unsigned)p.g.n1), kImgThreads,
                      plane_shape(p, kIotaGroup, 0, ppi, kIotaPT).smem, st, p, d, ppi, T1);
}

template <typename T, int TL, int RB>
cudaError_t launch_iota_plane_even(const Plan<T>& p, const IotaList<T>& d, const T* T1, cudaStream_t st) {
  const unsigned groups = (unsigned)((d.nf + kIotaGroup - 1) / kIotaGroup);
  const int ppi = iota_pairs(p);
  cudaError_t e = allow_smem<k_iota_plane_even<T, TL, RB>>();
  if (e != cudaSuccess) return e;
  return launch_chain(k_iota_plane_even<T, TL, RB>,
                      dim3((unsigned)((p.NT2 + ppi - 1) / ppi), groups, (unsigned)p.g.n1), kImgThreads,
                      plane_shape(p, kIotaGroup, 0, ppi, kIotaPT).smem, st, p, d, ppi, T1);
}

template <typename T, int KIND>
cudaError_t launch_pi_plane(const Plan<T>& p, const PiField<T>& s, int nf, T* P1, cudaStream_t st) {
  const PiSplit w = pi_split(p);
  const dim3 grid((unsigned)w.nparts, (unsigned)nf, (unsigned)p.g.n1);
  if (p.flat) return launch_chain(k_pi_plane_flat<T, KIND>, grid, kImgThreads, 0, st, p, s, w.ppi, P1);
  const size_t smem = plane_shape(p, 0, 1, w.ppi, 1).smem;
  cudaError_t e;
  if (w.reps > 1) {
    if ((e = allow_smem<k_pi_plane_seq<T, KIND>>()) != cudaSuccess) return e;
    return launch_chain(k_pi_plane_seq<T, KIND>, grid, kImgThreads, smem, st, p, s, w.ppi, w.reps, P1);
  }
  if ((e = allow_smem<k_pi_plane<T, KIND>>()) != cudaSuccess) return e;
  return launch_chain(k_pi_plane<T, KIND>, grid, kImgThreads, smem, st, p, s, w.ppi, P1);
}

}  // namespace

// Rows per plane item: the fewest waves of items over the SMs, each costing its
// rows plus a fixed chain (launch, first loads, barriers: about two row pairs'
// work), and a partial plane more to be summed for every part.
template <typename T>
EvalGeom eval_geom(const Plan<T>& p, PwMode mode) {
  EvalGeom g{1, p.NT2, 0};
  if (p.flat) {
    // Half a thread block of k2 -> x2 sums per item, while the items fit the SMs two to
    // one.  Band 8 x 512 has 12 planes of 385 row pairs: 28 of an item's rounds of sums on
    // 12 SMs took 490 us per evaluation of a product, 25 parts take 54.  Items of one sum
    // per thread leave the way back longer (band 2 x 300: 46 us; 34).  At 64 x 512 in FP64,
    // 96 planes: 1.3 ms whole, 0.75 in 3 parts.
    const int most = std::max(1, 2 * kSMs / p.g.n1);
    const int want = kPhaseThreads / (2 * fields_in(mode, true));
    const int parts = std::min((p.NT2 + want - 1) / want, most);
    g.ppc = (p.NT2 + parts - 1) / parts;
    g.nparts = (p.NT2 + g.ppc - 1) / g.ppc;
    return g;
  }
  double best = 1e300;
  for (int parts = 1; parts <= p.NT2; ++parts) {
    const int ppc = (p.NT2 + parts - 1) / parts;
    if ((p.NT2 + ppc - 1) / ppc != parts) continue;        // the same cut as with fewer parts
    if (plane_smem(p, mode, ppc) > (size_t)kMaxSmem) continue;
    const double waves = (double)(((long long)p.g.n1 * parts + kSMs - 1) / kSMs);
    const double cost = waves * (ppc + 2.0) + 0.3 * parts;
    if (cost < best) {
      best = cost;
      g.ppc = ppc;
      g.nparts = parts;
    }
  }
  g.tqs = band_tqs(p, mode);
  return g;
}

template <typename T>
cudaError_t band_phase(const Plan<T>& p, PwMode mode, const PiEpi<T>* prev, const T* P1, const T* A, const T* B, T* T1,
                       const T* Lhat, cudaStream_t st) {
  switch (mode) {
    case PW_F: return launch_band<T, PW_F>(p, prev, P1, A, B, T1, Lhat, st);
    case PW_T: return launch_band<T, PW_T>(p, prev, P1, A, B, T1, Lhat, st);
    case PW_TC: return launch_band<T, PW_TC>(p, prev, P1, A, B, T1, Lhat, st);
    case PW_GT: return launch_band<T, PW_GT>(p, prev, P1, A, B, T1, Lhat, st);
    case PW_D0: return launch_band<T, PW_D0>(p, prev, P1, A, B, T1, Lhat, st);
    case PW_D1: return launch_band<T, PW_D1>(p, prev, P1, A, B, T1, Lhat, st);
    default: return launch_band<T, PW_D2>(p, prev, P1, A, B, T1, Lhat, st);
  }
}

template <typename T>
cudaError_t plane_phase(const Plan<T>& p, PwMode mode, const T* T1, T* slot, T* slot2, T* P1, cudaStream_t st) {
  switch (mode) {
    case PW_F: return launch_plane<T, PW_F>(p, T1, slot, slot2, P1, st);
    case PW_T: return launch_plane<T, PW_T>(p, T1, slot, slot2, P1, st);
    case PW_TC: return launch_plane<T, PW_TC>(p, T1, slot, slot2, P1, st);
    case PW_GT: return launch_plane<T, PW_GT>(p, T1, slot, slot2, P1, st);
    case PW_D0: return launch_plane<T, PW_D0>(p, T1, slot, slot2, P1, st);
    case PW_D1: return launch_plane<T, PW_D1>(p, T1, slot, slot2, P1, st);
    default: return launch_plane<T, PW_D2>(p, T1, slot, slot2, P1, st);
  }
}

template <typename T>
long long eval_T1_elems(const Plan<T>& p) {
  return (long long)p.g.n1 * kMaxInFields * p.k.Kq() * 4;
}
template <typename T>
long long eval_P1_elems(const Plan<T>& p) {
  long long n = 0;
  for (int m = 0; m < PW_MODES; ++m)
    n = std::max(n, (long long)p.g.n1 * p.geom[m].nparts * mode_out(m) * p.k.Kq() * 4);
  return n;
}

template <typename T>
long long iota_T1_elems(const Plan<T>& p, int nf) {
  return (long long)p.g.n1 * nf * p.k.Kq() * 4;
}
template <typename T>
int iota_fields_at_once(const Plan<T>& p, int most) {
  int nf = std::min(most, 33);
  while (nf > 3 && iota_T1_elems(p, nf) > image_scratch(p)) nf -= 3;
  return nf;
}
template <typename T>
cudaError_t iota_fields(const Plan<T>& p, const IotaList<T>& d, T* T1, cudaStream_t st) {
  const int tqs = p.k.Kq() >= 4 ? 2 : 0;
  const size_t smem = (size_t)(up2(kIotaBandGroup * p.k.H1 * (4 << tqs)) + p.k.H1 * kChunk) * sizeof(V2<T>);
  cudaError_t e = allow_smem<k_iota_band<T>>();
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)((p.k.Kq() + (1 << tqs) - 1) >> tqs),
                  (unsigned)((d.nf + kIotaBandGroup - 1) / kIotaBandGroup));
  if ((e = launch_chain(k_iota_band<T>, grid, kImgThreads, smem, st, p, d, tqs, T1)) != cudaSuccess) return e;
  if (p.flat)
    return launch_chain(k_iota_plane_flat<T>,
                        dim3((unsigned)((p.NT2 + kImgThreads - 1) / kImgThreads), (unsigned)d.nf, (unsigned)p.g.n1),
                        kImgThreads, 0, st, p, d, (const T*)T1);
  // TL: the fewest lanes idle in one pass over t; RB: what 128 registers hold
  if (p.g.n3 % 2 == 0) {
    const int nq = p.g.n3 / 4 + 1;
    if (nq <= 16) return launch_iota_plane_even<T, 1, 8>(p, d, T1, st);
    if (nq <= 32) return launch_iota_plane_even<T, 2, 5>(p, d, T1, st);
    if (nq <= 48) return launch_iota_plane_even<T, 3, 4>(p, d, T1, st);
    return launch_iota_plane_even<T, 4, 3>(p, d, T1, st);
  }
  if (p.NT3 <= 32) return launch_iota_plane<T, 1, 8>(p, d, T1, st);
  if (p.NT3 <= 64) return launch_iota_plane<T, 2, 8>(p, d, T1, st);
  if (p.NT3 <= 96) return launch_iota_plane<T, 3, 6>(p, d, T1, st);
  return launch_iota_plane<T, 4, 4>(p, d, T1, st);
}

template <typename T>
long long pi_P1_elems(const Plan<T>& p) {
  return (long long)p.g.n1 * pi_split(p).nparts * 3 * p.k.Kq() * 4;
}
template <typename T>
cudaError_t pi_fields(const Plan<T>& p, PiKind kind, const PiField<T>& s, const PiEpi<T>& e, const T* Lhat, T* P1,
                      cudaStream_t st, cplx<T>* herm) {
  const int nf = e.ncomp, nparts = pi_split(p).nparts;
  cudaError_t rc;
  switch (kind) {
    case PI_FIELD: rc = launch_pi_plane<T, PI_FIELD>(p, s, nf, P1, st); break;
    case PI_RESIDUAL: rc = launch_pi_plane<T, PI_RESIDUAL>(p, s, nf, P1, st); break;
    case PI_INCREMENT: rc = launch_pi_plane<T, PI_INCREMENT>(p, s, nf, P1, st); break;
    default: rc = launch_pi_plane<T, PI_NEWTON>(p, s, nf, P1, st); break;
  }
  if (rc != cudaSuccess) return rc;
  const int tqs = p.k.Kq() >= 2 * kSMs ? 1 : 0, PC = 4 << tqs, H1 = p.k.H1;
  const size_t smem = (size_t)(kChunk * up4(H1) + 3 * kChunk * PC + 3 * H1 * PC) * sizeof(V2<T>);
  const dim3 grid((unsigned)((p.k.Kq() + (1 << tqs) - 1) >> tqs));
  auto launch = [&](auto kern) {
    return launch_chain(kern, grid, kImgThreads, smem, st, p, (const T*)P1, nf, nparts, tqs, e.coef[0], e.applyK[0],
                        Lhat, e.dst[0], herm);
  };
  if (herm != nullptr) {
    if ((rc = allow_smem<k_pi_band<T, true>>()) != cudaSuccess) return rc;
    return launch(k_pi_band<T, true>);
  }
  if ((rc = allow_smem<k_pi_band<T, false>>()) != cudaSuccess) return rc;
  return launch(k_pi_band<T, false>);
}

template <typename T>
void band_load(const cplx<T>* in, T* out, int ncomp, const Band& b, cudaStream_t st) {
  const long long n = ncomp * trig_of(b).vol();
  k_band_load<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(in, out, ncomp, b);
}
template <typename T>
void band_store(const T* in, cplx<T>* out, int ncomp, const Band& b, cudaStream_t st) {
  const long long n = ncomp * b.vol();
  k_band_store<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(in, out, ncomp, b);
}

// ---- accepted sizes -----------------------------------------------------------
// The interface takes the grids and bands whose complex half-spectrum tiles (two
// slabs and a twiddle table per axis, in the item sizes below) fit 200 KB of shared
// memory, N_3 nper <= 512 and K_1 <= 64, and lddmm_create K_j <= 512: a rule of the
// interface, kept as it is so that the same sizes run.  Every kernel above fits kMaxSmem
// within it (all accepted sizes evaluated: at most 224 KB in 3D, where eval_geom cuts the
// items to fit; a whole 2D plane 75 KB, in FP64 150).
template <typename T>
bool sizes_accepted(const Dims& g, const Band& b, int nper, bool brackets) {
  constexpr size_t lim = 200 * 1024, C = 2 * sizeof(T);
  constexpr int threads = 256;
  const size_t G1 = g.n1, G2 = g.n2, G3 = g.n3, H1 = b.h1, K2 = b.k2, K3 = b.k3;
  if ((size_t)nper * G3 > 2 * (size_t)threads || H1 > 32 || H1 * G1 * C > lim) return false;
  if (brackets && G1 > 2 * (size_t)threads) return false;
  const size_t G3e = G3 + (G3 & 1), G2e = G2 + (G2 & 1);
  const size_t ab0 = (K2 * K3 + K2 * G3e) * C + K2 * K3 * sizeof(T), ab1 = ab0 + (K3 * G3e + K2 * G2e) * C;
  if ((ab1 <= 64 * 1024 ? ab1 : ab0) > lim) return false;
  if (brackets) {
    auto cpw = [&](size_t TP) {
      return (24 * H1 * TP + H1 * ((G1 + 3) & ~size_t(3)) + G1 * ((H1 + 3) & ~size_t(3))) * C + 33 * G1 * TP * sizeof(T);
    };
    size_t TP = std::max<size_t>(1, std::min<size_t>(8, G2 * G3 / 152));
    while (TP > 1 && (cpw(TP) > lim || G1 * TP > 2 * (size_t)threads)) --TP;
    if (cpw(TP) > lim) return false;
  }
  constexpr size_t E = 128 / C;
  const size_t G3s = G3 + ((E / 2 + E - G3 % E) % E);
  for (size_t np = 1; np <= (size_t)nper; ++np) {
    const size_t want = std::max<size_t>(1, (304 + 36 * H1 - 1) / (36 * H1));
    size_t KC = std::min(std::min(std::max<size_t>(1, (K2 + want - 1) / want), size_t(8)), K2);
    const size_t R = std::max<size_t>(1, std::min<size_t>(8, threads / (np * G3)));
    const size_t row = np * G3 * C;
    auto fixed = [&]() { return (G2 * KC + G3s * K3 + R * np * KC * G3 + KC * K3 * 16) * C + KC * K3 * sizeof(T); };
    while (KC > 1 && fixed() + row * KC > lim) --KC;
    const size_t target = fixed() + 16 * row > 72 * 1024 ? 150 * 1024 : 72 * 1024;
    const size_t rows = fixed() < target ? (target - fixed()) / row : 0;
    if (fixed() + row * std::max(KC, std::min(G2, rows)) > lim) return false;
  }
  return true;
}

#define LDDMM_DFT_INST(T)                                                                                          \
  template EvalGeom eval_geom<T>(const Plan<T>&, PwMode);                                                          \
  template cudaError_t band_phase<T>(const Plan<T>&, PwMode, const PiEpi<T>*, const T*, const T*, const T*, T*,     \
                                     const T*, cudaStream_t);                                                      \
  template cudaError_t plane_phase<T>(const Plan<T>&, PwMode, const T*, T*, T*, T*, cudaStream_t);                 \
  template long long eval_T1_elems<T>(const Plan<T>&);                                                             \
  template long long eval_P1_elems<T>(const Plan<T>&);                                                             \
  template long long iota_T1_elems<T>(const Plan<T>&, int);                                                        \
  template int iota_fields_at_once<T>(const Plan<T>&, int);                                                        \
  template cudaError_t iota_fields<T>(const Plan<T>&, const IotaList<T>&, T*, cudaStream_t);                       \
  template long long pi_P1_elems<T>(const Plan<T>&);                                                               \
  template cudaError_t pi_fields<T>(const Plan<T>&, PiKind, const PiField<T>&, const PiEpi<T>&, const T*, T*,      \
                                    cudaStream_t, cplx<T>*);                                                       \
  template void band_load<T>(const cplx<T>*, T*, int, const Band&, cudaStream_t);                                  \
  template void band_store<T>(const T*, cplx<T>*, int, const Band&, cudaStream_t);                                 \
  template bool sizes_accepted<T>(const Dims&, const Band&, int, bool);
LDDMM_DFT_INST(float)
LDDMM_DFT_INST(double)

}  // namespace lddmm
