// Allocation-free variant of the band-limited -> grid transform (iota).
//
// Some callers cannot let a library call cudaMalloc: a host framework whose
// caching allocator already holds nearly all device memory, a latency-bound
// loop that cannot absorb the device-wide synchronisation cudaFree implies,
// or a plugin host that forbids libraries from allocating at all.  For them
// lddmm_iota_noalloc runs the transform with every intermediate in the
// fixed device array below instead of in buffers of a context.  The caller passes
// device inputs and outputs only.
//
// It contracts k3 -> x3 and k2 -> x2 of each complex half-spectrum slab (field,
// k1 >= 0) first and k1 -> x1 last: the intermediate [field][K1/2][N2][N3] is then
// bounded by the output, which is what the fixed array is sized for (the contexts'
// kernels hold [N1][field][K2][K3], which a long first axis can make larger).
#include <mutex>

#include "../../include/lddmm.h"
#include "internal.h"

namespace lddmm {
namespace {

constexpr int kThr = 256;
constexpr int kSmem = 200 * 1024;
constexpr int kMaxH1 = 32;

// sizes and twiddles: E3f[k3][x3], E2f[k2][x2] = exp(2 pi i f(k) x / G); E1f[h][x1]
// = w(h) exp(2 pi i h x1 / G1), w = 1 (h = 0) or 2
struct CPlan {
  Dims g;
  Band b;
  float2 *E3f, *E2f, *E1f;
};

// The kernels after the first are launched while their predecessor runs (programmatic
// dependent launch) and wait here for its end; the first one follows the stream's earlier
// work as usual.  What a predecessor wrote is read through plain pointers: loads through
// const __restrict__ ones could be moved before the wait.
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ bool nyq(int q, int K) { return (K % 2 == 0) && (2 * q == K); }
__device__ __forceinline__ void cmac(float2& acc, const float2& a, const float2& e) {
  acc.x = fmaf(a.x, e.x, fmaf(-a.y, e.y, acc.x));
  acc.y = fmaf(a.x, e.y, fmaf(a.y, e.x, acc.y));
}
__device__ __forceinline__ void ldpair(const float2* p, float2& a, float2& b) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  a = make_float2(v.x, v.y);
  b = make_float2(v.z, v.w);
}
__host__ __device__ __forceinline__ int even_up(int n) { return n + (n & 1); }

// (a(k) + conj a(-k)) / 2 with the Nyquist slots dropped
__global__ void k_hermitianize(const float2* __restrict__ in, float2* __restrict__ out, int ncomp, Band b) {
  chain_wait();
  const long long kvol = b.vol();
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= ncomp * kvol) return;
  const long long c = idx / kvol, r = idx % kvol;
  const int k3 = (int)(r % b.k3), k2 = (int)((r / b.k3) % b.k2), k1 = (int)(r / ((long long)b.k2 * b.k3));
  float2 v = make_float2(0.f, 0.f);
  if (!(nyq(k1, b.k1) || nyq(k2, b.k2) || nyq(k3, b.k3))) {
    const long long m = c * kvol +
        (((long long)((b.k1 - k1) % b.k1) * b.k2 + (b.k2 - k2) % b.k2) * b.k3 + (b.k3 - k3) % b.k3);
    const float2 a = in[idx], am = in[m];
    v = make_float2(0.5f * (a.x + am.x), 0.5f * (a.y - am.y));
  }
  out[idx] = v;
}

// stages A (k3 -> x3) and B (k2 -> x2) of one slab (field f, h), in 2 x 2 complex
// register tiles; shared memory: S0 [K2][K3], S1 [K2][G3e], with TWS the twiddles
template <bool TWS>
__global__ void __launch_bounds__(kThr) k_slab(CPlan p, const float2* src0, float2* T2) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int G2 = p.g.n2, G3 = p.g.n3, K2 = p.b.k2, K3 = p.b.k3, H1 = p.b.h1;
  const int G2e = even_up(G2), G3e = even_up(G3);
  const int f = blockIdx.x / H1, h = blockIdx.x % H1, tid = threadIdx.x;
  float2* S0 = reinterpret_cast<float2*>(smraw);
  float2* S1 = S0 + even_up(K2 * K3);
  float2* E3s = S1 + K2 * G3e;
  float2* E2s = E3s + K3 * G3e;
  const float2 zero = make_float2(0.f, 0.f);
  chain_wait();
  if (TWS) {
    for (int i = tid; i < K3 * G3e; i += kThr) {
      const int r = i / G3e, x = i - r * G3e;
      E3s[i] = x < G3 ? p.E3f[r * G3 + x] : zero;
    }
    for (int i = tid; i < K2 * G2e; i += kThr) {
      const int r = i / G2e, x = i - r * G2e;
      E2s[i] = x < G2 ? p.E2f[r * G2 + x] : zero;
    }
  }
  const float2* src = src0 + (long long)f * p.b.vol() + (long long)h * K2 * K3;
  for (int i = tid; i < K2 * K3; i += kThr) S0[i] = src[i];
  __syncthreads();
  const int n3p = G3e / 2, n2p = G2e / 2;
  for (int it = tid; it < (K2 / 2) * n3p; it += kThr) {
    const int kp = it / n3p, xp = it - kp * n3p, k2 = 2 * kp, x3 = 2 * xp;
    float2 c00 = zero, c01 = zero, c10 = zero, c11 = zero;
    const float2* s0 = S0 + k2 * K3;
#pragma unroll 4
    for (int k3 = 0; k3 < K3; ++k3) {
      const float2 a0 = s0[k3], a1 = s0[K3 + k3];
      float2 e0, e1;
      if (TWS) {
        ldpair(E3s + k3 * G3e + x3, e0, e1);
      } else {
        e0 = p.E3f[k3 * G3 + x3];
        e1 = x3 + 1 < G3 ? p.E3f[k3 * G3 + x3 + 1] : zero;
      }
      cmac(c00, a0, e0); cmac(c01, a0, e1); cmac(c10, a1, e0); cmac(c11, a1, e1);
    }
    S1[k2 * G3e + x3] = c00;
    S1[k2 * G3e + x3 + 1] = c01;
    S1[(k2 + 1) * G3e + x3] = c10;
    S1[(k2 + 1) * G3e + x3 + 1] = c11;
  }
  __syncthreads();
  float2* __restrict__ out = T2 + (long long)(f * H1 + h) * G2 * G3;
  for (int it = tid; it < n2p * n3p; it += kThr) {
    const int yp = it / n3p, xp = it - yp * n3p, x2 = 2 * yp, x3 = 2 * xp;
    float2 c00 = zero, c01 = zero, c10 = zero, c11 = zero;
#pragma unroll 4
    for (int k2 = 0; k2 < K2; ++k2) {
      float2 s0, s1, e0, e1;
      ldpair(S1 + k2 * G3e + x3, s0, s1);
      if (TWS) {
        ldpair(E2s + k2 * G2e + x2, e0, e1);
      } else {
        e0 = p.E2f[k2 * G2 + x2];
        e1 = x2 + 1 < G2 ? p.E2f[k2 * G2 + x2 + 1] : zero;
      }
      cmac(c00, s0, e0); cmac(c01, s1, e0); cmac(c10, s0, e1); cmac(c11, s1, e1);
    }
    out[(long long)x2 * G3 + x3] = c00;
    if (x3 + 1 < G3) out[(long long)x2 * G3 + x3 + 1] = c01;
    if (x2 + 1 < G2) {
      out[(long long)(x2 + 1) * G3 + x3] = c10;
      if (x3 + 1 < G3) out[(long long)(x2 + 1) * G3 + x3 + 1] = c11;
    }
  }
}

// stage C: each thread holds the H1 coefficients of one (x2, x3) position and
// walks all x1
template <int HR>
__global__ void __launch_bounds__(kThr) k_pencil(CPlan p, const float2* T2, float* __restrict__ f_out) {
  extern __shared__ __align__(16) unsigned char smraw[];
  float2* sE = reinterpret_cast<float2*>(smraw);           // [G1][H1]
  const int G1 = p.g.n1, H1 = p.b.h1;
  const long long inner = (long long)p.g.n2 * p.g.n3, nblk = (inner + kThr - 1) / kThr;
  const int f = (int)(blockIdx.x / nblk);
  const long long i = (blockIdx.x % nblk) * kThr + threadIdx.x;
  chain_wait();
  for (int j = threadIdx.x; j < H1 * G1; j += kThr) {
    const int x = j / H1, h = j - x * H1;
    sE[j] = p.E1f[h * G1 + x];
  }
  float2 a[HR];
  const bool live = i < inner;
  const float2* src = T2 + (long long)f * H1 * inner + i;
#pragma unroll
  for (int h = 0; h < HR; ++h) a[h] = (live && h < H1) ? src[(long long)h * inner] : make_float2(0.f, 0.f);
  __syncthreads();
  if (!live) return;
  float* __restrict__ dst = f_out + (long long)f * p.g.vol() + i;
  for (int x = 0; x < G1; ++x) {
    const float2* e = sE + x * H1;
    float v0 = 0.f, v1 = 0.f;
#pragma unroll
    for (int h = 0; h < HR; h += 2) {
      if (h < H1) v0 = fmaf(a[h].x, e[h].x, fmaf(-a[h].y, e[h].y, v0));
      if (h + 1 < H1) v1 = fmaf(a[h + 1].x, e[h + 1].x, fmaf(-a[h + 1].y, e[h + 1].y, v1));
    }
    dst[(long long)x * inner] = v0 + v1;
  }
}

template <typename... KArgs, typename... Args>
cudaError_t run(void (*kern)(KArgs...), long long grid, size_t smem, cudaStream_t st, Args... args) {
  // large items start as the predecessor ends: early ones would share the few SMs then free
  const bool large = smem > 32 * 1024;
  if (large) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kThr);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  cfg.attrs = at;
  cfg.numAttrs = large ? 0 : chain_attrs(at);
  return cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
}

// Fixed scratch: every GPU that loads this library holds it until exit.
constexpr size_t kNoAllocBytes = size_t(32) << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// Host code must not use g_noalloc_scratch as an address: its host name is a
// stand-in symbol.  The device address is looked up once per device.
struct DeviceScratch {
  std::once_flag once;
  cudaError_t err = cudaSuccess;
  unsigned char* ptr = nullptr;
};
constexpr int kMaxDevices = 64;
DeviceScratch g_scratch_of[kMaxDevices];

__device__ __forceinline__ int sfreq_dev(int q, int K) { return (2 * q < K) ? q : q - K; }

__device__ __forceinline__ float2 twiddle(long long p, int G, double w) {
  const long long r = ((p % G) + G) % G;
  double s, c;
  sincospi(2.0 * (double)r / (double)G, &s, &c);
  return make_float2((float)(w * c), (float)(w * s));
}

// The three twiddle tables of CPlan, one entry per thread.
__global__ void k_iota_twiddles(float2* E3f, float2* E2f, float2* E1f, Band b, Dims g) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long n3 = (long long)b.k3 * g.n3, n2 = (long long)b.k2 * g.n2,
                  n1 = (long long)b.h1 * g.n1;
  if (i < n3) {
    const int k = (int)(i / g.n3), x = (int)(i % g.n3);
    E3f[i] = twiddle((long long)sfreq_dev(k, b.k3) * x, g.n3, 1.0);
    return;
  }
  i -= n3;
  if (i < n2) {
    const int k = (int)(i / g.n2), x = (int)(i % g.n2);
    E2f[i] = twiddle((long long)sfreq_dev(k, b.k2) * x, g.n2, 1.0);
    return;
  }
  i -= n2;
  if (i < n1) {
    const int h = (int)(i / g.n1), x = (int)(i % g.n1);
    E1f[i] = twiddle((long long)h * x, g.n1, h == 0 ? 1.0 : 2.0);
  }
}

size_t align256(size_t n) { return (n + 255) & ~size_t(255); }

// device memory of device dev (or managed memory, which every device reaches)
bool is_device_pointer(const void* p, int dev) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (at.type == cudaMemoryTypeManaged) return true;
  return at.type == cudaMemoryTypeDevice && at.device == dev;
}

}  // namespace
}  // namespace lddmm

extern "C" int lddmm_iota_noalloc(int ndim, const int* grid, const int* K, const void* a, int ncomp,
                                  void* f_out, void* stream) {
  using namespace lddmm;
  if ((ndim != 2 && ndim != 3) || !grid || !K || !a || !f_out || ncomp < 1 || ncomp > kMaxIota)
    return LDDMM_EINVAL;
  for (int j = 0; j < ndim; ++j)
    if (grid[j] < 2 || K[j] < 2 || (K[j] & 1) || K[j] > grid[j] || grid[j] > (1 << 16))
      return LDDMM_EINVAL;
  const Dims N{grid[0], grid[1], ndim == 3 ? grid[2] : 1};
  Band b;
  b.k1 = K[0];
  b.k2 = K[1];
  b.k3 = ndim == 3 ? K[2] : 1;
  b.h1 = b.k1 / 2;
  const size_t c8 = sizeof(float2);
  const size_t s3 = align256((size_t)b.k3 * N.n3 * c8), s2 = align256((size_t)b.k2 * N.n2 * c8),
               s1 = align256((size_t)b.h1 * N.n1 * c8), sh = align256((size_t)ncomp * b.vol() * c8),
               st2 = align256((size_t)ncomp * b.h1 * N.n2 * N.n3 * c8);
  if (s3 + s2 + s1 + sh + st2 > kNoAllocBytes) return LDDMM_ENOMEM;

  // an error left pending by earlier work of the caller is not this call's:
  // report it without launching anything (and leave it for the caller)
  if (cudaPeekAtLastError() != cudaSuccess) return LDDMM_ECUDA;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return LDDMM_ECUDA;
  }
  DeviceScratch& ds = g_scratch_of[dev];
  std::call_once(ds.once, [&] {
    ds.err = cudaGetSymbolAddress(reinterpret_cast<void**>(&ds.ptr), g_noalloc_scratch);
  });
  if (ds.err != cudaSuccess || !ds.ptr) return LDDMM_ECUDA;
  if (!is_device_pointer(a, dev) || !is_device_pointer(f_out, dev)) return LDDMM_EINVAL;

  unsigned char* base = ds.ptr;
  CPlan p{};
  p.g = N;
  p.b = b;
  p.E3f = reinterpret_cast<float2*>(base);
  p.E2f = reinterpret_cast<float2*>(base + s3);
  p.E1f = reinterpret_cast<float2*>(base + s3 + s2);
  float2* herm = reinterpret_cast<float2*>(base + s3 + s2 + s1);
  float2* T2 = reinterpret_cast<float2*>(base + s3 + s2 + s1 + sh);
  if (!sizes_accepted<float>(N, b, 1, false)) return LDDMM_EINVAL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);

  const long long ntw = (long long)b.k3 * N.n3 + (long long)b.k2 * N.n2 + (long long)b.h1 * N.n1;
  k_iota_twiddles<<<(unsigned)((ntw + 255) / 256), 256, 0, st>>>(p.E3f, p.E2f, p.E1f, b, N);
  const long long nb = (long long)ncomp * b.vol();
  if (cudaGetLastError() != cudaSuccess) return LDDMM_ECUDA;   // nothing further is enqueued
  const float2* in = static_cast<const float2*>(a);
  cudaError_t e = run(k_hermitianize, (nb + kThr - 1) / kThr, 0, st, in, herm, ncomp, b);
  const size_t G2e = even_up(N.n2), G3e = even_up(N.n3);
  const size_t s0 = ((size_t)even_up(b.k2 * b.k3) + b.k2 * G3e) * c8, tw = (b.k3 * G3e + b.k2 * G2e) * c8;
  const long long slabs = (long long)ncomp * b.h1, pencils = ncomp * (((long long)N.n2 * N.n3 + kThr - 1) / kThr);
  if (e == cudaSuccess)
    e = s0 + tw <= (size_t)64 * 1024 ? run(k_slab<true>, slabs, s0 + tw, st, p, herm, T2)
                                     : run(k_slab<false>, slabs, s0, st, p, herm, T2);
  const size_t se = (size_t)b.h1 * N.n1 * c8;
  float* out = static_cast<float*>(f_out);
  if (e == cudaSuccess)
    e = b.h1 <= 8 ? run(k_pencil<8>, pencils, se, st, p, T2, out)
                  : (b.h1 <= 16 ? run(k_pencil<16>, pencils, se, st, p, T2, out)
                                : run(k_pencil<kMaxH1>, pencils, se, st, p, T2, out));
  return cudaGetLastError() == cudaSuccess ? LDDMM_OK : LDDMM_ECUDA;
}
