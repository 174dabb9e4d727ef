// Device bodies of a pseudo-spectral evaluation on the padded product grid
// (brackets of Eqs. 4, 48, 49 and the deformation products, with the truncated
// transforms of Eq. 46), shared by the stand-alone kernels (dft.cu) and the
// persistent sweep kernel (sweep.cu).
//
// A band-limited field is a tensor of real cosine/sine coefficients, and each
// transform is a real tensor contraction, one axis after another.  The k1 -> x1
// contraction comes first on the way to the grid and last on the way back, so
// an evaluation has two phases and two transposes:
//
//   band phase   item = tq quads (a, b) of axes 2 and 3, all k1, all fields:
//                x1 -> k1 of the product fields, the epilogue (K~, derivative of
//                the scalar products, Heun / Krylov combination: all local to a
//                quad), the spectral multipliers of the next evaluation's fields
//                and their k1 -> x1.
//   plane phase  item = part of one x1 plane (ppc pairs of rows x2, G2 - x2):
//                k2 -> x2 and k3 -> x3 of every field, the point products, and
//                x3 -> k3, x2 -> k2 back (a partial sum over the item's rows).
//
// Cosines are even and sines odd in x, so the points x and G - x share one sum of
// K/2 cosine and one of K/2 sine products (f = E + O and E - O), and on the way
// back the folded inputs f(x) +- f(G - x) are summed over half the axis: half of
// the products of the plain real sums, a quarter of the complex half-spectrum
// form.  (cos, sin) data and twiddles sit side by side, so one packed two-wide
// FMA advances both sums.
#pragma once

#include <algorithm>
#include <type_traits>

#include "internal.h"

namespace lddmm {
namespace dev {

constexpr double kTwoPi = 6.283185307179586476925286766559;
constexpr int kMaxSmem = 224 * 1024;
// FP32 sums back to the band are split over interleaved accumulators (four in k_pi_band): a
// sum of like signs (an image, the lowest frequencies) loses about the square root of a
// third of its length in roundings, and half of that in two halves.  Relative errors at
// 64^3, band 16^3: projection of images 1.24e-7 to 7.7e-8, ad~^dagger 1.49e-7 to 1.40e-7
// (complex half-spectrum sums: 7.4e-8 and 1.35e-7).  It costs no time, the chains being
// shorter; sums in blocks of eight, added to a total, cost 1-2% of a product.
template <typename T> constexpr int kSplit = sizeof(T) == 4 ? 2 : 1;
constexpr int kSMs = 152;   // sizing only: fixed, so that sums never depend on the device
// Threads of the two phases.  The contractions are bound by issue slots and by the
// register write-back of shared-memory reads (one pair per lane costs two packed
// FMAs), so a thread takes a register tile of several sums.
constexpr int kPhaseThreads = 256;
// Plane phase: on large items enough warps to overlap one's reads with another's
// sums (us per evaluation at 256 / 512 threads: band 32^3 19.5 / 18.7, 64^3 166 /
// 161); small ones have work for 256 only (16^3 9.8 / 10.3).
template <typename T> __host__ __device__ constexpr int plane_threads(int PT) { return sizeof(T) == 4 && PT > 5 ? 512 : 256; }

// Programmatic dependent launch: a kernel launched with programmatic stream
// serialisation may start while its predecessor runs; it stages its constant
// tables first and waits here before touching anything an earlier kernel wrote.
// Without that launch attribute (and inside the persistent sweep) it returns at once.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// lets the next kernel of the stream be scheduled (it still waits in pdl_wait)
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- pairs -------------------------------------------------------------------
// float pairs live in one 64-bit register pair, the operand of fma.rn.f32x2
template <typename T> struct V2;
template <> struct V2<float> { unsigned long long v; };
template <> struct alignas(16) V2<double> { double a, b; };

__device__ __forceinline__ V2<float> mk2(float x, float y) {
  V2<float> r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ V2<double> mk2(double x, double y) { return V2<double>{x, y}; }
__device__ __forceinline__ void un2(V2<float> p, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(p.v));
}
__device__ __forceinline__ void un2(V2<double> p, double& x, double& y) {
  x = p.a;
  y = p.b;
}
__device__ __forceinline__ V2<float> fma2(V2<float> a, V2<float> b, V2<float> c) {
  V2<float> r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ V2<double> fma2(V2<double> a, V2<double> b, V2<double> c) {
  return V2<double>{fma(a.a, b.a, c.a), fma(a.b, b.b, c.b)};
}
__device__ __forceinline__ V2<float> sum2(V2<float> a, V2<float> b) {
  V2<float> r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ V2<double> sum2(V2<double> a, V2<double> b) { return V2<double>{a.a + b.a, a.b + b.b}; }
template <typename T> __device__ __forceinline__ V2<T> zero2();
template <> __device__ __forceinline__ V2<float> zero2<float>() { return V2<float>{0ull}; }
template <> __device__ __forceinline__ V2<double> zero2<double>() { return V2<double>{0.0, 0.0}; }
// two consecutive pairs (16-byte aligned for float)
__device__ __forceinline__ void ld2(const V2<float>* p, V2<float>& a, V2<float>& b) {
  const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(p);
  a.v = q.x;
  b.v = q.y;
}
__device__ __forceinline__ void ld2(const V2<double>* p, V2<double>& a, V2<double>& b) {
  a = p[0];
  b = p[1];
}
// four consecutive reals of a quad: pairs (s2 = 0, 1) of s3 = 0 and of s3 = 1
template <typename T>
struct Quad {
  V2<T> c, s;
};
__device__ __forceinline__ Quad<float> ldq(const float* p) {
  const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(p);
  return Quad<float>{{q.x}, {q.y}};
}
__device__ __forceinline__ Quad<double> ldq(const double* p) {
  return Quad<double>{{p[0], p[1]}, {p[2], p[3]}};
}
__device__ __forceinline__ void stq(float* p, const Quad<float>& q) {
  ulonglong2 v;
  v.x = q.c.v;
  v.y = q.s.v;
  *reinterpret_cast<ulonglong2*>(p) = v;
}
__device__ __forceinline__ void stq(double* p, const Quad<double>& q) {
  p[0] = q.c.a;
  p[1] = q.c.b;
  p[2] = q.s.a;
  p[3] = q.s.b;
}

__host__ __device__ __forceinline__ int up4(int n) { return (n + 3) & ~3; }
__host__ __device__ __forceinline__ int up2(int n) { return n + (n & 1); }
__host__ __device__ __forceinline__ int up8(int n) { return (n + 7) & ~7; }

// n pairs global -> shared by all threads
template <typename T, int NT>
__device__ __forceinline__ void copy2(V2<T>* dst, const Pair<T>* src, int n) {
  const V2<T>* s = reinterpret_cast<const V2<T>*>(src);
  for (int i = threadIdx.x; i < n; i += NT) dst[i] = s[i];
}

// x / n for the kernels' index splits (exact while x * n < 2^32)
__device__ __forceinline__ int fdiv(int x, FastDiv d) { return d.m ? (int)__umulhi((unsigned)x, d.m) : x; }

// ============================================================================
// band phase
// ============================================================================
// Register tiles: HG k1 frequencies (x1 -> k1) or TG folded x1 points (k1 -> x1) of
// CP columns per thread.  A double FMA occupies its pipe for 64 cycles a warp
// whatever the lanes do, so double takes the most threads, one sum each.
template <typename T> struct BandTile { static constexpr int HG = 4, TG = 8, CP = 2; };
template <> struct BandTile<double> { static constexpr int HG = 1, TG = 1, CP = 1; };

template <typename T>
struct BandShape {
  int H1p, NT1p;            // table rows padded to kHG frequencies and kTG points
  int off_f, off_e, off_y;  // pair offsets: e1f table (e1b at 0), folded inputs / field coefficients, projections
  size_t smem;
};
template <typename T>
__host__ __device__ inline BandShape<T> band_shape(const Plan<T>& p, int tq, int NO, int NF) {
  BandShape<T> s;
  const int PC = 4 * tq, H1 = p.k.H1;
  s.H1p = up4(H1);
  s.NT1p = up8(p.NT1);
  s.off_f = up2(p.NT1 * s.H1p);
  s.off_e = up2(s.off_f + H1 * s.NT1p);
  const int e = NO * p.NT1, g = NF * H1;
  s.off_y = s.off_e + (e > g ? e : g) * PC;
  s.smem = (size_t)up2(s.off_y + NO * H1 * PC) * sizeof(V2<T>);
  return s;
}

// N sums of NS accumulators each (acc [NS][N]) into the first
template <typename T, int NS, int N>
__device__ __forceinline__ void add_sums(V2<T>* acc) {
  if constexpr (NS == 4) {
#pragma unroll
    for (int i = 0; i < 2 * N; ++i) acc[i] = sum2(acc[i], acc[2 * N + i]);
  }
  if constexpr (NS > 1) {
#pragma unroll
    for (int i = 0; i < N; ++i) acc[i] = sum2(acc[i], acc[N + i]);
  }
}

template <typename T>
__device__ __forceinline__ V2<T> scale2(V2<T> p, T s) {
  T a, b;
  un2(p, a, b);
  return mk2(a * s, b * s);
}
// p + s q
template <typename T>
__device__ __forceinline__ V2<T> add2(V2<T> p, V2<T> q, T s) {
  return fma2(q, mk2(s, s), p);
}
template <typename T>
__device__ __forceinline__ V2<T> shfl2(V2<T> p, int bit) {
  T a, b;
  un2(p, a, b);
  return mk2(__shfl_xor_sync(0xffffffffu, a, bit), __shfl_xor_sync(0xffffffffu, b, bit));
}
// d_1 of a coefficient pair (cos, sin over k1) at frequency h
template <typename T>
__device__ __forceinline__ V2<T> d1(V2<T> u, T w) {
  T x, y;
  un2(u, x, y);
  return mk2(w * y, -(w * x));
}

// the coefficients of mode MODE's input fields at one (h, column), from the
// sources' coefficients A and m = L~B there and at the partner columns (lanes
// whose columns differ in the cos/sin bit of axis 2 or 3); w: 2 pi times the
// frequencies, with the sign of this column's partner for axes 2 and 3
template <typename T, int MODE, bool FLAT>
__device__ __forceinline__ void mode_fields(const V2<T>* A, const V2<T>* m, const T* w, V2<T>* dst, int stride) {
  if constexpr (FLAT) {
    V2<T> D[2][2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      D[c][0] = d1<T>(A[c], w[0]);
      D[c][1] = scale2<T>(shfl2<T>(A[c], 1), w[1]);
    }
    int f = 0;
    if (MODE < PW_D0) {
      dst[f++ * stride] = A[0];
      dst[f++ * stride] = A[1];
    }
    if (MODE == PW_T) {
      dst[f++ * stride] = add2<T>(D[0][0], D[1][1], T(1));
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) dst[f++ * stride] = D[i / 2][i % 2];
    }
    dst[f++ * stride] = m[0];
    dst[f++ * stride] = m[1];
    const V2<T> m0y = scale2<T>(shfl2<T>(m[0], 1), w[1]);
    if (MODE < PW_D0) dst[f++ * stride] = add2<T>(d1<T>(m[1], w[0]), m0y, T(-1));
    return;
  }
  V2<T> DA[3][3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    DA[c][0] = d1<T>(A[c], w[0]);
    DA[c][1] = scale2<T>(shfl2<T>(A[c], 1), w[1]);
    DA[c][2] = scale2<T>(shfl2<T>(A[c], 2), w[2]);
  }
  int f = 0;
  if (MODE >= PW_D0) {                                    // DA, B
#pragma unroll
    for (int i = 0; i < 9; ++i) dst[f++ * stride] = DA[i / 3][i % 3];
#pragma unroll
    for (int c = 0; c < 3; ++c) dst[f++ * stride] = m[c];
    return;
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) dst[f++ * stride] = A[c];
  if constexpr (MODE == PW_T) {
    dst[f++ * stride] = add2<T>(add2<T>(DA[0][0], DA[1][1], T(1)), DA[2][2], T(1));
  } else {
#pragma unroll
    for (int i = 0; i < 9; ++i) dst[f++ * stride] = DA[i / 3][i % 3];
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) dst[f++ * stride] = m[c];
  V2<T> M1[3], M2[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    M1[c] = scale2<T>(shfl2<T>(m[c], 1), w[1]);
    M2[c] = scale2<T>(shfl2<T>(m[c], 2), w[2]);
  }
  dst[f++ * stride] = add2<T>(M1[2], M2[1], T(-1));        // curl m
  dst[f++ * stride] = add2<T>(M2[0], d1<T>(m[2], w[0]), T(-1));
  dst[f++ * stride] = add2<T>(d1<T>(m[1], w[0]), M1[0], T(-1));
}

// fold x1 of NO product fields (sums of nparts partial planes) for nq quads from
// q0: sE [NO][nt][PC], points t0 .. t0 + nt
template <typename T, int NT>
__device__ __forceinline__ void fold_planes(const Plan<T>& p, const T* P1, int NO, int nparts, int q0, int nq, int tqs,
                                            int t0, int nt, FastDiv dnt, V2<T>* sE) {
  const int G1 = p.g.n1, PC = 4 << tqs;
  const long long Kq = p.k.Kq(), pstride = NO * Kq * 4;   // pstride: one partial plane
  // A lane sums one side (x or G1 - x) of one (field, point, quad); neighbouring lanes
  // hold the two sides, exchange half of their sums and fold one pair of columns
  // each.  Two sums per thread and round, four partial planes of each in flight.
  const int n = (NO * nt) << (tqs + 1), side = threadIdx.x & 1;
  for (int i0 = 0; i0 < n; i0 += 2 * NT) {
    const T* a[2];
    V2<T>* d[2];
    bool two[2], live[2];
    V2<T> c[2], q[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int it = i0 + j * NT + (int)threadIdx.x, ix = min(it, n - 1) >> 1;
      const int ql = ix & ((1 << tqs) - 1), r = ix >> tqs;
      const int o = fdiv(r, dnt), t = r - o * nt, x = t0 + t;
      live[j] = it < n && ql < nq;
      two[j] = x > 0 && 2 * x != G1;
      a[j] = P1 + (long long)(side && two[j] ? G1 - x : x) * nparts * pstride +
             ((long long)o * Kq + q0 + min(ql, nq - 1)) * 4;
      d[j] = sE + (o * nt + t) * PC + 4 * ql + 2 * side;
      c[j] = q[j] = zero2<T>();
    }
    for (int k0 = 0; k0 < nparts; k0 += 4) {
      Quad<T> u[2][4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k0 + k < nparts) {
#pragma unroll
          for (int j = 0; j < 2; ++j) u[j][k] = ldq(a[j] + (k0 + k) * pstride);
        }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k0 + k < nparts) {
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            c[j] = sum2(c[j], u[j][k].c);
            q[j] = sum2(q[j], u[j][k].s);
          }
        }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const V2<T> got = shfl2<T>(side ? c[j] : q[j], 1);   // the other side of this lane's columns
      const V2<T> near = side ? got : c[j], far = side ? q[j] : got;
      T u0, u1, v0, v1;
      un2(near, u0, u1);                                   // side 0: x in near; side 1: x in got
      un2(far, v0, v1);
      if (live[j]) {
        d[j][0] = two[j] ? mk2(u0 + v0, u0 - v0) : mk2(u0, T(0));
        d[j][1] = two[j] ? mk2(u1 + v1, u1 - v1) : mk2(u1, T(0));
      }
    }
  }
}

// x1 -> k1 of the folded inputs sE [NO][nt][PC] with the table sW [nt][H1p], into
// (add: onto) sY [NO][H1][PC]; NS accumulators (kSplit)
template <typename T, int NT, bool FLAT, int NS>
__device__ __forceinline__ void contract_k1(const Plan<T>& p, int NO, int nt, int tqs, int H1p, const V2<T>* sE,
                                            const V2<T>* sW, bool add, V2<T>* sY) {
  constexpr int HG = BandTile<T>::HG, CP = BandTile<T>::CP;
  const int PC = 4 << tqs, H1 = p.k.H1, ng = (H1 + HG - 1) / HG;
  // columns in groups of CP (flat: the first two of every quad)
  const int cs = tqs + (FLAT ? 1 : 2) - (CP == 2 ? 1 : 0);
  for (int it = threadIdx.x; it < (NO * ng) << cs; it += NT) {
    const int ci = (it & ((1 << cs) - 1)) * CP, r = it >> cs;
    const int col = FLAT ? (ci >> 1) * 4 + (ci & 1) : ci;
    const int o = HG == 1 ? fdiv(r, p.dH1) : fdiv(r, p.dH1g), g = r - o * ng;
    const V2<T>* v = sE + o * nt * PC + col;
    const V2<T>* w = sW + g * HG;
    V2<T> acc[NS][HG][CP];
#pragma unroll
    for (int i = 0; i < NS * HG * CP; ++i) acc[i / (HG * CP)][i / CP % HG][i % CP] = zero2<T>();
    auto term = [&](int t, V2<T>(&sum)[HG][CP]) {
      V2<T> u[2];
      if (CP == 2) ld2(v + t * PC, u[0], u[1]);
      else u[0] = v[t * PC];
#pragma unroll
      for (int i = 0; i < HG; i += 2) {
        V2<T> w0, w1;
        if (HG > 1) ld2(w + t * H1p + i, w0, w1);
        else w0 = w[t * H1p];
#pragma unroll
        for (int c = 0; c < CP; ++c) {
          sum[i][c] = fma2(u[c], w0, sum[i][c]);
          if (HG > 1) sum[i + (HG > 1)][c] = fma2(u[c], w1, sum[i + (HG > 1)][c]);
        }
      }
    };
    if constexpr (NS == 1) {
#pragma unroll 4
      for (int t = 0; t < nt; ++t) term(t, acc[0]);
    } else if constexpr (NS == 2) {
      int t = 0;
#pragma unroll 2
      for (; t + 2 <= nt; t += 2) {
        term(t, acc[0]);
        term(t + 1, acc[1]);
      }
      if (t < nt) term(t, acc[0]);
    } else {
      int t = 0;
#pragma unroll 1
      for (; t + NS <= nt; t += NS)
#pragma unroll
        for (int k = 0; k < NS; ++k) term(t + k, acc[k]);
#pragma unroll 1
      for (; t < nt; ++t) term(t, acc[0]);
    }
    add_sums<T, NS, HG * CP>(&acc[0][0][0]);
#pragma unroll
    for (int i = 0; i < HG; ++i) {
      const int h = g * HG + i;
      if (h >= H1) break;
      V2<T>* y = sY + (o * H1 + h) * PC + col;
#pragma unroll
      for (int c = 0; c < CP; ++c) y[c] = add ? sum2(y[c], acc[0][i][c]) : acc[0][i][c];
    }
  }
}

// k1 -> x1 of the fields sG [NF][H1][PC] of nq quads from q0, folded points t0 ..
// t0 + nt (table sF [H1][ntp]): field f to plane field f0 + f of T1 [x1][nf][Kq][4]
template <typename T, int NT, bool FLAT>
__device__ __forceinline__ void band_to_planes(const Plan<T>& p, const V2<T>* sG, const V2<T>* sF, int NF, int f0,
                                               int nf, int q0, int nq, int tqs, int t0, int nt, int ntp, T* T1) {
  constexpr int TG = BandTile<T>::TG, CP = BandTile<T>::CP;
  const int H1 = p.k.H1, G1 = p.g.n1, PC = 4 << tqs, ng = (nt + TG - 1) / TG;
  const long long Kq = p.k.Kq();
  // (field, point group) pairs in lockstep: a thread's next pair by addition
  const int cs = tqs + (FLAT ? 1 : 2) - (CP == 2 ? 1 : 0);
  const int first = threadIdx.x >> cs, step = NT >> cs, dg = step / NF, df = step - dg * NF;
  int g = first / NF, f = first - g * NF;
  const int ci = (threadIdx.x & ((1 << cs) - 1)) * CP, col = FLAT ? (ci >> 1) * 4 + (ci & 1) : ci;
  if (col >= 4 * nq) return;
  const long long plane = nf * Kq * 4;
  while (g < ng) {
    const V2<T>* v = sG + f * H1 * PC + col;
    const V2<T>* w = sF + g * TG;
    V2<T> acc[TG][CP];
#pragma unroll
    for (int i = 0; i < TG; ++i)
#pragma unroll
      for (int c = 0; c < CP; ++c) acc[i][c] = zero2<T>();
#pragma unroll 4
    for (int h = 0; h < H1; ++h) {
      V2<T> u[2];
      if (CP == 2) ld2(v + h * PC, u[0], u[1]);
      else u[0] = v[h * PC];
#pragma unroll
      for (int i = 0; i < TG; i += 2) {
        V2<T> w0, w1;
        if (TG > 1) ld2(w + h * ntp + i, w0, w1);
        else w0 = w[h * ntp];
#pragma unroll
        for (int c = 0; c < CP; ++c) {
          acc[i][c] = fma2(u[c], w0, acc[i][c]);
          if (TG > 1) acc[i + (TG > 1)][c] = fma2(u[c], w1, acc[i + (TG > 1)][c]);
        }
      }
    }
    const int tb = t0 + g * TG;
    T* up = T1 + ((long long)(f0 + f) * Kq + q0) * 4 + col + tb * plane;
    T* dn = T1 + ((long long)(f0 + f) * Kq + q0) * 4 + col + (G1 - tb) * plane;
#pragma unroll
    for (int i = 0; i < TG; ++i) {
      const int t = tb + i;
      if (g * TG + i >= nt) break;
      const bool two = t > 0 && 2 * t != G1;
      T E[2], O[2];
#pragma unroll
      for (int c = 0; c < CP; ++c) un2(acc[i][c], E[c], O[c]);
      if (CP == 2) {
        *reinterpret_cast<V2<T>*>(up) = mk2(E[0] + O[0], E[1] + O[1]);
        if (two) *reinterpret_cast<V2<T>*>(dn) = mk2(E[0] - O[0], E[1] - O[1]);
      } else {
        *up = E[0] + O[0];
        if (two) *dn = E[0] - O[0];
      }
      up += plane;
      dn -= plane;
    }
    f += df;
    g += dg;
    if (f >= NF) {
      f -= NF;
      ++g;
    }
  }
}

// whether band-phase items of 2^tqs quads share an SM (FP32: more items than SMs)
// and then have the registers for one accumulator (two spill: band 64^3 0.7% slower)
template <typename T>
__host__ __device__ __forceinline__ bool shared_sms(const Plan<T>& p, int tqs) {
  return sizeof(T) == 4 && !p.flat && (p.k.Kq() >> tqs) > kSMs;
}

// one band-phase item of mode MODE: e != nullptr, the previous evaluation's
// projection and epilogue; A != nullptr, the fields of the next evaluation
template <typename T, int MODE, int NT, bool FLAT, int NS>
__device__ __forceinline__ void band_item(const Plan<T>& p, int tqs, const PiEpi<T>* e, int nparts, const T* P1,
                                          const T* A, const T* B, T* T1, const T* __restrict__ Lhat, int item,
                                          V2<T>* sm) {
  constexpr int NO = fields_out(MODE, FLAT), NF = fields_in(MODE, FLAT), C = FLAT ? 2 : 3;
  const int tq = 1 << tqs, PC = 4 << tqs, q0 = item << tqs, nq = min(tq, p.k.Kq() - q0), H1 = p.k.H1;
  const long long Kq = p.k.Kq(), kvol = Kq * H1 * 4;       // pairs of one component
  const BandShape<T> s = band_shape(p, tq, NO, NF);
  V2<T>*sB = sm, *sF = sm + s.off_f, *sE = sm + s.off_e, *sG = sE, *sY = sm + s.off_y;
  copy2<T, NT>(sB, p.e1b, p.NT1 * s.H1p);
  copy2<T, NT>(sF, p.e1f, H1 * s.NT1p);
  // this thread's coefficients: frequency h, column col of all components (threads
  // past H1 PC compute along with the last one, for the lane exchanges)
  const bool mine = (int)threadIdx.x < H1 * PC && (threadIdx.x & (PC - 1)) < 4 * nq;
  const int col = mine ? threadIdx.x & (PC - 1) : threadIdx.x & 3, h = mine ? threadIdx.x >> (tqs + 2) : 0;
  const int ql = col >> 2, sc = col & 3, q = q0 + ql, K3h = p.k.K3h, a = fdiv(q, p.dK3h), b = q - a * K3h;
  const long long at = ((long long)q * H1 + h) * 4 + sc;
  const T w[3] = {T(kTwoPi) * T(h), T(kTwoPi) * T(a) * ((sc & 1) ? T(-1) : T(1)),
                  T(kTwoPi) * T(b) * ((sc & 2) ? T(-1) : T(1))};
  const T L = Lhat[2 * at];
  pdl_wait();
  V2<T> vA[3], vB[3];
  if (e != nullptr) {
    // the epilogue's terms, in flight during the projection
    V2<T> X[kMaxTerm][3];
#pragma unroll
    for (int k = 0; k < kMaxTerm; ++k)
      if (k < e->nterm) {
        const V2<T>* x = reinterpret_cast<const V2<T>*>(e->X[k]) + at;
#pragma unroll
        for (int c = 0; c < C; ++c) X[k][c] = x[c * kvol];
      }
    if (A != nullptr && e->jA < 0) {
#pragma unroll
      for (int c = 0; c < C; ++c) vA[c] = reinterpret_cast<const V2<T>*>(A)[c * kvol + at];
    }
    if (A != nullptr && e->jB < 0) {
#pragma unroll
      for (int c = 0; c < C; ++c) vB[c] = reinterpret_cast<const V2<T>*>(B)[c * kvol + at];
    }
    fold_planes<T, NT>(p, P1, NO, nparts, q0, nq, tqs, 0, p.NT1, p.dNT1, sE);
    __syncthreads();
    contract_k1<T, NT, FLAT, NS>(p, NO, p.NT1, tqs, s.H1p, sE, sB, false, sY);
    __syncthreads();
    const bool dead2 = (a == 0 && (sc & 1)) || (b == 0 && (sc & 2));
    const T fac = dead2 ? T(0) : (h ? T(2) : T(1)) * (a ? T(2) : T(1)) * (b ? T(2) : T(1));
    const T kh = T(1) / L;
    const V2<T> f2 = mk2(fac, h ? fac : T(0));             // the sine slot of h = 0 is dead
    V2<T> yo[kMaxPer][3];
    const V2<T>* y = sY + h * PC + col;
    const int fs = H1 * PC, c1 = (col ^ 1) - col, c2 = (col ^ 2) - col;
#pragma unroll
    for (int o = 0; o < mode_nper(MODE); ++o)
#pragma unroll
      for (int c = 0; c < C; ++c) {
        V2<T> v;
        if (MODE >= PW_D0) {
          v = y[c * fs];
        } else if (o == 2) {
          v = y[(FLAT ? 6 + c : 8 + c) * fs];
        } else {                                           // grad of the scalar product + vector
          const V2<T>* g = y + (C + 1) * o * fs;
          const V2<T> d = c == 0 ? d1<T>(g[0], w[0]) : scale2<T>(g[c == 1 ? c1 : c2], w[c]);
          v = add2<T>(g[(1 + c) * fs], d, T(1));
        }
        T v0, v1, f0, f1;
        un2(v, v0, v1);
        un2(f2, f0, f1);
        yo[o][c] = mk2(f0 != T(0) ? f0 * v0 : T(0), f1 != T(0) ? f1 * v1 : T(0));
      }
#pragma unroll
    for (int j = 0; j < kMaxOut; ++j) {
      if (j >= e->nout) break;
      V2<T> v[3];
#pragma unroll
      for (int c = 0; c < C; ++c) v[c] = zero2<T>();
#pragma unroll
      for (int o = 0; o < mode_nper(MODE); ++o)
        if (e->cY[j][o] != T(0)) {
          const T cy = e->cY[j][o] * (e->applyK[o] ? kh : T(1));
#pragma unroll
          for (int c = 0; c < C; ++c) v[c] = add2<T>(v[c], yo[o][c], cy);
        }
#pragma unroll
      for (int k = 0; k < kMaxTerm; ++k)
        if (e->cX[j][k] != T(0)) {
#pragma unroll
          for (int c = 0; c < C; ++c) v[c] = add2<T>(v[c], X[k][c], e->cX[j][k]);
        }
      V2<T>* dst = reinterpret_cast<V2<T>*>(e->dst[j]) + at;
#pragma unroll
      for (int c = 0; c < C; ++c) {
        if (mine) dst[c * kvol] = v[c];
        if (j == e->jA) vA[c] = v[c];
        if (j == e->jB) vB[c] = v[c];
      }
      if (FLAT && mine) dst[2 * kvol] = zero2<T>();
    }
  } else {
#pragma unroll
    for (int c = 0; c < C; ++c) {
      vA[c] = reinterpret_cast<const V2<T>*>(A)[c * kvol + at];
      vB[c] = reinterpret_cast<const V2<T>*>(B)[c * kvol + at];
    }
    __syncthreads();
  }
  if (A == nullptr) return;
  if (MODE < PW_D0) {
#pragma unroll
    for (int c = 0; c < C; ++c) vB[c] = scale2<T>(vB[c], L);
  }
  // (inactive threads write into their own thread's column of a spare row: none,
  // they only take part in the lane exchanges)
  {
    V2<T> fld[NF];
    mode_fields<T, MODE, FLAT>(vA, vB, w, fld, 1);
    if (mine) {
#pragma unroll
      for (int f = 0; f < NF; ++f) sG[(f * H1 + h) * PC + col] = fld[f];
    }
  }
  __syncthreads();
  band_to_planes<T, NT, FLAT>(p, sG, sF, NF, 0, NF, q0, nq, tqs, 0, p.NT1, s.NT1p, T1);
}

// ============================================================================
// plane phase
// ============================================================================
template <typename T>
struct PlaneShape {
  int R, ppe, K3s;          // rows (2 ppc), row stride of the x2 twiddles, row stride of the k3 rows
  int off_3b, off_2f, off_2b, off_s, off_p;   // pair offsets
  size_t smem;
};
// PT: row pairs per thread of k2 -> x2.  (K3s = K3e + 2 keeps the rows that one
// warp reads in different banks.)
template <typename T>
__host__ __device__ inline PlaneShape<T> plane_shape(const Plan<T>& p, int NF, int NO, int ppc, int PT) {
  PlaneShape<T> s;
  s.R = 2 * ppc;
  s.ppe = (ppc + PT - 1) / PT * up2(PT);
  s.K3s = p.K3e + 2;
  s.off_3b = NF > 0 ? up2(p.K3e * p.NT3) : 0;
  s.off_2f = up2(s.off_3b + (NO > 0 ? p.NT3e * p.K3e : 0));
  s.off_2b = up2(s.off_2f + (NF > 0 ? p.k.K2h * s.ppe : 0));
  s.off_s = up2(s.off_2b + (NO > 0 ? ppc * up8(p.k.K2h) : 0));
  const int s1 = NF * s.R * s.K3s, z = NO * s.R * p.K3e;   // the folded k3 rows reuse the rows' place
  s.off_p = up2(s.off_s + (s1 > z ? s1 : z));
  s.smem = (size_t)up2(s.off_p + NO * s.R * p.NT3e) * sizeof(V2<T>);
  return s;
}

// k2 -> x2 of nf <= NF plane fields T1 [nf][Kq][4] for the np row pairs of tw2f
// [K2h][ppe]: rows 2 i (x2 = t) and 2 i + 1 (x2 = G2 - t) into S1 [NF][R][K3s].
// A thread sums PT row pairs of one (field, b), so the coefficients are read once.
template <typename T, int NT, int NF, int PT>
__device__ __forceinline__ void rows_from_band(const Plan<T>& p, const T* V, int nf, int np, const PlaneShape<T>& sh,
                                               const V2<T>* tw2f, V2<T>* S1) {
  constexpr int PTe = PT + (PT & 1), U = sizeof(T) == 4 ? (NF > 3 ? 16 : 8) : 4;
  const int K2h = p.k.K2h, K3h = p.k.K3h, K3e = p.K3e;
  const long long Kq = p.k.Kq();
  const int ng = (np + PT - 1) / PT;
  for (int it = threadIdx.x; it < NF * ng * K3h; it += NT) {
    const int r = fdiv(it, p.dK3h), b = it - r * K3h;
    const int g = r / NF, f = r - g * NF;
    if (f >= nf) continue;
    const T* v = V + ((long long)f * Kq + b) * 4;
    const V2<T>* w = tw2f + g * PTe;
    V2<T> c[PTe], s[PTe];
#pragma unroll
    for (int i = 0; i < PTe; ++i) c[i] = s[i] = zero2<T>();
    auto row = [&](const Quad<T>& q, const V2<T>* wa) {
#pragma unroll
      for (int i = 0; i < PT; i += 2) {
        V2<T> w0, w1;
        ld2(wa + i, w0, w1);
        c[i] = fma2(q.c, w0, c[i]);
        s[i] = fma2(q.s, w0, s[i]);
        if (i + 1 < PT) {
          c[i + 1] = fma2(q.c, w1, c[i + 1]);
          s[i + 1] = fma2(q.s, w1, s[i + 1]);
        }
      }
    };
    const int da = K3h * 4;
    int a = 0;
    auto rows = [&](auto n_) {                             // n loads in flight
      constexpr int N = decltype(n_)::value;
      for (; a + N <= K2h; a += N) {
        Quad<T> q[N];
#pragma unroll
        for (int u = 0; u < N; ++u) q[u] = ldq(v + u * da);
        v += N * da;
#pragma unroll
        for (int u = 0; u < N; ++u) row(q[u], w + u * sh.ppe);
        w += N * sh.ppe;
      }
    };
    rows(std::integral_constant<int, U>{});
    rows(std::integral_constant<int, 4>{});
    for (; a < K2h; ++a, v += da, w += sh.ppe) row(ldq(v), w);
#pragma unroll
    for (int i = 0; i < PT; ++i) {
      const int pr = g * PT + i;
      if (pr >= np) break;
      T Ec, Oc, Es, Os;
      un2(c[i], Ec, Oc);
      un2(s[i], Es, Os);
      V2<T>* d = S1 + (f * sh.R + 2 * pr) * sh.K3s + b;
      d[0] = mk2(Ec + Oc, Es + Os);
      d[sh.K3s] = mk2(Ec - Oc, Es - Os);
      if (b == K3h - 1 && K3e > K3h) d[1] = d[sh.K3s + 1] = zero2<T>();
    }
  }
}

// x2 -> k2 of the folded rows Z [NO][ppc][K3e][2] (the pairs over s2 of s3 = 0 and
// of s3 = 1) over np row pairs into (add: onto) the partial plane out [NO][Kq][4], AG
// frequencies per thread
template <typename T, int NT, int NO, int AG, int NS>
__device__ __forceinline__ void band_from_rows(const Plan<T>& p, const V2<T>* Z, int ppc, int np, const V2<T>* tw2b,
                                               T* out, bool add = false) {
  const int K2h = p.k.K2h, K2p = up8(K2h), K3h = p.k.K3h, K3e = p.K3e;
  const long long Kq = p.k.Kq();
  const int ng = (K2h + AG - 1) / AG;
  for (int it = threadIdx.x; it < NO * ng * K3h; it += NT) {
    const int r = fdiv(it, p.dK3h), b = it - r * K3h;
    const int g = r / NO, o = r - g * NO;
    const V2<T>* z = Z + (o * ppc * K3e + b) * 2;
    const V2<T>* w = tw2b + g * AG;
    V2<T> c[AG], s[AG];
#pragma unroll
    for (int i = 0; i < AG; ++i) c[i] = s[i] = zero2<T>();
    auto row = [&](V2<T>* c, V2<T>* s) {
      V2<T> qc, qs;
      ld2(z, qc, qs);
      z += 2 * K3e;
#pragma unroll
      for (int k = 0; k < AG; k += 2) {
        V2<T> w0, w1;
        ld2(w + k, w0, w1);
        c[k] = fma2(qc, w0, c[k]);
        s[k] = fma2(qs, w0, s[k]);
        c[k + 1] = fma2(qc, w1, c[k + 1]);
        s[k + 1] = fma2(qs, w1, s[k + 1]);
      }
      w += K2p;
    };
    if constexpr (NS == 1) {
#pragma unroll 3
      for (int i = 0; i < np; ++i) row(c, s);
    } else {
      V2<T> c2[AG], s2[AG];
#pragma unroll
      for (int k = 0; k < AG; ++k) c2[k] = s2[k] = zero2<T>();
#pragma unroll 2
      for (int i = 0; i < np / 2; ++i) {
        row(c, s);
        row(c2, s2);
      }
      if (np & 1) row(c, s);
#pragma unroll
      for (int k = 0; k < AG; ++k) {
        c[k] = sum2(c[k], c2[k]);
        s[k] = sum2(s[k], s2[k]);
      }
    }
    T* d = out + ((long long)o * Kq + (long long)(g * AG) * K3h + b) * 4;
#pragma unroll
    for (int k = 0; k < AG; ++k)
      if (g * AG + k < K2h) {
        if (add) {                                         // onto this thread's own sums
          const Quad<T> q = ldq(d + k * K3h * 4);
          c[k] = sum2(q.c, c[k]);
          s[k] = sum2(q.s, s[k]);
        }
        stq(d + k * K3h * 4, Quad<T>{c[k], s[k]});
      }
  }
}

// x3 -> k3 of the folded points sP [NO][R][NT3e] (table tw3b [NT3e][K3e]), then the
// fold of each row pair: Z [NO][ppc][K3e][2].  A thread takes both rows of a pair,
// two frequencies and OG fields; a self-paired x2 has one row only.
template <typename T, int NT, int NO, int OG, int NS>
__device__ __forceinline__ void rows_to_k3(const Plan<T>& p, const V2<T>* sP, int t0, int ppc, int np,
                                           const V2<T>* tw3b, V2<T>* Z) {
  constexpr int NG = (NO + OG - 1) / OG;
  const int K3e = p.K3e, NT3e = p.NT3e, G2 = p.g.n2, R = 2 * ppc;
  for (int it = threadIdx.x; it < NG * np * (K3e / 2); it += NT) {
    const int r = fdiv(it, p.dK3p), b = 2 * (it - r * (K3e / 2));
    const int i = r / NG, g = r - i * NG, t = t0 + i;
    const bool two = t > 0 && 2 * t != G2;
    const V2<T>* v = sP + (g * OG * R + 2 * i) * NT3e;
    const V2<T>* w = tw3b + b;
    const int second = two ? NT3e : 0;                     // (a missing row repeats the first)
    V2<T> acc[NS][OG][2][2];
#pragma unroll
    for (int o = 0; o < NS * OG * 4; ++o) acc[o / (OG * 4)][o / 4 % OG][o / 2 % 2][o % 2] = zero2<T>();
    for (int t3 = 0; t3 < NT3e; t3 += 2) {
      V2<T> w00, w01, w10, w11;
      ld2(w, w00, w01);
      ld2(w + K3e, w10, w11);
      w += 2 * K3e;
#pragma unroll
      for (int o = 0; o < OG; ++o) {
        if (NO % OG != 0 && g * OG + o >= NO) break;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          V2<T> a0, a1;
          ld2(v + o * R * NT3e + k * second + t3, a0, a1);
          acc[0][o][k][0] = fma2(a0, w00, acc[0][o][k][0]);
          acc[0][o][k][1] = fma2(a0, w01, acc[0][o][k][1]);
          acc[NS - 1][o][k][0] = fma2(a1, w10, acc[NS - 1][o][k][0]);
          acc[NS - 1][o][k][1] = fma2(a1, w11, acc[NS - 1][o][k][1]);
        }
      }
    }
    add_sums<T, NS, OG * 4>(&acc[0][0][0][0]);
#pragma unroll
    for (int o = 0; o < OG; ++o) {
      if (NO % OG != 0 && g * OG + o >= NO) break;
      V2<T>* z = Z + (((g * OG + o) * ppc + i) * K3e + b) * 2;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        T c1, s1, c2, s2;
        un2(acc[0][o][0][j], c1, s1);
        un2(acc[0][o][1][j], c2, s2);
        z[2 * j] = two ? mk2(c1 + c2, c1 - c2) : mk2(c1, T(0));
        z[2 * j + 1] = two ? mk2(s1 + s2, s1 - s2) : mk2(s1, T(0));
      }
    }
  }
}

// ---- point products ----------------------------------------------------------
// P(a, m) without its gradient part: -a x c + m d (c = curl m, d = div a)
template <typename T>
__device__ __forceinline__ void pvec(const T* a, const T* m, const T* c, T d, T* out) {
  out[0] += fma(m[0], d, fma(a[2], c[1], -(a[1] * c[2])));
  out[1] += fma(m[1], d, fma(a[0], c[2], -(a[2] * c[0])));
  out[2] += fma(m[2], d, fma(a[1], c[0], -(a[0] * c[1])));
}
template <typename T>
__device__ __forceinline__ T dot3(const T* a, const T* b) {
  return fma(a[0], b[0], fma(a[1], b[1], a[2] * b[2]));
}

// A stage-point slot keeps its fields point by point, so that a point is read with
// a few wide loads: [vol][12] (v, the diagonal of Dv, n, curl n: what PW_T needs),
// then [vol][6] (the rest of Dv, row by row); 12 fields (Du, v) for the deformation
// modes.
__host__ __device__ constexpr int mode_cached(int m) {
  return m == PW_T || m == PW_TC ? 12 : (m == PW_GT ? 18 : (m == PW_D1 ? 12 : 0));
}
template <int N>
__device__ __forceinline__ void ldv(const float* p, float* v) {
  if (N == 12) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float4 q = reinterpret_cast<const float4*>(p)[i];
      v[4 * i] = q.x;
      v[4 * i + 1] = q.y;
      v[4 * i + 2] = q.z;
      v[4 * i + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      const float2 q = reinterpret_cast<const float2*>(p)[i];
      v[2 * i] = q.x;
      v[2 * i + 1] = q.y;
    }
  }
}
template <int N>
__device__ __forceinline__ void ldv(const double* p, double* v) {
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = p[i];
}
template <int N>
__device__ __forceinline__ void stv(float* p, const float* v) {
  if (N == 12) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
      reinterpret_cast<float4*>(p)[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
  } else {
#pragma unroll
    for (int i = 0; i < N / 2; ++i) reinterpret_cast<float2*>(p)[i] = make_float2(v[2 * i], v[2 * i + 1]);
  }
}
template <int N>
__device__ __forceinline__ void stv(double* p, const double* v) {
#pragma unroll
  for (int i = 0; i < N; ++i) p[i] = v[i];
}
template <typename T, int MODE>
__device__ __forceinline__ void load_cached(const T* slot, long long vol, long long at, T* c) {
  if (mode_cached(MODE) >= 12) ldv<12>(slot + 12 * at, c);
  if (mode_cached(MODE) == 18) ldv<6>(slot + 12 * vol + 6 * at, c + 12);
}
// the fields x of a point as a slot keeps them
template <typename T, int MODE>
__device__ __forceinline__ void store_cached(T* slot, long long vol, long long at, const T* x) {
  if (MODE >= PW_D0) {
    stv<12>(slot + 12 * at, x);
    return;
  }
  const T a[12] = {x[0], x[1], x[2], x[3], x[7], x[11], x[12], x[13], x[14], x[15], x[16], x[17]};
  const T b[6] = {x[4], x[5], x[6], x[8], x[9], x[10]};
  stv<12>(slot + 12 * at, a);
  stv<6>(slot + 12 * vol + 6 * at, b);
}

// products of one point: x input fields, c cached fields, o outputs
template <typename T, int MODE>
__device__ __forceinline__ void products(const T* x, const T* c, T* o) {
#pragma unroll
  for (int i = 0; i < mode_out(MODE); ++i) o[i] = T(0);
  if (MODE == PW_F) {                                     // P(A, m)
    o[0] = dot3(x, x + 12);
    pvec(x, x + 12, x + 15, x[3] + x[7] + x[11], o + 1);
  } else if (MODE == PW_T || MODE == PW_TC) {             // P(A, n) + P(v, m)
    const T* m = MODE == PW_T ? x + 4 : x + 12;
    const T divA = MODE == PW_T ? x[3] : x[3] + x[7] + x[11];
    o[0] = dot3(x, c + 6) + dot3(c, m);
    pvec(x, c + 6, c + 9, divA, o + 1);
    pvec(c, m, m + 3, c[3] + c[4] + c[5], o + 1);
  } else if (MODE == PW_GT) {                             // P(v, m), P(A, n), Q(v, A)
    o[0] = dot3(c, x + 12);
    pvec(c, x + 12, x + 15, c[3] + c[4] + c[5], o + 1);
    o[4] = dot3(x, c + 6);
    pvec(x, c + 6, c + 9, x[3] + x[7] + x[11], o + 5);
    const T Dv[9] = {c[3], c[12], c[13], c[14], c[4], c[15], c[16], c[17], c[5]};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      T s = T(0);
#pragma unroll
      for (int j = 0; j < 3; ++j) s = fma(Dv[3 * i + j], x[j], fma(-x[3 + 3 * i + j], c[j], s));
      o[8 + i] = s;
    }
  } else if (MODE == PW_D0) {
#pragma unroll
    for (int i = 0; i < 3; ++i) o[i] = -(x[9 + i] + dot3(x + 3 * i, x + 9));
  } else if (MODE == PW_D1) {
#pragma unroll
    for (int i = 0; i < 3; ++i) o[i] = -(x[9 + i] + (dot3(x + 3 * i, c + 9) + dot3(c + 3 * i, x + 9)));
  } else {
#pragma unroll
    for (int i = 0; i < 3; ++i)
      o[i] = x[9 + i] + fma(x[i], x[9], fma(x[3 + i], x[10], x[6 + i] * x[11]));
  }
}

// product fields per thread of x3 -> k3: fewer on small items, for a thread per sum
__host__ __device__ constexpr int k3_fields(int NO, int PT) {
  return PT <= 3 || NO <= 4 ? 1 : (PT <= 5 ? 2 : 3);
}

// constant tables of one plane item (rows t0 .. t0 + np of axis 2)
template <typename T, int NT, int PT>
__device__ __forceinline__ void plane_tables(const Plan<T>& p, const PlaneShape<T>& s, int t0, int np, bool fwd,
                                             bool back, V2<T>* sm) {
  if (fwd) {
    constexpr int PTe = PT + (PT & 1);
    copy2<T, NT>(sm, p.e3f, p.K3e * p.NT3);
    const V2<T>* f = reinterpret_cast<const V2<T>*>(p.e2f);
    for (int a = threadIdx.x >> 3; a < p.k.K2h; a += NT / 8)
      for (int i = threadIdx.x & 7; i < s.ppe; i += 8) {
        const int g = i / PTe, k = i - g * PTe, t = g * PT + k;
        sm[s.off_2f + a * s.ppe + i] = k < PT && t < np ? f[(long long)a * p.NT2 + t0 + t] : zero2<T>();
      }
  }
  if (back) {
    copy2<T, NT>(sm + s.off_3b, p.e3b, p.NT3e * p.K3e);
    copy2<T, NT>(sm + s.off_2b, p.e2b + (long long)t0 * up8(p.k.K2h), np * up8(p.k.K2h));
  }
}

// one plane-phase item: plane x1, row pairs [part ppc, ...)
template <typename T, int MODE, int NT, int PT>
__device__ __forceinline__ void plane_item(const Plan<T>& p, int ppc, int nparts, const T* T1, T* slot, T* slot2, T* P1,
                                           int item, V2<T>* sm) {
  constexpr int NF = mode_in(MODE), NO = mode_out(MODE), NC = mode_cached(MODE);
  const int x1 = item / nparts, part = item - x1 * nparts;
  const int t0 = part * ppc, np = min(ppc, p.NT2 - t0);
  const PlaneShape<T> s = plane_shape(p, NF, NO, ppc, PT);
  const int R = s.R, K3e = p.K3e, K3s = s.K3s, NT3 = p.NT3, NT3e = p.NT3e, G2 = p.g.n2, G3 = p.g.n3;
  const long long Kq = p.k.Kq(), vol = p.g.vol();
  V2<T>* S1 = sm + s.off_s;
  V2<T>* sP = sm + s.off_p;
  plane_tables<T, NT, PT>(p, s, t0, np, true, true, sm);
  pdl_wait();
  __syncthreads();
  rows_from_band<T, NT, NF, PT>(p, T1 + (long long)x1 * NF * Kq * 4, NF, np, s, sm + s.off_2f, S1);
  __syncthreads();
  // k3 -> x3 and the products.  Two lanes 16 apart share a row and the x3 pairs tl and
  // tl + nth: each sums half of the fields at both (a row's coefficients are then read
  // once for two points), they exchange, and each finishes one pair.  The cached
  // fields are loaded before the sums.
  constexpr int FH = NF / 2;
  static_assert(NF % 2 == 0, "fields in two halves");
  const int nth = (NT3 + 1) / 2, half = (threadIdx.x >> 4) & 1;
  const int n = 2 * np * nth;                              // (row, tl) items, 16 per warp and round
  for (int i0 = 0; i0 < n; i0 += NT / 2) {
    const int it = i0 + (threadIdx.x >> 5) * 16 + (threadIdx.x & 15);
    const int ic = min(it, n - 1), row = fdiv(ic, p.dNT3h), tl = ic - row * nth;
    const int u = t0 + (row >> 1), tm = min(tl + half * nth, NT3 - 1);   // tm: the pair this lane finishes
    const bool two = tm > 0 && 2 * tm != G3;
    const bool mine = it < n && tl + half * nth < NT3 && !((row & 1) && (u == 0 || 2 * u == G2));
    const long long at = ((long long)x1 * G2 + ((row & 1) && u > 0 ? G2 - u : u)) * G3;
    T ca[NC > 0 ? NC : 1], cb[NC > 0 ? NC : 1];
    if (NC > 0) {
      load_cached<T, MODE>(slot, vol, at + tm, ca);
      load_cached<T, MODE>(slot, vol, at + (two ? G3 - tm : tm), cb);
    }
    V2<T> acc[2][FH];
#pragma unroll
    for (int f = 0; f < FH; ++f) acc[0][f] = acc[1][f] = zero2<T>();
    const V2<T>* v = S1 + (half * FH * R + row) * K3s;
    const V2<T>* w = sm + tl;
    const int t2 = min(tl + nth, NT3 - 1) - tl;            // to the second pair
    for (int b = 0; b < K3e; b += 2) {
      const V2<T> w00 = w[0], w01 = w[t2], w10 = w[NT3], w11 = w[NT3 + t2];
      w += 2 * NT3;
#pragma unroll
      for (int f = 0; f < FH; ++f) {
        V2<T> a0, a1;
        ld2(v + f * R * K3s + b, a0, a1);
        acc[0][f] = fma2(a1, w10, fma2(a0, w00, acc[0][f]));
        acc[1][f] = fma2(a1, w11, fma2(a0, w01, acc[1][f]));
      }
    }
    T xa[NF], xb[NF];
#pragma unroll
    for (int f = 0; f < FH; ++f) {
      const V2<T> own = half ? acc[1][f] : acc[0][f], got = shfl2<T>(half ? acc[0][f] : acc[1][f], 16);
      T E, O;
      un2(half ? got : own, E, O);
      xa[f] = E + O;
      xb[f] = E - O;
      un2(half ? own : got, E, O);
      xa[FH + f] = E + O;
      xb[FH + f] = E - O;
    }
    if (!mine) continue;
    T* out = MODE == PW_F || MODE == PW_D0 ? slot : (MODE == PW_TC ? slot2 : nullptr);
    if ((MODE == PW_F || MODE == PW_D0 || MODE == PW_TC) && out != nullptr) {
      store_cached<T, MODE>(out, vol, at + tm, xa);
      if (two) store_cached<T, MODE>(out, vol, at + G3 - tm, xb);
    }
    T oa[NO], ob[NO];
    products<T, MODE>(xa, ca, oa);
    products<T, MODE>(xb, cb, ob);
    V2<T>* d = sP + row * NT3e + tm;
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      d[o * R * NT3e] = two ? mk2(oa[o] + ob[o], oa[o] - ob[o]) : mk2(oa[o], T(0));
      if (tm == NT3 - 1 && NT3e > NT3) d[o * R * NT3e + 1] = zero2<T>();
    }
  }
  __syncthreads();
  rows_to_k3<T, NT, NO, k3_fields(NO, PT), k3_fields(NO, PT) == 1 ? kSplit<T> : 1>(p, sP, t0, ppc, np, sm + s.off_3b, S1);
  __syncthreads();
  T* out = P1 + ((long long)x1 * nparts + part) * NO * Kq * 4;
  if (p.k.K2h >= 16) band_from_rows<T, NT, NO, 8, 1>(p, S1, ppc, np, sm + s.off_2b, out);
  else band_from_rows<T, NT, NO, 4, 1>(p, S1, ppc, np, sm + s.off_2b, out);
}

// ---- 2D problems ---------------------------------------------------------------
// products of one point: x and c the flat fields (c: v_1, v_2, d_1 v_1, d_2 v_2, n_1,
// n_2, (curl n)_3, d_2 v_1, d_1 v_2)
template <typename T, int MODE>
__device__ __forceinline__ void products_flat(const T* x, const T* c, T* o) {
  auto dot = [](const T* a, const T* b) { return fma(a[0], b[0], a[1] * b[1]); };
  // -a x (curl m) + m div a, in the plane
  auto vec = [](const T* a, const T* m, T curl, T div, T* r) {
    r[0] = fma(m[0], div, -(a[1] * curl));
    r[1] = fma(m[1], div, a[0] * curl);
  };
  if (MODE == PW_F) {
    o[0] = dot(x, x + 6);
    vec(x, x + 6, x[8], x[2] + x[5], o + 1);
  } else if (MODE == PW_T || MODE == PW_TC) {
    const T* m = MODE == PW_T ? x + 3 : x + 6;
    T a[2], b[2];
    o[0] = dot(x, c + 4) + dot(c, m);
    vec(x, c + 4, c[6], MODE == PW_T ? x[2] : x[2] + x[5], a);
    vec(c, m, m[2], c[2] + c[3], b);
    o[1] = a[0] + b[0];
    o[2] = a[1] + b[1];
  } else if (MODE == PW_GT) {
    o[0] = dot(c, x + 6);
    vec(c, x + 6, x[8], c[2] + c[3], o + 1);
    o[3] = dot(x, c + 4);
    vec(x, c + 4, c[6], x[2] + x[5], o + 4);
    o[6] = fma(c[2], x[0], fma(c[7], x[1], -fma(x[2], c[0], x[3] * c[1])));
    o[7] = fma(c[8], x[0], fma(c[3], x[1], -fma(x[4], c[0], x[5] * c[1])));
  } else if (MODE == PW_D0) {
    o[0] = -(x[4] + dot(x, x + 4));
    o[1] = -(x[5] + dot(x + 2, x + 4));
  } else if (MODE == PW_D1) {                              // c: D u (row by row), v
    o[0] = -(x[4] + (dot(x, c + 4) + dot(c, x + 4)));
    o[1] = -(x[5] + (dot(x + 2, c + 4) + dot(c + 2, x + 4)));
  } else {
    o[0] = x[4] + fma(x[0], x[4], x[2] * x[5]);
    o[1] = x[5] + fma(x[1], x[4], x[3] * x[5]);
  }
}
__host__ __device__ constexpr int flat_cached(int m) { return m >= PW_D0 ? 6 : 9; }   // of a slot

template <typename T>
__host__ __device__ inline size_t plane_flat_smem(int mode, int ppc) {
  const int NF = fields_in(mode, true), NO = fields_out(mode, true);
  return (size_t)NO * ppc * sizeof(V2<T>) + (size_t)(NF + NO) * 2 * ppc * sizeof(T);
}

// acc += sum of a(i) b(i), i < n, eight loads of each in flight
template <typename T, typename A, typename B>
__device__ __forceinline__ void sum_flat(int n, V2<T>& acc, A&& a, B&& b) {
  int i = 0;
  for (; i + 8 <= n; i += 8) {
    V2<T> u[8], w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      u[k] = a(i + k);
      w[k] = b(i + k);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) acc = fma2(u[k], w[k], acc);
  }
#pragma unroll 4
  for (; i < n; ++i) acc = fma2(a(i), b(i), acc);
}

// one plane item of a 2D evaluation: x2 transforms of the row pairs [part ppc, ...) of
// plane x1, one sum per thread.  Rows i and np + i are x2 = t and G2 - t.
template <typename T, int MODE, int NT>
__device__ __forceinline__ void plane_item_flat(const Plan<T>& p, int ppc, int nparts, const T* T1, T* slot, T* slot2,
                                                T* P1, int item, V2<T>* sm) {
  constexpr int NF = fields_in(MODE, true), NO = fields_out(MODE, true), NS = flat_cached(MODE);
  const int K2h = p.k.K2h, NT2 = p.NT2, G2 = p.g.n2, K2p = up8(K2h);
  const int x1 = item / nparts, t0 = (item - x1 * nparts) * ppc, np = min(ppc, NT2 - t0), R = 2 * np;
  const V2<T>*tF = reinterpret_cast<const V2<T>*>(p.e2f) + t0,
             *tB = reinterpret_cast<const V2<T>*>(p.e2b) + (long long)t0 * K2p;
  V2<T>* sE = sm;                                          // folded products [o][i]
  T *sX = reinterpret_cast<T*>(sE + NO * np), *sO = sX + NF * R;
  auto single = [&](int t) { return t == 0 || 2 * t == G2; };
  pdl_wait();
  for (int it = threadIdx.x; it < NF * np; it += NT) {
    const int f = it / np, i = it - f * np;
    const T* v = T1 + ((long long)x1 * NF + f) * K2h * 4;
    V2<T> acc = zero2<T>();
    sum_flat<T>(K2h, acc, [&](int a) { return ldq(v + 4 * a).c; }, [&](int a) { return tF[a * NT2 + i]; });
    T E, O;
    un2(acc, E, O);
    sX[f * R + i] = E + O;
    sX[f * R + np + i] = E - O;
  }
  __syncthreads();
  for (int r = threadIdx.x; r < R; r += NT) {
    const int u = t0 + (r < np ? r : r - np);
    if (r >= np && single(u)) continue;
    const long long at = (long long)x1 * G2 + (r < np ? u : G2 - u);
    T x[NF], c[NS], o[NO];
#pragma unroll
    for (int f = 0; f < NF; ++f) x[f] = sX[f * R + r];
#pragma unroll
    for (int i = 0; i < NS; ++i)
      c[i] = MODE == PW_T || MODE == PW_TC || MODE == PW_GT || MODE == PW_D1 ? slot[NS * at + i] : T(0);
    T* out = MODE == PW_F || MODE == PW_D0 ? slot : (MODE == PW_TC ? slot2 : nullptr);
    if (out != nullptr) {
      constexpr int order[9] = {0, 1, 2, 5, 6, 7, 8, 3, 4};
#pragma unroll
      for (int i = 0; i < NS; ++i) out[NS * at + i] = x[MODE >= PW_D0 ? i : (order[i] < NF ? order[i] : 0)];
    }
    products_flat<T, MODE>(x, c, o);
#pragma unroll
    for (int i = 0; i < NO; ++i) sO[i * R + r] = o[i];
  }
  __syncthreads();
  for (int it = threadIdx.x; it < NO * np; it += NT) {
    const int o = it / np, i = it - o * np;
    const T u = sO[o * R + i];
    const bool two = !single(t0 + i);
    const T v = two ? sO[o * R + np + i] : T(0);
    sE[it] = two ? mk2(u + v, u - v) : mk2(u, T(0));
  }
  __syncthreads();
  for (int it = threadIdx.x; it < NO * K2h; it += NT) {
    const int o = it / K2h, a = it - o * K2h;
    V2<T> acc = zero2<T>();
    sum_flat<T>(np, acc, [&](int i) { return sE[o * np + i]; }, [&](int i) { return tB[(long long)i * K2p + a]; });
    stq(P1 + (((long long)item * NO + o) * K2h + a) * 4, Quad<T>{acc, zero2<T>()});
  }
}

}  // namespace dev
}  // namespace lddmm
