// Internal declarations of the GB300 LDDMM library: data layouts, transform
// plans, launch descriptors and kernel launchers.  Not part of the C interface.
//
// Internally every problem is three-dimensional with three velocity
// components: a 2D problem is the slab N_3 = 1, K_3 = 1 with a zero third
// component (the 3D formulas then reduce exactly to the 2D ones).
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

namespace lddmm {

// The kernels of a bracket evaluation launch with programmatic dependent
// launch (their prologues overlap the previous kernel); building with
// -DLDDMM_NO_PDL launches them plainly (same results, for comparison).
#ifdef LDDMM_NO_PDL
constexpr bool kUsePdl = false;
#else
constexpr bool kUsePdl = true;
#endif

// Launch attributes of the bracket-evaluation chain, written from at[0]:
// programmatic stream serialisation, unless built with LDDMM_NO_PDL.
// Returns the number of attributes written (at most 1).
inline unsigned chain_attrs(cudaLaunchAttribute* at) {
  if (!kUsePdl) return 0;
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  return 1;
}

template <typename T> struct CplxOf;
template <> struct CplxOf<float> { using type = float2; };
template <> struct CplxOf<double> { using type = double2; };
template <typename T> using cplx = typename CplxOf<T>::type;

// Grid sizes of one transform plan: the image grid N or the padded product
// grid M = ceil(3K/2).
struct Dims {
  int n1, n2, n3;
  __host__ __device__ long long vol() const { return (long long)n1 * n2 * n3; }
};

// Band sizes K_j and h1 = number of non-negative k1 slots kept by the
// Hermitian half-spectrum transforms (K_1/2, or 1 for a degenerate axis).
struct Band {
  int k1, k2, k3, h1;
  __host__ __device__ long long vol() const { return (long long)k1 * k2 * k3; }
};

// ---- band vectors ------------------------------------------------------------
// A band-limited field is held as its real cosine/sine coefficients
//   f(x) = sum V[q][h][2 s3 + s2][s1] phi_s1(h x1) phi_s2(a x2) phi_s3(b x3),
// phi_0(k x) = cos(2 pi k x / G), phi_1 = sin, q = a K3h + b ("quad" of the
// non-negative frequencies a, b of axes 2 and 3), h = 0..H1-1.  The K1 K2 K3
// real degrees of freedom of a Hermitian array are stored once; the slots of
// sin(0) are dead and hold zero (they take the place of the Nyquist slots).
// A band vector is [3][Kq][H1][4][2] reals.
struct Trig {
  int H1, K2h, K3h;   // non-negative frequencies per axis (K/2; 1 for a degenerate axis)
  __host__ __device__ int K1() const { return 2 * H1; }
  __host__ __device__ int Kq() const { return K2h * K3h; }
  __host__ __device__ long long vol() const { return (long long)Kq() * 2 * H1 * 4; }
};
__host__ __device__ inline Trig trig_of(const Band& b) { return Trig{b.h1, b.k2 / 2, b.k3 > 1 ? b.k3 / 2 : 1}; }

// division by a fixed divisor n through a 32-bit reciprocal (m = 0: n = 1)
struct FastDiv {
  unsigned m;
};
inline FastDiv fast_div(int n) { return FastDiv{n <= 1 ? 0u : (unsigned)(0xffffffffu / (unsigned)n + 1u)}; }

template <typename T>
struct alignas(2 * sizeof(T)) Pair {
  T x, y;
};

// ---- pseudo-spectral evaluations (dft.cu, sweep.cu) --------------------------
// One evaluation on the padded plan: the scalar fields of a band vector pair
// (A, B) on the product grid, point products, and the projection of the
// product fields back to the band.  Writing m = L~B, Du for a Jacobian
// (Du[i][j] = d_j u_i), the brackets are used in the form
//   P(a, m) = (Da)^T m + (Dm) a + m div a = grad(a.m) - a x curl m + m div a
//   Q(a, w) = Da w - Dw a
// (Eqs. 4, 49): the gradient is applied to the projected scalar a.m, exactly
// (truncated convolutions commute with spectral derivatives), so P needs ten
// transformed fields (a, div a, m, curl m) and four projections (a.m and a
// vector) in place of 24 and 3.  Modes, with their input and output fields:
//   PW_F   P(A, m): inputs A, DA, m, curl m (18; all cached in slot); outputs a.m, vec
//   PW_T   P(A, n) + P(v, m) with v, Dv, n, curl n cached: inputs A, div A, m,
//          curl m (10); outputs the scalar and the vector
//   PW_TC  the same from the 18 inputs of PW_F, which it stores in slot2
//   PW_GT  P(v, m), P(A, n), Q(v, A): 18 inputs; outputs 4 + 4 + 3
//   PW_D0  -(B + (DA) B): inputs DA, B (12; stored in slot unless null); outputs 3
//   PW_D1  -(B + (DA) v + (Du) B), {Du, v} cached in slot: 12 inputs, 3 outputs
//   PW_D2  B + (DA)^T B: 12 inputs, 3 outputs
// A stage-point cache slot holds the 18 (or 12) fields of every product-grid point.
enum PwMode : int { PW_F = 0, PW_T, PW_TC, PW_GT, PW_D0, PW_D1, PW_D2, PW_MODES };
__host__ __device__ constexpr int mode_in(int m) { return m == PW_T ? 10 : (m >= PW_D0 ? 12 : 18); }
__host__ __device__ constexpr int mode_out(int m) { return m == PW_GT ? 11 : (m >= PW_D0 ? 3 : 4); }
__host__ __device__ constexpr int mode_nper(int m) { return m == PW_GT ? 3 : 1; }
// 2D problems (one point and one frequency on axis 3, "flat") have no third
// component: their evaluations keep only the fields without one, in the order
//   PW_F, PW_TC, PW_GT  A_1, A_2, d_1 A_1, d_2 A_1, d_1 A_2, d_2 A_2, m_1, m_2, (curl m)_3
//   PW_T                A_1, A_2, div A, m_1, m_2, (curl m)_3
//   deformation         d_1 A_1, d_2 A_1, d_1 A_2, d_2 A_2, B_1, B_2
// and the sine columns of axis 3 are zero and skipped.
__host__ __device__ constexpr int fields_in(int m, bool flat) {
  return !flat ? mode_in(m) : (m == PW_T || m >= PW_D0 ? 6 : 9);
}
__host__ __device__ constexpr int fields_out(int m, bool flat) {
  return !flat ? mode_out(m) : (m == PW_GT ? 8 : (m >= PW_D0 ? 2 : 3));
}
constexpr int kSlotFields = 18, kDefFields = 12, kMaxOutFields = 11, kMaxInFields = 18;

// How an evaluation mode is cut into work items: the plane phase handles
// `ppc` folded x2 pairs of one x1 plane per item (nparts items per plane), the
// band phase 2^tqs quads per item.
struct EvalGeom {
  int ppc, nparts, tqs;
};

// Transform plan of one (grid, band) pair: the folded cosine/sine tables.  A
// real sum over an axis of G points pairs x = t with x = G - t (t = 0..G/2):
// cosines are even and sines odd in x, so both directions cost K/2 products
// per point and K/2 tables rows.  Entries are (cos, sin) pairs.
//   e1f[h][t], e1b[t][h]; e2f[a][t], e2b[t][a]; e3f[b][t], e3b[t][b]
// zero-padded as the kernels stage them: rows of e1f to a multiple of 8 points, of
// e1b to a multiple of 4 and of e2b to a multiple of 8 frequencies, of e3b to K3e
// (even); e3f to K3e frequencies and e3b to NT3e points.
template <typename T>
struct Plan {
  Dims g;
  Band b;
  Trig k;
  int NT1, NT2, NT3;      // folded points per axis, G/2 + 1
  int K3e, NT3e;          // even-rounded K3h and NT3
  bool flat;              // 2D: one point and one frequency on axis 3
  const Pair<T>*e1f, *e1b, *e2f, *e2b, *e3f, *e3b;
  EvalGeom geom[PW_MODES];   // of the plan's evaluations (padded plans)
  FastDiv dK3h, dK3p, dNT1, dNT3, dNT3h, dH1, dH1g;   // dK3p, dNT3h: pairs; dH1g: groups of 4 frequencies
};
inline int even_of(int n) { return n + (n & 1); }
template <typename T>
void plan_sizes(Plan<T>& p, Dims g, const Band& b) {
  p.g = g;
  p.b = b;
  p.k = trig_of(b);
  p.NT1 = g.n1 / 2 + 1;
  p.NT2 = g.n2 / 2 + 1;
  p.NT3 = g.n3 / 2 + 1;
  p.K3e = even_of(p.k.K3h);
  p.flat = b.k3 == 1 && g.n3 == 1;
  p.NT3e = even_of(p.NT3);
  p.dK3h = fast_div(p.k.K3h);
  p.dNT1 = fast_div(p.NT1);
  p.dNT3 = fast_div(p.NT3);
  p.dK3p = fast_div(p.K3e / 2);
  p.dNT3h = fast_div((p.NT3 + 1) / 2);
  p.dH1 = fast_div(p.k.H1);
  p.dH1g = fast_div((p.k.H1 + 3) / 4);
}

template <typename T>
EvalGeom eval_geom(const Plan<T>& p, PwMode mode);

// Epilogue of a projection.  The projected fields are first combined into
// ncomp-component fields Y_o (o < nper, see PwMode); then for band slot k of
// component c
//   dst_j(k) = sum_o cY[j][o] (applyK[o] ? 1/L^(k) : 1) Y_o(k) + sum_i cX[j][i] X_i(k)
// cY includes the 1/(G1 G2 G3) normalisation.  X and dst are band vectors; a dst
// may be one of the X terms.  jA, jB: outputs that are the sources A, B of the
// evaluation that follows in the same launch (-1: read from memory).
constexpr int kMaxPer = 3, kMaxOut = 4, kMaxTerm = 6;
template <typename T>
struct PiEpi {
  int ncomp, nper;
  int grp[kMaxPer];          // host side: the output group and coefficient of each Y_o,
  T coef[kMaxPer];           // folded into cY when an output is added
  int applyK[kMaxPer];
  int nout, nterm;
  int jA, jB;
  T* dst[kMaxOut];
  const T* X[kMaxTerm];
  T cY[kMaxOut][kMaxPer];
  T cX[kMaxOut][kMaxTerm];
};

// One evaluation of a sweep.
template <typename T>
struct EvalDesc {
  const T* A;
  const T* B;
  T* slot;
  T* slot2;
  PiEpi<T> epi;
};

// Band phase: projects the product fields P1 of the previous evaluation of the
// same mode (unless prev is null or has no outputs), applies its epilogue, and
// prepares the plane fields T1 of the next one (sources A and B, unless A is null).
template <typename T>
cudaError_t band_phase(const Plan<T>& p, PwMode mode, const PiEpi<T>* prev, const T* P1, const T* A, const T* B,
                       T* T1, const T* Lhat, cudaStream_t st);
// Plane phase: T1 -> fields on the product grid -> products -> P1.
template <typename T>
cudaError_t plane_phase(const Plan<T>& p, PwMode mode, const T* T1, T* slot, T* slot2, T* P1, cudaStream_t st);
// Every evaluation of a band-limited sweep in one cooperative launch
// (sweep.cu); ev is a device array of nev descriptors of one mode.  bar:
// kSweepBarWords device unsigned ints of barrier state; flag: device double set
// to 1 if a wait gave up.  stall > 0 is the test hook of the time-out path: the
// first grid barrier then waits for one arrival more than the grid has and
// every wait gives up after `stall` polls.
constexpr int kSweepBarWords = 32;
template <typename T>
cudaError_t sweep_launch(const Plan<T>& p, PwMode mode, const EvalDesc<T>* ev, int nev, const T* Lhat, T* T1,
                         T* P1, unsigned* bar, double* flag, cudaStream_t st, int stall = 0);
// elements of the two scratch arrays of evaluations on plan p
template <typename T>
long long eval_T1_elems(const Plan<T>& p);
template <typename T>
long long eval_P1_elems(const Plan<T>& p);

// ---- image-grid transforms (dft.cu) ---------------------------------------
// iota of nf scalar fields: band fields src[f] -> grid fields dst[f]
constexpr int kMaxIota = 36;
template <typename T>
struct IotaList {
  int nf;
  const T* src[kMaxIota];
  T* dst[kMaxIota];
};
template <typename T>
cudaError_t iota_fields(const Plan<T>& p, const IotaList<T>& d, T* T1, cudaStream_t st);
// pi of e.ncomp <= 3 grid fields with epilogue e (nper = 1); the fields, by kind:
//   PI_FIELD      f[0..2]
//   PI_RESIDUAL   c (m - y) d_j m                   (lambda(1) grad m(1))
//   PI_INCREMENT  c y d_j m                         (its Gauss-Newton increment, y = dm(1))
//   PI_NEWTON     c (dm d_j m + (m - y) d_j dm)     (the full-Newton increment)
// d_j: periodic central difference along axis j, taken while the rows are read
// The result goes to the epilogue's output, or to the Hermitian arrays herm if given.
enum PiKind { PI_FIELD = 0, PI_RESIDUAL, PI_INCREMENT, PI_NEWTON };
template <typename T>
struct PiField {
  const T* f[3];
  const T *m, *y, *dm;
  T c;
};
template <typename T>
cudaError_t pi_fields(const Plan<T>& p, PiKind kind, const PiField<T>& s, const PiEpi<T>& e, const T* Lhat, T* P1,
                      cudaStream_t st, cplx<T>* herm = nullptr);
// elements of the scratch: T1 of nf fields, P1 of three
template <typename T>
long long iota_T1_elems(const Plan<T>& p, int nf);
// fields of one iota_fields call (of at most `most`, in threes) that keep the scratch small
template <typename T>
int iota_fields_at_once(const Plan<T>& p, int most);
template <typename T>
long long pi_P1_elems(const Plan<T>& p);
constexpr int kIotaLaunches = 2, kPiLaunches = 2, kEvalLaunches = 2;

// Hermitian complex band arrays [ncomp][K1][K2][K3] (symmetrised on the way in)
// <-> band vectors; components beyond ncomp are not touched.
template <typename T>
void band_load(const cplx<T>* in, T* out, int ncomp, const Band& b, cudaStream_t st);
template <typename T>
void band_store(const T* in, cplx<T>* out, int ncomp, const Band& b, cudaStream_t st);

// whether a grid and band of these sizes are accepted: nper product fields per
// component are projected at once, `brackets`: evaluations run on the plan
template <typename T>
bool sizes_accepted(const Dims& g, const Band& b, int nper, bool brackets);

// ---- grid kernels (grid.cu) -----------------------------------------------
// Semi-Lagrangian state step (Eq. 52): m_next(x) = m(X_n(x)), foot point from
// v_next (at x) and v_cur (trilinear); also writes the displacement off[3].
template <typename T>
void transport_step(const T* m, const T* vnext, const T* vcur, T* mnext, T* off,
                    Dims g, double dt, cudaStream_t st);
// One step of the incremental state (Eq. 31): out = q(X) - c grad m . dv with the
// foot point X of the stored displacement, central differences; q null: q = 0.
// With q_n = dm_n - dt/2 grad m_n . dv_n this carries the trapezoid source along
// the characteristic (see grid.cu).
template <typename T>
void inc_step(const T* q, const T* m, const T* dv, const T* off, T* out, Dims g, double c, cudaStream_t st);
// ---- deformation-state form (Section 3.3) ----
// central-difference gradient of an image -> [3][vol]
template <typename T>
void central_grad(const T* m, T* g3, Dims g, cudaStream_t st);
// m1(x) = I0(x + u(x)), gs(x) = (grad I0)(x + u(x)) (trilinear, periodic); u [3][vol]
// in unit-box units
template <typename T>
void def_sample(const T* I0, const T* gI0, const T* u, T* m1, T* gs, Dims g, cudaStream_t st);
// f = c (m1 - I1) gs (du == nullptr), else dm = gs . du (-> dm_out if given) and
// f = c dm gs; f [3][vol]
template <typename T>
void def_force(const T* gs, const T* m1, const T* I1, const T* du, T* dm_out, double c, T* f, long long vol,
               cudaStream_t st);
// one reversed step of the exact discrete adjoint of the state transport:
// lam_out (zeroed by the caller) and gcur gain atomic scatters, gnext gains the
// per-voxel terms (see grid.cu); off is the step's stored displacement.
template <typename T>
void adjoint_step(const T* lam, const T* m, const T* vcur, const T* vnext, const T* off, T* lam_out, T* gnext,
                  T* gcur, Dims g, double dt, cudaStream_t st);
// out = c (a - b)
template <typename T>
void scaled_diff(const T* a, const T* b, double c, T* out, long long n, cudaStream_t st);

// ---- band vectors and reductions (grid.cu) --------------------------------
// out = a x + b y (band vectors of n reals; y may be null).
template <typename T>
void axpby(T* out, double a, const T* x, double bcoef, const T* y, long long n, cudaStream_t st);
// out = L^ x per band slot (V representative -> l2 gradient).
template <typename T>
void scale_L(T* out, const T* x, const T* Lhat, int ncomp, long long kvol, cudaStream_t st);
// FP64 reductions written to a device double (deterministic two-pass tree).
template <typename T>
void sum_sq_diff(const T* a, const T* b, long long n, double* partial, double* out,
                 cudaStream_t st);
// <a, b>_V = sum Lw a b, Lw = L^ times 1/2 per axis of nonzero frequency
template <typename T>
void inner_V(const T* a, const T* b, const T* Lw, int ncomp, long long kvol, double* partial, double* out,
             cudaStream_t st);
constexpr int kReduceBlocks = 304;   // 2 x 152 SMs
// device-resident conjugate-gradient scalars (grid.cu)
enum PcgSlot { PCG_R = 0, PCG_B, PCG_DQ, PCG_A, PCG_RN, PCG_BETA, PCG_DONE, PCG_ITS, PCG_K, PCG_COPY,
               PCG_SLOTS = 16 };
void pcg_init(double* s, cudaStream_t st);                 // ||b|| = sqrt(rho), counters reset
// one whole PCG step after q = H d in five launches: <d, q>_V partials; alpha
// (or the curvature stop) folded into their sum; x, r updates with the
// <r, r>_V partials; beta (or the residual stop) folded into their sum; d
template <typename T>
void pcg_step(T* x, T* r, T* d, const T* q, const T* Lw, long long kvol, int ncomp,
              double* partial, double* s, double tol, cudaStream_t st);

}  // namespace lddmm
