// Host side of the GB300 LDDMM library: the per-problem context behind the
// C interface of include/lddmm.h (internal; not part of the interface).
//
// A context owns, per problem, every device buffer of the method:
//   * the folded cosine/sine tables of the image-grid plan (N) and of the padded
//     product plan (M = ceil(3K/2)), and the symbol table L^(k);
//   * two trajectories ("lin", the Gauss-Newton linearisation point, and
//     "trial", used by energy evaluations and component calls), each with the
//     BL history v_n, the Heun predictors v*_{n+1}, the 18 padded-grid fields
//     (v, Dv, L v, curl L v) of every Heun stage point, the grid velocities
//     iota(v_n), the state history m_n and the characteristic displacements;
//   * the tangent history dv_n and its grid velocities, a ping-pong
//     pair for the incremental transport, the transform scratch and BL temporaries;
//   * with the deformation state equation (Section 3.3, opts.state_eq = 1):
//     per trajectory the band-limited inverse-map displacement u_n and its
//     predictors, the padded-grid fields {D u, v} of lin's stage points, and
//     grad I0 on the image grid.
// The time loops run on the host and enqueue kernels on one stream; the
// Hessian-vector product can be captured once per linearisation point into a
// CUDA graph and replayed.
//
// The members are defined by responsibility: host_context.cu (allocation,
// plans, probe), host_sweeps.cu (bracket evaluations and the time
// sweeps), host_deform.cu (the deformation-state form), host_objective.cu
// (energy, gradient, Hessian-vector products, graph capture), host_solver.cu
// (GN-Krylov), host_components.cu (the component calls); api.cu holds the C
// interface.
#pragma once

#include <algorithm>
#include <atomic>
#include <cmath>
#include <initializer_list>
#include <utility>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/lddmm.h"
#include "internal.h"

namespace lddmm {
namespace host {

constexpr double kPi = 3.141592653589793238462643383279;

struct Fail {
  int code;
};

enum ProbeClass { PR_TRANSPORT = 0, PR_INC, PR_IOTA_AB, PR_CPW, PR_PI_BA, PR_IOTA_FULL, PR_PI_FULL,
                  PR_SWEEP, PR_DEFORM, PR_COUNT };
const char* const kProbeNames[PR_COUNT] = {"transport", "inc_step", "iota_ab", "cpw", "pi_ba",
                                           "iota_full", "pi_full", "sweep", "deform"};

template <typename T>
struct State {
  T* vh = nullptr;          // [Nt+1][3][Kvol]
  T* vsh = nullptr;         // [Nt][3][Kvol]
  T* cache = nullptr;       // [2 Nt][18][Mvol]: padded-grid fields per stage point
  T* vgrid = nullptr;       // [Nt+1][3][Nvol]  (recompute: [2][3][Nvol], step n in n & 1)
  T* mh = nullptr;          // [Nt+1][Nvol]     (recompute: [2][Nvol])
  T* off = nullptr;         // [Nt][3][Nvol]    (recompute: [3][Nvol], the current step)
  // deformation-state form (Section 3.3): band-limited inverse-map displacement
  T* uh = nullptr;          // [Nt+1][3][Kvol]
  T* ush = nullptr;         // [Nt][3][Kvol]    Heun predictors u*_n
};

template <typename T>
struct Impl {
  using C = T;               // element of a band vector (internal.h): 3 Kvol reals
  using Z = cplx<T>;         // element of the caller's Hermitian arrays
  std::string* err = nullptr;
  int ndim = 3, duser = 3, device = 0;
  Dims N{}, M{};
  Band K{};
  int Nt = 1, s = 2;
  double alpha = 0, sigma = 1, dt = 1;
  long long Nvol = 0, Mvol = 0, Kvol = 0, Kuser = 0;   // Kuser: complex slots of a user component
  lddmm_opts opts{};
  cudaStream_t st = nullptr;
  Plan<T> full{}, pad{};
  T *Lhat = nullptr, *Lw = nullptr;   // L^ per slot; with the weights of the V product
  T *I0 = nullptr, *I1 = nullptr;
  State<T> lin, trial;
  bool have_images = false, have_lin = false, have_dm1 = false;
  T* T1 = nullptr;                    // transform scratch: plane fields; projected image planes
  T* P1 = nullptr;                    // projected planes of an evaluation
  int iota_nf = 33;                   // fields of one image-grid transform (T1 is sized for)
  Z *zin = nullptr, *zout = nullptr;  // [3][Kuser] staging of the caller's arrays
  C *k1 = nullptr, *aU = nullptr, *aW = nullptr, *Ut = nullptr, *Wt = nullptr, *U = nullptr,
    *W = nullptr, *vout = nullptr, *gbuf = nullptr;
  C *px = nullptr, *pr = nullptr, *vsol = nullptr, *vtry = nullptr;
  C* dvh = nullptr;          // [Nt+1][3][Kvol]
  C* srcs = nullptr;         // [Nt+1][3][Kvol] band sources of the exact discrete adjoint
  C* dvsh = nullptr;         // [Nt][3][Kvol] tangent predictor stages dv*_n
  C *Uh = nullptr, *Wh = nullptr;     // [Nt+1][3][Kvol] gradient sweep (U, W) per time level
  C *Uth = nullptr, *Wth = nullptr;   // [Nt][3][Kvol] gradient sweep stage values (U~, W~)
  C *bU = nullptr, *bW = nullptr;     // full-Newton sweep scratch
  T* tcache = nullptr;       // [2 Nt][18][Mvol] tangent stage-point fields (full Newton)
  C* zero3 = nullptr;        // [3][Kvol] zeros
  T* dvgrid = nullptr;       // [Nt+1][3][Nvol]  (recompute: [2][3][Nvol])
  T* dm[2] = {nullptr, nullptr};   // q_n of the incremental transport, ping-pong; dm(1) in dm[Nt & 1]
  T* fterm = nullptr;        // [3][Nvol]
  double *partial = nullptr, *dres = nullptr;   // dres[7]: sweep barrier time-out flag
  double* dpcg = nullptr;    // [PCG_SLOTS] device conjugate-gradient scalars
  double* hres = nullptr;    // pinned host mirror of dres
  // persistent sweeps: evaluation descriptors recorded once at creation
  std::vector<EvalDesc<T>>* rec = nullptr;
  EvalDesc<T> *ev_shoot_lin = nullptr, *ev_shoot_trial = nullptr, *ev_tangent = nullptr,
              *ev_backward = nullptr, *ev_exact = nullptr, *ev_tangent_c = nullptr,
              *ev_backward_hist = nullptr, *ev_newton = nullptr;
  unsigned* bar = nullptr;
  // the evaluation whose projection and epilogue the next band phase runs
  bool pending = false;
  PwMode pend_mode = PW_F;
  PiEpi<T> pend_epi{};
  long long launches = 0;
  std::vector<void*> allocs;
  unsigned long long device_bytes = 0;
  // graph of one Hessian-vector product (input dvh[0], output vout)
  cudaGraphExec_t hv_exec = nullptr, hv_exec_newton = nullptr;
  long long hv_nodes = 0, hv_nodes_newton = 0;
  bool have_zhist = false;   // Uh/Wh/Uth/Wth hold the last gradient's backward sweep
  // deformation-state form (Section 3.3)
  T* gI0 = nullptr;           // [3][Nvol] central-difference gradient of I0
  T* defcache = nullptr;      // [2 Nt][12][Mvol] {D u, v} at the stage points of lin's sweep
  C *dk1 = nullptr, *rhob = nullptr, *dua = nullptr, *dub = nullptr, *dup = nullptr;   // [3][Kvol]
  cudaStream_t cap = nullptr;
  cudaEvent_t ev = nullptr;
  bool capturing = false;
  // kernel-class probe: CUDA events around every launch of one class, read
  // back after each stream synchronisation (also inside the captured graph,
  // as external event-record nodes)
  int probe = -1;
  std::vector<cudaEvent_t> evpool;
  size_t evnext = 0;
  cudaEvent_t pstart = nullptr;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> pend_direct, graph_pairs;
  std::vector<cudaEvent_t> graph_events;
  bool graph_pending = false;
  double probe_ms = 0.0, probe_work = 0.0;
  long long probe_n = 0;
  std::vector<double> pend_work, graph_work;

  // ---------------------------------------------------------------- utils
  void cuda(cudaError_t e, const char* what) {
    if (e != cudaSuccess) {
      cudaGetLastError();   // reported here: not again by the next check_launch of this thread
      *err = std::string(what) + ": " + cudaGetErrorString(e);
      throw Fail{LDDMM_ECUDA};
    }
  }
  void check_launch(const char* what) { cuda(cudaGetLastError(), what); }
  template <typename P_>
  void alloc(P_*& p, size_t count) {
    void* q = nullptr;
    const size_t bytes = count * sizeof(P_);
    cudaError_t e = cudaMalloc(&q, bytes > 0 ? bytes : 16);
    if (e != cudaSuccess) {
      cudaGetLastError();
      *err = "cudaMalloc of " + std::to_string(bytes) + " bytes failed: " + cudaGetErrorString(e);
      throw Fail{LDDMM_ENOMEM};
    }
    allocs.push_back(q);
    device_bytes += bytes > 0 ? bytes : 16;
    p = static_cast<P_*>(q);
  }
  void release();

  // (cos, sin)(2 pi p / G), the sine exactly zero where it is
  static Pair<T> tw(long long p, int G) {
    const long long r = p % G;
    const double a = 2.0 * kPi * (double)r / (double)G;
    return Pair<T>{(T)std::cos(a), (2 * r) % G == 0 ? T(0) : (T)std::sin(a)};
  }

  void make_plan(Plan<T>& p, Dims g);

  void make_state(State<T>& S);
  // image-grid history accessors (step n of a kept or a two-step rolling history)
  long long hstep(int n) const { return opts.recompute ? (n & 1) : n; }
  T* mstate(State<T>& S, int n) { return S.mh + hstep(n) * Nvol; }
  T* m1(State<T>& S) { return mstate(S, Nt); }
  T* vgr(State<T>& S, int n) { return S.vgrid + hstep(n) * 3 * Nvol; }
  T* offp(State<T>& S, int n) { return S.off + (opts.recompute ? 0 : (long long)n) * 3 * Nvol; }
  T* dvg(int n) { return dvgrid + hstep(n) * 3 * Nvol; }

  void create(int nd, const int* grid, const int* band, double a, int s_, double sg, int nt,
              const lddmm_opts& o);

  // descriptors of every persistent sweep, recorded by running the sweep
  // loops once without launching anything
  void record_sweeps();

  // a persistent sweep whose barrier wait gave up left dres[7] = 1
  void check_flag(double f) {
    if (f != 0.0) {
      *err = "a bounded device wait (sweep barrier) timed out";
      throw Fail{LDDMM_ETIMEOUT};
    }
  }

  // ------------------------------------------------------------ staging
  // user BL vector (duser comps) -> hermitian 3-comp device vector
  bool in_place(const void* p, size_t bytes, size_t align);
  void load_bl(const void* user, C* dst);
  void store_bl(const C* src, void* user);
  void sync(const char* what) {
    cuda(cudaStreamSynchronize(st), what);
    collect();
  }

  // ------------------------------------------------------------- probe
  cudaEvent_t probe_event() {
    cudaEvent_t e = nullptr;
    if (capturing) {
      cuda(cudaEventCreate(&e), "probe event");
      graph_events.push_back(e);
      return e;
    }
    if (evnext == evpool.size()) {
      cuda(cudaEventCreate(&e), "probe event");
      evpool.push_back(e);
    }
    return evpool[evnext++];
  }
  void probe_record(cudaEvent_t e) {
    cuda(cudaEventRecordWithFlags(e, st, capturing ? cudaEventRecordExternal : cudaEventRecordDefault),
         "probe record");
  }
  void pb(int cls) {
    if (cls != probe) return;
    pstart = probe_event();
    probe_record(pstart);
  }
  // work: algorithmic flops (transforms, brackets) or bytes (transport steps)
  void pe(int cls, double work) {
    if (cls != probe) return;
    cudaEvent_t e = probe_event();
    probe_record(e);
    (capturing ? graph_pairs : pend_direct).push_back({pstart, e});
    (capturing ? graph_work : pend_work).push_back(work);
  }
  void collect();

  // -------------------------------------------------------- descriptors
  static PiEpi<T> epi(int ncomp, int nper) {
    PiEpi<T> e;
    std::memset(&e, 0, sizeof(e));
    e.ncomp = ncomp;
    e.nper = nper;
    return e;
  }
  // output dst = cR * (the fields of group r, each with its coefficient) + terms
  static void add_out(PiEpi<T>& e, C* dst, int r, double cR,
                      std::initializer_list<std::pair<const C*, double>> xs) {
    const int j = e.nout++;
    e.dst[j] = dst;
    for (int o = 0; o < e.nper; ++o) e.cY[j][o] = e.grp[o] == r ? (T)(cR * (double)e.coef[o]) : (T)0;
    for (auto& x : xs) {
      e.X[e.nterm] = x.first;
      e.cX[j][e.nterm++] = (T)x.second;
    }
  }
  // marks the outputs that the next evaluation reads as its sources
  static void link(PiEpi<T>& e, const C* A, const C* B) {
    e.jA = e.jB = -1;
    for (int j = 0; j < e.nout; ++j) {
      if (e.dst[j] == A) e.jA = j;
      if (e.dst[j] == B) e.jB = j;
    }
  }

  // operations of the transforms of nf scalar fields between the band and grid g
  // (folded cosine/sine sums: K/2 products per point and axis; 2D has no third axis)
  double grid_flops(const Dims& g, int nf) const {
    const double k1 = K.k1, k2 = K.k2, k3 = K.k3, n1 = g.n1;
    return nf * (k1 * n1 * k2 * k3 + n1 * k2 * g.n2 * k3 + (pad.flat ? 0.0 : n1 * (double)g.n2 * k3 * g.n3));
  }
  // fields that an evaluation transforms, in and out
  int eval_in(PwMode mode) const { return fields_in(mode, pad.flat); }
  int eval_out(PwMode mode) const { return fields_out(mode, pad.flat); }
  // operations of n fields of an evaluation in the band phase, and of its plane phase
  // (with, roughly, the point products)
  double band_flops(int n) const { return n * (double)Kuser * M.n1; }
  double plane_flops(PwMode mode) const {
    const double per_point[2][PW_MODES] = {{30, 60, 60, 90, 21, 39, 18}, {10, 22, 23, 34, 8, 16, 8}};
    const int n = eval_in(mode) + eval_out(mode);
    return grid_flops(M, n) - band_flops(n) + per_point[pad.flat][mode] * (double)Mvol;
  }

  // One evaluation of a pseudo-spectral expression (PwMode) with sources srcA,
  // srcB and projection epilogue e.  Its projection runs in the band phase of the
  // next evaluation (one launch for both); flush() runs it when none follows.
  void eval(PwMode mode, T* slot, const C* srcA, const C* srcB, const PiEpi<T>& e, T* slot2 = nullptr);
  void flush();

  // one band-limited sweep as a single persistent cooperative kernel
  void run_sweep(PwMode mode, const EvalDesc<T>* ev, int nev = 0);
  static constexpr long long kPersistentMaxPadded = 32768;   // M1 M2 M3
  bool deform() const { return opts.state_eq == 1; }
  void state_form_only(const char* what) {
    if (!deform()) return;
    *err = std::string(what) + " is defined for the image state form only (opts.state_eq = 0)";
    throw Fail{LDDMM_EINVAL};
  }
  // whether the options let sweeps run as persistent kernels (lddmm_batch_gn_solve
  // refuses such contexts)
  bool persistent() const {
    return opts.persistent == 2 || (opts.persistent == 1 && Mvol <= kPersistentMaxPadded);
  }
  // and whether they do: on request only.  Two launches per evaluation, each
  // starting as the one before drains, take less than the two grid barriers of a
  // persistent kernel (us per shoot evaluation, launches / persistent: 9.4 / 11.3 at
  // band 16^3, 50 / 51 at 2D 16^2 FP64).
  bool run_persistent() const { return rec == nullptr && opts.persistent == 2; }

  // iota of `count` BL vectors (3 comps each) onto the image grid
  void to_grid(const C* hist, int count, T* grid);

  // K~ pi (or pi alone) of a 3-component image-grid field -> band vector out
  void project(PiKind kind, const PiField<T>& f, C* out, double coef, bool applyK);
  void project_K(const T* f3, C* out, bool applyK = true);

  // K~ pi of a terminal field (PI_RESIDUAL, PI_INCREMENT or PI_NEWTON)
  void project_terminal(PiKind kind, const T* m, const T* y, const T* dm1, double c, C* out);

  // K~ sum_x f(x) e^{-2 pi i k.x} of a 3-component grid field: the V-representer
  // of the cotangent of iota (the adjoint of iota is N pi)
  void project_adjoint(const T* f3, C* out);

  // ------------------------------------------------------------- sweeps
  long long slot_elems() const { return (kSlotFields * Mvol + 3) / 4 * 4; }   // 16-byte aligned
  T* slot(State<T>& S, int k) { return S.cache + k * slot_elems(); }
  C* vec(C* base, int n) { return base + (long long)n * 3 * Kvol; }

  // Heun shoot of BL EPDiff (Eq. 51); S.vh[0] must hold v0
  void shoot(State<T>& S);

  // one semi-Lagrangian state step m_n -> m_{n+1} (Eq. 52) from the kept or
  // regenerated velocity grids of steps n and n + 1
  void state_step(State<T>& S, int n);

  // grid velocities and semi-Lagrangian transport of I0 (Eq. 52)
  void transport(State<T>& S);

  void forward(State<T>& S);

  // ------------------------------------- deformation-state form (Section 3.3)
  PiEpi<T> def_epi(bool applyK) const {
    PiEpi<T> e = epi(3, 1);
    e.grp[0] = 0;
    e.coef[0] = (T)(1.0 / (double)Mvol);
    e.applyK[0] = applyK ? 1 : 0;
    return e;
  }

  // padded-grid block {D u, v} of stage point k (2 n, 2 n + 1) of lin's sweep
  T* def_slot(int k) { return defcache + (long long)k * kDefFields * Mvol; }

  // Heun sweep of d/dt u~ = -v~ - D~u~ * v~ jointly with the shoot (stage 2 at
  // the EPDiff predictor v*_n), u~(0) = 0.  For lin the padded-grid fields of
  // each stage point stay in defcache for the tangent sweeps.
  void deform_sweep(State<T>& S);

  // m(1) = I0(x + u(1)(x)) into m1(S) and (grad I0)(x + u(1)(x)) into the first
  // three fields of S.vgrid (u(1) on the grid goes to the next three)
  void deform_sample(State<T>& S);

  // exact tangent of lin's deformation sweep along the shoot tangent (dvh,
  // dvsh), reading {D u, v} of each stage point from defcache; returns the
  // buffer holding delta u~(1)
  C* deform_tangent();

  // U~(1) = K~ pi[r + (D u)^T r] on the padded grid, r = iota(r~), u = u~(1)
  void terminal_deform(const C* r, const C* u, C* out);

  // energy pieces into dres[0] (<v0,v0>_V) and dres[1] (sum (m1 - I1)^2)
  void energy_terms(State<T>& S);
  double read_energy();
  double dot_V(const C* a, const C* b);

  // backward reduced adjoint Jacobi sweep (Eqs. 53-54) from (U, W) = (U, 0);
  // leaves W(0) in W
  void backward(State<T>& S);

  // incremental EPDiff (Eq. 30) from dvh[0], exact tangent of the Heun shoot
  T* tslot(int k) { return tcache + k * slot_elems(); }

  // incremental BL EPDiff (Eq. 30) from dvh[0]; with cache, also stores the
  // padded-grid fields of dv_n and dv*_n (full-Newton products)
  void tangent(State<T>& S, bool cache = false);

  // transpose of the Heun shoot tangent with a band source at every time level
  // (the exact discrete adjoint's band sweep): W_Nt = s_Nt, W_n = T_n^T W_{n+1}
  // + s_n with T_n^T the W part of the backward Jacobi sweep (U = 0); leaves
  // W_0 in W
  void backward_sources(State<T>& S);

  // the gradient's backward sweep (Eqs. 53-54) with its time levels and stage
  // values kept: level n in (Uh[n], Wh[n]) (Uh[Nt] = U~(1) set by the caller),
  // stage of step n in (Uth[n], Wth[n]); W(0) = Wh[0]
  void backward_hist(State<T>& S);

  // full-Newton incremental adjoint sweep (Eqs. 56-57 without the Gauss-Newton
  // drop): the derivative of the gradient's Heun-transposed recursion along the
  // tangent trajectory.  Per step four evaluations of the ad~ / ad~^dagger
  // bracket: G^T at v on (dU, dW) (the Gauss-Newton terms) and the same bracket
  // with dv in place of v on the gradient sweep's (U, W) (the dropped terms:
  // ad~^dagger_dv U, ad~^dagger_W dv - ad~_dv W), at the predictor and at the
  // step's start.  Starts from (U, W) = (dU(1), 0); leaves dW(0) in W.
  void newton_backward(State<T>& S);

  // V-gradient of the discretised energy itself (Section 2.5's route in
  // discrete form, Eqs. 12-14): the state transport reversed step by step on
  // the image grid, each time level's velocity sensitivity projected to the
  // band, then carried back to v0 by backward_sources.  Needs the kept
  // histories (every reversed step reads m_n, v_n, v_{n+1} and the displacement
  // in reverse time order).
  double exact_gradient_dev(const C* v0dev, C* gdev);

  // forward sweep of lin at v0 with the histories the exact adjoint reads
  void exact_forward(const C* v0dev);

  // reverse-mode sweep of the discrete map v0 -> m(1) from the cotangent
  // lambda(1) = dL/dm(1) held in dm[0]: the transport reversed step by step,
  // each level's velocity sensitivity projected to the band, the Heun shoot
  // transposed; leaves the V-representer of dL/dv0 in W
  void exact_backward();

  // enqueue one GN Hessian-vector product: input dvh[0], output vout
  void enqueue_hessvec(bool newton = false);

  // ------------------------------------------------------- public calls
  void need_images() {
    if (!have_images) {
      *err = "images not set (call lddmm_set_images first)";
      throw Fail{LDDMM_ESTATE};
    }
  }

  void set_images(const void* a, const void* b);

  double energy_dev(const C* v0dev);

  double energy(const void* v0);

  // gradient at the device vector v0dev (hermitian, 3 comps); g -> gdev
  double gradient_dev(const C* v0dev, C* gdev);

  // the rest of the gradient once lin holds the forward sweep of the point and
  // dres[0..1] its energy terms
  double gradient_tail(C* gdev);

  double gradient(const void* v0, void* g);

  double exact_gradient(const void* v0, void* g);

  void invalidate_graph();

  void set_probe(int cls);

  // Hessian-vector product with input already in dvh[0]; result in vout
  void hessvec_dev(bool newton = false);

  void build_graph(bool newton = false);

  void hessvec(const void* dv, void* out);

  void hessvec_newton(const void* dv, void* out);

  void gn_solve(void* v0, int n_gn, int n_pcg, lddmm_report* rep);

  // component calls ---------------------------------------------------------
  void iota_call(const void* a, int ncomp, void* out);

  void pi_call(const void* f, int ncomp, void* out);

  void ad_dagger_call(const void* v, const void* u, void* out);

  void ad_call(const void* v, const void* w, void* out);

  void shoot_call(const void* v0, void* v1);

  void transport_call(const void* v0, void* m1out);

  // l2 gradient of a loss of m(1) with respect to v0 (adjoint Jacobi sweep)
  void transport_vjp(const void* v0, const void* gm1, void* out);

  // the same vector-Jacobian product through the exact discrete adjoint of the
  // discretised map (the transposes of the semi-Lagrangian steps and of the Heun
  // shoot): the derivative of the discrete m(1) itself
  void transport_vjp_exact(const void* v0, const void* gm1, void* out);

  void last_dm1(void* out);
};

}  // namespace host
}  // namespace lddmm
