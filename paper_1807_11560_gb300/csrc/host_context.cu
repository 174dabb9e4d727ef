// Host side, context resources: the per-problem allocations and plans
// (create / release), the cosine/sine tables, the recorded persistent-sweep
// descriptors, host<->device marshalling of band vectors and the kernel-class
// probe.
#include "impl.h"

namespace lddmm {
namespace host {

template <typename T>
void Impl<T>::release() {
  if (hv_exec) cudaGraphExecDestroy(hv_exec);
  hv_exec = nullptr;
  if (hv_exec_newton) cudaGraphExecDestroy(hv_exec_newton);
  hv_exec_newton = nullptr;
  if (cap) cudaStreamDestroy(cap);
  cap = nullptr;
  if (ev) cudaEventDestroy(ev);
  ev = nullptr;
  for (cudaEvent_t e : evpool) cudaEventDestroy(e);
  evpool.clear();
  for (cudaEvent_t e : graph_events) cudaEventDestroy(e);
  graph_events.clear();
  for (void* q : allocs) cudaFree(q);
  allocs.clear();
  if (hres) cudaFreeHost(hres);
  hres = nullptr;
}

template <typename T>
void Impl<T>::make_plan(Plan<T>& p, Dims g) {
  plan_sizes(p, g, K);
  // (cos, sin)(2 pi k x / G) of nk frequencies and nt folded points, frequency-major
  // ([nkp][ntp]) and point-major ([ntb][nkb]), zero-padded
  auto table = [&](int G, int nk, int nt, int nkp, int ntp, int ntb, int nkb, const Pair<T>*& fk, const Pair<T>*& ft) {
    std::vector<Pair<T>> a((size_t)nkp * ntp, Pair<T>{T(0), T(0)}), b((size_t)ntb * nkb, Pair<T>{T(0), T(0)});
    for (int k = 0; k < nk; ++k)
      for (int x = 0; x < nt; ++x) {
        const Pair<T> w = tw((long long)k * x, G);
        a[(size_t)k * ntp + x] = w;
        b[(size_t)x * nkb + k] = w;
      }
    Pair<T>*da = nullptr, *db = nullptr;
    alloc(da, a.size());
    alloc(db, b.size());
    cuda(cudaMemcpy(da, a.data(), a.size() * sizeof(Pair<T>), cudaMemcpyHostToDevice), "tables");
    cuda(cudaMemcpy(db, b.data(), b.size() * sizeof(Pair<T>), cudaMemcpyHostToDevice), "tables");
    fk = da;
    ft = db;
  };
  auto up = [](int n, int m) { return (n + m - 1) / m * m; };
  table(g.n1, p.k.H1, p.NT1, p.k.H1, up(p.NT1, 8), p.NT1, up(p.k.H1, 4), p.e1f, p.e1b);
  table(g.n2, p.k.K2h, p.NT2, p.k.K2h, p.NT2, p.NT2, up(p.k.K2h, 8), p.e2f, p.e2b);
  table(g.n3, p.k.K3h, p.NT3, p.K3e, p.NT3, p.NT3e, p.K3e, p.e3f, p.e3b);
  for (int m = 0; m < PW_MODES; ++m) p.geom[m] = eval_geom(p, (PwMode)m);
}

template <typename T>
void Impl<T>::make_state(State<T>& S) {
  alloc(S.vh, (size_t)(Nt + 1) * 3 * Kvol);
  alloc(S.vsh, (size_t)Nt * 3 * Kvol);
  alloc(S.cache, (size_t)2 * Nt * slot_elems());
  const size_t steps = opts.recompute ? 2 : (size_t)Nt + 1;
  alloc(S.vgrid, steps * 3 * Nvol);
  alloc(S.mh, steps * Nvol);
  alloc(S.off, (opts.recompute ? 1 : (size_t)Nt) * 3 * Nvol);
  if (deform()) {
    alloc(S.uh, (size_t)(Nt + 1) * 3 * Kvol);
    alloc(S.ush, (size_t)Nt * 3 * Kvol);
  }
}

template <typename T>
void Impl<T>::create(int nd, const int* grid, const int* band, double a, int s_, double sg, int nt,
              const lddmm_opts& o) {
  ndim = nd;
  duser = nd;
  N = Dims{grid[0], grid[1], nd == 3 ? grid[2] : 1};
  K.k1 = band[0];
  K.k2 = band[1];
  K.k3 = nd == 3 ? band[2] : 1;
  K.h1 = K.k1 / 2;
  auto padn = [](int k) { return k == 1 ? 1 : (3 * k + 1) / 2; };
  M = Dims{padn(K.k1), padn(K.k2), padn(K.k3)};
  Nt = nt;
  s = s_;
  alpha = a;
  sigma = sg;
  dt = 1.0 / nt;
  Nvol = N.vol();
  Mvol = M.vol();
  Kvol = trig_of(K).vol();
  Kuser = K.vol();
  opts = o;
  st = (cudaStream_t)o.stream;
  cuda(cudaGetDevice(&device), "device");
  cuda(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "stream");
  cuda(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming), "event");

  if (!sizes_accepted<T>(N, K, 1, false) || !sizes_accepted<T>(M, K, 3, true)) {
    *err = "grid or band too large for the transform tiles (N_3 <= 512, K_3 <= 112, shared memory)";
    throw Fail{LDDMM_EINVAL};
  }
  make_plan(full, N);
  make_plan(pad, M);
  // L^ per slot of a band component, and L^ times 1/2 per axis of nonzero
  // frequency (the squared norms of the cosine and sine modes)
  const Trig tk = trig_of(K);
  std::vector<T> L((size_t)Kvol), Lv((size_t)Kvol);
  for (int f2 = 0; f2 < tk.K2h; ++f2)
    for (int f3 = 0; f3 < tk.K3h; ++f3)
      for (int f1 = 0; f1 < tk.H1; ++f1) {
        const double l = std::pow(1.0 + 4.0 * kPi * kPi * alpha * ((double)f1 * f1 + (double)f2 * f2 + (double)f3 * f3),
                                  (double)s);
        const double w = (f1 ? 0.5 : 1.0) * (f2 ? 0.5 : 1.0) * (f3 ? 0.5 : 1.0);
        for (int i = 0; i < 8; ++i) {
          const size_t at = ((size_t)(f2 * tk.K3h + f3) * tk.H1 + f1) * 8 + i;
          L[at] = (T)l;
          Lv[at] = (T)w * (T)l;
        }
      }
  alloc(Lhat, (size_t)Kvol);
  alloc(Lw, (size_t)Kvol);
  cuda(cudaMemcpy(Lhat, L.data(), L.size() * sizeof(T), cudaMemcpyHostToDevice), "Lhat");
  cuda(cudaMemcpy(Lw, Lv.data(), Lv.size() * sizeof(T), cudaMemcpyHostToDevice), "Lw");

  alloc(I0, (size_t)Nvol);
  alloc(I1, (size_t)Nvol);
  iota_nf = iota_fields_at_once<T>(full, opts.recompute || deform() ? 3 : 3 * (Nt + 1));
  alloc(T1, (size_t)std::max({iota_T1_elems<T>(full, iota_nf), pi_P1_elems<T>(full), eval_T1_elems<T>(pad)}));
  alloc(P1, (size_t)eval_P1_elems<T>(pad));
  alloc(zin, (size_t)3 * Kuser);
  alloc(zout, (size_t)3 * Kuser);
  for (C** b : {&k1, &aU, &aW, &Ut, &Wt, &U, &W, &vout, &gbuf, &px, &pr,
                &vsol, &vtry})
    alloc(*b, (size_t)3 * Kvol);
  alloc(dvh, (size_t)(Nt + 1) * 3 * Kvol);
  alloc(srcs, (size_t)(Nt + 1) * 3 * Kvol);
  alloc(dvsh, (size_t)Nt * 3 * Kvol);
  alloc(Uh, (size_t)(Nt + 1) * 3 * Kvol);
  alloc(Wh, (size_t)(Nt + 1) * 3 * Kvol);
  alloc(Uth, (size_t)Nt * 3 * Kvol);
  alloc(Wth, (size_t)Nt * 3 * Kvol);
  alloc(bU, (size_t)3 * Kvol);
  alloc(bW, (size_t)3 * Kvol);
  alloc(zero3, (size_t)3 * Kvol);
  cuda(cudaMemset(zero3, 0, (size_t)3 * Kvol * sizeof(C)), "memset");
  alloc(dvgrid, (opts.recompute ? 2 : (size_t)Nt + 1) * 3 * Nvol);
  for (int i = 0; i < 2; ++i) alloc(dm[i], (size_t)Nvol);
  alloc(fterm, (size_t)3 * Nvol);
  if (deform()) {
    alloc(gI0, (size_t)3 * Nvol);
    alloc(defcache, (size_t)2 * Nt * kDefFields * Mvol);
    for (C** b : {&dk1, &rhob, &dua, &dub, &dup}) alloc(*b, (size_t)3 * Kvol);
  }
  alloc(partial, (size_t)kReduceBlocks);
  alloc(dres, 8);
  alloc(dpcg, PCG_SLOTS);
  cuda(cudaMemset(dres, 0, 8 * sizeof(double)), "memset");
  cuda(cudaMallocHost(&hres, 8 * sizeof(double)), "cudaMallocHost");
  make_state(lin);
  make_state(trial);
  alloc(tcache, (size_t)2 * Nt * slot_elems());
  alloc(bar, kSweepBarWords);
  record_sweeps();
  cuda(cudaDeviceSynchronize(), "create");
}

template <typename T>
void Impl<T>::record_sweeps() {
  std::vector<EvalDesc<T>> v;
  rec = &v;
  auto upload = [&](EvalDesc<T>*& dst) {
    alloc(dst, v.size());
    cuda(cudaMemcpy(dst, v.data(), v.size() * sizeof(EvalDesc<T>), cudaMemcpyHostToDevice), "descriptors");
    v.clear();
  };
  shoot(lin);
  upload(ev_shoot_lin);
  shoot(trial);
  upload(ev_shoot_trial);
  tangent(lin);
  upload(ev_tangent);
  backward(lin);
  upload(ev_backward);
  backward_sources(lin);
  upload(ev_exact);
  tangent(lin, true);
  upload(ev_tangent_c);
  backward_hist(lin);
  upload(ev_backward_hist);
  newton_backward(lin);
  upload(ev_newton);
  rec = nullptr;
}

namespace {
// the allocation that holds a device address (driver call, looked up once)
using AddressRange = int (*)(unsigned long long* base, size_t* size, unsigned long long p);
AddressRange address_range() {
  static const AddressRange f = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &p, 12000, cudaEnableDefault, &q) !=
            cudaSuccess || q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      p = nullptr;
    }
    return reinterpret_cast<AddressRange>(p);
  }();
  return f;
}
}  // namespace

// Whether the kernels can read or write the bytes at p in place: memory of this
// context's device, aligned as the element, all of it inside one allocation.
// Anything else (host and managed arrays, another device, a range that is too
// short) goes through the staging buffers and the copy's own checks.
template <typename T>
bool Impl<T>::in_place(const void* p, size_t bytes, size_t align) {
  const unsigned long long a = reinterpret_cast<uintptr_t>(p);
  if (a % align != 0 || !address_range()) return false;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (at.type != cudaMemoryTypeDevice || at.device != device) return false;
  unsigned long long base = 0;
  size_t size = 0;
  return address_range()(&base, &size, a) == 0 && a + bytes <= base + size;
}

template <typename T>
void Impl<T>::load_bl(const void* user, C* dst) {
  const Z* src = static_cast<const Z*>(user);
  if (!in_place(user, (size_t)duser * Kuser * sizeof(Z), sizeof(Z))) {
    cuda(cudaMemcpyAsync(zin, user, (size_t)duser * Kuser * sizeof(Z), cudaMemcpyDefault, st), "copy BL input");
    src = zin;
  }
  if (duser < 3)
    cuda(cudaMemsetAsync(dst + (size_t)duser * Kvol, 0, (size_t)(3 - duser) * Kvol * sizeof(T), st), "memset");
  band_load<T>(src, dst, duser, K, st);
  ++launches;
  check_launch("band load");
}

template <typename T>
void Impl<T>::store_bl(const C* src, void* user) {
  const bool direct = in_place(user, (size_t)duser * Kuser * sizeof(Z), sizeof(Z));
  band_store<T>(src, direct ? static_cast<Z*>(user) : zout, duser, K, st);
  ++launches;
  check_launch("band store");
  if (!direct)
    cuda(cudaMemcpyAsync(user, zout, (size_t)duser * Kuser * sizeof(Z), cudaMemcpyDefault, st), "copy BL output");
}

template <typename T>
void Impl<T>::collect() {
  float ms = 0.f;
  for (size_t i = 0; i < pend_direct.size(); ++i) {
    cuda(cudaEventElapsedTime(&ms, pend_direct[i].first, pend_direct[i].second), "probe elapsed");
    probe_ms += ms;
    probe_work += pend_work[i];
    ++probe_n;
  }
  pend_direct.clear();
  pend_work.clear();
  evnext = 0;
  if (graph_pending) {
    for (size_t i = 0; i < graph_pairs.size(); ++i) {
      cuda(cudaEventElapsedTime(&ms, graph_pairs[i].first, graph_pairs[i].second), "probe elapsed");
      probe_ms += ms;
      probe_work += graph_work[i];
      ++probe_n;
    }
    graph_pending = false;
  }
}

template <typename T>
void Impl<T>::invalidate_graph() {
  if (hv_exec_newton) {
    cudaGraphExecDestroy(hv_exec_newton);
    hv_exec_newton = nullptr;
  }
  if (hv_exec) {
    cudaGraphExecDestroy(hv_exec);
    hv_exec = nullptr;
  }
  for (cudaEvent_t e : graph_events) cudaEventDestroy(e);
  graph_events.clear();
  graph_pairs.clear();
  graph_work.clear();
  graph_pending = false;
}

template <typename T>
void Impl<T>::set_probe(int cls) {
  sync("probe");
  if (cls != probe) invalidate_graph();
  probe = cls;
  probe_ms = 0.0;
  probe_work = 0.0;
  probe_n = 0;
}

// the members defined here, for both precisions
template void Impl<float>::release();
template void Impl<float>::make_plan(Plan<float>& p, Dims g);
template void Impl<float>::make_state(State<float>& S);
template void Impl<float>::create(int nd, const int* grid, const int* band, double a, int s_, double sg, int nt, const lddmm_opts& o);
template void Impl<float>::record_sweeps();
template bool Impl<float>::in_place(const void* p, size_t bytes, size_t align);
template bool Impl<double>::in_place(const void* p, size_t bytes, size_t align);
template void Impl<float>::load_bl(const void* user, C* dst);
template void Impl<float>::store_bl(const C* src, void* user);
template void Impl<float>::collect();
template void Impl<float>::invalidate_graph();
template void Impl<float>::set_probe(int cls);
template void Impl<double>::release();
template void Impl<double>::make_plan(Plan<double>& p, Dims g);
template void Impl<double>::make_state(State<double>& S);
template void Impl<double>::create(int nd, const int* grid, const int* band, double a, int s_, double sg, int nt, const lddmm_opts& o);
template void Impl<double>::record_sweeps();
template void Impl<double>::load_bl(const void* user, C* dst);
template void Impl<double>::store_bl(const C* src, void* user);
template void Impl<double>::collect();
template void Impl<double>::invalidate_graph();
template void Impl<double>::set_probe(int cls);

}  // namespace host
}  // namespace lddmm
