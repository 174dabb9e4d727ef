// Host side, the deformation-state form (Section 3.3): the band-limited
// inverse-map sweep, its tangent, the terminal sampling and U~(1).
#include "impl.h"

namespace lddmm {
namespace host {

template <typename T>
void Impl<T>::deform_sweep(State<T>& S) {
  const bool keep = &S == &lin;
  cuda(cudaMemsetAsync(S.uh, 0, (size_t)3 * Kvol * sizeof(C), st), "memset u0");
  for (int n = 0; n < Nt; ++n) {
    C* un = vec(S.uh, n);
    C* us = vec(S.ush, n);
    PiEpi<T> e1 = def_epi(false);
    add_out(e1, dk1, 0, 1.0, {});
    add_out(e1, us, 0, dt, {{un, 1.0}});
    eval(PW_D0, keep ? def_slot(2 * n) : nullptr, un, vec(S.vh, n), e1);
    PiEpi<T> e2 = def_epi(false);
    add_out(e2, vec(S.uh, n + 1), 0, 0.5 * dt, {{un, 1.0}, {dk1, 0.5 * dt}});
    eval(PW_D0, keep ? def_slot(2 * n + 1) : nullptr, us, vec(S.vsh, n), e2);
  }
  flush();
}

template <typename T>
void Impl<T>::deform_sample(State<T>& S) {
  T* u1 = S.vgrid + 3 * Nvol;
  to_grid(vec(S.uh, Nt), 1, u1);
  def_sample<T>(I0, gI0, u1, m1(S), S.vgrid, N, st);
  ++launches;
  check_launch("deformation terminal sampling");
}

template <typename T>
auto Impl<T>::deform_tangent() -> C* {
  C* cur = dua;
  C* nxt = dub;
  cuda(cudaMemsetAsync(cur, 0, (size_t)3 * Kvol * sizeof(C), st), "memset du0");
  for (int n = 0; n < Nt; ++n) {
    PiEpi<T> e1 = def_epi(false);
    add_out(e1, dk1, 0, 1.0, {});
    add_out(e1, dup, 0, dt, {{cur, 1.0}});
    eval(PW_D1, def_slot(2 * n), cur, vec(dvh, n), e1);
    PiEpi<T> e2 = def_epi(false);
    add_out(e2, nxt, 0, 0.5 * dt, {{cur, 1.0}, {dk1, 0.5 * dt}});
    eval(PW_D1, def_slot(2 * n + 1), dup, vec(dvsh, n), e2);
    std::swap(cur, nxt);
  }
  flush();
  return cur;
}

template <typename T>
void Impl<T>::terminal_deform(const C* r, const C* u, C* out) {
  PiEpi<T> e = def_epi(true);
  add_out(e, out, 0, 1.0, {});
  eval(PW_D2, nullptr, u, r, e);
  flush();
}

// the members defined here, for both precisions
template void Impl<float>::deform_sweep(State<float>& S);
template void Impl<float>::deform_sample(State<float>& S);
template auto Impl<float>::deform_tangent() -> C*;
template void Impl<float>::terminal_deform(const C* r, const C* u, C* out);
template void Impl<double>::deform_sweep(State<double>& S);
template void Impl<double>::deform_sample(State<double>& S);
template auto Impl<double>::deform_tangent() -> C*;
template void Impl<double>::terminal_deform(const C* r, const C* u, C* out);

}  // namespace host
}  // namespace lddmm
