// Element-local arithmetic of the face form of the right-hand side, on the generated operators
// Ops<N> (gen_face.cpp): a thread holds one element's nodal row in registers.
//
// The flux through an edge is split into one part per side: each element evaluates, for each of
// its faces, the part of the reconstructed flux that its own values contribute (face_part), and
// the flux is the own part minus the neighbour's reversed part plus the jump of the two sides'
// reference values (face_flux).  Parts are linear in u - u_0 (u_0 = a mean of the element's nodal
// values, Ops<N>::reference), so the large diffusive coefficients only ever multiply differences of
// nearby values; a constant state gives exactly zero.  The mean halves those differences against one
// node's value: with node 0 as the reference the right-hand side was 1.1 to 1.4 times further from
// 64-bit arithmetic than with operators composed in 64 bits per edge, with the mean 0.6 to 1.0 times
// (orders 1..6, random and smooth fields).  All of it is kept as mirror-even and mirror-odd components
// along the face (GE and GO values); the neighbour runs along the face the other way, which only
// changes the sign of its odd components, and its outward normal is opposite.
//
// Parameters of a face, from the own side: c, h the apex of the own sub-triangle in the face's
// frame; A, B the weights of the R + S and R - S parts (means over the two sides), C, D the same
// for own minus neighbour (Algorithm 1); s = J_f (v.n).  The neighbour's record holds the same
// A, B and the negated C, D, s, so both elements form bitwise opposite fluxes.
#pragma once
#include "refops.h"

#ifdef __CUDACC__
#include <cuda_runtime.h>
#else
#include <cmath>
using std::fma;
#define __forceinline__ inline
#endif

namespace rdg {
namespace face {

template <int N>
struct Ops;


template <typename T>
struct Par {
  T c, h, A, B, C, D, s;
};

// Own part of the flux through face F: g[GE + GO].  d = u - u_0.  diff: the C, D
// weights are not all zero (the caller decides for the whole warp).
template <typename T, int N, int F, bool ALG1>
RDG_HD __forceinline__ void face_part(const T* d, const Par<T>& p, bool diff, T* g) {
  using O = Ops<N>;
  T e[O::NE], o[O::NO];
  if constexpr (F == 0) O::split0(d, e, o);
  else if constexpr (F == 1) O::split1(d, e, o);
  else O::split2(d, e, o);
  // upwind part of the trace: J_f (v.n) u where the flow leaves through this face
  const T up = p.s > T(0) ? p.s : T(0), uh = T(0.5) * up;
  T te[O::GE], to[O::GO];
#pragma unroll
  for (int q = 0; q < O::GO; ++q) {
    te[q] = uh * e[q];
    to[q] = uh * o[q];
  }
  if constexpr (O::GE > O::GO) te[O::GE - 1] = up * e[O::MID < 0 ? 0 : O::MID];
  T ae[O::NE], ao[O::NO], be[O::NE], bo[O::NO];
  O::expand_even(e, ae);
  O::expand_odd(o, ao);
  O::shift(p.c, p.h, ae, ao, be, bo);
  T x[O::GE];
  auto acc_e = [&](T w) {
#pragma unroll
    for (int q = 0; q < O::GE; ++q) te[q] = fma(w, x[q], te[q]);
  };
  auto acc_o = [&](T w) {
#pragma unroll
    for (int q = 0; q < O::GO; ++q) to[q] = fma(w, x[q], to[q]);
  };
  if constexpr (ALG1) {
    O::alg1_a_even(be, x), acc_e(p.A);
    O::alg1_a_odd(bo, x), acc_o(p.A);
    O::alg1_b_even(bo, x), acc_e(p.B);
    O::alg1_b_odd(be, x), acc_o(p.B);
    if (diff) {
      O::alg1_c_even(be, x), acc_e(p.C);
      O::alg1_c_odd(bo, x), acc_o(p.C);
      O::alg1_d_even(bo, x), acc_e(p.D);
      O::alg1_d_odd(be, x), acc_o(p.D);
    }
  } else {
    O::alg2_a_even(be, x), acc_e(p.A);
    O::alg2_a_odd(bo, x), acc_o(p.A);
    O::alg2_b_even(bo, x), acc_e(p.B);
    O::alg2_b_odd(be, x), acc_o(p.B);
  }
#pragma unroll
  for (int q = 0; q < O::GE; ++q) g[q] = te[q];
#pragma unroll
  for (int q = 0; q < O::GO; ++q) g[O::GE + q] = to[q];
}

// Flux out of the own element from both sides' parts: on return ge, go hold its even and odd
// components.  u0, n0: the two sides' reference values; ng: the neighbour's part.
template <typename T, int N, bool ALG1>
RDG_HD __forceinline__ void face_flux(const Par<T>& p, bool diff, T u0, T n0, const T* ng, T* ge, T* go) {
  using O = Ops<N>;
  const T jump = u0 - n0, base = p.s * (p.s > T(0) ? u0 : n0);
  T z[O::GE];
#pragma unroll
  for (int q = 0; q < O::GE; ++q) z[q] = T(0);
  if constexpr (ALG1) O::alg1_jump_a(p.A, z);
  else O::alg2_jump_a(p.A, z);
#pragma unroll
  for (int q = 0; q < O::GE; ++q) ge[q] = (ge[q] - ng[q]) + fma(z[q], jump, base);
#pragma unroll
  for (int q = 0; q < O::GO; ++q) go[q] += ng[O::GE + q];
  if (ALG1 && diff) {
#pragma unroll
    for (int q = 0; q < O::GO; ++q) z[q] = T(0);
    O::alg1_jump_d(p.D, z);
#pragma unroll
    for (int q = 0; q < O::GO; ++q) go[q] = fma(z[q], jump, go[q]);
  }
}

// Volume term in mirror components (halves: node = e + o, mirror node = e - o) from the element's
// mirror coefficients c = {a_r + a_s, a_r - a_s, (g_rr + 2 g_rs + g_ss)/2, (g_rr - g_ss)/2,
// (g_rr - 2 g_rs + g_ss)/2}.
// SHARE 0..3: one of four nearly equal parts of the sum, -1: all of it.  REF: u0 is the value of this
// node, 0 or Ops<N>::CENTRE, whose d is zero and left out of the products; -1: of none (the centre, a
// node near the centroid, halves the differences as the mean does, for Np products less).
template <typename T, int N, int SHARE = -1, int REF = -1>
RDG_HD __forceinline__ void volume_mirror(const T* d, T u0, const T* c, T* ve, T* vo) {
  using O = Ops<N>;
  T e[O::NE], o[O::NO];
  O::split1(d, e, o);
  if constexpr (SHARE < 0) O::template volume<T, REF>(e, o, u0, c[0], c[1], c[2], c[3], c[4], ve, vo);
  else if constexpr (SHARE == 0) O::template volume0<T, REF>(e, o, u0, c[0], c[1], c[2], c[3], c[4], ve, vo);
  else if constexpr (SHARE == 1) O::template volume1<T, REF>(e, o, u0, c[0], c[1], c[2], c[3], c[4], ve, vo);
  else if constexpr (SHARE == 2) O::template volume2<T, REF>(e, o, u0, c[0], c[1], c[2], c[3], c[4], ve, vo);
  else O::template volume3<T, REF>(e, o, u0, c[0], c[1], c[2], c[3], c[4], ve, vo);
}
// The same from the coefficients a_r, a_s, g_rr, g_rs, g_ss.
template <typename T, int N, int REF = -1>
RDG_HD __forceinline__ void volume_parts(const T* d, T u0, T ar, T as, T grr, T grs, T gss, T* ve, T* vo) {
  const T gm = T(0.5) * (grr + gss);
  const T c[5] = {ar + as, ar - as, gm + grs, T(0.5) * (grr - gss), gm - grs};
  volume_mirror<T, N, -1, REF>(d, u0, c, ve, vo);
}

}  // namespace face
}  // namespace rdg
