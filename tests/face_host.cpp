// Host build of the face form's element-local arithmetic (csrc/face_ops.h on the generated
// operators), the same sequence as face_parts_kernel and face_stage_kernel, for the CPU test.
#include <cstdint>

#include "face_ops.h"
namespace rdg {
namespace face {
#include FACE_OPS
}  // namespace face
}  // namespace rdg

using namespace rdg;

// par [K][3][7] (c, h, A, B, C, D, s), nbr [K][3] = 4 element + face, geo [K][6]; rec [K][3][N + 2] is scratch
template <typename T, int N, bool ALG1>
void rhs(int64_t K, const T* u, const double* par, const int64_t* nbr, const double* geo, T* out, T* rec) {
  using O = face::Ops<N>;
  constexpr int NP = O::NP, G = O::GE + O::GO, R = G + 1;
  auto P = [&](int64_t k, int f) {
    const double* q = par + (k * 3 + f) * 7;
    return face::Par<T>{(T)q[0], (T)q[1], (T)q[2], (T)q[3], (T)q[4], (T)q[5], (T)q[6]};
  };
  for (int64_t k = 0; k < K; ++k) {
    T d[NP];
    for (int j = 0; j < NP; ++j) d[j] = u[k * NP + j] - u[k * NP];
    const bool diff = par[k * 21 + 4] != 0 || par[k * 21 + 11] != 0 || par[k * 21 + 18] != 0 || par[k * 21 + 5] != 0 ||
                      par[k * 21 + 12] != 0 || par[k * 21 + 19] != 0;
    face::face_part<T, N, 0, ALG1>(d, P(k, 0), diff, rec + (k * 3 + 0) * R);
    face::face_part<T, N, 1, ALG1>(d, P(k, 1), diff, rec + (k * 3 + 1) * R);
    face::face_part<T, N, 2, ALG1>(d, P(k, 2), diff, rec + (k * 3 + 2) * R);
    for (int f = 0; f < 3; ++f) rec[(k * 3 + f) * R + G] = u[k * NP];
  }
  for (int64_t k = 0; k < K; ++k) {
    T d[NP], v[NP], ve[O::NE], vo[O::NO];
    const T u0 = u[k * NP];
    for (int j = 0; j < NP; ++j) d[j] = u[k * NP + j] - u0;
    const double* g = geo + k * 6;
    face::volume_parts<T, N>(d, u0, (T)g[0], (T)g[1], (T)g[2], (T)g[3], (T)g[4], ve, vo);
    auto lift = [&](int f) {
      const T *own = rec + (k * 3 + f) * R, *nb = rec + ((nbr[k * 3 + f] >> 2) * 3 + (nbr[k * 3 + f] & 3)) * R;
      T ge[O::GE], go[O::GO];
      for (int q = 0; q < O::GE; ++q) ge[q] = own[q];
      for (int q = 0; q < O::GO; ++q) go[q] = own[O::GE + q];
      face::face_flux<T, N, ALG1>(P(k, f), true, u0, nb[G], nb, ge, go);
      for (int q = 0; q < O::GE; ++q) ge[q] *= -(T)g[5];
      for (int q = 0; q < O::GO; ++q) go[q] *= -(T)g[5];
      O::lift_even(ge, ve);
      O::lift_odd(go, vo);
    };
    auto clear = [&]() {
      for (int q = 0; q < O::NE; ++q) ve[q] = 0;
      for (int q = 0; q < O::NO; ++q) vo[q] = 0;
    };
    lift(1);
    O::nodes(ve, vo, v);
    clear();
    lift(0);
    O::join0(ve, vo, v);
    clear();
    lift(2);
    O::join2(ve, vo, v);
    for (int j = 0; j < NP; ++j) out[k * NP + j] = v[j];
  }
}

extern "C" void rhs64(int alg1, int64_t K, const double* u, const double* par, const int64_t* nbr, const double* geo,
                      double* out, double* rec) {
  alg1 ? rhs<double, ORDER, true>(K, u, par, nbr, geo, out, rec) : rhs<double, ORDER, false>(K, u, par, nbr, geo, out, rec);
}
extern "C" void rhs32(int alg1, int64_t K, const float* u, const double* par, const int64_t* nbr, const double* geo,
                      float* out, float* rec) {
  alg1 ? rhs<float, ORDER, true>(K, u, par, nbr, geo, out, rec) : rhs<float, ORDER, false>(K, u, par, nbr, geo, out, rec);
}
