// Face form of a right-hand-side stage (FP32, element-wise D): one kernel per Runge-Kutta stage,
// one thread per element, no per-edge operators.  The element-local arithmetic is face_ops.h.
//
//  face_parts_kernel  each element's part of the flux through its three faces, from a stage input
//  face_stage_kernel  volume term of the stage input, fluxes from the own and the neighbours' parts,
//                     LIFT, sources, the stage update, and the new values' parts for the next stage
//
// Face records (the parts and the element's reference value) are planes of float2 [3 RP][K], so a
// warp stores and reads its own elements' records in whole sectors; two buffers alternate between
// stages, since a block reads its neighbours' records while others already write the next stage's.
#pragma once
#include <cuda_runtime.h>

#include "face_ops.h"
#include "internal.h"
#include "kernel_common.cuh"

namespace rdg {
namespace dev {

template <int N>
__host__ __device__ constexpr int face_block() {
  return 128;
}
template <int N>
__host__ __device__ constexpr int face_min_blocks() {
  return N <= 2 ? 6 : (N <= 4 ? 4 : (N == 5 ? 3 : 2));
}

// Row of NP values in shared memory, read or written with the widest aligned access (NP = 6, 10: 8
// bytes, 28: 16), which is also free of bank conflicts: the row is an odd number of such words.
template <int NP>
__device__ __forceinline__ void row_get(const float* p, float (&v)[NP]) {
  if constexpr (NP % 4 == 0) {
#pragma unroll
    for (int j = 0; j < NP; j += 4) {
      const float4 t = *reinterpret_cast<const float4*>(p + j);
      v[j] = t.x, v[j + 1] = t.y, v[j + 2] = t.z, v[j + 3] = t.w;
    }
  } else if constexpr (NP % 2 == 0) {
#pragma unroll
    for (int j = 0; j < NP; j += 2) {
      const float2 t = *reinterpret_cast<const float2*>(p + j);
      v[j] = t.x, v[j + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < NP; ++j) v[j] = p[j];
  }
}
template <int NP>
__device__ __forceinline__ void row_put(float* p, const float (&v)[NP]) {
  if constexpr (NP % 4 == 0) {
#pragma unroll
    for (int j = 0; j < NP; j += 4) *reinterpret_cast<float4*>(p + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
  } else if constexpr (NP % 2 == 0) {
#pragma unroll
    for (int j = 0; j < NP; j += 2) *reinterpret_cast<float2*>(p + j) = make_float2(v[j], v[j + 1]);
  } else {
#pragma unroll
    for (int j = 0; j < NP; ++j) p[j] = v[j];
  }
}

// A face's parameters: {c, h, A, B}, {C, D, s, neighbour}.
__device__ __forceinline__ face::Par<float> face_par(float4 a, float4 b) {
  return face::Par<float>{a.x, a.y, a.z, a.w, b.x, b.y, b.z};
}

// Parts of element k (values v) through its three faces into the record planes.
template <int N, bool ALG1>
__device__ __forceinline__ void store_parts(const float (&v)[np_of(N)], const float4 (&pa)[3], const float4 (&pb)[3],
                                            float2* out, int64_t K, int64_t k, bool active) {
  using O = face::Ops<N>;
  constexpr int NP = np_of(N), RP = face::rec_pairs(N), G = O::GE + O::GO;
  float d[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) d[j] = v[j] - v[0];
  auto one = [&](auto face_c) {
    constexpr int F = decltype(face_c)::value;
    float g[2 * RP];
    // the own-minus-neighbour weights are zero wherever D does not jump: skipped for whole warps
    const bool diff = ALG1 && __any_sync(0xffffffffu, pb[F].x != 0.f || pb[F].y != 0.f);
    face::face_part<float, N, F, ALG1>(d, face_par(pa[F], pb[F]), diff, g);
    g[G] = v[0];
    if constexpr (G + 1 < 2 * RP) g[G + 1] = 0.f;
    if (active) {
#pragma unroll
      for (int c = 0; c < RP; ++c) out[(int64_t)(F * RP + c) * K + k] = make_float2(g[2 * c], g[2 * c + 1]);
    }
  };
  one(std::integral_constant<int, 0>{});
  one(std::integral_constant<int, 1>{});
  one(std::integral_constant<int, 2>{});
}

// Parts of the stage input's elements [a.k_begin, a.K) (k_begin a multiple of 4: 16-byte rows).
template <int N, bool ALG1>
__global__ void __launch_bounds__(face_block<N>(), face_min_blocks<N>()) face_parts_kernel(FaceArgs a) {
  constexpr int NP = np_of(N), BLK = face_block<N>();
  __shared__ __align__(16) float shs[BLK * NP];
  const int64_t k0 = a.k_begin + (int64_t)blockIdx.x * BLK;
  const int nk = (int)min((int64_t)BLK, a.k_end - k0);
  const int tid = threadIdx.x;
  const bool active = tid < nk;
  const int64_t k = k0 + (active ? tid : nk - 1);
  float4 pa[3], pb[3];
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    pa[f] = __ldg(a.par + (int64_t)(2 * f) * a.K + k);
    pb[f] = __ldg(a.par + (int64_t)(2 * f + 1) * a.K + k);
  }
  wait_for_predecessor();
  allow_dependents();
  {
    Staged<float, BLK, NP> gs;
    gs.load(a.us + k0 * NP, nk * NP);
    gs.store(shs, nk * NP);
  }
  __syncthreads();
  float v[NP];
  row_get<NP>(shs + (active ? tid : nk - 1) * NP, v);
  store_parts<N, ALG1>(v, pa, pb, a.fout, a.K, k, active);
}

// Parts of the Dirichlet ghosts' data, one thread per forcing term and boundary edge: the flux is
// linear in the ghost values sum_m G_m tau_m(t), so their parts are formed once per data set.  A
// ghost's shared face is its second, whose node order is the element's own.
template <int N, bool ALG1>
__global__ void __launch_bounds__(128) face_ghost_kernel(const float* G, const float4* gpar, int64_t B, int64_t n, float* out) {
  using O = face::Ops<N>;
  constexpr int NP = np_of(N), RP = face::rec_pairs(N), NG = O::GE + O::GO;
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (i >= n) return;
  const int64_t b = i % B;
  float d[NP], g[2 * RP];
  const float v0 = G[i * NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) d[j] = G[i * NP + j] - v0;
  face::face_part<float, N, 1, ALG1>(d, face_par(gpar[2 * b], gpar[2 * b + 1]), true, g);
  g[NG] = v0;
  if constexpr (NG + 1 < 2 * RP) g[NG + 1] = 0.f;
#pragma unroll
  for (int c = 0; c < 2 * RP; ++c) out[i * 2 * RP + c] = g[c];
}

template <int N, bool ALG1>
__global__ void __launch_bounds__(face_block<N>(), face_min_blocks<N>()) face_stage_kernel(FaceArgs a) {
  using O = face::Ops<N>;
  constexpr int NP = np_of(N), BLK = face_block<N>(), RP = face::rec_pairs(N), NG = O::GE + O::GO;
  __shared__ __align__(16) float shs[BLK * NP];
  __shared__ __align__(16) float shn[BLK * NP];
  __shared__ float tau_s[RDG_MAX_FORCING_TERMS], tau_g[RDG_MAX_FORCING_TERMS];
  const int64_t k0 = (int64_t)blockIdx.x * BLK;
  const int nk = (int)min((int64_t)BLK, a.K - k0);
  const int tid = threadIdx.x;
  const bool active = tid < nk;
  const int row = active ? tid : nk - 1;
  const int64_t k = k0 + row;
  // the parameters and coefficients are written by no stage: loaded before the dependency wait
  float4 pa[3], pb[3];
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    pa[f] = __ldg(a.par + (int64_t)(2 * f) * a.K + k);
    pb[f] = __ldg(a.par + (int64_t)(2 * f + 1) * a.K + k);
  }
  float geo[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) geo[c] = __ldg(a.geo + c * a.K + k);
  const bool need_un = a.mode == 2 || a.mode == 3 || (a.mode == 4 && a.rka != 0.f);
  wait_for_predecessor();
  allow_dependents();
  float2 own[3][RP], nb[3][RP];
  {
    Staged<float, BLK, NP> gs, gn;
    gs.load(a.us + k0 * NP, nk * NP);
    if (need_un) gn.load(a.un + k0 * NP, nk * NP);
#pragma unroll
    for (int f = 0; f < 3; ++f) {
#pragma unroll
      for (int c = 0; c < RP; ++c) own[f][c] = a.fin[(int64_t)(f * RP + c) * a.K + k];
      const unsigned r = __float_as_uint(pb[f].w), fn = r & 3u;
      int64_t kn = r >> 2;
      if (fn != 3u && kn >= a.K) {   // self-check: record and read the own record instead
        report(a.err, kErrBadIndex);
        kn = k;
      }
#pragma unroll
      for (int c = 0; c < RP; ++c)
        nb[f][c] = fn != 3u ? a.fin[(int64_t)(fn * RP + c) * a.K + kn] : make_float2(0.f, 0.f);
    }
    gs.store(shs, nk * NP);
    if (need_un) gn.store(shn, nk * NP);
  }
  if (tid < a.frc.nsrc) tau_s[tid] = (float)tau_of(a.frc.kind[tid], a.frc.omega[tid], stage_time(a.time));
  if (tid < a.frc.nghost) tau_g[tid] = (float)tau_of(a.frc.gkind[tid], a.frc.gomega[tid], stage_time(a.time));
  __syncthreads();
  float rhs[NP], u0;
  {
    float ve[O::NE], vo[O::NO];
    {
      float d[NP];
      row_get<NP>(shs + row * NP, d);
      u0 = d[0];
#pragma unroll
      for (int j = 0; j < NP; ++j) d[j] -= u0;
      face::volume_parts<float, N>(d, u0, geo[0], geo[1], geo[2], geo[3], geo[4], ve, vo);
    }
    auto flux = [&](int f, float (&ge)[O::GE], float (&go)[O::GO]) {
      float ng[2 * RP], og[2 * RP];
#pragma unroll
      for (int c = 0; c < RP; ++c) {
        og[2 * c] = own[f][c].x, og[2 * c + 1] = own[f][c].y;
        ng[2 * c] = nb[f][c].x, ng[2 * c + 1] = nb[f][c].y;
      }
      const unsigned r = __float_as_uint(pb[f].w);
      if ((r & 3u) == 3u && a.frc.nghost > 0) {   // Dirichlet: the ghost data's parts at the stage time
        const int64_t b = r >> 2;
        if (b < a.B) {
          for (int m = 0; m < a.frc.nghost; ++m) {
            const float* gp = a.gpart + ((int64_t)m * a.B + b) * 2 * RP;
            const float tm = tau_g[m];
#pragma unroll
            for (int c = 0; c <= NG; ++c) ng[c] = fmaf(tm, gp[c], ng[c]);
          }
        } else {
          report(a.err, kErrBadIndex);
        }
      }
#pragma unroll
      for (int q = 0; q < O::GE; ++q) ge[q] = og[q];
#pragma unroll
      for (int q = 0; q < O::GO; ++q) go[q] = og[O::GE + q];
      face::face_flux<float, N, ALG1>(face_par(pa[f], pb[f]), u0, ng[NG], ng, ge, go);
      const float mj = -geo[5];
#pragma unroll
      for (int q = 0; q < O::GE; ++q) ge[q] *= mj;
#pragma unroll
      for (int q = 0; q < O::GO; ++q) go[q] *= mj;
    };
    float ge[O::GE], go[O::GO];
    flux(1, ge, go);              // the second face's order is the element's own
    O::lift_even(ge, ve);
    O::lift_odd(go, vo);
    O::nodes(ve, vo, rhs);
#pragma unroll
    for (int q = 0; q < O::NE; ++q) ve[q] = 0.f;
#pragma unroll
    for (int q = 0; q < O::NO; ++q) vo[q] = 0.f;
    flux(0, ge, go);
    O::lift_even(ge, ve);
    O::lift_odd(go, vo);
    O::join0(ve, vo, rhs);
#pragma unroll
    for (int q = 0; q < O::NE; ++q) ve[q] = 0.f;
#pragma unroll
    for (int q = 0; q < O::NO; ++q) vo[q] = 0.f;
    flux(2, ge, go);
    O::lift_even(ge, ve);
    O::lift_odd(go, vo);
    O::join2(ve, vo, rhs);
  }
  for (int m = 0; m < a.frc.nsrc; ++m) {
    float S[NP];
    row_get<NP>(a.S + ((int64_t)m * a.K + k) * NP, S);
    const float tm = tau_s[m];
#pragma unroll
    for (int i = 0; i < NP; ++i) rhs[i] = fmaf(tm, S[i], rhs[i]);
  }
  if (a.mode >= 1) {
    float us[NP], un[NP];
    row_get<NP>(shs + row * NP, us);
    if (a.mode == 4) {
      // low-storage stage: du' = rka du + dt L, u' = u + rkb du'
      if (need_un) {
        row_get<NP>(shn + row * NP, un);
#pragma unroll
        for (int i = 0; i < NP; ++i) un[i] = fmaf(a.rka, un[i], a.dt * rhs[i]);
      } else {
#pragma unroll
        for (int i = 0; i < NP; ++i) un[i] = a.dt * rhs[i];
      }
#pragma unroll
      for (int i = 0; i < NP; ++i) rhs[i] = fmaf(a.rkb, un[i], us[i]);
      if (active) row_put<NP>(shn + tid * NP, un);
    } else {
#pragma unroll
      for (int i = 0; i < NP; ++i) rhs[i] = fmaf(a.dt, rhs[i], us[i]);
      if (need_un) {
        const float c = a.mode == 2 ? 0.25f : (float)(2.0 / 3.0);   // see rk_combine
        row_get<NP>(shn + row * NP, un);
#pragma unroll
        for (int i = 0; i < NP; ++i) rhs[i] = fmaf(c, rhs[i] - un[i], un[i]);
      }
    }
  }
  if (active) row_put<NP>(shs + tid * NP, rhs);   // a thread rewrites only its own row
  __syncthreads();
  stage_out(a.out + k0 * NP, shs, nk * NP);
  if (a.mode == 4) stage_out(a.out2 + k0 * NP, shn, nk * NP);
  if (a.fout) store_parts<N, ALG1>(rhs, pa, pb, a.fout, a.K, k, active);
}

}  // namespace dev
}  // namespace rdg
