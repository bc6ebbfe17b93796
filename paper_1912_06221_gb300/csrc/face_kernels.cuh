// Face form of a right-hand-side stage (FP32, element-wise D): one kernel per Runge-Kutta stage,
// one thread per element, no per-edge operators.  The element-local arithmetic is face_ops.h.
//
//  face_parts_kernel  each element's part of the flux through its three faces, from a stage input
//  face_stage_kernel  volume term of the stage input, fluxes from the own and the neighbours' parts,
//                     LIFT, sources, the stage update, and the new values' parts for the next stage
//
// A warp owns 32 consecutive elements and never waits for another warp: its rows go through a slice
// of shared memory of its own (cp.async in, 16-byte stores out).  A face record is the N + 1 components of
// the part; records lie in planes [3][K] of 4, 2 and 1 floats (N = 4: a plane of float4 and one of
// float), then one plane [K] of the reference values, so a warp stores and reads its own elements'
// records in whole sectors and each record costs one or two loads.  Two buffers alternate between
// stages, since a warp reads its neighbours' records while others already write the next stage's.
#pragma once
#include <cuda_runtime.h>

#include "face_ops.h"
#include "internal.h"
#include "kernel_common.cuh"

namespace rdg {
namespace dev {

constexpr int kFaceWarps = 4;
constexpr int kFaceBlock = 32 * kFaceWarps;

// How face_stage_kernel is built for a range of sizes (launch_stage in face_order.cu chooses).
//  early: bit 0, the own and the neighbours' records, bit 1, the face parameters are held in registers
//         from before the volume term; otherwise each is loaded where it is used;
//  blocks: resident blocks of 4 warps per SM asked of the compiler;
//  roll: the three faces in a loop over one copy of the code (the values rotate from face to face).
// Few tiles (small): one warp per scheduler hides no latency by itself, so everything is loaded early;
// at orders 5 and 6 a lone warp waits for instructions (70 KB of straight-line code at order 6), so
// the loop is faster there (order 6, 20402 elements: 7.9 against 8.9 us per stage; order 4 no gain).
// More tiles than those warps (large): all tiles resident at once beats two uneven waves.  131072
// elements, small / large: order 1 4.2 / 3.4 us, 2 5.5 / 4.5, 3 7.2 / 6.1, 4 10.8 / 9.2; 65522
// elements: order 5 10.9 / 9.2, 6 14.7 / 13.5 (all with node 0 as the reference value; its mean adds 0 to 2.5%).
struct FaceBuild {
  int early, blocks;
  bool roll;
};
template <int N, bool LARGE>
__host__ __device__ constexpr FaceBuild face_build() {
  if (!LARGE) return N <= 3 ? FaceBuild{3, 5, false} : N == 4 ? FaceBuild{3, 4, false} : FaceBuild{3, N == 5 ? 3 : 2, true};
  return N <= 2 ? FaceBuild{1, 7, false} : N <= 4 ? FaceBuild{0, 7, false} : FaceBuild{N == 5 ? 3 : 0, 4, N == 5};
}
// Resident four-warp blocks per SM of face_team_kernel.
template <int N>
__host__ __device__ constexpr int team_blocks() {
  return N == 4 ? 6 : (N == 5 ? 5 : 4);
}

// Load of stage data.  LIVE: written by other blocks of the same launch (the persistent batch kernel),
// so it is read through L2; otherwise by an earlier kernel.
template <bool LIVE, typename V>
__device__ __forceinline__ V ld_stage(const V* p) {
  if constexpr (LIVE) return __ldcg(p);
  else return *p;
}

// Rows of a warp's elements (n values from a 16-byte aligned start) into its shared slice.
template <int NP, bool LIVE = false>
__device__ __forceinline__ void rows_in(float* sh, const float* g, int n, int lane) {
  const int nv = n / 4;
#pragma unroll
  for (int it = 0; it < (NP + 3) / 4; ++it) {
    const int i = lane + 32 * it;
    if (i < nv)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(sh + 4 * i)),
                   "l"(g + 4 * i)
                   : "memory");
  }
  const int i = nv * 4 + lane;
  if (i < n) sh[i] = ld_stage<LIVE>(g + i);
}
template <int NP>
__device__ __forceinline__ void rows_out(float* g, const float* sh, int n, int lane) {
  const int nv = n / 4;
#pragma unroll
  for (int it = 0; it < (NP + 3) / 4; ++it) {
    const int i = lane + 32 * it;
    if (i < nv) reinterpret_cast<float4*>(g)[i] = reinterpret_cast<const float4*>(sh)[i];
  }
  const int i = nv * 4 + lane;
  if (i < n) g[i] = sh[i];
}
__device__ __forceinline__ void rows_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void rows_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
  __syncwarp();
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

// Element k's face parameters: {c, h, A, B}, s and, where the caller's warp has a jump of D, {C, D}.
__device__ __forceinline__ face::Par<float> face_par(const FaceArgs& a, int f, unsigned k, bool diff) {
  const float4 p = __ldg(a.p4 + (size_t)f * a.K + k);
  const float2 q = diff ? __ldg(a.p2 + (size_t)f * a.K + k) : make_float2(0.f, 0.f);
  return face::Par<float>{p.x, p.y, p.z, p.w, q.x, q.y, __ldg(a.p1 + (size_t)f * a.K + k)};
}

// The own-minus-neighbour weights are zero wherever D does not jump; the face's neighbour word says so,
// and a warp without a jump skips their loads and products.
template <bool ALG1>
__device__ __forceinline__ bool jump_in_warp(unsigned nbr) {
  return ALG1 && __any_sync(0xffffffffu, (nbr & kFaceJump) != 0);
}

// Record r of a buffer of 3 K records: planes of 4, 2 and 1 floats.
template <int NG, bool LIVE>
__device__ __forceinline__ void record_get(const float* buf, size_t K3, unsigned r, float (&v)[NG]) {
  constexpr int N4 = NG / 4 * 4, N2 = N4 + (NG - N4) / 2 * 2;
  if constexpr (NG >= 4) {
    const float4 t = ld_stage<LIVE>(reinterpret_cast<const float4*>(buf) + r);
    v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
  }
  if constexpr (N2 > N4) {
    const float2 t = ld_stage<LIVE>(reinterpret_cast<const float2*>(buf + N4 * K3) + r);
    v[N4] = t.x, v[N4 + 1] = t.y;
  }
  if constexpr (NG > N2) v[N2] = ld_stage<LIVE>(buf + N2 * K3 + r);
}
// The neighbour's record (word r of the neighbour table) and its reference value; of a boundary edge,
// whose data ghost_get supplies, or a corrupt table, any valid one.
template <int NG, bool LIVE>
__device__ __forceinline__ void neighbour_get(const FaceArgs& a, unsigned r, unsigned k, float (&v)[NG + 1]) {
  const unsigned K = (unsigned)a.K, K3 = 3u * K;
  if (r >= K3) {
    if (r >= K3 + (unsigned)a.B) report(a.err, kErrBadIndex);
    r = k;
  }
  float g[NG];
  record_get<NG, LIVE>(a.fin, K3, r, g);
#pragma unroll
  for (int c = 0; c < NG; ++c) v[c] = g[c];
  r -= r >= K ? K : 0u;
  r -= r >= K ? K : 0u;
  v[NG] = ld_stage<LIVE>(a.fin + (size_t)NG * K3 + r);
}
__device__ __forceinline__ float stage_tau(const FaceArgs& a, int m) { return a.tau_row ? a.tau_row[m] : a.tau[m]; }
// Dirichlet: the ghost data's parts at the stage time.
template <int NG>
__device__ __forceinline__ void ghost_get(const FaceArgs& a, unsigned b, float (&v)[NG + 1]) {
#pragma unroll
  for (int c = 0; c <= NG; ++c) v[c] = 0.f;
  if (b >= (unsigned)a.B) return;
  for (int m = 0; m < a.nghost; ++m) {
    const float* gp = a.gpart + ((int64_t)m * a.B + b) * (NG + 1);
    const float tm = stage_tau(a, RDG_MAX_FORCING_TERMS + m);
#pragma unroll
    for (int c = 0; c <= NG; ++c) v[c] = fmaf(tm, gp[c], v[c]);
  }
}
template <int NG>
__device__ __forceinline__ void record_put(float* buf, size_t K3, unsigned r, const float (&v)[NG]) {
  constexpr int N4 = NG / 4 * 4, N2 = N4 + (NG - N4) / 2 * 2;
  if constexpr (NG >= 4) reinterpret_cast<float4*>(buf)[r] = make_float4(v[0], v[1], v[2], v[3]);
  if constexpr (N2 > N4) reinterpret_cast<float2*>(buf + N4 * K3)[r] = make_float2(v[N4], v[N4 + 1]);
  if constexpr (NG > N2) (buf + N2 * K3)[r] = v[N2];
}

// Parts of element k (values v) through its three faces into the record planes.
template <int N, bool ALG1, bool ROLL>
__device__ __forceinline__ void store_parts(const FaceArgs& a, const float (&v)[np_of(N)], const face::Par<float> (&par)[3],
                                            const bool (&diff)[3], unsigned k, bool active) {
  constexpr int NP = np_of(N), NG = N + 1;
  const size_t K3 = 3 * (size_t)a.K;
  const float v0 = face::Ops<N>::reference(v);
  float d[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) d[j] = v[j] - v0;
  auto one = [&](auto face_c) {
    constexpr int F = decltype(face_c)::value;
    float g[NG];
    face::face_part<float, N, F, ALG1>(d, par[F], diff[F], g);
    if (active) record_put<NG>(a.fout, K3, (unsigned)F * (unsigned)a.K + k, g);
  };
  if constexpr (ROLL) {
    face::Par<float> p = par[1];
    bool df = diff[1];
#pragma unroll 1
    for (int i = 0; i < 3; ++i) {
      const int f = i == 2 ? 0 : i + 1;
      float g[NG];
      face::face_part<float, N, 1, ALG1>(d, p, df, g);
      if (active) record_put<NG>(a.fout, K3, (unsigned)f * (unsigned)a.K + k, g);
      face::Ops<N>::rotate(d);
      p = i == 0 ? par[2] : par[0];
      df = i == 0 ? diff[2] : diff[0];
    }
  } else {
    one(std::integral_constant<int, 0>{});
    one(std::integral_constant<int, 1>{});
    one(std::integral_constant<int, 2>{});
  }
  if (active) (a.fout + NG * K3)[k] = v0;
}

// Parts of the nk (>= 1) stage input elements from k0 on, by one warp; sh: 32 rows.
template <int N, bool ALG1, bool ROLL, bool LIVE>
__device__ __forceinline__ void parts_tile(const FaceArgs& a, int64_t k0, int nk, float* sh) {
  constexpr int NP = np_of(N);
  const int lane = threadIdx.x & 31;
  const bool active = lane < nk;
  const int row = active ? lane : nk - 1;
  const unsigned k = (unsigned)(k0 + row);
  face::Par<float> par[3];
  bool diff[3];
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    diff[f] = jump_in_warp<ALG1>(__ldg(a.nbr + (size_t)f * a.K + k));
    par[f] = face_par(a, f, k, diff[f]);
  }
  if constexpr (!LIVE) {
    wait_for_predecessor();
    allow_dependents();
  }
  rows_in<NP, LIVE>(sh, a.us + k0 * NP, nk * NP, lane);
  rows_commit();
  rows_wait<0>();
  float v[NP];
  row_get<NP>(sh + row * NP, v);
  store_parts<N, ALG1, ROLL>(a, v, par, diff, k, active);
}

// Parts of the stage input's elements [k_begin, k_end) (k_begin a multiple of 4: 16-byte rows).
template <int N, bool ALG1>
__global__ void __launch_bounds__(kFaceBlock, face_build<N, false>().blocks)
    face_parts_kernel(const __grid_constant__ FaceArgs a) {
  __shared__ __align__(16) float sh[kFaceWarps][32 * np_of(N)];
  const int warp = threadIdx.x >> 5;
  const int64_t k0 = a.k_begin + ((int64_t)blockIdx.x * kFaceWarps + warp) * 32;
  const int nk = (int)min((int64_t)32, a.k_end - k0);
  if (nk > 0) parts_tile<N, ALG1, face_build<N, false>().roll, false>(a, k0, nk, sh[warp]);
}

// Parts of the Dirichlet ghosts' data, one thread per forcing term and boundary edge: the flux is
// linear in the ghost values sum_m G_m tau_m(t), so their parts are formed once per data set.  A
// ghost's shared face is its second, whose node order is the element's own.
template <int N, bool ALG1>
__global__ void __launch_bounds__(128) face_ghost_kernel(const float* G, const float4* gpar, int64_t B, int64_t n, float* out) {
  constexpr int NP = np_of(N), NG = N + 1;
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (i >= n) return;
  const int64_t b = i % B;
  float d[NP], g[NG];
#pragma unroll
  for (int j = 0; j < NP; ++j) d[j] = G[i * NP + j];
  const float v0 = face::Ops<N>::reference(d);
#pragma unroll
  for (int j = 0; j < NP; ++j) d[j] -= v0;
  const float4 p = gpar[2 * b], q = gpar[2 * b + 1];
  face::face_part<float, N, 1, ALG1>(d, face::Par<float>{p.x, p.y, p.z, p.w, q.x, q.y, q.z}, true, g);
#pragma unroll
  for (int c = 0; c < NG; ++c) out[i * (NG + 1) + c] = g[c];
  out[i * (NG + 1) + NG] = v0;
}

// The neighbour's part (as neighbour_get's record) evaluated from its row of the stage input: the same
// arithmetic as its own parts, so the same bits.  p: the own face's parameters; the neighbour's are the
// same but for its apex (c, h) and the signs of C, D and s.
template <int N, bool ALG1>
__device__ __forceinline__ void neighbour_part(const FaceArgs& a, unsigned r, unsigned k, const face::Par<float>& p, bool diff,
                                               float (&ng)[N + 2]) {
  using O = face::Ops<N>;
  constexpr int NP = np_of(N), NG = N + 1;
  const unsigned K = (unsigned)a.K, K3 = 3u * K;
  if (r >= K3) {
    if (r >= K3 + (unsigned)a.B) report(a.err, kErrBadIndex);
    r = k;
  }
  const int fn = r >= 2u * K ? 2 : (r >= K ? 1 : 0);
  const unsigned kn = r - (unsigned)fn * K;
  const float2 apex = __ldg(reinterpret_cast<const float2*>(a.p4 + r));
  float v[NP], w[NP], n[NG];
  row_get<NP>(a.us + (int64_t)kn * NP, v);
  const float n0 = O::reference(v);
#pragma unroll
  for (int j = 0; j < NP; ++j) w[j] = v[j] -= n0;
  O::rotate(w);
#pragma unroll
  for (int j = 0; j < NP; ++j) v[j] = fn == 1 ? v[j] : w[j];
  O::rotate(w);
#pragma unroll
  for (int j = 0; j < NP; ++j) v[j] = fn == 0 ? w[j] : v[j];
  face::face_part<float, N, 1, ALG1>(v, face::Par<float>{apex.x, apex.y, p.A, p.B, -p.C, -p.D, -p.s}, diff, n);
#pragma unroll
  for (int c = 0; c < NG; ++c) ng[c] = n[c];
  ng[NG] = n0;
}

// One stage of the nk (>= 1) elements from k0 on, by one warp; shs, shn: 32 rows each.  EARLY, ROLL: see
// FaceBuild.  LONE: no records are read, the own and the neighbours' parts are evaluated here (EARLY 3;
// not for the low-storage stage, which updates the rows that other warps still read).
template <int N, bool ALG1, int EARLY, bool ROLL, bool LIVE, bool LONE = false>
__device__ __forceinline__ void stage_tile(const FaceArgs& a, int64_t k0, int nk, float* shs, float* shn) {
  static_assert(!LONE || (EARLY == 3 && !ROLL && !LIVE), "see above");
  using O = face::Ops<N>;
  constexpr bool RECS = EARLY & 1, PARS = EARLY & 2;
  constexpr int NP = np_of(N), NG = N + 1;
  static_assert(NG == O::GE + O::GO, "record size");
  const int lane = threadIdx.x & 31;
  const bool active = lane < nk;
  const int row = active ? lane : nk - 1;
  const unsigned k = (unsigned)(k0 + row), K3 = 3u * (unsigned)a.K;
  // neighbours, coefficients and parameters are written by no stage: loaded before the dependency wait
  unsigned nbr[3];
#pragma unroll
  for (int f = 0; f < 3; ++f) nbr[f] = __ldg(a.nbr + (size_t)f * a.K + k);
  float geo[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) geo[c] = __ldg(a.geo + (size_t)c * a.K + k);
  bool diff[3];
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    diff[f] = jump_in_warp<ALG1>(nbr[f]);
    nbr[f] &= ~kFaceJump;
  }
  face::Par<float> par[3] = {};
  if constexpr (PARS) {
#pragma unroll
    for (int f = 0; f < 3; ++f) par[f] = face_par(a, f, k, diff[f]);
  }
  const bool need_un = a.mode == 2 || a.mode == 3 || (a.mode == 4 && a.rka != 0.f);
  if constexpr (!LIVE) {
    wait_for_predecessor();
    allow_dependents();
  }
  rows_in<NP, LIVE>(shs, a.us + k0 * NP, nk * NP, lane);
  rows_commit();
  if (need_un) rows_in<NP, LIVE>(shn, a.un + k0 * NP, nk * NP, lane);
  rows_commit();
  float own[RECS ? 3 : 1][NG], nb[RECS ? 3 : 1][NG + 1];
  auto records = [&](int f, float (&og)[NG], float (&ng)[NG + 1]) {
    record_get<NG, LIVE>(a.fin, K3, (unsigned)f * (unsigned)a.K + k, og);
    neighbour_get<NG, LIVE>(a, nbr[f], k, ng);
  };
  if constexpr (RECS && !LONE) {
#pragma unroll
    for (int f = 0; f < 3; ++f) records(f, own[f], nb[f]);
  }
  float u0;
  if constexpr (!LONE) u0 = ld_stage<LIVE>(a.fin + (size_t)NG * K3 + k);   // the reference value, with the own record
  rows_wait<1>();
  if constexpr (LONE) {
    float d[NP];
    row_get<NP>(shs + row * NP, d);
    u0 = O::reference(d);
#pragma unroll
    for (int j = 0; j < NP; ++j) d[j] -= u0;
    face::face_part<float, N, 0, ALG1>(d, par[0], diff[0], own[0]);
    face::face_part<float, N, 1, ALG1>(d, par[1], diff[1], own[1]);
    face::face_part<float, N, 2, ALG1>(d, par[2], diff[2], own[2]);
#pragma unroll
    for (int f = 0; f < 3; ++f) neighbour_part<N, ALG1>(a, nbr[f], k, par[f], diff[f], nb[f]);
  }
  float rhs[NP];
  {
    float ve[O::NE], vo[O::NO];
    {
      float d[NP];
      row_get<NP>(shs + row * NP, d);
      const float uc = d[O::CENTRE];
#pragma unroll
      for (int j = 0; j < NP; ++j) d[j] -= uc;
      face::volume_mirror<float, N, -1, O::CENTRE>(d, uc, geo, ve, vo);
    }
    auto flux = [&](int f, float (&ge)[O::GE], float (&go)[O::GO]) {
      float (&og)[NG] = own[RECS ? f : 0], (&ng)[NG + 1] = nb[RECS ? f : 0];
      if constexpr (!RECS) records(f, og, ng);
      const face::Par<float> p = PARS ? par[f] : face_par(a, f, k, diff[f]);
      if (nbr[f] >= K3) ghost_get<NG>(a, nbr[f] - K3, ng);
#pragma unroll
      for (int q = 0; q < O::GE; ++q) ge[q] = og[q];
#pragma unroll
      for (int q = 0; q < O::GO; ++q) go[q] = og[O::GE + q];
      face::face_flux<float, N, ALG1>(p, diff[f], u0, ng[NG], ng, ge, go);
      const float mj = -geo[5];
#pragma unroll
      for (int q = 0; q < O::GE; ++q) ge[q] *= mj;
#pragma unroll
      for (int q = 0; q < O::GO; ++q) go[q] *= mj;
    };
    float ge[O::GE], go[O::GO];
    if constexpr (ROLL) {
      O::nodes(ve, vo, rhs);
#pragma unroll 1
      for (int i = 0; i < 3; ++i) {
        if (i == 0) flux(1, ge, go);
        else if (i == 1) flux(2, ge, go);
        else flux(0, ge, go);
#pragma unroll
        for (int q = 0; q < O::NE; ++q) ve[q] = 0.f;
#pragma unroll
        for (int q = 0; q < O::NO; ++q) vo[q] = 0.f;
        O::lift_even(ge, ve);
        O::lift_odd(go, vo);
        O::join1(ve, vo, rhs);
        O::rotate(rhs);
      }
    } else {
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
  }
  for (int m = 0; m < a.nsrc; ++m) {
    float S[NP];
    row_get<NP>(a.S + ((int64_t)m * a.K + k) * NP, S);
    const float tm = stage_tau(a, m);
#pragma unroll
    for (int i = 0; i < NP; ++i) rhs[i] = fmaf(tm, S[i], rhs[i]);
  }
  rows_wait<0>();
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
      __syncwarp();
      if (active) row_put<NP>(shn + lane * NP, un);
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
  __syncwarp();
  if (active) row_put<NP>(shs + lane * NP, rhs);
  __syncwarp();
  rows_out<NP>(a.out + k0 * NP, shs, nk * NP, lane);
  if (a.mode == 4) rows_out<NP>(a.out2 + k0 * NP, shn, nk * NP, lane);
  if (a.fout) {
    if constexpr (!PARS) {
#pragma unroll
      for (int f = 0; f < 3; ++f) par[f] = face_par(a, f, k, diff[f]);
    }
    store_parts<N, ALG1, ROLL>(a, rhs, par, diff, k, active);
  }
}

template <int N, bool ALG1, bool LARGE>
__global__ void __launch_bounds__(kFaceBlock, face_build<N, LARGE>().blocks)
    face_stage_kernel(const __grid_constant__ FaceArgs a) {
  constexpr FaceBuild build = face_build<N, LARGE>();
  __shared__ __align__(16) float shs[kFaceWarps][32 * np_of(N)];
  __shared__ __align__(16) float shn[kFaceWarps][32 * np_of(N)];
  const int warp = threadIdx.x >> 5;
  for (int64_t tile = (int64_t)blockIdx.x * kFaceWarps + warp; tile * 32 < a.K; tile += (int64_t)gridDim.x * kFaceWarps) {
    stage_tile<N, ALG1, build.early, build.roll, false>(a, tile * 32, (int)min((int64_t)32, a.K - tile * 32), shs[warp],
                                                       shn[warp]);
    __syncwarp();   // the rows before the next tile's
  }
}

// The same stage with four warps on 32 elements: each warp takes a quarter of the volume term, and
// the last three one face each (flux and LIFT before the update, the new parts after it).  A thread of
// face_stage_kernel walks the whole chain alone (N = 4: 1900 instructions, about 1.8 us for a lone
// warp), which sets the stage time where there are few warps per scheduler; here the chain is about a
// third as long.
template <int N, bool ALG1, bool LIVE>
__device__ __forceinline__ void team_tile(const FaceArgs& a, int64_t k0, int nk, float* su, float (*sp)[32 * np_of(N)]) {
  using O = face::Ops<N>;
  constexpr int NP = np_of(N), NG = N + 1, V4 = (NP * 8 + 127) / 128;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = nk * NP, nv = n / 4;
  const bool active = lane < nk;
  const int row = active ? lane : nk - 1;
  const unsigned k = (unsigned)(k0 + row), K = (unsigned)a.K, K3 = 3u * K;
  const int f = warp - 1;               // this warp's face (none for warp 0)
  unsigned nbr = 0;
  bool diff = false;
  face::Par<float> par{};
  if (f >= 0) {
    nbr = __ldg(a.nbr + (size_t)f * K + k);
    diff = jump_in_warp<ALG1>(nbr);
    nbr &= ~kFaceJump;
    par = face_par(a, f, k, diff);
  }
  float geo[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) geo[c] = __ldg(a.geo + (size_t)c * K + k);
  const bool need_un = a.mode == 2 || a.mode == 3 || (a.mode == 4 && a.rka != 0.f);
  if constexpr (!LIVE) {
    wait_for_predecessor();
    allow_dependents();
  }
  const float4* us4 = reinterpret_cast<const float4*>(a.us + k0 * NP);
  float4 un4[V4];
#pragma unroll
  for (int j = 0; j < V4; ++j) {
    const int i = tid + 128 * j;
    if (i < nv)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(su + 4 * i)),
                   "l"(us4 + i)
                   : "memory");
    un4[j] = need_un && i < nv ? ld_stage<LIVE>(reinterpret_cast<const float4*>(a.un + k0 * NP) + i)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if (nv * 4 + tid < n) su[nv * 4 + tid] = ld_stage<LIVE>(a.us + k0 * NP + nv * 4 + tid);
  rows_commit();
  float own[NG], nb[NG + 1];
  const float u0 = ld_stage<LIVE>(a.fin + (size_t)NG * K3 + k);
  if (f >= 0) {
    record_get<NG, LIVE>(a.fin, K3, (unsigned)f * K + k, own);
    neighbour_get<NG, LIVE>(a, nbr, k, nb);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  {
    float d[NP], rhs[NP], ve[O::NE], vo[O::NO], ge[O::GE], go[O::GO];
    row_get<NP>(su + row * NP, d);
    const float uc = d[O::CENTRE];
#pragma unroll
    for (int j = 0; j < NP; ++j) d[j] -= uc;
    auto flux = [&]() {
      if (nbr >= K3) ghost_get<NG>(a, nbr - K3, nb);
#pragma unroll
      for (int q = 0; q < O::GE; ++q) ge[q] = own[q];
#pragma unroll
      for (int q = 0; q < O::GO; ++q) go[q] = own[O::GE + q];
      face::face_flux<float, N, ALG1>(par, diff, u0, nb[NG], nb, ge, go);
#pragma unroll
      for (int q = 0; q < O::GE; ++q) ge[q] *= -geo[5];
#pragma unroll
      for (int q = 0; q < O::GO; ++q) go[q] *= -geo[5];
    };
    auto clear = [&]() {
#pragma unroll
      for (int q = 0; q < O::NE; ++q) ve[q] = 0.f;
#pragma unroll
      for (int q = 0; q < O::NO; ++q) vo[q] = 0.f;
    };
    auto lift = [&]() {
      O::lift_even(ge, ve);
      O::lift_odd(go, vo);
    };
    if (warp == 0) {
      face::volume_mirror<float, N, 0, O::CENTRE>(d, uc, geo, ve, vo);
      O::nodes(ve, vo, rhs);
    } else if (warp == 1) {
      face::volume_mirror<float, N, 1, O::CENTRE>(d, uc, geo, ve, vo);
      O::nodes(ve, vo, rhs);
      flux();
      clear();
      lift();
      O::join0(ve, vo, rhs);
    } else if (warp == 2) {
      face::volume_mirror<float, N, 2, O::CENTRE>(d, uc, geo, ve, vo);
      flux();
      lift();                           // the second face's order is the element's own
      O::nodes(ve, vo, rhs);
    } else {
      face::volume_mirror<float, N, 3, O::CENTRE>(d, uc, geo, ve, vo);
      O::nodes(ve, vo, rhs);
      flux();
      clear();
      lift();
      O::join2(ve, vo, rhs);
    }
    if (active) row_put<NP>(sp[warp] + lane * NP, rhs);
  }
  __syncthreads();
  // the update, value by value: any thread, any value of the tile
  const int64_t g0 = k0 * NP;
  auto update = [&](int i, float un, float& du) {
    float v = (sp[0][i] + sp[1][i]) + (sp[2][i] + sp[3][i]);
    for (int m = 0; m < a.nsrc; ++m) v = fmaf(stage_tau(a, m), a.S[(int64_t)m * a.K * NP + g0 + i], v);
    if (a.mode == 0) return v;
    const float us = su[i];
    if (a.mode == 4) {
      // low-storage stage: du' = rka du + dt L, u' = u + rkb du'
      du = need_un ? fmaf(a.rka, un, a.dt * v) : a.dt * v;
      return fmaf(a.rkb, du, us);
    }
    v = fmaf(a.dt, v, us);
    return need_un ? fmaf(a.mode == 2 ? 0.25f : (float)(2.0 / 3.0), v - un, un) : v;   // see rk_combine
  };
#pragma unroll
  for (int j = 0; j < V4; ++j) {
    const int i = tid + 128 * j;
    if (i < nv) {
      float4 v, du;
      v.x = update(4 * i, un4[j].x, du.x);
      v.y = update(4 * i + 1, un4[j].y, du.y);
      v.z = update(4 * i + 2, un4[j].z, du.z);
      v.w = update(4 * i + 3, un4[j].w, du.w);
      reinterpret_cast<float4*>(su)[i] = v;
      reinterpret_cast<float4*>(a.out + g0)[i] = v;
      if (a.mode == 4) reinterpret_cast<float4*>(a.out2 + g0)[i] = du;
    }
  }
  if (nv * 4 + tid < n) {
    const int i = nv * 4 + tid;
    float du = 0.f;
    const float v = update(i, need_un ? ld_stage<LIVE>(a.un + g0 + i) : 0.f, du);
    su[i] = v;
    a.out[g0 + i] = v;
    if (a.mode == 4) a.out2[g0 + i] = du;
  }
  if (!a.fout) return;
  __syncthreads();
  float d[NP];
  row_get<NP>(su + row * NP, d);
  const float v0 = face::Ops<N>::reference(d);
  if (f >= 0) {
    float g[NG];
#pragma unroll
    for (int j = 0; j < NP; ++j) d[j] -= v0;
    if (f == 0) face::face_part<float, N, 0, ALG1>(d, par, diff, g);
    else if (f == 1) face::face_part<float, N, 1, ALG1>(d, par, diff, g);
    else face::face_part<float, N, 2, ALG1>(d, par, diff, g);
    if (active) record_put<NG>(a.fout, K3, (unsigned)f * K + k, g);
  } else if (active) {
    (a.fout + (size_t)NG * K3)[k] = v0;
  }
}

template <int N, bool ALG1>
__global__ void __launch_bounds__(128, team_blocks<N>()) face_team_kernel(const __grid_constant__ FaceArgs a) {
  __shared__ __align__(16) float su[32 * np_of(N)];
  __shared__ __align__(16) float sp[4][32 * np_of(N)];
  const int64_t k0 = (int64_t)blockIdx.x * 32;
  team_tile<N, ALG1, false>(a, k0, (int)min((int64_t)32, a.K - k0), su, sp);
}

// Order 1, where two launches cost more than the arithmetic: a stage without records in one launch
// (us per stage called on its own, one launch / parts and stage: up to 32768 triangles 2.8 / 4.6, 131072
// 4.7 / 5.8; a right-hand side of 32768 3.8 / 5.9, of 524288 12.8 / 15.4).
template <int N, bool ALG1>
__global__ void __launch_bounds__(kFaceBlock, 5) face_lone_kernel(const __grid_constant__ FaceArgs a) {
  __shared__ __align__(16) float shs[kFaceWarps][32 * np_of(N)];
  __shared__ __align__(16) float shn[kFaceWarps][32 * np_of(N)];
  const int warp = threadIdx.x >> 5;
  const int64_t k0 = ((int64_t)blockIdx.x * kFaceWarps + warp) * 32;
  if (k0 < a.K) stage_tile<N, ALG1, 3, false, false, true>(a, k0, (int)min((int64_t)32, a.K - k0), shs[warp], shn[warp]);
}

// A lone right-hand side of a small mesh in one launch: a thread evaluates its neighbours' parts beside
// its own (the same arithmetic on the neighbour's row, so the same bits) instead of reading records of a
// first launch.  Twice the parts' work, which is free while there is at most a warp per scheduler; what
// bounds such a call is its launches (order 2, 512 triangles).
template <int N, bool ALG1>
__global__ void __launch_bounds__(kFaceBlock) face_rhs_kernel(const __grid_constant__ FaceArgs a) {
  using O = face::Ops<N>;
  constexpr int NP = np_of(N), NG = N + 1;
  __shared__ __align__(16) float sh_all[kFaceWarps][32 * NP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float* sh = sh_all[warp];
  const int64_t k0 = ((int64_t)blockIdx.x * kFaceWarps + warp) * 32;
  const int nk = (int)min((int64_t)32, a.K - k0);
  if (nk <= 0) return;
  const bool active = lane < nk;
  const int row = active ? lane : nk - 1;
  const unsigned k = (unsigned)(k0 + row), K = (unsigned)a.K, K3 = 3u * K;
  unsigned nbr[3];
  bool diff[3];
  float geo[6];
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    nbr[f] = __ldg(a.nbr + (size_t)f * K + k);
    diff[f] = jump_in_warp<ALG1>(nbr[f]);
    nbr[f] &= ~kFaceJump;
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) geo[c] = __ldg(a.geo + (size_t)c * K + k);
  wait_for_predecessor();
  allow_dependents();
  rows_in<NP>(sh, a.us + k0 * NP, nk * NP, lane);
  rows_commit();
  rows_wait<0>();
  float d[NP], rhs[NP];
  row_get<NP>(sh + row * NP, d);
  const float u0 = face::Ops<N>::reference(d);
#pragma unroll
  for (int j = 0; j < NP; ++j) d[j] -= u0;
  {
    float ve[O::NE], vo[O::NO];
    face::volume_mirror<float, N>(d, u0, geo, ve, vo);
    O::nodes(ve, vo, rhs);
  }
#pragma unroll 1
  for (int i = 0; i < 3; ++i) {         // faces 1, 2, 0: d and rhs rotate into the face's order
    const int f = i == 2 ? 0 : i + 1;
    const unsigned r = i == 0 ? nbr[1] : (i == 1 ? nbr[2] : nbr[0]);
    const bool df = i == 0 ? diff[1] : (i == 1 ? diff[2] : diff[0]);
    const face::Par<float> p = face_par(a, f, k, df);
    float g[NG], ng[NG + 1];
    face::face_part<float, N, 1, ALG1>(d, p, df, g);
    neighbour_part<N, ALG1>(a, r, k, p, df, ng);
    if (r >= K3) ghost_get<NG>(a, r - K3, ng);
    float ge[O::GE], go[O::GO], ve[O::NE], vo[O::NO];
#pragma unroll
    for (int q = 0; q < O::GE; ++q) ge[q] = g[q];
#pragma unroll
    for (int q = 0; q < O::GO; ++q) go[q] = g[O::GE + q];
    face::face_flux<float, N, ALG1>(p, df, u0, ng[NG], ng, ge, go);
#pragma unroll
    for (int q = 0; q < O::GE; ++q) ge[q] *= -geo[5];
#pragma unroll
    for (int q = 0; q < O::GO; ++q) go[q] *= -geo[5];
#pragma unroll
    for (int q = 0; q < O::NE; ++q) ve[q] = 0.f;
#pragma unroll
    for (int q = 0; q < O::NO; ++q) vo[q] = 0.f;
    O::lift_even(ge, ve);
    O::lift_odd(go, vo);
    O::join1(ve, vo, rhs);
    O::rotate(rhs);
    O::rotate(d);
  }
  for (int m = 0; m < a.nsrc; ++m) {
    float S[NP];
    row_get<NP>(a.S + ((int64_t)m * a.K + k) * NP, S);
    const float tm = stage_tau(a, m);
#pragma unroll
    for (int i = 0; i < NP; ++i) rhs[i] = fmaf(tm, S[i], rhs[i]);
  }
  __syncwarp();
  if (active) row_put<NP>(sh + lane * NP, rhs);
  __syncwarp();
  rows_out<NP>(a.out + k0 * NP, sh, nk * NP, lane);
}

}  // namespace dev
}  // namespace rdg
