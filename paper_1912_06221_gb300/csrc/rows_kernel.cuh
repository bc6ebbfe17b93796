// One-kernel FP64 stage of small meshes: a lane per (element, node) instead of a thread per element.
// An FP64 warp instruction holds its quarter of the SM for 64 cycles here (2 multiply-adds per clock
// per SM), so a thread that walks an element's products alone sets the stage time where there are few
// elements: order 2, 512 triangles, two kernels 13.3 us per stage (about 190 serial multiply-adds on
// 16 of 608 schedulers).  With a lane per node a warp holds 32 / Np elements and its chain is one row
// of each product: 70 FP64 instructions at order 2, 115 at order 4.  The price is dense rows and every
// edge's flux evaluated by both of its elements (bitwise the same, the operator's rows in the same
// order), about twice the pipe time per element, which is free while schedulers are idle.
// Included by rhs_order.cu for FP64, after rhs_kernels.cuh.
#pragma once

namespace rdg {
namespace dev {

template <int N>
struct RowsShape {
  static constexpr int NP = np_of(N), NFP = nfp_of(N), NQ = 3 * NFP;
  static constexpr int EPW = 32 / NP;                       // elements per warp
  static constexpr int WARPS = 4;
  static constexpr int TAB = 4 * NP * NP + NQ * NP;         // Dr^T, Ds^T, Wr^T, Ws^T, LIFT^T: lanes read along a row
};

template <int N, int MODE>
__global__ void __launch_bounds__(32 * RowsShape<N>::WARPS) rows_stage_kernel(const __grid_constant__ EdgeArgs<double> ea,
                                                                              const __grid_constant__ ElemArgs<double> a,
                                                                              const double* __restrict__ table) {
  static_assert(MODE >= 0 && MODE <= 3, "other lanes gather from the stage input: it may not be updated in place");
  using R = RowsShape<N>;
  constexpr int NP = R::NP, NFP = R::NFP, NQ = R::NQ, EPW = R::EPW, RW = 2 * NP - 1;
  constexpr int QW = EdgeWords<double, N>::QW, NWS = EdgeWords<double, N>::NWS;
  __shared__ __align__(16) double tab[R::TAB];
  __shared__ double sv[R::WARPS][4][EPW * NP];              // the element's values, its three neighbours'
  __shared__ double sx[R::WARPS][3][2][EPW * NP];           // per face, both sides' values less the edge's u_0
  __shared__ double sd[R::WARPS][EPW * NP], sf[R::WARPS][2][EPW * NP], sq[R::WARPS][EPW * NQ];
  __shared__ double tau_s[RDG_MAX_FORCING_TERMS], tau_g[RDG_MAX_FORCING_TERMS];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int e = lane / NP, i = lane % NP, at = lane < EPW * NP ? lane : 0;
  const int64_t k = ((int64_t)blockIdx.x * R::WARPS + w) * EPW + e;
  const bool on = e < EPW && k < a.K;
  // what no stage writes, before the dependency wait
  for (int j = tid; j < R::TAB / 2; j += 32 * R::WARPS)
    reinterpret_cast<double2*>(tab)[j] = __ldg(reinterpret_cast<const double2*>(table) + j);
  if (R::TAB % 2 && tid == 0) tab[R::TAB - 1] = __ldg(table + R::TAB - 1);
  int er[3] = {0, 0, 0}, kn[3] = {0, 0, 0};
  double geo[6] = {};
  if (on) {
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      er[f] = a.eref[(int64_t)f * a.K + k];
      if (er[f] < 0 || (er[f] >> 1) >= a.E) {   // self-check: record and use edge 0 instead
        report(a.err, kErrBadIndex);
        er[f] = 0;
      }
      kn[f] = (er[f] & 1) ? ea.k1[er[f] >> 1] : ea.k2[er[f] >> 1];
      if (kn[f] >= 0 ? kn[f] >= a.K : (-1 - (int64_t)kn[f]) >= ea.B) {
        report(a.err, kErrBadIndex);
        kn[f] = 0;
      }
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) geo[c] = a.geo[(int64_t)c * a.K + k];
  }
  wait_for_predecessor();
  allow_dependents();
  if (tid < a.frc.nsrc) tau_s[tid] = tau_of(a.frc.kind[tid], a.frc.omega[tid], stage_time(a.time));
  if (tid >= 16 && tid - 16 < a.frc.nghost)
    tau_g[tid - 16] = tau_of(a.frc.gkind[tid - 16], a.frc.gomega[tid - 16], stage_time(a.time));
  __syncthreads();
  double u = 0.0;
  if (on) {
    u = a.us[k * NP + i];
    sv[w][0][at] = u;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      double v = 0.0;
      if (kn[f] >= 0) {
        v = a.us[(int64_t)kn[f] * NP + i];
      } else {                                   // Dirichlet: the ghost data at the stage time
        const int64_t b = -1 - (int64_t)kn[f];
        for (int m = 0; m < a.frc.nghost; ++m) v += tau_g[m] * ea.G[((int64_t)m * ea.B + b) * NP + i];
      }
      sv[w][1 + f][at] = v;
    }
  }
  __syncwarp();
  if (on) {
    sd[w][at] = u - sv[w][0][e * NP];
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      const bool side2 = er[f] & 1;
      const double ub = side2 ? sv[w][1 + f][e * NP] : sv[w][0][e * NP], v = sv[w][1 + f][at];
      sx[w][f][0][at] = (side2 ? v : u) - ub;
      sx[w][f][1][at] = (side2 ? u : v) - ub;
    }
  }
  __syncwarp();
  if (on) {
    // volume flux at node i
    double ur = 0.0, us = 0.0;
#pragma unroll
    for (int j = 1; j < NP; ++j) {
      ur = fma(tab[j * NP + i], sd[w][e * NP + j], ur);
      us = fma(tab[NP * NP + j * NP + i], sd[w][e * NP + j], us);
    }
    double pr = geo[2] * ur + geo[3] * us, ps = geo[3] * ur + geo[4] * us;
    if (ea.Dn) {                                 // D given at the nodes
      const double dn = __ldg(ea.Dn + k * NP + i);
      pr *= dn;
      ps *= dn;
    }
    sf[w][0][at] = geo[0] * u - pr;
    sf[w][1][at] = geo[1] * u - ps;
    // face fluxes i, i + Np, ... of the element's 3 Nfp, in its own face orders
    for (int q = i; q < NQ; q += NP) {
      const int f = q / NFP, c = q % NFP;
      const int ef = f == 0 ? er[0] : (f == 1 ? er[1] : er[2]);
      const bool side2 = ef & 1;
      const int64_t id = ef >> 1;
      const int r = side2 ? NFP - 1 - c : c;
      const double* W = static_cast<const double*>(ea.W) + ((id >> 5) * QW * kTile + (id & 31)) * 2;
      const double *x1 = &sx[w][f][0][e * NP], *x2 = &sx[w][f][1][e * NP];
      double acc = 0.0;
#pragma unroll
      for (int j = 0; j < RW; ++j) {
        const int idx = r * RW + j;
        acc = fma(__ldg(W + (idx >> 1) * (2 * kTile) + (idx & 1)), j < NP - 1 ? x1[j + 1] : x2[j - (NP - 1)], acc);
      }
      acc = fma(__ldg(W + ((NWS - 1) >> 1) * (2 * kTile) + ((NWS - 1) & 1)),
                side2 ? sv[w][1 + f][e * NP] : sv[w][0][e * NP], acc);
      sq[w][e * NQ + q] = side2 ? -acc : acc;
    }
  }
  __syncwarp();
  if (!on) return;
  double vr = 0.0, vs = 0.0, sl = 0.0;
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    vr = fma(tab[2 * NP * NP + j * NP + i], sf[w][0][e * NP + j], vr);
    vs = fma(tab[3 * NP * NP + j * NP + i], sf[w][1][e * NP + j], vs);
  }
#pragma unroll
  for (int q = 0; q < NQ; ++q) sl = fma(tab[4 * NP * NP + q * NP + i], sq[w][e * NQ + q], sl);
  double rhs = fma(-geo[5], sl, vr + vs);
  for (int m = 0; m < a.frc.nsrc; ++m) rhs = fma(tau_s[m], a.S[((int64_t)m * a.K + k) * NP + i], rhs);
  if (MODE >= 1) rhs = fma(a.dt, rhs, u);
  if (MODE >= 2) rhs = rk_combine<double, MODE>(a.un[k * NP + i], rhs);
  a.out[k * NP + i] = rhs;
}

}  // namespace dev

template <int N>
inline int launch_rows_t(int mode, const EdgeArgs<double>& ea, const ElemArgs<double>& a, const double* table, cudaStream_t s) {
  using R = dev::RowsShape<N>;
  if (a.K == 0) return RDG_OK;
  const unsigned g = (unsigned)((a.K + R::WARPS * R::EPW - 1) / (R::WARPS * R::EPW));
  constexpr unsigned b = 32 * R::WARPS;
  switch (mode) {
    case 0: return launch_pdl(dev::rows_stage_kernel<N, 0>, g, b, s, ea, a, table);
    case 1: return launch_pdl(dev::rows_stage_kernel<N, 1>, g, b, s, ea, a, table);
    case 2: return launch_pdl(dev::rows_stage_kernel<N, 2>, g, b, s, ea, a, table);
    case 3: return launch_pdl(dev::rows_stage_kernel<N, 3>, g, b, s, ea, a, table);
    default: return RDG_EINVAL;   // the low-storage stage updates its input in place
  }
}

}  // namespace rdg
