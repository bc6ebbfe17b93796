// Build-time generator of the face-form arithmetic of one order (face_ops_<N>.h): the constant
// matrices of the method, split by the mirror symmetry of the reference triangle and written out
// as straight-line multiply-adds with literal coefficients.
//
// Why literals: the matrices are the same for every element, so a thread that owns an element
// needs one coefficient per multiply-add.  As immediates they cost nothing beside the instruction
// itself; from constant memory a run of a few hundred different coefficients misses the small
// immediate-constant cache at every line, and from shared memory each costs a load slot.
//
// Why the mirror symmetry: every operator commutes (or anticommutes) with the mirror that swaps
// r and s, so acting on sums e = u_i + u_mirror(i) and differences o = u_i - u_mirror(i) halves
// the multiply-adds of every product.
//
// Frame of a face (the rotated frame of Sec. 4.4 with the face on the hypotenuse): x = (s - r)/2
// runs along the face, t = -(r + s)/2 away from it.  A nodal field is expanded in t^j P_k(x),
// j + k <= N.  The sub-triangle of the enclosed parallelogram has its apex at (x, t) = (c, h) and
// shares the face, so its own coordinates are x = x' + c t', t = h t': the projection of Eq.
// totalProjection is b_{J,K} = sum_s c^s h^(J-s) sum_k S^s_{K,k} a_{J-s,k}, about 3 Np
// multiply-adds instead of the 2 Np^2 of V_p V^{-1}.  The reconstruction, its gradient on the
// diagonal and the interface rule are then fixed Nfp x Np matrices on b, weighted by up to four
// numbers of the edge.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "refops.h"

using namespace rdg;
using Mat = std::vector<double>;

namespace {

Mat mul(const Mat& A, const Mat& B, int n, int k, int m) {
  Mat C((size_t)n * m, 0.0);
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < m; ++j) {
      long double s = 0;
      for (int l = 0; l < k; ++l) s += (long double)A[(size_t)i * k + l] * B[(size_t)l * m + j];
      C[(size_t)i * m + j] = (double)s;
    }
  return C;
}

Mat inverse(const Mat& A, int n) {
  std::vector<long double> a(A.begin(), A.end()), b((size_t)n * n, 0.0L);
  for (int i = 0; i < n; ++i) b[(size_t)i * n + i] = 1;
  for (int c = 0; c < n; ++c) {
    int p = c;
    for (int r = c + 1; r < n; ++r)
      if (std::fabs(a[(size_t)r * n + c]) > std::fabs(a[(size_t)p * n + c])) p = r;
    if (a[(size_t)p * n + c] == 0) { std::fprintf(stderr, "singular basis\n"); std::exit(1); }
    for (int j = 0; j < n; ++j) {
      std::swap(a[(size_t)p * n + j], a[(size_t)c * n + j]);
      std::swap(b[(size_t)p * n + j], b[(size_t)c * n + j]);
    }
    const long double d = 1 / a[(size_t)c * n + c];
    for (int j = 0; j < n; ++j) { a[(size_t)c * n + j] *= d; b[(size_t)c * n + j] *= d; }
    for (int r = 0; r < n; ++r) {
      const long double f = a[(size_t)r * n + c];
      if (r == c || f == 0) continue;
      for (int j = 0; j < n; ++j) { a[(size_t)r * n + j] -= f * a[(size_t)c * n + j]; b[(size_t)r * n + j] -= f * b[(size_t)c * n + j]; }
    }
  }
  return Mat(b.begin(), b.end());
}

// Legendre P_k(x) and the coefficients of d/dx in the Legendre basis: P_k' = sum (2m+1) P_m, m = k-1, k-3, ...
double legendre(int k, double x) {
  double p0 = 1, p1 = x;
  if (k == 0) return 1;
  for (int n = 1; n < k; ++n) { const double p2 = ((2 * n + 1) * x * p1 - n * p0) / (n + 1); p0 = p1; p1 = p2; }
  return p1;
}

struct Gen {
  int N, Np, Nfp;
  const RefOps* o;
  std::vector<int> mir, er, eo;      // mirror; even and odd components' representatives (pairs first)
  int NE, NO, GE, GO;
  std::vector<std::pair<int, int>> jk;
  std::vector<int> ae, ao;           // expansion terms with k even / odd (indices into jk)
  std::vector<int> P[3];             // rotated node l of face f is element node P[f][l]

  std::string lit(double v) const {
    char buf[64];
    std::snprintf(buf, sizeof buf, "T(%a)", v);
    return buf;
  }
  // y = M x (or y += M x), column by column, zeros left out
  void product(const Mat& M, int n, int m, const char* x, const char* y, bool add, double scale = 0) const {
    double top = scale;
    for (double v : M) top = std::max(top, std::fabs(v));
    std::vector<bool> begun(n, add);
    for (int j = 0; j < m; ++j)
      for (int i = 0; i < n; ++i) {
        const double v = M[(size_t)i * m + j];
        if (std::fabs(v) <= 1e-13 * top) continue;
        if (begun[i]) std::printf("    %s[%d] = fma(%s, %s[%d], %s[%d]);\n", y, i, lit(v).c_str(), x, j, y, i);
        else std::printf("    %s[%d] = %s * %s[%d];\n", y, i, lit(v).c_str(), x, j);
        begun[i] = true;
      }
    for (int i = 0; i < n; ++i)
      if (!begun[i]) std::printf("    %s[%d] = T(0);\n", y, i);
  }
  void open(const char* sig, const char* more = "", const char* ret = "void") const {
    std::printf("  template <typename T%s>\n  static RDG_HD __forceinline__ %s %s {\n", more, ret, sig);
  }
  void close() const { std::printf("  }\n"); }

  int rep(bool even, int c) const { return even ? er[c] : eo[c]; }
  // Nodal matrix M [rows nodes][cols nodes] between mirror components.  Inputs are sums/differences
  // (fixed nodes: the value), or halves of them ("values": node = e' + o') when in_val; outputs are halves.
  Mat comp(const Mat& M, bool out_even, bool in_even, bool in_val) const {
    const int n = out_even ? NE : NO, m = in_even ? NE : NO;
    Mat R((size_t)n * m, 0.0);
    for (int a = 0; a < n; ++a)
      for (int b = 0; b < m; ++b) {
        const int i = rep(out_even, a), j = rep(in_even, b);
        auto at = [&](int ii) {
          if (mir[j] == j) return M[(size_t)ii * Np + j];
          const double v = M[(size_t)ii * Np + j] + (in_even ? 1 : -1) * M[(size_t)ii * Np + mir[j]];
          return in_val ? v : 0.5 * v;
        };
        R[(size_t)a * m + b] = mir[i] == i ? at(i) : 0.5 * (at(i) + (out_even ? 1 : -1) * at(mir[i]));
      }
    return R;
  }

  void run() {
    Np = o->Np;
    Nfp = o->Nfp;
    for (int i = 0; i < Np; ++i) {
      int best = -1;
      for (int j = 0; j < Np; ++j)
        if (std::hypot(o->r[j] - o->s[i], o->s[j] - o->r[i]) < 1e-10) best = j;
      if (best < 0) { std::fprintf(stderr, "node set not mirror symmetric\n"); std::exit(1); }
      mir.push_back(best);
    }
    // pairs: the face's own nodes first, oriented along the face, then the others, then fixed nodes
    std::vector<bool> seen(Np, false);
    for (int q = 0; q < Nfp / 2; ++q) {
      const int i = o->hyp[q];
      if (mir[i] != o->hyp[Nfp - 1 - q]) { std::fprintf(stderr, "face nodes not mirror symmetric\n"); std::exit(1); }
      er.push_back(i);
      seen[i] = seen[mir[i]] = true;
    }
    for (int i = 0; i < Np; ++i)
      if (!seen[i] && mir[i] != i) { er.push_back(i); seen[i] = seen[mir[i]] = true; }
    eo = er;
    NO = (int)eo.size();
    for (int i = 0; i < Np; ++i)
      if (mir[i] == i) er.push_back(i);
    NE = (int)er.size();
    GE = (Nfp + 1) / 2;
    GO = Nfp / 2;
    for (int j = 0; j <= N; ++j)
      for (int k = 0; k <= N - j; ++k) {
        (k % 2 ? ao : ae).push_back((int)jk.size());
        jk.push_back({j, k});
      }
    if ((int)ae.size() != NE || (int)ao.size() != NO) { std::fprintf(stderr, "parity counts differ\n"); std::exit(1); }
    for (int f = 0; f < 3; ++f) {
      P[f].assign(Np, -1);
      for (int i = 0; i < Np; ++i) P[f][o->perm[f * Np + i]] = i;
    }
    for (int l = 0; l < Np; ++l)
      if (P[1][l] != l) { std::fprintf(stderr, "face 2's ordering is not the element's\n"); std::exit(1); }

    int fixed_face = -1;   // the face's middle node among the even components
    int centre = -1;       // the node of the mirror axis nearest the centroid
    for (int i = 0; i < Np; ++i)
      if (mir[i] == i && (centre < 0 || std::fabs(o->r[i] + 1.0 / 3) < std::fabs(o->r[centre] + 1.0 / 3) - 1e-9)) centre = i;
    for (int c = 0; c < NE; ++c) {
      if (Nfp % 2 && er[c] == o->hyp[Nfp / 2]) fixed_face = c;
    }
    std::printf("template <>\nstruct Ops<%d> {\n", N);
    std::printf("  static constexpr int NP = %d, NE = %d, NO = %d, GE = %d, GO = %d, MID = %d, CENTRE = %d;\n", Np, NE, NO, GE, GO,
                fixed_face, centre);

    // the reference value: the mean over the vertices and the innermost ring of three nodes (order 1: the
    // vertices), taken of differences so that a constant state's is exactly its value.  All Np nodes gave
    // the same error for 3 to 5 times the operations.
    {
      std::vector<int> L;
      double inner = 1e30;
      for (int i = 0; i < Np; ++i) {
        const double d = std::hypot(std::hypot(o->r[i] + 1.0 / 3, o->s[i] + 1.0 / 3), o->r[i] + o->s[i] + 2.0 / 3);
        if (P[2][i] != i && d < inner - 1e-9) {
          inner = d;
          L = {i, P[2][i], P[2][P[2][i]]};
        }
      }
      if (N > 1) L.insert(L.end(), {0, P[2][0], P[2][P[2][0]]});
      const double w = 1.0 / (double)L.size();
      open("reference(const T* v)", "", "T");
      std::printf("    T s[2] = {T(0), T(0)};\n");
      int c = 0;
      for (int i : L)
        if (i != 0) {
          std::printf("    s[%d] = fma(v[%d] - v[0], %s, s[%d]);\n", c % 2, i, lit(w).c_str(), c % 2);
          ++c;
        }
      std::printf("    return v[0] + (s[0] + s[1]);\n");
      close();
    }

    // mirror sums and differences of d in face f's order (face 1: the element's own)
    for (int f = 0; f < 3; ++f) {
      char sig[96];
      std::snprintf(sig, sizeof sig, "split%d(const T* d, T* e, T* o)", f);
      open(sig);
      for (int c = 0; c < NE; ++c) {
        const int i = P[f][er[c]], j = P[f][mir[er[c]]];
        if (i == j) std::printf("    e[%d] = d[%d];\n", c, i);
        else std::printf("    e[%d] = d[%d] + d[%d];\n    o[%d] = d[%d] - d[%d];\n", c, i, j, c, i, j);
      }
      close();
      // nodal values from halves, added to v
      std::snprintf(sig, sizeof sig, "join%d(const T* e, const T* o, T* v)", f);
      open(sig);
      for (int c = 0; c < NE; ++c) {
        const int i = P[f][er[c]], j = P[f][mir[er[c]]];
        if (i == j) std::printf("    v[%d] += e[%d];\n", i, c);
        else std::printf("    v[%d] += e[%d] + o[%d];\n    v[%d] += e[%d] - o[%d];\n", i, c, c, j, c, c);
      }
      close();
    }
    // the element's values in the next face's order: faces 1, 2, 0 (and back to 1) in turn
    for (int l = 0; l < Np; ++l)
      if (P[2][P[2][l]] != P[0][l] || P[2][P[0][l]] != l) { std::fprintf(stderr, "face orderings are not a rotation\n"); std::exit(1); }
    open("rotate(T* v)");
    for (int l = 0; l < Np; ++l) {   // cycles of three
      const int b = P[2][l], c = P[2][b];
      if (l < b && l < c) std::printf("    { const T t = v[%d]; v[%d] = v[%d]; v[%d] = v[%d]; v[%d] = t; }\n", l, l, b, b, c, c);
    }
    close();
    open("nodes(const T* e, const T* o, T* v)");
    for (int c = 0; c < NE; ++c) {
      const int i = er[c], j = mir[er[c]];
      if (i == j) std::printf("    v[%d] = e[%d];\n", i, c);
      else std::printf("    v[%d] = e[%d] + o[%d];\n    v[%d] = e[%d] - o[%d];\n", i, c, c, j, c, c);
    }
    close();

    // expansion coefficients of the face frame from sums and differences
    Mat B((size_t)Np * Np);
    for (int i = 0; i < Np; ++i) {
      const double x = (o->s[i] - o->r[i]) / 2, t = -(o->r[i] + o->s[i]) / 2;
      for (int c = 0; c < Np; ++c) B[(size_t)i * Np + c] = std::pow(t, jk[c].first) * legendre(jk[c].second, x);
    }
    const Mat Ti = inverse(B, Np);
    for (int odd = 0; odd < 2; ++odd) {
      const auto& rows = odd ? ao : ae;
      const int n = (int)rows.size();
      Mat M((size_t)n * n, 0.0);
      for (int a = 0; a < n; ++a)
        for (int c = 0; c < n; ++c) {
          const int j = odd ? eo[c] : er[c];
          const double v = Ti[(size_t)rows[a] * Np + j];
          M[(size_t)a * n + c] = mir[j] == j ? v : 0.5 * (v + (odd ? -1 : 1) * Ti[(size_t)rows[a] * Np + mir[j]]);
        }
      open(odd ? "expand_odd(const T* o, T* a)" : "expand_even(const T* e, T* a)");
      product(M, n, n, odd ? "o" : "e", "a", false);
      close();
    }

    // sub-triangle coefficients: t^j scaled by h^j, then the shift x' + c t', Horner in c
    open("shift(T c, T h, T* ae, T* ao, T* be, T* bo)");
    std::vector<std::string> name(Np), bname(Np);
    for (int i = 0; i < NE; ++i) { name[ae[i]] = "ae[" + std::to_string(i) + "]"; bname[ae[i]] = "be[" + std::to_string(i) + "]"; }
    for (int i = 0; i < NO; ++i) { name[ao[i]] = "ao[" + std::to_string(i) + "]"; bname[ao[i]] = "bo[" + std::to_string(i) + "]"; }
    std::printf("    T hp = h;\n");
    for (int j = 1; j <= N; ++j) {
      for (int q = 0; q < Np; ++q)
        if (jk[q].first == j) std::printf("    %s *= hp;\n", name[q].c_str());
      if (j < N) std::printf("    hp *= h;\n");
    }
    // D[s][k] = Legendre coefficients of P_k^(s) / s!
    std::vector<std::vector<std::vector<double>>> D(N + 1, std::vector<std::vector<double>>(N + 1, std::vector<double>(N + 1, 0.0)));
    for (int k = 0; k <= N; ++k) D[0][k][k] = 1;
    for (int s = 1; s <= N; ++s)
      for (int k = 0; k <= N; ++k)
        for (int m = 0; m <= N; ++m)
          for (int q = m - 1; q >= 0; q -= 2) D[s][k][q] += D[s - 1][k][m] * (2 * q + 1) / s;
    for (int q = 0; q < Np; ++q) {
      const int J = jk[q].first, K = jk[q].second;
      bool begun = false;
      std::printf("    {\n      T v;\n");
      for (int s = std::min(J, N); s >= 0; --s) {
        bool first = true;
        for (int p = 0; p < Np; ++p) {
          if (jk[p].first != J - s) continue;
          const double v = D[s][jk[p].second][K];
          if (v == 0) continue;
          if (first && begun) std::printf("      v = fma(v, c, %s);\n", v == 1 ? name[p].c_str() : (lit(v) + " * " + name[p]).c_str());
          else if (first) std::printf("      v = %s;\n", v == 1 ? name[p].c_str() : (lit(v) + " * " + name[p]).c_str());
          else std::printf("      v = fma(%s, %s, v);\n", lit(v).c_str(), name[p].c_str());
          first = false;
          begun = true;
        }
        if (first && begun) std::printf("      v *= c;\n");
      }
      std::printf("      %s = v;\n    }\n", bname[q].c_str());
    }
    close();

    // flux contributions of the own side: weights A, B (means over the two sides) and, for Algorithm 1,
    // C, D (own minus neighbour); A and C multiply the R + S parts, B and D the R - S parts
    auto flux_rows = [&](const Mat& Z, bool cross, double scale, const char* fn) {
      const Mat F = mul(Z, B, Nfp, Np, Np);
      for (int outo = 0; outo < 2; ++outo) {
        const bool in_odd = cross ? !outo : outo;
        const auto& in = in_odd ? ao : ae;
        const int n = outo ? GO : GE, m = (int)in.size();
        Mat M((size_t)n * m);
        for (int i = 0; i < n; ++i)
          for (int c = 0; c < m; ++c) {
            const double v1 = F[(size_t)i * Np + in[c]], v2 = F[(size_t)(Nfp - 1 - i) * Np + in[c]];
            M[(size_t)i * m + c] = (i == Nfp - 1 - i) ? (outo ? 0 : v1) : 0.5 * (v1 + (outo ? -1 : 1) * v2);
          }
        double top = scale, bad = 0;
        for (double v : F) top = std::max(top, std::fabs(v));
        const auto& other = in_odd ? ae : ao;   // the parity that must not appear
        for (int i = 0; i < n; ++i)
          for (int c : other) {
            const double v1 = F[(size_t)i * Np + c], v2 = F[(size_t)(Nfp - 1 - i) * Np + c];
            if (!(i == Nfp - 1 - i && outo)) bad = std::max(bad, std::fabs(v1 + (outo ? -1 : 1) * v2));
          }
        if (bad > 1e-10 * top) { std::fprintf(stderr, "%s: mirror symmetry broken (%g of %g)\n", fn, bad, top); std::exit(1); }
        char sig[128];
        std::snprintf(sig, sizeof sig, "%s_%s(const T* b, T* g)", fn, outo ? "odd" : "even");
        open(sig);
        product(M, n, m, "b", "g", false, scale);
        close();
      }
      return F;
    };
    auto add = [&](const Mat& a, const Mat& b, double f) {
      Mat c(a);
      for (size_t i = 0; i < c.size(); ++i) c[i] += f * b[i];
      return c;
    };
    auto constant_rows = [&](const Mat& F, bool odd, const char* fn) {
      // a constant on the own side (b_{00} = 1): the jump's flux, mirror even for A and odd for D
      char sig[64];
      std::snprintf(sig, sizeof sig, "%s(T w, T* g)", fn);
      open(sig);
      for (int i = 0; i < (odd ? GO : GE); ++i) {
        const double v1 = F[(size_t)i * Np], v2 = F[(size_t)(Nfp - 1 - i) * Np];
        std::printf("    g[%d] = fma(%s, w, g[%d]);\n", i, lit(i == Nfp - 1 - i ? v1 : 0.5 * (v1 + (odd ? -1 : 1) * v2)).c_str(), i);
      }
      close();
    };
    double scale = 0;
    for (double v : o->QRV[0]) scale = std::max(scale, std::fabs(v));
    const Mat sum2 = add(o->QRV[0], o->QSV[0], 1), dif2 = add(o->QRV[0], o->QSV[0], -1);
    constant_rows(flux_rows(sum2, false, scale, "alg2_a"), false, "alg2_jump_a");
    flux_rows(dif2, true, scale, "alg2_b");
    const Mat ow_s = add(o->ZR[0][0], o->ZS[0][0], 1), ow_d = add(o->ZR[0][0], o->ZS[0][0], -1);
    const Mat nb_s = add(o->ZR[1][0], o->ZS[1][0], 1), nb_d = add(o->ZR[1][0], o->ZS[1][0], -1);
    constant_rows(flux_rows(add(ow_s, nb_s, 1), false, scale, "alg1_a"), false, "alg1_jump_a");
    flux_rows(add(ow_d, nb_d, 1), true, scale, "alg1_b");
    flux_rows(add(ow_s, nb_s, -1), false, scale, "alg1_c");
    constant_rows(flux_rows(add(ow_d, nb_d, -1), true, scale, "alg1_d"), true, "alg1_jump_d");

    // LIFT of one face in its rotated order, the same for every face
    for (int odd = 0; odd < 2; ++odd) {
      const int n = odd ? NO : NE, m = odd ? GO : GE;
      Mat M((size_t)n * m);
      for (int a = 0; a < n; ++a)
        for (int q = 0; q < m; ++q) {
          const int l = odd ? eo[a] : er[a];
          double v1 = 0, v2 = 0;
          for (int f = 0; f < 3; ++f) {
            v1 += o->LIFT[(size_t)P[f][l] * 3 * Nfp + f * Nfp + q] / 3;
            v2 += o->LIFT[(size_t)P[f][l] * 3 * Nfp + f * Nfp + Nfp - 1 - q] / 3;
          }
          M[(size_t)a * m + q] = (q == Nfp - 1 - q) ? v1 : v1 + (odd ? -1 : 1) * v2;
        }
      open(odd ? "lift_odd(const T* g, T* v)" : "lift_even(const T* g, T* v)");
      product(M, n, m, "g", "v", true);
      close();
    }

    // volume term in halves (ve, vo): p = D+ d, m = D- d with D+- = Dr +- Ds, F+- = F_r +- F_s,
    // vol = (W+ F+ + W- F-) / 2; component by component, so only d, vol and four scalars are live.
    // al = a_r + a_s, am = a_r - a_s, be = (g_rr + 2 g_rs + g_ss)/2, ga = (g_rr - g_ss)/2, de = (g_rr - 2 g_rs + g_ss)/2
    // REF: the node that d is taken from (0 or the centre), whose own entry is zero and left out, or -1
    const Mat Dp = add(o->Dr, o->Ds, 1), Dm = add(o->Dr, o->Ds, -1);
    Mat Wp = add(o->Wr, o->Ws, 1), Wm = add(o->Wr, o->Ws, -1);
    for (auto& v : Wp) v *= 0.5;
    for (auto& v : Wm) v *= 0.5;
    // volume: all components; volume0..3: the components' products split into four nearly equal shares
    // for four warps that work on the same elements, the last three also having a face's flux and LIFT
    std::vector<int> share(NE + NO, 0);
    {
      std::vector<double> load = {0.0, 1, 1, 1};
      const double face = 3.0 * GE + 3.0 * GO + NE * GE + NO * GO + NE + 2.0 * NO + 8;
      for (int w = 1; w < 4; ++w) load[w] = face;
      for (int q = 0; q < NE + NO; ++q) {
        int best = 0;
        for (int w = 1; w < 4; ++w)
          if (load[w] < load[best]) best = w;
        share[q] = best;
        load[best] += 2.0 * Np + 7;
      }
    }
    for (int part = -1; part < 4; ++part) {
      char sig[160];
      std::snprintf(sig, sizeof sig, "volume%s(const T* e, const T* o, T u0, T al, T am, T be, T ga, T de, T* ve, T* vo)",
                    part < 0 ? "" : std::to_string(part).c_str());
      open(sig, ", int REF");
      bool bege = false, bego = false;
      for (int odd = 0; odd < 2; ++odd) {
        const Mat Rp = comp(Dp, !odd, !odd, false), Rm = comp(Dm, !odd, odd, false);
        const Mat Cp = comp(Wp, !odd, !odd, true), Cm = comp(Wm, odd, !odd, true);
        const int n = odd ? NO : NE, mo = odd ? NE : NO;   // this parity's components, the other's
        for (int q = 0; q < n; ++q) {
          if (part >= 0 && share[odd * NE + q] != part) continue;
          std::printf("    {\n      T p, m;\n");
          auto row = [&](const Mat& R, int cols, const char* x, const char* y, bool skip0) {
            double top = 0;
            for (double v : R) top = std::max(top, std::fabs(v));
            bool begun = false;
            for (int c = 0; c < cols; ++c) {
              const double v = R[(size_t)q * cols + c];
              if (std::fabs(v) <= 1e-13 * top) continue;
              const int ref = skip0 && (er[c] == 0 || er[c] == centre) ? er[c] : -1;
              if (ref >= 0 && !begun)
                std::printf("      if constexpr (REF == %d) %s = T(0);\n      else %s = %s * %s[%d];\n", ref, y, y, lit(v).c_str(), x, c);
              else if (ref >= 0)
                std::printf("      if constexpr (REF != %d) %s = fma(%s, %s[%d], %s);\n", ref, y, lit(v).c_str(), x, c, y);
              else if (begun) std::printf("      %s = fma(%s, %s[%d], %s);\n", y, lit(v).c_str(), x, c, y);
              else std::printf("      %s = %s * %s[%d];\n", y, lit(v).c_str(), x, c);
              begun = true;
            }
            if (!begun) std::printf("      %s = T(0);\n", y);
          };
          row(Rp, n, odd ? "o" : "e", "p", !odd);
          row(Rm, mo, odd ? "e" : "o", "m", odd);
          if (odd) std::printf("      const T u = T(0.5) * o[%d];\n", q);
          else if (mir[er[q]] == er[q]) std::printf("      const T u = e[%d] + u0;\n", q);
          else std::printf("      const T u = fma(T(0.5), e[%d], u0);\n", q);
          std::printf("      const T fp = al * u - (be * p + ga * m), fm = am * u - (ga * p + de * m);\n");
          auto col = [&](const Mat& C, int rows, const char* f, const char* y, bool& begun) {
            double top = 0;
            for (double v : C) top = std::max(top, std::fabs(v));
            for (int i = 0; i < rows; ++i) {
              const double v = C[(size_t)i * n + q];
              if (!begun) std::printf("      %s[%d] = %s * %s;\n", y, i, lit(v).c_str(), f);
              else if (std::fabs(v) > 1e-13 * top) std::printf("      %s[%d] = fma(%s, %s, %s[%d]);\n", y, i, lit(v).c_str(), f, y, i);
            }
            begun = true;
          };
          col(Cp, n, "fp", odd ? "vo" : "ve", odd ? bego : bege);
          col(Cm, mo, "fm", odd ? "ve" : "vo", odd ? bege : bego);
          std::printf("    }\n");
        }
      }
      for (int i = 0; i < NE && !bege; ++i) std::printf("    ve[%d] = T(0);\n", i);
      for (int i = 0; i < NO && !bego; ++i) std::printf("    vo[%d] = T(0);\n", i);
      close();
    }
    std::printf("};\n");
  }
};

}  // namespace

int main(int argc, char** argv) {
  const int N = argc > 1 ? std::atoi(argv[1]) : 0;
  const char* msg = "order out of range";
  const RefOps* o = get_refops(N, &msg);
  if (!o) { std::fprintf(stderr, "%s\n", msg); return 1; }
  Gen g;
  g.N = N;
  g.o = o;
  g.run();
  return 0;
}
