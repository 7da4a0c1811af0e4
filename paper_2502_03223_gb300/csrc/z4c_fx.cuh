// The pointwise Z4c right-hand side of one cell in block fixed point
// (softfp.cuh): the algebra of z4c.cuh (Lam & Shibata, arXiv:2502.03223,
// Eq. bssn, Eq. K, Eq. moving_puncture) with its contractions of metric,
// Christoffel symbols, derivatives and At_ij as integer sums, and the few
// operations on scalars and the assembly of the 25 outputs in FP64.
//
// In FP64 the pass executed 1350 FP64 instructions per warp at 16 SM cycles
// each, with the integer units idle.  Here the products of the Christoffel
// symbols, of At_ij and of the shift's derivatives (about 530, three mad.wide
// each) run on the integer units; the contractions whose operands would only
// be converted for one use (the second derivatives) stay in FP64, so that both
// pipes are busy for about the same time.
//
// Identities used on the way (exact; gt^ij the inverse of gt_ij):
//  * Gt_{i,jk} + Gt_{j,ik} = d_k gt_ij, so Gt_d^k Gt_(ij)k = Gt_d^k d_k gt_ij / 2;
//  * terms proportional to gt_ij drop out of the trace-free part: X_ij leaves
//    out P gt_ij / W^2, gt_ij (tr DDW / W - 2 dW^2 / W^2) and gt_ij d alpha . dW / W;
//    the traces take them in closed form (3 times the factor);
//  * gt^ij Gt^k_ij = Gt_d^k, so tr DDW = gt^ij d_i d_j W - Gt_d^k d_k W (and for alpha);
//  * alpha DDW_ij / W - D~_i D~_j alpha takes one product with Gt^k_ij, of the
//    vector (alpha / W) d_k W - d_k alpha;
//  * tr S = rho h (w^2 - 1) + 3 P, rho h = rho (1 + eps) + P.
#pragma once

#include "softfp.cuh"
#include "z4c.cuh"

namespace sacra {

// symmetric-pair index as a compile-time function
SF_HD constexpr int sq(int i, int j) {
  return (i == j) ? (i == 0 ? 0 : (i == 1 ? 3 : 5)) : (i + j == 1 ? 1 : (i + j == 2 ? 2 : 4));
}
SF_HD constexpr bool diag6(int a) { return a == 0 || a == 3 || a == 5; }

// gt^ij s_ij style contraction of a group gi2 (off-diagonal entries doubled)
SF_HD sf::i64 tr6(const sf::Bf (&gi2)[6], const sf::Bf *s) {
  sf::Acc a;
#pragma unroll
  for (int q = 0; q < 6; ++q) sf::mac(a, gi2[q], s[q]);
  return sf::fin(a);
}

struct Z4cPar {               // the star's parameters as the cell takes them
  double kappa, eta_B;
  int bssn;
};

// The algebra runs in two passes, because its straight-line code (10 000
// instructions, 160 KB) does not stay in the SM's instruction cache: as one
// kernel it waited for instructions most of the time (0.52 ms per launch on a
// migration star of 3 x 256^2, where the FP64 form took 0.57 ms).  Pass A (the
// Christoffel symbols and the quadratic Ricci terms) is bound by the integer
// and multiply-add pipes, pass B (second derivatives, matter, assembly) by the
// FP64 pipe: 0.15 and 0.19 ms there; 13.3 -> 7.2 ms per step of the migration
// star 5 x 512^2 (FP64).
//
// U(f): state field f; D1(a, k), D2(a, q): derivative scratch; AK(f):
// advection and dissipation; PR(f): primitives; fz = exp(-r^2 / r_Z4^2).
// out(f, value) receives the 25 right-hand sides, rs the Ricci scalar.
// Both passes return false where the form does not apply (a non-finite input,
// |h_ij| >= 2^20, det gt <= 0); pass B has then written nothing, and pass A
// marks the cell in its scratch plane zOK.

// What pass A leaves for pass B, in planes of the right-hand side that pass B
// overwrites: gt^ij, X_ij, gt^ij R_ij so far, At_ij At^ij, Gt_d^i, the source
// of Gt^i so far, and 1.0 (or 0.0: the cell goes to the FP64 algebra).
enum : int { zGI = 0, zX = 6, zTR = 12, zAA = 13, zGD = 14, zS = 17, zOK = 20, zN = 21 };

template <class FU, class F1, class FO>
SF_HD bool z4c_fx_a(FU U, F1 D1, FO put) {
  using namespace sf;
  int top = 0;
  // ---- the metric and its inverse
  Grp<6> g, gi;
  double hd[6], gd[6];                              // h_ij, gt^ij
  {
#pragma unroll
    for (int a = 0; a < 6; ++a) hd[a] = U(fHXX + a);
    i64 det, R[6];
    int edet, eR;
    if (!metric_group(hd, g) || !metric_inverse(g, gi, R, eR, det, edet)) { put(zOK, 0.0); return false; }
#pragma unroll
    for (int a = 0; a < 6; ++a) gd[a] = to_double(R[a], eR);
  }
#pragma unroll
  for (int a = 0; a < 6; ++a) put(zGI + a, gd[a]);
  const double W = U(fW), al = U(fAL);
  const double iW = srcp(W);

  // ---- At_i^k, At^ij, At_ij At^ij, At_i^l At_lj
  double AmA[6];
  Grp<6> Au;
  {
    double Ad[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) Ad[q] = U(fAXX + q);
    Grp<6> A;
    load(Ad, A, top);
    Grp<9> Am;                                      // At_i^k at [3 i + k]
    i64 R[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        Acc q;
#pragma unroll
        for (int l = 0; l < 3; ++l) mac(q, A.v[sq(i, l)], gi.v[sq(l, k)]);
        R[3 * i + k] = fin(q);
      }
    norm(R, A.e + gi.e + kUnit, Am);
    Acc d, o;
    mac(d, Am.v[0], Am.v[0]); mac(d, Am.v[4], Am.v[4]); mac(d, Am.v[8], Am.v[8]);
    mac(o, Am.v[1], Am.v[3]); mac(o, Am.v[2], Am.v[6]); mac(o, Am.v[5], Am.v[7]);
    put(zAA, to_double(fin(d) + 2 * fin(o), 2 * Am.e + kUnit));
    i64 Q[6];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        Acc a, b;
#pragma unroll
        for (int l = 0; l < 3; ++l) {
          mac(a, gi.v[sq(i, l)], Am.v[3 * l + j]);
          mac(b, Am.v[3 * i + l], A.v[sq(l, j)]);
        }
        Q[sq(i, j)] = fin(a);
        AmA[sq(i, j)] = to_double(fin(b), Am.e + A.e + kUnit);
      }
    norm(Q, gi.e + Am.e + kUnit, Au);
  }

  // ---- Christoffel symbols: 2 Gt_{k,ij} (Gl), Gt^k_ij, Gt_d^i
  double dWd[3], dald[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) { dWd[k] = D1(0, k); dald[k] = D1(12, k); }
  const double aW = al * iW;
  double X[6];
  i64 S[6];
  int eS;
  {
    Grp<18> dh;                                     // d_k gt_a at [3 a + k]
    {
      double x[18];
#pragma unroll
      for (int a = 0; a < 6; ++a)
#pragma unroll
        for (int k = 0; k < 3; ++k) x[3 * a + k] = D1(1 + a, k);
      load(x, dh, top);
    }
    Bf Gl[3][6];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
          // for k = i two of the three terms cancel and d_j gt_kk is left, for k = j d_i gt_kk
          if (k == i) Gl[k][sq(i, j)] = dh.v[3 * sq(k, i) + j];
          else if (k == j) Gl[k][sq(i, j)] = dh.v[3 * sq(k, j) + i];
          else Gl[k][sq(i, j)] = dh.v[3 * sq(k, j) + i] + dh.v[3 * sq(k, i) + j] - dh.v[3 * sq(i, j) + k];
        }
    const int eGl = dh.e - 1;
    Grp<18> G2;                                     // Gt^k_a at [6 k + a]
    {
      i64 R[18];
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int a = 0; a < 6; ++a) {
          Acc q;
#pragma unroll
          for (int l = 0; l < 3; ++l) mac(q, gi.v[sq(k, l)], Gl[l][a]);
          R[6 * k + a] = fin(q);
        }
      norm(R, gi.e + eGl + kUnit, G2);
    }
    // Gt_d^i, and Gt^i_jk At^jk with At^ij (d_j alpha + 3 alpha d_j W / W) of the Gt^i source
    Grp<3> Gd;
    {
      double y[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) y[j] = dald[j] + 3.0 * aW * dWd[j];
      Grp<3> yg;
      load(y, yg, top);
      i64 R[3];
      const int e = gi.e + G2.e + kUnit;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        Acc d, o, ud, uo, ay;
#pragma unroll
        for (int a = 0; a < 6; ++a) {
          mac(diag6(a) ? d : o, gi.v[a], G2.v[6 * i + a]);
          mac(diag6(a) ? ud : uo, Au.v[a], G2.v[6 * i + a]);
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) mac(ay, Au.v[sq(i, j)], yg.v[j]);
        R[i] = fin(d) + 2 * fin(o);
        put(zGD + i, to_double(R[i], e));
        put(zS + i, 2.0 * (al * to_double(fin(ud) + 2 * fin(uo), Au.e + G2.e + kUnit)
                           - to_double(fin(ay), Au.e + yg.e + kUnit)));
      }
      norm(R, e, Gd);
    }
    // (alpha / W) d_k W - d_k alpha, times Gt^k_ij
    {
      double c[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) c[k] = dald[k] - aW * dWd[k];
      Grp<3> cg;
      load(c, cg, top);
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        Acc a;
#pragma unroll
        for (int k = 0; k < 3; ++k) mac(a, G2.v[6 * k + q], cg.v[k]);
        X[q] = to_double(fin(a), G2.e + cg.e + kUnit);
      }
    }
    // the conformal Ricci tensor but its second derivatives.  The quadratic
    // terms by the first index a of M[a][k][l] = gt^lm Gt_{a,km}:
    // Q_ia = Gt^k_li M[a][k][l] enters ia twice, Gt^a_im M[a][j][m] enters ij
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      i64 R[9];
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int l = 0; l < 3; ++l) {
          Acc q;
#pragma unroll
          for (int m = 0; m < 3; ++m) mac(q, gi.v[sq(l, m)], Gl[a][sq(k, m)]);
          R[3 * k + l] = fin(q);
        }
      Grp<9> M;
      norm(R, gi.e + eGl + kUnit, M);
      i64 T[6], Q[3];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        Acc q;
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
          for (int l = 0; l < 3; ++l) mac(q, G2.v[6 * k + sq(l, i)], M.v[3 * k + l]);
        Q[i] = fin(q);
      }
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
          Acc q;
#pragma unroll
          for (int m = 0; m < 3; ++m) mac(q, G2.v[6 * a + sq(i, m)], M.v[3 * j + m]);
          i64 t = fin(q);
          if (j == a) t += Q[i];
          if (i == a) t += Q[j];
          T[sq(i, j)] = t;
        }
      const int eT = G2.e + M.e + kUnit;
      if (a == 0) {
#pragma unroll
        for (int q = 0; q < 6; ++q) S[q] = T[q];
        eS = eT;
      } else {
        align_add(S, eS, T, eT);
      }
    }
    i64 T[6];
    // Gt_d^k d_k gt_ij / 2
#pragma unroll
    for (int a = 0; a < 6; ++a) {
      Acc q;
#pragma unroll
      for (int k = 0; k < 3; ++k) mac(q, Gd.v[k], dh.v[3 * a + k]);
      T[a] = fin(q);
    }
    align_add(S, eS, T, Gd.e + dh.e + kUnit - 1);
  }
  // X_ij so far: alpha times these Ricci terms, the product with Gt^k_ij, and
  // -2 alpha At_i^l At_lj / W^2 (pass B multiplies by W^2); the Ricci trace
  {
    Grp<6> R;
    norm(S, eS, R);
    Acc d, o;
#pragma unroll
    for (int q = 0; q < 6; ++q) mac(diag6(q) ? d : o, gi.v[q], R.v[q]);
    put(zTR, to_double(fin(d) + 2 * fin(o), gi.e + R.e + kUnit));
    const double c = -2.0 * aW * iW;
#pragma unroll
    for (int q = 0; q < 6; ++q) put(zX + q, X[q] + al * to_double(S[q], eS) + c * AmA[q]);
  }
  const bool ok = top < 2047;
  put(zOK, ok ? 1.0 : 0.0);
  return ok;
}

template <class FU, class F1, class F2, class FA, class FP, class FS, class FO>
SF_HD bool z4c_fx_b(const Z4cPar &p, FU U, F1 D1, F2 D2, FA AK, FP PR, FS scr, double fz, FO out, double *rs) {
  using namespace sf;
  if (scr(zOK) != 1.0) return false;
  int top = 0;
  double gd[6], hd[6];                              // gt^ij, h_ij
#pragma unroll
  for (int a = 0; a < 6; ++a) gd[a] = scr(zGI + a);
  // gt^ij t_ij of a symmetric tensor
  const double g1 = 2.0 * gd[1], g2 = 2.0 * gd[2], g4 = 2.0 * gd[4];
  auto trd = [&](const double (&t)[6]) {
    return gd[0] * t[0] + gd[3] * t[3] + gd[5] * t[5] + g1 * t[1] + g2 * t[2] + g4 * t[4];
  };
  Grp<6> g;
  {
#pragma unroll
    for (int a = 0; a < 6; ++a) hd[a] = U(fHXX + a);
    metric_group(hd, g);                            // in range: pass A
  }
  const double W = U(fW), al = U(fAL), iW = srcp(W), aW = al * iW, W2 = W * W;
  double Rc[6];                                     // gt_k(i d_j) Gt^k - gt^lm d_l d_m gt_ij / 2
  {
    // gt_k(i d_j) Gt^k
    double x[9];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int j = 0; j < 3; ++j) x[3 * k + j] = D1(8 + k, j);
    Grp<9> dG;
    load(x, dG, top);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        Acc q;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          mac(q, g.v[sq(k, i)], dG.v[3 * k + j]);
          if (i != j) mac(q, g.v[sq(k, j)], dG.v[3 * k + i]);
        }
        Rc[sq(i, j)] = to_double(i == j ? 2 * fin(q) : fin(q), g.e + dG.e + kUnit - 1);
      }
  }

  // ---- X_ij = alpha R_ij - D_i D_j alpha without terms in gt_ij, and the traces
  double dWd[3], dald[3], Gdd[3], s[3], X[6];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    dWd[k] = D1(0, k);
    dald[k] = D1(12, k);
    Gdd[k] = scr(zGD + k);
    s[k] = scr(zS + k);
  }
  const double AA = scr(zAA);
  double Rs, D2a, trX;
  {
    double w[6], a[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      double dd[6];
#pragma unroll
      for (int r = 0; r < 6; ++r) dd[r] = D2(1 + q, r);
      Rc[q] -= 0.5 * trd(dd);
      w[q] = D2(0, q);
      a[q] = D2(7, q);
    }
    double v[3], dW2 = 0.0, daW = 0.0, gW = 0.0, ga = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      v[i] = gd[sq(i, 0)] * dWd[0] + gd[sq(i, 1)] * dWd[1] + gd[sq(i, 2)] * dWd[2];
      dW2 += v[i] * dWd[i];
      daW += v[i] * dald[i];
      gW += Gdd[i] * dWd[i];
      ga += Gdd[i] * dald[i];
    }
    const double trDDW = trd(w) - gW, trD = trd(a) - ga, trRc = scr(zTR) + trd(Rc);
    const double iWd = iW * daW;
    // gt^ij R_ij: R_ij = Rc_ij + DDW_ij / W + gt_ij (tr DDW / W - 2 dW^2 / W^2)
    Rs = W2 * (trRc + iW * (4.0 * trDDW - 6.0 * iW * dW2));
    D2a = W2 * (trD - iWd);
    trX = al * (trRc + iW * trDDW) - (trD + 2.0 * iWd);
    double aw[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) aw[i] = iW * dald[i];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        const int q = sq(i, j);
        const double mix = i == j ? 2.0 * aw[i] * dWd[i] : aw[i] * dWd[j] + aw[j] * dWd[i];
        X[q] = scr(zX + q) + al * Rc[q] + (aW * w[q] - a[q]) - mix;
      }
  }

  // ---- matter
  constexpr double PI = 3.14159265358979323846;
  double E, SE, Si[3] = {0.0, 0.0, 0.0};            // E, tr S + E, S_i
  {
    const double P = PR(pP);
    const double ud[3] = {PR(pUX), PR(pUY), PR(pUZ)};
    const double rh = PR(pRHO) * (1.0 + PR(pEPS)) + P;
    E = rh - P;
    SE = rh + 2.0 * P;
    if (ud[0] != 0.0 || ud[1] != 0.0 || ud[2] != 0.0) {
      double u2 = 0.0;
#pragma unroll
      for (int i = 0; i < 3; ++i)
        u2 += ud[i] * (gd[sq(i, 0)] * ud[0] + gd[sq(i, 1)] * ud[1] + gd[sq(i, 2)] * ud[2]);
      const double z2 = W2 * u2, w2 = 1.0 + z2, w = ssqrt(w2);
      E = rh * w2 - P;
      SE = rh * (z2 + w2) + 2.0 * P;
      const double c = -8.0 * PI * al * rh;
#pragma unroll
      for (int i = 0; i < 3; ++i) Si[i] = rh * w * ud[i];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) X[sq(i, j)] += c * ud[i] * ud[j];
      trX += c * u2;
    }
    top = imax(top, field(E + SE) >> 20);
  }

  // ---- the shift's derivatives
  double dbd[9];                                    // d_k beta^i at [3 i + k]
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) dbd[3 * i + k] = D1(13 + i, k);
  Grp<9> db;
  load(dbd, db, top);
  double Ad[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) Ad[q] = U(fAXX + q);
  Grp<6> A;
  load(Ad, A, top);
  if (top >= 2047) return false;
  const double Kh = U(fKH), Th = U(fTH);
  const double K = Kh + 2.0 * Th;
  const double kap = p.kappa * fz;
  const double divb = dbd[0] + dbd[4] + dbd[8];
  {
    double z[3], gr[3] = {0.0, 0.0, 0.0}, lap[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      double dd[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) dd[q] = D2(8 + i, q);
      lap[i] = trd(dd);
#pragma unroll
      for (int j = 0; j < 3; ++j) gr[j] += dd[sq(i, j)];
    }
    // gt^ij (d_j d_k beta^k / 3 - (2/3) alpha (2 d_j Kh + d_j Theta) - 16 pi alpha S_j)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      z[j] = (1.0 / 3.0) * (gr[j] - 2.0 * al * (2.0 * D1(7, j) + D1(11, j))) - 16.0 * PI * al * Si[j];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      s[i] += lap[i] + (gd[sq(i, 0)] * z[0] + gd[sq(i, 1)] * z[1] + gd[sq(i, 2)] * z[2]);
      s[i] -= Gdd[0] * dbd[3 * i] + Gdd[1] * dbd[3 * i + 1] + Gdd[2] * dbd[3 * i + 2];
      s[i] += (2.0 / 3.0) * Gdd[i] * divb - 2.0 * al * kap * (U(fGX + i) - Gdd[i]);
      const double Bi = U(fBBX + i);
      out(fGX + i, s[i] + AK(fGX + i));
      out(fBBX + i, s[i] - p.eta_B * Bi + AK(fBBX + i));
      out(fBX + i, 0.75 * Bi + AK(fBX + i));
    }
  }
  out(fW, W * (al * K - divb) * (1.0 / 3.0) + AK(fW));
  out(fKH, -D2a + al * (AA + K * K * (1.0 / 3.0)) + 4.0 * PI * al * SE + al * kap * Th + AK(fKH));
  out(fTH, (p.bssn ? 0.0
                   : fz * (0.5 * al * (Rs - AA + (2.0 / 3.0) * K * K) - 8.0 * PI * al * E) - 2.0 * al * kap * Th) + AK(fTH));
  out(fAL, -2.0 * al * Kh + AK(fAL));
  const double t3 = trX * (1.0 / 3.0), cA = al * K - (2.0 / 3.0) * divb, cg = -(2.0 / 3.0) * divb;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      const int q = sq(i, j);
      Acc a2, a3;                                   // gt_ik d_j beta^k + gt_jk d_i beta^k, At_kj d_i beta^k + At_ki d_j beta^k
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        mac(a2, g.v[sq(i, k)], db.v[3 * k + j]);
        mac(a3, A.v[sq(k, j)], db.v[3 * k + i]);
        if (i != j) {
          mac(a2, g.v[sq(j, k)], db.v[3 * k + i]);
          mac(a3, A.v[sq(k, i)], db.v[3 * k + j]);
        }
      }
      const int two = i == j ? 1 : 0;
      const double gq = diag6(q) ? 1.0 + hd[q] : hd[q];
      const double gb = to_double(fin(a2), g.e + db.e + kUnit + two);
      const double Ab = to_double(fin(a3), A.e + db.e + kUnit + two);
      out(fHXX + q, -2.0 * al * Ad[q] + cg * gq + gb + AK(fHXX + q));
      out(fAXX + q, W2 * (X[q] - gq * t3) + cA * Ad[q] + Ab + AK(fAXX + q));
    }
  if (rs) *rs = Rs;
  return true;
}

}  // namespace sacra
