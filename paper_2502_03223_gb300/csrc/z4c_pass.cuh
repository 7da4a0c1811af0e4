// The pointwise Z4c right-hand side of one cell in FP64, in two passes: the
// algebra of z4c.cuh (Lam & Shibata, arXiv:2502.03223, Eq. bssn, Eq. K,
// Eq. moving_puncture) with fewer operations, by identities that hold exactly
// (gt^ij the inverse of gt_ij):
//  * Gt_{i,jk} + Gt_{j,ik} = d_k gt_ij, so Gt_d^k Gt_(ij)k = Gt_d^k d_k gt_ij / 2;
//  * terms proportional to gt_ij drop out of the trace-free part: X_ij leaves
//    out P gt_ij / W^2, gt_ij (tr DDW / W - 2 dW^2 / W^2) and gt_ij d alpha . dW / W;
//    the traces take them in closed form (3 times the factor);
//  * gt^ij Gt^k_ij = Gt_d^k, so tr DDW = gt^ij d_i d_j W - Gt_d^k d_k W (and for alpha);
//  * alpha DDW_ij / W - D~_i D~_j alpha takes one product with Gt^k_ij, of the
//    vector (alpha / W) d_k W - d_k alpha;
//  * tr S = rho h (w^2 - 1) + 3 P, rho h = rho (1 + eps) + P.
//
// Every value keeps its own exponent: h_ij - small off-diagonal entries, a
// conformal metric stretched in one direction - may differ by many orders
// within a cell, and a contraction of small entries must keep its digits.  (On
// one integer grid per group of values the cofactors of a stretched metric
// lost accuracy as the cube of its largest entry.)
//
// Bound by the FP64 pipe.  Two passes, because the straight-line code of one
// does not stay in the SM's instruction cache beside its loads and its live
// values do not fit the registers; pass A's twenty results wait in the
// right-hand side's planes.  9.8 ms per step of the migration star 5 x 512^2,
// 13.3 ms with the algebra of z4c.cuh as written in one pass.
#pragma once

#include "fields.h"
#include "softfp.cuh"

namespace sacra {

// symmetric-pair index as a compile-time function
SF_HD constexpr int sq(int i, int j) {
  return (i == j) ? (i == 0 ? 0 : (i == 1 ? 3 : 5)) : (i + j == 1 ? 1 : (i + j == 2 ? 2 : 4));
}

// gt^ij t_ij of a symmetric tensor
template <class T>
SF_HD T trace6(const T (&gi)[6], const T (&t)[6]) {
  return gi[0] * t[0] + gi[3] * t[3] + gi[5] * t[5] + T(2) * (gi[1] * t[1] + gi[2] * t[2] + gi[4] * t[4]);
}

SF_HD double z4c_rcp(double v) { return sf::srcp(v); }
SF_HD double z4c_sqrt(double v) { return sf::ssqrt(v); }

template <class T>
struct Z4cPar {               // the star's parameters as the cell takes them
  T kappa, eta_B;
  int bssn;
};

// What pass A leaves for pass B, in planes of the right-hand side that pass B
// overwrites: gt^ij, X_ij so far, gt^ij R_ij so far, At_ij At^ij, Gt_d^i, the
// source of Gt^i so far.
enum : int { zGI = 0, zX = 6, zTR = 12, zAA = 13, zGD = 14, zS = 17, zN = 20 };

// U(f): state field f; D1(a, k), D2(a, q): derivative scratch; AK(f):
// advection and dissipation; PR(f): primitives; fz = exp(-r^2 / r_Z4^2).
// put(plane, value) writes pass A's results, scr(plane) reads them back;
// out(f, value) receives the 25 right-hand sides, rs the Ricci scalar.
template <class T, class FU, class F1, class FO>
SF_HD void z4c_pass_a(FU U, F1 D1, FO put) {
  // ---- gt^ij
  T gi[6];
  {
    T g[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) g[a] = U(fHXX + a);
    g[0] += T(1); g[3] += T(1); g[5] += T(1);
    const T cxx = g[3] * g[5] - g[4] * g[4];
    const T cxy = g[2] * g[4] - g[1] * g[5];
    const T cxz = g[1] * g[4] - g[2] * g[3];
    const T id = z4c_rcp(g[0] * cxx + g[1] * cxy + g[2] * cxz);
    gi[0] = cxx * id; gi[1] = cxy * id; gi[2] = cxz * id;
    gi[3] = (g[0] * g[5] - g[2] * g[2]) * id;
    gi[4] = (g[1] * g[2] - g[0] * g[4]) * id;
    gi[5] = (g[0] * g[3] - g[1] * g[1]) * id;
  }
#pragma unroll
  for (int a = 0; a < 6; ++a) put(zGI + a, gi[a]);
  const T al = U(fAL), iW = z4c_rcp(U(fW)), aW = al * iW;

  // ---- At_i^k, At^ij, At_ij At^ij; X_ij starts with -2 alpha At_i^l At_lj / W^2
  // (pass B multiplies by W^2)
  T X[6], Au[6];
  {
    T A[6], Am[3][3];
#pragma unroll
    for (int q = 0; q < 6; ++q) A[q] = U(fAXX + q);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int k = 0; k < 3; ++k)
        Am[i][k] = A[sq(i, 0)] * gi[sq(0, k)] + A[sq(i, 1)] * gi[sq(1, k)] + A[sq(i, 2)] * gi[sq(2, k)];
    put(zAA, Am[0][0] * Am[0][0] + Am[1][1] * Am[1][1] + Am[2][2] * Am[2][2]
                 + T(2) * (Am[0][1] * Am[1][0] + Am[0][2] * Am[2][0] + Am[1][2] * Am[2][1]));
    const T c = T(-2) * aW * iW;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        Au[sq(i, j)] = gi[sq(i, 0)] * Am[0][j] + gi[sq(i, 1)] * Am[1][j] + gi[sq(i, 2)] * Am[2][j];
        X[sq(i, j)] = c * (Am[i][0] * A[sq(0, j)] + Am[i][1] * A[sq(1, j)] + Am[i][2] * A[sq(2, j)]);
      }
  }

  // ---- Christoffel symbols: 2 Gt_{k,ij} (Gl), Gt^k_ij, Gt_d^i
  T dW[3], dal[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) { dW[k] = D1(0, k); dal[k] = D1(12, k); }
  T dh[6][3], Gl[3][6], G2[3][6], Gd[3], hg[6];     // d_k gt_a, ..., gt^ij / 2
#pragma unroll
  for (int a = 0; a < 6; ++a) {
    hg[a] = T(0.5) * gi[a];
#pragma unroll
    for (int k = 0; k < 3; ++k) dh[a][k] = D1(1 + a, k);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        // for k = i two of the three terms cancel and d_j gt_kk is left, for k = j d_i gt_kk
        if (k == i) Gl[k][sq(i, j)] = dh[sq(k, i)][j];
        else if (k == j) Gl[k][sq(i, j)] = dh[sq(k, j)][i];
        else Gl[k][sq(i, j)] = dh[sq(k, j)][i] + dh[sq(k, i)][j] - dh[sq(i, j)][k];
      }
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int a = 0; a < 6; ++a)
      G2[k][a] = hg[sq(k, 0)] * Gl[0][a] + hg[sq(k, 1)] * Gl[1][a] + hg[sq(k, 2)] * Gl[2][a];
  // Gt_d^i, and Gt^i_jk At^jk with At^ij (d_j alpha + 3 alpha d_j W / W) of the Gt^i source
  {
    T y[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) y[j] = dal[j] + T(3) * aW * dW[j];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      Gd[i] = trace6(gi, G2[i]);
      put(zGD + i, Gd[i]);
      put(zS + i, T(2) * (al * trace6(Au, G2[i]) - (Au[sq(i, 0)] * y[0] + Au[sq(i, 1)] * y[1] + Au[sq(i, 2)] * y[2])));
    }
  }
  // the conformal Ricci tensor but its second derivatives: Gt_d^k d_k gt_ij / 2 and the
  // quadratic terms, by the first index a of M[a][k][l] = gt^lm Gt_{a,km}:
  // Q_ia = Gt^k_li M[a][k][l] enters ia twice, Gt^a_im M[a][j][m] enters ij
  T S[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) S[q] = T(0.5) * (Gd[0] * dh[q][0] + Gd[1] * dh[q][1] + Gd[2] * dh[q][2]);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    T M[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int l = 0; l < 3; ++l)
        M[k][l] = hg[sq(l, 0)] * Gl[a][sq(k, 0)] + hg[sq(l, 1)] * Gl[a][sq(k, 1)] + hg[sq(l, 2)] * Gl[a][sq(k, 2)];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      T q = T(0);
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int l = 0; l < 3; ++l) q += G2[k][sq(l, i)] * M[k][l];
      S[sq(i, a)] += i == a ? T(2) * q : q;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j)
        S[sq(i, j)] += G2[a][sq(i, 0)] * M[j][0] + G2[a][sq(i, 1)] * M[j][1] + G2[a][sq(i, 2)] * M[j][2];
  }
  // X_ij so far: also alpha times these Ricci terms and (d_k alpha - (alpha / W) d_k W) Gt^k_ij
  put(zTR, trace6(gi, S));
  T c[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) c[k] = dal[k] - aW * dW[k];
#pragma unroll
  for (int q = 0; q < 6; ++q) put(zX + q, X[q] + al * S[q] + (c[0] * G2[0][q] + c[1] * G2[1][q] + c[2] * G2[2][q]));
}

template <class T, class FU, class F1, class F2, class FA, class FP, class FS, class FO, class FR>
SF_HD void z4c_pass_b(const Z4cPar<T> &p, FU U, F1 D1, F2 D2, FA AK, FP PR, FS scr, T fz, FO out, FR rs) {
  T gi[6], g[6];                                    // gt^ij, gt_ij
#pragma unroll
  for (int a = 0; a < 6; ++a) { gi[a] = scr(zGI + a); g[a] = U(fHXX + a); }
  g[0] += T(1); g[3] += T(1); g[5] += T(1);
  const T W = U(fW), al = U(fAL), iW = z4c_rcp(W), aW = al * iW, W2 = W * W;
  T Rc[6];                                          // gt_k(i d_j) Gt^k - gt^lm d_l d_m gt_ij / 2
  {
    T dG[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int j = 0; j < 3; ++j) dG[k][j] = D1(8 + k, j);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        T q = T(0);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          q += g[sq(k, i)] * dG[k][j];
          if (i != j) q += g[sq(k, j)] * dG[k][i];
        }
        Rc[sq(i, j)] = i == j ? q : T(0.5) * q;
      }
  }

  // ---- X_ij = alpha R_ij - D_i D_j alpha without terms in gt_ij, and the traces
  T dW[3], dal[3], Gd[3], s[3], X[6];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    dW[k] = D1(0, k);
    dal[k] = D1(12, k);
    Gd[k] = scr(zGD + k);
    s[k] = scr(zS + k);
  }
  const T AA = scr(zAA);
  T Rs, D2a, trX;
  {
    T w[6], a[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      T dd[6];
#pragma unroll
      for (int r = 0; r < 6; ++r) dd[r] = D2(1 + q, r);
      Rc[q] -= T(0.5) * trace6(gi, dd);
      w[q] = D2(0, q);
      a[q] = D2(7, q);
    }
    T dW2 = T(0), daW = T(0), gW = T(0), ga = T(0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const T v = gi[sq(i, 0)] * dW[0] + gi[sq(i, 1)] * dW[1] + gi[sq(i, 2)] * dW[2];
      dW2 += v * dW[i];
      daW += v * dal[i];
      gW += Gd[i] * dW[i];
      ga += Gd[i] * dal[i];
    }
    const T trDDW = trace6(gi, w) - gW, trD = trace6(gi, a) - ga, trRc = scr(zTR) + trace6(gi, Rc);
    const T iWd = iW * daW;
    // gt^ij R_ij: R_ij = Rc_ij + DDW_ij / W + gt_ij (tr DDW / W - 2 dW^2 / W^2)
    Rs = W2 * (trRc + iW * (T(4) * trDDW - T(6) * iW * dW2));
    D2a = W2 * (trD - iWd);
    trX = al * (trRc + iW * trDDW) - (trD + T(2) * iWd);
    T aw[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) aw[i] = iW * dal[i];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        const int q = sq(i, j);
        const T mix = i == j ? T(2) * aw[i] * dW[i] : aw[i] * dW[j] + aw[j] * dW[i];
        X[q] = scr(zX + q) + al * Rc[q] + (aW * w[q] - a[q]) - mix;
      }
  }

  // ---- matter
  const T PI = T(3.14159265358979323846L);
  T E, SE, Si[3];                                   // E, tr S + E, S_i
  {
    const T P = PR(pP);
    const T ud[3] = {PR(pUX), PR(pUY), PR(pUZ)};
    const T rh = PR(pRHO) * (T(1) + PR(pEPS)) + P;
    const T none = T(0) * rh;                       // NaN where rho, eps or P is not finite
    Si[0] = Si[1] = Si[2] = none;
    trX += none;
    E = rh - P;
    SE = rh + T(2) * P;
    if (ud[0] != T(0) || ud[1] != T(0) || ud[2] != T(0)) {
      T u2 = T(0);
#pragma unroll
      for (int i = 0; i < 3; ++i)
        u2 += ud[i] * (gi[sq(i, 0)] * ud[0] + gi[sq(i, 1)] * ud[1] + gi[sq(i, 2)] * ud[2]);
      const T z2 = W2 * u2, w2 = T(1) + z2, w = z4c_sqrt(w2);
      E = rh * w2 - P;
      SE = rh * (z2 + w2) + T(2) * P;
      const T c = T(-8) * PI * al * rh;
#pragma unroll
      for (int i = 0; i < 3; ++i) Si[i] = rh * w * ud[i];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) X[sq(i, j)] += c * ud[i] * ud[j];
      trX += c * u2;
    }
  }

  // ---- the shift's derivatives
  T db[3][3];                                       // d_k beta^i
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) db[i][k] = D1(13 + i, k);
  T A[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) A[q] = U(fAXX + q);
  const T Kh = U(fKH), Th = U(fTH);
  const T K = Kh + T(2) * Th;
  const T kap = p.kappa * fz;
  const T divb = db[0][0] + db[1][1] + db[2][2];
  {
    T z[3], gr[3] = {T(0), T(0), T(0)}, lap[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      T dd[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) dd[q] = D2(8 + i, q);
      lap[i] = trace6(gi, dd);
#pragma unroll
      for (int j = 0; j < 3; ++j) gr[j] += dd[sq(i, j)];
    }
    // gt^ij (d_j d_k beta^k / 3 - (2/3) alpha (2 d_j Kh + d_j Theta) - 16 pi alpha S_j)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      z[j] = (T(1) / T(3)) * (gr[j] - T(2) * al * (T(2) * D1(7, j) + D1(11, j))) - T(16) * PI * al * Si[j];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      s[i] += lap[i] + (gi[sq(i, 0)] * z[0] + gi[sq(i, 1)] * z[1] + gi[sq(i, 2)] * z[2]);
      s[i] -= Gd[0] * db[i][0] + Gd[1] * db[i][1] + Gd[2] * db[i][2];
      s[i] += (T(2) / T(3)) * Gd[i] * divb - T(2) * al * kap * (U(fGX + i) - Gd[i]);
      const T Bi = U(fBBX + i);
      out(fGX + i, s[i] + AK(fGX + i));
      out(fBBX + i, s[i] - p.eta_B * Bi + AK(fBBX + i));
      out(fBX + i, T(0.75) * Bi + AK(fBX + i));
    }
  }
  out(fW, W * (al * K - divb) * (T(1) / T(3)) + AK(fW));
  out(fKH, -D2a + al * (AA + K * K * (T(1) / T(3))) + T(4) * PI * al * SE + al * kap * Th + AK(fKH));
  out(fTH, (p.bssn ? T(0)
                   : fz * (T(0.5) * al * (Rs - AA + (T(2) / T(3)) * K * K) - T(8) * PI * al * E) - T(2) * al * kap * Th) + AK(fTH));
  out(fAL, T(-2) * al * Kh + AK(fAL));
  const T t3 = trX * (T(1) / T(3)), cA = al * K - (T(2) / T(3)) * divb, cg = (T(-2) / T(3)) * divb;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      const int q = sq(i, j);
      // gt_ik d_j beta^k + gt_jk d_i beta^k and At_kj d_i beta^k + At_ki d_j beta^k (for i = j the two
      // sums are one: the other terms are halved and the result doubled)
      const T half = i == j ? T(0.5) : T(1), two = i == j ? T(2) : T(1);
      T sh = half * (cg * g[q] - T(2) * al * A[q]), sa = half * (cA * A[q] + W2 * (X[q] - g[q] * t3));
      sh += g[sq(i, 0)] * db[0][j] + g[sq(i, 1)] * db[1][j] + g[sq(i, 2)] * db[2][j];
      sa += A[sq(j, 0)] * db[0][i] + A[sq(j, 1)] * db[1][i] + A[sq(j, 2)] * db[2][i];
      if (i != j) {
        sh += g[sq(j, 0)] * db[0][i] + g[sq(j, 1)] * db[1][i] + g[sq(j, 2)] * db[2][i];
        sa += A[sq(i, 0)] * db[0][j] + A[sq(i, 1)] * db[1][j] + A[sq(i, 2)] * db[2][j];
      }
      out(fHXX + q, two * sh + AK(fHXX + q));
      out(fAXX + q, two * sa + AK(fAXX + q));
    }
  rs(Rs);
}

}  // namespace sacra
