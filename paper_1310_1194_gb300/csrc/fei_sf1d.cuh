// fei_sf1d.cuh -- one-dimensional factors of the collapsed tensor-product
// basis as compile-time constants, and the layout of the factor tables that
// the sum-factorised kernels (forward and adjoint) keep in shared memory.
//
// With the collapsed coordinates xi1 = (1+u)(1-v)/4, xi2 = (1+v)/2, zeta the
// basis is phi_{(m,n),k} = A_m(u) B_mn(v) L_k(zeta), and its derivatives in
// (u, v, zeta) are products too:
//   F_0 = A B L,  F_1 = A' B L,  F_2 = A (2 B') L,  F_3 = A B L'.
// The reference gradient is a pointwise combination of them,
//   d/dxi1 = g F_1,  d/dxi2 = s g F_1 + F_2,  d/dzeta = F_3,
//   g = 4 / (1-v),  s = (1+u) / 2,
// so with the adjugate rows (adj_0, adj_1, adj_2) replaced by
// (g (adj_0 + s adj_1), adj_1, adj_2) the point operator of fei_geom.cuh
// couples the separable F_a, 13 pairs (a, b) in all, each direction with two
// kinds of factor (the function or its derivative).  Pairs with the same v
// and zeta factors share their v and zeta sums: nine combinations
// (v kind of the row, v kind of the column, zeta kinds), kCombo below.
#pragma once

#include <stdint.h>

namespace fei {

// Gauss-Legendre nodes of M points and the Legendre factors on them, by
// constant evaluation: Newton's method on P_M from the previous root's
// neighbourhood (the roots interlace those of P_{M-1}; bisection brackets
// them), all in FP64.
template <int M>
struct Leg1D {
  double x[M] = {}, w[M] = {};
  double P[M][M] = {}, dP[M][M] = {};  // [degree][node], Legendre, unnormalised
  double L[M][M] = {}, dL[M][M] = {};  // normalised on [-1, 1]

  __host__ __device__ static constexpr double legendre(int n, double t, double *d) {
    double pm = 1.0, pc = t, dm = 0.0, dc = 1.0;
    if (n == 0) {
      *d = 0.0;
      return 1.0;
    }
    for (int k = 1; k < n; ++k) {
      const double pn = ((2 * k + 1) * t * pc - k * pm) / (k + 1);
      const double dn = dm + (2 * k + 1) * pc;
      pm = pc, pc = pn, dm = dc, dc = dn;
    }
    *d = dc;
    return pc;
  }
  __host__ __device__ static constexpr double root(double a) {  // Newton's square root
    double r = a > 1.0 ? a : 1.0;
    for (int i = 0; i < 60; ++i) r = 0.5 * (r + a / r);
    return r;
  }
  constexpr Leg1D() {
    // negative roots by scanning for sign changes, then bisection + Newton
    int found = 0;
    const int steps = 4000;
    double d = 0.0;
    for (int i = 0; i < steps && found < M / 2; ++i) {
      double lo = -1.0 + i * (1.0 / steps), hi = -1.0 + (i + 1) * (1.0 / steps);
      const double fl = legendre(M, lo, &d), fh = legendre(M, hi, &d);
      if (fl * fh >= 0.0 && fh != 0.0) continue;
      double t = 0.5 * (lo + hi);
      for (int it = 0; it < 8; ++it) t -= legendre(M, t, &d) / d;
      if (t > -1e-9) continue;
      x[found] = t;
      x[M - 1 - found] = -t;
      ++found;
    }
    if (M % 2) x[M / 2] = 0.0;
    for (int i = 0; i < M; ++i) {
      legendre(M, x[i], &d);
      w[i] = 2.0 / ((1.0 - x[i] * x[i]) * d * d);
      for (int k = 0; k < M; ++k) {
        double dk = 0.0;
        P[k][i] = legendre(k, x[i], &dk);
        dP[k][i] = dk;
        const double nk = root((2.0 * k + 1.0) / 2.0);
        L[k][i] = nk * P[k][i];
        dL[k][i] = nk * dk;
      }
    }
  }
  // value of factor kind (0: function, 1: derivative) of degree k at node i
  __host__ __device__ constexpr double U(int kind, int k, int i) const { return kind ? dP[k][i] : P[k][i]; }
  // product of two zeta factors in the discrete Legendre basis of the nodes:
  // Z_a,k Z_b,k' = sum_l zz(...) L_l on the nodes, so that
  // sum_i Z_a,k(x_i) Z_b,k'(x_i) d_i = sum_l zz d^_l with
  // d^_l = sum_i L_l(x_i) d_i.  Zero by parity for odd k + a + k' + b + l,
  // and by degree for many of the low functions.
  constexpr double zz(int a, int b, int k, int k2, int l) const {
    if ((k + a + k2 + b + l) % 2) return 0.0;
    double s = 0.0;
    for (int i = 0; i < M; ++i) s += w[i] * (a ? dL[k][i] : L[k][i]) * (b ? dL[k2][i] : L[k2][i]) * L[l][i];
    return (s < 1e-11 && s > -1e-11) ? 0.0 : s;
  }
};
template <int M>
struct Leg {
  static constexpr Leg1D<M> tab{};
};
// every product coefficient once (constant evaluation is slow)
template <int M>
struct ZzTab {
  double c[2][2][M][M][M] = {};
  constexpr ZzTab() {
    for (int a = 0; a < 2; ++a)
      for (int b = 0; b < 2; ++b)
        for (int k = 0; k < M; ++k)
          for (int k2 = 0; k2 < M; ++k2)
            for (int l = 0; l < M; ++l) c[a][b][k][k2][l] = Leg<M>::tab.zz(a, b, k, k2, l);
  }
};
template <int M>
struct Zz {
  static constexpr ZzTab<M> tab{};
};

// compile-time loop: f(integral_constant<int, I>) for I = 0 .. N-1
template <int I>
struct IntC {
  static constexpr int value = I;
  constexpr operator int() const { return I; }
};
template <int N, int I = 0, typename F>
__device__ __forceinline__ void static_for(F &&f) {
  if constexpr (I < N) {
    f(IntC<I>{});
    static_for<N, I + 1>(static_cast<F &&>(f));
  }
}

// Combination c: v kind of the row (va) and of the column (vb) function and
// the zeta kinds (za, zb).  Its pairs of terms (index of the point operator
// in fei_geom.cuh's layout, u kinds of row and column):
//   0: va 0 vb 0 z 00: Dt00 (0,0), Dt01 (0,1), Dt11 (1,1)
//   1: va 0 vb 1 z 00: Dt02 (0,0), Dt12 (1,0)
//   2: va 1 vb 0 z 00: Dt21 (0,1)
//   3: va 1 vb 1 z 00: Dt22 (0,0)
//   4: va 0 vb 0 z 01: Dt03 (0,0), Dt13 (1,0)
//   5: va 1 vb 0 z 01: Dt23 (0,0)
//   6: va 0 vb 0 z 10: Dt31 (0,1)
//   7: va 0 vb 1 z 10: Dt32 (0,0)
//   8: va 0 vb 0 z 11: Dt33 (0,0)
constexpr int kCombos = 9;
constexpr int kOps = 13;  // point operators Dt00, Dt01..03, Dt11..33

// Layout of the factor tables of one degree (values of type T), M = p+1
// nodes, NT triangle functions, half nodes i < (M+1)/2 (the factors of u are
// even or odd, so the other half of the nodes follows by symmetry):
//   UH[2][M m][4 iu]   U_kind(m) at the half nodes (zero-padded)
//   U0[M m][M iu], U1  A_m and A_m' at every node
//   VC[M iv][NT t][2]  B, 2 B' by triangle function
//   VR[M iv][NT r][2]  the same in row order (m ascending, then n)
//   ZL[M iz][M k], ZD  L_k and L_k'
//   GV[M iv]           g = 4 / (1-v)
//   SU[M iu]           s = (1+u) / 2
//   MT[NT]             m of t
template <int P>
struct SfTab {
  static constexpr int M = P + 1, NT = M * (M + 1) / 2;
  static constexpr int O_UH = 0, O_U0 = O_UH + 2 * M * 4, O_U1 = O_U0 + (M * M + 3) / 4 * 4,
                       O_VC = O_U1 + (M * M + 3) / 4 * 4,
                       O_VR = O_VC + (2 * M * NT + 3) / 4 * 4, O_ZL = O_VR + (2 * M * NT + 3) / 4 * 4,
                       O_ZD = O_ZL + M * M,
                       O_GV = O_ZD + M * M, O_SU = O_GV + M, O_MT = O_SU + M;
  static constexpr int SIZE = (O_MT + NT + 3) / 4 * 4;
};
// Index of the triangle function (m, n): total degree ascending, then n; and
// its place in row order.
__host__ __device__ constexpr int tri_index(int m, int n) { return (m + n) * (m + n + 1) / 2 + n; }
__host__ __device__ constexpr int row_start(int M, int m) { return m * M - m * (m - 1) / 2; }

}  // namespace fei
