// fei_sf.cuh -- sum-factorised forward kernel, FP32 or FP64 (fei_sf1d.cuh has
// the factors).
//
// The paper points to sum factorisation as the way to cut the O(p^9) cost of
// the double loop for high orders (Sec. 1.2-1.3, the special integration it
// cites for p >= 4-5).  Per element, with the point operators Dt of the
// collapsed coordinates at the M^3 nodes (iz, iv, iu):
//   X_c[iv][m][m'][l]  = sum over the pairs of combination c, sum_iu
//                        U(m,iu) U(m',iu) Dt^[l][iv][iu]
//   Y_zz[t][t'][l]     = sum_c sum_iv V(t,iv) V(t',iv) X_c[iv][m(t)][m(t')][l]
//   A[(k,t),(k',t')]   = sum_zz sum_l zz(k,k',l) Y_zz[t][t'][l]
// where Dt^ is Dt in the discrete Legendre basis of the zeta nodes.  In that
// basis the product of two zeta factors has few terms (by parity, and by
// degree for the low functions): at p = 7 the last sum takes about 7 terms
// per entry instead of 32.  Even l meet only the entries with k + k' even
// through the zeta pairs LL and L'L' and odd l through LL' and L'L (and the
// other way round), so an entry class (k + k' even or odd) is a thread's
// work of its own.
//
// Per element 0.23 MFLOP at p = 4 and 3.0 MFLOP at p = 7 (the dense
// contraction: 5.7 and 340).
//
// Blocks are persistent over batches of E elements.  Stages, with one block
// barrier between two:
//   1 one warp per element: the record (fetched one batch ahead), element
//     vectors and node columns, beside the last sums of the batch before;
//   2 point operators of every point, into shared memory;
//   3 the zeta transform of the operators, in place;
//   then per group of rows (m = g and m = M-1-g: M+1 rows t, so groups are
//   alike): 4 the u sums into X (one group of X at a time keeps a block's
//   shared memory small enough for several blocks per SM), 5 the v and zeta
//   sums in registers, with direct stores.
// In stage 5 a thread owns one column t', up to R rows t of one m, and one
// entry class.  X is read as 16-byte vectors, each value feeding about six
// multiply-adds per row; lanes run over t', so that the stores of one
// (k, k') are contiguous and lanes that share m' read the same X.
#pragma once

#include <atomic>
#include <type_traits>

#include "fei_elem32.cuh"
#include "fei_geom.cuh"
#include "fei_internal.cuh"
#include "fei_sf_ops.cuh"

namespace fei {

// Elements per block (E), rows per thread (R), blocks per SM the register
// budget is set for (MINB).  E > 1 where one element's columns and row blocks
// do not fill warps.  Larger R reads X less often; the choices are the fastest
// measured (GB300, FP32; in brackets the kernels that this one replaced: the
// dense one at p = 2, the one with 21 term pairs above):
//   p = 2, 200 000 prisms: 0.49 ms (2.51); MINB = 8: 0.54
//   p = 3,  60 000: 0.31 ms (1.67); R = 2: 0.36
//   p = 4, 100 000: 1.34 ms (5.41); R = 5: 1.68, MINB = 5: 1.48 (both before
//                   the element setup's checks, which took 1.336 to 1.344)
//   p = 5,  20 000: 0.68 ms (1.81); R = 2: 0.71, MINB = 6: 0.71
//   p = 6,  16 384: 1.28 ms (3.8); R = 3: 1.41, MINB = 3: 1.9
//   p = 7,  16 384: 2.12 ms (6.25); R = 2: 2.26, R = 4: 2.15
// What bounds it (ncu): issue (p = 4: 68 % of slots, 11.4 k warp instructions
// an element; p = 7: 54 %, 90 k), with barriers and shared-memory latency as
// the largest stalls; without its stores it takes the same time, DRAM writes
// are the outputs.  FP64: the FP64 pipe (p = 4, 4096 prisms: 1.25 ms; the
// dense kernel 23.2 ms).
template <typename T, int P>
struct SfShape;
template <> struct SfShape<float, 2> { static constexpr int E = 4, R = 3, MINB = 6; };
template <> struct SfShape<float, 3> { static constexpr int E = 3, R = 4, MINB = 6; };
template <> struct SfShape<float, 4> { static constexpr int E = 2, R = 3, MINB = 4; };
template <> struct SfShape<float, 5> { static constexpr int E = 1, R = 3, MINB = 5; };
template <> struct SfShape<float, 6> { static constexpr int E = 1, R = 4, MINB = 2; };
template <> struct SfShape<float, 7> { static constexpr int E = 1, R = 3, MINB = 2; };
template <> struct SfShape<double, 2> { static constexpr int E = 4, R = 3, MINB = 2; };
template <> struct SfShape<double, 3> { static constexpr int E = 3, R = 4, MINB = 2; };
template <> struct SfShape<double, 4> { static constexpr int E = 2, R = 3, MINB = 2; };
template <> struct SfShape<double, 5> { static constexpr int E = 1, R = 4, MINB = 2; };
template <> struct SfShape<double, 6> { static constexpr int E = 1, R = 4, MINB = 1; };
template <> struct SfShape<double, 7> { static constexpr int E = 1, R = 4, MINB = 1; };

template <typename T, int P>
struct SfCfg {
  static constexpr bool F32 = std::is_same<T, float>::value;
  static constexpr int M = P + 1, NT = M * (M + 1) / 2, NSH = nsh_of(P), NQ = nq_of(P), NT2 = M * M;
  static constexpr int E = SfShape<T, P>::E, R = SfShape<T, P>::R, MINB = SfShape<T, P>::MINB;
  static constexpr int NE = (M + 1) / 2, NO = M / 2;  // even and odd l (and half nodes of u)
  // packed FP32 multiply-adds in the v sums; not where odd counts of l would
  // leave halves of the packs unused and cost registers (M = 5, 6)
  static constexpr bool PACKED = F32 && M != 5 && M != 6;
  static constexpr int NG = (M + 1) / 2;              // row groups
  static constexpr int nblk(int g) {                  // row blocks of group g
    const int c0 = M - g, c1 = g + 1;
    return (c0 + R - 1) / R + (M - 1 - g != g ? (c1 + R - 1) / R : 0);
  }
  static constexpr int NBLK = [] {
    int b = 0;
    for (int g = 0; g < NG; ++g) b = nblk(g) > b ? nblk(g) : b;
    return b;
  }();
  static constexpr int WPC = (E * NBLK * NT + 31) / 32;  // warps per entry class
  static constexpr int NW = 2 * WPC, NTH = 32 * NW;
  // an l row of X: even l, then odd l from XO (padded for vector loads)
  static constexpr int XR = M == 5 ? 6 : NE > 2 ? 8 : 4, XO = M == 5 ? 4 : XR / 2;
  // stride of an (m, m') chunk of X: an odd multiple of the vector loads'
  // size, so that the chunks of consecutive m' start in different banks
  static constexpr int XS = M == 3 ? 20 : M == 5 ? 34 : M * XR + 4;
  static constexpr int XC = 2 * M * XS;     // one combination of a group
  // shared memory, in values of T
  static constexpr int O_D = SfTab<P>::SIZE;             // [E] operators (OpPos)
  static constexpr int DE = (kOps * M * (F32 && M == 8 ? 72 : M * M) + 3) / 4 * 4;
  static constexpr int O_X = O_D + E * DE;               // [E][9][2][M m'][XS]
  static constexpr int XE = kCombos * XC;
  static constexpr int O_F = O_X + E * XE;               // [E][NQ] load weights
  static constexpr int O_F1 = O_F + (E * NQ + 3) / 4 * 4;
  static constexpr int O_F2 = O_F1 + (E * NQ + 3) / 4 * 4;
  // v factors as packs: columns [M iv][NT t], then rows [M iv][NT r]
  static constexpr int O_FAC = O_F2 + (E * M * NT + 3) / 4 * 4;
  static constexpr int VALUES = O_FAC + (PACKED ? 8 : 4) * M * NT;
  // lookup tables: per lane of the u sums its operators' and X's offsets,
  // per column of the zeta transform its offset
  static constexpr int PER = E * NT2, W0 = (PER + 31) / 32, W1 = W0 + (2 * PER + 31) / 32,
                       W2 = W1 + (2 * PER + 31) / 32, W3 = W2 + (4 * PER + 31) / 32;
  static constexpr int B_U = VALUES * (int)sizeof(T), B_Z = B_U + 4 * 32 * W3;
  static constexpr int DYN_SMEM = B_Z + (2 * E * kOps * NT2 + 15) / 16 * 16;
  static_assert(E * DE < 65536 && E * XE < 65535, "16-bit offsets");
  static_assert(E <= NW, "one warp per element in the setup");
};

// Element data of one slot.
template <typename T, int P>
struct SfElem {
  std::conditional_t<std::is_same<T, float>::value, Elem32<P>, Elem64<P>> el;
  double cd[14];
  T cf[14];
  int status;
};
// Stage 4: the X values of one (iv, l) for the row functions m = g and
// m = M-1-g and every m', x[j][m'] += sum_iu U_UA(m, iu) U_UB(m', iu) d[iu].
// The factors are even or odd in u, so the sum runs over half the nodes on
// e = d(u) + d(-u) or o = d(u) - d(-u).
// p <= 5: the products of the two factors are constants of the code
template <typename T, int P, int G, int UA, int UB>
__device__ __forceinline__ void u_sum_const(const T *e, const T *o, T (*x)[P + 1]) {
  constexpr int M = P + 1, NE = (M + 1) / 2;
  static_for<(2 * G == M - 1 ? 1 : 2)>([&](auto j) {
    constexpr int m = j.value ? M - 1 - G : G;
    static_for<M>([&](auto m2) {
      static_for<NE>([&](auto i) {
        constexpr double c = Leg<M>::tab.U(UA, m, i.value) * Leg<M>::tab.U(UB, m2.value, i.value);
        if constexpr (c != 0.0) x[j.value][m2.value] += T(c) * ((m + UA + m2.value + UB) % 2 ? o[i.value] : e[i.value]);
      });
    });
  });
}
// p >= 6: the row factor from the table (u: its half-node values), so that
// the code does not grow with the row; PAR is the row factor's parity
template <typename T, int P, int UB, int PAR>
__device__ __forceinline__ void u_sum_row(const T *e, const T *o, const T *u, T *x) {
  constexpr int M = P + 1, NE = (M + 1) / 2;
  T ue[NE], uo[NE];
#pragma unroll
  for (int i = 0; i < NE; ++i) ue[i] = u[i] * e[i], uo[i] = u[i] * o[i];
  static_for<M>([&](auto m2) {
    static_for<NE>([&](auto i) {
      constexpr double c = Leg<M>::tab.U(UB, m2.value, i.value);
      if constexpr (c != 0.0) x[m2.value] += T(c) * ((m2.value + UB + PAR) % 2 ? uo[i.value] : ue[i.value]);
    });
  });
}
template <typename T, int P, int UA, int UB>
__device__ __forceinline__ void u_sum(const T *D, int sw, const T *tab, int g, T (*x)[P + 1]) {
  constexpr int M = P + 1, NE = (M + 1) / 2, NG = (M + 1) / 2;
  T d[M], e[NE], o[NE];
  load_u_row<M>(D, sw, d);
  even_odd<T, M>(d, e, o);
  if constexpr (P <= 5) {
    static_for<NG>([&](auto gg) {
      if (g == gg.value) u_sum_const<T, P, gg.value, UA, UB>(e, o, x);
    });
  } else {
    const bool single = 2 * g == M - 1;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (j && single) break;
      const int m = j ? M - 1 - g : g;
      T u[4];
      load_vec<NE>(tab + SfTab<P>::O_UH + (UA * M + m) * 4, u);
      if ((m + UA) & 1) u_sum_row<T, P, UB, 1>(e, o, u, x[j]);
      else u_sum_row<T, P, UB, 0>(e, o, u, x[j]);
    }
  }
}

// Packs of values for the v sums.  FP32: pairs with packed multiply-adds (half
// the issue slots), the v factors stored twice ({B, B, 2B', 2B'}) so that they
// need no move into a pair.
template <typename T, bool PACKED>
struct Pack;
template <>
struct Pack<float, true> {
  using type = float2;
  using factors = float4;
  static constexpr int W = 2;
  static __device__ __forceinline__ float2 zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ float2 first(float4 f) { return make_float2(f.x, f.y); }
  static __device__ __forceinline__ float2 second(float4 f) { return make_float2(f.z, f.w); }
  static __device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
  static __device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
  static __device__ __forceinline__ float get(float2 v, int i) { return i ? v.y : v.x; }
  template <int N, bool A16>
  static __device__ __forceinline__ void load(const float *s, float2 *v) {
    if constexpr (N == 2 && A16) {
      const float4 f = *reinterpret_cast<const float4 *>(s);
      v[0] = make_float2(f.x, f.y), v[1] = make_float2(f.z, f.w);
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) v[i] = reinterpret_cast<const float2 *>(s)[i];
    }
  }
  static __device__ __forceinline__ void put(float *f, int i, float b, float d) {
    reinterpret_cast<float4 *>(f)[i] = make_float4(b, b, d, d);
  }
};
template <typename T>
struct Pack<T, false> {
  using type = T;
  using factors = typename Vec2<T>::type;
  static constexpr int W = 1;
  static __device__ __forceinline__ T zero() { return T(0); }
  static __device__ __forceinline__ T first(factors f) { return f.x; }
  static __device__ __forceinline__ T second(factors f) { return f.y; }
  static __device__ __forceinline__ T mul(T a, T b) { return a * b; }
  static __device__ __forceinline__ T fma(T a, T b, T c) { return a * b + c; }
  static __device__ __forceinline__ T get(T v, int) { return v; }
  template <int N, bool A16>
  static __device__ __forceinline__ void load(const T *s, T *v) {
    if constexpr (A16 || N <= 2) {
      load_vec<N>(s, v);
    } else {
      load_vec<2>(s, v);
      v[2] = s[2];
    }
  }
  static __device__ __forceinline__ void put(T *f, int i, T b, T d) {
    factors v;
    v.x = b, v.y = d;
    reinterpret_cast<factors *>(f)[i] = v;
  }
};

// Stage 5 for one entry class CL (parity of k + k'): nr rows from n0 of
// (m, ml) and column t2 = (m2, ...), results stored at o (row t of the first
// row, column t2), or zeros for a flagged element.
template <typename T, int P, int CL, bool UP>
__device__ __forceinline__ void v_zeta_sums(const T *X, const T *fac, int ml, int m, int n0, int nr, int t2, int m2,
                                            T *A, bool flagged) {
  using C = SfCfg<T, P>;
  constexpr int M = C::M, NT = C::NT, NSH = C::NSH, R = C::R, XR = C::XR, XS = C::XS, XC = C::XC;
  // values of l that meet LL and L'L' (same parity as the class) and LL', L'L
  constexpr int NA = CL ? C::NO : C::NE, NB = CL ? C::NE : C::NO;
  constexpr int OA = CL ? C::XO : 0, OB = CL ? 0 : C::XO;
  auto row_of = [&](int r) { return tri_index(m, n0 + r); };
  // entry (k, k') of row t; o: A_e[t][t2] (full layout)
  auto store = [&](T *o, int k, int k2, int t, T v) {
    if constexpr (UP) {
      // column k' NT + t2 >= row k NT + t: every k' > k, none below, and at
      // k' = k the columns t2 >= t
      if (k2 > k || (k2 == k && t2 >= t)) {
        const int row = k * NT + t;
        A[row * NSH - row * (row + 1) / 2 + k2 * NT + t2] = v;
      }
    } else {
      o[k * NT * NSH + k2 * NT] = v;
    }
  };
  if (flagged) {
    for (int r = 0; r < nr; ++r)
      for (int k = 0; k < M; ++k)
        for (int k2 = (k + CL) & 1; k2 < M; k2 += 2) store(A + (row_of(r) * NSH + t2), k, k2, row_of(r), T(0));
    return;
  }
  // PA, PB: the values of l as packs of W (FP32: pairs, one packed
  // multiply-add each; an odd count leaves the last half unused)
  using Pk = Pack<T, C::PACKED>;
  constexpr bool A16 = XR % 4 == 0, ROLL = P >= 4;
  using V = typename Pk::type;
  constexpr int W = Pk::W, PA = (NA + W - 1) / W, PB = (NB + W - 1) / W;
  V a00[R][PA], a11[R][PA], a01[R][PB], a10[R][PB];
#pragma unroll
  for (int r = 0; r < R; ++r) {
#pragma unroll
    for (int i = 0; i < PA; ++i) a00[r][i] = a11[r][i] = Pk::zero();
#pragma unroll
    for (int i = 0; i < PB; ++i) a01[r][i] = a10[r][i] = Pk::zero();
  }
  const T *x0 = X + (ml * M + m2) * XS;
  const typename Pk::factors *vc = reinterpret_cast<const typename Pk::factors *>(fac) + t2;
  const typename Pk::factors *vr = reinterpret_cast<const typename Pk::factors *>(fac) + M * NT + row_start(M, m) + n0;
#pragma unroll 1
  for (int iv = 0; iv < M; ++iv) {
    const typename Pk::factors fb = vc[iv * NT];
    const V b0 = Pk::first(fb), b1 = Pk::second(fb);
    const T *xa = x0 + iv * XR + OA, *xb = x0 + iv * XR + OB;
    V za[PA], zb[PA], zc[PA], zd[PB], ze[PB], zf[PB];
    {
      V p[PA], q[PA];
      Pk::template load<PA, A16>(xa, p);
      Pk::template load<PA, A16>(xa + XC, q);
#pragma unroll
      for (int i = 0; i < PA; ++i) za[i] = Pk::fma(b1, q[i], Pk::mul(b0, p[i]));
      Pk::template load<PA, A16>(xa + 2 * XC, p);
      Pk::template load<PA, A16>(xa + 3 * XC, q);
#pragma unroll
      for (int i = 0; i < PA; ++i) zb[i] = Pk::fma(b1, q[i], Pk::mul(b0, p[i]));
      Pk::template load<PA, A16>(xa + 8 * XC, p);
#pragma unroll
      for (int i = 0; i < PA; ++i) zc[i] = Pk::mul(b0, p[i]);
    }
    {
      V p[PB], q[PB];
      Pk::template load<PB, A16>(xb + 4 * XC, p);
      Pk::template load<PB, A16>(xb + 5 * XC, q);
#pragma unroll
      for (int i = 0; i < PB; ++i) zd[i] = Pk::mul(b0, p[i]), ze[i] = Pk::mul(b0, q[i]);
      Pk::template load<PB, A16>(xb + 6 * XC, p);
      Pk::template load<PB, A16>(xb + 7 * XC, q);
#pragma unroll
      for (int i = 0; i < PB; ++i) zf[i] = Pk::fma(b1, q[i], Pk::mul(b0, p[i]));
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (r < nr) {
        const typename Pk::factors fa = vr[iv * NT + r];
        const V c0 = Pk::first(fa), c1 = Pk::second(fa);
#pragma unroll
        for (int i = 0; i < PA; ++i) {
          a00[r][i] = Pk::fma(c0, za[i], a00[r][i]);
          a00[r][i] = Pk::fma(c1, zb[i], a00[r][i]);
          a11[r][i] = Pk::fma(c0, zc[i], a11[r][i]);
        }
#pragma unroll
        for (int i = 0; i < PB; ++i) {
          a01[r][i] = Pk::fma(c0, zd[i], a01[r][i]);
          a01[r][i] = Pk::fma(c1, ze[i], a01[r][i]);
          a10[r][i] = Pk::fma(c0, zf[i], a10[r][i]);
        }
      }
    }
  }
  // zeta sums of one row: the entries (k, k') of the class.  LL and L'L'
  // contribute alike to (k, k') and (k', k), and LL' to one what L'L does to
  // the other: with the sum and the difference of Y01 and Y10 an entry pair
  // takes half the terms of its two entries.
  auto zeta_row = [&](int t, const V *v00, const V *v11, const V *v01, const V *v10) {
    T *o = A + (t * NSH + t2);
    T r00[NA], r11[NA], ps[NB], pd[NB];
#pragma unroll
    for (int i = 0; i < NA; ++i) r00[i] = Pk::get(v00[i / W], i % W), r11[i] = Pk::get(v11[i / W], i % W);
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const T y01 = Pk::get(v01[i / W], i % W), y10 = Pk::get(v10[i / W], i % W);
      ps[i] = y01 + y10, pd[i] = y01 - y10;
    }
    static_for<M>([&](auto k) {
      static_for<M - k.value>([&](auto dk) {
        constexpr int ka = k.value, kb = ka + dk.value;
        if constexpr ((ka + kb) % 2 == CL) {
          T s = T(0), d = T(0);
          static_for<NA>([&](auto i) {
            constexpr int l = 2 * i.value + CL;
            constexpr double c00 = Zz<M>::tab.c[0][0][ka][kb][l], c11 = Zz<M>::tab.c[1][1][ka][kb][l];
            if constexpr (c00 != 0.0) s += T(c00) * r00[i.value];
            if constexpr (c11 != 0.0) s += T(c11) * r11[i.value];
          });
          static_for<NB>([&](auto i) {
            constexpr int l = 2 * i.value + 1 - CL;
            constexpr double ca = Zz<M>::tab.c[0][1][ka][kb][l], cb = Zz<M>::tab.c[0][1][kb][ka][l];
            constexpr double hs = 0.5 * (ca + cb), hd = 0.5 * (ca - cb);
            if constexpr (hs > 1e-11 || hs < -1e-11) s += T(hs) * ps[i.value];
            if constexpr (ka != kb && (hd > 1e-11 || hd < -1e-11)) d += T(hd) * pd[i.value];
          });
          if constexpr (ka == kb) {
            store(o, ka, ka, t, s);
          } else {
            store(o, ka, kb, t, s + d);
            store(o, kb, ka, t, s - d);
          }
        }
      });
    });
  };
  if constexpr (ROLL) {
    // the next row's values move down: the code of the entries exists once
    // (unrolled rows miss the instruction cache: p = 4 1.38, p = 7 2.21 ms)
#pragma unroll 1
    for (int r = 0; r < nr; ++r) {
      zeta_row(row_of(r), a00[0], a11[0], a01[0], a10[0]);
#pragma unroll
      for (int j = 0; j + 1 < R; ++j) {
#pragma unroll
        for (int i = 0; i < PA; ++i) a00[j][i] = a00[j + 1][i], a11[j][i] = a11[j + 1][i];
#pragma unroll
        for (int i = 0; i < PB; ++i) a01[j][i] = a01[j + 1][i], a10[j][i] = a10[j + 1][i];
      }
    }
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (r < nr) zeta_row(row_of(r), a00[r], a11[r], a01[r], a10[r]);
  }
}

template <typename T, int P, bool UP>
__global__ void __launch_bounds__(SfCfg<T, P>::NTH, SfCfg<T, P>::MINB) sf_forward_kernel(FwdArgs a, const T *gtab) {
  using C = SfCfg<T, P>;
  constexpr bool F32 = C::F32;
  constexpr int M = C::M, NT = C::NT, NSH = C::NSH, NQ = C::NQ, NT2 = C::NT2, E = C::E, NTH = C::NTH, NW = C::NW,
                XR = C::XR, XS = C::XS, XC = C::XC, R = C::R;
  extern __shared__ __align__(16) unsigned char smraw[];
  T *sm = reinterpret_cast<T *>(smraw);
  __shared__ SfElem<T, P> ELS[2][E];  // this batch's and the next one's
  __shared__ std::conditional_t<F32, NodeTab32<P>, SfNodes64<P>> nodes;
  T *D = sm + C::O_D, *X = sm + C::O_X, *F = sm + C::O_F, *F1 = sm + C::O_F1, *F2 = sm + C::O_F2;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int i = tid; i < SfTab<P>::SIZE; i += NTH) sm[i] = gtab[i];
  if constexpr (F32) {
    load_node_tab32<P>(nodes, a.znode, a.tnode, tid, NTH);
  } else {
    for (int t = tid; t < NT2; t += NTH)
      nodes.tx[t][0] = a.tnode[4 * t], nodes.tx[t][1] = a.tnode[4 * t + 1], nodes.tw[t] = a.tnode[4 * t + 2];
    for (int z = tid; z < M; z += NTH) nodes.zz[z] = a.znode[2 * z], nodes.zw[z] = a.znode[2 * z + 1];
  }
  T *fac = sm + C::O_FAC;
  for (int i = tid; i < 2 * M * NT; i += NTH) {
    const T *v = gtab + SfTab<P>::O_VC + 2 * i;  // VC, then VR (M NT pairs each)
    static_assert(SfTab<P>::O_VR == SfTab<P>::O_VC + (2 * M * NT + 3) / 4 * 4, "VR after VC");
    const T *w = i < M * NT ? v : gtab + SfTab<P>::O_VR + 2 * (i - M * NT);
    Pack<T, C::PACKED>::put(fac, i, w[0], w[1]);
  }
  uint32_t *tabu = reinterpret_cast<uint32_t *>(smraw + C::B_U);
  uint16_t *tabz = reinterpret_cast<uint16_t *>(smraw + C::B_Z);
  // u sums: combinations with the same kinds of pairs share warps: 0 | 1 4 |
  // 2 6 | 3 5 7 8 (most pairs first); entry: the offset of the first pair's
  // u row (its low bits l & 4 where halves are swapped) and of X
  for (int i = tid; i < 32 * C::W3; i += NTH) {
    const int wt = i >> 5, kind = (wt >= C::W0) + (wt >= C::W1) + (wt >= C::W2);
    const int li = i - 32 * (kind == 0 ? 0 : kind == 1 ? C::W0 : kind == 2 ? C::W1 : C::W2), j = li / C::PER,
              i0 = li - j * C::PER, sl = i0 / NT2, t = i0 - sl * NT2, iv = t / M, l = t - iv * M;
    const int op = kind == 0 ? 0 : kind == 1 ? 2 + j : kind == 2 ? 7 + 3 * j : (0xCB98 >> (4 * j)) & 15;
    const int ci = kind == 0 ? 0 : kind == 1 ? 1 + 3 * j : kind == 2 ? 2 + 4 * j : (0x8753 >> (4 * j)) & 15;
    const uint32_t dof = sl * C::DE + OpPos<T, M>::row(op, iv, l) + (OpPos<T, M>::SWZ ? l & 4 : 0);
    const uint32_t xof = sl * C::XE + ci * XC + iv * XR + (l & 1) * C::XO + (l >> 1);
    tabu[i] = j < (kind == 0 ? 1 : kind == 3 ? 4 : 2) ? dof | xof << 16 : 0xffffffffu;
  }
  for (int i = tid; i < E * kOps * NT2; i += NTH) {
    const int sl = i / (kOps * NT2), i0 = i - sl * (kOps * NT2), k = i0 / NT2, t = i0 - k * NT2, iv = t / M;
    tabz[i] = (uint16_t)(sl * C::DE + OpPos<T, M>::row(k, iv, 0) + t - iv * M);
  }
  const T *gv = sm + SfTab<P>::O_GV, *su = sm + SfTab<P>::O_SU, *mtf = sm + SfTab<P>::O_MT;
  const int64_t items = a.count ? (int64_t)(*a.count) : a.n_work;
  const bool per_elem = a.coef_mode == FEI_COEF_PER_ELEMENT;

  // Slot of this warp in the element setup (the last warps: the ones with the
  // least work in the last group of rows), and its share of the record of
  // the batch at it: a vertex coordinate (lanes 0..17) or a per-element
  // coefficient.
  const int slot = NW - 1 - warp;
  auto fetch = [&](int64_t it) -> double {
    it += slot;
    if (slot >= E || it >= items) return 0.0;
    const int64_t e = a.list ? (int64_t)a.list[it] : it;
    if (lane < 18) return a.geom[18 * e + lane];
    if (!per_elem) return 0.0;
    const int j = lane - 18;
    return j < 9 ? a.K[9 * e + j] : j < 12 ? a.b[3 * e + j - 9] : j == 12 ? a.c[e] : a.f[e];
  };
  // ---- 1: the record and the node data of one element, one warp
  auto setup = [&](SfElem<T, P> &S, double rec) {
    const bool bad = __any_sync(0xffffffffu, !finite64(rec));
    if (lane < 18) {
      S.el.X[lane] = rec;
    } else {
      S.cd[lane - 18] = rec;
      if constexpr (F32) S.cf[lane - 18] = f64_to_f32_bits(rec);
      else S.cf[lane - 18] = rec;
    }
    __syncwarp();
    if (lane == 0)
      S.status = bad ? FEI_ERR_NONFINITE : UP && per_elem && !coef_symmetric(S.cd, S.cd + 9) ? FEI_ERR_INVALID_ARG : 0;
    if constexpr (F32) {
      elem_setup32<P>(S.el, nodes, lane);
      __syncwarp();
      for (int j = lane; j < 3 * NT2; j += 32) {
        const int t = j / 3, k = j - 3 * t;
        S.el.tc3f[t][k] = tri_column32<P>(S.el, nodes, t, k);
      }
    } else {
      for (int i = lane; i < M + NT2; i += 32) {
        if (i < M) z_columns_from_vertices(S.el.X, nodes.zz[i], S.el.zc1[i], S.el.zc2[i], S.el.zn3[i]);
        else t_column_from_vertices(S.el.X, nodes.tx[i - M][0], nodes.tx[i - M][1], S.el.tc3[i - M]);
      }
    }
  };
  const int64_t step = (int64_t)gridDim.x * E;
  double rec = fetch((int64_t)blockIdx.x * E);
  __syncthreads();
  if (slot < E && (int64_t)blockIdx.x * E + slot < items) setup(ELS[0][slot], rec);
  rec = fetch((int64_t)blockIdx.x * E + step);
  __syncthreads();

  int cur = 0;
  for (int64_t base = (int64_t)blockIdx.x * E; base < items; base += step, cur ^= 1) {
    const int nel = items - base < E ? (int)(items - base) : E;
    SfElem<T, P> *EL = ELS[cur];
    // the next batch's per-point records on their way to the L2
    if (!per_elem)
      for (int sl = 0; sl < E && base + step + sl < items; ++sl) {
        const int64_t it = base + step + sl, e = a.list ? (int64_t)a.list[it] : it;
        const int64_t r = a.q_off ? a.q_off[e] : e * (int64_t)NQ;
        prefetch_l2(a.K + 9 * r, 72 * NQ, tid, NTH);
        prefetch_l2(a.b + 3 * r, 24 * NQ, tid, NTH);
        prefetch_l2(a.c + r, 8 * NQ, tid, NTH);
        prefetch_l2(a.f + r, 8 * NQ, tid, NTH);
      }
    // ---- 2: point operators
    for (int o = tid; o < nel * NQ; o += NTH) {
      // points in the order (iv, iz, iu) of the operators' layout
      const int sl = o / NQ, i0 = o - sl * NQ, iv = i0 / NT2, i1 = i0 - iv * NT2, iz = i1 / M, iu = i1 - iz * M,
                t = iv * M + iu, q = iz * NT2 + t;
      SfElem<T, P> &S = EL[sl];
      T K[9], b[3], cf, ff;
      int pst = 0;
      if (!per_elem) {
        const int64_t e = a.list ? (int64_t)a.list[base + sl] : base + sl;
        const int64_t r = (a.q_off ? a.q_off[e] : e * (int64_t)NQ) + q;
        double cq[14];
#pragma unroll
        for (int k = 0; k < 9; ++k) cq[k] = a.K[9 * r + k];
#pragma unroll
        for (int k = 0; k < 3; ++k) cq[9 + k] = a.b[3 * r + k];
        cq[12] = a.c[r];
        cq[13] = a.f[r];
        T cv[14];
        bool fin = true;
        if constexpr (F32) {
          fin = coef_to_f32<14>(cq, cv);
        } else {
#pragma unroll
          for (int k = 0; k < 14; ++k) fin &= finite64(cv[k] = cq[k]);
        }
        if (!fin) pst = FEI_ERR_NONFINITE;
        else if (UP && !coef_symmetric(cq, cq + 9)) pst = FEI_ERR_INVALID_ARG;
#pragma unroll
        for (int k = 0; k < 9; ++k) K[k] = cv[k];
#pragma unroll
        for (int k = 0; k < 3; ++k) b[k] = cv[9 + k];
        cf = cv[12], ff = cv[13];
      } else {
#pragma unroll
        for (int k = 0; k < 9; ++k) K[k] = S.cf[k];
#pragma unroll
        for (int k = 0; k < 3; ++k) b[k] = S.cf[9 + k];
        cf = S.cf[12], ff = S.cf[13];
      }
      T a0[3], a1[3], a2[3], Dq[16], s, w;
      if constexpr (F32) {
        int st;
        w = nodes.zwf[iz] * nodes.twf[t];
        s = point_wdet32<P>(S.el, nodes, iz, t, w, a.tnode, &st);
        pst = merge_status(pst, st);
        cross3(S.el.zc2f[iz], S.el.tc3f[t], a0);
        cross3(S.el.tc3f[t], S.el.zc1f[iz], a1);
#pragma unroll
        for (int k = 0; k < 3; ++k) a2[k] = S.el.zn3f[iz][k];
      } else {
        w = nodes.zw[iz] * nodes.tw[t];
        s = w * dot3(S.el.zn3[iz], S.el.tc3[t]);
        pst = merge_status(pst, point_status(s));
        cross3(S.el.zc2[iz], S.el.tc3[t], a0);
        cross3(S.el.tc3[t], S.el.zc1[iz], a1);
#pragma unroll
        for (int k = 0; k < 3; ++k) a2[k] = S.el.zn3[iz][k];
      }
      // adjugate row of the u derivative: g (adj_0 + s adj_1)
#pragma unroll
      for (int k = 0; k < 3; ++k) a0[k] = gv[iv] * (a0[k] + su[iu] * a1[k]);
      dt_from_adj<T>(a0, a1, a2, w, s, w * w / s, K, b, cf, ff, Dq);
      T *dst = D + sl * C::DE;
#pragma unroll
      for (int k = 0; k < kOps; ++k) dst[OpPos<T, M>::at(k, iv, iz, iu)] = Dq[k];
      F[sl * NQ + q] = Dq[13];
      if (pst) atomicMax(&S.status, pst);
    }
    __syncthreads();
    // ---- 3: zeta transform, d^_l = sum_i L_l(z_i) d_i, even and odd l
    for (int o = tid; o < nel * kOps * NT2; o += NTH) {
      // the column (op, iv, iu) at stride M in l (halves swapped by l & 4)
      const int c0 = tabz[o];
      auto at = [&](int l) { return (OpPos<T, M>::SWZ ? c0 ^ (l & 4) : c0) + l * M; };
      T d[M];
#pragma unroll
      for (int i = 0; i < M; ++i) d[i] = D[at(i)];
      T ev[C::NE], od[C::NE];
#pragma unroll
      for (int i = 0; i < C::NE; ++i) {
        const bool mid = 2 * i == M - 1;
        ev[i] = mid ? d[i] : d[i] + d[M - 1 - i];
        od[i] = mid ? T(0) : d[i] - d[M - 1 - i];
      }
      static_for<M>([&](auto l) {
        T s = T(0);
        static_for<C::NE>([&](auto i) {
          constexpr double c = Leg<M>::tab.L[l.value][i.value];
          if constexpr (c != 0.0) s += T(c) * (l.value % 2 ? od[i.value] : ev[i.value]);
        });
        D[at(l.value)] = s;
      });
    }
    __syncthreads();

#pragma unroll 1
    for (int g = 0; g < C::NG; ++g) {
      const bool single = 2 * g == M - 1;
      // ---- 4: u sums, lanes over (combination, iv, l)
      {
        for (int wt = warp; wt < C::W3; wt += NW) {
          const uint32_t ent = tabu[32 * wt + lane];
          const int dof = ent & 0xffffu, xof = ent >> 16;
          if (ent == 0xffffffffu || dof >= nel * C::DE) continue;
          T x[2][M];
#pragma unroll
          for (int i = 0; i < M; ++i) x[0][i] = x[1][i] = T(0);
          constexpr int OP = OpPos<T, M>::OP;
          const int sw = OpPos<T, M>::SWZ ? dof & 4 : 0;
          const T *Dd = D + dof - sw;
          if (wt < C::W0) {
            u_sum<T, P, 0, 0>(Dd, sw, sm, g, x);
            u_sum<T, P, 0, 1>(Dd + OP, sw, sm, g, x);
            u_sum<T, P, 1, 1>(Dd + 4 * OP, sw, sm, g, x);
          } else if (wt < C::W1) {
            u_sum<T, P, 0, 0>(Dd, sw, sm, g, x);
            u_sum<T, P, 1, 0>(Dd + 3 * OP, sw, sm, g, x);
          } else if (wt < C::W2) {
            u_sum<T, P, 0, 1>(Dd, sw, sm, g, x);
          } else {
            u_sum<T, P, 0, 0>(Dd, sw, sm, g, x);
          }
          T *dst = X + xof;
#pragma unroll
          for (int m2 = 0; m2 < M; ++m2) dst[m2 * XS] = x[0][m2];
          if (!single) {
#pragma unroll
            for (int m2 = 0; m2 < M; ++m2) dst[(M + m2) * XS] = x[1][m2];
          }
        }
        // load vector: the u sums beside group 0's, the zeta sums beside group 1's
        if (g == 0) {
          for (int o = tid; o < nel * NQ; o += NTH) {
            const int sl = o / NQ, q = o - sl * NQ, row = q / M, m = q - row * M;
            T acc = T(0);
#pragma unroll
            for (int iu = 0; iu < M; ++iu) acc += sm[SfTab<P>::O_U0 + m * M + iu] * F[sl * NQ + row * M + iu];
            F1[sl * NQ + q] = acc;
          }
        } else if (g == 1) {
          for (int o = tid; o < nel * NSH; o += NTH) {
            const int sl = o / NSH, i = o - sl * NSH, k = i / NT, t = i - k * NT;
            const int64_t e = a.list ? (int64_t)a.list[base + sl] : base + sl;
            T acc = T(0);
#pragma unroll
            for (int iz = 0; iz < M; ++iz) acc += sm[SfTab<P>::O_ZL + iz * M + k] * F2[(sl * M + iz) * NT + t];
            reinterpret_cast<T *>(a.bv)[out_b(a, base + sl, e, NSH) + i] = EL[sl].status ? T(0) : acc;
          }
        }
      }
      __syncthreads();
      // ---- 5: v and zeta sums, stores
      {
        const int nb0 = (M - g + R - 1) / R, nb = nb0 + (single ? 0 : (g + R) / R), tasks = nel * nb * NT;
        const int cl = warp >= C::WPC;
        for (int lt = (warp - cl * C::WPC) * 32 + lane; lt < tasks; lt += C::WPC * 32) {
          const int sl = lt / (nb * NT), i0 = lt - sl * (nb * NT), blk = i0 / NT, t2 = i0 - blk * NT;
          const int ml = blk >= nb0, m = ml ? M - 1 - g : g, n0 = (ml ? blk - nb0 : blk) * R;
          const int nr = M - m - n0 < R ? M - m - n0 : R;
          const int64_t e = a.list ? (int64_t)a.list[base + sl] : base + sl;
          T *A = reinterpret_cast<T *>(a.A) + out_a(a, base + sl, e, NSH);
          const T *Xs = X + sl * C::XE;
          const int m2 = (int)mtf[t2];
          const bool flagged = EL[sl].status != 0;
          if (cl == 0) v_zeta_sums<T, P, 0, UP>(Xs, fac, ml, m, n0, nr, t2, m2, A, flagged);
          else v_zeta_sums<T, P, 1, UP>(Xs, fac, ml, m, n0, nr, t2, m2, A, flagged);
        }
        if (g == 0) {
          for (int o = tid; o < nel * M * NT; o += NTH) {
            const int sl = o / (M * NT), i = o - sl * (M * NT), iz = i / NT, t = i - iz * NT, m = (int)mtf[t];
            T acc = T(0);
#pragma unroll
            for (int iv = 0; iv < M; ++iv)
              acc += sm[SfTab<P>::O_VC + 2 * (iv * NT + t)] * F1[sl * NQ + (iz * M + iv) * M + m];
            F2[o] = acc;
          }
        }
        if (g == C::NG - 1 && tid < nel) {
          const int64_t e = a.list ? (int64_t)a.list[base + tid] : base + tid;
          a.status[e] = EL[tid].status;
        }
        // the next batch's setup beside the last group's sums
        if (g == C::NG - 1 && slot < E) {
          if (base + step + slot < items) setup(ELS[cur ^ 1][slot], rec);
          rec = fetch(base + 2 * step);
        }
      }
      __syncthreads();
    }
  }
}

template <typename T, int P, bool UP>
fei_status launch_sf_one(const T *tab, const FwdArgs &a, int64_t grid_work, cudaStream_t s, int64_t grid_cap) {
  using C = SfCfg<T, P>;
  FEI_CUDA_TRY(cudaFuncSetAttribute(sf_forward_kernel<T, P, UP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    C::DYN_SMEM),
               "cudaFuncSetAttribute(sf_forward)");
  // resident blocks of this kernel on the device, asked once per device
  static std::atomic<int> resident[64];
  int dev;
  FEI_CUDA_TRY(cudaGetDevice(&dev), "cudaGetDevice");
  int fit = dev < 64 ? resident[dev].load(std::memory_order_relaxed) : 0;
  if (!fit) {
    int sms, per_sm = 1;
    FEI_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "cudaDeviceGetAttribute");
    FEI_CUDA_TRY(
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sf_forward_kernel<T, P, UP>, C::NTH, C::DYN_SMEM),
        "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
    fit = sms * (per_sm < 1 ? 1 : per_sm);
    if (dev < 64) resident[dev].store(fit, std::memory_order_relaxed);
  }
  const int64_t batches = (grid_work + C::E - 1) / C::E;
  int64_t blocks = grid_cap > 0 ? grid_cap : fit;
  if (!a.count && blocks > batches) blocks = batches;
  if (blocks < 1) blocks = 1;
  sf_forward_kernel<T, P, UP><<<(unsigned)blocks, C::NTH, C::DYN_SMEM, s>>>(a, tab);
  FEI_CUDA_TRY(cudaGetLastError(), "sf_forward_kernel launch");
  return FEI_OK;
}

template <typename T, int P>
fei_status launch_sf(const T *tab, const FwdArgs &a, int64_t grid_work, cudaStream_t s, int64_t grid_cap) {
  using C = SfCfg<T, P>;
  static_assert(2 * C::E * sizeof(SfElem<T, P>) + 4096 + C::DYN_SMEM <= 232448, "shared memory of one block (227 KB)");
  if (!tab) return set_error(FEI_ERR_UNSUPPORTED, "no sum-factorised tables for degree %d", P);
  return a.upper ? launch_sf_one<T, P, true>(tab, a, grid_work, s, grid_cap)
                 : launch_sf_one<T, P, false>(tab, a, grid_work, s, grid_cap);
}

}  // namespace fei
