// fei_backward.cu -- reverse pass of the element integration.
//
// L = <gA, A> + <gb, b>.  With A_e = sum_q G_q^T Dt_q G_q (fei_geom.cuh):
//   dL/dDt_q[a][b] = (G_q gA G_q^T)[a][b],  dL/d(w det J f)_q = sum_i gb_i phi_i(q).
// The contraction is the transpose of the sum-factorised forward
// (fei_sf.cuh, fei_sf1d.cuh): per element, with F_a the separable factors of
// the collapsed coordinates,
//   Y_zz[t][t'][l]    = sum over (k,k') zz(k,k',l) gA[(k,t),(k',t')]
//   X_c[m][m'][iv][l] = sum over t of m, t' of m': V(t,iv) V(t',iv) Y_zz[t][t'][l]
//   g^_ab[iv][l][iu]  = sum over (m,m') U(m,iu) U(m',iu) X_c[m][m'][iv][l]
// then the zeta transform's transpose, and per point the step from the
// collapsed operators to Dt.  Rows are taken in groups of one or two m (Y and X
// of a group at a time).  It costs what the forward costs: 0.23 MFLOP per
// element at p = 4, 3.0 at p = 7 (the dense W = gA G^T: 5.7 and 340).
//
// The Jacobian is recomputed at every point (never stored) and the chain
// from dL/dDt to the coefficients, to the adjugate rows and det J, to the
// Jacobian columns c1, c2, c3, to the element vectors and finally to the 18
// vertex coordinates is:
//   Dt00 = w det c, Dt0l = w adj_l.b, Dt_lm = (w/det) adj_l K adj_m^T,
//   adj_0 = c2 x c3, adj_1 = c3 x c1, adj_2 = c1 x c2, det = adj_2 . c3,
//   c1 = A1 + zeta B1, c2 = A2 + zeta B2, c3 = C + xi1 D1 + xi2 D2.
// One element per thread block; blocks are persistent.
#include <atomic>
#include <type_traits>

#include "fei_elem32.cuh"
#include "fei_geom.cuh"
#include "fei_internal.cuh"
#include "fei_sf_ops.cuh"

namespace fei {
namespace {

// Threads and blocks per SM: small blocks, several per SM, one to two points a
// thread.  Rows in groups of two m (m = g and M-1-g, alike in size); at p = 7
// and p = 5 of one m (the shared memory of two and of five blocks per SM; at
// p = 4 and 6 the further barriers cost more).  GB300, p = 5, 20 000 prisms with
// per-point fields: 1.19 ms (gA requested a whole element ahead 1.27, groups of
// two m 1.35, 224 threads and 3 blocks 1.6); the dense adjoint on the tensor
// cores took 5.0.  The parts, by leaving
// them out: zeta sums 0.32 ms (their loads of gA: 0.19 ms of HBM time), v sums
// 0.16, u sums 0.18, the chain 0.31; the rest is barriers and latency (issue
// 53 % of slots, 20 warps an SM).  Since then the forward's check of w det J:
// 1.28 -> 1.31 ms by a profiler's (cold) times.
template <typename T, int P>
struct AdjCfg {
  static constexpr bool F32 = std::is_same<T, float>::value;
  static constexpr int M = P + 1, NT = M * (M + 1) / 2, NSH = nsh_of(P), NQ = nq_of(P), NT2 = M * M;
  static constexpr int NTH = P <= 2 ? 32 : P == 3 ? 64 : P <= 5 ? 128 : 256;
  static constexpr int MINB = F32 ? (P <= 2 ? 24 : P == 3 ? 12 : P == 4 ? 6 : P == 5 ? 5 : 2)
                                  : (P <= 2 ? 8 : P == 3 ? 4 : P == 4 ? 2 : 1);
  static constexpr int NW = NTH / 32;
  static constexpr int GM = P == 7 || P == 5 ? 1 : 2, NG = GM == 1 ? M : (M + 1) / 2;
  static constexpr int RM = GM == 1 ? M : M + 1;  // most rows of a group
  static constexpr int NE = (M + 1) / 2, NP = (M + 1) / 2;  // NP: pairs (m', M-1-m')
  // gA is requested into the L2 one element ahead, or where two elements' gA
  // of every block would fill it (p = 5: 97 MB of 129, and DRAM reads were
  // twice gA) one row group ahead.  Forward and adjoint: p = 5, 20 000 prisms
  // 1.91 -> 1.86 ms, p = 6, 8000 1.67 -> 1.63, p = 7, 4000 1.55 -> 1.37; at p = 4
  // the whole element is better, 1.76 against 1.80 (40 000)
  static constexpr bool BY_GROUP = P >= 5;
  // Y [row][t'][l] of 4 values (LL, L'L', LL', L'L); the stride of t' an odd
  // multiple of 4 values against bank conflicts
  static constexpr int YS = 4 * (M % 2 ? M : M + 1);
  static constexpr int O_Y = SfTab<P>::SIZE, YV = RM * NT * YS;
  static constexpr int O_X = O_Y + YV, XV = kCombos * GM * M * NT2;  // [9][GM][M m'][M iv][M l]
  static constexpr int O_D = O_X + (XV + 3) / 4 * 4;
  static constexpr int DV = (kOps * OpPos<T, M>::OP + 3) / 4 * 4;
  static constexpr int O_G1 = O_D + DV;                         // [2][M][NT]
  static constexpr int O_G2 = O_G1 + (2 * M * NT + 3) / 4 * 4;  // [NQ]
  static constexpr int O_GF = O_G2 + (NQ + 3) / 4 * 4;          // [NQ]
  static constexpr int END = O_GF + (NQ + 3) / 4 * 4;
  // quadratic-loss adjoint: the tables, G1 [2][M][NT] (FP32: pairs), G2
  // [3][NQ], and in FP32 the rounding errors of VC, of ZL .. SU and of U0, U1
  static constexpr int Q_G1 = SfTab<P>::SIZE, Q_G2 = Q_G1 + (F32 ? 2 : 1) * (O_G2 - O_G1),
                       Q_LO = Q_G2 + (3 * NQ + 3) / 4 * 4,
                       Q_LZ = Q_LO + 2 * M * NT, Q_LU = Q_LZ + 2 * M * M + 2 * M,
                       Q_END = F32 ? (Q_LU + 2 * M * M + 3) / 4 * 4 : Q_LO;
};

// The rows of gA of row group g on their way to the L2: a point every 128
// bytes of each row, and its last value.
template <typename T, int P>
__device__ __forceinline__ void prefetch_rows(const T *gA, int g, int tid) {
  using C = AdjCfg<T, P>;
  constexpr int M = C::M, NT = C::NT, NSH = C::NSH, STEP = 128 / (int)sizeof(T), L = (NSH + STEP - 1) / STEP + 1;
  const bool single = C::GM == 1 || 2 * g == M - 1;
  const int n0 = M - g, rows = n0 + (single ? 0 : g + 1);
  for (int o = tid; o < rows * M * L; o += C::NTH) {
    const int i = o / L, j = o - i * L, k = i / rows, r = i - k * rows;
    const int t = r < n0 ? tri_index(g, r) : tri_index(M - 1 - g, r - n0);
    const T *p = gA + (int64_t)(k * NT + t) * NSH + (j * STEP < NSH - 1 ? j * STEP : NSH - 1);
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
  }
}

template <typename T, int P>
struct AdjElem {
  std::conditional_t<std::is_same<T, float>::value, Elem32<P>, Elem64<P>> el;
  T cf[14];
  int status;
  double gev[21];
};

__device__ __forceinline__ int point_status_f(float s) {
  if (!(fabsf(s) <= 3.402823466e38f)) return FEI_ERR_NONFINITE;
  if (!(s > 0.f)) return FEI_ERR_NEGATIVE_JACOBIAN;
  return 0;
}

// The coefficient record r as T; false if a value is not finite.
template <typename T>
__device__ __forceinline__ bool load_coef_b(const BwdArgs &a, int64_t r, T *cf) {
  double cd[14];
#pragma unroll
  for (int k = 0; k < 9; ++k) cd[k] = a.K[9 * r + k];
#pragma unroll
  for (int k = 0; k < 3; ++k) cd[9 + k] = a.b[3 * r + k];
  cd[12] = a.c[r];
  cd[13] = a.f[r];
  if constexpr (std::is_same<T, float>::value) return coef_to_f32<14>(cd, cf);
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 14; ++k) ok &= finite64(cf[k] = cd[k]);
  return ok;
}

// (s, e) with s + e = a + b exactly (Knuth's two-sum), FP32.
__device__ __forceinline__ float2 two_sum_f(float a, float b) {
  const float s = a + b, bb = s - a;
  return make_float2(s, (a - (s - bb)) + (b - bb));
}
// x + y for unevaluated FP32 pairs (hi, lo), normalised.
__device__ __forceinline__ float2 add_pair_f(float2 x, float2 y) {
  const float2 s = two_sum_f(x.x, y.x);
  const float lo = s.y + x.y + y.y;
  const float hi = s.x + lo;
  return make_float2(hi, lo - (hi - s.x));
}

// ---------------------------------------------------------------------------
// Sums over the points of the 21 element-vector and 14 coefficient gradients.
// Each thread holds its points' sums of 32 values; a warp adds them by
// halving: lanes exchange half of their values and add the other half, so
// that lane k ends with value k.  FP32 values are added as unevaluated FP32
// pairs (two-sum, about 2^-44 relative), in a fixed order.
// ---------------------------------------------------------------------------
struct Pair32 {
  using type = float2;
  static __device__ __forceinline__ float2 first(float a, float b) { return two_sum_f(a, b); }
  static __device__ __forceinline__ float2 add(float2 a, float2 b) { return add_pair_f(a, b); }
  static __device__ __forceinline__ float2 shfl(float2 v, int off) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, off), __shfl_xor_sync(0xffffffffu, v.y, off));
  }
  static __device__ __forceinline__ double value(float2 v) { return (double)v.x + (double)v.y; }
};
struct Plain64 {
  using type = double;
  static __device__ __forceinline__ double first(double a, double b) { return a + b; }
  static __device__ __forceinline__ double add(double a, double b) { return a + b; }
  static __device__ __forceinline__ double shfl(double v, int off) { return __shfl_xor_sync(0xffffffffu, v, off); }
  static __device__ __forceinline__ double value(double v) { return v; }
};
template <typename T>
using SumOf = std::conditional_t<std::is_same<T, float>::value, Pair32, Plain64>;

// lane k (k < N): the warp's sum of value k (N a power of two; lanes k + j N
// hold the same sums)
template <int N, typename T>
__device__ __forceinline__ typename SumOf<T>::type warp_sums(const T *v, int lane) {
  using S = SumOf<T>;
  typename S::type w[N == 1 ? 1 : N / 2];
  {
    const bool up = lane & (N / 2);
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      const T keep = up ? v[i + N / 2] : v[i], send = up ? v[i] : v[i + N / 2];
      w[i] = S::first(keep, __shfl_xor_sync(0xffffffffu, send, N / 2));
    }
  }
#pragma unroll
  for (int h = N / 4; h >= 1; h >>= 1) {
    const bool up = lane & h;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const typename S::type keep = up ? w[i + h] : w[i], send = up ? w[i] : w[i + h];
      w[i] = S::add(keep, S::shfl(send, h));
    }
  }
  // the rest of the lanes' bits
#pragma unroll
  for (int off = N; off < 32; off <<= 1) w[0] = S::add(w[0], S::shfl(w[0], off));
  return w[0];
}


// ---------------------------------------------------------------------------
// The transposed sums
// ---------------------------------------------------------------------------

// Y of one row t, column t' and entry class CL (parity of k + k') from gA's
// entries at g (row (k,t) of column (k',t') at k NT NSH + k' NT).
template <typename T, int P, int CL>
__device__ __forceinline__ void zeta_adjoint(const T *g, T *y) {
  constexpr int M = P + 1, NT = M * (M + 1) / 2, NSH = nsh_of(P);
  constexpr int NA = CL ? M / 2 : (M + 1) / 2, NB = CL ? (M + 1) / 2 : M / 2;
  T y00[NA], y11[NA], ps[NB], pd[NB];
#pragma unroll
  for (int i = 0; i < NA; ++i) y00[i] = y11[i] = T(0);
#pragma unroll
  for (int i = 0; i < NB; ++i) ps[i] = pd[i] = T(0);
  static_for<M>([&](auto k) {
    static_for<M - k.value>([&](auto dk) {
      constexpr int ka = k.value, kb = ka + dk.value;
      if constexpr ((ka + kb) % 2 == CL) {
        const T g1 = g[ka * NT * NSH + kb * NT], g2 = ka == kb ? T(0) : g[kb * NT * NSH + ka * NT];
        const T s = g1 + g2, d = g1 - g2;
        static_for<NA>([&](auto i) {
          constexpr int l = 2 * i.value + CL;
          constexpr double c00 = Zz<M>::tab.c[0][0][ka][kb][l], c11 = Zz<M>::tab.c[1][1][ka][kb][l];
          if constexpr (c00 != 0.0) y00[i.value] += T(c00) * s;
          if constexpr (c11 != 0.0) y11[i.value] += T(c11) * s;
        });
        static_for<NB>([&](auto i) {
          constexpr int l = 2 * i.value + 1 - CL;
          constexpr double ca = Zz<M>::tab.c[0][1][ka][kb][l], cb = Zz<M>::tab.c[0][1][kb][ka][l];
          constexpr double hs = 0.5 * (ca + cb), hd = 0.5 * (ca - cb);
          if constexpr (hs > 1e-11 || hs < -1e-11) ps[i.value] += T(hs) * s;
          if constexpr (ka != kb && (hd > 1e-11 || hd < -1e-11)) pd[i.value] += T(hd) * d;
        });
      }
    });
  });
  using V2 = typename Vec2<T>::type;
#pragma unroll
  for (int i = 0; i < NA; ++i) {
    V2 v;
    v.x = y00[i], v.y = y11[i];
    *reinterpret_cast<V2 *>(y + 4 * (2 * i + CL)) = v;
  }
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    V2 v;
    v.x = ps[i] + pd[i], v.y = ps[i] - pd[i];
    *reinterpret_cast<V2 *>(y + 4 * (2 * i + 1 - CL) + 2) = v;
  }
}

__device__ __forceinline__ void load4(const float *s, float *d) {
  const float4 v = *reinterpret_cast<const float4 *>(s);
  d[0] = v.x, d[1] = v.y, d[2] = v.z, d[3] = v.w;
}
__device__ __forceinline__ void load4(const double *s, double *d) {
  const double2 v = *reinterpret_cast<const double2 *>(s), w = *reinterpret_cast<const double2 *>(s + 2);
  d[0] = v.x, d[1] = v.y, d[2] = w.x, d[3] = w.y;
}

// X_c of one (iv, l): the nr rows of m (Y rows from y, vr their v factors)
// against the functions t' of m2 (vb their v factors at iv, from vc).
// HALF: 0 both halves of the combinations, 1 those of LL and L'L' (0..3, 8), 2 those
// of LL' and L'L (4..7).
template <typename T, int P, int HALF>
__device__ __forceinline__ void v_adjoint(const T *y, const typename Vec2<T>::type *vr, int nr,
                                          const typename Vec2<T>::type *vc, int m2, T *x) {
  using C = AdjCfg<T, P>;
  constexpr bool HA = HALF != 2, HB = HALF != 1;
  constexpr int M = C::M, NT = C::NT, YS = C::YS;
  using V2 = typename Vec2<T>::type;
  const int cnt = M - m2;
  V2 vb[M];
#pragma unroll
  for (int n = 0; n < M; ++n)
    if (n < cnt) vb[n] = vc[tri_index(m2, n)];
  T acc[kCombos];
#pragma unroll
  for (int c = 0; c < kCombos; ++c) acc[c] = T(0);
  const T *y0 = y + tri_index(m2, 0) * YS;
#pragma unroll 1
  for (int r = 0; r < nr; ++r, y0 += NT * YS) {
    T i00a = T(0), i00b = T(0), i11 = T(0), i01 = T(0), i10a = T(0), i10b = T(0);
    const T *yp = y0;
#pragma unroll
    for (int n = 0; n < M; ++n) {
      if (n >= cnt) break;
      T v[4];
      if constexpr (HALF == 0) load4(yp, v);
      else load_vec<2>(yp + (HB ? 2 : 0), v + (HB ? 2 : 0));
      if constexpr (HA) {
        i00a += vb[n].x * v[0];
        i00b += vb[n].y * v[0];
        i11 += vb[n].x * v[1];
      }
      if constexpr (HB) {
        i01 += vb[n].x * v[2];
        i10a += vb[n].x * v[3];
        i10b += vb[n].y * v[3];
      }
      yp += (m2 + n + 2) * YS;  // to tri_index(m2, n + 1)
    }
    const V2 va = vr[r];
    if constexpr (HA) {
      acc[0] += va.x * i00a;
      acc[1] += va.x * i00b;
      acc[2] += va.y * i00a;
      acc[3] += va.y * i00b;
      acc[8] += va.x * i11;
    }
    if constexpr (HB) {
      acc[4] += va.x * i01;
      acc[5] += va.y * i01;
      acc[6] += va.x * i10a;
      acc[7] += va.x * i10b;
    }
  }
#pragma unroll
  for (int c = 0; c < kCombos; ++c)
    if ((c < 4 || c == 8) ? HA : HB) x[c * (C::GM * M * C::NT2)] = acc[c];
}

template <int M>
__device__ __forceinline__ void store_u_row(float *D, int sw, const float *d) {
  if constexpr (M == 8) {
    *reinterpret_cast<float4 *>(D + sw) = make_float4(d[0], d[1], d[2], d[3]);
    *reinterpret_cast<float4 *>(D + (sw ^ 4)) = make_float4(d[4], d[5], d[6], d[7]);
  } else if constexpr (M == 4) {
    *reinterpret_cast<float4 *>(D) = make_float4(d[0], d[1], d[2], d[3]);
  } else if constexpr (M % 2 == 0) {
#pragma unroll
    for (int c = 0; c < M / 2; ++c) reinterpret_cast<float2 *>(D)[c] = make_float2(d[2 * c], d[2 * c + 1]);
  } else {
#pragma unroll
    for (int c = 0; c < M; ++c) D[c] = d[c];
  }
}
template <int M>
__device__ __forceinline__ void store_u_row(double *D, int, const double *d) {
#pragma unroll
  for (int c = 0; c < M; ++c) D[c] = d[c];
}

// One pair of terms of one (iv, l): the u row D (accumulated over the
// groups) += sum over (m, m') U_UA(m, iu) U_UB(m', iu) x[m][m'], the products
// even or odd in u.
template <typename T, int P, int UA, int UB>
__device__ __forceinline__ void u_adjoint(const T (*x)[P + 1], int g, bool single, const T *tab, bool first, T *D,
                                          int sw) {
  using C = AdjCfg<T, P>;
  constexpr int M = C::M, NE = C::NE;
  T e[NE], o[NE];
#pragma unroll
  for (int i = 0; i < NE; ++i) e[i] = o[i] = T(0);
#pragma unroll
  for (int j = 0; j < C::GM; ++j) {
    if (j && single) break;
    const int m = j ? M - 1 - g : g;
    T qe[NE], qo[NE], u[4];
#pragma unroll
    for (int i = 0; i < NE; ++i) qe[i] = qo[i] = T(0);
    static_for<M>([&](auto m2) {
      static_for<NE>([&](auto i) {
        constexpr double c = Leg<M>::tab.U(UB, m2.value, i.value);
        if constexpr (c != 0.0) {
          if constexpr ((m2.value + UB) % 2) qo[i.value] += T(c) * x[j][m2.value];
          else qe[i.value] += T(c) * x[j][m2.value];
        }
      });
    });
    load_vec<NE>(tab + SfTab<P>::O_UH + (UA * M + m) * 4, u);
    const bool odd = (m + UA) & 1;
#pragma unroll
    for (int i = 0; i < NE; ++i) {
      e[i] += u[i] * (odd ? qo[i] : qe[i]);
      o[i] += u[i] * (odd ? qe[i] : qo[i]);
    }
  }
  T d[M];
  if (first) {
#pragma unroll
    for (int i = 0; i < M; ++i) d[i] = T(0);
  } else {
    load_u_row<M>(D, sw, d);
  }
#pragma unroll
  for (int i = 0; i < NE; ++i) {
    if (2 * i == M - 1) {
      d[i] += e[i];
    } else {
      d[i] += e[i] + o[i];
      d[M - 1 - i] += e[i] - o[i];
    }
  }
  store_u_row<M>(D, sw, d);
}

// ---------------------------------------------------------------------------
// The chain at one point
// ---------------------------------------------------------------------------

// From dL/dDt (gD00, gD0, gDm) and dL/d(w det J f) (gs): the 14 coefficient
// gradients gco and the gradients of the columns gc1, gc2, gc3.
template <typename T>
__device__ __forceinline__ void chain_point(T w, T s, T det, const T (*adj)[3], const T *cx1, const T *cx2,
                                            const T *cx3, const T *cf, T gD00, const T *gD0, const T (*gDm)[3], T gs,
                                            T *gco, T *gc1, T *gc2, T *gc3) {
  const T *K = cf, *bvec = cf + 9;
  const T cc = cf[12], ff = cf[13], wd = w / det, wdd = wd / det;
  T Ka[3][3], Kta[3][3];
#pragma unroll
  for (int m = 0; m < 3; ++m)
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      Ka[m][r] = K[3 * r] * adj[m][0] + K[3 * r + 1] * adj[m][1] + K[3 * r + 2] * adj[m][2];
      Kta[m][r] = K[r] * adj[m][0] + K[3 + r] * adj[m][1] + K[6 + r] * adj[m][2];
    }
  T U[3][3], V[3][3], Tm[3][3];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      U[r][k] = gDm[r][0] * Ka[0][k] + gDm[r][1] * Ka[1][k] + gDm[r][2] * Ka[2][k];
      V[r][k] = gDm[0][r] * Kta[0][k] + gDm[1][r] * Kta[1][k] + gDm[2][r] * Kta[2][k];
      Tm[r][k] = gDm[r][0] * adj[0][k] + gDm[r][1] * adj[1][k] + gDm[r][2] * adj[2][k];
    }
  // dL/dK = (w / det) adj^T gDm adj, dL/db = w adj^T gD0, dL/dc = w det gD00,
  // dL/df = w det gs
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c)
      gco[3 * r + c] = wd * (adj[0][r] * Tm[0][c] + adj[1][r] * Tm[1][c] + adj[2][r] * Tm[2][c]);
#pragma unroll
  for (int k = 0; k < 3; ++k) gco[9 + k] = w * (gD0[0] * adj[0][k] + gD0[1] * adj[1][k] + gD0[2] * adj[2][k]);
  gco[12] = s * gD00;
  gco[13] = s * gs;
  // through det J and the adjugate rows: with the quadratic form
  // sum_lm gDm[l][m] adj_l K adj_m^T = sum_{l,r} adj[l][r] U[l][r]
  T quad = T(0);
#pragma unroll
  for (int l = 0; l < 3; ++l) quad += adj[l][0] * U[l][0] + adj[l][1] * U[l][1] + adj[l][2] * U[l][2];
  const T gdet = w * (cc * gD00 + ff * gs) - wdd * quad;
  T gadj[3][3];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int k = 0; k < 3; ++k) gadj[r][k] = w * gD0[r] * bvec[k] + wd * (U[r][k] + V[r][k]);
  T tmp[3], gn3[3];
  cross3(cx3, gadj[0], gc2);  // adj0 = c2 x c3
  cross3(gadj[0], cx2, gc3);
  cross3(cx1, gadj[1], tmp);  // adj1 = c3 x c1
#pragma unroll
  for (int k = 0; k < 3; ++k) gc3[k] += tmp[k];
  cross3(gadj[1], cx3, gc1);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    gn3[k] = gadj[2][k] + gdet * cx3[k];  // adj2 = n3, det = n3 . c3
    gc3[k] += gdet * adj[2][k];
  }
  cross3(cx2, gn3, tmp);  // n3 = c1 x c2
#pragma unroll
  for (int k = 0; k < 3; ++k) gc1[k] += tmp[k];
  cross3(gn3, cx1, tmp);
#pragma unroll
  for (int k = 0; k < 3; ++k) gc2[k] += tmp[k];
}

template <typename T, int P, bool Q>
__global__ void __launch_bounds__(AdjCfg<T, P>::NTH, AdjCfg<T, P>::MINB) backward_kernel(BwdArgs a, const T *gtab,
                                                                                              const double *gtab64) {
  using C = AdjCfg<T, P>;
  using S = SumOf<T>;
  using V2 = typename Vec2<T>::type;
  constexpr bool F32 = C::F32;
  constexpr int M = C::M, NT = C::NT, NSH = C::NSH, NQ = C::NQ, NT2 = C::NT2, NTH = C::NTH, NW = C::NW, YS = C::YS;
  extern __shared__ __align__(16) unsigned char dsm[];
  T *sm = reinterpret_cast<T *>(dsm);
  __shared__ AdjElem<T, P> E;
  __shared__ std::conditional_t<F32, NodeTab32<P>, SfNodes64<P>> nodes;
  __shared__ typename S::type red[NW][36], sum[36];
  T *G1 = sm + (Q ? C::Q_G1 : C::O_G1), *G2 = sm + (Q ? C::Q_G2 : C::O_G2), *GF = sm + C::O_GF;
  T *Y = sm + C::O_Y, *X = sm + C::O_X, *D = sm + C::O_D;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int i = tid; i < SfTab<P>::SIZE; i += NTH) sm[i] = gtab[i];
  if constexpr (F32) {
    load_node_tab32<P>(nodes, a.znode, a.tnode, tid, NTH);
  } else {
    for (int t = tid; t < NT2; t += NTH)
      nodes.tx[t][0] = a.tnode[4 * t], nodes.tx[t][1] = a.tnode[4 * t + 1], nodes.tw[t] = a.tnode[4 * t + 2];
    for (int z = tid; z < M; z += NTH) nodes.zz[z] = a.znode[2 * z], nodes.zw[z] = a.znode[2 * z + 1];
  }
  if constexpr (Q && F32) {
    // the factors' rounding errors
    auto err = [&](int at, int from, int n) {
      for (int i = tid; i < n; i += NTH) sm[at + i] = (float)(gtab64[from + i] - (double)gtab[from + i]);
    };
    err(C::Q_LO, SfTab<P>::O_VC, 2 * M * NT);
    err(C::Q_LZ, SfTab<P>::O_ZL, 2 * M * M + 2 * M);
    err(C::Q_LU, SfTab<P>::O_U0, M * M);
    err(C::Q_LU + M * M, SfTab<P>::O_U1, M * M);
  }
  const T *gv = sm + SfTab<P>::O_GV, *su = sm + SfTab<P>::O_SU, *u0 = sm + SfTab<P>::O_U0, *u1 = sm + SfTab<P>::O_U1,
          *zl = sm + SfTab<P>::O_ZL, *zd = sm + SfTab<P>::O_ZD;
  const V2 *vc = reinterpret_cast<const V2 *>(sm + SfTab<P>::O_VC), *vr = reinterpret_cast<const V2 *>(sm + SfTab<P>::O_VR);
  const T *gAg = reinterpret_cast<const T *>(a.gA), *gbg = reinterpret_cast<const T *>(a.gb);
  const int64_t items = a.count ? (int64_t)(*a.count) : a.n_work;
  const bool perq = a.coef_mode == FEI_COEF_PER_POINT;
  // this lane's share of an element's record (last warp): a vertex coordinate
  // or a per-element coefficient
  auto fetch = [&](int64_t it) -> double {
    if (warp != NW - 1 || it >= items) return 0.0;
    const int64_t e = a.list ? (int64_t)a.list[it] : it;
    if (lane < 18) return a.geom[18 * e + lane];
    if (perq) return 0.0;
    const int j = lane - 18;
    return j < 9 ? a.K[9 * e + j] : j < 12 ? a.b[3 * e + j - 9] : j == 12 ? a.c[e] : a.f[e];
  };
  double rec = fetch(blockIdx.x);
  __syncthreads();

  for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const int64_t e = a.list ? (int64_t)a.list[item] : item;
    const int64_t aoff = a.A_off ? a.A_off[e] : e * (int64_t)(NSH * NSH);
    const int64_t boff = a.b_off ? a.b_off[e] : e * (int64_t)NSH;
    const int64_t qoff = a.q_off ? a.q_off[e] : e * (int64_t)NQ;
    // the next element's inputs on their way to the L2
    int64_t anext = -1;
    if (item + gridDim.x < items) {
      const int64_t it = item + gridDim.x, en = a.list ? (int64_t)a.list[it] : it;
      anext = a.A_off ? a.A_off[en] : en * (int64_t)(NSH * NSH);
      if (!Q && !C::BY_GROUP) prefetch_l2(gAg + anext, (int)sizeof(T) * NSH * NSH, tid, NTH);
      if (perq) {
        const int64_t r = a.q_off ? a.q_off[en] : en * (int64_t)NQ;
        prefetch_l2(a.K + 9 * r, 72 * NQ, tid, NTH);
        prefetch_l2(a.b + 3 * r, 24 * NQ, tid, NTH);
        prefetch_l2(a.c + r, 8 * NQ, tid, NTH);
        prefetch_l2(a.f + r, 8 * NQ, tid, NTH);
      }
    }
    // the element's record (fetched one element ahead) and node data, by the
    // last warp beside the first sums
    if (warp == NW - 1) {
      const bool bad = __any_sync(0xffffffffu, !finite64(rec));
      if (lane < 18) {
        E.el.X[lane] = rec;
      } else {
        if constexpr (F32) E.cf[lane - 18] = f64_to_f32_bits(rec);
        else E.cf[lane - 18] = rec;
      }
      if (lane == 0) E.status = bad ? FEI_ERR_NONFINITE : 0;
      __syncwarp();
      if constexpr (F32) {
        elem_setup32<P>(E.el, nodes, lane);
        __syncwarp();
        for (int j = lane; j < 3 * NT2; j += 32) {
          const int t = j / 3, k = j - 3 * t;
          E.el.tc3f[t][k] = tri_column32<P>(E.el, nodes, t, k);
        }
      } else {
        for (int i = lane; i < M + NT2; i += 32) {
          if (i < M) z_columns_from_vertices(E.el.X, nodes.zz[i], E.el.zc1[i], E.el.zc2[i], E.el.zn3[i]);
          else t_column_from_vertices(E.el.X, nodes.tx[i - M][0], nodes.tx[i - M][1], E.el.tc3[i - M]);
        }
      }
      rec = fetch(item + gridDim.x);
    }
    if constexpr (!Q) {
#pragma unroll 1
      for (int g = 0; g < C::NG; ++g) {
        const bool single = C::GM == 1 || 2 * g == M - 1;
        const int n0 = M - g, rows = n0 + (single ? 0 : g + 1);
        if constexpr (C::BY_GROUP) {
          const bool last = g == C::NG - 1;
          if (!last || anext >= 0) prefetch_rows<T, P>(gAg + (last ? anext : aoff), last ? 0 : g + 1, tid);
        }
        // zeta sums: rows of the group, columns t', entry classes
        const int tasks = rows * NT, padded = (tasks + 31) / 32 * 32;
        for (int o = tid; o < 2 * padded; o += NTH) {
          const int cl = o >= padded, lt = o - cl * padded;
          if (lt >= tasks) continue;
          const int r = lt / NT, t2 = lt - r * NT;
          const int t = r < n0 ? tri_index(g, r) : tri_index(M - 1 - g, r - n0);
          const T *src = gAg + aoff + (int64_t)t * NSH + t2;
          T *y = Y + (r * NT + t2) * YS;
          if (cl == 0) zeta_adjoint<T, P, 0>(src, y);
          else zeta_adjoint<T, P, 1>(src, y);
        }
        if (g == 0) {
          for (int o = tid; o < M * NT; o += NTH) {
            const int iz = o / NT, t = o - iz * NT;
            T s = T(0);
#pragma unroll
            for (int k = 0; k < M; ++k) s += zl[iz * M + k] * gbg[boff + k * NT + t];
            G1[o] = s;
          }
        }
        __syncthreads();
        // v sums: lanes over (pair m', M-1-m'; iv; l), and over the two halves
        // of the combinations where one would leave half of the threads idle
        constexpr int VT = C::NP * NT2, SPLIT = VT <= NTH / 2 ? 2 : 1;
        for (int o = tid; o < SPLIT * VT; o += NTH) {
          const int hb = o >= VT, o1 = o - hb * VT, j = o1 / NT2, i0 = o1 - j * NT2, iv = i0 / M, l = i0 - iv * M;
#pragma unroll 1
          for (int ml = 0; ml < (single ? 1 : 2); ++ml) {
            const int m = ml ? M - 1 - g : g;
#pragma unroll 1
            for (int jj = 0; jj < 2; ++jj) {
              const int m2 = jj ? M - 1 - j : j;
              if (jj && m2 == j) break;
              const T *ys = Y + (ml ? n0 * NT * YS : 0) + 4 * l;
              const V2 *rows = vr + iv * NT + row_start(M, m), *cols = vc + iv * NT;
              T *dst = X + (ml * M + m2) * NT2 + i0;
              if constexpr (SPLIT == 1) {
                v_adjoint<T, P, 0>(ys, rows, M - m, cols, m2, dst);
              } else {
                if (hb) v_adjoint<T, P, 2>(ys, rows, M - m, cols, m2, dst);
                else v_adjoint<T, P, 1>(ys, rows, M - m, cols, m2, dst);
              }
            }
          }
        }
        if (g == 0) {
          for (int o = tid; o < NQ; o += NTH) {
            const int iz = o / NT2, i0 = o - iz * NT2, iv = i0 / M, m = i0 - iv * M;
            T s = T(0);
            for (int n = 0; n < M - m; ++n) {
              const int t = tri_index(m, n);
              s += vc[iv * NT + t].x * G1[iz * NT + t];
            }
            G2[o] = s;
          }
        }
        __syncthreads();
        // u sums, accumulated over the groups; lanes over (combination, iv,
        // l), combinations with the same kinds of pairs side by side
        constexpr int per = NT2, w0 = (per + 31) / 32, w1 = w0 + (2 * per + 31) / 32, w2 = w1 + (2 * per + 31) / 32,
                      w3 = w2 + (4 * per + 31) / 32;
        for (int wt = warp; wt < w3; wt += NW) {
          const int kind = (wt >= w0) + (wt >= w1) + (wt >= w2);
          const int li = (wt - (kind == 0 ? 0 : kind == 1 ? w0 : kind == 2 ? w1 : w2)) * 32 + lane, j = li / per,
                    i0 = li - j * per, iv = i0 / M, l = i0 - iv * M;
          if (j >= (kind == 0 ? 1 : kind == 3 ? 4 : 2)) continue;
          const int ci = kind == 0 ? 0 : kind == 1 ? 1 + 3 * j : kind == 2 ? 2 + 4 * j : (0x8753 >> (4 * j)) & 15;
          T x[C::GM][M];
          const T *src = X + ci * (C::GM * M * NT2) + i0;
#pragma unroll
          for (int m2 = 0; m2 < M; ++m2) x[0][m2] = src[m2 * NT2];
          if (C::GM == 2 && !single) {
#pragma unroll
            for (int m2 = 0; m2 < M; ++m2) x[C::GM - 1][m2] = src[(M + m2) * NT2];
          }
          constexpr int OP = OpPos<T, M>::OP;
          T *Dd = D + OpPos<T, M>::row(0, iv, l);
          const int sw = l & 4;
          const bool first = g == 0;
          if (kind == 0) {
            u_adjoint<T, P, 0, 0>(x, g, single, sm, first, Dd, sw);
            u_adjoint<T, P, 0, 1>(x, g, single, sm, first, Dd + OP, sw);
            u_adjoint<T, P, 1, 1>(x, g, single, sm, first, Dd + 4 * OP, sw);
          } else if (kind == 1) {
            u_adjoint<T, P, 0, 0>(x, g, single, sm, first, Dd + (2 + j) * OP, sw);
            u_adjoint<T, P, 1, 0>(x, g, single, sm, first, Dd + (5 + j) * OP, sw);
          } else if (kind == 2) {
            u_adjoint<T, P, 0, 1>(x, g, single, sm, first, Dd + (7 + 3 * j) * OP, sw);
          } else {
            u_adjoint<T, P, 0, 0>(x, g, single, sm, first, Dd + ((0xCB98 >> (4 * j)) & 15) * OP, sw);
          }
        }
        if (g == 0) {
          for (int o = tid; o < NQ; o += NTH) {
            const int row = o / M, iu = o - row * M;
            T s = T(0);
#pragma unroll
            for (int m = 0; m < M; ++m) s += u0[m * M + iu] * G2[row * M + m];
            GF[o] = s;
          }
        }
      }
      __syncthreads();
      // the zeta transform's transpose, in place
      for (int o = tid; o < kOps * NT2; o += NTH) {
        const int k = o / NT2, i0 = o - k * NT2, iv = i0 / M, iu = i0 - iv * M;
        T d[M];
#pragma unroll
        for (int l = 0; l < M; ++l) d[l] = D[OpPos<T, M>::at(k, iv, l, iu)];
        static_for<C::NE>([&](auto i) {
          T ev = T(0), od = T(0);
          static_for<M>([&](auto l) {
            constexpr double c = Leg<M>::tab.L[l.value][i.value];
            if constexpr (c != 0.0) {
              if constexpr (l.value % 2) od += T(c) * d[l.value];
              else ev += T(c) * d[l.value];
            }
          });
          D[OpPos<T, M>::at(k, iv, i.value, iu)] = ev + od;
          if constexpr (2 * i.value != M - 1) D[OpPos<T, M>::at(k, iv, M - 1 - i.value, iu)] = ev - od;
        });
      }
      __syncthreads();
    } else {
      // L_e = u^T A_e u - u^T b_e: with v_q = G_q u (4 values per point),
      // dL/dDt_q = v_q v_q^T and dL/d(w det f)_q = -v_q[0], so gA = u u^T is
      // never formed; v_q by the three one-dimensional sums, the last of
      // them at the point
      if constexpr (F32) {
        // the first two sums in double-FP32 (factors and sums as pairs), so
        // that v_q carries no more rounding than one dense FP32 sum
        float2 *W = reinterpret_cast<float2 *>(G1);
        const float2 *vlo = reinterpret_cast<const float2 *>(sm + C::Q_LO);
        const float *zlo = sm + C::Q_LZ;
        for (int o = tid; o < M * NT; o += NTH) {
          const int iz = o / NT, t = o - iz * NT;
          float2 p = make_float2(0.f, 0.f), d = p;
#pragma unroll
          for (int k = 0; k < M; ++k) {
            const float2 uv = make_float2(f64_to_f32_bits(a.u[boff + k * NT + t]), 0.f);
            p = add_ff(p, mul_ff(uv, make_float2(zl[iz * M + k], zlo[iz * M + k])));
            d = add_ff(d, mul_ff(uv, make_float2(zd[iz * M + k], zlo[M * M + iz * M + k])));
          }
          W[o] = norm_ff(p);
          W[M * NT + o] = norm_ff(d);
        }
        __syncthreads();
        for (int o = tid; o < NQ; o += NTH) {
          const int iz = o / NT2, i0 = o - iz * NT2, iv = i0 / M, m = i0 - iv * M;
          float2 s0 = make_float2(0.f, 0.f), s1 = s0, s2 = s0;
          for (int n = 0; n < M - m; ++n) {
            const int t = tri_index(m, n);
            const float2 v = vc[iv * NT + t], vl = vlo[iv * NT + t], w0 = W[iz * NT + t], w1 = W[(M + iz) * NT + t];
            s0 = add_ff(s0, mul_ff(make_float2(v.x, vl.x), w0));
            s1 = add_ff(s1, mul_ff(make_float2(v.y, vl.y), w0));
            s2 = add_ff(s2, mul_ff(make_float2(v.x, vl.x), w1));
          }
          G2[o] = s0.x + s0.y;
          G2[NQ + o] = s1.x + s1.y;
          G2[2 * NQ + o] = s2.x + s2.y;
        }
      } else {
        for (int o = tid; o < M * NT; o += NTH) {
          const int iz = o / NT, t = o - iz * NT;
          T p = T(0), d = T(0);
#pragma unroll
          for (int k = 0; k < M; ++k) {
            const T uv = a.u[boff + k * NT + t];
            p += zl[iz * M + k] * uv;
            d += zd[iz * M + k] * uv;
          }
          G1[o] = p;
          G1[M * NT + o] = d;
        }
        __syncthreads();
        for (int o = tid; o < NQ; o += NTH) {
          const int iz = o / NT2, i0 = o - iz * NT2, iv = i0 / M, m = i0 - iv * M;
          T s0 = T(0), s1 = T(0), s2 = T(0);
          for (int n = 0; n < M - m; ++n) {
            const int t = tri_index(m, n);
            const V2 v = vc[iv * NT + t];
            const T w0 = G1[iz * NT + t], w1 = G1[(M + iz) * NT + t];
            s0 += v.x * w0;
            s1 += v.y * w0;
            s2 += v.x * w1;
          }
          G2[o] = s0;
          G2[NQ + o] = s1;
          G2[2 * NQ + o] = s2;
        }
      }
      __syncthreads();
    }

    int pst = 0;
    // the chain, one thread per point; acc: 21 element-vector gradients,
    // 11 coefficient gradients, then 3 more (per-element coefficients)
    T acc[36];
#pragma unroll
    for (int k = 0; k < 36; ++k) acc[k] = T(0);
#pragma unroll 1
    for (int q = tid; q < NQ; q += NTH) {
      const int iz = q / NT2, t = q - iz * NT2, iv = t / M, iu = t - iv * M;
      T cf[14];
      if (perq) {
        if (!load_coef_b<T>(a, qoff + q, cf)) pst = FEI_ERR_NONFINITE;
      } else {
#pragma unroll
        for (int k = 0; k < 14; ++k) cf[k] = E.cf[k];
      }
      T w, s, det, adj[3][3], cx1[3], cx2[3], cx3[3], z, x1, x2;
      if constexpr (F32) {
        const float2 wp = mul_ff(nodes.ztab2[iz][1], nodes.ttab2[t][0]);  // rounded once
        w = wp.x + wp.y;
        int st;
        s = point_wdet32<P>(E.el, nodes, iz, t, nodes.zwf[iz] * nodes.twf[t], a.tnode, &st, &det);
        pst = merge_status(pst, merge_status(st, point_status_f(s)));
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          cx1[k] = E.el.zc1f[iz][k];
          cx2[k] = E.el.zc2f[iz][k];
          cx3[k] = E.el.tc3f[t][k];
          adj[2][k] = E.el.zn3f[iz][k];
        }
        z = nodes.ztab2[iz][0].x, x1 = nodes.txi2[t][0].x, x2 = nodes.txi2[t][1].x;
      } else {
        w = nodes.zw[iz] * nodes.tw[t];
        det = dot3(E.el.zn3[iz], E.el.tc3[t]);
        s = w * det;
        pst = merge_status(pst, point_status(s));
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          cx1[k] = E.el.zc1[iz][k];
          cx2[k] = E.el.zc2[iz][k];
          cx3[k] = E.el.tc3[t][k];
          adj[2][k] = E.el.zn3[iz][k];
        }
        z = nodes.zz[iz], x1 = nodes.tx[t][0], x2 = nodes.tx[t][1];
      }
      cross3(cx2, cx3, adj[0]);
      cross3(cx3, cx1, adj[1]);
      // dL/dDt at the point: with G_1 = g F_1, G_2 = s g F_1 + F_2 and
      // G_0, G_3 = F_0, F_3
      T gD00, gD0[3], gDm[3][3], gs;
      const T gp = gv[iv], sp = su[iu];
      if constexpr (Q) {
        T v0 = T(0), v1 = T(0), v2 = T(0), v3 = T(0);
        const T *p = G2 + (iz * M + iv) * M;
        if constexpr (F32) {
          // the factors' rounding errors first: the same for every element and
          // point, they would not average out of the sums over the points
          const T *ul = sm + C::Q_LU + iu;
#pragma unroll
          for (int m = 0; m < M; ++m) {
            v0 += ul[m * M] * p[m];
            v1 += ul[(M + m) * M] * p[m];
            v2 += ul[m * M] * p[NQ + m];
            v3 += ul[m * M] * p[2 * NQ + m];
          }
        }
#pragma unroll
        for (int m = 0; m < M; ++m) {
          const T um = u0[m * M + iu];
          v0 += um * p[m];
          v1 += u1[m * M + iu] * p[m];
          v2 += um * p[NQ + m];
          v3 += um * p[2 * NQ + m];
        }
        if constexpr (F32) {
          v1 = fmaf(gp, v1, sm[C::Q_LZ + 2 * M * M + iv] * v1);
          v2 += sm[C::Q_LZ + 2 * M * M + M + iu] * v1;
        } else {
          v1 *= gp;
        }
        v2 += sp * v1;
        const T v[3] = {v1, v2, v3};
        gD00 = v0 * v0;
        gs = -v0;
#pragma unroll
        for (int l = 0; l < 3; ++l) {
          gD0[l] = v0 * v[l];
#pragma unroll
          for (int m = 0; m < 3; ++m) gDm[l][m] = v[l] * v[m];
        }
      } else {
        auto at = [&](int k) { return D[OpPos<T, M>::at(k, iv, iz, iu)]; };
        gs = GF[q];
        gD00 = at(0);
        gD0[0] = gp * at(1);
        gD0[1] = sp * gD0[0] + at(2);
        gD0[2] = at(3);
        T r[3][3];
#pragma unroll
        for (int l = 0; l < 3; ++l) {
          r[l][0] = gp * at(4 + 3 * l);
          r[l][1] = sp * r[l][0] + at(5 + 3 * l);
          r[l][2] = at(6 + 3 * l);
        }
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          gDm[0][m] = gp * r[0][m];
          gDm[1][m] = sp * gDm[0][m] + r[1][m];
          gDm[2][m] = r[2][m];
        }
      }
      T gco[14], gc1[3], gc2[3], gc3[3];
      chain_point<T>(w, s, det, adj, cx1, cx2, cx3, cf, gD00, gD0, gDm, gs, gco, gc1, gc2, gc3);
      if (perq) {
        const int64_t r = qoff + q;
#pragma unroll
        for (int k = 0; k < 9; ++k) a.gK[9 * r + k] = gco[k];
#pragma unroll
        for (int k = 0; k < 3; ++k) a.gbc[3 * r + k] = gco[9 + k];
        a.gc[r] = gco[12];
        a.gf[r] = gco[13];
      } else {
#pragma unroll
        for (int k = 0; k < 14; ++k) acc[21 + k] += gco[k];
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        acc[0 + k] += gc1[k];
        acc[3 + k] += z * gc1[k];
        acc[6 + k] += gc2[k];
        acc[9 + k] += z * gc2[k];
        acc[12 + k] += gc3[k];
        acc[15 + k] += x1 * gc3[k];
        acc[18 + k] += x2 * gc3[k];
      }
    }
    if (pst) atomicMax(&E.status, pst);
    // sums over the points: per warp, then over the warps in order
    const typename S::type wsum = warp_sums<32>(acc, lane);
    red[warp][lane] = wsum;
    if (!perq) {
      const typename S::type rest = warp_sums<4>(acc + 32, lane);
      if (lane < 4) red[warp][32 + lane] = rest;
    }
    __syncthreads();
    const int nval = perq ? 21 : 35;
    for (int k = tid; k < nval; k += NTH) {
      typename S::type v = red[0][k];
      for (int j = 1; j < NW; ++j) v = S::add(v, red[j][k]);
      sum[k] = v;
      if (k < 21) E.gev[k] = S::value(v);
    }
    __syncthreads();
    const int st = E.status;
    // element vectors -> vertices (transpose of the element vectors'
    // differences): vertex component (vertex i / 3, coordinate i % 3)
    for (int i = tid; i < 18; i += NTH) {
      const int vx = i / 3, k = i - 3 * vx;
      // signs of (A1, B1, A2, B2, C, D1, D2) for P0, P1, P2, Q0, Q1, Q2,
      // two bits each (0: none, 1: +, 2: -)
      const unsigned sg = vx == 0 ? 0x1666u : vx == 1 ? 0x809u : vx == 2 ? 0x2090u : vx == 3 ? 0x29AAu
                          : vx == 4 ? 0x405u : 0x1050u;
      double val;
      if constexpr (F32) {
        float2 v = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 7; ++c) {
          const unsigned b = (sg >> (2 * c)) & 3u;
          if (b) {
            const float2 g = sum[3 * c + k];
            v = add_pair_f(v, b == 1u ? g : make_float2(-g.x, -g.y));
          }
        }
        val = 0.5 * ((double)v.x + (double)v.y);
      } else {
        double v = 0.0;
#pragma unroll
        for (int c = 0; c < 7; ++c) {
          const unsigned b = (sg >> (2 * c)) & 3u;
          if (b) v += b == 1u ? E.gev[3 * c + k] : -E.gev[3 * c + k];
        }
        val = 0.5 * v;
      }
      a.g_geom[18 * e + i] = st ? 0.0 : val;
    }
    if (!perq) {
      for (int k = tid; k < 14; k += NTH) {
        const double v = st ? 0.0 : S::value(sum[21 + k]);
        if (k < 9) a.gK[9 * e + k] = v;
        else if (k < 12) a.gbc[3 * e + (k - 9)] = v;
        else if (k == 12) a.gc[e] = v;
        else a.gf[e] = v;
      }
    } else if (st) {
      // flagged element: overwrite the per-point gradients with zeros
      for (int q = tid; q < NQ; q += NTH) {
        const int64_t r = qoff + q;
        for (int k = 0; k < 9; ++k) a.gK[9 * r + k] = 0.0;
        for (int k = 0; k < 3; ++k) a.gbc[3 * r + k] = 0.0;
        a.gc[r] = 0.0;
        a.gf[r] = 0.0;
      }
    }
    __syncthreads();
  }
}

template <typename T, int P, bool Q>
fei_status launch_bwd(const T *tab, const double *tab64, const BwdArgs &a, int64_t grid_work, cudaStream_t s) {
  using C = AdjCfg<T, P>;
  constexpr int SMEM = (Q ? C::Q_END : C::END) * (int)sizeof(T);
  static_assert(sizeof(AdjElem<T, P>) + 8192 + SMEM <= 232448, "shared memory of one block (227 KB)");
  if (!tab) return set_error(FEI_ERR_UNSUPPORTED, "no sum-factorised tables for degree %d", P);
  FEI_CUDA_TRY(cudaFuncSetAttribute(backward_kernel<T, P, Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM),
               "cudaFuncSetAttribute(backward)");
  // resident blocks of this kernel on the device, asked once per device
  static std::atomic<int> resident[64];
  int dev;
  FEI_CUDA_TRY(cudaGetDevice(&dev), "cudaGetDevice");
  int fit = dev < 64 ? resident[dev].load(std::memory_order_relaxed) : 0;
  if (!fit) {
    int sms, per_sm = 1;
    FEI_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "cudaDeviceGetAttribute");
    FEI_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, backward_kernel<T, P, Q>, C::NTH, SMEM),
                 "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
    fit = sms * (per_sm < 1 ? 1 : per_sm);
    if (dev < 64) resident[dev].store(fit, std::memory_order_relaxed);
  }
  int64_t blocks = grid_work < fit ? grid_work : fit;
  if (blocks < 1) blocks = 1;
  backward_kernel<T, P, Q><<<(unsigned)blocks, C::NTH, SMEM, s>>>(a, tab, tab64);
  FEI_CUDA_TRY(cudaGetLastError(), "backward_kernel launch");
  return FEI_OK;
}

template <typename T, bool Q>
fei_status launch_bwd_typed(int p, const T *tab, const double *tab64, const BwdArgs &a, int64_t grid_work, cudaStream_t s) {
  switch (p) {
    case 1: return launch_bwd<T, 1, Q>(tab, tab64, a, grid_work, s);
    case 2: return launch_bwd<T, 2, Q>(tab, tab64, a, grid_work, s);
    case 3: return launch_bwd<T, 3, Q>(tab, tab64, a, grid_work, s);
    case 4: return launch_bwd<T, 4, Q>(tab, tab64, a, grid_work, s);
    case 5: return launch_bwd<T, 5, Q>(tab, tab64, a, grid_work, s);
    case 6: return launch_bwd<T, 6, Q>(tab, tab64, a, grid_work, s);
    case 7: return launch_bwd<T, 7, Q>(tab, tab64, a, grid_work, s);
  }
  return set_error(FEI_ERR_INVALID_DEGREE, "degree %d outside 1..7", p);
}

}  // namespace

fei_status launch_cc_backward(int p, bool fp64, const fei_reference *ref, const BwdArgs &a, int64_t grid_work,
                              cudaStream_t s, bool quadratic) {
  if (grid_work <= 0) return FEI_OK;
  if (quadratic)
    return fp64 ? launch_bwd_typed<double, true>(p, ref->sf64, ref->sf64, a, grid_work, s)
                : launch_bwd_typed<float, true>(p, ref->sf, ref->sf64, a, grid_work, s);
  return fp64 ? launch_bwd_typed<double, false>(p, ref->sf64, ref->sf64, a, grid_work, s)
              : launch_bwd_typed<float, false>(p, ref->sf, ref->sf64, a, grid_work, s);
}

}  // namespace fei
