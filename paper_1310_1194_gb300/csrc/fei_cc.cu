// fei_cc.cu -- element integration on the CUDA cores: the FP64 and FP32
// paths.  Degrees 2 to 7 run the sum-factorised kernels (fei_sf.cuh) in FP64
// or FP32; this file holds the p = 1 kernels.
//
// Algorithm 1 of the paper at p = 1 (6 shape functions, 8 points): the
// element's geometry is read once (step 2), the point operators Dt_q are
// formed (steps 7-8, fei_geom.cuh), then the double loop over shape
// functions (steps 9-13).
//
// FEI_FP64: everything in FP64.  FEI_FP32: the vertex differences in FP64,
// element vectors, the vertical-node sums of det J and w det J at every point
// in double-FP32 (the first two in FP64 where they cancel, p1_safe), w det J
// rounded once; the adjugate rows, the point operator and the contraction in
// FP32.
#include <type_traits>

#include "fei_geom.cuh"
#include "fei_internal.cuh"

namespace fei {
namespace {

__device__ __forceinline__ int64_t n_items(const FwdArgs &a) {
  return a.count ? (int64_t)(*a.count) : a.n_work;
}

// Loads the 14 coefficient values of record r (K 9, b 3, c, f) and reports
// whether all are finite.
__device__ __forceinline__ bool load_coef(const FwdArgs &a, int64_t r, double *cd) {
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    cd[k] = a.K[9 * r + k];
    ok &= finite64(cd[k]);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    cd[9 + k] = a.b[3 * r + k];
    ok &= finite64(cd[9 + k]);
  }
  cd[12] = a.c[r];
  cd[13] = a.f[r];
  ok &= finite64(cd[12]) && finite64(cd[13]);
  return ok;
}

// Point operator directly from the element vectors, FP64.
__device__ __forceinline__ int point_direct64(const double *ev, const double *pt, const double *cd, double *D) {
  double c1[3], c2[3], n3[3], c3[3];
  znode_columns(ev, pt[2], c1, c2, n3);
  tnode_column(ev, pt[0], pt[1], c3);
  const double w = pt[3];
  const double det = dot3(n3, c3);
  const double s = w * det;
  double a0[3], a1[3];
  cross3(c2, c3, a0);
  cross3(c3, c1, a1);
  dt_from_adj<double>(a0, a1, n3, w, s, w / det, cd, cd + 9, cd[12], cd[13], D);
  return point_status(s);
}

// ---------------------------------------------------------------------------
// FP64: four elements of 8 points per warp, so that every lane takes a point;
// lanes then run over the entries of the A_e.
// ---------------------------------------------------------------------------

// One component (j = vector * 3 + axis) of the element vectors A1, B1, A2,
// B2, C, D1, D2 from the bottom (P) and top (Q) vertices, FP64:
// 0.5 ((X_a - X_b) + s (X_c - X_d)) with the vertices a, b, c, d and the
// sign s of each vector picked by integer selects, so that lanes holding
// different vectors run the same FP64 instructions (a branch per vector
// would run every branch's FP64 work in every lane of the warp).
__device__ __forceinline__ double elem_vec_comp(const double *X, int j) {
  const int v = j / 3, k = j - 3 * v;
  // a | b << 4 | c << 8 | d << 12 | (s + 1) << 16, vertices P0..P2 = 0..2,
  // Q0..Q2 = 3..5: A1 = (P1-P0) + (Q1-Q0), B1 = (Q1-Q0) - (P1-P0),
  // A2 = (P2-P0) + (Q2-Q0), B2 = (Q2-Q0) - (P2-P0), C = Q0-P0,
  // D1 = (Q1-P1) - (Q0-P0), D2 = (Q2-P2) - (Q0-P0), each halved
  const int code = v == 0 ? (1 | 0 << 4 | 4 << 8 | 3 << 12 | 2 << 16)
                   : v == 1 ? (4 | 3 << 4 | 1 << 8 | 0 << 12 | 0 << 16)
                   : v == 2 ? (2 | 0 << 4 | 5 << 8 | 3 << 12 | 2 << 16)
                   : v == 3 ? (5 | 3 << 4 | 2 << 8 | 0 << 12 | 0 << 16)
                   : v == 4 ? (3 | 0 << 4 | 0 << 8 | 0 << 12 | 1 << 16)
                   : v == 5 ? (4 | 1 << 4 | 3 << 8 | 0 << 12 | 0 << 16)
                            : (5 | 2 << 4 | 3 << 8 | 0 << 12 | 0 << 16);
  const double xa = X[3 * (code & 15) + k], xb = X[3 * ((code >> 4) & 15) + k];
  const double xc = X[3 * ((code >> 8) & 15) + k], xd = X[3 * ((code >> 12) & 15) + k];
  const int sg = code >> 16;  // s + 1
  const long long t = __double_as_longlong(xc - xd);
  // s (X_c - X_d) by the sign bit (s = -1) or zero (s = 0): integer work
  const double st = sg == 1 ? 0.0 : __longlong_as_double(sg == 0 ? t ^ (1LL << 63) : t);
  return 0.5 * ((xa - xb) + st);
}

struct SmallCfg {
  static constexpr int P = 1, NSH = nsh_of(P), NQ = nq_of(P), K4 = 4 * NQ, NT = (P + 1) * (P + 1);
  static constexpr int EPW = 32 / NQ;  // elements per warp
  static constexpr int WPB = 4;
  // per element slot: X[18], ev[21], cd[14], D[NQ][16], H[K4][NSH], status
  static constexpr int SLOT_BYTES = (sizeof(double) * (18 + 21 + 14 + NQ * 16 + K4 * NSH) + 16 + 15) / 16 * 16;
  static constexpr int WARP_BYTES = EPW * SLOT_BYTES;
  static constexpr int SMEM = ((sizeof(double) * K4 * NSH + 15) / 16) * 16 + WPB * WARP_BYTES;
};

__global__ void __launch_bounds__(SmallCfg::WPB * 32) cc_small_kernel(FwdArgs a) {
  using C = SmallCfg;
  constexpr int NSH = C::NSH, NQ = C::NQ, K4 = C::K4, EPW = C::EPW, NT = C::NT;
  static_assert(NQ <= 32, "one point per lane");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double *Gs = reinterpret_cast<double *>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char *wb = smem_raw + ((sizeof(double) * K4 * NSH + 15) / 16) * 16 + warp * C::WARP_BYTES;
  auto Xs = [&](int sl) { return reinterpret_cast<double *>(wb + sl * C::SLOT_BYTES); };
  auto evs = [&](int sl) { return Xs(sl) + 18; };
  auto cds = [&](int sl) { return Xs(sl) + 39; };
  auto Ds = [&](int sl) { return Xs(sl) + 53; };
  auto Hs = [&](int sl) { return Ds(sl) + NQ * 16; };
  auto Ss = [&](int sl) { return reinterpret_cast<int *>(Hs(sl) + K4 * NSH); };

  const double *G = a.G64;
  for (int k = threadIdx.x; k < K4 * NSH; k += blockDim.x) Gs[k] = G[k];
  __syncthreads();

  const int64_t items = n_items(a);
  const int64_t nwarps = (int64_t)gridDim.x * C::WPB;
  for (int64_t item0 = ((int64_t)blockIdx.x * C::WPB + warp) * EPW; item0 < items; item0 += nwarps * EPW) {
    const int nel = items - item0 < EPW ? (int)(items - item0) : EPW;
    // geometry and coefficients of the warp's elements, spread over lanes
    for (int idx = lane; idx < nel * 32; idx += 32) {
      const int sl = idx >> 5, k = idx & 31;
      const int64_t e = a.list ? (int64_t)a.list[item0 + sl] : item0 + sl;
      bool ok = true;
      if (k < 18) {
        const double x = a.geom[18 * e + k];
        Xs(sl)[k] = x;
        ok = finite64(x);
      } else if (a.coef_mode == FEI_COEF_PER_ELEMENT) {
        const int c = k - 18;
        const double x = c < 9 ? a.K[9 * e + c] : c < 12 ? a.b[3 * e + (c - 9)] : c == 12 ? a.c[e] : a.f[e];
        cds(sl)[c] = x;
        ok = finite64(x);
      }
      // lanes of one element are one aligned group of 32: the whole warp
      const unsigned bad = __ballot_sync(0xffffffffu, !ok);
      // upper layout: K symmetric (K01 = K10, K02 = K20, K12 = K21: lanes
      // 19/21, 20/24, 23/25) and b = 0 (lanes 27-29), per-element records
      bool sym = true;
      if (a.upper && a.coef_mode == FEI_COEF_PER_ELEMENT) {
        const double xk = k >= 18 ? cds(sl)[k - 18] : 0.0;
        const int c = k - 18;
        const int partner = c == 1 ? 21 : c == 3 ? 19 : c == 2 ? 24 : c == 6 ? 20 : c == 5 ? 25 : c == 7 ? 23 : k;
        const double xp = __shfl_sync(0xffffffffu, xk, partner);
        sym = (c >= 9 && c <= 11) ? xk == 0.0 : xk == xp;
      }
      const unsigned nonsym = __ballot_sync(0xffffffffu, !sym);
      if (k == 0) Ss(sl)[0] = bad ? 2 * FEI_ERR_NONFINITE : (nonsym ? FEI_ERR_INVALID_ARG : 0);
    }
    __syncwarp();
    // element vectors, one component per lane (FP64)
    for (int idx = lane; idx < nel * 21; idx += 32) {
      const int sl = idx / 21, j = idx - sl * 21;
      const double v = elem_vec_comp(Xs(sl), j);
      evs(sl)[j] = v;
    }
    __syncwarp();
    // point operators: lane = (element slot, point)
    const int psl = lane / NQ, q = lane - psl * NQ;
    int pst = 0;
    if (psl < nel) {
      const int64_t e = a.list ? (int64_t)a.list[item0 + psl] : item0 + psl;
      // quadrature point from the node tables: q = iz*(p+1)^2 + t
      const int iz = q / NT, t = q % NT;
      double cq[14];
      if (a.coef_mode == FEI_COEF_PER_POINT) {
        const int64_t r = (a.q_off ? a.q_off[e] : e * (int64_t)NQ) + q;
        if (!load_coef(a, r, cq)) pst = FEI_ERR_NONFINITE;
        else if (a.upper && !coef_symmetric(cq, cq + 9)) pst = FEI_ERR_INVALID_ARG;
      }
      const double ptv[4] = {a.tnode[4 * t], a.tnode[4 * t + 1], a.znode[2 * iz],
                             a.tnode[4 * t + 2] * a.znode[2 * iz + 1]};
      const bool perq = a.coef_mode == FEI_COEF_PER_POINT;
      pst = merge_status(pst, point_direct64(evs(psl), ptv, perq ? cq : cds(psl), Ds(psl) + 16 * q));
      if (pst) atomicMax(Ss(psl), pst == FEI_ERR_NONFINITE ? 2 * FEI_ERR_NONFINITE : pst);
    }
    __syncwarp();
    // H[(q, b)][i] = sum_a Dt_q[a][b] G[q][a][i], per element
    for (int idx = lane; idx < nel * NQ * NSH; idx += 32) {
      const int sl = idx / (NQ * NSH), rem = idx - sl * (NQ * NSH);
      const int qq = rem / NSH, i = rem - qq * NSH;
      const double *Dq = Ds(sl) + 16 * qq;
      double *H = Hs(sl);
      const double g0 = Gs[(4 * qq + 0) * NSH + i], g1 = Gs[(4 * qq + 1) * NSH + i];
      const double g2 = Gs[(4 * qq + 2) * NSH + i], g3 = Gs[(4 * qq + 3) * NSH + i];
      H[(4 * qq + 0) * NSH + i] = Dq[0] * g0;
#pragma unroll
      for (int m = 0; m < 3; ++m)
        H[(4 * qq + 1 + m) * NSH + i] = Dq[1 + m] * g0 + Dq[4 + m] * g1 + Dq[7 + m] * g2 + Dq[10 + m] * g3;
    }
    __syncwarp();
    // A_e = H^T G and b_e, lanes over (element, entry)
    for (int idx = lane; idx < nel * NSH * NSH; idx += 32) {
      const int sl = idx / (NSH * NSH), ij = idx - sl * (NSH * NSH);
      const int i = ij / NSH, j = ij - i * NSH;
      const int64_t e = a.list ? (int64_t)a.list[item0 + sl] : item0 + sl;
      const int64_t aoff = out_a(a, item0 + sl, e, NSH);
      if (a.upper && j < i) continue;  // the upper layout keeps j >= i
      const double *H = Hs(sl);
      double acc = 0.0;
#pragma unroll 4
      for (int k = 0; k < K4; ++k) acc += H[k * NSH + i] * Gs[k * NSH + j];
      reinterpret_cast<double *>(a.A)[aoff + a_pos(i, j, NSH, a.upper)] = Ss(sl)[0] ? 0.0 : acc;
    }
    for (int idx = lane; idx < nel * NSH; idx += 32) {
      const int sl = idx / NSH, i = idx - sl * NSH;
      const int64_t e = a.list ? (int64_t)a.list[item0 + sl] : item0 + sl;
      const int64_t boff = out_b(a, item0 + sl, e, NSH);
      const double *D = Ds(sl);
      double acc = 0.0;
      for (int qq = 0; qq < NQ; ++qq) acc += D[16 * qq + 13] * Gs[(4 * qq) * NSH + i];
      reinterpret_cast<double *>(a.bv)[boff + i] = Ss(sl)[0] ? 0.0 : acc;
    }
    for (int sl = lane; sl < nel; sl += 32) {
      const int64_t e = a.list ? (int64_t)a.list[item0 + sl] : item0 + sl;
      const int v = Ss(sl)[0];
      // NONFINITE is recorded as 2 * NONFINITE so that it wins the max
      a.status[e] = v == 2 * FEI_ERR_NONFINITE ? FEI_ERR_NONFINITE : v;
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// p = 1, FP32 path: one thread per element.  A p = 1 element is small (6
// shape functions, 8 points, 36 entries), so a thread keeps A_e and b_e in
// registers and runs the points in turn.  Records and results pass through
// shared memory, so that consecutive threads touch consecutive addresses (a
// thread's own record or matrix is a line of its own in every load and
// store).  1 000 000 prisms (GB300): 0.277 ms, 1.53 TB/s of inputs and
// outputs; with FP64 node sums and per-thread loads and stores 0.467 ms.  It
// is bound by issue (55 % of slots with the 12 warps an SM that the
// registers allow); more blocks per SM spill (4: 0.30, 5: 0.38 ms).
// ---------------------------------------------------------------------------
constexpr int kP1Threads = 128;

// The two p = 1 kernels below (one thread per element for large batches,
// eight lanes per element for small ones) give the same bits: their
// node sums and their sums over points run in one fixed order of
// rounded operations (the host-memory entry cuts a batch into chunks of
// any size and must equal the device entry bit for bit).
//
// FP64 node sums (p1_setup64): n3_k and its products p_k rounded one by one,
// value v summed as (p_v + p_v+1) + p_v+2.
__device__ __forceinline__ double p1_node_sum(const double *n3, const double *w, int v) {
  const double a = __dmul_rn(n3[v], w[v]), b = __dmul_rn(n3[(v + 1) % 3], w[(v + 1) % 3]);
  const double c = __dmul_rn(n3[(v + 2) % 3], w[(v + 2) % 3]);
  return __dadd_rn(__dadd_rn(a, b), c);
}
__device__ __forceinline__ double p1_cross_comp(double a1, double a2, double b1, double b2) {
  return __dsub_rn(__dmul_rn(a1, b2), __dmul_rn(a2, b1));  // a1 b2 - a2 b1
}
// The gradient components of p = 1 function i = 3 k + t that are not zero
// everywhere, as bits (1: d/dxi1, 2: d/dxi2, 4: d/dzeta): t = (0,0), (1,0),
// (0,1) with L_0 constant and L_1 linear in zeta.
__host__ __device__ constexpr int p1_grad(int i) { return (i % 3 == 1 ? 3 : i % 3 == 2 ? 2 : 0) | (i >= 3 ? 4 : 0); }
// One point's contribution to A_e (36 values, row-major) and b_e (6):
// G_q^T Dt_q G_q and (w det J f) G_q0, every operation rounded in turn, the
// zero components left out (15 of 24 values remain).
__device__ __forceinline__ void p1_point_contrib(const float *D, const float *G, float *c) {
  constexpr int NSH = 6;
#pragma unroll
  for (int i = 0; i < NSH; ++i) {
    const float g0 = G[i];
    const float h0 = __fmul_rn(D[0], g0);
    float h1 = __fmul_rn(D[1], g0), h2 = __fmul_rn(D[2], g0), h3 = __fmul_rn(D[3], g0);
    if (p1_grad(i) & 1) {
      const float g = G[NSH + i];
      h1 = __fmaf_rn(D[4], g, h1), h2 = __fmaf_rn(D[5], g, h2), h3 = __fmaf_rn(D[6], g, h3);
    }
    if (p1_grad(i) & 2) {
      const float g = G[2 * NSH + i];
      h1 = __fmaf_rn(D[7], g, h1), h2 = __fmaf_rn(D[8], g, h2), h3 = __fmaf_rn(D[9], g, h3);
    }
    if (p1_grad(i) & 4) {
      const float g = G[3 * NSH + i];
      h1 = __fmaf_rn(D[10], g, h1), h2 = __fmaf_rn(D[11], g, h2), h3 = __fmaf_rn(D[12], g, h3);
    }
#pragma unroll
    for (int j = 0; j < NSH; ++j) {
      float v = __fmul_rn(h0, G[j]);
      if (p1_grad(j) & 1) v = __fmaf_rn(h1, G[NSH + j], v);
      if (p1_grad(j) & 2) v = __fmaf_rn(h2, G[2 * NSH + j], v);
      if (p1_grad(j) & 4) v = __fmaf_rn(h3, G[3 * NSH + j], v);
      c[i * NSH + j] = v;
    }
    c[NSH * NSH + i] = __fmul_rn(D[13], g0);
  }
}

// Element setup.  The vertex differences are FP64 subtractions, split from
// their bit fields into FP32 pairs; everything after them is double-FP32
// arithmetic in operations that are rounded one by one (no contraction), so
// that both kernels give the same bits: 21 FP64 instructions an element
// instead of about 190 (this part's FP64 rate bound the kernel), at an error
// of about 2^-44 before the single rounding of w det J where nothing cancels;
// the others take FP64 (p1_safe: 1 000 000 prisms 270 -> 274 us).
__device__ __forceinline__ float2 p1_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  float e = __fmaf_rn(a.x, b.x, -p);
  e = __fmaf_rn(a.x, b.y, e);
  e = __fmaf_rn(a.y, b.x, e);
  return make_float2(p, e);
}
__device__ __forceinline__ float2 p1_add(float2 a, float2 b) {
  const float s = __fadd_rn(a.x, b.x), bb = __fadd_rn(s, -a.x);
  const float err = __fadd_rn(__fadd_rn(a.x, -__fadd_rn(s, -bb)), __fadd_rn(b.x, -bb));
  return make_float2(s, __fadd_rn(__fadd_rn(err, a.y), b.y));
}
__device__ __forceinline__ float2 p1_norm(float2 a) {
  const float s = __fadd_rn(a.x, a.y), bb = __fadd_rn(s, -a.x);
  return make_float2(s, __fadd_rn(__fadd_rn(a.x, -__fadd_rn(s, -bb)), __fadd_rn(a.y, -bb)));
}
// half of t1 + t2
__device__ __forceinline__ float2 p1_half_sum(float2 t1, float2 t2) {
  const float2 v = p1_norm(p1_add(t1, t2));
  return make_float2(__fmul_rn(0.5f, v.x), __fmul_rn(0.5f, v.y));
}
// Component j = 3 v + axis of the element vectors A1, B1, A2, B2, C, D1, D2 as
// a pair (the vertices and signs of elem_vec_comp); clears *in_range where a
// difference is outside the pairs' range.
__device__ __forceinline__ float2 elem_vec_pair(const double *X, int j, bool *in_range) {
  const int v = j / 3, k = j - 3 * v;
  const int code = v == 0 ? (1 | 0 << 4 | 4 << 8 | 3 << 12 | 2 << 16)
                   : v == 1 ? (4 | 3 << 4 | 1 << 8 | 0 << 12 | 0 << 16)
                   : v == 2 ? (2 | 0 << 4 | 5 << 8 | 3 << 12 | 2 << 16)
                   : v == 3 ? (5 | 3 << 4 | 2 << 8 | 0 << 12 | 0 << 16)
                   : v == 4 ? (3 | 0 << 4 | 0 << 8 | 0 << 12 | 1 << 16)
                   : v == 5 ? (4 | 1 << 4 | 3 << 8 | 0 << 12 | 0 << 16)
                            : (5 | 2 << 4 | 3 << 8 | 0 << 12 | 0 << 16);
  const double d1 = X[3 * (code & 15) + k] - X[3 * ((code >> 4) & 15) + k];
  const double d2 = X[3 * ((code >> 8) & 15) + k] - X[3 * ((code >> 12) & 15) + k];
  bool r1, r2;
  const float2 t1 = split_f64_bits(d1, &r1), t2 = split_f64_bits(d2, &r2);
  *in_range &= r1 && r2;
  return p1_half_sum(t1, code >> 16 == 0 ? neg_ff(t2) : t2);
}
// component z B + A of a column
__device__ __forceinline__ float2 p1_column(float2 z, float2 A, float2 B) { return p1_norm(p1_add(A, p1_mul(z, B))); }
// a1 b2 - a2 b1
__device__ __forceinline__ float2 p1_cross_pair(float2 a1, float2 a2, float2 b1, float2 b2) {
  return p1_norm(p1_add(p1_mul(a1, b2), neg_ff(p1_mul(a2, b1))));
}
// (p_v + p_v+1) + p_v+2
__device__ __forceinline__ float2 p1_sum3(float2 a, float2 b, float2 c) { return p1_norm(p1_add(p1_add(a, b), c)); }

// Whether the pairs' det J is safe at every point.  The pairs lose what the
// differences of products in n3 and the sums n3.C, n3.D1, n3.D2 cancel (their
// error is about 2^-42 of q = sum_k (|c1||c2| terms of n3_k) (|C_k| + |D1_k| +
// |D2_k|) bounds, which cancel nothing): an element whose det J is not above
// 2^-14 q at the corners of both node triangles (the points are inside), thin,
// flat, collapsed or mirrored, or near the ends of the FP32 range, takes the
// FP64 setup, where n3 of a collapsed triangle is 0.  Rounded operations only,
// in one order: both p = 1 kernels decide alike.
__device__ __forceinline__ float p1_gate(const float *ev) {
  float m1[3], m2[3], md[3], q = 0.f;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    m1[k] = __fadd_rn(fabsf(ev[k]), fabsf(ev[3 + k]));
    m2[k] = __fadd_rn(fabsf(ev[6 + k]), fabsf(ev[9 + k]));
    // |v0|, |v1|, |v2| / 2 in terms of C, D1, D2
    md[k] = __fadd_rn(__fmaf_rn(5.f, fabsf(ev[12 + k]), fabsf(ev[15 + k])), fabsf(ev[18 + k]));
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int i = (k + 1) % 3, j = (k + 2) % 3;
    q = __fmaf_rn(__fmaf_rn(m1[i], m2[j], __fmul_rn(m1[j], m2[i])), md[k], q);
  }
  return __fmul_rn(6.103515625e-5f, q);  // 2^-14 q
}
// one vertical node: (a, b, g) = w_z (n3.C, n3.D1, n3.D2)
__device__ __forceinline__ bool p1_safe(const float2 *zab, float wz, float gate) {
  const float a = zab[0].x, b = zab[1].x, g = zab[2].x;
  const float lo = fminf(a, fminf(__fadd_rn(a, b), __fadd_rn(a, g)));
  return lo > __fmul_rn(wz, gate) && lo > 1e-28f && gate < 1e28f;
}

// The same setup in FP64, for an element that p1_safe refuses or with a vertex
// difference outside 2^-60 <= |d| < 2^60 (other than 0): ev32 [21], then the
// node sums [2][3] as pairs (12 values).  Not inlined: the compiler would
// execute its FP64 instructions ahead of the branch.
__device__ __noinline__ void p1_setup64(const double *X, const double *zd, const double *zwd, float *out) {
  double ev[21];
  elem_vectors(X, ev);
#pragma unroll
  for (int k = 0; k < 21; ++k) out[k] = (float)ev[k];
#pragma unroll
  for (int iz = 0; iz < 2; ++iz) {
    double c1[3], c2[3], n3[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      c1[k] = fma(zd[iz], ev[3 + k], ev[k]);
      c2[k] = fma(zd[iz], ev[9 + k], ev[6 + k]);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
      n3[k] = p1_cross_comp(c1[(k + 1) % 3], c1[(k + 2) % 3], c2[(k + 1) % 3], c2[(k + 2) % 3]);
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      const float2 z = split_f64(__dmul_rn(zwd[iz], p1_node_sum(n3, ev + 12 + 3 * v, v)));
      out[21 + 6 * iz + 2 * v] = z.x;
      out[22 + 6 * iz + 2 * v] = z.y;
    }
  }
}

__global__ void __launch_bounds__(kP1Threads, 3) cc_p1_kernel(FwdArgs a) {
  constexpr int NSH = 6, NQ = 8, M = 2, NT = 4;
  constexpr int IN = 33, OUT = 43;  // odd strides: a column of the tile in distinct banks
  // a tile's records (18 vertex coordinates, 14 coefficients), then its outputs
  __shared__ __align__(16) double tile[kP1Threads * IN];
  __shared__ int32_t eid[kP1Threads];
  float *outs = reinterpret_cast<float *>(tile);
  __shared__ float Gs[4 * NQ * NSH];  // G32 [q][a][i]
  __shared__ float2 ttab[NT][3];      // w_t, w_t xi1, w_t xi2 as FP32 pairs
  __shared__ float ttabf[NT][3];      // w_t, xi1, xi2
  __shared__ float zf[M], zwf[M];
  __shared__ double zd[M], zwd[M];
  __shared__ float2 zp[M], zwp[M];
  for (int k = threadIdx.x; k < 4 * NQ * NSH; k += blockDim.x) Gs[k] = a.G32[k];
  if (threadIdx.x < NT) {
    const int t = threadIdx.x;
    const double x1 = a.tnode[4 * t], x2 = a.tnode[4 * t + 1], wt = a.tnode[4 * t + 2];
    ttab[t][0] = split_f64(wt);
    ttab[t][1] = split_f64(wt * x1);
    ttab[t][2] = split_f64(wt * x2);
    ttabf[t][0] = (float)wt;
    ttabf[t][1] = (float)x1;
    ttabf[t][2] = (float)x2;
  } else if (threadIdx.x >= 32 && threadIdx.x < 32 + M) {
    const int iz = threadIdx.x - 32;
    zd[iz] = a.znode[2 * iz];
    zwd[iz] = a.znode[2 * iz + 1];
    zf[iz] = (float)zd[iz];
    zwf[iz] = (float)zwd[iz];
    zp[iz] = split_f64(zd[iz]);
    zwp[iz] = split_f64(zwd[iz]);
  }
  const int64_t items = n_items(a);
  const int tid = threadIdx.x;
  const bool perq = a.coef_mode == FEI_COEF_PER_POINT;
  const bool flat = !a.A_off && !a.b_off && !a.list && !a.upper && ((uintptr_t)a.A & 15) == 0 && ((uintptr_t)a.bv & 7) == 0;
  for (int64_t base = blockIdx.x * (int64_t)kP1Threads; base < items; base += (int64_t)gridDim.x * kP1Threads) {
    const int nt = items - base < kP1Threads ? (int)(items - base) : kP1Threads;
    // the tile's records by consecutive threads (one thread per element would
    // touch a line per lane and load)
    if (tid < nt) eid[tid] = a.list ? a.list[base + tid] : (int32_t)(base + tid);
    __syncthreads();
    // (all loads of a tile in flight before the first store)
    double in_reg[32];
    auto gather = [&](const double *src, auto width, int at) {
      constexpr int W = decltype(width)::value;
#pragma unroll
      for (int j = 0; j < W; ++j) {
        const int i = tid + j * kP1Threads, el = i / W, k = i - el * W;
        in_reg[at + j] = i < nt * W ? src[(int64_t)eid[el] * W + k] : 0.0;
      }
    };
    auto spread = [&](auto width, int at) {
      constexpr int W = decltype(width)::value;
#pragma unroll
      for (int j = 0; j < W; ++j) {
        const int i = tid + j * kP1Threads, el = i / W, k = i - el * W;
        tile[el * IN + at + k] = in_reg[at + j];
      }
    };
    using W18 = std::integral_constant<int, 18>;
    using W9 = std::integral_constant<int, 9>;
    using W3 = std::integral_constant<int, 3>;
    using W1 = std::integral_constant<int, 1>;
    gather(a.geom, W18{}, 0);
    if (!perq) {
      gather(a.K, W9{}, 18);
      gather(a.b, W3{}, 27);
      gather(a.c, W1{}, 30);
      gather(a.f, W1{}, 31);
    }
    spread(W18{}, 0);
    if (!perq) {
      spread(W9{}, 18);
      spread(W3{}, 27);
      spread(W1{}, 30);
      spread(W1{}, 31);
    }
    __syncthreads();
    // threads past the tile compute on its first record and store nothing
    const int slot = tid < nt ? tid : 0;
    const int64_t e = eid[slot];
    const double *in = tile + slot * IN;
    bool ok = true, sym = true;
    float ev32[21];   // element vectors rounded once
    float2 zab[M][3];  // per vertical node w_z (n3.C, n3.D1, n3.D2), FP32 pairs
    {
      double X[18];
#pragma unroll
      for (int k = 0; k < 18; ++k) {
        X[k] = in[k];
        ok &= finite64(X[k]);
      }
      bool in_range = true;
      float2 ev[21];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        auto diff = [&](int i, int j) {
          bool r;
          const float2 d = split_f64_bits(X[3 * i + k] - X[3 * j + k], &r);
          in_range &= r;
          return d;
        };
        const float2 e1p = diff(1, 0), e1q = diff(4, 3), e2p = diff(2, 0), e2q = diff(5, 3);
        const float2 v0 = diff(3, 0), v1 = diff(4, 1), v2 = diff(5, 2);
        ev[0 + k] = p1_half_sum(e1p, e1q);
        ev[3 + k] = p1_half_sum(e1q, neg_ff(e1p));
        ev[6 + k] = p1_half_sum(e2p, e2q);
        ev[9 + k] = p1_half_sum(e2q, neg_ff(e2p));
        ev[12 + k] = p1_half_sum(v0, make_float2(0.f, 0.f));
        ev[15 + k] = p1_half_sum(v1, neg_ff(v0));
        ev[18 + k] = p1_half_sum(v2, neg_ff(v0));
      }
#pragma unroll
      for (int k = 0; k < 21; ++k) ev32[k] = ev[k].x;
#pragma unroll
      for (int iz = 0; iz < M; ++iz) {
        float2 c1[3], c2[3], n3[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          c1[k] = p1_column(zp[iz], ev[k], ev[3 + k]);
          c2[k] = p1_column(zp[iz], ev[6 + k], ev[9 + k]);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k)
          n3[k] = p1_cross_pair(c1[(k + 1) % 3], c1[(k + 2) % 3], c2[(k + 1) % 3], c2[(k + 2) % 3]);
#pragma unroll
        for (int v = 0; v < 3; ++v) {
          float2 p[3];
#pragma unroll
          for (int k = 0; k < 3; ++k) p[k] = p1_mul(n3[k], ev[12 + 3 * v + k]);
          zab[iz][v] = p1_norm(p1_mul(zwp[iz], p1_sum3(p[v], p[(v + 1) % 3], p[(v + 2) % 3])));
        }
      }
      const float gate = p1_gate(ev32);
#pragma unroll
      for (int iz = 0; iz < M; ++iz) in_range &= p1_safe(zab[iz], zwf[iz], gate);
      if (!in_range) {
        float t[33];
        p1_setup64(in, zd, zwd, t);
#pragma unroll
        for (int k = 0; k < 21; ++k) ev32[k] = t[k];
#pragma unroll
        for (int j = 0; j < 6; ++j) zab[j / 3][j % 3] = make_float2(t[21 + 2 * j], t[22 + 2 * j]);
      }
    }
    // FP32 columns c1, c2 and n3 per vertical node
    float zc[M][9];
#pragma unroll
    for (int iz = 0; iz < M; ++iz) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        zc[iz][k] = fmaf(zf[iz], ev32[3 + k], ev32[k]);
        zc[iz][3 + k] = fmaf(zf[iz], ev32[9 + k], ev32[6 + k]);
      }
      cross3(zc[iz], zc[iz] + 3, zc[iz] + 6);
    }
    float cf[14];
    if (!perq) {
      double cd[14];
#pragma unroll
      for (int k = 0; k < 14; ++k) cd[k] = in[18 + k];
      sym = !a.upper || coef_symmetric(cd, cd + 9);
      ok &= coef_to_f32<14>(cd, cf);
    }
    int st = !ok ? FEI_ERR_NONFINITE : (!sym ? FEI_ERR_INVALID_ARG : 0);
    float A[NSH][NSH], bv[NSH];
#pragma unroll
    for (int i = 0; i < NSH; ++i) {
      bv[i] = 0.f;
#pragma unroll
      for (int j = 0; j < NSH; ++j) A[i][j] = 0.f;
    }
#pragma unroll
    for (int iz = 0; iz < M; ++iz)
#pragma unroll 1
    for (int t = 0; t < NT; ++t) {
      const int q = iz * NT + t;
      if (perq) {
        double cd[14];
        const int64_t r = (a.q_off ? a.q_off[e] : e * (int64_t)NQ) + q;
        int pst = 0;
        if (!load_coef(a, r, cd)) pst = FEI_ERR_NONFINITE;
        else if (a.upper && !coef_symmetric(cd, cd + 9)) pst = FEI_ERR_INVALID_ARG;
        st = merge_status(st, pst);
#pragma unroll
        for (int k = 0; k < 14; ++k) cf[k] = (float)cd[k];
      }
      // w det J in double-FP32, rounded once
      const float2 sd = add_ff(add_ff(mul_ff(ttab[t][0], zab[iz][0]), mul_ff(ttab[t][1], zab[iz][1])),
                               mul_ff(ttab[t][2], zab[iz][2]));
      const float sf = sd.x + sd.y;
      st = merge_status(st, !(fabsf(sf) <= 3.402823466e38f) ? FEI_ERR_NONFINITE
                            : !(sf > 0.f)                    ? FEI_ERR_NEGATIVE_JACOBIAN
                                                             : 0);
      float c3[3], a0[3], a1[3], D[16];
#pragma unroll
      for (int k = 0; k < 3; ++k)
        c3[k] = fmaf(ttabf[t][2], ev32[18 + k], fmaf(ttabf[t][1], ev32[15 + k], ev32[12 + k]));
      cross3(zc[iz] + 3, c3, a0);
      cross3(c3, zc[iz], a1);
      const float wf = ttabf[t][0] * zwf[iz];
      dt_from_adj<float>(a0, a1, zc[iz] + 6, wf, sf, wf * wf / sf, cf, cf + 9, cf[12], cf[13], D);
      // A_e += G_q^T Dt_q G_q, b_e += (w det J f) G_q0
      float c[NSH * NSH + NSH];
      p1_point_contrib(D, Gs + q * 4 * NSH, c);
#pragma unroll
      for (int i = 0; i < NSH; ++i) {
#pragma unroll
        for (int j = 0; j < NSH; ++j) A[i][j] = __fadd_rn(A[i][j], c[i * NSH + j]);
        bv[i] = __fadd_rn(bv[i], c[NSH * NSH + i]);
      }
    }
    // the tile's outputs by consecutive threads, as 16-byte values where the
    // tile's matrices are one aligned range
    if (tid < nt) a.status[e] = st;
    __syncthreads();
    if (flat) {
      float4 *o4 = reinterpret_cast<float4 *>(tile);
      float2 *o2 = reinterpret_cast<float2 *>(o4 + kP1Threads * 9);
#pragma unroll
      for (int v = 0; v < 9; ++v) {
        const float *r = &A[0][0] + 4 * v;
        o4[tid * 9 + v] = st ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(r[0], r[1], r[2], r[3]);
      }
#pragma unroll
      for (int v = 0; v < 3; ++v) o2[tid * 3 + v] = st ? make_float2(0.f, 0.f) : make_float2(bv[2 * v], bv[2 * v + 1]);
      __syncthreads();
      float4 *A4 = reinterpret_cast<float4 *>(reinterpret_cast<float *>(a.A) + base * 36);
      float2 *b2 = reinterpret_cast<float2 *>(reinterpret_cast<float *>(a.bv) + base * 6);
#pragma unroll
      for (int v = 0; v < 9; ++v)
        if (tid + v * kP1Threads < nt * 9) A4[tid + v * kP1Threads] = o4[tid + v * kP1Threads];
#pragma unroll
      for (int v = 0; v < 3; ++v)
        if (tid + v * kP1Threads < nt * 3) b2[tid + v * kP1Threads] = o2[tid + v * kP1Threads];
    } else {
#pragma unroll
      for (int i = 0; i < NSH; ++i) {
#pragma unroll
        for (int j = 0; j < NSH; ++j) outs[tid * OUT + i * NSH + j] = st ? 0.f : A[i][j];
        outs[tid * OUT + NSH * NSH + i] = st ? 0.f : bv[i];
      }
      __syncthreads();
      for (int i = tid; i < nt * 36; i += kP1Threads) {
        const int el = i / 36, k = i - el * 36, r = k / NSH, c = k - r * NSH;
        if (!a.upper || c >= r)
          reinterpret_cast<float *>(a.A)[out_a(a, base + el, eid[el], NSH) + a_pos(r, c, NSH, a.upper)] = outs[el * OUT + k];
      }
      for (int i = tid; i < nt * 6; i += kP1Threads) {
        const int el = i / 6, k = i - el * 6;
        reinterpret_cast<float *>(a.bv)[out_b(a, base + el, eid[el], NSH) + k] = outs[el * OUT + 36 + k];
      }
    }
    __syncthreads();
  }
}

// p = 1, FP32 path, small batches: eight lanes per element (one per
// point), so that a batch that fills only part of the GPU (4096 prisms:
// 32 blocks of the kernel above) is not bound by one thread walking its
// eight points in turn.  The setup is spread over the lanes (three
// element-vector components per lane, three lanes per vertical node for
// the node sums), each lane forms its point's contribution to A_e and b_e
// in registers, and a butterfly over the eight lanes adds them up.
__global__ void __launch_bounds__(kP1Threads) cc_p1_small_kernel(FwdArgs a) {
  constexpr int NSH = 6, NQ = 8, M = 2, NT = 4;
  __shared__ float Gs[4 * NQ * NSH];  // G32 [q][a][i]
  __shared__ float2 ttab[NT][3];
  __shared__ float ttabf[NT][3];
  __shared__ float zf[M], zwf[M];
  __shared__ double zd[M], zwd[M];
  __shared__ float2 zp[M], zwp[M];
  for (int k = threadIdx.x; k < 4 * NQ * NSH; k += blockDim.x) Gs[k] = a.G32[k];
  if (threadIdx.x < NT) {
    const int t = threadIdx.x;
    const double x1 = a.tnode[4 * t], x2 = a.tnode[4 * t + 1], wt = a.tnode[4 * t + 2];
    ttab[t][0] = split_f64(wt);
    ttab[t][1] = split_f64(wt * x1);
    ttab[t][2] = split_f64(wt * x2);
    ttabf[t][0] = (float)wt;
    ttabf[t][1] = (float)x1;
    ttabf[t][2] = (float)x2;
  } else if (threadIdx.x >= 32 && threadIdx.x < 32 + M) {
    const int iz = threadIdx.x - 32;
    zd[iz] = a.znode[2 * iz];
    zwd[iz] = a.znode[2 * iz + 1];
    zf[iz] = (float)zd[iz];
    zwf[iz] = (float)zwd[iz];
    zp[iz] = split_f64(zd[iz]);
    zwp[iz] = split_f64(zwd[iz]);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, g = lane & 7, gbase = lane & 24;
  const int64_t items = n_items(a);
  const int64_t groups = (int64_t)gridDim.x * (blockDim.x / 8);
  // every lane of the warp runs every iteration (the shuffles need the
  // whole warp); a group past the end computes on a clamped element and
  // stores nothing
  const int64_t first = (int64_t)blockIdx.x * (blockDim.x / 8) + (threadIdx.x >> 3);
  const int64_t warp_first = first - (lane >> 3);
  for (int64_t it0 = warp_first; it0 < items; it0 += groups) {
    const int64_t item = it0 + (lane >> 3);
    const bool live = item < items;
    const int64_t e = live ? (a.list ? (int64_t)a.list[item] : item) : (a.list ? (int64_t)a.list[0] : 0);
    // vertices: lane g checks coordinates g, g + 8, g + 16 (the group's AND
    // below); the element-vector components g, g + 8, g + 16 read theirs
    // from global memory (the group's 144 bytes, cached), in FP64
    const double *X = a.geom + 18 * e;
    bool ok = finite64(X[g]) && finite64(X[g + 8]) && (g >= 2 || finite64(X[g + 16]));
    float2 evm[3];
    bool in_range = true;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int j = g + 8 * r;
      evm[r] = elem_vec_pair(X, j < 21 ? j : 20, &in_range);
    }
    auto ev2 = [&](int j) {
      return make_float2(__shfl_sync(0xffffffffu, evm[j / 8].x, gbase + (j & 7)),
                         __shfl_sync(0xffffffffu, evm[j / 8].y, gbase + (j & 7)));
    };
    float2 ev[21];
    float ev32[21];
#pragma unroll
    for (int j = 0; j < 21; ++j) {
      ev[j] = ev2(j);
      ev32[j] = ev[j].x;
    }
    // node sums: lanes 0..5 of the group, three per vertical node
    float2 zab[M][3];
    {
      const int iz = g < 3 ? 0 : 1, k = g < 6 ? g - 3 * iz : 0;
      const int l1 = gbase + 3 * iz + (k + 1) % 3, l2 = gbase + 3 * iz + (k + 2) % 3;
      auto shfl2 = [](float2 v, int src) {
        return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
      };
      // component k of a vector
      auto comp = [&](int v) { return k == 0 ? ev[3 * v] : k == 1 ? ev[3 * v + 1] : ev[3 * v + 2]; };
      const float2 z = zp[iz], wz = zwp[iz];
      const float2 c1 = p1_column(z, comp(0), comp(1)), c2 = p1_column(z, comp(2), comp(3));
      const float2 c1a = shfl2(c1, l1), c1b = shfl2(c1, l2), c2a = shfl2(c2, l1), c2b = shfl2(c2, l2);
      const float2 n3 = p1_cross_pair(c1a, c1b, c2a, c2b);
      // lane k of the node keeps value k, summed as (p_k + p_k+1) + p_k+2
      float2 sum[3];
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        const float2 p = p1_mul(n3, comp(4 + v)), pa = shfl2(p, l1), pb = shfl2(p, l2);
        sum[v] = p1_sum3(p, pa, pb);
      }
      const float2 mine = p1_norm(p1_mul(wz, k == 0 ? sum[0] : k == 1 ? sum[1] : sum[2]));
#pragma unroll
      for (int n = 0; n < M; ++n)
#pragma unroll
        for (int v = 0; v < 3; ++v) zab[n][v] = shfl2(mine, gbase + 3 * n + v);
    }
#pragma unroll
    for (int off = 4; off >= 1; off >>= 1) in_range &= __shfl_xor_sync(0xffffffffu, (int)in_range, off) != 0;
    // (the same in every lane of the group)
    const float gate = p1_gate(ev32);
#pragma unroll
    for (int n = 0; n < M; ++n) in_range &= p1_safe(zab[n], zwf[n], gate);
    if (!in_range) {
      float t[33];
      p1_setup64(X, zd, zwd, t);
#pragma unroll
      for (int k = 0; k < 21; ++k) ev32[k] = t[k];
#pragma unroll
      for (int j = 0; j < 6; ++j) zab[j / 3][j % 3] = make_float2(t[21 + 2 * j], t[22 + 2 * j]);
    }
    // coefficients: components g and g + 8 per lane, shared in FP32
    float cf[14];
    const bool perq = a.coef_mode == FEI_COEF_PER_POINT;
    bool sym = true;
    if (!perq) {
      float cm[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int c = g + 8 * r;
        double x = 0.0;
        if (c < 14) x = c < 9 ? a.K[9 * e + c] : c < 12 ? a.b[3 * e + c - 9] : c == 12 ? a.c[e] : a.f[e];
        ok &= finite64(x);
        cm[r] = (float)x;
      }
#pragma unroll
      for (int c = 0; c < 14; ++c) cf[c] = __shfl_sync(0xffffffffu, cm[c / 8], gbase + (c & 7));
      if (a.upper) {
        // K symmetric and b = 0, compared in FP64 (as the other kernels)
        const double k01 = a.K[9 * e + 1], k10 = a.K[9 * e + 3], k02 = a.K[9 * e + 2], k20 = a.K[9 * e + 6];
        const double k12 = a.K[9 * e + 5], k21 = a.K[9 * e + 7];
        sym = k01 == k10 && k02 == k20 && k12 == k21 && a.b[3 * e] == 0.0 && a.b[3 * e + 1] == 0.0 &&
              a.b[3 * e + 2] == 0.0;
      }
    }
    // the point of this lane
    const int q = g, iz = q / NT, t = q - iz * NT;
    int st = 0;
    if (perq) {
      double cd[14];
      const int64_t r = (a.q_off ? a.q_off[e] : e * (int64_t)NQ) + q;
      if (!load_coef(a, r, cd)) st = FEI_ERR_NONFINITE;
      else if (a.upper && !coef_symmetric(cd, cd + 9)) st = FEI_ERR_INVALID_ARG;
#pragma unroll
      for (int k = 0; k < 14; ++k) cf[k] = (float)cd[k];
    }
    const float2 *zq = iz ? zab[1] : zab[0];
    const float2 sd = add_ff(add_ff(mul_ff(ttab[t][0], zq[0]), mul_ff(ttab[t][1], zq[1])), mul_ff(ttab[t][2], zq[2]));
    const float sf = sd.x + sd.y;
    st = merge_status(st, !(fabsf(sf) <= 3.402823466e38f) ? FEI_ERR_NONFINITE
                          : !(sf > 0.f)                    ? FEI_ERR_NEGATIVE_JACOBIAN
                                                           : 0);
    float zc[9];
    {
      const float zz = zf[iz];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        zc[k] = fmaf(zz, ev32[3 + k], ev32[k]);
        zc[3 + k] = fmaf(zz, ev32[9 + k], ev32[6 + k]);
      }
      cross3(zc, zc + 3, zc + 6);
    }
    float c3[3], a0[3], a1[3], D[16];
#pragma unroll
    for (int k = 0; k < 3; ++k) c3[k] = fmaf(ttabf[t][2], ev32[18 + k], fmaf(ttabf[t][1], ev32[15 + k], ev32[12 + k]));
    cross3(zc + 3, c3, a0);
    cross3(c3, zc, a1);
    const float wf = ttabf[t][0] * zwf[iz];
    dt_from_adj<float>(a0, a1, zc + 6, wf, sf, wf * wf / sf, cf, cf + 9, cf[12], cf[13], D);
    float c[NSH * NSH + NSH];  // this point's G_q^T Dt_q G_q, then its share of b
    p1_point_contrib(D, Gs + q * 4 * NSH, c);
    // the sums over the group's points in point order (q = lane), as the
    // one-thread kernel adds them
    float A[NSH * NSH + NSH];
#pragma unroll
    for (int v = 0; v < NSH * NSH + NSH; ++v) A[v] = 0.f;
#pragma unroll
    for (int qq = 0; qq < NQ; ++qq)
#pragma unroll
      for (int v = 0; v < NSH * NSH + NSH; ++v) A[v] = __fadd_rn(A[v], __shfl_sync(0xffffffffu, c[v], gbase + qq));
    int code = st == FEI_ERR_NONFINITE ? 2 * FEI_ERR_NONFINITE : st;
    if (!ok) code = 2 * FEI_ERR_NONFINITE;  // any lane's coordinate or coefficient
    else if (!sym && code == 0) code = FEI_ERR_INVALID_ARG;
#pragma unroll
    for (int off = 4; off >= 1; off >>= 1) code = max(code, __shfl_xor_sync(0xffffffffu, code, off));
    const int fst = code == 2 * FEI_ERR_NONFINITE ? FEI_ERR_NONFINITE : code;
    if (live) {
      float *Ao = reinterpret_cast<float *>(a.A) + out_a(a, item, e, NSH);
      float *bo = reinterpret_cast<float *>(a.bv) + out_b(a, item, e, NSH);
#pragma unroll
      for (int v = 0; v < NSH * NSH + NSH; ++v) {
        if ((v & 7) != g) continue;
        if (v < NSH * NSH) {
          const int i = v / NSH, j = v - i * NSH;
          if (!a.upper || j >= i) Ao[a_pos(i, j, NSH, a.upper)] = fst ? 0.f : A[v];
        } else {
          bo[v - NSH * NSH] = fst ? 0.f : A[v];
        }
      }
      if (g == 0) a.status[e] = fst;
    }
  }
}

// Below this many elements the batch fills little of the GPU with one
// thread per element, and eight lanes per element finish sooner.
constexpr int64_t kP1SmallBatch = 16384;

fei_status launch_p1(const FwdArgs &a, int64_t grid_work, cudaStream_t s, int64_t grid_cap) {
  if (!a.count && grid_work <= kP1SmallBatch) {
    int64_t blocks = (grid_work * 8 + kP1Threads - 1) / kP1Threads;
    if (grid_cap > 0 && blocks > grid_cap) blocks = grid_cap;
    cc_p1_small_kernel<<<(unsigned)blocks, kP1Threads, 0, s>>>(a);
    FEI_CUDA_TRY(cudaGetLastError(), "cc_p1_small_kernel launch");
    return FEI_OK;
  }
  int64_t blocks = (grid_work + kP1Threads - 1) / kP1Threads;
  const int64_t cap = grid_cap > 0 ? grid_cap : 152 * 3;  // resident blocks: the tables are loaded once
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  cc_p1_kernel<<<(unsigned)blocks, kP1Threads, 0, s>>>(a);
  FEI_CUDA_TRY(cudaGetLastError(), "cc_p1_kernel launch");
  return FEI_OK;
}

fei_status launch_small(const FwdArgs &a, int64_t grid_work, cudaStream_t s, int64_t grid_cap) {
  using C = SmallCfg;
  FEI_CUDA_TRY(cudaFuncSetAttribute(cc_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM),
               "cudaFuncSetAttribute(cc_small)");
  int64_t blocks = (grid_work + C::WPB * C::EPW - 1) / (C::WPB * C::EPW);
  const int64_t cap = grid_cap > 0 ? grid_cap : (a.count ? 152 * 4 : 0);
  if (cap > 0 && blocks > cap) blocks = cap;
  if (blocks > 2147483647LL) blocks = 2147483647LL;
  if (blocks < 1) blocks = 1;
  cc_small_kernel<<<(unsigned)blocks, C::WPB * 32, C::SMEM, s>>>(a);
  FEI_CUDA_TRY(cudaGetLastError(), "cc_small_kernel launch");
  return FEI_OK;
}

}  // namespace

fei_status launch_cc_forward(int p, bool fp64, const fei_reference *ref, const FwdArgs &a, int64_t grid_work,
                             cudaStream_t s, int64_t grid_cap) {
  if (grid_work <= 0) return FEI_OK;
  if (p < 1 || p > kPMax) return set_error(FEI_ERR_INVALID_DEGREE, "degree %d outside 1..7", p);
  if (p == 1) return fp64 ? launch_small(a, grid_work, s, grid_cap) : launch_p1(a, grid_work, s, grid_cap);
  return fp64 ? launch_sf64_forward(p, ref, a, grid_work, s, grid_cap)
              : launch_sf_forward(p, ref, a, grid_work, s, grid_cap);
}

}  // namespace fei
