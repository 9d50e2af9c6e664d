// fei_elem32.cuh -- element setup of the FP32-class paths: vertex
// differences in FP64, everything after them in double-FP32 arithmetic
// (fei_geom.cuh), rounded once where an FP32 value is used.
#pragma once

#include "fei_geom.cuh"
#include "fei_internal.cuh"

namespace fei {

// Node tables of one degree in shared memory: vertical nodes (zeta, w_z) and
// triangle nodes (w_t, w_t xi1, w_t xi2) as FP32 hi + lo pairs, FP32 copies.
template <int P>
struct NodeTab32 {
  static constexpr int M = P + 1, NT = M * M;
  double zz[M], zw[M];
  float2 ztab2[M][2];   // (zeta, w_z)
  float2 ttab2[NT][3];  // (w_t, w_t xi1, w_t xi2)
  float2 txi2[NT][2];   // (xi1, xi2)
  float zwf[M], twf[NT];
};

template <int P>
__device__ __forceinline__ void load_node_tab32(NodeTab32<P> &tb, const double *znode, const double *tnode, int tid,
                                                int nth) {
  for (int t = tid; t < NodeTab32<P>::NT; t += nth) {
    const double x1 = tnode[4 * t], x2 = tnode[4 * t + 1], wt = tnode[4 * t + 2];
    tb.ttab2[t][0] = split_f64(wt);
    tb.ttab2[t][1] = split_f64(wt * x1);
    tb.ttab2[t][2] = split_f64(wt * x2);
    tb.txi2[t][0] = split_f64(x1);
    tb.txi2[t][1] = split_f64(x2);
    tb.twf[t] = (float)wt;
  }
  for (int z = tid; z < P + 1; z += nth) {
    tb.zz[z] = znode[2 * z];
    tb.zw[z] = znode[2 * z + 1];
    tb.ztab2[z][0] = split_f64(znode[2 * z]);
    tb.ztab2[z][1] = split_f64(znode[2 * z + 1]);
    tb.zwf[z] = (float)znode[2 * z + 1];
  }
}

// Per element: the vertices, the element vectors as pairs, and per vertical
// node c1, c2, n3 = c1 x c2 in FP32, (n3.C, n3.D1, n3.D2) and w_z times them
// as pairs.
template <int P>
struct Elem32 {
  static constexpr int M = P + 1, NT = M * M;
  double X[18];
  float2 ev2[21];
  float2 zsum[M][3], zabg[M][3];
  float zc1f[M][3], zc2f[M][3], zn3f[M][3];
  float tc3f[NT][3];
  float gate;  // w det J above w times this is accurate as a pair (elem_setup32)
};

// One warp: element vectors (lanes 0-20, component k = j % 3 of vector
// v = j / 3) and vertical-node data (lane = 3 iz + k) of one element.  The
// vertex differences are FP64 subtractions (two per lane, one warp's worth of
// independent subtractions), split from their bit fields into FP32 pairs,
// the rest in double-FP32 arithmetic: a dependent FP64 instruction takes
// hundreds of cycles on this part, an FP32 one a few.  Differences outside
// 2^-60 <= |d| < 2^60 (other than 0) take the same steps in FP64, and so does
// an element whose n3 cancels (thin, collapsed or mirrored triangles): the
// pairs' n3 is good to about 2^-44 of the terms T = |c1a c2b| + |c1b c2a| of its
// components, so at every node a component has to be above 2^-14 of the largest
// T of all nodes (all: c1 or c2 may cancel at one of them).
//
// gate = 3 2^-14 q, q the largest T_k (5 |C_k| + |D1_k| + |D2_k|), so that 3 q bounds
// the terms of n3 . c3 in which nothing cancels: w det J as a pair has an error
// of about 2^-42 w 3 q, at most 2^-28 of a value above w gate.  One reduction
// each; with sums over k by shuffles the setup cost 3 % of the forward at p = 3.
// (p = 4, 100 000 prisms: 1.357 -> 1.364 ms with these checks, by shuffles 1.369.)
template <int P>
__device__ __noinline__ void elem_setup32(Elem32<P> &el, const NodeTab32<P> &tb, int lane) {
  constexpr int NZ = P + 1;
  const double x = lane < 18 ? el.X[lane] : 0.0;
  const int v = lane < 21 ? lane / 3 : 0, kv = lane < 21 ? lane % 3 : 0;
  // vertices (a, b, c, d) of vector v, 3 bits each, 12 bits per vector:
  //   A1 (1,0,4,3)  B1 (4,3,1,0)  A2 (2,0,5,3)  B2 (5,3,2,0)
  //   C  (3,0,0,0)  D1 (4,1,3,0)  D2 (5,2,3,0)
  // each (X_a - X_b) +- (X_c - X_d), halved
  constexpr unsigned long long kTab =
      (0x223ull << 0) | (0x8C8ull << 12) | (0x42Bull << 24) | (0xAD0ull << 36) | (0x600ull << 48);
  constexpr unsigned long long kTab2 = (0x858ull << 0) | (0xA98ull << 12);  // D1, D2
  constexpr unsigned kNeg = 0x6Au;                                          // B1, B2, D1, D2 subtract
  const unsigned tv = (unsigned)((v < 5 ? kTab >> (12 * v) : kTab2 >> (12 * (v - 5))) & 0xFFFu);
  const int la = 3 * ((tv >> 9) & 7u) + kv, lb = 3 * ((tv >> 6) & 7u) + kv;
  const int lc = 3 * ((tv >> 3) & 7u) + kv, ld = 3 * (tv & 7u) + kv;
  const bool subtract = (kNeg >> v) & 1u;
  const bool act = lane < 3 * NZ;
  const int iz = act ? lane / 3 : 0, k = act ? lane % 3 : 0;
  const int g0 = lane - k, l1 = g0 + (k + 1) % 3, l2 = g0 + (k + 2) % 3;
  const double xa = __shfl_sync(0xffffffffu, x, la), xb = __shfl_sync(0xffffffffu, x, lb);
  const double xc = __shfl_sync(0xffffffffu, x, lc), xd = __shfl_sync(0xffffffffu, x, ld);
  const double t1 = xa - xb, t2 = xc - xd;
  bool r1 = true, r2 = true;
  const float2 t1s = split_f64_bits(t1, &r1), t2s = split_f64_bits(t2, &r2);
  // gate and whether n3 cancels, from the terms of the lane's component of n3,
  // its part of (5 |C| + |D1| + |D2|) and the component (values >= 0 order as their
  // bits, a NaN above them)
  auto cancels = [&](float terms, float vert, float n3, float *gate) {
    const float T = act ? terms : 0.f;
    const float tm = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(T)));
    const float q = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(T * vert)));
    *gate = q < 3e29f ? 1.8310546875e-4f * q : __int_as_float(0x7f800000);  // infinity: always FP64
    unsigned ok = __ballot_sync(0xffffffffu, fabsf(n3) > 6.103515625e-5f * tm);
    ok |= ok >> 1 | ok >> 2;  // bit 3 iz: one of node iz's components
    constexpr unsigned nodes = 0x249249u & ((1u << 3 * NZ) - 1u);
    return (ok & nodes) != nodes;
  };
  bool pairs = __all_sync(0xffffffffu, lane >= 21 || (r1 && r2));
  if (pairs) {
    auto shfl2 = [](float2 q, int src) {
      return make_float2(__shfl_sync(0xffffffffu, q.x, src), __shfl_sync(0xffffffffu, q.y, src));
    };
    float2 ev = norm_ff(add_ff(t1s, subtract ? neg_ff(t2s) : t2s));
    ev = make_float2(0.5f * ev.x, 0.5f * ev.y);
    const float2 z2 = tb.ztab2[iz][0], wz2 = tb.ztab2[iz][1];
    const float2 a1 = shfl2(ev, k), b1 = shfl2(ev, 3 + k), a2 = shfl2(ev, 6 + k), b2 = shfl2(ev, 9 + k);
    const float2 vc = shfl2(ev, 12 + k), vd1 = shfl2(ev, 15 + k), vd2 = shfl2(ev, 18 + k);
    const float2 c1 = norm_ff(add_ff(a1, mul_ff(z2, b1)));
    const float2 c2 = norm_ff(add_ff(a2, mul_ff(z2, b2)));
    const float2 c1a = shfl2(c1, l1), c1b = shfl2(c1, l2), c2a = shfl2(c2, l1), c2b = shfl2(c2, l2);
    const float2 n3 = norm_ff(add_ff(mul_ff(c1a, c2b), neg_ff(mul_ff(c1b, c2a))));
    float2 ab = mul_ff(n3, vc);
    float2 bb = mul_ff(n3, vd1);
    float2 gb = mul_ff(n3, vd2);
    ab = norm_ff(add_ff(ab, add_ff(shfl2(ab, l1), shfl2(ab, l2))));
    bb = norm_ff(add_ff(bb, add_ff(shfl2(bb, l1), shfl2(bb, l2))));
    gb = norm_ff(add_ff(gb, add_ff(shfl2(gb, l1), shfl2(gb, l2))));
    float gate;
    pairs = !cancels(fabsf(c1a.x * c2b.x) + fabsf(c1b.x * c2a.x), 5.f * fabsf(vc.x) + fabsf(vd1.x) + fabsf(vd2.x), n3.x,
                   &gate);
    if (pairs) {
      if (lane == 0) el.gate = gate;
      if (lane < 21) el.ev2[lane] = ev;
      if (act) {
        const float2 sk = k == 0 ? ab : k == 1 ? bb : gb;
        el.zsum[iz][k] = sk;
        el.zabg[iz][k] = norm_ff(mul_ff(wz2, sk));
        el.zc1f[iz][k] = c1.x;
        el.zc2f[iz][k] = c2.x;
        el.zn3f[iz][k] = n3.x;
      }
    }
  }
  if (!pairs) {
    const double ev = 0.5 * (subtract ? t1 - t2 : t1 + t2);
    const double z = tb.zz[iz], wz = tb.zw[iz];
    const double a1 = __shfl_sync(0xffffffffu, ev, k), b1 = __shfl_sync(0xffffffffu, ev, 3 + k);
    const double a2 = __shfl_sync(0xffffffffu, ev, 6 + k), b2 = __shfl_sync(0xffffffffu, ev, 9 + k);
    const double vc = __shfl_sync(0xffffffffu, ev, 12 + k), vd1 = __shfl_sync(0xffffffffu, ev, 15 + k);
    const double vd2 = __shfl_sync(0xffffffffu, ev, 18 + k);
    const double c1 = fma(z, b1, a1);
    const double c2 = fma(z, b2, a2);
    const double c1a = __shfl_sync(0xffffffffu, c1, l1), c1b = __shfl_sync(0xffffffffu, c1, l2);
    const double c2a = __shfl_sync(0xffffffffu, c2, l1), c2b = __shfl_sync(0xffffffffu, c2, l2);
    const double n3 = c1a * c2b - c1b * c2a;
    double ab = n3 * vc;
    double bb = n3 * vd1;
    double gb = n3 * vd2;
    ab += __shfl_sync(0xffffffffu, ab, l1) + __shfl_sync(0xffffffffu, ab, l2);
    bb += __shfl_sync(0xffffffffu, bb, l1) + __shfl_sync(0xffffffffu, bb, l2);
    gb += __shfl_sync(0xffffffffu, gb, l1) + __shfl_sync(0xffffffffu, gb, l2);
    float gate;
    cancels((float)(fabs(c1a * c2b) + fabs(c1b * c2a)), (float)(5.0 * fabs(vc) + fabs(vd1) + fabs(vd2)), (float)n3, &gate);
    if (lane == 0) el.gate = gate;
    if (lane < 21) el.ev2[lane] = split_f64(ev);
    if (act) {
      const double sk = k == 0 ? ab : k == 1 ? bb : gb;
      el.zsum[iz][k] = split_f64(sk);
      el.zabg[iz][k] = split_f64(wz * sk);
      el.zc1f[iz][k] = (float)c1;
      el.zc2f[iz][k] = (float)c2;
      el.zn3f[iz][k] = (float)n3;
    }
  }
}

// Component k of the triangle-node column c3 = C + xi1 D1 + xi2 D2, rounded once.
template <int P>
__device__ __forceinline__ float tri_column32(const Elem32<P> &el, const NodeTab32<P> &tb, int t, int k) {
  const float2 c3 = add_ff(add_ff(el.ev2[12 + k], mul_ff(tb.txi2[t][0], el.ev2[15 + k])),
                           mul_ff(tb.txi2[t][1], el.ev2[18 + k]));
  return c3.x + c3.y;
}

// Columns c1, c2 and n3 = c1 x c2 at the vertical node z from the vertex
// coordinates (the element vectors A1, B1, A2, B2 formed on the spot), FP64.
__device__ __forceinline__ void z_columns_from_vertices(const double *X, double z, double *c1, double *c2,
                                                        double *n3) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double e1p = X[3 + k] - X[k], e1q = X[12 + k] - X[9 + k];
    const double e2p = X[6 + k] - X[k], e2q = X[15 + k] - X[9 + k];
    c1[k] = fma(z, 0.5 * (e1q - e1p), 0.5 * (e1p + e1q));
    c2[k] = fma(z, 0.5 * (e2q - e2p), 0.5 * (e2p + e2q));
  }
  cross3(c1, c2, n3);
}
// Column c3 at the triangle node (xi1, xi2) (element vectors C, D1, D2).
__device__ __forceinline__ void t_column_from_vertices(const double *X, double xi1, double xi2, double *c3) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double v0 = X[9 + k] - X[k], v1 = X[12 + k] - X[3 + k], v2 = X[15 + k] - X[6 + k];
    c3[k] = fma(xi2, 0.5 * (v2 - v0), fma(xi1, 0.5 * (v1 - v0), 0.5 * v0));
  }
}

// det J at vertical node iz and triangle node t in FP64, from the vertices.
template <int P>
__device__ __noinline__ double point_det64(const Elem32<P> &el, const NodeTab32<P> &tb, int iz, int t,
                                           const double *tnode) {
  double c1[3], c2[3], n3[3], c3[3];
  z_columns_from_vertices(el.X, tb.zz[iz], c1, c2, n3);
  t_column_from_vertices(el.X, tnode[4 * t], tnode[4 * t + 1], c3);
  return dot3(n3, c3);
}

// w det J at vertical node iz and triangle node t, rounded once to FP32, and
// the point's status; w: the point's weight.  w det J = w_t (a + xi1 b + xi2 g)
// from the node sums in double-FP32; a value that is not above w times the
// element's gate (elem_setup32), or near the lower end of the FP32 range, is
// formed again in FP64 from the vertices, so that a value that an FP32 pair
// could get wrong, in sign or in its FP32 digits, is an FP64 one.  With det: det J
// too (the adjoint's, with the forward's status).
template <int P>
__device__ __forceinline__ float point_wdet32(const Elem32<P> &el, const NodeTab32<P> &tb, int iz, int t, float w,
                                              const double *tnode, int *status, float *det = nullptr) {
  const float2 sd = add_ff(add_ff(mul_ff(tb.ttab2[t][0], el.zabg[iz][0]), mul_ff(tb.ttab2[t][1], el.zabg[iz][1])),
                           mul_ff(tb.ttab2[t][2], el.zabg[iz][2]));
  const float s = sd.x + sd.y;
  *status = 0;
  if (s > w * el.gate && s > 1e-30f) {
    if (det) {
      const float2 dd = add_ff(add_ff(el.zsum[iz][0], mul_ff(tb.txi2[t][0], el.zsum[iz][1])),
                               mul_ff(tb.txi2[t][1], el.zsum[iz][2]));
      *det = dd.x + dd.y;
    }
    return s;
  }
  const double d = point_det64<P>(el, tb, iz, t, tnode), sw = tb.zw[iz] * tnode[4 * t + 2] * d;
  // p = 2: a value outside the FP32 range is flagged as well
  *status = point_status(P <= 2 ? (double)(float)sw : sw);
  if (det) *det = (float)d;
  return (float)sw;
}

}  // namespace fei
