// fei_sf_ops.cuh -- what the sum-factorised forward (fei_sf.cuh) and adjoint
// (fei_backward.cu) share: FP64 element data, the point operators' layout in
// shared memory, small vector loads.
#pragma once

#include <type_traits>

#include "fei_elem32.cuh"
#include "fei_sf1d.cuh"

namespace fei {

// FP64 element data: the vertices and the node columns.
template <int P>
struct Elem64 {
  static constexpr int M = P + 1;
  double X[18];
  double zc1[M][3], zc2[M][3], zn3[M][3], tc3[M * M][3];
};
template <int P>
struct SfNodes64 {
  double zz[P + 1], zw[P + 1], tx[(P + 1) * (P + 1)][2], tw[(P + 1) * (P + 1)];
};

// Operators in shared memory: [op][iv][l][iu], the M values of a u row
// without a pad.  Rows of one quarter-warp fall in distinct banks for M = 4, 6
// (16- and 8-byte loads) and odd M (4-byte loads); for M = 8 the 16-byte
// halves are swapped by bit 2 of l, and iv has a stride of 72, so that the
// columns of the zeta transform are free of conflicts too.
template <typename T, int M>
struct OpPos {
  static constexpr bool SWZ = std::is_same<T, float>::value && M == 8;
  static constexpr int IV = SWZ ? 72 : M * M, OP = M * IV;
  static __device__ __forceinline__ int row(int op, int iv, int l) { return op * OP + iv * IV + l * M; }
  static __device__ __forceinline__ int at(int op, int iv, int l, int iu) {
    return row(op, iv, l) + (SWZ ? iu ^ (l & 4) : iu);
  }
};
// the u row of (op, iv, l); sw = l & 4 for the swapped halves
template <int M>
__device__ __forceinline__ void load_u_row(const float *D, int sw, float *d) {
  if constexpr (M == 8) {
    const float4 v = *reinterpret_cast<const float4 *>(D + sw), w = *reinterpret_cast<const float4 *>(D + (sw ^ 4));
    d[0] = v.x, d[1] = v.y, d[2] = v.z, d[3] = v.w, d[4] = w.x, d[5] = w.y, d[6] = w.z, d[7] = w.w;
  } else if constexpr (M == 4) {
    const float4 v = *reinterpret_cast<const float4 *>(D);
    d[0] = v.x, d[1] = v.y, d[2] = v.z, d[3] = v.w;
  } else if constexpr (M % 2 == 0) {
#pragma unroll
    for (int c = 0; c < M / 2; ++c) {
      const float2 v = reinterpret_cast<const float2 *>(D)[c];
      d[2 * c] = v.x, d[2 * c + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int c = 0; c < M; ++c) d[c] = D[c];
  }
}
template <int M>
__device__ __forceinline__ void load_u_row(const double *D, int, double *d) {
#pragma unroll
  for (int c = 0; c < M; ++c) d[c] = D[c];
}
// N values from a 16-byte aligned address (the pad after them may be read)
template <int N>
__device__ __forceinline__ void load_vec(const float *s, float *d) {
  if constexpr (N > 2) {
    const float4 v = *reinterpret_cast<const float4 *>(s);
    d[0] = v.x, d[1] = v.y, d[2] = v.z;
    if constexpr (N > 3) d[3] = v.w;
  } else if constexpr (N == 2) {
    const float2 v = *reinterpret_cast<const float2 *>(s);
    d[0] = v.x, d[1] = v.y;
  } else {
    d[0] = s[0];
  }
}
template <int N>
__device__ __forceinline__ void load_vec(const double *s, double *d) {
#pragma unroll
  for (int i = 0; i < N; i += 2) {
    if (i + 1 < N) {
      const double2 v = *reinterpret_cast<const double2 *>(s + i);
      d[i] = v.x, d[i + 1] = v.y;
    } else {
      d[i] = s[i];
    }
  }
}
template <typename T>
struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };

// Even and odd parts in u of the M values d: e on the half nodes u <= 0, o.
template <typename T, int M>
__device__ __forceinline__ void even_odd(const T *d, T *e, T *o) {
#pragma unroll
  for (int i = 0; i < (M + 1) / 2; ++i) {
    const bool mid = 2 * i == M - 1;
    e[i] = mid ? d[i] : d[i] + d[M - 1 - i];
    o[i] = mid ? T(0) : d[i] - d[M - 1 - i];
  }
}
}  // namespace fei
