// fei_sf.cu -- tables of the sum-factorised paths and the FP32 forward
// (FEI_SF_FP32; fei_sf.cuh has the kernel, fei_sf64.cu its FP64 instances).
//
// The 1D factors of the collapsed tensor-product basis are tabulated once per
// degree in FP64 from the library's own Gauss nodes and checked against the
// library's 3D reference table when the reference is created; a degree whose
// check fails has no sum-factorised path (FEI_ERR_UNSUPPORTED).
#include <math.h>
#include <string.h>

#include "fei_internal.cuh"
#include "fei_sf.cuh"

namespace fei {

namespace {

// ---------------------------------------------------------------------------
// 1D factor tables
// ---------------------------------------------------------------------------
// Layout while tabulated (FP64), M = p+1, T = the triangle functions
// (total degree ascending, then n ascending):
//   U[3][M iu][M m], V[4][M iv][T t], Z[2][M k][M iz], mt[T] (m of t).
__host__ __device__ constexpr int sf_tab_size(int p) {
  return 3 * (p + 1) * (p + 1) + 4 * (p + 1) * ((p + 1) * (p + 2) / 2) + 2 * (p + 1) * (p + 1) +
         (p + 1) * (p + 2) / 2;
}
// Legendre P_0..P_n and derivatives at x.
__device__ void legendre_all(int n, double x, double *P, double *dP) {
  P[0] = 1.0;
  dP[0] = 0.0;
  if (n >= 1) {
    P[1] = x;
    dP[1] = 1.0;
  }
  for (int k = 1; k < n; ++k) {
    P[k + 1] = ((2 * k + 1) * x * P[k] - k * P[k - 1]) / (k + 1);
    dP[k + 1] = dP[k - 1] + (2 * k + 1) * P[k];
  }
}

// Jacobi P_n^{(al, 0)}(x) by the three-term recurrence.
__device__ double jacobi(int n, double al, double x) {
  if (n == 0) return 1.0;
  double pm = 1.0, pc = 0.5 * ((al + 2.0) * x + al);
  for (int k = 2; k <= n; ++k) {
    const double a1 = 2.0 * k * (k + al) * (2.0 * k + al - 2.0);
    const double a2 = (2.0 * k + al - 1.0) * (al * al);
    const double a3 = (2.0 * k + al - 2.0) * (2.0 * k + al - 1.0) * (2.0 * k + al);
    const double a4 = 2.0 * (k + al - 1.0) * (k - 1.0) * (2.0 * k + al);
    const double pn = ((a2 + a3 * x) * pc - a4 * pm) / a1;
    pm = pc;
    pc = pn;
  }
  return pc;
}
// d/dx P_n^{(al, 0)} = (n + al + 1) / 2 P_{n-1}^{(al + 1, 1)}; the (al+1, 1)
// polynomial by the general three-term recurrence.
__device__ double jacobi_deriv(int n, double al, double x) {
  if (n == 0) return 0.0;
  const double a = al + 1.0, b = 1.0;
  const int m = n - 1;
  double pm = 1.0, pc = 0.5 * ((a + b + 2.0) * x + (a - b));
  if (m == 0) pc = 1.0;
  for (int k = 2; k <= m; ++k) {
    const double s = 2.0 * k + a + b;
    const double a1 = 2.0 * k * (k + a + b) * (s - 2.0);
    const double a2 = (s - 1.0) * (a * a - b * b);
    const double a3 = (s - 2.0) * (s - 1.0) * s;
    const double a4 = 2.0 * (k + a - 1.0) * (k + b - 1.0) * s;
    const double pn = ((a2 + a3 * x) * pc - a4 * pm) / a1;
    pm = pc;
    pc = pn;
  }
  return 0.5 * (n + al + 1.0) * pc;
}

// One thread: every table entry (FP64) from the 1D Gauss-Legendre nodes.
__global__ void sf_tables_kernel(int p, const double *znode, double *tab) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int M = p + 1, T = (p + 1) * (p + 2) / 2;
  double *U = tab, *V = U + 3 * M * M, *Z = V + 4 * M * T, *mt = Z + 2 * M * M;
  double P[8], dP[8];
  for (int i = 0; i < M; ++i) {
    const double x = znode[2 * i];
    legendre_all(p, x, P, dP);
    for (int m = 0; m < M; ++m) {
      U[(0 * M + i) * M + m] = P[m];
      U[(1 * M + i) * M + m] = dP[m];
      U[(2 * M + i) * M + m] = (1.0 + x) * dP[m];
    }
    for (int k = 0; k < M; ++k) {
      const double nk = sqrt((2.0 * k + 1.0) / 2.0);
      Z[(0 * M + k) * M + i] = nk * P[k];
      Z[(1 * M + k) * M + i] = nk * dP[k];
    }
    int t = 0;
    for (int d = 0; d <= p; ++d)
      for (int n = 0; n <= d; ++n, ++t) {
        const int m = d - n;
        const double c = sqrt(2.0 * (2 * m + 1) * (m + n + 1));
        const double h = 0.5 * (1.0 - x);
        const double hm = pow(h, m), jn = jacobi(n, 2.0 * m + 1.0, x), djn = jacobi_deriv(n, 2.0 * m + 1.0, x);
        const double B = c * hm * jn;
        const double dB = c * (m > 0 ? -0.5 * m * pow(h, m - 1) * jn : 0.0) + c * hm * djn;
        V[(0 * M + i) * T + t] = B;
        V[(1 * M + i) * T + t] = 4.0 * B / (1.0 - x);
        V[(2 * M + i) * T + t] = 2.0 * B / (1.0 - x);
        V[(3 * M + i) * T + t] = 2.0 * dB;
        if (i == 0) mt[t] = m;
      }
  }
}

// max |G(from the factors) - G64| over the whole reference table, and max
// |G64|, as the bits of non-negative doubles (atomicMax orders them).
__global__ void sf_check_kernel(int p, const double *tab, const double *G64, unsigned long long *out) {
  const int M = p + 1, T = (p + 1) * (p + 2) / 2, nsh = T * M, nq = M * M * M;
  const double *U = tab, *V = U + 3 * M * M, *Z = V + 4 * M * T, *mt = Z + 2 * M * M;
  double dmax = 0.0, gmax = 0.0;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < nq * nsh; idx += gridDim.x * blockDim.x) {
    const int q = idx / nsh, i = idx % nsh;
    const int iz = q / (M * M), iv = (q / M) % M, iu = q % M;
    const int k = i / T, t = i % T, m = (int)mt[t];
    const double A = U[iu * M + m], A1 = U[(M + iu) * M + m], A2 = U[(2 * M + iu) * M + m];
    const double B = V[iv * T + t], B1 = V[(M + iv) * T + t], B2 = V[(2 * M + iv) * T + t],
                 B3 = V[(3 * M + iv) * T + t];
    const double L = Z[k * M + iz], L1 = Z[(M + k) * M + iz];
    const double g[4] = {A * B * L, A1 * B1 * L, A2 * B2 * L + A * B3 * L, A * B * L1};
    for (int a = 0; a < 4; ++a) {
      const double ref = G64[(size_t)(4 * q + a) * nsh + i];
      dmax = fmax(dmax, fabs(g[a] - ref));
      gmax = fmax(gmax, fabs(ref));
    }
  }
  atomicMax(&out[0], (unsigned long long)__double_as_longlong(dmax));
  atomicMax(&out[1], (unsigned long long)__double_as_longlong(gmax));
}

// The FP64 tables in the kernels' layout (SfTab), as T.
template <typename T>
__global__ void pack_tables_kernel(int p, const double *t64, const double *znode, T *out) {
  const int M = p + 1, NT = M * (M + 1) / 2;
  const double *U = t64, *V = U + 3 * M * M, *Z = V + 4 * M * NT;
  // SfTab's offsets for a run-time degree
  const int o_u0 = 2 * M * 4, o_u1 = o_u0 + (M * M + 3) / 4 * 4, o_vc = o_u1 + (M * M + 3) / 4 * 4, o_vr = o_vc + (2 * M * NT + 3) / 4 * 4,
            o_zl = o_vr + (2 * M * NT + 3) / 4 * 4, o_zd = o_zl + M * M, o_gv = o_zd + M * M, o_su = o_gv + M, o_mt = o_su + M;
  const int stride = gridDim.x * blockDim.x, i0 = blockIdx.x * blockDim.x + threadIdx.x;
  for (int i = i0; i < 2 * M * 4; i += stride) {
    const int kind = i / (M * 4), m = i / 4 % M, iu = i % 4;
    out[i] = iu < (M + 1) / 2 ? (T)U[(kind * M + iu) * M + m] : T(0);
  }
  for (int i = i0; i < M * M; i += stride) {
    out[o_u0 + i] = (T)U[(i % M) * M + i / M];
    out[o_u1 + i] = (T)U[(M + i % M) * M + i / M];
    out[o_zl + i] = (T)Z[(i % M) * M + i / M];
    out[o_zd + i] = (T)Z[(M + i % M) * M + i / M];
  }
  for (int i = i0; i < M * NT; i += stride) {
    const int iv = i / NT, t = i % NT;
    // t = (m, n): its place in row order (m ascending, then n)
    int d = 0;
    while ((d + 1) * (d + 2) / 2 <= t) ++d;
    const int n = t - d * (d + 1) / 2, m = d - n, r = row_start(M, m) + n;
    const T v0 = (T)V[iv * NT + t], v1 = (T)V[(3 * M + iv) * NT + t];
    out[o_vc + 2 * i] = v0;
    out[o_vc + 2 * i + 1] = v1;
    out[o_vr + 2 * (iv * NT + r)] = v0;
    out[o_vr + 2 * (iv * NT + r) + 1] = v1;
    if (iv == 0) out[o_mt + t] = (T)m;
  }
  for (int i = i0; i < M; i += stride) {
    out[o_gv + i] = (T)(4.0 / (1.0 - znode[2 * i]));
    out[o_su + i] = (T)(0.5 * (1.0 + znode[2 * i]));
  }
}
int sf_table_size(int p) {
  switch (p) {
    case 1: return SfTab<1>::SIZE;
    case 2: return SfTab<2>::SIZE;
    case 3: return SfTab<3>::SIZE;
    case 4: return SfTab<4>::SIZE;
    case 5: return SfTab<5>::SIZE;
    case 6: return SfTab<6>::SIZE;
    default: return SfTab<7>::SIZE;
  }
}

}  // namespace

fei_status build_sf_tables(fei_reference *r) {
  r->sf = nullptr;
  r->sf64 = nullptr;
  const int n = sf_tab_size(r->p), nk = sf_table_size(r->p);
  double *t64 = nullptr;
  unsigned long long *dd = nullptr;
  cudaError_t e = cudaMalloc(&t64, sizeof(double) * n);
  if (e == cudaSuccess) e = cudaMalloc(&dd, 2 * sizeof(unsigned long long));
  if (e == cudaSuccess) e = cudaMemset(dd, 0, 2 * sizeof(unsigned long long));
  if (e == cudaSuccess) {
    sf_tables_kernel<<<1, 32>>>(r->p, r->znode, t64);
    sf_check_kernel<<<64, 256>>>(r->p, t64, r->G64, dd);
    e = cudaGetLastError();
  }
  unsigned long long h[2] = {0, 0};
  if (e == cudaSuccess) e = cudaMemcpy(h, dd, sizeof(h), cudaMemcpyDeviceToHost);
  float *t32 = nullptr;
  double *tab64 = nullptr;
  if (e == cudaSuccess) {
    double dmax, gmax;
    memcpy(&dmax, &h[0], 8);
    memcpy(&gmax, &h[1], 8);
    // the factors must reproduce the reference table (same basis, same
    // ordering, same signs) to FP64 rounding; otherwise no sum-factorised
    // path for this degree
    if (dmax <= 1e-12 * gmax) {
      e = cudaMalloc(&t32, sizeof(float) * nk);
      if (e == cudaSuccess) e = cudaMalloc(&tab64, sizeof(double) * nk);
      if (e == cudaSuccess) e = cudaMemset(t32, 0, sizeof(float) * nk);
      if (e == cudaSuccess) e = cudaMemset(tab64, 0, sizeof(double) * nk);
      if (e == cudaSuccess) {
        pack_tables_kernel<float><<<8, 256>>>(r->p, t64, r->znode, t32);
        pack_tables_kernel<double><<<8, 256>>>(r->p, t64, r->znode, tab64);
        e = cudaGetLastError();
      }
      if (e == cudaSuccess) e = cudaDeviceSynchronize();
    }
  }
  if (t64) cudaFree(t64);
  if (dd) cudaFree(dd);
  if (e != cudaSuccess) {
    if (t32) cudaFree(t32);
    if (tab64) cudaFree(tab64);
    return cuda_error(e, "sum-factorisation tables");
  }
  r->sf = t32;
  r->sf64 = tab64;
  return FEI_OK;
}

void free_sf_tables(fei_reference *r) {
  if (r->sf) cudaFree(r->sf);
  if (r->sf64) cudaFree(r->sf64);
  r->sf = nullptr;
  r->sf64 = nullptr;
}

fei_status launch_sf_forward(int p, const fei_reference *ref, const FwdArgs &a, int64_t grid_work, cudaStream_t s,
                             int64_t grid_cap) {
  if (grid_work <= 0) return FEI_OK;
  switch (p) {
    case 2: return launch_sf<float, 2>(ref->sf, a, grid_work, s, grid_cap);
    case 3: return launch_sf<float, 3>(ref->sf, a, grid_work, s, grid_cap);
    case 4: return launch_sf<float, 4>(ref->sf, a, grid_work, s, grid_cap);
    case 5: return launch_sf<float, 5>(ref->sf, a, grid_work, s, grid_cap);
    case 6: return launch_sf<float, 6>(ref->sf, a, grid_work, s, grid_cap);
    case 7: return launch_sf<float, 7>(ref->sf, a, grid_work, s, grid_cap);
  }
  return set_error(FEI_ERR_UNSUPPORTED, "sum-factorised path for degree %d", p);
}

}  // namespace fei
