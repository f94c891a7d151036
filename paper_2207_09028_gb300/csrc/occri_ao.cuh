// occri_ao.cuh -- device functions of the AO kernels: solid harmonics, displacements of grid
// points from atoms, the double-float Gaussian argument and the point blocks.
#pragma once

#include "occri_device.cuh"
#include "occri_internal.h"

namespace occri {
namespace ao {

using dev::cis_frac;
using dev::exp_t;

// Unnormalised real solid harmonics, m = -l..l (p: x, y, z).
template <typename T, int L>
__device__ __forceinline__ void solid(T x, T y, T z, T (&P)[2 * L + 1]) {
  if constexpr (L == 0) {
    P[0] = T(1);
  } else if constexpr (L == 1) {
    P[0] = x; P[1] = y; P[2] = z;
  } else if constexpr (L == 2) {
    P[0] = x * y;
    P[1] = y * z;
    P[2] = T(2) * z * z - x * x - y * y;
    P[3] = x * z;
    P[4] = x * x - y * y;
  } else {
    const T x2 = x * x, y2 = y * y, z2 = z * z;
    P[0] = y * (T(3) * x2 - y2);
    P[1] = x * y * z;
    P[2] = y * (T(4) * z2 - x2 - y2);
    P[3] = z * (T(2) * z2 - T(3) * x2 - T(3) * y2);
    P[4] = x * (T(4) * z2 - x2 - y2);
    P[5] = z * (x2 - y2);
    P[6] = x * (x2 - T(3) * y2);
  }
}

// r_n - A - T0 for one grid point and atom, in the working precision.
template <typename T> struct Disp;
template <> struct Disp<double> { double x, y, z; };
template <> struct Disp<float> { float xh, yh, zh, xl, yl, zl; };

__device__ __forceinline__ void load_disp(const AOParams& p, int atom, long long n, Disp<double>* d) {
  const double* b = p.d0_d + (size_t)atom * 3 * p.ng;
  d->x = b[n];
  d->y = b[p.ng + n];
  d->z = b[2 * p.ng + n];
}
__device__ __forceinline__ void load_disp(const AOParams& p, int atom, long long n, Disp<float>* d) {
  const float* h = p.d0_hi + (size_t)atom * 3 * p.ng;
  const float* l = p.d0_lo + (size_t)atom * 3 * p.ng;
  d->xh = h[n]; d->yh = h[p.ng + n]; d->zh = h[2 * p.ng + n];
  d->xl = l[n]; d->yl = l[p.ng + n]; d->zl = l[2 * p.ng + n];
}

// Exact-argument Gaussian for FP32: x = (d0 - T') as an unevaluated hi + lo sum (two-diff
// of the hi parts plus the lo parts), r^2 and alpha r^2 as hi + lo pairs (FMA
// two-products, two-sums), and e^{-alpha r^2} = e^{-ah} (1 - al). Returns r^2 (hi) for
// the cutoff test and the coordinates rounded to FP32 for the polynomial.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
// d - T rounded to FP32 in *x, *y, *z, and r^2 as *r2h + *r2l.
__device__ __forceinline__ void exact_r2(const Disp<float>& d, float txh, float tyh, float tzh,
                                         float txl, float tyl, float tzl, float* r2h, float* r2l,
                                         float* x, float* y, float* z) {
  float c[3], cl[3];
  const float dh[3] = {d.xh, d.yh, d.zh}, dl[3] = {d.xl, d.yl, d.zl};
  const float th[3] = {txh, tyh, tzh}, tl[3] = {txl, tyl, tzl};
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    float s, e;
    two_sum(dh[q], -th[q], s, e);
    c[q] = s;
    cl[q] = e + (dl[q] - tl[q]);
  }
  float ph[3], pl[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    ph[q] = c[q] * c[q];
    pl[q] = fmaf(c[q], c[q], -ph[q]) + 2.0f * c[q] * cl[q];
  }
  float s1, e1, s2, e2;
  two_sum(ph[0], ph[1], s1, e1);
  two_sum(s1, ph[2], s2, e2);
  *r2l = (e1 + e2) + (pl[0] + pl[1] + pl[2]);
  *r2h = s2;
  *x = c[0] + cl[0];
  *y = c[1] + cl[1];
  *z = c[2] + cl[2];
}
__device__ __forceinline__ float exact_gauss(const Disp<float>& d, float txh, float tyh,
                                             float tzh, float txl, float tyl, float tzl,
                                             float ah_, float al_, float* r2h, float* x,
                                             float* y, float* z) {
  float r2l;
  exact_r2(d, txh, tyh, tzh, txl, tyl, tzl, r2h, &r2l, x, y, z);
  const float ah = ah_ * *r2h;
  const float al = fmaf(ah_, *r2h, -ah) + ah_ * r2l + al_ * *r2h;
  return expf(-ah) * (1.0f - al);
}

// Grid point of `lane` in point block `blk` (2 x 4 x 4 points, ragged at the grid edge);
// lanes outside the grid get a clamped in-range point and *valid = false.
// Point `lane` of block `blk`: its natural index n = (n1 N2 + n2) N3 + n3 (the
// geometry tables) and its index in the orbital/accumulator fields, which are stored
// with the third axis outermost, q = (n3 N1 + n1) N2 + n2 (see occri_internal.h).
// Lanes run along n2 first so that four consecutive lanes touch contiguous elements.
// Points past the grid edge (ragged blocks) are clamped and flagged invalid.
__device__ __forceinline__ long long block_point(const AOParams& p, int blk, int lane, bool* valid,
                                                 long long* q) {
  const int b3 = blk % p.nb[2], b2 = (blk / p.nb[2]) % p.nb[1], b1 = blk / (p.nb[1] * p.nb[2]);
  int n1 = 2 * b1 + (lane >> 4), n2 = 4 * b2 + (lane & 3), n3 = 4 * b3 + ((lane >> 2) & 3);
  *valid = n1 < p.N[0] && n2 < p.N[1] && n3 < p.N[2];
  n1 = min(n1, p.N[0] - 1);
  n2 = min(n2, p.N[1] - 1);
  n3 = min(n3, p.N[2] - 1);
  *q = ((long long)n3 * p.N[0] + n1) * p.N[1] + n2;
  return ((long long)n1 * p.N[1] + n2) * p.N[2] + n3;
}

// e^{sign i k.r} at grid point (n1, n2, n3): the phase 2 pi sum_d kint_d n_d / (D_d N) of k = kint / D,
// reduced exactly in integers.
template <typename T>
__device__ __forceinline__ cplx_t<T> point_phase(const int* kint, int D0, int D1, int D2, int N,
                                                 int n1, int n2, int n3, int sign) {
  const long long Dc = (long long)D0 * D1 * D2;
  const long long num = (long long)kint[0] * n1 * (Dc / D0) + (long long)kint[1] * n2 * (Dc / D1) +
                        (long long)kint[2] * n3 * (Dc / D2);
  return cis_frac<T>(num, Dc * N, sign);
}

}  // namespace ao
}  // namespace occri
