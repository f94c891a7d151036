// occri_chi.cu -- Bloch AOs on the grid in tiles, and the two products with them:
//   (a) chi_{mu k}(r) = sum_T e^{i k.T} phi_mu(r - A - T)                     (Sec. II.A)
//   (b) psi_{ik}(r) = sum_mu C^k_{mu i} chi_{mu k}(r)                          (Eq. occmo)
//   (e) K_{mu i}(k) = -(Omega/(N_k N_g)) sum_r conj(chi_{mu k}(r)) Y_{ik}(r)   (Eq. occrik)
//
// chi_kernel forms chi for a run of point blocks (2 x 4 x 4 points each) and every k at once:
// the Gaussian of an image is evaluated once, summed with the other images of its residue
// class (lattice vectors equal modulo the k-mesh's supercell share e^{i k.T}), and only the
// class sums meet the phases. orb_kernel and con_kernel are the products, one block per warp
// with a point per lane. Blocks keep only the AOs that reach them: an atom's shells are
// ordered by screening radius, so the AOs that reach a block are a prefix of the atom's slots.
//
// Before this, each step evaluated the Gaussians itself, once per four k-points in (b) and
// once per k-point in (e), with every image's phases applied on the spot.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <numeric>
#include <type_traits>
#include <vector>

#include "fft_reg.cuh"
#include "occri_ao.cuh"
#include "occri_chi.cuh"
#include "occri_device.cuh"
#include "occri_internal.h"

namespace occri {
namespace chi {

using ao::Disp;

constexpr int kWarps = 8;       // most warps of a chi_kernel CTA
constexpr int kFoldWarps = 4;   // warps of its CTAs where no class sums cross warps
constexpr int kFold = 8;        // most classes of a mesh whose shells take a warp each
constexpr int kRows = 7 * kFold;   // entry rows of a warp (a value per lane each)
constexpr int kCols = 10;       // AOs that the CTA takes together (wide shells)
constexpr int kWide = 12;       // images from which a shell counts as wide

template <typename T> struct Rec;
template <> struct alignas(16) Rec<float> { float xh, yh, zh; int cls; float xl, yl, zl; int pad; };
template <> struct alignas(16) Rec<double> { double x, y, z; int cls, pad; };

template <typename T> struct CsT;
template <> struct CsT<double> { using type = double2; };
template <> struct CsT<float> { using type = float4; };

template <typename T>
__device__ __forceinline__ Rec<T> load_rec(const Params& p, size_t list0, const int* cls, int j) {
  const int id = p.a.blist[list0 + j];
  Rec<T> r;
  if constexpr (sizeof(T) == 4) {
    r.xh = p.a.img_hi[id];
    r.yh = p.a.img_hi[p.a.nimg + id];
    r.zh = p.a.img_hi[2 * p.a.nimg + id];
    r.xl = p.a.img_lo[id];
    r.yl = p.a.img_lo[p.a.nimg + id];
    r.zl = p.a.img_lo[2 * p.a.nimg + id];
  } else {
    r.x = p.a.img_d[id];
    r.y = p.a.img_d[p.a.nimg + id];
    r.z = p.a.img_d[2 * p.a.nimg + id];
  }
  r.cls = cls[id];
  r.pad = 0;
  return r;
}

// The 2L + 1 functions of a shell (without their norms) at displacement d - T, 0 past the
// screening radius.
template <int L>
__device__ __forceinline__ void eval(const ChiShell& sh, const Disp<float>& d,
                                     const Rec<float>& r, float (&v)[2 * L + 1]) {
  float x, y, z, r2, e;
  if (sh.exact) {
    e = ao::exact_gauss(d, r.xh, r.yh, r.zh, r.xl, r.yl, r.zl, sh.alpha, sh.alpha_lo, &r2, &x, &y,
                        &z);
  } else {
    x = (d.xh - r.xh) + (d.xl - r.xl);
    y = (d.yh - r.yh) + (d.yl - r.yl);
    z = (d.zh - r.zh) + (d.zl - r.zl);
    r2 = x * x + y * y + z * z;
    e = expf(-(sh.alpha * r2 + sh.alpha_lo * r2));
  }
  if (!(r2 <= sh.rcut2)) e = 0.f;
  ao::solid<float, L>(x, y, z, v);
#pragma unroll
  for (int m = 0; m < 2 * L + 1; ++m) v[m] *= e;
}
template <int L>
__device__ __forceinline__ void eval(const ChiShell& sh, const Disp<double>& d,
                                     const Rec<double>& r, double (&v)[2 * L + 1]) {
  const double x = d.x - r.x, y = d.y - r.y, z = d.z - r.z;
  const double r2 = x * x + y * y + z * z;
  double e = exp(-(sh.alpha_d * r2));
  if (!(r2 <= sh.rcut2_d)) e = 0.0;
  ao::solid<double, L>(x, y, z, v);
#pragma unroll
  for (int m = 0; m < 2 * L + 1; ++m) v[m] *= e;
}

// acc[b][m] += phases of KT k-points times the entries' values
template <typename T, int KT, int NM>
__device__ __forceinline__ void phase_sums(const cplx_t<T>* ph, int nkp, const T* ent,
                                           const int* ecls, int ne, int k0, int lane,
                                           T (&xr)[KT][NM], T (&xi)[KT][NM]) {
  for (int e = 0; e < ne; ++e) {
    const cplx_t<T>* row = ph + (size_t)ecls[e] * nkp + k0;
    cplx_t<T> w[KT];
    if constexpr (sizeof(T) == 4 && KT % 2 == 0) {
#pragma unroll
      for (int b = 0; b < KT; b += 2) {
        const float4 q = __ldg(reinterpret_cast<const float4*>(row + b));
        w[b] = cplx_t<T>{q.x, q.y};
        w[b + 1] = cplx_t<T>{q.z, q.w};
      }
    } else {
#pragma unroll
      for (int b = 0; b < KT; ++b) w[b] = __ldg(row + b);
    }
    T v[NM];
#pragma unroll
    for (int m = 0; m < NM; ++m) v[m] = ent[(e * NM + m) * 32 + lane];
#pragma unroll
    for (int b = 0; b < KT; ++b)
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        xr[b][m] += w[b].x * v[m];
        xi[b][m] += w[b].y * v[m];
      }
  }
}

// A narrow shell, one warp: every image its own entry (a lane reads back only what it wrote),
// then chi of the k-points [ka, kb). Where the entries run out, the sums so far go to chi and the rest is
// added.
template <typename T, int L, int KT, typename GetRec>
__device__ __forceinline__ void narrow_shell(const Params& p, const ChiShell& sh,
                                             const Disp<T>& d, int np, const GetRec& rec, T* ent,
                                             int* ecls, cplx_t<T>* out, int kstride, int lane,
                                             int ka, int kb) {
  constexpr int NM = 2 * L + 1;
  constexpr int CAP = kRows / NM;
  const cplx_t<T>* ph = reinterpret_cast<const cplx_t<T>*>(p.phase);
  for (int j0 = 0; j0 < np; j0 += CAP) {
    const int ne = min(CAP, np - j0);
    for (int e = 0; e < ne; ++e) {
      const Rec<T> r = rec(j0 + e);
      T v[NM];
      eval<L>(sh, d, r, v);
#pragma unroll
      for (int m = 0; m < NM; ++m) ent[(e * NM + m) * 32 + lane] = v[m];
      if (lane == 0) ecls[e] = r.cls;
    }
    __syncwarp();
    for (int k0 = ka; k0 < kb; k0 += KT) {
      T xr[KT][NM], xi[KT][NM];
#pragma unroll
      for (int b = 0; b < KT; ++b)
#pragma unroll
        for (int m = 0; m < NM; ++m) xr[b][m] = xi[b][m] = T(0);
      phase_sums<T, KT, NM>(ph, p.nkp, ent, ecls, ne, k0, lane, xr, xi);
#pragma unroll
      for (int b = 0; b < KT; ++b) {
        if (k0 + b >= kb) break;
        cplx_t<T>* o = out + (size_t)(k0 + b) * kstride + lane;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
          cplx_t<T> v{xr[b][m], xi[b][m]};
          if (j0 > 0) {
            const cplx_t<T> u = o[32 * m];
            v.x += u.x;
            v.y += u.y;
          }
          o[32 * m] = v;
        }
      }
    }
    __syncwarp();
  }
}

// A shell on a mesh of at most kFold classes, one warp: class sums in the warp's rows (row
// class NM + m; a lane reads back only what it wrote), then chi of every k. Where every axis
// has one or two points the phases are signs and chi is real: sums and differences over the axes
// (a Walsh-Hadamard transform), and the buffer holds real values; else the classes' phases as in
// narrow_shell.
template <typename T, int L, int KT, typename GetRec>
__device__ __forceinline__ void fold_shell(const Params& p, const ChiShell& sh, const Disp<T>& d,
                                           int np, const GetRec& rec, T* ent, int* ecls,
                                           cplx_t<T>* out, int kstride, int lane) {
  constexpr int NM = 2 * L + 1;
  const int nc = p.ncls, nk = p.a.nk;
  T* e0 = ent + lane;
  for (int x = 0; x < nc * NM; ++x) e0[x * 32] = T(0);
  Rec<T> next = rec(0);
  for (int j = 0; j < np; ++j) {
    const Rec<T> r = next;
    if (j + 1 < np) next = rec(j + 1);
    T v[NM];
    eval<L>(sh, d, r, v);
    T* o = e0 + r.cls * (NM * 32);
#pragma unroll
    for (int m = 0; m < NM; ++m) o[m * 32] += v[m];
  }
  if (p.signs) {
    int off[kFold];   // where each class index's k goes, or -1
#pragma unroll
    for (int c = 0; c < kFold; ++c) {
      const int k = c < nc ? p.kidx[c] : -1;
      off[c] = k >= 0 ? k * kstride + lane : -1;
    }
    // rolled: the straight-line form missed the instruction cache
#pragma unroll 1
    for (int m = 0; m < NM; ++m) {
      T f[kFold];
#pragma unroll
      for (int c = 0; c < kFold; ++c) f[c] = c < nc ? e0[(c * NM + m) * 32] : T(0);
#pragma unroll
      for (int st = 1; st < kFold; st *= 2) {
        if (st >= nc) break;
#pragma unroll
        for (int c = 0; c < kFold; ++c)
          if (!(c & st)) {
            const T u = f[c], w = f[c + st];
            f[c] = u + w;
            f[c + st] = u - w;
          }
      }
#pragma unroll
      for (int c = 0; c < kFold; ++c)
        if (off[c] >= 0) reinterpret_cast<T*>(out)[off[c] + 32 * m] = f[c];
    }
    return;
  }
  __syncwarp();
  if (lane < nc) ecls[lane] = lane;
  __syncwarp();
  for (int k0 = 0; k0 < nk; k0 += KT) {
    T xr[KT][NM], xi[KT][NM];
#pragma unroll
    for (int b = 0; b < KT; ++b)
#pragma unroll
      for (int m = 0; m < NM; ++m) xr[b][m] = xi[b][m] = T(0);
    phase_sums<T, KT, NM>(reinterpret_cast<const cplx_t<T>*>(p.phase), p.nkp, ent, ecls, nc, k0,
                          lane, xr, xi);
#pragma unroll
    for (int b = 0; b < KT; ++b) {
      if (k0 + b >= nk) break;
#pragma unroll
      for (int m = 0; m < NM; ++m)
        out[(size_t)(k0 + b) * kstride + 32 * m + lane] = cplx_t<T>{xr[b][m], xi[b][m]};
    }
  }
}

// ---- wide shells: the class sums of up to kCols AOs in shared memory, then a discrete Fourier
// transform over the classes, axis by axis (chi_k = sum_l e^{2 pi i k.l/D} Phi_l, Phi real: only
// the non-negative half of the first axis is kept, the rest are conjugates). A column holds
// one AO: rows ((l_0 D_1 + l_1) D_2 + l_2), a value per lane; after the first axis, row pairs
// 2 k_0 (re) and 2 k_0 + 1 (im) in the place of l_0.
template <typename F>
__device__ __forceinline__ void by_length(int D, F&& f) {
  switch (D) {
    case 1: f(std::integral_constant<int, 1>{}); break;
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5: f(std::integral_constant<int, 5>{}); break;
    case 6: f(std::integral_constant<int, 6>{}); break;
    default: f(std::integral_constant<int, 8>{}); break;
  }
}

// One column's transform; chi of every k of the mesh goes to out.
template <typename T>
__device__ __forceinline__ void mesh_dft(const Params& p, T* col, cplx_t<T>* out, int kstride,
                                         int lane) {
  const int D0 = p.a.D[0], D1 = p.a.D[1], D2 = p.a.D[2], H = D0 / 2 + 1, P = D1 * D2;
  T* c = col + lane;
  by_length(D0, [&](auto ND) {
    constexpr int N = decltype(ND)::value;
    for (int j = 0; j < P; ++j) {
      T re[N], im[N];
      fft::static_for<N>([&](auto I) {
        constexpr int n = decltype(I)::value;
        re[n] = c[(n * P + j) * 32];
        im[n] = T(0);
      });
      fft::pfa<N, 1>(re, im);
      fft::static_for<N>([&](auto I) {
        constexpr int q = decltype(I)::value, k = fft::pfa_out(N, q);
        if constexpr (k < N / 2 + 1) {
          c[(2 * k * P + j) * 32] = re[q];
          c[((2 * k + 1) * P + j) * 32] = im[q];
        }
      });
    }
  });
  if (D1 > 1)
    by_length(D1, [&](auto ND) {
      constexpr int N = decltype(ND)::value;
      for (int j = 0; j < H * D2; ++j) {
        T* r = c + ((size_t)(j / D2) * 2 * P + j % D2) * 32;
        T re[N], im[N];
        fft::static_for<N>([&](auto I) {
          constexpr int n = decltype(I)::value;
          re[n] = r[n * D2 * 32];
          im[n] = r[(P + n * D2) * 32];
        });
        fft::pfa<N, 1>(re, im);
        fft::static_for<N>([&](auto I) {
          constexpr int q = decltype(I)::value, k = fft::pfa_out(N, q);
          r[k * D2 * 32] = re[q];
          r[(P + k * D2) * 32] = im[q];
        });
      }
    });
  by_length(D2, [&](auto ND) {
    constexpr int N = decltype(ND)::value;
    for (int j = 0; j < H * D1; ++j) {
      const int k0 = j / D1, k1 = j % D1;
      const T* r = c + ((size_t)k0 * 2 * P + k1 * D2) * 32;
      T re[N], im[N];
      fft::static_for<N>([&](auto I) {
        constexpr int n = decltype(I)::value;
        re[n] = r[n * 32];
        im[n] = r[(P + n) * 32];
      });
      fft::pfa<N, 1>(re, im);
      const int g0 = (D0 - k0) % D0, g1 = (D1 - k1) % D1;   // -k on the first two axes
      const int* at = p.kidx + (k0 * D1 + k1) * D2;
      const int* neg = p.kidx + (g0 * D1 + g1) * D2;
      fft::static_for<N>([&](auto I) {
        constexpr int q = decltype(I)::value, k = fft::pfa_out(N, q);
        const int i = at[k];
        if (i >= 0) out[(size_t)i * kstride + lane] = cplx_t<T>{re[q], im[q]};
        if (g0 != k0) {
          const int n = neg[k == 0 ? 0 : N - k];
          if (n >= 0) out[(size_t)n * kstride + lane] = cplx_t<T>{re[q], -im[q]};
        }
      });
    }
  });
}

// Displacement, r^2 and what the shells need of them for one image. In FP32 shells with an exact
// exponent want r^2 as a hi + lo pair (see ao::exact_gauss); the others take lo = 0 and alpha
// r^2 in one rounding less.
template <typename T> struct Geo;
template <> struct Geo<float> {
  float x, y, z, rh, rl;
  __device__ __forceinline__ Geo(const Disp<float>& d, const Rec<float>& r, bool exact) {
    if (exact) {
      ao::exact_r2(d, r.xh, r.yh, r.zh, r.xl, r.yl, r.zl, &rh, &rl, &x, &y, &z);
    } else {
      x = (d.xh - r.xh) + (d.xl - r.xl);
      y = (d.yh - r.yh) + (d.yl - r.yl);
      z = (d.zh - r.zh) + (d.zl - r.zl);
      rh = x * x + y * y + z * z;
      rl = 0.f;
    }
  }
  __device__ __forceinline__ float gauss(float alpha, float alpha_lo, float rcut2,
                                         bool exact) const {
    float e;
    if (exact) {
      const float ah = alpha * rh;
      const float al = fmaf(alpha, rh, -ah) + alpha * rl + alpha_lo * rh;
      e = expf(-ah) * (1.0f - al);
    } else {
      e = expf(-(alpha * rh + alpha_lo * rh));
    }
    return rh <= rcut2 ? e : 0.f;
  }
};
template <> struct Geo<double> {
  double x, y, z, r2;
  __device__ __forceinline__ Geo(const Disp<double>& d, const Rec<double>& r, bool)
      : x(d.x - r.x), y(d.y - r.y), z(d.z - r.z) {
    r2 = x * x + y * y + z * z;
  }
  __device__ __forceinline__ double gauss(double alpha, double, double rcut2, bool) const {
    const double e = exp(-(alpha * r2));
    return r2 <= rcut2 ? e : 0.0;
  }
};

// Shells of one angular momentum that share their images' displacements: as many as fit the
// columns and the registers.
template <int L> constexpr int group_shells() { return L == 0 ? 8 : (L == 1 ? 3 : (L == 2 ? 2 : 1)); }

// Class sums of ns shells (functions [m0, m0 + nm) of each) over a stretch [t0, t1) of the list
// in order of class. A class that may continue from the stretch before (the first one of a
// stretch) goes to `edge`, its number to *edge_cls; the others are this warp's alone. The
// shells come by falling reach, np[s] images each.
template <typename T, int L, typename GetRec, typename GetOrder>
__device__ __forceinline__ void class_sums(const ChiShell* shells, const int* np, int ns,
                                           const Disp<T>& d, int t0, int t1, int m0, int nm,
                                           const GetRec& rec, const GetOrder& order, T* cols,
                                           int col_rows, T* edge, int* edge_cls, int lane) {
  constexpr int NM = 2 * L + 1, NS = group_shells<L>();
  T acc[NS][NM], alpha[NS], alpha_lo[NS], rcut2[NS];
  int n[NS];
  bool exact = false;   // one exact exponent: all of the group's
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    const int q = min(s, ns - 1);
    exact = exact || shells[q].exact;
    n[s] = s < ns ? np[s] : 0;
    if constexpr (sizeof(T) == 4) {
      alpha[s] = shells[q].alpha;
      alpha_lo[s] = shells[q].alpha_lo;
      rcut2[s] = shells[q].rcut2;
    } else {
      alpha[s] = shells[q].alpha_d;
      alpha_lo[s] = T(0);
      rcut2[s] = shells[q].rcut2_d;
    }
#pragma unroll
    for (int m = 0; m < NM; ++m) acc[s][m] = T(0);
  }
  int cur = -1, first = -1;
  auto close = [&]() {
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      if (s >= ns) break;
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        const int c = s * nm + m - m0;
        if (m >= m0 && m < m0 + nm) {
          T* o = cur == first ? edge + c * 32 : cols + ((size_t)c * col_rows + cur) * 32;
          o[lane] = acc[s][m];
        }
        acc[s][m] = T(0);
      }
    }
  };
  int next = t0 < t1 ? order(t0) : 0;
  for (int t = t0; t < t1; ++t) {
    const int j = next;
    if (t + 1 < t1) next = order(t + 1);
    if (j >= n[0]) continue;   // past every shell's reach (uniform)
    const Rec<T> r = rec(j);
    if (r.cls != cur) {
      if (cur >= 0) close();
      cur = r.cls;
      if (first < 0) first = cur;
    }
    const Geo<T> g(d, r, exact);
    T P[NM];
    ao::solid<T, L>(g.x, g.y, g.z, P);
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      if (j < n[s]) {
        const T e = g.gauss(alpha[s], alpha_lo[s], rcut2[s], exact);
#pragma unroll
        for (int m = 0; m < NM; ++m) acc[s][m] += P[m] * e;
      }
    }
  }
  if (cur >= 0) close();
  if (lane == 0) *edge_cls = first;
}

// chi of the blocks [blk0, blk0 + gridDim.x) for one atom; a lane is a grid point. Every Gaussian
// is evaluated once for all k. The atom's wide shells come first (they are a prefix of its
// shells): the CTA takes a few of one angular momentum, which share their images' distances,
// each warp a stretch of the images, then a warp per AO transforms. The phases of a narrow
// shell's few images are applied one by one.
// What bounds it: the stores at many k-points, the Gaussians at few. Phases times class sums
// (a dense product over classes) instead of the transform took 43 ms per pass at 64 k, 350
// AOs, 60^3: each broadcast phase costs the load path as much as a full vector.
// FOLD: meshes of up to kFold classes (fold_shell alone, CTAs of kFoldWarps: with fewer registers
// more of them fit; at six CTAs the phases' kernel spills and is 3 % slower).
template <typename T, int KS, int KL, bool FOLD>
__global__ void __launch_bounds__(32 * (FOLD ? kFoldWarps : kWarps),
                                  !FOLD ? 2 : (sizeof(T) == 8 ? 4 : (KS == 1 ? 6 : 5)))
chi_kernel(Params p, cplx_t<T>* __restrict__ chi, int blk0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ T edge[kWarps][kCols][32];
  __shared__ int edge_cls[kWarps];
  T* buf = reinterpret_cast<T*>(smem_raw);   // entry rows of the warps, or columns
  int* eclss = reinterpret_cast<int*>(buf + p.buf_rows * 32);
  Rec<T>* recs = reinterpret_cast<Rec<T>*>(eclss + kWarps * kRows);
  int* lnp = reinterpret_cast<int*>(recs + p.lsm);   // images << 2 | l of the atom's shells
  unsigned short* ord = reinterpret_cast<unsigned short*>(lnp + p.a.nsa);
  const int blk = blk0 + blockIdx.x, a = blockIdx.y;
  const size_t ab = (size_t)a * p.a.nblk + blk;
  const int nact = p.nsh[ab];
  if (nact == 0) return;
  const int s0 = p.a.atom_shell0[a];
  const unsigned short* pre = p.a.bpre + ab * p.a.nsa;
  const size_t list0 = ab * p.a.lmax;
  const int n_all = pre[p.shells[s0].orig - s0];   // the widest shell's images
  const int* cls = p.cls + (size_t)p.t0i[ab] * p.a.nimg;
  const bool in_smem = p.lsm > 0;
  for (int x = threadIdx.x; x < nact; x += blockDim.x) {
    const ChiShell& sh = p.shells[s0 + x];
    lnp[x] = pre[sh.orig - s0] << 2 | sh.l;
  }
  if (in_smem) {
    for (int j = threadIdx.x; j < n_all; j += blockDim.x) {
      recs[j] = load_rec<T>(p, list0, cls, j);
      if (p.order) ord[j] = p.order[list0 + j];
    }
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  bool valid;
  long long q;
  const long long n = ao::block_point(p.a, blk, lane, &valid, &q);
  Disp<T> d;
  ao::load_disp(p.a, a, n, &d);
  const int* aoff = p.aoff + (size_t)blk * (p.a.natm + 1);
  const int kstride = 32 * aoff[p.a.natm];
  const size_t base0 = (size_t)(p.boff[blk] * p.a.nk + aoff[a]) * 32;
  // (real values: the same offsets in T)
  cplx_t<T>* base = p.signs ? reinterpret_cast<cplx_t<T>*>(reinterpret_cast<T*>(chi) + base0)
                            : chi + base0;
  auto rec = [&](int j) -> Rec<T> { return in_smem ? recs[j] : load_rec<T>(p, list0, cls, j); };
  auto order = [&](int t) -> int { return in_smem ? ord[t] : p.order[list0 + t]; };
  __shared__ ChiShell gsh[8];
  __shared__ int gnp[8], gidx[8], gslot[kCols], gns, gm0, gnm, gnext, gl;
  int wide = 0;   // wide shells (a prefix)
  if constexpr (!FOLD) if (p.ncol > 0) {
    while (wide < nact && lnp[wide] >> 2 >= kWide) ++wide;
    // Groups of one angular momentum, in turn over the CTAs of the (block, atom)
    const int t0 = n_all * warp / nw, t1 = n_all * (warp + 1) / nw;
    int at = 0, m0 = 0, l = 0;   // next shell to look at, its first function
    for (int group = 0; l < 4; ++group) {
      __syncthreads();   // the group before is done with the columns and the list
      if (threadIdx.x == 0) {
        int ns = 0, x = at;
        const int full = 2 * l + 1, nm = min(full - m0, p.ncol);   // functions of each shell
        const int most = max(1, min(l == 0 ? group_shells<0>() : (l == 1 ? group_shells<1>() :
                                    (l == 2 ? group_shells<2>() : 1)), p.ncol / full));
        for (; x < wide && ns < most; ++x) {
          if ((lnp[x] & 3) != l) continue;
          gnp[ns] = lnp[x] >> 2;
          gidx[ns++] = s0 + x;
          if (m0 + nm < full) break;   // a part of one shell: the rest of it next
        }
        gns = ns;
        gm0 = m0;
        gnm = nm;
        gl = l;
        gnext = ns > 0 && m0 + nm < full ? x : -1 - x;
      }
      __syncthreads();
      const int ns = gns, nm = gnm, gm = gm0;
      if (gnext >= 0) {   // stay at this shell
        at = gnext;
        m0 = gm + nm;
      } else {
        at = -1 - gnext;
        m0 = 0;
        if (ns == 0) {    // no more of this angular momentum
          ++l;
          at = 0;
          --group;
          continue;
        }
      }
      if (group % gridDim.z != blockIdx.z) continue;
      const int cols = ns * nm;
      if ((int)threadIdx.x < ns) {
        const ChiShell sh = p.shells[gidx[threadIdx.x]];
        gsh[threadIdx.x] = sh;
        for (int m = 0; m < nm; ++m) gslot[threadIdx.x * nm + m] = sh.slot + gm + m;
      }
      for (int c = 0; c < cols; ++c)   // the classes' rows (the transform fills the others)
        for (int x = threadIdx.x; x < p.ncls * 32; x += blockDim.x)
          buf[(size_t)c * p.col_rows * 32 + x] = T(0);
      __syncthreads();
      T* eb = &edge[warp][0][0];
      int* ec = &edge_cls[warp];
      switch (gl) {
        case 0: class_sums<T, 0>(gsh, gnp, ns, d, t0, t1, gm, nm, rec, order, buf, p.col_rows, eb, ec, lane); break;
        case 1: class_sums<T, 1>(gsh, gnp, ns, d, t0, t1, gm, nm, rec, order, buf, p.col_rows, eb, ec, lane); break;
        case 2: class_sums<T, 2>(gsh, gnp, ns, d, t0, t1, gm, nm, rec, order, buf, p.col_rows, eb, ec, lane); break;
        default: class_sums<T, 3>(gsh, gnp, ns, d, t0, t1, gm, nm, rec, order, buf, p.col_rows, eb, ec, lane); break;
      }
      __syncthreads();
      for (int x = warp; x < cols; x += nw) {   // a warp per AO: the stretches' edges in
        T* col = buf + (size_t)x * p.col_rows * 32;   // order, then the transform
        for (int w = 0; w < nw; ++w) {
          const int c = edge_cls[w];
          if (c >= 0) col[c * 32 + lane] += edge[w][x][lane];
        }
        mesh_dft<T>(p, col, base + 32 * (size_t)gslot[x], kstride, lane);
      }
    }
    __syncthreads();
  }
  T* ent = buf + warp * kRows * 32;
  int* ecls = eclss + warp * kRows;
  const int kz = FOLD ? 1 : p.kslices, per = (p.a.nk + 8 * kz - 1) / (8 * kz) * 8;
  for (int it = warp + nw * blockIdx.z; it < (nact - wide) * kz; it += nw * gridDim.z) {
    const int s = wide + it / kz, ka = per * (it % kz), kb = min(p.a.nk, ka + per);
    const ChiShell sh = p.shells[s0 + s];
    const int np = pre[sh.orig - s0];
    cplx_t<T>* out = p.signs ? reinterpret_cast<cplx_t<T>*>(reinterpret_cast<T*>(base) + 32 * sh.slot)
                             : base + 32 * (size_t)sh.slot;
    if constexpr (FOLD) {
      switch (sh.l) {
        case 0: fold_shell<T, 0, KS>(p, sh, d, np, rec, ent, ecls, out, kstride, lane); break;
        case 1: fold_shell<T, 1, KS>(p, sh, d, np, rec, ent, ecls, out, kstride, lane); break;
        case 2: fold_shell<T, 2, KL>(p, sh, d, np, rec, ent, ecls, out, kstride, lane); break;
        default: fold_shell<T, 3, KL>(p, sh, d, np, rec, ent, ecls, out, kstride, lane); break;
      }
    } else {
      switch (sh.l) {
        case 0: narrow_shell<T, 0, KS>(p, sh, d, np, rec, ent, ecls, out, kstride, lane, ka, kb); break;
        case 1: narrow_shell<T, 1, KS>(p, sh, d, np, rec, ent, ecls, out, kstride, lane, ka, kb); break;
        case 2: narrow_shell<T, 2, KL>(p, sh, d, np, rec, ent, ecls, out, kstride, lane, ka, kb); break;
        default: narrow_shell<T, 3, KL>(p, sh, d, np, rec, ent, ecls, out, kstride, lane, ka, kb); break;
      }
    }
  }
  if (blockIdx.z == 0 && warp == nw - 1) {   // padding slots of the atom's last group
    const ChiShell& last = p.shells[s0 + nact - 1];
    for (int x = last.slot + 2 * last.l + 1; x < aoff[a + 1] - aoff[a]; ++x)
      for (int k = 0; k < p.a.nk; ++k) {
        const size_t o = (size_t)k * kstride + 32 * x + lane;
        if (p.signs) reinterpret_cast<T*>(base)[o] = T(0);
        else base[o] = cplx_t<T>{T(0), T(0)};
      }
  }
}

// chi on meshes of many k-points that the transform does not take (shifted meshes, other axis
// lengths), FP32: neighbouring shells of an atom, up to kDense AOs, at once. The warps evaluate a
// batch of images into shared memory, then share the k-points, each with the sums of KD of them
// and all kDense AOs in registers, so that a phase serves kDense products and chi is written
// once per batch (every batch but the first adds). A group's shells have nearly the same reach;
// the images that one lacks are zeros, and what its unused columns hold is not stored.
// What bounds it: the phases (four wavefronts of the load path per 16 bytes that all lanes read) and
// the products, about equally by count. One shell and warp at a time, a phase per product and chi read
// and written again every 8 to 56 images: orbitals of 104 AOs at 9^3 k, 24^3, 23.0 ms against 8.1
// (15.1 when they were summed without tiles).
constexpr int kDense = 8;      // AOs of a group
constexpr int KD = 4;          // k-points per warp
// Least k-points of a mesh that takes it. Orbitals at 36^3, 104 and 350 AOs, narrow_shell against
// this kernel: 12 k 642 / 719 and 1992 / 2355 us, 16 k 784 / 783 and 2498 / 2623, 20 k 964 / 953 and
// 3178 / 3276, 27 k 1538 / 1151 and 5190 / 4043; at 12^3 it is ahead from 9 k on.
constexpr int kDenseK = 16;
constexpr int kDenseImages = 96;   // most images of a batch (1 KB each; two CTAs per SM)
__global__ void __launch_bounds__(32 * kWarps, 2)
chi_dense_kernel(Params p, float2* __restrict__ chi, int blk0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* val = reinterpret_cast<float*>(smem_raw);   // [image][column][lane]
  int* ecls = reinterpret_cast<int*>(val + (size_t)p.batch * kDense * 32);
  int* lnp = ecls + p.batch;                         // images << 2 | l of the atom's shells
  const int blk = blk0 + blockIdx.x, a = blockIdx.y;
  const size_t ab = (size_t)a * p.a.nblk + blk;
  const int nact = p.nsh[ab];
  if (nact == 0) return;
  const int s0 = p.a.atom_shell0[a];
  const unsigned short* pre = p.a.bpre + ab * p.a.nsa;
  const size_t list0 = ab * p.a.lmax;
  const int* cls = p.cls + (size_t)p.t0i[ab] * p.a.nimg;
  for (int x = threadIdx.x; x < nact; x += blockDim.x) {
    const ChiShell& sh = p.shells[s0 + x];
    lnp[x] = pre[sh.orig - s0] << 2 | sh.l;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  bool valid;
  long long q;
  const long long n = ao::block_point(p.a, blk, lane, &valid, &q);
  Disp<float> d;
  ao::load_disp(p.a, a, n, &d);
  const int* aoff = p.aoff + (size_t)blk * (p.a.natm + 1);
  const int kstride = 32 * aoff[p.a.natm];
  float2* base = chi + (size_t)(p.boff[blk] * p.a.nk + aoff[a]) * 32 + lane;
  // the CTA's k-points
  const int nk = p.a.nk, per = (nk + KD * (int)gridDim.z - 1) / (KD * (int)gridDim.z) * KD;
  const int ka = min(nk, per * (int)blockIdx.z), kb = min(nk, ka + per);
  const float2* ph = reinterpret_cast<const float2*>(p.phase);
  int last = 0;   // slots of the atom so far
  for (int s = 0; s < nact;) {
    int e = s, cols = 0;   // the group's shells [s, e)
    while (e < nact && cols + 2 * (lnp[e] & 3) + 1 <= kDense) cols += 2 * (lnp[e++] & 3) + 1;
    const int slot = p.shells[s0 + s].slot, images = lnp[s] >> 2;
    for (int j0 = 0; j0 < images; j0 += p.batch) {
      const int ne = min(p.batch, images - j0);
      for (int j = warp; j < ne; j += kWarps) {
        const Rec<float> r = load_rec<float>(p, list0, cls, j0 + j);
        float* o = val + (size_t)j * kDense * 32 + lane;
        for (int x = s; x < e; ++x) {
          const ChiShell& sh = p.shells[s0 + x];
          const bool in = j0 + j < lnp[x] >> 2;   // (past the shell's radius eval gives 0)
          auto put = [&](auto L) {
            constexpr int l = decltype(L)::value;
            float v[2 * l + 1];
            if (in) eval<l>(sh, d, r, v);
#pragma unroll
            for (int m = 0; m < 2 * l + 1; ++m) o[32 * m] = in ? v[m] : 0.f;
            o += 32 * (2 * l + 1);
          };
          switch (lnp[x] & 3) {
            case 0: put(std::integral_constant<int, 0>{}); break;
            case 1: put(std::integral_constant<int, 1>{}); break;
            case 2: put(std::integral_constant<int, 2>{}); break;
            default: put(std::integral_constant<int, 3>{}); break;
          }
        }
        if (lane == 0) ecls[j] = r.cls;
      }
      __syncthreads();
      for (int k0 = ka + KD * warp; k0 < kb; k0 += KD * kWarps) {
        float xr[KD][kDense], xi[KD][kDense];
#pragma unroll
        for (int b = 0; b < KD; ++b)
#pragma unroll
          for (int c = 0; c < kDense; ++c) xr[b][c] = xi[b][c] = 0.f;
        // whole groups of KD: the table's rows are zero past the last k-point
#pragma unroll 2
        for (int j = 0; j < ne; ++j) {
          const float4* row = reinterpret_cast<const float4*>(ph + (size_t)ecls[j] * p.nkp + k0);
          const float* v = val + (size_t)j * kDense * 32 + lane;
          float4 w[KD / 2];
#pragma unroll
          for (int b = 0; b < KD / 2; ++b) w[b] = __ldg(row + b);
#pragma unroll
          for (int c = 0; c < kDense; ++c) {
            const float x = v[32 * c];
#pragma unroll
            for (int b = 0; b < KD / 2; ++b) {
              xr[2 * b][c] += w[b].x * x;
              xi[2 * b][c] += w[b].y * x;
              xr[2 * b + 1][c] += w[b].z * x;
              xi[2 * b + 1][c] += w[b].w * x;
            }
          }
        }
#pragma unroll
        for (int b = 0; b < KD; ++b) {
          if (k0 + b >= kb) break;
          float2* o = base + (size_t)(k0 + b) * kstride + 32 * (size_t)slot;
#pragma unroll
          for (int c = 0; c < kDense; ++c) {
            if (c >= cols) break;
            float2 y = make_float2(xr[b][c], xi[b][c]);
            if (j0 > 0) {
              const float2 u = o[32 * c];
              y.x += u.x;
              y.y += u.y;
            }
            o[32 * c] = y;
          }
        }
      }
      __syncthreads();   // the batch's values are free
    }
    last = slot + cols;
    s = e;
  }
  for (int x = last; x < aoff[a + 1] - aoff[a]; ++x)   // padding slots of the atom's last group
    for (int k = ka + warp; k < kb; k += kWarps)
      base[(size_t)k * kstride + 32 * (size_t)x] = make_float2(0.f, 0.f);
}

// List positions of every (atom, block) in order of class, once at plan creation: a warp per
// list, which appends the images of one class after another.
__global__ void __launch_bounds__(256)
order_kernel(Params p, unsigned short* __restrict__ order) {
  const int ab = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int a = ab / p.a.nblk, s0 = p.a.atom_shell0[min(a, p.a.natm - 1)];
  if (a >= p.a.natm || p.nsh[ab] == 0) return;
  const size_t list0 = (size_t)ab * p.a.lmax;
  const int n = p.a.bpre[(size_t)ab * p.a.nsa + p.shells[s0].orig - s0];
  const int* cls = p.cls + (size_t)p.t0i[ab] * p.a.nimg;
  int at = 0;
  for (int c = 0; c < p.ncls && at < n; ++c)
    for (int j0 = 0; j0 < n; j0 += 32) {
      const int j = j0 + lane;
      const bool in = j < n && cls[p.a.blist[list0 + j]] == c;
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (in) order[list0 + at + __popc(m & ((1u << lane) - 1u))] = (unsigned short)j;
      at += __popc(m);
    }
}

// chi is read once: past L1, which holds what is shared (coefficients, orbital fields).
__device__ __forceinline__ float2 stream_ld(const float2* p) {
  float2 v;
  asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ double2 stream_ld(const double2* p) {
  double2 v;
  asm volatile("ld.global.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
  return v;
}

__device__ __forceinline__ float stream_ld(const float* p) {
  float v;
  asm volatile("ld.global.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double stream_ld(const double* p) {
  double v;
  asm volatile("ld.global.L1::no_allocate.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}

// chi as the products read it: real on meshes whose phases are signs (half the bytes and half
// the products)
template <typename T, bool REAL> using chi_t = std::conditional_t<REAL, T, cplx_t<T>>;

// t += c x; in FP32 the coefficient is a hi/lo pair
__device__ __forceinline__ void cmac(const double2& c, const double2& x, double2& t) {
  t.x += c.x * x.x - c.y * x.y;
  t.y += c.x * x.y + c.y * x.x;
}
__device__ __forceinline__ void cmac(const float4& c, const float2& x, float2& t) {
  t.x = fmaf(c.x, x.x, fmaf(-c.y, x.y, fmaf(c.z, x.x, fmaf(-c.w, x.y, t.x))));
  t.y = fmaf(c.x, x.y, fmaf(c.y, x.x, fmaf(c.z, x.y, fmaf(c.w, x.x, t.y))));
}

__device__ __forceinline__ void cmac(const double2& c, double x, double2& t) {
  t.x += c.x * x;
  t.y += c.y * x;
}
__device__ __forceinline__ void cmac(const float4& c, float x, float2& t) {
  t.x = fmaf(c.x, x, fmaf(c.z, x, t.x));
  t.y = fmaf(c.y, x, fmaf(c.w, x, t.y));
}

// psi_ik at NB consecutive blocks per warp: kPad AOs are summed on their own before they join
// the orbital's sum, so that few roundings happen at its full size. In FP32 a coefficient,
// the same for every lane, costs the load path as much as a value per lane: up to four
// orbitals take two blocks (64 k, 200 AOs, 48^3, nocc 4: orbitals and AOs 5.5 -> 5.0 ms); with
// eight the wider tile's registers cost what it saves (350 AOs, 8 k, 60^3: 1.52 against 1.50 ms).
template <typename T, int NI, bool REAL> constexpr int orb_blocks() {
  return sizeof(T) == 4 && (REAL || NI == 4) ? 2 : 1;
}
template <typename T, int NI, int NB, bool REAL>
__global__ void __launch_bounds__(128)
orb_kernel(Params p, const chi_t<T, REAL>* __restrict__ chi, const typename CsT<T>::type* __restrict__ cs,
           cplx_t<T>* __restrict__ psi, int blk0, int nb, int i0, int periodic) {
  const int w = NB * (blockIdx.x * 4 + (threadIdx.x >> 5));
  if (w >= nb) return;
  const int k = blockIdx.y, lane = threadIdx.x & 31;
  const int nocc = p.a.nocc, blk = blk0 + w, nlast = min(NB, nb - w) - 1;
  using X = chi_t<T, REAL>;
  const int* aoff[NB];
  const X* x0[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) {   // past the last block: the last one again, not stored
    const int q = blk + min(b, nlast);
    aoff[b] = p.aoff + (size_t)q * (p.a.natm + 1);
    x0[b] = chi + ((size_t)p.boff[q] * p.a.nk + (size_t)k * aoff[b][p.a.natm]) * 32 + lane;
  }
  cplx_t<T> acc[NB][NI];
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int i = 0; i < NI; ++i) acc[b][i] = cplx_t<T>{T(0), T(0)};
  // slots [s, s + kPad) of an atom for the blocks [b0, b1) of the warp
  auto group = [&](const X* (&xa)[NB], const typename CsT<T>::type* ca, int s, auto B0,
                   auto B1) {
    constexpr int b0 = decltype(B0)::value, b1 = decltype(B1)::value;
    X x[NB][kPad];
#pragma unroll
    for (int b = b0; b < b1; ++b)
#pragma unroll
      for (int u = 0; u < kPad; ++u) x[b][u] = stream_ld(xa[b] + (size_t)(s + u) * 32);
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      if (i0 + i >= nocc) break;
      cplx_t<T> t[NB];
#pragma unroll
      for (int b = b0; b < b1; ++b) t[b] = cplx_t<T>{T(0), T(0)};
#pragma unroll
      for (int u = 0; u < kPad; ++u) {
        const typename CsT<T>::type c = __ldg(ca + (size_t)(s + u) * nocc + i);
#pragma unroll
        for (int b = b0; b < b1; ++b) cmac(c, x[b][u], t[b]);
      }
#pragma unroll
      for (int b = b0; b < b1; ++b) {
        acc[b][i].x += t[b].x;
        acc[b][i].y += t[b].y;
      }
    }
  };
  using Zero = std::integral_constant<int, 0>;
  using One = std::integral_constant<int, 1>;
  using All = std::integral_constant<int, NB>;
  for (int a = 0; a < p.a.natm; ++a) {
    int n[NB], both = 1 << 30;
    const X* xa[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      n[b] = aoff[b][a + 1] - aoff[b][a];
      xa[b] = x0[b] + (size_t)aoff[b][a] * 32;
      both = min(both, n[b]);
    }
    const typename CsT<T>::type* ca = cs + ((size_t)k * p.nslots + p.slot0[a]) * nocc + i0;
#pragma unroll 2
    for (int s = 0; s < both; s += kPad) group(xa, ca, s, Zero{}, All{});
    if constexpr (NB == 2) {   // what only one of the blocks has
      for (int s = both; s < n[0]; s += kPad) group(xa, ca, s, Zero{}, One{});
      for (int s = both; s < n[1]; s += kPad) group(xa, ca, s, One{}, All{});
    }
  }
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if (b > nlast) break;
    bool valid;
    long long q;
    const long long n = ao::block_point(p.a, blk + b, lane, &valid, &q);
    if (!valid) continue;
    if (periodic) {   // u = e^{-ik.r} psi
      const int N = p.a.N[0];
      const int n3 = (int)(n % N), n2 = (int)(n / N % N), n1 = (int)(n / ((long long)N * N));
      const cplx_t<T> ph = ao::point_phase<T>(p.a.kint + 3 * k, p.a.D[0], p.a.D[1], p.a.D[2], N,
                                              n1, n2, n3, -1);
#pragma unroll
      for (int i = 0; i < NI; ++i) acc[b][i] = dev::cmul<T>(acc[b][i], ph);
    }
#pragma unroll
    for (int i = 0; i < NI; ++i)
      if (i0 + i < nocc) psi[((size_t)k * nocc + i0 + i) * p.a.fs + q] = acc[b][i];
  }
}

// Sums over the lanes of a warp of NV values per lane, by halving: after the exchange over lane
// bit b each lane keeps half of its values. Lane l ends with the sums of the values
// l (NV / 32) + j. NV words of shared memory per warp.
//
// FP64 values are added as they are. FP32 values are added as 64-bit integers in units of
// 2^-57 of the largest lane's power of two, value by value: of a lane's 24 bits only those below
// that unit are lost, so the sums are those of FP64 or better, and integer additions run at full
// rate, where an SM adds two FP64 values per cycle (45^3, 8 k, nocc 8, items of 16 blocks: a build
// 3.42 ms with FP64 sums of the lanes, 3.31 with these).
__device__ __forceinline__ long long lane_fixed(unsigned bits, int e) {   // e: largest lane's exponent
  const int x = bits >> 23 & 255;
  const unsigned m = (bits & 0x7fffffu) | (x ? 0x800000u : 0u);
  const unsigned long long q = ((unsigned long long)m << 40) >> min(7 + e - max(x, 1), 63);
  return (int)bits < 0 ? -(long long)q : (long long)q;
}
template <int NV>
__device__ __forceinline__ void halve_lanes(const double (&v)[NV], double (&out)[NV / 32], int lane,
                                            unsigned*) {
  double w[NV];
#pragma unroll
  for (int j = 0; j < NV; ++j) w[j] = v[j];
#pragma unroll
  for (int step = 0; step < 5; ++step) {
    const int half = NV >> (step + 1);
    const bool up = (lane >> (4 - step)) & 1;
#pragma unroll
    for (int j = 0; j < half; ++j) {
      const double mine = up ? w[j + half] : w[j], other = up ? w[j] : w[j + half];
      w[j] = mine + __shfl_xor_sync(0xffffffffu, other, 16 >> step);
    }
  }
#pragma unroll
  for (int j = 0; j < NV / 32; ++j) out[j] = w[j];
}
template <int NV>
__device__ __forceinline__ void halve_lanes(const float (&v)[NV], double (&out)[NV / 32], int lane,
                                            unsigned* top) {
  constexpr unsigned kAll = 0xffffffffu, kInf = 0x7f800000u;
  // the largest lane's bits of value j go to top; where a lane holds an infinity or NaN, the sum's
  auto largest = [&](int j) {
    unsigned t = __reduce_max_sync(kAll, __float_as_uint(v[j]) & 0x7fffffffu);
    if (t >= kInf) {   // (uniform)
      double s = v[j];
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kAll, s, o);
      t = __float_as_uint((float)s);
    }
    if (lane == 0) top[j] = t;
    return (int)max(t >> 23 & 255u, 1u);
  };
  long long w[NV / 2];
  const bool up0 = (lane >> 4) & 1;
#pragma unroll
  for (int j = 0; j < NV / 2; ++j) {
    const int e0 = largest(j), e1 = largest(j + NV / 2), e = up0 ? e1 : e0;
    const float mine = up0 ? v[j + NV / 2] : v[j], other = up0 ? v[j] : v[j + NV / 2];
    w[j] = lane_fixed(__float_as_uint(mine), e) +
           lane_fixed(__float_as_uint(__shfl_xor_sync(kAll, other, 16)), e);
  }
#pragma unroll
  for (int step = 1; step < 5; ++step) {
    const int half = NV >> (step + 1);
    const bool up = (lane >> (4 - step)) & 1;
#pragma unroll
    for (int j = 0; j < half; ++j) {
      const long long mine = up ? w[j + half] : w[j], other = up ? w[j] : w[j + half];
      w[j] = mine + __shfl_xor_sync(kAll, other, 16 >> step);
    }
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < NV / 32; ++j) {
    const unsigned t = top[lane * (NV / 32) + j];
    const int e = (int)max(t >> 23 & 255u, 1u);   // the unit is 2^(e - 183)
    out[j] = (t & 0x7fffffffu) >= kInf ? (double)__uint_as_float(t)
                                       : (double)w[j] * __hiloint2double((e + 840) << 20, 0);
  }
}

// Partial sums over r of conj(chi) F: a warp takes kPad AOs of an atom over a run of the blocks
// they reach (work items, made with the plan), sums per lane in the working precision, then
// over the lanes exactly or in FP64. sum_kernel adds the items in a fixed order, so that the result
// does not depend on the order in which they ran. What bounds it: issue and the load path, both
// about half busy (60^3, 8 k, 94 AOs, real tiles: 0.51 ms); evaluating the AOs at each k-point
// instead made the contraction over half of a build at 8 k, 104 AOs, 36^3.
template <typename T, int NI, bool REAL>
__global__ void __launch_bounds__(256, 2)
con_kernel(Params p, const chi_t<T, REAL>* __restrict__ chi, const cplx_t<T>* __restrict__ F,
           int item0, int nitems, int i0) {
  const int w = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (w >= nitems) return;
  const int k = blockIdx.y, lane = threadIdx.x & 31;
  const int4 it = p.items[item0 + w];
  const int nocc = p.a.nocc;
  const cplx_t<T>* f0 = F + ((size_t)k * nocc + i0) * p.a.fs;
  constexpr int NV = 2 * kPad * NI;
  T acc[NV];   // [slot][i][re, im]
#pragma unroll
  for (int j = 0; j < NV; ++j) acc[j] = T(0);
#pragma unroll 1
  for (int b = 0; b < it.w; ++b) {
    const int blk = p.border[it.z + b];
    const int* aoff = p.aoff + (size_t)blk * (p.a.natm + 1);
    const chi_t<T, REAL>* x0 = chi + ((size_t)p.boff[blk] * p.a.nk + (size_t)k * aoff[p.a.natm] +
                                      aoff[it.x] + it.y) * 32 + lane;
    chi_t<T, REAL> x[kPad];
#pragma unroll
    for (int u = 0; u < kPad; ++u) x[u] = stream_ld(x0 + 32 * u);
    bool valid;
    long long q;
    ao::block_point(p.a, blk, lane, &valid, &q);
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      cplx_t<T> y{T(0), T(0)};
      if (valid && i0 + i < nocc) y = __ldg(f0 + (size_t)i * p.a.fs + q);
#pragma unroll
      for (int u = 0; u < kPad; ++u) {   // conj(x) y
        T& re = acc[2 * (u * NI + i)];
        T& im = acc[2 * (u * NI + i) + 1];
        if constexpr (REAL) {
          re += x[u] * y.x;
          im += x[u] * y.y;
        } else {
          re += x[u].x * y.x + x[u].y * y.y;
          im += x[u].x * y.y - x[u].y * y.x;
        }
      }
    }
  }
  double sum[NV / 32];
  __shared__ unsigned top[8][NV];
  halve_lanes<NV>(acc, sum, lane, top[threadIdx.x >> 5]);
  // lane l holds the values l (NV / 32) + j
  double* o = p.part + ((size_t)k * nitems + w) * NV + lane * (NV / 32);
#pragma unroll
  for (int j = 0; j < NV / 32; ++j) o[j] = sum[j];
}

// out[k][mu][i] = scale N_mu (sum of the items), or += after the first chunk: one CTA per (slot
// group, k), a thread per value and every kSumSplit-th run, the shares added in order.
constexpr int kSumSplit = 8;
template <int NI>
__global__ void __launch_bounds__(2 * kPad * NI * kSumSplit)
sum_kernel(Params p, double2* __restrict__ out, double2* __restrict__ copy, int row_of0, int nitems, int i0, double scale, int add) {
  constexpr int NV = 2 * kPad * NI;
  __shared__ double share[kSumSplit][NV];
  const int v = threadIdx.x % NV, z = threadIdx.x / NV, k = blockIdx.y;
  int a = 0;
  while ((int)blockIdx.x * kPad >= p.slot0[a + 1]) ++a;
  const int g = (int)blockIdx.x - p.slot0[a] / kPad;
  const int2 ro = p.rows_of[row_of0 + a];
  const double* src = p.part + (size_t)k * nitems * NV + v;
  double t = 0.0;
#pragma unroll 4
  for (int r = z; r < ro.y; r += kSumSplit) {
    const int2 row = p.rows[ro.x + r];
    if (g < row.y) t += src[(size_t)(row.x + g) * NV];
  }
  share[z][v] = t;
  __syncthreads();
  if (z != 0) return;
  const int u = v / (2 * NI), i = (v / 2) % NI;
  const int mu = p.slot_ao[blockIdx.x * kPad + u];
  if (mu < 0 || i0 + i >= p.a.nocc) return;
#pragma unroll
  for (int y = 1; y < kSumSplit; ++y) t += share[y][v];
  const size_t at = 2 * (((size_t)k * p.a.nao + mu) * p.a.nocc + i0 + i) + (v & 1);
  double* dst = reinterpret_cast<double*>(out) + at;
  t *= scale * p.ao_norm[mu];
  if (add) t += *dst;
  *dst = t;
  if (copy) reinterpret_cast<double*>(copy)[at] = t;
}

// Coefficients factor N_mu X^k_{mu i} in slot order, formed in FP64 (hi/lo floats in FP32), 0
// in padding slots.
template <typename T>
__global__ void slot_c_kernel(const double2* __restrict__ X, const double* __restrict__ nrm,
                              const int* __restrict__ slot_ao, typename CsT<T>::type* __restrict__ out,
                              int nao, int nocc, int nslots, long long n, double factor) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e % nocc);
    const long long ks = e / nocc;
    const int mu = slot_ao[ks % nslots];
    double x = 0.0, y = 0.0;
    if (mu >= 0) {
      const double2 c = X[((ks / nslots) * nao + mu) * nocc + i];
      const double s = factor * nrm[mu];
      x = s * c.x;
      y = s * c.y;
    }
    if constexpr (sizeof(T) == 4) {
      const float xh = (float)x, yh = (float)y;
      out[e] = make_float4(xh, yh, (float)(x - (double)xh), (float)(y - (double)yh));
    } else {
      out[e] = make_double2(x, y);
    }
  }
}

Params params(const Plan& p) {
  const ChiTables& t = *p.chi;
  Params q;
  q.a = p.ao_params();
  q.shells = t.shells;
  q.slot0 = t.slot0;
  q.slot_ao = t.slot_ao;
  q.nsh = t.nsh;
  q.aoff = t.aoff;
  q.boff = t.boff;
  q.t0i = t.t0i;
  q.cls = t.cls;
  q.order = t.order;
  q.phase = t.phase;
  q.items = t.items;
  q.border = t.border;
  q.rows = t.rows;
  q.rows_of = t.rows_of;
  q.part = t.part;
  q.row_scale = t.row_scale;
  q.ao_norm = p.ao_norm;
  q.nslots = t.nslots;
  q.ncls = t.ncls;
  q.nkp = t.nkp;
  q.lsm = t.lsm;
  q.parts = t.parts;
  q.kidx = t.kidx;
  q.ncol = t.ncol;
  q.col_rows = t.col_rows;
  q.buf_rows = t.buf_rows;
  q.warps = t.warps;
  q.signs = t.signs;
  q.batch = t.batch;
  q.kslices = t.kslices;
  return q;
}

template <typename T> size_t chi_smem(int buf_rows, int lsm, int nsa) {
  return (size_t)buf_rows * 32 * sizeof(T) + (size_t)(kWarps * kRows + nsa) * sizeof(int) +
         (size_t)lsm * (sizeof(Rec<T>) + sizeof(unsigned short));
}

size_t dense_smem(int batch, int nsa) {
  return (size_t)batch * (kDense * 32 * sizeof(float) + sizeof(int)) + (size_t)nsa * sizeof(int);
}

// A kernel's dynamic shared memory limit on each device, raised where a launch needs more.
struct SmemLimit {
  std::mutex mu;
  size_t have[kMaxDevices] = {};
  template <typename K>
  cudaError_t raise(K kernel, int device, size_t bytes) {
    std::lock_guard<std::mutex> lock(mu);
    size_t& h = have[(device >= 0 && device < kMaxDevices) ? device : 0];
    if (bytes <= h) return cudaSuccess;
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) h = bytes;
    return e;
  }
};

template <typename T, int KS, int KL, bool FOLD>
cudaError_t run_chi_as(const Plan& p, const Params& q, const ChiChunk& c, cudaStream_t s) {
  const size_t sm = chi_smem<T>(q.buf_rows, q.lsm, q.a.nsa);
  static SmemLimit limit;
  const cudaError_t e = limit.raise(chi_kernel<T, KS, KL, FOLD>, p.device, sm);
  if (e != cudaSuccess) return e;
  chi_kernel<T, KS, KL, FOLD><<<dim3(c.b1 - c.b0, p.natm, q.parts), 32 * q.warps, sm, s>>>(
      q, (cplx_t<T>*)p.chi->chi, c.b0);
  return cudaGetLastError();
}
cudaError_t run_dense(const Plan& p, const Params& q, const ChiChunk& c, cudaStream_t s) {
  const size_t sm = dense_smem(q.batch, q.a.nsa);
  static SmemLimit limit;
  const cudaError_t e = limit.raise(chi_dense_kernel, p.device, sm);
  if (e != cudaSuccess) return e;
  chi_dense_kernel<<<dim3(c.b1 - c.b0, p.natm, q.parts), 32 * kWarps, sm, s>>>(
      q, (float2*)p.chi->chi, c.b0);
  return cudaGetLastError();
}
template <typename T, int KS, int KL>
cudaError_t run_chi(const Plan& p, const Params& q, const ChiChunk& c, cudaStream_t s) {
  if constexpr (sizeof(T) == 4)
    if (q.batch > 0) return run_dense(p, q, c, s);
  return q.ncls <= kFold ? run_chi_as<T, KS, KL, true>(p, q, c, s)
                         : run_chi_as<T, KS, KL, false>(p, q, c, s);
}

// k-points per pass over a shell's entries: as many as the registers hold, fewer for meshes
// that would leave them idle
template <typename T>
cudaError_t fill(const Plan& p, const Params& q, const ChiChunk& c, cudaStream_t s) {
  if (p.nk == 1) return run_chi<T, 1, 1>(p, q, c, s);
  if constexpr (sizeof(T) == 4) {
    if (p.nk <= 4) return run_chi<T, 4, 4>(p, q, c, s);
    return run_chi<T, 8, 4>(p, q, c, s);
  } else {
    return run_chi<T, 4, 2>(p, q, c, s);
  }
}

template <typename T, int NI, bool REAL>
void run_orb_as(const Params& q, const void* chi, const void* cs, void* out, const ChiChunk& c,
                int i0, int periodic, cudaStream_t s) {
  // one block per warp where two would leave SMs without work
  const int nb = c.b1 - c.b0;
  constexpr int NB = orb_blocks<T, NI, REAL>();
  const auto* x = (const chi_t<T, REAL>*)chi;
  const auto* cf = (const typename CsT<T>::type*)cs;
  if (NB == 1 || (long long)nb * q.a.nk < 152 * 64)
    orb_kernel<T, NI, 1, REAL><<<dim3((nb + 3) / 4, q.a.nk), 128, 0, s>>>(
        q, x, cf, (cplx_t<T>*)out, c.b0, nb, i0, periodic);
  else
    orb_kernel<T, NI, NB, REAL><<<dim3((nb + 7) / 8, q.a.nk), 128, 0, s>>>(
        q, x, cf, (cplx_t<T>*)out, c.b0, nb, i0, periodic);
}
template <typename T, int NI>
void run_orb(const Params& q, const void* chi, const void* cs, void* out, const ChiChunk& c,
             int i0, int periodic, cudaStream_t s) {
  if (q.signs) run_orb_as<T, NI, true>(q, chi, cs, out, c, i0, periodic, s);
  else run_orb_as<T, NI, false>(q, chi, cs, out, c, i0, periodic, s);
}

template <typename T>
cudaError_t product_b(const Plan& p, const Params& q, const ChiChunk& c, const void* cs,
                      void* out, int periodic, cudaStream_t s) {
  const void* x = p.chi->chi;
  for (int i0 = 0; i0 < p.nocc;) {
    const int left = p.nocc - i0;
    if (left <= 4) run_orb<T, 4>(q, x, cs, out, c, i0, periodic, s);
    else if (left <= 8) run_orb<T, 8>(q, x, cs, out, c, i0, periodic, s);
    else run_orb<T, 16>(q, x, cs, out, c, i0, periodic, s);
    i0 += left <= 4 ? 4 : (left <= 8 ? 8 : 16);
  }
  return cudaGetLastError();
}

template <typename T, int NI>
void run_con(const Plan& p, const Params& q, const ChiChunk& c, const void* F, double2* out,
             double2* copy, int i0, double scale, cudaStream_t s) {
  const dim3 grid((c.con.nitems + 7) / 8, p.nk);
  if (c.con.nitems > 0 && q.signs)
    con_kernel<T, NI, true><<<grid, 256, 0, s>>>(q, (const T*)p.chi->chi, (const cplx_t<T>*)F,
                                                 c.con.item0, c.con.nitems, i0);
  else if (c.con.nitems > 0)
    con_kernel<T, NI, false><<<grid, 256, 0, s>>>(q, (const cplx_t<T>*)p.chi->chi,
                                                  (const cplx_t<T>*)F, c.con.item0, c.con.nitems, i0);
  sum_kernel<NI><<<dim3(q.nslots / kPad, p.nk), 2 * kPad * NI * kSumSplit, 0, s>>>(
      q, out, copy, c.con.row_of0, c.con.nitems, i0, scale, c.b0 > 0 ? 1 : 0);
}

// orbitals per pass of con_kernel
inline int con_width(int left, bool fp64) { return (fp64 || left <= 4) ? 4 : 8; }

template <typename T>
cudaError_t product_e(const Plan& p, const Params& q, const ChiChunk& c, const void* F,
                      double2* out, double2* copy, double scale, cudaStream_t s) {
  for (int i0 = 0; i0 < p.nocc;) {
    const int ni = con_width(p.nocc - i0, sizeof(T) == 8);
    if (ni == 4) {
      run_con<T, 4>(p, q, c, F, out, copy, i0, scale, s);
    } else if constexpr (sizeof(T) == 4) {
      run_con<T, 8>(p, q, c, F, out, copy, i0, scale, s);
    }
    i0 += ni;
  }
  return cudaGetLastError();
}

template cudaError_t fill<float>(const Plan&, const Params&, const ChiChunk&, cudaStream_t);
template cudaError_t fill<double>(const Plan&, const Params&, const ChiChunk&, cudaStream_t);

}  // namespace chi

template <typename T>
cudaError_t launch_slot_c(const Plan& p, const double2* X, void* out, double factor,
                          cudaStream_t s) {
  const long long n = (long long)p.nk * p.chi->nslots * p.nocc;
  chi::slot_c_kernel<T><<<2 * 152, 256, 0, s>>>(X, p.ao_norm, p.chi->slot_ao,
                                                (typename chi::CsT<T>::type*)out, p.nao, p.nocc,
                                                p.chi->nslots, n, factor);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_orbitals(const Plan& p, int nsets, const void* const* cs, void* const* out,
                            bool periodic, cudaStream_t s) {
  const chi::Params q = chi::params(p);
  for (const ChiChunk& c : p.chi->chunks) {
    cudaError_t e = chi::fill<T>(p, q, c, s);
    for (int i = 0; i < nsets && e == cudaSuccess; ++i)
      e = chi::product_b<T>(p, q, c, cs[i], out[i], periodic, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <typename T>
cudaError_t launch_contract_field(const Plan& p, const void* F, double2* out, double2* copy,
                                  double scale, cudaStream_t s) {
  const chi::Params q = chi::params(p);
  for (const ChiChunk& c : p.chi->chunks) {
    // one chunk: the buffer still holds chi from the orbitals of this call
    cudaError_t e = p.chi->chunks.size() > 1 ? chi::fill<T>(p, q, c, s) : cudaSuccess;
    if (e == cudaSuccess) e = chi::product_e<T>(p, q, c, F, out, copy, scale, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

int chi_launches(const Plan& p, bool contract) {
  const int nc = (int)p.chi->chunks.size();
  const int per = contract ? (p.precision == OCCRI_FP64 ? 4 : 8) : 16;
  const int products = (contract ? 2 : 1) * ((p.nocc + per - 1) / per);
  return nc * (products + (contract && nc == 1 ? 0 : 1));
}

int chi_slots(const Plan& p) { return p.chi->nslots; }

void chi_free(ChiTables* t) {
  if (!t) return;
  if (t->arena) cudaFree(t->arena);
  if (t->chunk_arena) cudaFree(t->chunk_arena);
  delete t;
}

namespace {

// Tables laid out one after another (256-byte steps) for one allocation and one copy.
struct Arena {
  std::vector<unsigned char> bytes;
  static size_t align(size_t x) { return (x + 255) / 256 * 256; }
  template <typename X>
  size_t put(const std::vector<X>& v) {
    const size_t at = align(bytes.size());
    bytes.resize(at + v.size() * sizeof(X));
    if (!v.empty()) std::memcpy(bytes.data() + at, v.data(), v.size() * sizeof(X));
    return at;
  }
};

}  // namespace

// Upper bound of |P_lm(d)| e^{-alpha d^2} over d: c_l (l / (2 alpha e))^{l/2}.
static double shell_peak(int l, double alpha) {
  static const double cl[4] = {1.0, 1.0, 2.0, 4.0};
  if (l == 0) return 1.0;
  return cl[l] * std::pow(l / (2.0 * alpha * std::exp(1.0)), 0.5 * l);
}

cudaError_t chi_create(Plan* p, const std::vector<ShellDev>& sh, const std::vector<double>& rcut,
                       const std::vector<unsigned short>& bpre, const std::vector<int>& img_n,
                       const std::vector<int>& t0, const std::vector<int>& atom_shell0,
                       size_t* total) {
  ChiTables* t = new (std::nothrow) ChiTables();
  if (!t) return cudaErrorMemoryAllocation;
  p->chi = t;
  t->tile = tc_contraction(*p) ? kTcTile : 0;
  const int natm = p->natm, nblk = p->nblk, nsa = p->nsa, lmax = p->lmax;
  const bool fp64 = p->precision == OCCRI_FP64;
  // slots: per atom, shells by falling screening radius
  std::vector<ChiShell> shells(p->nshell);
  std::vector<int> slot0(natm + 1, 0), slot_ao;
  for (int a = 0; a < natm; ++a) {
    slot0[a] = (int)slot_ao.size();
    std::vector<int> idx(atom_shell0[a + 1] - atom_shell0[a]);
    std::iota(idx.begin(), idx.end(), atom_shell0[a]);
    std::stable_sort(idx.begin(), idx.end(), [&](int x, int y) { return rcut[x] > rcut[y]; });
    for (size_t i = 0; i < idx.size(); ++i) {
      const ShellDev& s = sh[idx[i]];
      ChiShell& c = shells[atom_shell0[a] + i];
      std::memset(&c, 0, sizeof(c));
      c.alpha_d = s.alpha;
      c.rcut2_d = s.rcut2;
      c.alpha = s.alpha_f;
      c.alpha_lo = s.alpha_lo;
      c.rcut2 = s.rcut2_f;
      c.l = s.l;
      c.slot = (int)slot_ao.size() - slot0[a];
      c.orig = idx[i];
      c.exact = s.exact_arg;
      for (int m = 0; m < 2 * s.l + 1; ++m) slot_ao.push_back(s.ao + m);
    }
    while ((slot_ao.size() - slot0[a]) % chi::kPad) slot_ao.push_back(-1);
  }
  slot0[natm] = (int)slot_ao.size();
  t->nslots = slot0[natm];
  // FP16 scale of each slot: 2^13 over a bound of |chi| (the shell's largest value times the
  // images that reach a block)
  std::vector<float> row_scale(slot_ao.size(), 1.f);
  if (t->tile > 0)
    for (int a = 0; a < natm; ++a)
      for (int i = atom_shell0[a]; i < atom_shell0[a + 1]; ++i) {
        const ChiShell& c = shells[i];
        int np = 1;
        for (int b = 0; b < nblk; ++b)
          np = std::max<int>(np, bpre[((size_t)a * nblk + b) * nsa + (c.orig - atom_shell0[a])]);
        int e2 = 0;
        std::frexp(shell_peak(c.l, c.alpha_d) * np, &e2);
        for (int m = 0; m < 2 * c.l + 1; ++m)
          row_scale[slot0[a] + c.slot + m] = (float)std::ldexp(1.0, 13 - e2);
      }
  // active shells and slots per (atom, block)
  std::vector<unsigned short> nsh((size_t)natm * nblk, 0);
  std::vector<int> aoff((size_t)nblk * (natm + 1), 0);
  for (int b = 0; b < nblk; ++b)
    for (int a = 0; a < natm; ++a) {
      const size_t ab = (size_t)a * nblk + b;
      int n = 0, slots = 0;
      const int ns = atom_shell0[a + 1] - atom_shell0[a];
      while (n < ns && bpre[ab * nsa + (shells[atom_shell0[a] + n].orig - atom_shell0[a])] > 0) {
        const ChiShell& c = shells[atom_shell0[a] + n];
        slots = c.slot + 2 * c.l + 1;
        ++n;
      }
      nsh[ab] = (unsigned short)n;
      slots = (slots + chi::kPad - 1) / chi::kPad * chi::kPad;
      aoff[(size_t)b * (natm + 1) + a + 1] = aoff[(size_t)b * (natm + 1) + a] + slots;
    }
  // Wide shells go through the transform over classes where the mesh is (nearly) full, its
  // k-points are distinct and its lengths are compiled; columns as the shared memory allows.
  const int Dc = p->D[0] * p->D[1] * p->D[2], nimg = p->nimg;
  bool dft = Dc <= 4096 && Dc <= 4 * p->nk;
  for (int d = 0; d < 3; ++d) dft = dft && (p->D[d] <= 6 || p->D[d] == 8);
  std::vector<int> kidx(dft ? Dc : 1, -1);
  for (int k = 0; k < p->nk && dft; ++k) {
    const int r = (p->kint_h[3 * k] * p->D[1] + p->kint_h[3 * k + 1]) * p->D[2] + p->kint_h[3 * k + 2];
    if (kidx[r] >= 0) dft = false;
    kidx[r] = k;
  }
  t->signs = dft && Dc <= chi::kFold && p->D[0] <= 2 && p->D[1] <= 2 && p->D[2] <= 2;
  // residue classes of T0 + T' modulo the k-mesh's supercell, a table row per distinct T0; the
  // transform takes class = residue, other meshes number the residues in use
  std::vector<int> id(Dc, -1), residue, cls, seen;
  if (dft) {
    residue.resize(Dc);
    std::iota(residue.begin(), residue.end(), 0);
    id = residue;
  }
  std::vector<unsigned short> t0i((size_t)natm * nblk);
  for (size_t ab = 0; ab < t0i.size(); ++ab) {
    size_t row = 0;
    while (row < seen.size() && seen[row] != t0[ab]) ++row;
    t0i[ab] = (unsigned short)row;
    if (row < seen.size()) continue;
    seen.push_back(t0[ab]);
    int s0[3];
    dev::unpack_t0(t0[ab], &s0[0], &s0[1], &s0[2]);
    for (int j = 0; j < nimg; ++j) {
      int r = 0;
      for (int d = 0; d < 3; ++d) {
        const int D = p->D[d];
        r = r * D + ((s0[d] + img_n[3 * (size_t)j + d]) % D + D) % D;
      }
      if (id[r] < 0) {
        id[r] = (int)residue.size();
        residue.push_back(r);
      }
      cls.push_back(id[r]);
    }
  }
  t->ncls = std::max(1, (int)residue.size());
  t->nkp = (p->nk + 7) / 8 * 8;
  std::vector<double2> phase((size_t)t->ncls * t->nkp, make_double2(0.0, 0.0));
  std::vector<double2> unit(residue.size() * p->nk > (size_t)Dc ? Dc : 0);   // e^{2 pi i n / Dc}
  auto root = [&](long long num) {
    const double ang = 2.0 * 3.14159265358979323846 * (double)num / (double)Dc;
    return make_double2(std::cos(ang), std::sin(ang));
  };
  for (size_t n = 0; n < unit.size(); ++n) unit[n] = root((long long)n);
  for (size_t c = 0; c < residue.size(); ++c) {
    const int n[3] = {residue[c] / (p->D[1] * p->D[2]), residue[c] / p->D[2] % p->D[1],
                      residue[c] % p->D[2]};
    for (int k = 0; k < p->nk; ++k) {
      long long num = 0;
      for (int d = 0; d < 3; ++d) num += (long long)p->kint_h[k * 3 + d] * n[d] * (Dc / p->D[d]);
      num %= Dc;
      phase[c * t->nkp + k] = unit.empty() ? root(num) : unit[num];
    }
  }
  // Up to kFold classes every shell takes one warp (fold_shell). With few shells in all, a CTA
  // per atom and block would transform its columns on a nearly idle GPU: on many k-points
  // chi_dense_kernel spreads those instead (6x6x8 k, 10 AOs, 8^3: orbitals 100 -> 68 us).
  const long long shells_all = (long long)nblk * natm * nsa;
  dft = dft && Dc > chi::kFold && (fp64 || p->nk < 128 || shells_all >= 152 * 8);
  t->aoff_h = aoff;
  const int row_bytes = 32 * (fp64 ? 8 : 4);
  t->col_rows = 2 * (p->D[0] / 2 + 1) * p->D[1] * p->D[2];
  // 88 KB of columns leave room for two CTAs per SM; where that is under four AOs, one CTA
  const long long col_bytes = (long long)t->col_rows * row_bytes;
  const long long cols = (88 * 1024 / col_bytes >= 4 ? 88 : 176) * 1024 / col_bytes;
  t->ncol = dft ? (int)std::min<long long>(chi::kCols, cols) : 0;
  // without the transform nothing crosses warps: smaller CTAs
  t->warps = t->ncol > 0 ? chi::kWarps : chi::kFoldWarps;
  t->buf_rows = std::max(t->ncol * t->col_rows, t->warps * chi::kRows);
  const size_t need = fp64 ? chi::chi_smem<double>(t->buf_rows, lmax, nsa)
                           : chi::chi_smem<float>(t->buf_rows, lmax, nsa);
  t->lsm = need <= 200 * 1024 ? lmax : 0;
  // several CTAs per (block, atom) where there are few of them (a Gamma cell)
  long long parts = 152LL * 4 / ((long long)nblk * natm);
  if (!fp64 && !dft && p->nk >= chi::kDenseK) {
    // batches of about equal size; the CTAs of a (block, atom) share the k-points
    const int nb = (lmax + chi::kDenseImages - 1) / chi::kDenseImages;
    t->batch = (lmax + nb - 1) / nb;
    parts = std::min<long long>(parts, p->nk / (chi::KD * chi::kWarps));
  } else {
    // many k-points on a small grid: slices of them for narrow shells, a warp each
    t->kslices = (int)std::max(1LL, std::min(p->nk / 32LL, 152LL * 16 / shells_all));
    parts = std::min<long long>(std::max(4, (nsa * t->kslices + t->warps - 1) / t->warps), parts);
  }
  t->parts = (int)std::max(1LL, parts);

  std::vector<float2> phase_f;
  if (!fp64)
    for (const double2& z : phase) phase_f.push_back(make_float2((float)z.x, (float)z.y));
  Arena tab;
  const size_t o_sh = tab.put(shells), o_s0 = tab.put(slot0), o_ao = tab.put(slot_ao),
               o_nsh = tab.put(nsh), o_aoff = tab.put(aoff), o_t0i = tab.put(t0i),
               o_cls = tab.put(cls), o_ph = fp64 ? tab.put(phase) : tab.put(phase_f),
               o_rs = tab.put(row_scale), o_ki = tab.put(kidx);
  // then the lists in order of class (for the wide shells)
  const bool sorted = t->ncol > 0;
  const size_t o_ord = Arena::align(tab.bytes.size());
  const size_t bytes = o_ord + (sorted ? sizeof(short) * (size_t)natm * nblk * lmax : 0);
  *total += bytes;
  cudaError_t e = device_malloc(&t->arena, bytes);
  if (e != cudaSuccess) return e;
  e = cudaMemcpy(t->arena, tab.bytes.data(), tab.bytes.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return e;
  unsigned char* d = (unsigned char*)t->arena;
  t->shells = (ChiShell*)(d + o_sh);
  t->slot0 = (int*)(d + o_s0);
  t->slot_ao = (int*)(d + o_ao);
  t->nsh = (unsigned short*)(d + o_nsh);
  t->aoff = (int*)(d + o_aoff);
  t->t0i = (unsigned short*)(d + o_t0i);
  t->cls = (int*)(d + o_cls);
  t->phase = d + o_ph;
  t->row_scale = (float*)(d + o_rs);
  t->kidx = (int*)(d + o_ki);
  if (sorted) {
    t->order = (unsigned short*)(d + o_ord);   // after the copies, on their stream
    chi::order_kernel<<<(natm * nblk + 7) / 8, 256>>>(chi::params(*p), t->order);
    e = cudaGetLastError();
  }
  return e;
}

namespace {

// Chunks of blocks of at most `budget` bytes of chi (one block at least), the contractions' work
// items in them, and their memory, whose device addresses go to t.
cudaError_t chi_layout(Plan* p, size_t budget, size_t slot_bytes, size_t* total) {
  ChiTables* t = p->chi;
  const int natm = p->natm, nblk = p->nblk;
  const bool fp64 = p->precision == OCCRI_FP64;
  const std::vector<int>& aoff = t->aoff_h;
  t->chunks.clear();
  t->chi_bytes = t->part_bytes = 0;
  t->item_pairs = 0;
  std::vector<long long> boff(nblk, 0);
  {
    ChiChunk c;
    long long slots = 0;
    for (int b = 0; b < nblk; ++b) {
      const int n = aoff[(size_t)b * (natm + 1) + natm];
      if (b > c.b0 && slot_bytes * (slots + n) > budget) {
        c.b1 = b;
        t->chunks.push_back(c);
        c.b0 = b;
        slots = 0;
      }
      boff[b] = slots;
      slots += n;
      t->chi_bytes = std::max(t->chi_bytes, slot_bytes * (size_t)slots);
    }
    c.b1 = nblk;
    t->chunks.push_back(c);
  }
  // The contraction's items: a group of slots of an atom (kPad of them, or a tensor-core tile)
  // over up to `run` of the blocks that reach the group. `run` gives enough items to fill the
  // GPU (about 16 warps per scheduler, or three rounds of CTAs); a lane's FP32 sums go over
  // 16 blocks at most (with 64 the bands' columns at 40^3, 8 k were 1.7e-7 from FP64, with 16
  // 1.5e-7).
  std::vector<int4> items;
  std::vector<int> border;
  std::vector<int2> rows, rows_of;
  auto slots = [&](int a, int b) {
    return aoff[(size_t)b * (natm + 1) + a + 1] - aoff[(size_t)b * (natm + 1) + a];
  };
  auto run_length = [&](int width, long long want, long long most) {
    long long groups = 0;
    for (int b = 0; b < nblk; ++b)
      for (int a = 0; a < natm; ++a) groups += (slots(a, b) + width - 1) / width;
    const int run = (int)std::max<long long>(4, std::min(most, groups * p->nk / want));
    return (run + 1) / 2 * 2;
  };
  const int con_run = run_length(chi::kPad, 152 * 64, fp64 ? 64 : 16);
  const int tc_run = t->tile > 0 ? run_length(t->tile, 152 * 9, tc_item_blocks(p->nocc)) : 0;
  std::vector<int> first(natm);   // the chunk's blocks by falling number of the atom's slots
  auto make_items = [&](const ChiChunk& c, ChiItems* it, int width, int run, size_t values,
                        long long* pairs) {
    it->item0 = (int)items.size();
    it->row_of0 = (int)rows_of.size();
    const int nb = c.b1 - c.b0;
    for (int a = 0; a < natm; ++a) {
      const int row0 = (int)rows.size(), o0 = first[a];
      for (int r0 = 0; r0 < nb && slots(a, border[o0 + r0]) > 0; r0 += run) {
        const int ns = slots(a, border[o0 + r0]);
        rows.push_back(make_int2((int)items.size() - it->item0, (ns + width - 1) / width));
        for (int s = 0; s < ns; s += width) {
          int n = 0;
          while (n < run && r0 + n < nb && slots(a, border[o0 + r0 + n]) > s) ++n;
          items.push_back(make_int4(a, s, o0 + r0, n));
          if (pairs) *pairs += (n + 1) / 2;
        }
      }
      rows_of.push_back(make_int2(row0, (int)rows.size() - row0));
    }
    it->nitems = (int)items.size() - it->item0;
    t->part_bytes =
        std::max(t->part_bytes, sizeof(double) * values * (size_t)it->nitems * p->nk);
  };
  for (ChiChunk& c : t->chunks) {
    for (int a = 0; a < natm; ++a) {
      std::vector<int> bl(c.b1 - c.b0);
      std::iota(bl.begin(), bl.end(), c.b0);
      std::stable_sort(bl.begin(), bl.end(),
                       [&](int x, int y) { return slots(a, x) > slots(a, y); });
      first[a] = (int)border.size();
      border.insert(border.end(), bl.begin(), bl.end());
    }
    make_items(c, &c.con, chi::kPad, con_run,
               2 * (size_t)chi::kPad * chi::con_width(p->nocc, fp64), nullptr);
    if (t->tile > 0)
      make_items(c, &c.tc, t->tile, tc_run, tc_item_values(p->nocc), &t->item_pairs);
  }
  Arena tab;
  const size_t o_boff = tab.put(boff), o_it = tab.put(items), o_bd = tab.put(border),
               o_rows = tab.put(rows), o_ro = tab.put(rows_of);
  const size_t o_part = Arena::align(tab.bytes.size());   // the items' sums, then chi
  const size_t o_chi = Arena::align(o_part + t->part_bytes);
  const size_t bytes = o_chi + std::max<size_t>(t->chi_bytes, 16);
  cudaError_t e = device_malloc(&t->chunk_arena, bytes);
  if (e != cudaSuccess) return e;
  e = cudaMemcpy(t->chunk_arena, tab.bytes.data(), tab.bytes.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return e;
  *total += bytes;
  unsigned char* d = (unsigned char*)t->chunk_arena;
  t->boff = (long long*)(d + o_boff);
  t->items = (int4*)(d + o_it);
  t->border = (int*)(d + o_bd);
  t->rows = (int2*)(d + o_rows);
  t->rows_of = (int2*)(d + o_ro);
  t->part = (double*)(d + o_part);
  t->chi = d + o_chi;
  return cudaSuccess;
}

}  // namespace

cudaError_t chi_reserve(Plan* p, size_t later, size_t* total) {
  const ChiTables& t = *p->chi;
  const size_t csz = (p->precision == OCCRI_FP64 ? sizeof(double) : sizeof(float)) * (t.signs ? 1 : 2);
  const size_t slot_bytes = csz * 32 * (size_t)p->nk;
  size_t all = 0, widest = 0;
  for (int b = 0; b < p->nblk; ++b) {
    const size_t n = slot_bytes * t.aoff_h[(size_t)b * (p->natm + 1) + p->natm];
    all += n;
    widest = std::max(widest, n);
  }
  size_t free_b = 0, dev_b = 0;
  if (cudaMemGetInfo(&free_b, &dev_b) != cudaSuccess) return cudaGetLastError();
  const size_t room = free_b > later ? free_b - later : 0;
  size_t budget = all <= std::min(kChiKeepBytes, room / 4)
                      ? std::max<size_t>(all, 1)
                      : std::max(widest, std::min(kChiChunkBytes, room / 8));
  while (true) {
    const cudaError_t e = chi_layout(p, budget, slot_bytes, total);
    // no memory: smaller chunks, down to one block
    if (e != cudaErrorMemoryAllocation || t.chi_bytes <= widest) return e;
    cudaGetLastError();
    budget = std::max(widest, t.chi_bytes / 2);
  }
}

template cudaError_t launch_slot_c<float>(const Plan&, const double2*, void*, double, cudaStream_t);
template cudaError_t launch_slot_c<double>(const Plan&, const double2*, void*, double, cudaStream_t);
template cudaError_t launch_orbitals<float>(const Plan&, int, const void* const*, void* const*,
                                            bool, cudaStream_t);
template cudaError_t launch_orbitals<double>(const Plan&, int, const void* const*, void* const*,
                                             bool, cudaStream_t);
template cudaError_t launch_contract_field<float>(const Plan&, const void*, double2*, double2*,
                                                  double, cudaStream_t);
template cudaError_t launch_contract_field<double>(const Plan&, const void*, double2*, double2*,
                                                   double, cudaStream_t);

}  // namespace occri
