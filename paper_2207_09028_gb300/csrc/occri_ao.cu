// occri_ao.cu -- the orbitals without allocation, the fields' phases and output order.
//   (a)+(b) psi_{ik}(r) = sum_mu C^k_{mu i} chi_{mu k}(r)                  (Eq. occmo)
// with chi_{mu k}(r) = sum_T e^{i k.T} phi_mu(r - A - T) (Sec. II.A). orbitals_kernel evaluates
// chi where it is used and stores none of it, for occri_orbitals_noalloc alone, which has no
// memory for AO tiles; every other call takes the tiles of occri_chi.cu.
//
// The image sum is split as T = T0(r, A) + T': T0 brings r - A into the
// Wigner-Seitz cell (precomputed per grid point and atom), T' runs over one
// master list of lattice vectors sorted by length. Every thread of a warp walks
// the same prefix of that list (a shell's prefix covers its screening radius
// plus the largest |r - A - T0|), so the image offsets and the phase table
// e^{i k.T'} are warp-uniform loads.
//
// In FP32 the displacement r - A - T is formed from hi/lo float pairs so that
// it is accurate to an ulp of its own size, not of |T|.
#include <cuda_runtime.h>

#include <mutex>

#include "occri_ao.cuh"

namespace occri {
namespace ao {

__device__ __forceinline__ void image_disp(const AOParams& p, const Disp<double>& d, int j,
                                           double* x, double* y, double* z) {
  *x = d.x - p.img_d[j];
  *y = d.y - p.img_d[p.nimg + j];
  *z = d.z - p.img_d[2 * p.nimg + j];
}
__device__ __forceinline__ void image_disp(const AOParams& p, const Disp<float>& d, int j,
                                           float* x, float* y, float* z) {
  *x = (d.xh - p.img_hi[j]) + (d.xl - p.img_lo[j]);
  *y = (d.yh - p.img_hi[p.nimg + j]) + (d.yl - p.img_lo[p.nimg + j]);
  *z = (d.zh - p.img_hi[2 * p.nimg + j]) + (d.zl - p.img_lo[2 * p.nimg + j]);
}

template <typename T> __device__ __forceinline__ T sh_alpha(const ShellDev& s);
template <> __device__ __forceinline__ double sh_alpha<double>(const ShellDev& s) { return s.alpha; }
template <> __device__ __forceinline__ float sh_alpha<float>(const ShellDev& s) { return s.alpha_f; }
template <typename T> __device__ __forceinline__ T sh_alpha_lo(const ShellDev& s);
template <> __device__ __forceinline__ double sh_alpha_lo<double>(const ShellDev&) { return 0.0; }
template <> __device__ __forceinline__ float sh_alpha_lo<float>(const ShellDev& s) { return s.alpha_lo; }
template <typename T> __device__ __forceinline__ T sh_rcut2(const ShellDev& s);
template <> __device__ __forceinline__ double sh_rcut2<double>(const ShellDev& s) { return s.rcut2; }
template <> __device__ __forceinline__ float sh_rcut2<float>(const ShellDev& s) { return s.rcut2_f; }

// e^{i k.T0} for the T0 shared by the points of block `blk` for this atom.
template <typename T>
__device__ __forceinline__ cplx_t<T> phase_t0(const AOParams& p, int atom, int blk, int k) {
  int t[3];
  dev::unpack_t0(p.t0[(size_t)atom * p.nblk + blk], &t[0], &t[1], &t[2]);
  long long num = 0;
#pragma unroll
  for (int d = 0; d < 3; ++d)
    num += (long long)p.kint[k * 3 + d] * t[d] * (p.Dc / p.D[d]);
  return cis_frac<T>(num, p.Dc, +1);
}

// chi_{mu k}(r_n)/N_mu for KB consecutive k-points (rows k0..k0+KB-1 of the padded
// phase table); the image geometry, exponential and polynomial are computed once.
template <typename T, int L, int KB>
__device__ __forceinline__ void shell_values_kb(const AOParams& p, const ShellDev& sh, int k0,
                                                const Disp<T>& d, const unsigned short* list,
                                                int np, T (&cr)[KB][2 * L + 1],
                                                T (&ci)[KB][2 * L + 1]) {
  const cplx_t<T>* ph = reinterpret_cast<const cplx_t<T>*>(p.img_phase) + (size_t)k0 * p.nimg;
  const T alpha = sh_alpha<T>(sh), alo = sh_alpha_lo<T>(sh), rc2 = sh_rcut2<T>(sh);
#pragma unroll
  for (int b = 0; b < KB; ++b)
#pragma unroll
    for (int m = 0; m < 2 * L + 1; ++m) {
      cr[b][m] = T(0);
      ci[b][m] = T(0);
    }
  const bool exact = (sizeof(T) == 4) && sh.exact_arg;
  for (int j = 0; j < np; ++j) {
    const int idx = list[j];
    T x, y, z, r2, e;
    if constexpr (sizeof(T) == 4) {
      if (exact) {
        e = exact_gauss(d, p.img_hi[idx], p.img_hi[p.nimg + idx], p.img_hi[2 * p.nimg + idx],
                        p.img_lo[idx], p.img_lo[p.nimg + idx], p.img_lo[2 * p.nimg + idx], alpha,
                        alo, &r2, &x, &y, &z);
      } else {
        image_disp(p, d, idx, &x, &y, &z);
        r2 = x * x + y * y + z * z;
        e = exp_t(-(alpha * r2 + alo * r2));
      }
    } else {
      image_disp(p, d, idx, &x, &y, &z);
      r2 = x * x + y * y + z * z;
      e = exp_t(-(alpha * r2 + alo * r2));
    }
    if (r2 <= rc2) {
      T P[2 * L + 1];
      solid<T, L>(x, y, z, P);
#pragma unroll
      for (int m = 0; m < 2 * L + 1; ++m) P[m] *= e;
#pragma unroll
      for (int b = 0; b < KB; ++b) {
        const cplx_t<T> w = ph[(size_t)b * p.nimg + idx];
#pragma unroll
        for (int m = 0; m < 2 * L + 1; ++m) {
          cr[b][m] += w.x * P[m];
          ci[b][m] += w.y * P[m];
        }
      }
    }
  }
}


// psi += (N_mu C_mu i) chi_mu / N_mu; in FP32 the scaled coefficient is a hi/lo pair.
__device__ __forceinline__ void cmac(const double2* cs, size_t idx, double xr, double xi,
                                     double& ar, double& ai) {
  const double2 c = cs[idx];
  ar += c.x * xr - c.y * xi;
  ai += c.x * xi + c.y * xr;
}
__device__ __forceinline__ void cmac(const float4* cs, size_t idx, float xr, float xi, float& ar,
                                     float& ai) {
  const float4 c = cs[idx];
  ar += (c.x * xr - c.y * xi) + (c.z * xr - c.w * xi);
  ai += (c.x * xi + c.y * xr) + (c.z * xi + c.w * xr);
}
template <typename T> struct CsType;
template <> struct CsType<double> { using type = double2; };
template <> struct CsType<float> { using type = float4; };

template <typename T, int L, int NI, int KB>
__device__ __forceinline__ void orbital_shell(const AOParams& p, const ShellDev& sh, int k0,
                                              const Disp<T>& d, const unsigned short* list,
                                              int np, const cplx_t<T> (&ph0)[KB], int i0,
                                              T (&ar)[KB][NI], T (&ai)[KB][NI]) {
  using CS = typename CsType<T>::type;
  const CS* cs = reinterpret_cast<const CS*>(p.cs);
  T cr[KB][2 * L + 1], ci[KB][2 * L + 1];
  shell_values_kb<T, L, KB>(p, sh, k0, d, list, np, cr, ci);
#pragma unroll
  for (int b = 0; b < KB; ++b) {
    if (k0 + b >= p.nk) break;
#pragma unroll
    for (int m = 0; m < 2 * L + 1; ++m) {
      const T xr = cr[b][m] * ph0[b].x - ci[b][m] * ph0[b].y;
      const T xi = cr[b][m] * ph0[b].y + ci[b][m] * ph0[b].x;
      const size_t row = ((size_t)(k0 + b) * p.nao + sh.ao + m) * p.nocc;
#pragma unroll
      for (int i = 0; i < NI; ++i)
        if (i0 + i < p.nocc) cmac(cs, row + i0 + i, xr, xi, ar[b][i], ai[b][i]);
    }
  }
}

// Scaled coefficients N_mu C^k_{mu i}, formed in FP64 (and split hi/lo for FP32).
__global__ void scale_c_kernel_d(const double2* __restrict__ C, const double* __restrict__ nrm,
                                 double2* __restrict__ out, int nao, int nocc, long long n) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const double s = nrm[(e / nocc) % nao];
    out[e] = make_double2(s * C[e].x, s * C[e].y);
  }
}
__global__ void scale_c_kernel_f(const double2* __restrict__ C, const double* __restrict__ nrm,
                                 float4* __restrict__ out, int nao, int nocc, long long n) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const double s = nrm[(e / nocc) % nao];
    const double x = s * C[e].x, y = s * C[e].y;
    const float xh = (float)x, yh = (float)y;
    out[e] = make_float4(xh, yh, (float)(x - (double)xh), (float)(y - (double)yh));
  }
}

// One warp per point block, four blocks per CTA; KB k-points per thread. Three CTAs per SM
// (168 registers, a 104-byte spill in FP32) were 7 % faster than two (255 registers).
template <typename T, int NI, int KB>
__global__ void __launch_bounds__(128, 3)
orbitals_kernel(AOParams p, cplx_t<T>* __restrict__ psi, int i0) {
  const int blk = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (blk >= p.nblk) return;
  bool valid;
  long long q;
  const long long n = block_point(p, blk, threadIdx.x & 31, &valid, &q);
  const int k0 = blockIdx.y * KB;
  T ar[KB][NI], ai[KB][NI];
#pragma unroll
  for (int b = 0; b < KB; ++b)
#pragma unroll
    for (int i = 0; i < NI; ++i) { ar[b][i] = T(0); ai[b][i] = T(0); }
  for (int a = 0; a < p.natm; ++a) {
    Disp<T> d;
    load_disp(p, a, n, &d);
    cplx_t<T> ph0[KB];
#pragma unroll
    for (int b = 0; b < KB; ++b)
      ph0[b] = (k0 + b < p.nk) ? phase_t0<T>(p, a, blk, k0 + b) : cplx_t<T>{T(0), T(0)};
    const size_t ab = (size_t)a * p.nblk + blk;
    const unsigned short* list = p.blist + ab * p.lmax;
    const unsigned short* pre = p.bpre + ab * p.nsa;
    const int s0 = p.atom_shell0[a];
    for (int s = s0; s < p.atom_shell0[a + 1]; ++s) {
      const ShellDev sh = p.shells[s];
      const int np = pre[s - s0];
      switch (sh.l) {
        case 0: orbital_shell<T, 0, NI, KB>(p, sh, k0, d, list, np, ph0, i0, ar, ai); break;
        case 1: orbital_shell<T, 1, NI, KB>(p, sh, k0, d, list, np, ph0, i0, ar, ai); break;
        case 2: orbital_shell<T, 2, NI, KB>(p, sh, k0, d, list, np, ph0, i0, ar, ai); break;
        default: orbital_shell<T, 3, NI, KB>(p, sh, k0, d, list, np, ph0, i0, ar, ai); break;
      }
    }
  }
  if (!valid) return;
#pragma unroll
  for (int b = 0; b < KB; ++b) {
    if (k0 + b >= p.nk) break;
#pragma unroll
    for (int i = 0; i < NI; ++i)
      if (i0 + i < p.nocc)
        psi[((size_t)(k0 + b) * p.nocc + i0 + i) * p.fs + q] = cplx_t<T>{ar[b][i], ai[b][i]};
  }
}

// Widen the fields to c128 and put them back in natural point order:
// out[f][(n1 N + n2) N + n3] = in[f][(n3 N + n1) N + n2] (cubic grid of edge N; input
// fields fs points apart, output fields N^3 apart).
template <typename T>
__global__ void widen_kernel(const cplx_t<T>* __restrict__ in, double2* __restrict__ out,
                             long long n, int N, long long fs) {
  const long long ng = (long long)N * N * N;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const long long f = e / ng, r = e - f * ng;
    const int n3 = (int)(r % N), n2 = (int)((r / N) % N), n1 = (int)(r / ((long long)N * N));
    const cplx_t<T> v = in[f * fs + ((long long)n3 * N + n1) * N + n2];
    out[e] = make_double2(double(v.x), double(v.y));
  }
}


// F[k][i][q] = (F + a + b) e^{i k.r_q} for every orbital field of every k-point (fields' point order
// q = (n3 N + n1) N + n2, cubic grid of edge N): the streams' sums of periodic parts become Y_ik.
template <typename T>
__global__ void phase_fields_kernel(cplx_t<T>* __restrict__ F, const cplx_t<T>* __restrict__ a,
                                    const cplx_t<T>* __restrict__ b, const int* __restrict__ kint,
                                    int nk, int nocc, int N, long long fs, int D0, int D1, int D2) {
  const long long ng = (long long)N * N * N;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < nk * ng;
       e += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(e / ng);
    const long long q = e - (long long)k * ng;
    const int n3 = (int)(q / ((long long)N * N));
    const int rem = (int)(q - (long long)n3 * N * N);
    const cplx_t<T> ph = point_phase<T>(kint + 3 * k, D0, D1, D2, N, rem / N, rem % N, n3, +1);
    const size_t at = (size_t)k * nocc * fs + q;
    for (int i = 0; i < nocc; ++i) {
      const size_t f = at + (size_t)i * fs;
      cplx_t<T> v = F[f];
      if (a) {
        cplx_t<T> u = a[f];
        if (b) {
          const cplx_t<T> w = b[f];
          u.x += w.x;
          u.y += w.y;
        }
        v.x += u.x;
        v.y += u.y;
      }
      F[f] = dev::cmul<T>(v, ph);
    }
  }
}

}  // namespace ao

template <typename T>
cudaError_t launch_phase_fields(const Plan& p, void* F, const void* a, const void* b,
                                cudaStream_t s) {
  ao::phase_fields_kernel<T><<<8 * 152, 256, 0, s>>>((cplx_t<T>*)F, (const cplx_t<T>*)a,
                                                      (const cplx_t<T>*)b, p.kint, p.nk, p.nocc,
                                                      p.N[0], p.fs, p.D[0], p.D[1], p.D[2]);
  return cudaGetLastError();
}
template cudaError_t launch_phase_fields<float>(const Plan&, void*, const void*, const void*,
                                                cudaStream_t);
template cudaError_t launch_phase_fields<double>(const Plan&, void*, const void*, const void*,
                                                 cudaStream_t);

template <typename T>
cudaError_t launch_widen(const Plan& p, void* out, cudaStream_t s) {
  const long long n = (long long)p.nk * p.nocc * p.ng;
  ao::widen_kernel<T><<<4 * 152, 256, 0, s>>>((const cplx_t<T>*)p.psi, (double2*)out, n, p.N[0],
                                               p.fs);
  return cudaGetLastError();
}

template cudaError_t launch_widen<float>(const Plan&, void*, cudaStream_t);
template cudaError_t launch_widen<double>(const Plan&, void*, cudaStream_t);

}  // namespace occri

// ------------------------------------------------------------------ orbitals without allocation
//
// occri_orbitals_noalloc evaluates the AOs where it uses them and keeps its
// scratch -- the normalised coefficients N_mu C^k_{mu i} and the orbitals in the
// plan's working precision before widening -- in this file-scope device array
// instead of the plan's workspaces. Every GPU that loads the library reserves
// OCCRI_STATIC_SCRATCH_BYTES of device memory for it until the process exits.
static __device__ __align__(256) unsigned char occri_static_scratch[OCCRI_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
void* g_scratch_addr[kMaxDevices] = {};
std::mutex g_scratch_mutex;

size_t round_up_256(size_t x) { return (x + 255) & ~size_t(255); }

// Device address of the static array for the current device (looked up once per device,
// with that device current; the host-side symbol itself is not a device address). The
// caller has made the plan's device current.
int static_scratch_address(void** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return OCCRI_ECUDA;
  }
  if (dev < 0 || dev >= kMaxDevices) return OCCRI_EUNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (!g_scratch_addr[dev]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, occri_static_scratch) != cudaSuccess || ptr == nullptr) {
      cudaGetLastError();
      return OCCRI_ECUDA;
    }
    g_scratch_addr[dev] = ptr;
  }
  *out = g_scratch_addr[dev];
  return OCCRI_OK;
}

template <typename T>
int orbitals_noalloc_impl(const occri::Plan& p, const double2* C, void* psi_out, void* base) {
  using namespace occri;
  using CS = typename ao::CsType<T>::type;
  const long long ncs = (long long)p.nk * p.nao * p.nocc;
  const long long npsi = (long long)p.nk * p.nocc * p.ng;   // outputs (natural order)
  CS* cs = reinterpret_cast<CS*>(base);
  cplx_t<T>* psi = reinterpret_cast<cplx_t<T>*>(static_cast<unsigned char*>(base) +
                                                round_up_256(sizeof(CS) * ncs));
  cudaStream_t s = p.stream;
  if constexpr (sizeof(T) == 8)
    ao::scale_c_kernel_d<<<2 * 152, 256, 0, s>>>(C, p.ao_norm, cs, p.nao, p.nocc, ncs);
  else
    ao::scale_c_kernel_f<<<2 * 152, 256, 0, s>>>(C, p.ao_norm, cs, p.nao, p.nocc, ncs);
  AOParams ap = p.ao_params();
  ap.cs = cs;
  constexpr int KB = orbital_kbatch<T>();
  const dim3 grid((unsigned)((p.nblk + 3) / 4), (p.nk + KB - 1) / KB);
  for (int i0 = 0; i0 < p.nocc; i0 += kOrbChunk)
    ao::orbitals_kernel<T, kOrbChunk, KB><<<grid, 128, 0, s>>>(ap, psi, i0);
  ao::widen_kernel<T><<<4 * 152, 256, 0, s>>>(psi, (double2*)psi_out, npsi, p.N[0], p.fs);
  return cudaGetLastError() == cudaSuccess ? OCCRI_OK : OCCRI_ECUDA;
}

}  // namespace

extern "C" int occri_orbitals_noalloc(const occri_plan* plan, const void* C_dev, void* psi_dev) {
  if (!plan || !C_dev || !psi_dev) return OCCRI_EINVAL;
  const occri::Plan& p = *plan->p;
  // the plan's device is made current, so the scratch address below is that device's
  occri::DeviceGuard guard(p.device);
  if (!guard.ok) return OCCRI_ECUDA;
  const bool fp64 = p.precision == OCCRI_FP64;
  const size_t ncs = (size_t)p.nk * p.nao * p.nocc;
  const size_t npsi = (size_t)p.nk * p.nocc * p.fs;   // internal fields, fs points apart
  const size_t need = round_up_256((fp64 ? sizeof(double2) : sizeof(float4)) * ncs) +
                      (fp64 ? sizeof(double2) : sizeof(float2)) * npsi;
  if (need > (size_t)OCCRI_STATIC_SCRATCH_BYTES) return OCCRI_EINVAL;
  void* base = nullptr;
  const int st = static_scratch_address(&base);
  if (st != OCCRI_OK) return st;
  return fp64 ? orbitals_noalloc_impl<double>(p, (const double2*)C_dev, psi_dev, base)
              : orbitals_noalloc_impl<float>(p, (const double2*)C_dev, psi_dev, base);
}
