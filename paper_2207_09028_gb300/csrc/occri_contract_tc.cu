// occri_contract_tc.cu -- step (e), K_{mu i}(k) = -(Omega/(N_k N_g)) sum_r conj(chi_{mu k}(r))
// Y_ik(r) (Eq. occrik, the last step of Algorithm 3), on the tensor cores.
//
// Per k it is a real GEMM: rows Re chi and Im chi of 64 AO slots (M = 128), columns Re Y and
// Im Y of the occupied orbitals (N = 16, 32 or 64), reduction over the points of the blocks that
// reach the slots. The four real products of a slot and an orbital give
//   Re K = chi_r.Y_r + chi_i.Y_i,   Im K = chi_r.Y_i - chi_i.Y_r.
// A stage is a pair of point blocks (K = 64). The CTA reads chi and Y as FP32, splits both into
// FP16 hi + lo (power-of-two scales per slot and per orbital) while it writes them to shared
// memory in the tensor cores' layout, and one thread issues the stage's three FP16 products
// (hi.hi + hi.lo + lo.hi) into tensor memory, 16 points to an accumulator, which leave it after
// the stage for FP32 sums in registers: sums in tensor memory round toward zero (64 points to
// an accumulator biased E_x by 1.1e-7 relative, long sums by 1e-6). After 16 blocks these go on
// in FP64; the items' sums are added in a fixed order.
//
// What bounds it: issue (66 % at 27 k, 94 AOs, 60^3: 1.39 ms), which is the split of chi, read
// once, into its FP16 halves; with N = 16 the tensor pipe is 4 % busy. The earlier form
// generated the AOs of the k-mesh's supercell in FP16 blocks instead (D_1 D_2 D_3 / 2 times the
// products of this one, 36 % of them in reach): 2.09 of 3.43 ms of a build at 8 k, 104 AOs,
// 36^3, 5.5 of 7.9 ms at 6 k, 50^3, and 50 of 426 ms at 64 k, 350 AOs, 60^3.
// Every mbarrier wait is bounded by the plan's wait limit; on timeout the kernel records
// OCCRI_ETIMEOUT, stops issuing and waits once more (bounded too) for the products in flight.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "occri_ao.cuh"
#include "occri_chi.cuh"
#include "occri_device.cuh"
#include "occri_internal.h"
#include "occri_tc.cuh"

namespace occri {
namespace tcc {

constexpr int kM = 128;              // rows of a tile: Re, then Im, of kTcTile slots
constexpr int kK = 64;               // points per stage (two blocks)
constexpr int kSlices = kK / 16;     // MMA steps of a stage, each with its own accumulator
constexpr int kThreads = 256;
static_assert(kM == 2 * kTcTile, "rows of a tile");
// Operand layout (K-major, no swizzle): core matrices of 8 rows x 8 points (128 bytes) of one
// 8-point column one after another, columns 32 bytes past a multiple of 128 apart, so that a
// warp's stores of 2 points x 16 lanes x 2 rows hit 32 banks.
constexpr int kSBO = 128;
constexpr int lbo(int rows) { return rows / 8 * kSBO + 32; }
constexpr int op_bytes(int rows) { return kK / 8 * lbo(rows); }
__device__ __forceinline__ int op_off(int rows, int row, int k) {
  return (k >> 3) * lbo(rows) + (row >> 3) * kSBO + (row & 7) * 16 + (k & 7) * 2;
}

__device__ __forceinline__ void fail(int* status) {
  if (status && atomicCAS(status, 0, (int)OCCRI_ETIMEOUT) == 0) status[1] = -1;
}

// A warp's bounded wait: lane 0 waits and the warp follows its verdict (what comes next is
// warp-wide: tensor-memory loads need all 32 lanes), then every lane sees the phase itself.
__device__ __forceinline__ bool warp_wait(uint32_t bar, unsigned parity, long long limit_ns,
                                          int lane) {
  int ok = 1;
  if (lane == 0) ok = tc::mbar_wait(bar, parity, limit_ns) ? 1 : 0;
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (ok && lane != 0) tc::mbar_try_wait(bar, parity);
  return ok != 0;
}
constexpr long long kDrainNs = 2000000000LL;   // after a timeout: for the products in flight

// FP16 hi/lo split of two values, packed as two 32-bit words (x0 in the low half)
__device__ __forceinline__ void split2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(x0, x1);
  const float2 back = __half22float2(h);
  const __half2 l = __floats2half2_rn(x0 - back.x, x1 - back.y);
  memcpy(&hi, &h, 4);
  memcpy(&lo, &l, 4);
}

// 2^(13 - e) for a column whose largest |Re| + |Im| has exponent e (frexp)
__device__ __forceinline__ int col_exp(unsigned bits) {
  int e2 = 0;
  const float m = __uint_as_float(bits);
  if (m > 0.f) frexpf(m, &e2);
  return e2;
}

// largest |Re| + |Im| of every (k, i) field of Y, as float bits (cleared before)
__global__ void __launch_bounds__(256)
colmax_kernel(const float2* __restrict__ Y, unsigned* __restrict__ colmax, long long ng,
              long long fs) {
  float m = 0.f;
  for (long long q = (long long)blockIdx.y * 256 + threadIdx.x; q < ng; q += 256LL * gridDim.y) {
    const float2 v = Y[(size_t)blockIdx.x * fs + q];
    m = fmaxf(m, fabsf(v.x) + fabsf(v.y));
  }
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(colmax + blockIdx.x, __float_as_uint(m));
}

struct Smem {
  unsigned long long done;
  uint32_t tmem;
};

// FP32 sums end after kTcBlocks blocks. With 16 columns an item goes on over up to 64, its FP64 sums
// added to in place (27 k, 94 AOs, 60^3: 1.39 ms against 1.52 with items of kTcBlocks; 48^3, 64 k
// builds 44.2 -> 43.7 ms); wider kernels have no registers for that (nocc 20, 27 k, 30^3: 0.54
// against 0.44 ms) and take items of kTcBlocks.
template <int N> constexpr bool kFlush = N == 16;

// One work item per CTA: kTcTile slots of an atom over a run of blocks, at one k.
template <int N, bool REAL>
__global__ void __launch_bounds__(kThreads, N == 64 ? 2 : 3)
con_tc_kernel(chi::Params p, const void* __restrict__ chi, const float2* __restrict__ Y,
              const unsigned* __restrict__ colmax, int item0, int nitems, int* status,
              long long wait_ns, int fault) {
  constexpr int NI = N / 2;                       // orbitals, padded
  constexpr int AB = op_bytes(kM), BB = op_bytes(N);
  constexpr uint32_t kIdesc = tc::idesc_f16_f32(kM, N);
  constexpr int COLS = kSlices * N;               // an accumulator per 16-point slice
  constexpr int HB = NI / 16;                     // orbital pairs per warp and block (NI > 8)
  extern __shared__ __align__(1024) unsigned char sm[];
  unsigned char* a_hi = sm;
  unsigned char* a_lo = sm + AB;
  unsigned char* b_hi = sm + 2 * AB;
  unsigned char* b_lo = b_hi + BB;
  Smem& bar = *reinterpret_cast<Smem*>(b_lo + BB);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int w = blockIdx.x, k = blockIdx.y, nocc = p.a.nocc;
  const int4 it = p.items[item0 + w];
  const int nst = (it.w + 1) / 2;
  if (tid == 0) {
    tc::mbar_init(tc::smem_u32(&bar.done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) tc::tmem_alloc(tc::smem_u32(&bar.tmem), COLS);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = bar.tmem;

  // A lane's share of a stage: points 2 (lane mod 16) and the next one of block h, for the slots
  // (2 s + lane / 16) of the warp's eight, and the orbitals 2 (warp + 8 j) + lane / 16
  const int pt = 2 * (lane & 15), odd = lane >> 4;
  float4 av[2][4], bv[2][HB > 0 ? HB : 1];
  auto load = [&](int st) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const bool have = 2 * st + h < it.w;
      const int blk = have ? p.border[it.z + 2 * st + h] : 0;
      const int* aoff = p.aoff + (size_t)blk * (p.a.natm + 1);
      const int n = have ? aoff[it.x + 1] - aoff[it.x] - it.y : 0;   // slots of the tile here
      const size_t x = ((size_t)p.boff[blk] * p.a.nk + (size_t)k * aoff[p.a.natm] + aoff[it.x] +
                        it.y) * 32 + pt;
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int slot = 8 * warp + 2 * s + odd;
        av[h][s] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (slot < n) {
          if constexpr (REAL) {
            const float2 v = __ldg(reinterpret_cast<const float2*>((const float*)chi + x + 32 * slot));
            av[h][s] = make_float4(v.x, 0.f, v.y, 0.f);
          } else {
            av[h][s] = __ldg(reinterpret_cast<const float4*>((const float2*)chi + x + 32 * slot));
          }
        }
      }
      if constexpr (HB == 0) continue;
      bool v0, v1;
      long long q0, q1;
      ao::block_point(p.a, blk, pt, &v0, &q0);
      ao::block_point(p.a, blk, pt + 1, &v1, &q1);
#pragma unroll
      for (int j = 0; j < HB; ++j) {
        const int i = 2 * (warp + 8 * j) + odd;
        float2 y0 = make_float2(0.f, 0.f), y1 = y0;
        if (have && i < nocc) {
          const float2* f = Y + ((size_t)k * nocc + i) * p.a.fs;
          if (v0) y0 = __ldg(f + q0);
          if (v1) y1 = __ldg(f + q1);
        }
        bv[h][j] = make_float4(y0.x, y0.y, y1.x, y1.y);
      }
    }
  };
  // NI = 8: four orbital pairs, one per warp 0-3 of block 0 and per warp 4-7 of block 1
  const int i8 = 2 * (warp & 3) + odd;
  float4 b8 = make_float4(0.f, 0.f, 0.f, 0.f);
  auto load8 = [&](int st) {
    const int h = warp >> 2;
    b8 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (2 * st + h >= it.w || i8 >= nocc) return;
    const int blk = p.border[it.z + 2 * st + h];
    bool v0, v1;
    long long q0, q1;
    ao::block_point(p.a, blk, pt, &v0, &q0);
    ao::block_point(p.a, blk, pt + 1, &v1, &q1);
    const float2* f = Y + ((size_t)k * nocc + i8) * p.a.fs;
    if (v0) { const float2 y = __ldg(f + q0); b8.x = y.x; b8.y = y.y; }
    if (v1) { const float2 y = __ldg(f + q1); b8.z = y.x; b8.w = y.y; }
  };
  float rs[4], cs[HB > 0 ? HB : 1];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int slot = p.slot0[it.x] + it.y + 8 * warp + 2 * s + odd;
    rs[s] = slot < p.slot0[it.x + 1] ? p.row_scale[slot] : 1.f;
  }
  auto col_scale = [&](int i) {
    return i < nocc ? ldexpf(1.f, 13 - col_exp(colmax[(size_t)k * nocc + i])) : 1.f;
  };
  if constexpr (NI == 8) {
    cs[0] = col_scale(i8);
  } else {
#pragma unroll
    for (int j = 0; j < HB; ++j) cs[j] = col_scale(2 * (warp + 8 * j) + odd);
  }
  auto put = [&](unsigned char* hi, unsigned char* lo, int rows, int row_re, int row_im, int kp,
                 float4 v, float s) {
    uint32_t h, l;
    split2(v.x * s, v.z * s, h, l);
    const int o = op_off(rows, row_re, kp);
    *reinterpret_cast<uint32_t*>(hi + o) = h;
    *reinterpret_cast<uint32_t*>(lo + o) = l;
    split2(v.y * s, v.w * s, h, l);
    const int o2 = op_off(rows, row_im, kp);
    *reinterpret_cast<uint32_t*>(hi + o2) = h;
    *reinterpret_cast<uint32_t*>(lo + o2) = l;
  };
  auto store = [&]() {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int row = 8 * warp + 2 * s + odd;
        put(a_hi, a_lo, kM, row, kTcTile + row, 32 * h + pt, av[h][s], rs[s]);
      }
      if constexpr (NI > 8) {
#pragma unroll
        for (int j = 0; j < HB; ++j) {
          const int i = 2 * (warp + 8 * j) + odd;
          if (i < NI) put(b_hi, b_lo, N, i, NI + i, 32 * h + pt, bv[h][j], cs[j]);
        }
      }
    }
    if constexpr (NI == 8) put(b_hi, b_lo, N, i8, NI + i8, 32 * (warp >> 2) + pt, b8, cs[0]);
  };

  // a warp takes its lane quarter's rows: the first four warps the columns of Re Y, the others
  // those of Im Y
  float sum[NI];
#pragma unroll
  for (int j = 0; j < NI; ++j) sum[j] = 0.f;
  const uint32_t mine = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(NI * (warp >> 2));
  auto take = [&]() {
    tc::tc_fence_after();
#pragma unroll
    for (int c = 0; c < NI; c += 8) {
      uint32_t v[kSlices][8];
#pragma unroll
      for (int s = 0; s < kSlices; ++s) tc::tmem_ld8(mine + s * N + c, v[s]);
      tc::tmem_wait_ld();
#pragma unroll
      for (int j = 0; j < 8; ++j)
        sum[c + j] += (__uint_as_float(v[0][j]) + __uint_as_float(v[1][j])) +
                      (__uint_as_float(v[2][j]) + __uint_as_float(v[3][j]));
    }
    tc::tc_fence_before();
  };
  // the item's FP64 sums, part[k][item][row][column]; this thread adds to its own
  double* o = p.part + ((size_t)k * nitems + w) * kM * N +
              (size_t)(32 * (warp & 3) + lane) * N + NI * (warp >> 2);
  bool stored = false;
  auto flush = [&]() {
#pragma unroll
    for (int j = 0; j < NI; j += 2) {
      double2 t = make_double2((double)sum[j], (double)sum[j + 1]);
      double2* d = reinterpret_cast<double2*>(o + j);
      if (stored) {
        const double2 u = *d;
        t.x += u.x;
        t.y += u.y;
      }
      *d = t;
      sum[j] = sum[j + 1] = 0.f;
    }
    stored = true;
  };
  bool ok = true;
  auto fetch = [&](int st) {
    load(st);
    if constexpr (NI == 8) load8(st);
  };
  fetch(0);
  int st = 0;   // stages issued
#pragma unroll 1
  for (; st < nst; ++st) {
    if (st > 0) {
      ok = warp_wait(tc::smem_u32(&bar.done), (unsigned)((st - 1) & 1), wait_ns, lane);
      if (ok) take();
      if constexpr (kFlush<N>)
        if (st % (kTcBlocks / 2) == 0) flush();
    }
    if (ok) store();
    tc::fence_proxy_async_smem();
    if (!__syncthreads_and(ok ? 1 : 0)) {   // one warp's timeout ends the CTA's work
      ok = false;
      break;
    }
    if (tid == 0 && fault != OCCRI_FAULT_WAIT) {   // (test-only fault: nothing is issued)
      tc::tc_fence_after();
      const uint32_t ah = tc::smem_u32(a_hi), al = tc::smem_u32(a_lo), bh = tc::smem_u32(b_hi),
                     bl = tc::smem_u32(b_lo);
      // per 16-point slice, the small cross terms first: one addition rounds at full size
#pragma unroll
      for (int s = 0; s < kSlices; ++s) {
        const uint32_t ao = 2 * s * lbo(kM), bo = 2 * s * lbo(N), acc = tmem + s * N;
        const uint64_t da = tc::smem_desc(ah + ao, lbo(kM), kSBO);
        const uint64_t db = tc::smem_desc(bh + bo, lbo(N), kSBO);
        tc::mma_f16(acc, da, tc::smem_desc(bl + bo, lbo(N), kSBO), kIdesc, 0u);
        tc::mma_f16(acc, tc::smem_desc(al + ao, lbo(kM), kSBO), db, kIdesc, 1u);
        tc::mma_f16(acc, da, db, kIdesc, 1u);
      }
      tc::mma_commit(tc::smem_u32(&bar.done));
    }
    if (st + 1 < nst) fetch(st + 1);
  }
  // the last stage issued
  const unsigned parity = (unsigned)((st - 1) & 1);
  if (ok) {
    ok = warp_wait(tc::smem_u32(&bar.done), parity, wait_ns, lane);
    if (ok) take();
  }
  if (!ok) {
    // the sums are void; the products in flight still read shared memory and write tensor
    // memory, so the CTA keeps both until they are done (or this longer limit has passed too)
    if (fault != OCCRI_FAULT_WAIT)
      warp_wait(tc::smem_u32(&bar.done), parity, wait_ns > kDrainNs ? wait_ns : kDrainNs, lane);
    if (lane == 0) fail(status);
  }
  flush();
  tc::tc_fence_before();
  __syncthreads();   // every warp has read the accumulator
  if (warp == 0) tc::tmem_dealloc(tmem, COLS);
}

// kc[k][mu][i] = scale N_mu (sum of the items), or += after the first chunk: a CTA per (slot, k),
// a lane per orbital and part, every eighth run of items per warp, the warps' shares added in
// order.
template <int N>
__global__ void __launch_bounds__(256)
sum_tc_kernel(chi::Params p, const unsigned* __restrict__ colmax, double2* __restrict__ kc,
              double2* __restrict__ copy, int row_of0, int nitems, double scale, int add) {
  constexpr int NI = N / 2, Z = 8;
  __shared__ double share[Z][2 * NI];
  const int slot = blockIdx.x, k = blockIdx.y, nocc = p.a.nocc;
  const int mu = p.slot_ao[slot];
  if (mu < 0) return;
  int a = 0;
  while (slot >= p.slot0[a + 1]) ++a;
  const int s = slot - p.slot0[a], g = s / kTcTile, r = s % kTcTile;
  const int2 ro = p.rows_of[row_of0 + a];
  const int z = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double* src = p.part + ((size_t)k * nitems * kM + r) * N;
  for (int v = lane; v < 2 * nocc; v += 32) {
    const int i = v >> 1, im = v & 1;
    double t = 0.0;
#pragma unroll 4
    for (int y = z; y < ro.y; y += Z) {
      const int2 row = p.rows[ro.x + y];
      if (g >= row.y) continue;
      const double* q = src + (size_t)(row.x + g) * kM * N;
      t += im ? q[NI + i] - q[kTcTile * N + i] : q[i] + q[kTcTile * N + NI + i];
    }
    share[z][v] = t;
  }
  __syncthreads();
  if (z != 0) return;
  for (int v = lane; v < 2 * nocc; v += 32) {
    const int i = v >> 1, im = v & 1;
    double t = 0.0;
#pragma unroll
    for (int y = 0; y < Z; ++y) t += share[y][v];
    const double f = scale * p.ao_norm[mu] / (double)p.row_scale[slot] *
                     ldexp(1.0, col_exp(colmax[(size_t)k * nocc + i]) - 13);
    const size_t at = 2 * (((size_t)k * p.a.nao + mu) * nocc + i) + im;
    double* dst = reinterpret_cast<double*>(kc) + at;
    t = add ? *dst + f * t : f * t;
    *dst = t;
    if (copy) reinterpret_cast<double*>(copy)[at] = t;
  }
}

constexpr int width(int nocc) { return nocc <= 8 ? 16 : (nocc <= 16 ? 32 : 64); }

template <int N>
cudaError_t run(const Plan& p, const chi::Params& q, const ChiChunk& c, double2* copy,
                double scale, cudaStream_t s, LaunchHook* hook) {
  constexpr size_t smem = 2 * (size_t)(op_bytes(kM) + op_bytes(N)) + sizeof(Smem);
  static_assert(smem <= 75 * 1024, "three CTAs per SM");
  static DeviceCache attr;
  attr.get(p.device, [&] {
    cudaFuncSetAttribute(con_tc_kernel<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
    cudaFuncSetAttribute(con_tc_kernel<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem);
    return 1;
  });
  const dim3 grid(c.tc.nitems, p.nk);
  if (hook) hook->before();
  if (c.tc.nitems > 0 && q.signs)
    con_tc_kernel<N, true><<<grid, kThreads, smem, s>>>(q, p.chi->chi, (const float2*)p.Y, p.colmax,
                                                        c.tc.item0, c.tc.nitems, p.status, p.wait_ns,
                                                        p.fault);
  else if (c.tc.nitems > 0)
    con_tc_kernel<N, false><<<grid, kThreads, smem, s>>>(q, p.chi->chi, (const float2*)p.Y,
                                                         p.colmax, c.tc.item0, c.tc.nitems, p.status,
                                                         p.wait_ns, p.fault);
  if (hook) hook->after();
  sum_tc_kernel<N><<<dim3(q.nslots, p.nk), 256, 0, s>>>(q, p.colmax, p.kc, copy, c.tc.row_of0,
                                                                  c.tc.nitems, scale,
                                                                  c.b0 > 0 ? 1 : 0);
  return cudaGetLastError();
}

}  // namespace tcc

int tc_item_blocks(int nocc) { return tcc::width(nocc) == 16 ? 64 : kTcBlocks; }
size_t tc_item_values(int nocc) { return (size_t)tcc::kM * tcc::width(nocc); }
double tc_flops_per_stage(int nocc) { return 3.0 * 2.0 * tcc::kM * tcc::width(nocc) * tcc::kK; }
long long tc_plan_stages(const Plan& p) { return p.chi->item_pairs * p.nk; }
int tc_plan_launches(const Plan& p) {
  const int nc = (int)p.chi->chunks.size();
  return 1 + 2 * nc + (nc > 1 ? nc : 0);
}

cudaError_t launch_contract_tc(const Plan& p, double2* copy, cudaStream_t s, LaunchHook* hook) {
  using namespace tcc;
  const chi::Params q = chi::params(p);
  // Y carries N_g/(4 pi) (see PairParams), hence -Omega 4 pi / (N_k N_g^2)
  const double scale = -p.omega_cell * 4.0 * 3.14159265358979323846 /
                       ((double)p.nk * (double)p.ng * (double)p.ng);
  const int ncol = p.nk * p.nocc;
  cudaError_t e = cudaMemsetAsync(p.colmax, 0, sizeof(unsigned) * (size_t)ncol, s);
  if (e != cudaSuccess) return e;
  const int split = std::max(1, std::min((int)((p.ng + 1023) / 1024), 152 * 16 / ncol));
  colmax_kernel<<<dim3(ncol, split), 256, 0, s>>>((const float2*)p.Y, p.colmax, p.ng, p.fs);
  for (const ChiChunk& c : p.chi->chunks) {
    // one chunk: the buffer still holds chi from the orbitals of this build
    e = p.chi->chunks.size() > 1 ? chi::fill<float>(p, q, c, s) : cudaGetLastError();
    if (e != cudaSuccess) return e;
    switch (width(p.nocc)) {
      case 16: e = run<16>(p, q, c, copy, scale, s, hook); break;
      case 32: e = run<32>(p, q, c, copy, scale, s, hook); break;
      default: e = run<64>(p, q, c, copy, scale, s, hook); break;
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace occri
