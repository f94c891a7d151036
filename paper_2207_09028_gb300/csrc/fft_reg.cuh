// fft_reg.cuh -- one-thread, register-resident FFT of compile-time length.
//
// A length-N transform lives in registers. N = q_1 q_2 q_3 (its powers of 2, 3 and 5, which are
// coprime) is split by the prime-factor algorithm (Good 1958): with n = sum n_i N/q_i and
// k = the residues k_i (Chinese remainder theorem), e^{2 pi i n k/N} is the product of the
// factors' own exponentials, so no twiddles stand between the factors. A prime power q runs the
// decimation-in-frequency recursion q = R*M (R in {4,2,3,5}). Everything is unrolled at
// compile time: every index, every twiddle and the output permutation are constants.
// X[k] = sum_n x[n] e^{SIGN 2 pi i n k / N} with SIGN = -1 (forward) or +1 (inverse,
// unnormalised).
//
// Twiddle values come from a constexpr sine/cosine (Taylor series after exact
// integer octant reduction), evaluated by the compiler in double precision.
#pragma once
#include <utility>

#if defined(__CUDACC__)
#define OCCRI_HDI __host__ __device__ __forceinline__
#else
#define OCCRI_HDI inline
#endif

namespace occri {
namespace fft {

// ---------------------------------------------------------------- constexpr trig

constexpr double kPi = 3.14159265358979323846264338327950288;

constexpr double taylor_sin(double x) {
  double term = x, sum = x;
  for (int n = 1; n < 16; ++n) {
    term *= -x * x / ((2.0 * n) * (2.0 * n + 1.0));
    sum += term;
  }
  return sum;
}

constexpr double taylor_cos(double x) {
  double term = 1.0, sum = 1.0;
  for (int n = 1; n < 16; ++n) {
    term *= -x * x / ((2.0 * n - 1.0) * (2.0 * n));
    sum += term;
  }
  return sum;
}

// cos and sin of 2*pi*num/den with the angle reduced to [0, pi/4] exactly.
struct CS { double c, s; };

constexpr CS cs2pi(long long num, long long den) {
  long long r = num % den;
  if (r < 0) r += den;
  long long u = 8 * r;
  long long o = u / den;
  long long rem = u - o * den;
  double phi = (kPi / 4.0) * (double)rem / (double)den;
  double psi = (kPi / 4.0) * (double)(den - rem) / (double)den;
  double sp = taylor_sin(phi), cp = taylor_cos(phi);
  double sq = taylor_sin(psi), cq = taylor_cos(psi);
  switch (o) {
    case 0: return CS{cp, sp};
    case 1: return CS{sq, cq};
    case 2: return CS{-sp, cp};
    case 3: return CS{-cq, sq};
    case 4: return CS{-cp, -sp};
    case 5: return CS{-sq, -cq};
    case 6: return CS{sp, -cp};
    default: return CS{cq, -sq};
  }
}

// ---------------------------------------------------------------- compile-time loops

template <typename F, int... Is>
OCCRI_HDI void static_for_impl(F&& f, std::integer_sequence<int, Is...>) {
  (f(std::integral_constant<int, Is>{}), ...);
}

template <int N, typename F>
OCCRI_HDI void static_for(F&& f) {
  static_for_impl(f, std::make_integer_sequence<int, N>{});
}

// ---------------------------------------------------------------- radix plan

constexpr bool is_base(int n) { return n == 1 || n == 2 || n == 3 || n == 4 || n == 5; }

constexpr int pick_radix(int n) {
  return is_base(n) ? n : (n % 4 == 0 ? 4 : (n % 2 == 0 ? 2 : (n % 3 == 0 ? 3 : 5)));
}

constexpr bool smooth235(int n) {
  if (n < 1) return false;
  while (n % 2 == 0) n /= 2;
  while (n % 3 == 0) n /= 3;
  while (n % 5 == 0) n /= 5;
  return n == 1;
}

// Register position p holds output X[dif_rev(N, p)] after dif<N>.
constexpr int dif_rev(int n, int p) {
  if (is_base(n)) return p;
  int r = pick_radix(n), m = n / r;
  return r * dif_rev(m, p % m) + p / m;
}

// Coprime factors of a {2,3,5}-smooth N: its powers of 2, 3 and 5 (those above 1), in order.
constexpr int prime_part(int n, int p) {
  int q = 1;
  while (n % p == 0) { q *= p; n /= p; }
  return q;
}
constexpr int pf_count(int n) {
  return (prime_part(n, 2) > 1) + (prime_part(n, 3) > 1) + (prime_part(n, 5) > 1);
}
constexpr int pf(int n, int i) {
  for (int p : {2, 3, 5})
    if (prime_part(n, p) > 1 && i-- == 0) return prime_part(n, p);
  return 1;
}
constexpr int inv_mod(int a, int m) {
  for (int x = 0; x < m; ++x)
    if ((a * x) % m == 1 % m) return x;
  return 0;
}
// The k modulo n with k = 1 modulo its factor q and 0 modulo the others.
constexpr int crt_unit(int n, int q) { return (n / q) * inv_mod((n / q) % q, q) % n; }

// Register p = sum n_i N/q_i (mod N) holds output X[pfa_out(N, p)] after pfa<N>.
constexpr int pfa_out(int n, int p) {
  int k = 0;
  for (int i = 0; i < pf_count(n); ++i) {
    const int q = pf(n, i);
    const int ni = (p % q) * inv_mod((n / q) % q, q) % q;
    k = (k + dif_rev(q, ni) * crt_unit(n, q)) % n;
  }
  return k;
}

// ---------------------------------------------------------------- butterflies

// Elements A, A + S, ... of the TOT registers, indices modulo TOT.
template <int SIGN, int A, int S, typename T, int TOT>
OCCRI_HDI void dft2(T (&re)[TOT], T (&im)[TOT]) {
  constexpr int a = A % TOT, b = (A + S) % TOT;
  const T ar = re[a], ai = im[a], br = re[b], bi = im[b];
  re[a] = ar + br; im[a] = ai + bi;
  re[b] = ar - br; im[b] = ai - bi;
}

template <int SIGN, int A, int S, typename T, int TOT>
OCCRI_HDI void dft3(T (&re)[TOT], T (&im)[TOT]) {
  constexpr int a = A % TOT, b = (A + S) % TOT, c = (A + 2 * S) % TOT;
  constexpr T h = T(SIGN * 0.86602540378443864676372317075293618);  // sqrt(3)/2
  const T t1r = re[b] + re[c], t1i = im[b] + im[c];
  const T dr = re[b] - re[c], di = im[b] - im[c];
  const T t2r = fma(T(-0.5), t1r, re[a]), t2i = fma(T(-0.5), t1i, im[a]);
  re[a] = re[a] + t1r; im[a] = im[a] + t1i;
  // t2 +- i SIGN h d
  re[b] = fma(-h, di, t2r); im[b] = fma(h, dr, t2i);
  re[c] = fma(h, di, t2r); im[c] = fma(-h, dr, t2i);
}

template <int SIGN, int A, int S, typename T, int TOT>
OCCRI_HDI void dft4(T (&re)[TOT], T (&im)[TOT]) {
  constexpr int a = A % TOT, b = (A + S) % TOT, c = (A + 2 * S) % TOT, d = (A + 3 * S) % TOT;
  const T s0r = re[a] + re[c], s0i = im[a] + im[c];
  const T d0r = re[a] - re[c], d0i = im[a] - im[c];
  const T s1r = re[b] + re[d], s1i = im[b] + im[d];
  const T d1r = re[b] - re[d], d1i = im[b] - im[d];
  // SIGN * i * d1 = (-SIGN d1i, SIGN d1r)
  const T jr = (SIGN > 0) ? -d1i : d1i;
  const T ji = (SIGN > 0) ? d1r : -d1r;
  re[a] = s0r + s1r; im[a] = s0i + s1i;
  re[c] = s0r - s1r; im[c] = s0i - s1i;
  re[b] = d0r + jr; im[b] = d0i + ji;
  re[d] = d0r - jr; im[d] = d0i - ji;
}

// Five points: the sines enter as s_1 (t3 + (s_2/s_1) t4) and s_1 ((s_2/s_1) t3 - t4), the outer
// factor in the last multiply-adds: 32 operations. In FP32 fl(s_1) fl(s_2/s_1) makes the
// transform's gain 1.6e-8 too large, which no sum averages out. Where two stages of five follow
// each other (25 points) that is more than rounding each constant by itself costs (3.3e-8 against
// 1.9e-8): there the second row is s_2 (t3 - (s_1/s_2) t4) (0.8e-8 a stage, 1.7e-8). With one
// stage the gains of whole lines stay within 0.3e-8 of those of rounded constants, and a 45-point
// line in one thread's registers would be 2 % slower with the two constants more.
template <int TOT> constexpr bool two_sines() { return TOT % 25 == 0; }
template <int SIGN, int A, int S, typename T, int TOT>
OCCRI_HDI void dft5(T (&re)[TOT], T (&im)[TOT]) {
  constexpr CS w1 = cs2pi(1, 5), w2 = cs2pi(2, 5);
  constexpr int e0 = A % TOT, e1 = (A + S) % TOT, e2 = (A + 2 * S) % TOT, e3 = (A + 3 * S) % TOT,
                e4 = (A + 4 * S) % TOT;
  const T ar = re[e0], ai = im[e0];
  const T t1r = re[e1] + re[e4], t1i = im[e1] + im[e4];
  const T t2r = re[e2] + re[e3], t2i = im[e2] + im[e3];
  const T t3r = re[e1] - re[e4], t3i = im[e1] - im[e4];
  const T t4r = re[e2] - re[e3], t4i = im[e2] - im[e3];
  constexpr T c1 = T(w1.c), c2 = T(w2.c), s1 = T(SIGN * w1.s), s2 = T(SIGN * w2.s),
              r1 = T(w2.s / w1.s), r2 = T(w1.s / w2.s);
  const T p1r = fma(c2, t2r, fma(c1, t1r, ar)), p1i = fma(c2, t2i, fma(c1, t1i, ai));
  const T p2r = fma(c1, t2r, fma(c2, t1r, ar)), p2i = fma(c1, t2i, fma(c2, t1i, ai));
  const T q1r = fma(r1, t4r, t3r), q1i = fma(r1, t4i, t3i);    // times i s_1 below
  constexpr T so = two_sines<TOT>() ? s2 : s1;                 // times i s_o
  const T q2r = two_sines<TOT>() ? fma(-r2, t4r, t3r) : fma(r1, t3r, -t4r);
  const T q2i = two_sines<TOT>() ? fma(-r2, t4i, t3i) : fma(r1, t3i, -t4i);
  re[e0] = ar + (t1r + t2r); im[e0] = ai + (t1i + t2i);
  re[e1] = fma(-s1, q1i, p1r); im[e1] = fma(s1, q1r, p1i);
  re[e4] = fma(s1, q1i, p1r); im[e4] = fma(-s1, q1r, p1i);
  re[e2] = fma(-so, q2i, p2r); im[e2] = fma(so, q2r, p2i);
  re[e3] = fma(so, q2i, p2r); im[e3] = fma(-so, q2r, p2i);
}

template <int R, int SIGN, int A, int S, typename T, int TOT>
OCCRI_HDI void small_dft(T (&re)[TOT], T (&im)[TOT]) {
  if constexpr (R == 2) dft2<SIGN, A, S>(re, im);
  else if constexpr (R == 3) dft3<SIGN, A, S>(re, im);
  else if constexpr (R == 4) dft4<SIGN, A, S>(re, im);
  else if constexpr (R == 5) dft5<SIGN, A, S>(re, im);
}

// x[P] *= e^{SIGN 2 pi i E / N}
template <int N, int SIGN, int E, int PP, typename T, int TOT>
OCCRI_HDI void twiddle(T (&re)[TOT], T (&im)[TOT]) {
  constexpr int e = E % N, P = PP % TOT;
  if constexpr (e == 0) {
  } else if constexpr (2 * e == N) {
    re[P] = -re[P]; im[P] = -im[P];
  } else if constexpr (4 * e == N || 4 * e == 3 * N) {
    // multiply by (+/-) i
    constexpr int sgn = (4 * e == N) ? SIGN : -SIGN;
    const T r = re[P], i = im[P];
    if constexpr (sgn > 0) { re[P] = -i; im[P] = r; } else { re[P] = i; im[P] = -r; }
  } else {
    constexpr CS w = cs2pi(e, N);
    const T c = T(w.c), s = T(SIGN * w.s);
    const T r = re[P], i = im[P];
    re[P] = r * c - i * s;
    im[P] = r * s + i * c;
  }
}

// In-place DIF of the N elements at positions A + S*idx (modulo TOT).
template <int N, int SIGN, int A, int S, typename T, int TOT>
OCCRI_HDI void dif(T (&re)[TOT], T (&im)[TOT]) {
  if constexpr (N == 1) {
  } else if constexpr (is_base(N)) {
    small_dft<N, SIGN, A, S>(re, im);
  } else {
    constexpr int R = pick_radix(N), M = N / R;
    static_for<M>([&](auto I1) {
      constexpr int n1 = decltype(I1)::value;
      small_dft<R, SIGN, A + S * n1, S * M>(re, im);
      static_for<R>([&](auto K1) {
        constexpr int k1 = decltype(K1)::value;
        twiddle<N, SIGN, n1 * k1, A + S * (n1 + M * k1)>(re, im);
      });
    });
    static_for<R>([&](auto K1) {
      constexpr int k1 = decltype(K1)::value;
      dif<M, SIGN, A + S * M * k1, S>(re, im);
    });
  }
}

// Full transform: after the call, register p holds X[pfa_out(N, p)].
template <int N, int SIGN, typename T>
OCCRI_HDI void pfa(T (&re)[N], T (&im)[N]) {
  static_assert(smooth235(N), "FFT length must be {2,3,5}-smooth");
  static_for<pf_count(N)>([&](auto F) {
    constexpr int q = pf(N, decltype(F)::value), S = N / q;
    // the transforms of length q: one per value of the other factors' indices, i.e. per
    // multiple of q modulo N
    static_for<S>([&](auto J) { dif<q, SIGN, (decltype(J)::value * q) % N, S>(re, im); });
  });
}

// ---------------------------------------------------------------- packed FP32 form
// The same decimation-in-frequency recursion for FP32 with each complex value held as
// one 64-bit register pair {re, im}. Operations that act alike on both halves (sums,
// differences, scaling by a real constant) are single packed f32x2 instructions
// (add/sub/mul/fma.rn.f32x2, sm_100 and later); products with +-i and the twiddles,
// which mix the halves, are scalar operations on the pair's halves. Every packed
// instruction rounds each half exactly as the scalar instruction would.
#if defined(__CUDACC__)
namespace pk {
using u64 = unsigned long long;
__device__ __forceinline__ u64 pack(float re, float im) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(re), "f"(im));
  return r;
}
__device__ __forceinline__ void unpack(u64 v, float& re, float& im) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(re), "=f"(im) : "l"(v));
}
__device__ __forceinline__ u64 add(u64 a, u64 b) {
  u64 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 sub(u64 a, u64 b) {
  u64 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 mul(u64 a, u64 b) {
  u64 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 fma(u64 a, u64 b, u64 c) {   // a * b + c
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ u64 splat(float c) { return pack(c, c); }
// SGN * i * x = (-SGN x.im, SGN x.re)
template <int SGN>
__device__ __forceinline__ u64 mul_i(u64 x) {
  float r, i;
  unpack(x, r, i);
  return SGN > 0 ? pack(-i, r) : pack(i, -r);
}
// (a - b) with its halves exchanged, for a later multiply-add by (-s, s) = i s
__device__ __forceinline__ u64 sub_swap(u64 a, u64 b) {
  float ar, ai, br, bi;
  unpack(a, ar, ai);
  unpack(b, br, bi);
  return pack(ai - bi, ar - br);
}
// x * (c + i s), scalar on the halves so that c and s stay instruction immediates
__device__ __forceinline__ u64 cmul_const(u64 x, float c, float s) {
  float r, i;
  unpack(x, r, i);
  return pack(r * c - i * s, r * s + i * c);
}
}  // namespace pk

template <int SIGN, int A, int S, int TOT>
__device__ __forceinline__ void pdft2(pk::u64 (&x)[TOT]) {
  constexpr int e0 = A % TOT, e1 = (A + S) % TOT;
  const pk::u64 a = x[e0], b = x[e1];
  x[e0] = pk::add(a, b);
  x[e1] = pk::sub(a, b);
}

template <int SIGN, int A, int S, int TOT>
__device__ __forceinline__ void pdft3(pk::u64 (&x)[TOT]) {
  constexpr int e0 = A % TOT, e1 = (A + S) % TOT, e2 = (A + 2 * S) % TOT;
  constexpr float h = float(SIGN * 0.86602540378443864676372317075293618);  // sqrt(3)/2
  const pk::u64 a = x[e0];
  const pk::u64 t1 = pk::add(x[e1], x[e2]);
  const pk::u64 d = pk::sub_swap(x[e1], x[e2]);
  const pk::u64 t2 = pk::fma(t1, pk::splat(-0.5f), a);
  x[e0] = pk::add(a, t1);
  x[e1] = pk::fma(d, pk::pack(-h, h), t2);   // t2 + i h (x1 - x2)
  x[e2] = pk::fma(d, pk::pack(h, -h), t2);
}

template <int SIGN, int A, int S, int TOT>
__device__ __forceinline__ void pdft4(pk::u64 (&x)[TOT]) {
  constexpr int e0 = A % TOT, e1 = (A + S) % TOT, e2 = (A + 2 * S) % TOT, e3 = (A + 3 * S) % TOT;
  constexpr float h = float(SIGN);
  const pk::u64 s0 = pk::add(x[e0], x[e2]);
  const pk::u64 d0 = pk::sub(x[e0], x[e2]);
  const pk::u64 s1 = pk::add(x[e1], x[e3]);
  const pk::u64 d1 = pk::sub_swap(x[e1], x[e3]);
  x[e0] = pk::add(s0, s1);
  x[e2] = pk::sub(s0, s1);
  x[e1] = pk::fma(d1, pk::pack(-h, h), d0);   // d0 + i SIGN (x1 - x3)
  x[e3] = pk::fma(d1, pk::pack(h, -h), d0);
}

// As dft5, the terms that multiply i with their halves exchanged.
template <int SIGN, int A, int S, int TOT>
__device__ __forceinline__ void pdft5(pk::u64 (&x)[TOT]) {
  constexpr CS w1 = cs2pi(1, 5), w2 = cs2pi(2, 5);
  constexpr int e0 = A % TOT, e1 = (A + S) % TOT, e2 = (A + 2 * S) % TOT, e3 = (A + 3 * S) % TOT,
                e4 = (A + 4 * S) % TOT;
  const pk::u64 a = x[e0];
  const pk::u64 t1 = pk::add(x[e1], x[e4]);
  const pk::u64 t2 = pk::add(x[e2], x[e3]);
  const pk::u64 t3 = pk::sub_swap(x[e1], x[e4]);
  const pk::u64 t4 = pk::sub_swap(x[e2], x[e3]);
  const pk::u64 c1 = pk::splat(float(w1.c)), c2 = pk::splat(float(w2.c));
  constexpr float s1 = float(SIGN * w1.s), s2 = float(SIGN * w2.s);
  constexpr float r1 = float(w2.s / w1.s), r2 = float(w1.s / w2.s);
  const pk::u64 p1 = pk::fma(t2, c2, pk::fma(t1, c1, a));
  const pk::u64 p2 = pk::fma(t2, c1, pk::fma(t1, c2, a));
  const pk::u64 q1 = pk::fma(t4, pk::splat(r1), t3);
  // -q2 where s_o = s_1: one multiply-add either way
  const pk::u64 q2 = two_sines<TOT>() ? pk::fma(t4, pk::splat(-r2), t3)
                                      : pk::fma(t3, pk::splat(-r1), t4);
  constexpr float so = two_sines<TOT>() ? s2 : -s1;
  x[e0] = pk::add(pk::add(t1, t2), a);
  x[e1] = pk::fma(q1, pk::pack(-s1, s1), p1);   // p1 + i s_1 q1
  x[e4] = pk::fma(q1, pk::pack(s1, -s1), p1);
  x[e2] = pk::fma(q2, pk::pack(-so, so), p2);
  x[e3] = pk::fma(q2, pk::pack(so, -so), p2);
}

template <int R, int SIGN, int A, int S, int TOT>
__device__ __forceinline__ void psmall_dft(pk::u64 (&x)[TOT]) {
  if constexpr (R == 2) pdft2<SIGN, A, S>(x);
  else if constexpr (R == 3) pdft3<SIGN, A, S>(x);
  else if constexpr (R == 4) pdft4<SIGN, A, S>(x);
  else if constexpr (R == 5) pdft5<SIGN, A, S>(x);
}

// x[P] *= e^{SIGN 2 pi i E / N}
template <int N, int SIGN, int E, int PP, int TOT>
__device__ __forceinline__ void ptwiddle(pk::u64 (&x)[TOT]) {
  constexpr int e = E % N, P = PP % TOT;
  if constexpr (e == 0) {
  } else if constexpr (2 * e == N) {
    x[P] = pk::sub(pk::splat(0.0f), x[P]);
  } else if constexpr (4 * e == N || 4 * e == 3 * N) {
    constexpr int sgn = (4 * e == N) ? SIGN : -SIGN;
    x[P] = pk::mul_i<sgn>(x[P]);
  } else {
    constexpr CS w = cs2pi(e, N);
    x[P] = pk::cmul_const(x[P], float(w.c), float(SIGN * w.s));
  }
}

template <int N, int SIGN, int A, int S, int TOT>
__device__ __forceinline__ void pdif(pk::u64 (&x)[TOT]) {
  if constexpr (N == 1) {
  } else if constexpr (is_base(N)) {
    psmall_dft<N, SIGN, A, S>(x);
  } else {
    constexpr int R = pick_radix(N), M = N / R;
    static_for<M>([&](auto I1) {
      constexpr int n1 = decltype(I1)::value;
      psmall_dft<R, SIGN, A + S * n1, S * M>(x);
      static_for<R>([&](auto K1) {
        constexpr int k1 = decltype(K1)::value;
        ptwiddle<N, SIGN, n1 * k1, A + S * (n1 + M * k1)>(x);
      });
    });
    static_for<R>([&](auto K1) {
      constexpr int k1 = decltype(K1)::value;
      pdif<M, SIGN, A + S * M * k1, S>(x);
    });
  }
}

// Packed FP32 transform: after the call, x[p] holds X[pfa_out(N, p)].
template <int N, int SIGN>
__device__ __forceinline__ void ppfa(pk::u64 (&x)[N]) {
  static_assert(smooth235(N), "FFT length must be {2,3,5}-smooth");
  static_for<pf_count(N)>([&](auto F) {
    constexpr int q = pf(N, decltype(F)::value), S = N / q;
    static_for<S>([&](auto J) { pdif<q, SIGN, (decltype(J)::value * q) % N, S>(x); });
  });
}
#endif

}  // namespace fft
}  // namespace occri
