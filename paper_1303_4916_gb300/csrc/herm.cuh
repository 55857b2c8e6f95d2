// herm.cuh -- contracted [e0|f0] block of one shell quartet with the bra in
// Hermite Gaussians (McMurchie and Davidson, J. Comput. Phys. 26, 218 (1978)),
// for the thread-per-quartet classes in FP64 and df64.
//
// What bounds these kernels in FP64 is the count of FP64 instructions: on
// GB300 one of them holds a sub-partition's FP64 pipe for 64 cycles however
// many lanes it serves, and everything else (FP32, integer, loads) issues
// beside it.  So the scheme here spends FP32 and integer instructions to
// save FP64 ones:
//  * The primitive loop runs bra outer, ket inner, and per bra primitive the
//    inner loop only accumulates H[t][f] = sum_ket K rs [t|f0], t the Hermite
//    indices up to la + lb; the expansion of the bra's [e0| in them (the
//    E coefficients in PA and 1/(2p), the bra prefactor) is applied once per
//    bra primitive, outside the inner loop.  The Obara-Saika form carried
//    it through every primitive quartet.
//  * Exponents enter through s = 1/(2p) + 1/(2q) alone: with rs = s^(-1/2),
//    w = rs^2 = 2 rho and y = w |PQ|^2 = 2 T, (-2 rho)^m F_m(T) =
//    w^m S_m(y), S_m(y) = (-1)^m F_m(y / 2); the remaining sqrt(1 / (pq)) is
//    in the records' prefactors.
//  * 1/sqrt is the hardware estimate and one third-order correction, four
//    FP64 instructions (hf_rsqrt).
//  * S_m is a tabulated FP64 value plus a Taylor tail of at most 2^-7 of it
//    (2^-5.9 in the far rows), evaluated in double-float arithmetic (48 bits) on
//    the FP32 pipe: two FP64 additions per order instead of an eight-term FP64
//    Horner.  The table index and the offset come from the bits of y, without
//    FP64 conversions.  Against 40-digit values the worst relative error is
//    1.9 x 2^-53 below T = 60 and, above it, 2.0 up to m = 6, 4.2 at m = 7 and
//    6.9 at m = 8, where the first term left out of the tail shows.  (The FP64
//    Horner with downward recursion: 1.8 to 10.8 below T = 60 from L = 0 to 8,
//    and the upward recursion 2.4 to 28 above it.)  In df64, in units of 2^-48:
//    at most 1.9 for all orders (before: 1.4 to 5 below T = 60, 4.5 to 45 above).
// (ps|ss), FP64: 0.0489 ns per primitive quartet on the whole GPU, from 0.0996
// (the pipe's rate is 629e9 FP64 instructions x lanes per second: the time of
// 31 of them, of which 27 are executed; 63 before).
#pragma once
#include <type_traits>
#include <utility>

#include "df64.cuh"
#include "hf_device.h"

namespace hfk {

// ------------------------------------------------------------- compile-time indices
template <int N>
using ic = std::integral_constant<int, N>;
template <class F, int... I>
__device__ __forceinline__ void sfor_impl(F&& f, std::integer_sequence<int, I...>) {
  (f(ic<I>{}), ...);
}
// f(0), ..., f(N - 1) with each index a constant expression
template <int N, class F>
__device__ __forceinline__ void sfor(F&& f) {
  sfor_impl(f, std::make_integer_sequence<int, N>{});
}

__host__ __device__ constexpr int nherm(int L) { return (L + 1) * (L + 2) * (L + 3) / 6; }
// (t, u, v) of total n at nherm(n - 1) + its place among the Cartesian
// components of l = n (x power descending, then y)
__host__ __device__ constexpr int hidx(int t, int u, int v) {
  const int n = t + u + v, r = u + v;
  return nherm(n - 1) + r * (r + 1) / 2 + v;
}
__host__ __device__ constexpr int hpow(int idx, int dir) {
  int n = 0;
  while (nherm(n) <= idx) ++n;
  int k = idx - nherm(n - 1), r = 0;
  while ((r + 1) * (r + 2) / 2 <= k) ++r;
  const int v = k - r * (r + 1) / 2, t = n - r, u = r - v;
  return dir == 0 ? t : dir == 1 ? u : v;
}
// the e0 (or f0) set of a pair (la, lb): components of l = la .. la + lb in
// order; they are the Hermite indices from nherm(la - 1) on
__host__ __device__ constexpr int set0(int la) { return nherm(la - 1); }

// ------------------------------------------------------------- arithmetic
__device__ __forceinline__ double zero_of(double) { return 0.0; }
__device__ __forceinline__ df64 zero_of(df64) { return df64(0.0f, 0.0f); }
__device__ __forceinline__ double times_int(double a, int k) { return k * a; }
__device__ __forceinline__ df64 times_int(df64 a, int k) { return df_mulf(a, (float)k); }
__device__ __forceinline__ double fmah(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ df64 fmah(df64 a, df64 b, df64 c) { return df_fma(a, b, c); }

// y^2 for a positive normal y whose low word is zero, exact: the square of the
// 21-bit significand in integers, so no FP64 instruction
__device__ __forceinline__ double square_high(double y) {
  const unsigned h = (unsigned)__double2hiint(y), m = (h & 0xfffffu) | 0x100000u;
  const unsigned long long q = (unsigned long long)m * m;  // in [2^40, 2^42)
  const int up = (int)(q >> 41);                           // 1: at least 2^41
  const unsigned long long f = q << (12 - up);             // in [2^52, 2^53)
  return __longlong_as_double((long long)(((unsigned long long)(2 * (int)(h >> 20) - 1024 + up) << 52) + f));
}

// 1/sqrt(a), a normal and positive: the hardware estimate y0 (its low word is
// zero: 21 bits) and the binomial series of (1 - e)^(-1/2), e = 1 - a y0^2, to
// second order in e; the neglected 5/16 e^3 is below 2^-57.
__device__ __forceinline__ double hf_rsqrt(double a) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double e = fma(-a, square_high(y), 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ df64 hf_rsqrt(df64 a) { return rsqrt(a); }

// A float as a double by moving its bits (no conversion instruction, which
// would take an FP64 slot).  Zero and subnormals come out as values below
// 2^-126, which vanish in the sums they enter.
__device__ __forceinline__ double bits_to_double(float f) {
  const unsigned u = __float_as_uint(f);
  return __hiloint2double((int)((((u & 0x7fffffffu) >> 3) + 0x38000000u) | (u & 0x80000000u)), (int)(u << 29));
}

// ------------------------------------------------------------- S_m(y)
__device__ __forceinline__ void ldg256u(const unsigned* __restrict__ p, unsigned* v) {
  asm("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
      : "l"(p));
}

// a b + c in double-float for |a b| below |c|: one product, a quick two-sum
__device__ __forceinline__ df64 df_fma_small(df64 a, df64 b, df64 c) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  const float s = __fadd_rn(c.hi, p);
  const float r = __fsub_rn(p, __fsub_rn(s, c.hi));
  return df64(s, __fadd_rn(r, __fadd_rn(e, c.lo)));
}

// S_{m+1} + z/2 (S_{m+2} + z/3 (S_{m+3} + z/4 g)): the Taylor tail over z, g
// the sum of the higher terms (below 2^-24 of the tail).
__device__ __forceinline__ df64 taylor_tail(df64 z, df64 z3, df64 s1, df64 s2, df64 s3, float g) {
  df64 f = df_quick_two_sum(s3.hi, __fmaf_rn(g, z.hi * 0.25f, s3.lo));
  f = df_fma_small(f, z3, s2);
  return df_fma_small(f, df64(z.hi * 0.5f, z.lo * 0.5f), s1);
}
// z / 3
__device__ __forceinline__ df64 third(df64 z) {
  constexpr float h = (float)(1.0 / 3.0), l = (float)(1.0 / 3.0 - (double)(float)(1.0 / 3.0));
  return z * df64(h, l);
}
// 2^e as a float, zero below the normal range
__device__ __forceinline__ float pow2f(int e) { return e < -126 ? 0.0f : __int_as_float((e + 127) << 23); }

// S_0 .. S_L at y >= 0.  Below 120 from the rows y_i = i / 32; from there on
// F_m(T) is its large-T form (what is neglected is below e^-60), a power of
// T, so y / 4^k in [32, 128) is looked up in rows y_i = i / 8 of that form
// and S_m is scaled by 2^(-k (2m + 1)): the same instructions for both, where
// a branch made most warps of a spread-out molecule run both sides (0.0439
// against 0.0352 ns per (ss|ss) primitive quartet of a 40-atom one).
template <int L>
__device__ __forceinline__ void boys_y(double y, const KernelCommon& kc, double* S) {
  constexpr int ROW = BOYSY64_ROW(L), P0 = 2 * (L + 1), F0 = P0 + 2 * (L + 3);
  const unsigned hi = (unsigned)__double2hiint(y), lo = (unsigned)__double2loint(y);
  const bool far = hi >= 0x405e0000u;  // y >= 120
  const int k = far ? (int)((hi >> 20) - 1028u) >> 1 : 0;
  // y / 4^k in units of 2^-57 (it is below 2^7): the 53-bit significand,
  // shifted to its place
  const unsigned sh = 1029u - ((hi >> 20) - 2 * k);
  const unsigned long long M = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 43) | ((unsigned long long)lo << 11);
  const unsigned long long Y = sh > 63u ? 0ull : M >> sh;
  const unsigned yh = (unsigned)(Y >> 32), yl = (unsigned)Y;
  const unsigned i = far ? ((yh >> 1) + (1u << 20)) >> 21 : (yh + (1u << 19)) >> 20;
  // z = (y / 4^k - y_i) / 2 in units of 2^-58: the upper part exact in a float
  const int xh = (int)(yh - (i << (far ? 22 : 20)));
  const float zh = (float)(int)(((unsigned)xh << 3) | (yl >> 29)) * 0x1p-29f;
  const float zl = (float)(int)(yl & 0x1fffffffu) * 0x1p-58f;
  const df64 z = df_quick_two_sum(zh, zl), z3 = third(z);
  unsigned r[ROW];
  unsigned at = far ? i + (BOYSY64_NNEAR - 256) : i;
  if (!HF_BCHECK(kc, at < BOYSY64_NNEAR + BOYSY_NFAR, HF_BC_BOYS, at)) at = 0;
  const unsigned* const row = kc.boysy64 + boysy64_off(L) + (size_t)at * ROW;
#pragma unroll
  for (int j = 0; j < ROW; j += 8) ldg256u(row + j, r + j);
  auto pr = [&](int j) { return df64(__uint_as_float(r[P0 + 2 * (j - 1)]), __uint_as_float(r[P0 + 2 * (j - 1) + 1])); };
  auto fl = [&](int j) { return __uint_as_float(j <= L + 3 ? r[P0 + 2 * (j - 1)] : r[F0 + j - L - 4]); };
#pragma unroll
  for (int m = 0; m <= L; ++m) {
    float g = __fmaf_rn(fl(m + 6), z.hi * (1.0f / 6.0f), fl(m + 5));
    g = __fmaf_rn(g, z.hi * 0.2f, fl(m + 4));
    const df64 t = taylor_tail(z, z3, pr(m + 1), pr(m + 2), pr(m + 3), g);
    const float p = __fmul_rn(t.hi, z.hi);
    float e = __fmaf_rn(t.hi, z.hi, -p);
    e = __fmaf_rn(t.hi, z.lo, e);
    e = __fmaf_rn(t.lo, z.hi, e);
    const double v = (__hiloint2double((int)r[2 * m + 1], (int)r[2 * m]) + bits_to_double(e)) + bits_to_double(p);
    // times 2^(-k (2m + 1)) in the exponent field
    const int vh = __double2hiint(v), drop = k * (2 * m + 1);
    S[m] = drop < ((vh >> 20) & 0x7ff) ? __hiloint2double(vh - (drop << 20), __double2loint(v)) : 0.0;
  }
}

// The same in double-float throughout, with rows y_i = i / 8 in both ranges
// (|z| <= 2^-5, one more float term): a table a quarter of the FP64 one's
// size, since here the row loads are a larger share of the time.  The far index
// is bounded: centres far enough apart (1e16 bohr) overflow y.
template <int L>
__device__ __forceinline__ void boys_y(df64 y, const KernelCommon& kc, df64* S) {
  const bool far = y.hi >= 120.0f;
  const int k = far ? ((__float_as_int(y.hi) >> 23) - 132) >> 1 : 0;
  const float sc = pow2f(-2 * k);
  const float yh = y.hi * sc, yl = y.lo * sc;  // exact
  if constexpr (L == 0) {
    // (ss|ss) is bound by L1 (each lane's row is a wavefront of its own), so
    // its row is one 32-byte load on a finer grid (|z| <= 2^-8, far 2^-7 with
    // T >= 16): terms to S_4
    const float gs = far ? 32.0f : 64.0f;
    const int i = __float2int_rn(yh * gs);
    const float xh = __fsub_rn(yh, (float)i * (far ? 1.0f / 32.0f : 1.0f / 64.0f));  // exact (Sterbenz)
    const df64 z = df_quick_two_sum(0.5f * xh, 0.5f * yl);
    unsigned r[8];
    int at = far ? min(i, 4096) + (BOYSYDF0_NNEAR - 1024) : i;
    if (!HF_BCHECK(kc, at >= 0 && at < BOYSYDF0_NNEAR + BOYSYDF0_NFAR, HF_BC_BOYS, at)) at = 0;
    ldg256u(kc.boysydf + (size_t)at * 8, r);
    auto w = [&](int j) { return __uint_as_float(r[j]); };
    const float g = __fmaf_rn(w(7), z.hi * 0.25f, w(6));
    df64 f = df_quick_two_sum(w(4), __fmaf_rn(g, z.hi * (1.0f / 3.0f), w(5)));
    f = df_fma_small(f, df64(0.5f * z.hi, 0.5f * z.lo), df64(w(2), w(3)));
    f = df_fma_small(f, z, df64(w(0), w(1)));
    f = df_quick_two_sum(f.hi, f.lo);
    const float s = pow2f(-k);
    S[0] = df64(f.hi * s, f.lo * s);
    return;
  }
  constexpr int ROW = BOYSYDF_ROW(L), F0 = 2 * (L + 4);
  const int i = __float2int_rn(yh * 8.0f);
  const float xh = __fsub_rn(yh, (float)i * 0.125f);  // exact (Sterbenz)
  const df64 z = df_quick_two_sum(0.5f * xh, 0.5f * yl), z3 = third(z);
  unsigned r[ROW];
  int at = far ? min(i, 1024) + (BOYSYDF_NNEAR - 256) : i;
  if (!HF_BCHECK(kc, at >= 0 && at < BOYSYDF_NNEAR + BOYSY_NFAR, HF_BC_BOYS, at)) at = 0;
  const unsigned* const row = kc.boysydf + boysydf_off(L) + (size_t)at * ROW;
#pragma unroll
  for (int j = 0; j < ROW; j += 8) ldg256u(row + j, r + j);
  auto pr = [&](int j) { return df64(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1])); };
  auto fl = [&](int j) { return __uint_as_float(j <= L + 3 ? r[2 * j] : r[F0 + j - L - 4]); };
#pragma unroll
  for (int m = 0; m <= L; ++m) {
    float g = __fmaf_rn(fl(m + 7), z.hi * (1.0f / 7.0f), fl(m + 6));
    g = __fmaf_rn(g, z.hi * (1.0f / 6.0f), fl(m + 5));
    g = __fmaf_rn(g, z.hi * 0.2f, fl(m + 4));
    const df64 f = df_fma_small(taylor_tail(z, z3, pr(m + 1), pr(m + 2), pr(m + 3), g), z, pr(m));
    const df64 v = df_quick_two_sum(f.hi, f.lo);
    const float s = pow2f(-k * (2 * m + 1));
    S[m] = df64(v.hi * s, v.lo * s);
  }
}

// ------------------------------------------------------------- records
// 1/(2p), P, PA, K'' (the pair's prefactor with the exponent factor folded in)
template <typename R>
struct HPrim {
  R o2, P[3], PA[3], K;
};
__device__ __forceinline__ void load_hprim(const PairSet& s, int idx, HPrim<double>& q) {
  const double* p = s.prim64 + (size_t)idx * PRIM64_STRIDE;
  double v[8];
  asm("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(p));
  asm("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(v[4]), "=d"(v[5]), "=d"(v[6]), "=d"(v[7]) : "l"(p + 4));
  q.o2 = v[0]; q.P[0] = v[1]; q.P[1] = v[2]; q.P[2] = v[3];
  q.PA[0] = v[4]; q.PA[1] = v[5]; q.PA[2] = v[6]; q.K = v[7];
}
__device__ __forceinline__ void load_hprim(const PairSet& s, int idx, HPrim<df64>& q) {
  const unsigned* p = reinterpret_cast<const unsigned*>(s.primdf + (size_t)idx * PRIMDF_STRIDE);
  unsigned v[16];
  ldg256u(p, v);
  ldg256u(p + 8, v + 8);
  auto g = [&](int k) { return df64(__uint_as_float(v[2 * k]), __uint_as_float(v[2 * k + 1])); };
  q.o2 = g(0); q.P[0] = g(1); q.P[1] = g(2); q.P[2] = g(3);
  q.PA[0] = g(4); q.PA[1] = g(5); q.PA[2] = g(6); q.K = g(7);
}

// ------------------------------------------------------------- Hermite integrals
// r[hidx] = R_tuv from B[m] = R^(m)_000 (m = 0..L), in place from the highest
// order: R^(m)_{t+1} = PQ R^(m+1)_t + t R^(m+1)_{t-1} along the axis with the
// smallest power (no second term where that is one).
__host__ __device__ constexpr int herm_axis(int idx) {
  int best = -1;
  for (int d = 0; d < 3; ++d)
    if (hpow(idx, d) > 0 && (best < 0 || hpow(idx, d) < hpow(idx, best))) best = d;
  return best;
}
__host__ __device__ constexpr int hdown(int idx, int dir, int k) {
  return hidx(hpow(idx, 0) - (dir == 0 ? k : 0), hpow(idx, 1) - (dir == 1 ? k : 0), hpow(idx, 2) - (dir == 2 ? k : 0));
}
template <int L, typename R>
__device__ __forceinline__ void herm_r(const R* B, const R* PQ, R* r) {
  r[0] = B[L];
  sfor<L>([&](auto step) {
    constexpr int m = L - 1 - decltype(step)::value, N = nherm(L - m);
    sfor<N - 1>([&](auto k) {
      constexpr int idx = N - 1 - decltype(k)::value, ax = herm_axis(idx), pw = hpow(idx, ax);
      constexpr int d1 = hdown(idx, ax, 1);
      if constexpr (pw == 1) {
        r[idx] = PQ[ax] * r[d1];
      } else {
        constexpr int d2 = hdown(idx, ax, 2);
        if constexpr (pw == 2) r[idx] = fmah(PQ[ax], r[d1], r[d2]);
        else r[idx] = fmah(PQ[ax], r[d1], times_int(r[d2], pw - 1));
      }
    });
    r[0] = B[m];
  });
}

// One-dimensional expansion coefficients of (x - X0)^i in Hermite Gaussians,
// times SGN^n (SGN = -1 on the ket, whose derivatives act on -Q):
// e^{i+1}_n = SGN h e^i_{n-1} + X e^i_n + SGN (n + 1) e^i_{n+1}, n <= i + 1,
// with h = 1/(2p).  e[0][0] = 1 is not stored: its factor is skipped.
template <int I, int SGN, typename R>
__device__ __forceinline__ void herm_e(R X, R h, R (&e)[I + 1][I + 1]) {
  const R hs = SGN > 0 ? h : -h;
  if constexpr (I >= 1) {
    e[1][0] = X;
    e[1][1] = hs;
  }
  sfor<I - 1 < 0 ? 0 : I - 1>([&](auto ii) {
    constexpr int i = decltype(ii)::value + 1;
    sfor<i + 2>([&](auto nn) {
      constexpr int n = decltype(nn)::value;
      R v;
      if constexpr (n > i) v = hs * e[i][n - 1];
      else if constexpr (n == 0) v = fmah(X, e[i][0], SGN > 0 ? e[i][1] : -e[i][1]);
      else if constexpr (n == i) v = fmah(hs, e[i][n - 1], X * e[i][n]);
      else v = fmah(hs, e[i][n - 1], fmah(X, e[i][n], times_int(e[i][n + 1], SGN * (n + 1))));
      e[i + 1][n] = v;
    });
  });
}

// acc[e * NF + f] += over bra records [b0, b0 + nb) and ket records [k0, k0 +
// nk) (nk differs per lane; 0 for an inactive lane).
template <class C>
__device__ __forceinline__ void contracted_herm(const PairSet& ps, const KernelCommon& kc, int b0, int nb, int k0,
                                                int nk, double* acc) {
  using R = double;
  constexpr int LBR = C::LA + C::LB, LK = C::LC + C::LD, L = LBR + LK;
  constexpr int NT = nherm(LBR), NF = C::NF, NE = C::NE;
  const R zero = zero_of(R{});
#pragma unroll
  for (int x = 0; x < NE * NF; ++x) acc[x] = zero;
  for (int ib = 0; ib < nb; ++ib) {
    HPrim<R> a;
    load_hprim(ps, b0 + ib, a);
    R H[NT * NF];
#pragma unroll
    for (int x = 0; x < NT * NF; ++x) H[x] = zero;
    for (int ik = 0; ik < nk; ++ik) {
      HPrim<R> c;
      load_hprim(ps, k0 + ik, c);
      const R rs = hf_rsqrt(a.o2 + c.o2);
      const R w = rs * rs;
      R PQ[3];
#pragma unroll
      for (int x = 0; x < 3; ++x) PQ[x] = a.P[x] - c.P[x];
      const R y = w * fmah(PQ[0], PQ[0], fmah(PQ[1], PQ[1], PQ[2] * PQ[2]));
      R B[L + 1];
      boys_y<L>(y, kc, B);
      R g = c.K * rs;
      if constexpr (L == 0) {
        H[0] = fmah(g, B[0], H[0]);
      } else {
        if constexpr (LK == 0) H[0] = fmah(g, B[0], H[0]);  // R_000 goes nowhere else
        else B[0] = g * B[0];
#pragma unroll
        for (int m = 1; m <= L; ++m) {
          g = g * w;
          B[m] = g * B[m];
        }
        R r[nherm(L)];
        herm_r<L>(B, PQ, r);
        if constexpr (LK == 0) {
#pragma unroll
          for (int t = 1; t < NT; ++t) H[t] = H[t] + r[t];
        } else {
          R e[3][LK + 1][LK + 1];
#pragma unroll
          for (int d = 0; d < 3; ++d) herm_e<LK, -1>(c.PA[d], c.o2, e[d]);
          // H[t][f] += sum_u (-1)^u E_f^u R_{t+u}
          sfor<NF>([&](auto fc) {
            constexpr int f = decltype(fc)::value, fi = set0(C::LC) + f;
            constexpr int fx = hpow(fi, 0), fy = hpow(fi, 1), fz = hpow(fi, 2);
            sfor<(fx + 1) * (fy + 1) * (fz + 1)>([&](auto uc) {
              constexpr int k = decltype(uc)::value;
              constexpr int uz = k % (fz + 1), uy = (k / (fz + 1)) % (fy + 1), ux = k / ((fz + 1) * (fy + 1));
              if constexpr (fx + fy + fz == 0) {
#pragma unroll
                for (int t = 0; t < NT; ++t) H[t * NF + f] = H[t * NF + f] + r[t];
              } else {
                R co = zero;
                if constexpr (fx > 0) co = e[0][fx][ux];
                if constexpr (fy > 0) {
                  if constexpr (fx > 0) co = co * e[1][fy][uy];
                  else co = e[1][fy][uy];
                }
                if constexpr (fz > 0) {
                  if constexpr (fx + fy > 0) co = co * e[2][fz][uz];
                  else co = e[2][fz][uz];
                }
                sfor<NT>([&](auto tc) {
                  constexpr int t = decltype(tc)::value;
                  constexpr int s = hidx(hpow(t, 0) + ux, hpow(t, 1) + uy, hpow(t, 2) + uz);
                  H[t * NF + f] = fmah(co, r[s], H[t * NF + f]);
                });
              }
            });
          });
        }
      }
    }
    // the bra's [e0| in Hermite Gaussians, with its prefactor
    R e[3][LBR + 1][LBR + 1];
#pragma unroll
    for (int d = 0; d < 3; ++d) herm_e<LBR, 1>(a.PA[d], a.o2, e[d]);
    sfor<NE>([&](auto ec) {
      constexpr int ei = set0(C::LA) + decltype(ec)::value;
      constexpr int ex = hpow(ei, 0), ey = hpow(ei, 1), ez = hpow(ei, 2);
      sfor<(ex + 1) * (ey + 1) * (ez + 1)>([&](auto uc) {
        constexpr int k = decltype(uc)::value;
        constexpr int uz = k % (ez + 1), uy = (k / (ez + 1)) % (ey + 1), ux = k / ((ez + 1) * (ey + 1));
        R co = a.K;
        if constexpr (ex > 0) co = co * e[0][ex][ux];
        if constexpr (ey > 0) co = co * e[1][ey][uy];
        if constexpr (ez > 0) co = co * e[2][ez][uz];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          constexpr int t = hidx(ux, uy, uz);
          R& v = acc[decltype(ec)::value * NF + f];
          v = fmah(co, H[t * NF + f], v);
        }
      });
    });
  }
}

// The same by the class's generated Obara-Saika recurrence (ket outer, bra
// inner), with the set-up and S_m of the Hermite form: rho / p = w / (2p),
// rho / q = w / (2q), 1 / (2(p+q)) = (rho / p) / (2q).
template <class C, typename R>
__device__ __forceinline__ void contracted_os(const PairSet& ps, const KernelCommon& kc, int b0, int nb, int k0, int nk,
                                              R* acc) {
  const R zero = zero_of(R{});
#pragma unroll
  for (int x = 0; x < C::NE * C::NF; ++x) acc[x] = zero;
  for (int ik = 0; ik < nk; ++ik) {
    HPrim<R> c;
    load_hprim(ps, k0 + ik, c);
    for (int ib = 0; ib < nb; ++ib) {
      HPrim<R> a;
      load_hprim(ps, b0 + ib, a);
      const R rs = hf_rsqrt(a.o2 + c.o2);
      const R w = rs * rs;
      const R rp = w * a.o2, rq = w * c.o2;
      R PQ[3], WP[3], WQ[3];
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        PQ[x] = a.P[x] - c.P[x];
        WP[x] = -(rp * PQ[x]);
        WQ[x] = rq * PQ[x];
      }
      R B[C::L + 1];
      boys_y<C::L>(w * fmah(PQ[0], PQ[0], fmah(PQ[1], PQ[1], PQ[2] * PQ[2])), kc, B);
      const R g = a.K * c.K * rs;
#pragma unroll
      for (int m = 0; m <= C::L; ++m) B[m] = (m & 1 ? -g : g) * B[m];
      C::template vrr<R>(acc, B, a.PA, WP, c.PA, WQ, a.o2, c.o2, rp * c.o2, rp, rq);
    }
  }
}

// Which form a class takes, as measured.  FP64 is bound by its FP64 instruction
// count, of which the Hermite form has fewer; (ds|pp), with 10 Hermite indices
// over 9 ket components, is the one class where the Obara-Saika form is faster
// all the same ((pp|pp) has as many sums, spills 2 KB and still gains).  df64 is bound by FP32 issue and by L1 (a lane's own ket record per
// primitive quartet, as the ket loop is the inner one): the Obara-Saika order,
// with the ket record loaded once, is the faster.  Hermite against
// Obara-Saika, ns per primitive quartet on the whole GPU (40-atom s+p and
// 9- and 20-atom s+p+d molecules):
//   FP64  (ss|ss) .0352/.0369  (ps|ss) .0508/.0613  (ps|ps) .126/.131  (pp|ss) .0954/.115  (pp|ps) .256/.284
//         (pp|pp) .99/1.07  (ds|ss) .115/.137  (ds|ps) .310/.319  (ds|ds) 1.52/1.53  (ds|pp) 1.16/1.06
//         (dp|ss) .228/.313  (dp|ps) .64/.75  (dd|ss) .60/.74
//   df64  (ss|ss) .0142/.0090  (ps|ss) .0154/.0130  (ps|ps) .0299/.0281  (pp|ss) .0257/.0257  (pp|ps) .128/.087
//         (ds|ds) .76/.42  (ds|pp) 1.40/.53  (dp|ps) .55/.32  (dd|ss) .43/.27
template <class C, typename R>
__device__ __forceinline__ void contracted(const PairSet& ps, const KernelCommon& kc, int b0, int nb, int k0, int nk,
                                           R* acc) {
  constexpr bool ds_pp = C::LA == 2 && C::LB == 0 && C::LC == 1 && C::LD == 1;
  if constexpr (std::is_same<R, double>::value && !ds_pp) contracted_herm<C>(ps, kc, b0, nb, k0, nk, acc);
  else contracted_os<C, R>(ps, kc, b0, nb, k0, nk, acc);
}

}  // namespace hfk
