// Host build of the tabulated S_m(y) of the Hermite kernels (csrc/herm.cuh) for
// tests/test_herm_host.py (test infrastructure).  The test copies the header
// with its three inline-assembly statements replaced (the 32-byte loads by plain
// ones); the device intrinsics it uses are IEEE-754 operations or moves of bits.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

template <class T, class U>
static inline T same_bits(U u) {
  static_assert(sizeof(T) == sizeof(U), "size");
  T t;
  std::memcpy(&t, &u, sizeof t);
  return t;
}
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static inline float __double2float_rn(double x) { return (float)x; }
static inline float rsqrtf(float x) { return 1.0f / std::sqrt(x); }
// the device's conversion saturates, and gives 0 for a NaN
static inline int __float2int_rn(float x) { return x != x ? 0 : x >= 2147483648.0f ? 2147483647 : (int)std::nearbyint(x); }
static inline int __double2hiint(double x) { return (int)(same_bits<long long>(x) >> 32); }
static inline int __double2loint(double x) { return (int)same_bits<long long>(x); }
static inline double __hiloint2double(int h, int l) { return same_bits<double>((long long)(((unsigned long long)(unsigned)h << 32) | (unsigned)l)); }
static inline double __longlong_as_double(long long x) { return same_bits<double>(x); }
static inline unsigned __float_as_uint(float x) { return same_bits<unsigned>(x); }
static inline int __float_as_int(float x) { return same_bits<int>(x); }
static inline float __uint_as_float(unsigned x) { return same_bits<float>(x); }
static inline float __int_as_float(int x) { return same_bits<float>(x); }
// the hardware's estimate: the low word is zero
static inline double host_rsqrt_estimate(double a) { return same_bits<double>(same_bits<long long>(1.0 / std::sqrt(a)) & ~0xffffffffll); }
static inline int min(int a, int b) { return a < b ? a : b; }
#include "herm_host.cuh"

// S_0 .. S_L at y in FP64 (s) and df64 (d: hi, lo pairs; y is split into a pair)
template <int L>
static void all(const unsigned* t64, const unsigned* tdf, double y, double* s, float* d) {
  KernelCommon kc{};
  kc.boysy64 = t64;
  kc.boysydf = tdf;
  hfk::boys_y<L>(y, kc, s);
  df64 q[L + 1];
  hfk::boys_y<L>(df64(y), kc, q);
  for (int m = 0; m <= L; ++m) {
    d[2 * m] = q[m].hi;
    d[2 * m + 1] = q[m].lo;
  }
}
extern "C" void s_all(int L, const unsigned* t64, const unsigned* tdf, double y, double* s, float* d) {
  void (*const f[])(const unsigned*, const unsigned*, double, double*, float*) = {all<0>, all<1>, all<2>, all<3>, all<4>,
                                                                                  all<5>, all<6>, all<7>, all<8>};
  f[L](t64, tdf, y, s, d);
}
extern "C" int words64() { return (int)boysy64_off(BOYSY_LMAX + 1); }
extern "C" int wordsdf() { return (int)boysydf_off(BOYSY_LMAX + 1); }
extern "C" double rsqrt64(double a) { return hfk::hf_rsqrt(a); }
