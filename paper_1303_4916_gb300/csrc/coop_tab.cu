// coop_tab.cu -- host side of herm_coop.cuh: the index tables of the
// warp-cooperative Hermite kernels, one per class, behind an index of HF_NCLASS
// words.  The device reads them; their order is CoopTab's.
#include <algorithm>
#include <vector>

#include "eri_classes.cuh"
#include "herm_coop.cuh"
#include "hf_internal.h"

namespace {

using hfk::hidx;
using hfk::hpow;
using hfk::nherm;

struct Term {
  int u;              // Hermite index
  uint32_t factors;   // places in the e row
};
// expansion of component idx (a Hermite index) of a pair whose powers reach I
std::vector<Term> terms(int idx, int I) {
  const int f[3] = {hpow(idx, 0), hpow(idx, 1), hpow(idx, 2)};
  auto place = [&](int d, int n) { return f[d] == 0 ? 0u : (uint32_t)(1 + d * hfk::e_size(I) + f[d] * (f[d] + 1) / 2 - 1 + n); };
  std::vector<Term> t;
  for (int x = 0; x <= f[0]; ++x)
    for (int y = 0; y <= f[1]; ++y)
      for (int z = 0; z <= f[2]; ++z) t.push_back(Term{hidx(x, y, z), place(0, x) | place(1, y) << 8 | place(2, z) << 16});
  return t;
}

template <class C>
void add_class(std::vector<uint32_t>& out) {
  using T = hfk::CoopTab<C>;
  std::vector<uint32_t> t(T::END, 0u);
  for (int i = 1; i < T::NR; ++i) {
    const int ax = hfk::herm_axis(i), pw = hpow(i, ax);
    t[T::R0 + i - 1] = (uint32_t)i | (uint32_t)hfk::hdown(i, ax, 1) << 8 |
                       (pw > 1 ? (uint32_t)hfk::hdown(i, ax, 2) << 16 : 0u) | (uint32_t)ax << 24 | (uint32_t)(pw - 1) << 26;
  }
  // inside a total power the entries without a second term first (even rounds)
  for (int n = 1; n <= T::L; ++n)
    std::stable_sort(t.begin() + T::R0 + nherm(n - 1) - 1, t.begin() + T::R0 + nherm(n) - 1,
                     [](uint32_t a, uint32_t b) { return (a >> 26) < (b >> 26); });
  int n = 0;
  for (int f = 0; f < C::NF; ++f)
    for (const Term& x : terms(hfk::set0(C::LC) + f, T::LK)) t[T::K0 + n++] = x.factors;
  n = 0;
  for (int e = 0; e < C::NE; ++e) {
    const std::vector<Term> b = terms(hfk::set0(C::LA) + e, T::LB);
    for (int f = 0; f < C::NF; ++f)
      t[T::A0 + e * C::NF + f] = (uint32_t)b.size() | (uint32_t)n << 4 | (uint32_t)f << 12;
    for (const Term& x : b) {
      t[T::AU0 + n] = (uint32_t)x.u;
      t[T::B0 + n++] = x.factors;
    }
  }
  for (int h = 0; h < T::NT; ++h)
    for (int u = 0; u < T::NU; ++u)
      t[T::P0 + h * T::NUW + u / 4] |=
          (uint32_t)hidx(hpow(h, 0) + hpow(u, 0), hpow(h, 1) + hpow(u, 1), hpow(h, 2) + hpow(u, 2)) << 8 * (u % 4);
  out[class_index(C::LA, C::LB, C::LC, C::LD)] = (uint32_t)out.size();
  out.insert(out.end(), t.begin(), t.end());
}

}  // namespace

std::vector<uint32_t> hf_coop_tables() {
  std::vector<uint32_t> t(HF_NCLASS, 0u);
  add_class<hfgen::C_dp_pp>(t);
  add_class<hfgen::C_dp_ds>(t);
  add_class<hfgen::C_dp_dp>(t);
  add_class<hfgen::C_dd_ps>(t);
  add_class<hfgen::C_dd_pp>(t);
  add_class<hfgen::C_dd_ds>(t);
  add_class<hfgen::C_dd_dp>(t);
  add_class<hfgen::C_dd_dd>(t);
  return t;
}
