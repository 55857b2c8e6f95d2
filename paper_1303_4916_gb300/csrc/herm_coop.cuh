// herm_coop.cuh -- the contracted [e0|f0] set of one shell quartet by one warp,
// the bra in Hermite Gaussians (herm.cuh), for the classes with L >= 5 in
// FP64 and df64.
//
// Per bra primitive the warp sums H[t][f] = sum over a group of ket primitives
// of K rs sum_u (-1)^u E_f^u R_{t+u}, a lane per t with the f in registers and
// every index a constant but R's place; then one pass applies the bra's
// expansion.  The Hermite integrals R are built level by level in shared
// memory, their set-up (as in herm.cuh) 32 primitive quartets at a time, the
// ket's coefficients once per group.  The Obara-Saika node lists this replaces
// evaluated every node of the bra and of the ket per primitive quartet
// (a J/K build of a 9-atom s+p+d molecule 22.7 -> 20.2 ms in FP64, of a 20-atom
// one in df64 with an FP32 split 45 -> 36.4 ms, 36.6 with the range rule below).
// Index tables (coop_tab.cu) are kept with the context.
//
// Range in df64: the set-up forms w^m, m <= 8, w = 2 rho up to twice the smaller
// exponent, and floats end at 2^127: plain d shells of exponent 2500 overflow
// (and a NaN follows), diffuse ones of 1e-3 lose their low words.  So a
// quartet whose exponents leave the range where that cannot happen is taken in
// powers of two: lengths in units of 2^-a, 4^a near its largest w, so that the
// expansion coefficients are of order one; and per primitive quartet with k,
// 4^k near w in those units, R^(m)_N is formed times 2^(-k (N + 2m)), which the
// recursion keeps (PQ times 2^k, w times 4^-k), and the finished R_N is put
// back by 2^(k N).  Only exponents change, so nothing is rounded by it.  It is an
// instantiation of its own (SCALED): woven into the plain one, where it does
// nothing, it cost a 20-atom build 1.4 %.
#pragma once
#include "herm.cuh"

namespace hfk {

// one-dimensional coefficients e[i][n], 1 <= i <= I, n <= i, in a row:
// e[i][n] at i (i + 1) / 2 - 1 + n
__host__ __device__ constexpr int e_size(int I) { return (I + 1) * (I + 2) / 2 - 1; }
// terms of the expansion of every component of l = la .. la + lb
__host__ __device__ constexpr int herm_terms(int la, int lb) {
  int n = 0;
  for (int i = nherm(la - 1); i < nherm(la + lb); ++i) n += (hpow(i, 0) + 1) * (hpow(i, 1) + 1) * (hpow(i, 2) + 1);
  return n;
}
// terms of the components of l >= la that come before Hermite index idx
__host__ __device__ constexpr int nherm_terms_before(int la, int idx) {
  int n = 0;
  for (int i = nherm(la - 1); i < idx; ++i) n += (hpow(i, 0) + 1) * (hpow(i, 1) + 1) * (hpow(i, 2) + 1);
  return n;
}

// Shape of a class: NT Hermite indices t of the bra on TM lanes (the power of
// two below NT) for PM = 32 / TM primitive quartets side by side, the TL left
// over on TL lanes each of the up to KC quartets of a group, so that both
// passes fill the warp (20 = 16 + 4 and 35 = 32 + 3 for dp and dd).  KC, the
// ket primitives of a group, is what shared memory allows.
template <class C>
struct CoopTab {
  static constexpr int LB = C::LA + C::LB, LK = C::LC + C::LD, L = LB + LK;
  static constexpr int NT = nherm(LB), NU = nherm(LK), NF = C::NF, NA = C::NE * C::NF, NR = nherm(L);
  static constexpr int TM = NT >= 32 ? 32 : NT >= 16 ? 16 : NT >= 8 ? 8 : 4, PM = 32 / TM, TL = NT - TM;
  static constexpr int NCK = herm_terms(C::LC, C::LD), NCB = herm_terms(C::LA, C::LB);
  // Bra primitives outermost where the pass that applies the bra's expansion
  // (NA outputs) is long: it then runs once per bra primitive, and the ket's
  // coefficients are formed again for each; else ket groups outermost, the
  // coefficients formed once.  KC and ROWS let two blocks share an SM.
  static constexpr bool BRA_OUTER = NA > 300;
  static constexpr int KC = BRA_OUTER ? 4 : 8, ROWS = NA > 600 ? 16 : 32;
  static constexpr int NUW = (NU + 3) / 4;
  // word offsets of the class's table
  static constexpr int R0 = 0;               // [NR - 1] dst | d1 << 8 | d2 << 16 | axis << 24 | (power - 1) << 26, by total
  static constexpr int K0 = R0 + NR - 1;     // [NCK] x | y << 8 | z << 16: places of the factors in the e row (0: one)
  static constexpr int B0 = K0 + NCK;        // [NCB]
  static constexpr int A0 = B0 + NCB;        // [NA] terms | coefficient << 4 | f << 12
  static constexpr int AU0 = A0 + NA;        // [NCB] the Hermite index of each bra term
  static constexpr int P0 = AU0 + NCB;       // [NT][NUW] places of R_{t+u}, four u to a word
  static constexpr int END = P0 + NT * NUW;
  // a warp's shared slice, in R: the [e0|f0] sums, set-up rows, coefficients,
  // Hermite integrals of a group (H overlays them), left-over sums
  static constexpr int ROW = (3 + L + 1) | 1, NEK = 1 + 3 * e_size(LK), NEB = 1 + 3 * e_size(LB);
  static constexpr int RG = KC * NR > NT * NF ? KC * NR : NT * NF;
  static constexpr int SX = KC * NR > KC * TL * NF ? KC * NR : KC * TL * NF;   // second integral buffer, left-over sums
  static constexpr int SC = BRA_OUTER && KC * NCK > SX ? KC * NCK : SX;        // and, bra outermost, the coefficients
  static constexpr int oA = 0, oRow = oA + NA, oE = oRow + ROWS * ROW, oCB = oE + (KC * NEK > NEB ? KC * NEK : NEB),
                       oR = oCB + NCB, oS = oR + RG, oX = oS, oCK = BRA_OUTER ? oS : oS + SC,
                       WS = oS + SC + (BRA_OUTER ? 0 : KC * NCK);
};

// k a for the second term of the recursion, k = power - 1 (0 where it has none)
static __constant__ double kSmallInt[8] = {0.0, 1.0, 2.0, 3.0, 4.0, 5.0, 6.0, 7.0};
__device__ __forceinline__ double times_small(double a, int k) { return kSmallInt[k] * a; }  // no conversion
__device__ __forceinline__ df64 times_small(df64 a, int k) { return df_mulf(a, (float)k); }

// H[f] += sum_u c[f, u] R_{t+u} for one t: every index but R's place is a
// constant, so the multiply-adds of different f follow each other freely.
template <class C, typename R>
__device__ __forceinline__ void herm_terms_add(const R* __restrict__ Rq, const R* __restrict__ c, const uint32_t* place,
                                               R* H) {
  using T = CoopTab<C>;
  sfor<T::NU>([&](auto uc) {
    constexpr int u = decltype(uc)::value, ux = hpow(u, 0), uy = hpow(u, 1), uz = hpow(u, 2);
    const R r = Rq[(place[u / 4] >> (8 * (u % 4))) & 255u];
    sfor<C::NF>([&](auto fc) {
      constexpr int f = decltype(fc)::value, fi = set0(C::LC) + f;
      constexpr int fx = hpow(fi, 0), fy = hpow(fi, 1), fz = hpow(fi, 2);
      if constexpr (ux <= fx && uy <= fy && uz <= fz) {
        constexpr int at = nherm_terms_before(C::LC, fi) + (ux * (fy + 1) + uy) * (fz + 1) + uz;
        H[f] = fmah(c[at], r, H[f]);
      }
    });
  });
}

// product of the up to three factors a coefficient word names in the e row
template <typename R>
__device__ __forceinline__ R coef_of(uint32_t w, const R* er, R first) {
  R v = first;
  if (w & 255u) v = v * er[w & 255u];
  if ((w >> 8) & 255u) v = v * er[(w >> 8) & 255u];
  if (w >> 16) v = v * er[w >> 16];
  return v;
}
// times a power of two
__device__ __forceinline__ df64 times_pow2(df64 a, float s) { return df64(a.hi * s, a.lo * s); }
// The plain range of a quartet (all bounds on the exponent e of 2p, 2^e <= 2p):
// w < 2^10 and >= 2^-7, prefactors of pairs below 2^14 (g w^8 of two d pairs
// there is below 1e33 and, at the diffuse end, above 1e-25).
__device__ __forceinline__ bool plain_range(const PairInfo& bra, const PairInfo& ket) {
  return min(bra.emax, ket.emax) <= 9 && max(bra.emax, ket.emax) <= 13 && min(bra.emin, ket.emin) >= -6;
}
__device__ __forceinline__ double one_of(double) { return 1.0; }
__device__ __forceinline__ df64 one_of(df64) { return df64(1.0f, 0.0f); }

// e row of dimension d of a record
template <int I, int SGN, typename R>
__device__ __forceinline__ void store_e(R X, R h, R* er, int d) {
  R e[I + 1][I + 1];
  herm_e<I, SGN>(X, h, e);
  sfor<I>([&](auto ii) {
    constexpr int i = decltype(ii)::value + 1;
#pragma unroll
    for (int n = 0; n <= i; ++n) er[1 + d * e_size(I) + i * (i + 1) / 2 - 1 + n] = e[i][n];
  });
}

// The [e0|f0] of (bra|ket) over the primitive quartets [q_lo, q_hi) (bra
// primitive major) into s[oA ..]; SCALED outside the plain range.
template <class C, typename R, bool SCALED>
__device__ __forceinline__ void coop_herm(const PairSet& P, const KernelCommon& kc, const PairInfo& bra,
                                          const PairInfo& ket, int q_lo, int q_hi, R* const s, const int lane) {
  using T = CoopTab<C>;
  constexpr int L = T::L, LK = T::LK, LB = T::LB, NF = C::NF;
  const R zero = zero_of(R{});
  for (int k = lane; k < T::NA; k += 32) s[T::oA + k] = zero;
  if (q_hi <= q_lo) {  // an empty part, or a pair without significant primitives
    __syncwarp();
    return;
  }
  const uint32_t* __restrict__ tab = kc.cooptab + __ldg(kc.cooptab + class_index(C::LA, C::LB, C::LC, C::LD));
  const int nk = ket.nprim;
  const int tm = lane % T::TM, sm = lane / T::TM;                   // main pass: t, quartet of the pass
  const int tl = T::TL > 0 ? T::TM + lane % (T::TL > 0 ? T::TL : 1) : 0, sl = lane / (T::TL > 0 ? T::TL : 1);  // left-over pass
  uint32_t pm[T::NUW], pl[T::NUW];
#pragma unroll
  for (int k = 0; k < T::NUW; ++k) {
    pm[k] = __ldg(tab + T::P0 + tm * T::NUW + k);
    pl[k] = __ldg(tab + T::P0 + tl * T::NUW + k);
  }
  const int ib_lo = q_lo / nk, ib_hi = (q_hi - 1) / nk + 1;
  // lengths in units of 2^-ua; the bound keeps 2^(7 ua) a float
  [[maybe_unused]] const int ua = SCALED ? max(-18, min(18, min(bra.emax, ket.emax) >> 1)) : 0;
  [[maybe_unused]] int kq = 0;  // k of the primitive quartet of this lane's set-up row
  auto len = [&](R x) { if constexpr (SCALED) return times_pow2(x, pow2f(ua)); else return x; };       // a length
  auto area = [&](R x) { if constexpr (SCALED) return times_pow2(x, pow2f(2 * ua)); else return x; };  // 1 / (2p)
  R H[NF], X[NF];
  // e rows of the ket primitives [kb, ke), at most KC
  auto ket_rows = [&](int kb, int ke) {
    if (lane < 3 * T::KC) {
      const int k = lane / 3, d = lane - 3 * k;
      if (kb + k < ke) {
        HPrim<R> c;
        load_hprim(P, ket.prim0 + kb + k, c);
        store_e<LK, -1>(len(d == 0 ? c.PA[0] : d == 1 ? c.PA[1] : c.PA[2]), area(c.o2), s + T::oE + k * T::NEK, d);
      }
    }
  };
  auto ket_coefs = [&](int n) {
    for (int x = lane; x < n * T::NCK; x += 32) {
      const int k = x / T::NCK, j = x - k * T::NCK;
      s[T::oCK + x] = coef_of(__ldg(tab + T::K0 + j), s + T::oE + k * T::NEK, one_of(R{}));
    }
  };
  // PQ and R^(m)_000 of one primitive quartet
  auto setup = [&](int ib, int ik, R* row) {
    HPrim<R> a, c;
    load_hprim(P, bra.prim0 + ib, a);
    load_hprim(P, ket.prim0 + ik, c);
    const R rs = hf_rsqrt(area(a.o2 + c.o2));
    R w = rs * rs;
    R PQ[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      PQ[x] = len(a.P[x] - c.P[x]);
      row[x] = PQ[x];
    }
    R B[L + 1];
    boys_y<L>(w * fmah(PQ[0], PQ[0], fmah(PQ[1], PQ[1], PQ[2] * PQ[2])), kc, B);
    if constexpr (SCALED) {
      kq = ((__float_as_int(w.hi) >> 23) - 127) >> 1;
      w = times_pow2(w, pow2f(-2 * kq));
#pragma unroll
      for (int x = 0; x < 3; ++x) row[x] = times_pow2(PQ[x], pow2f(kq));
    }
    R g = c.K * rs;
#pragma unroll
    for (int m = 0; m <= L; ++m) {
      row[3 + m] = g * B[m];
      if (m < L) g = g * w;
    }
  };
  // Hermite integrals of n quartets from their rows (row0 on), level by level,
  // the lanes over all their entries (one quartet alone fills a third of them)
  auto integrals = [&](int row0, int n) {
    const R* const rows = s + T::oRow + row0 * T::ROW;
    R* prev = L % 2 == 0 ? s + T::oR : s + T::oS;
    R* next = L % 2 == 0 ? s + T::oS : s + T::oR;
    if (lane < n) prev[lane * T::NR] = rows[lane * T::ROW + 3 + L];
    __syncwarp();
    sfor<L>([&](auto step) {
      constexpr int m = L - 1 - decltype(step)::value, N = nherm(L - m) - 1;
      for (int x = lane; x < n * N; x += 32) {
        const int j = x / N;
        const uint32_t d = __ldg(tab + T::R0 + x - j * N);
        const R* const pj = prev + j * T::NR;
        next[j * T::NR + (d & 255u)] = fmah(rows[j * T::ROW + ((d >> 24) & 3u)], pj[(d >> 8) & 255u],
                                            times_small(pj[(d >> 16) & 255u], (int)(d >> 26)));
      }
      if (lane < n) next[lane * T::NR] = rows[lane * T::ROW + 3 + m];
      __syncwarp();
      R* const t = prev;
      prev = next;
      next = t;
    });
    if constexpr (SCALED) {
      for (int x0 = 0; x0 < n * T::NR; x0 += 32) {
        const int x = x0 + lane, j = min(x / T::NR, n - 1), i = x - j * T::NR;
        const int k = __shfl_sync(0xffffffffu, kq, row0 + j);
        if (x < n * T::NR) {
          int N = 0;
#pragma unroll
          for (int l = 0; l < L; ++l) N += i >= nherm(l);
          s[T::oR + x] = times_pow2(s[T::oR + x], pow2f(k * N));
        }
      }
      __syncwarp();
    }
  };
  // H and the left-over X of n quartets, coefficients from ck on.  Both passes
  // go through one copy of the unrolled sums (they change places in between):
  // two copies of the df64 code overran the instruction cache (issue active
  // 13 % in (dd|dd), 25 % in (dd|dp), waiting for instructions).
  auto add_terms = [&](const R* ck, int n) {
#pragma unroll 1
    for (int ps = 0; ps < (T::TL > 0 ? 2 : 1); ++ps) {
#pragma unroll 1
      for (int j = ps ? sl : sm; j < n; j += ps ? 32 : T::PM)
        herm_terms_add<C, R>(s + T::oR + j * T::NR, ck + j * T::NCK, pm, H);
      if constexpr (T::TL > 0) {
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          const R t = H[f];
          H[f] = X[f];
          X[f] = t;
        }
#pragma unroll
        for (int k = 0; k < T::NUW; ++k) {
          const uint32_t t = pm[k];
          pm[k] = pl[k];
          pl[k] = t;
        }
      }
    }
  };
  auto clear = [&]() {
#pragma unroll
    for (int f = 0; f < NF; ++f) H[f] = X[f] = zero;
  };
  // applies the bra primitive's expansion to the lanes' sums (n: left-over
  // slots in use) and adds them to s[oA ..]
  auto flush = [&](int ib, int n) {
    HPrim<R> a;
    load_hprim(P, bra.prim0 + ib, a);
    __syncwarp();
    if (lane < 3) store_e<LB, 1>(len(lane == 0 ? a.PA[0] : lane == 1 ? a.PA[1] : a.PA[2]), area(a.o2), s + T::oE, lane);
    R* const Hs = s + T::oR;  // the integrals are done with
    if (sm == 0)
#pragma unroll
      for (int f = 0; f < NF; ++f) Hs[tm * NF + f] = H[f];
    if (T::TL > 0 && sl < n)
#pragma unroll
      for (int f = 0; f < NF; ++f) s[T::oX + (sl * T::TL + tl - T::TM) * NF + f] = X[f];
    __syncwarp();
    for (int k = lane; k < T::NCB; k += 32) s[T::oCB + k] = coef_of(__ldg(tab + T::B0 + k), s + T::oE, a.K);
#pragma unroll
    for (int p = 1; p < T::PM; ++p) {
      if (sm == p)
#pragma unroll
        for (int f = 0; f < NF; ++f) Hs[tm * NF + f] = Hs[tm * NF + f] + H[f];
      __syncwarp();
    }
    for (int o = lane; o < T::TL * NF; o += 32) {
      R v = s[T::oX + o];
      for (int j = 1; j < n; ++j) v = v + s[T::oX + j * T::TL * NF + o];
      Hs[T::TM * NF + o] = v;
    }
    __syncwarp();
    for (int o = lane; o < T::NA; o += 32) {
      const uint32_t w = __ldg(tab + T::A0 + o);
      const int f = (w >> 12) & 63u;
      const R* c = s + T::oCB + ((w >> 4) & 255u);
      const uint32_t* u = tab + T::AU0 + ((w >> 4) & 255u);
      R v = s[T::oA + o];
      for (int j = w & 15u; j > 0; --j) v = fmah(*c++, Hs[__ldg(u++) * NF + f], v);
      s[T::oA + o] = v;
    }
    __syncwarp();
  };
  if constexpr (T::BRA_OUTER) {
    for (int ib = ib_lo; ib < ib_hi; ++ib) {
      const int ka = max(0, q_lo - ib * nk), kz = min(nk, q_hi - ib * nk);  // not empty
      clear();
      for (int kr = ka; kr < kz; kr += T::ROWS) {
        const int kt = min(kr + T::ROWS, kz);
        if (kr + lane < kt) setup(ib, kr + lane, s + T::oRow + lane * T::ROW);
        __syncwarp();
        const int ng = (kt - kr + T::KC - 1) / T::KC;
        for (int g = 0; g < ng; ++g) {
          const int kb = kr + g * (kt - kr) / ng, ke = kr + (g + 1) * (kt - kr) / ng;
          ket_rows(kb, ke);
          integrals(kb - kr, ke - kb);
          ket_coefs(ke - kb);  // over the second integral buffer
          __syncwarp();
          add_terms(s + T::oCK, ke - kb);
          __syncwarp();
        }
      }
      flush(ib, min(T::KC, kz - ka));
    }
  } else {
    constexpr int NB = T::ROWS / T::KC;
    const int ngrp = (nk + T::KC - 1) / T::KC;
    for (int gk = 0; gk < ngrp; ++gk) {
      const int kb = gk * nk / ngrp, ke = (gk + 1) * nk / ngrp;
      ket_rows(kb, ke);
      __syncwarp();
      ket_coefs(ke - kb);
      __syncwarp();
      for (int ib0 = ib_lo; ib0 < ib_hi; ib0 += NB) {
        const int ibx = ib0 + lane / T::KC, ikx = kb + lane % T::KC;
        if (ibx < ib_hi && ikx < ke) setup(ibx, ikx, s + T::oRow + lane * T::ROW);
        __syncwarp();
        for (int ib = ib0; ib < min(ib0 + NB, ib_hi); ++ib) {
          // this part's ket primitives of the group
          const int k0 = max(kb, q_lo - ib * nk), k1 = min(ke, q_hi - ib * nk), n = k1 - k0;
          if (n <= 0) continue;  // warp-uniform
          clear();
          integrals((ib - ib0) * T::KC + k0 - kb, n);
          add_terms(s + T::oCK + (k0 - kb) * T::NCK, n);
          flush(ib, n);
        }
      }
    }
  }
  if constexpr (SCALED)  // [e0|f0] have the dimension length^(e + f - 1)
    for (int o = lane; o < T::NA; o += 32) {
      const int e = set0(C::LA) + o / NF, f = set0(C::LC) + o % NF;
      int l = 0;
#pragma unroll
      for (int i = 0; i < LB; ++i) l += e >= nherm(i);
#pragma unroll
      for (int i = 0; i < LK; ++i) l += f >= nherm(i);
      s[T::oA + o] = times_pow2(s[T::oA + o], pow2f(ua * (1 - l)));
    }
}

}  // namespace hfk
