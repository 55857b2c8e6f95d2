// rys_grad.cu -- the two-electron part of the analytic RHF gradient by Rys
// quadrature, every class (the recurrences and the tables are those of
// rys.cu, one power higher on A, B and C).
//
// A primitive's derivative with respect to its centre is d/dA_x [x_A^a
// e^(-alpha x_A^2)] = 2 alpha x_A^(a+1) e - a x_A^(a-1) e, so per direction
// the one-dimensional factor of (ab|cd) with respect to A becomes
// 2 alpha I(a+1, b, c, d) - a I(a-1, b, c, d) (likewise b, beta for B and c,
// gamma for C); D follows by translational invariance, dD = -(dA + dB + dC).
// The quartet's derivative integrals are contracted on the fly with
//     Gamma = 8 w [2 D_ab D_cd - (D_ac D_bd + D_ad D_bc) / 2]
// (w the symmetry weight of the unique quartet), the two-electron part of
// dE/dR = sum over unique quartets of Gamma d(ab|cd)/dR with the energy
// E_2e = 2 Tr[D J] - Tr[D K].
//
// FP64 instructions bound it (one holds a sub-partition's pipe for 64 cycles
// whatever the number of live lanes), so the kernel is laid out for full
// lanes and few of them:
//  * A task is one (primitive quartet, root), and a group of g lanes (a power
//    of two, chosen per class) takes it, 32 / g tasks side by side in the
//    warp: one lane per task for (ss|ss), the whole warp for the d, f and g
//    blocks.  A warp on one task, as it was before, left most lanes idle in
//    the classes of s and p shells.
//  * The derivative of direction x needs, for each one-dimensional index
//    i = (a_x, b_x, c_x, d_x), only W_x(i) = sum over the outputs of that i
//    of Gamma Iy Iz: a product and a multiply-add per output and direction,
//    then dI(i) W(i) for A, B and C once per i.  The outputs come sorted by i
//    (host-built streams, cut into segments of even length for the lanes).
//    Forming nine products per output took 40 instructions where this takes
//    6 and a share of the 9 per segment.
// Whole gradient on GB300, with the classes on side streams: of a 5-atom s+p+d
// molecule (49 functions) 201 -> 34.6 ms, of QZ-shaped water (140 functions, s
// to g) 321 -> 35.0 ms.
#include <algorithm>
#include <array>
#include <cstring>
#include <map>
#include <vector>

#include "eri.cuh"
#include "hf_internal.h"
#include "per_device.h"
#include "rys_class.cuh"

namespace hfr {

// One class with g lanes per task: sizes, and the device table's offsets (in
// words).  Table: transfer entries of H and I, then per (chunk, direction)
// the stream of segments.
struct GradClass {
  RysClass base;        // the J/K class: chunks and work-list shape
  int n;                // roots
  int NG, MG;           // highest G powers: la + lb + 1, lc + ld + 1
  int SG, SH, SI;       // per-direction table sizes
  int oH, oI, ws;       // offsets in a task's tables (doubles), their size
  int g, lg;            // lanes per task, log2
  int nH, nI;           // transfer entries, multiples of g
  int tH, tI, tS;       // word offsets: entries, and the chunk x direction index of stream starts
};

inline GradClass grad_class(const RysClass& rc, int g) {
  GradClass c{};
  c.base = rc;
  c.n = (rc.la + rc.lb + rc.lc + rc.ld + 1) / 2 + 1;
  c.NG = rc.nmax + 1;
  c.MG = rc.mmax + 1;
  c.SG = (c.NG + 1) * (c.MG + 1);
  c.SH = (rc.la + 2) * (rc.lb + 2) * (c.MG + 1);
  c.SI = (rc.la + 2) * (rc.lb + 2) * (rc.lc + 2) * (rc.ld + 1);
  c.oH = 3 * c.SG;
  c.oI = rc.ld == 0 ? c.oH : c.oH + 3 * c.SH;  // ld = 0: I is H (ic = m)
  c.ws = (rc.ld == 0 ? c.oH + 3 * c.SH : c.oI + 3 * c.SI) | 1;  // odd: the tasks' tables start in different banks
  c.g = g;
  c.lg = 0;
  while ((1 << c.lg) < g) ++c.lg;
  return c;
}

// Entry of a transfer: dst (12 bits) | src (11) | power moved (3) | direction (2)
inline uint32_t move_entry(int dst, int src, int pw, int dir) {
  return (uint32_t)dst | (uint32_t)src << 12 | (uint32_t)pw << 23 | (uint32_t)dir << 26;
}

// Host table of a class with g lanes per task.
inline std::vector<uint32_t> grad_table(GradClass* gc) {
  const RysClass& rc = gc->base;
  const int g = gc->g, M1 = gc->MG + 1;
  std::vector<uint32_t> t;
  auto flush = [&](std::vector<uint32_t>& e) {  // by power (even rounds), padded with copies
    std::stable_sort(e.begin(), e.end(), [](uint32_t a, uint32_t b) { return ((a >> 23) & 7) < ((b >> 23) & 7); });
    while (e.size() % g) e.push_back(e.back());
    t.insert(t.end(), e.begin(), e.end());
    return (int)e.size();
  };
  {  // H(ia, ib, m) from G(ia .. ia + ib, m)
    std::vector<uint32_t> e;
    for (int dir = 0; dir < 3; ++dir)
      for (int ia = 0; ia <= rc.la + 1; ++ia)
        for (int ib = 0; ib <= rc.lb + 1 && ia + ib <= gc->NG; ++ib)
          for (int m = 0; m < M1; ++m)
            e.push_back(move_entry(dir * gc->SH + (ia * (rc.lb + 2) + ib) * M1 + m, dir * gc->SG + ia * M1 + m, ib, dir));
    gc->tH = 0;
    gc->nH = flush(e);
  }
  gc->tI = (int)t.size();
  gc->nI = 0;
  if (rc.ld > 0) {  // I(ia, ib, ic, id) from H(ia, ib, ic .. ic + id); at most one of the powers is raised
    std::vector<uint32_t> e;
    for (int dir = 0; dir < 3; ++dir)
      for (int ia = 0; ia <= rc.la + 1; ++ia)
        for (int ib = 0; ib <= rc.lb + 1; ++ib)
          for (int ic = 0; ic <= rc.lc + 1; ++ic) {
            if ((ia > rc.la) + (ib > rc.lb) + (ic > rc.lc) > 1) continue;
            for (int id = 0; id <= rc.ld; ++id) {
              const int ab = ia * (rc.lb + 2) + ib;
              e.push_back(move_entry(dir * gc->SI + (ab * (rc.lc + 2) + ic) * (rc.ld + 1) + id,
                                     dir * gc->SH + ab * M1 + ic, id, dir));
            }
          }
    gc->nI = flush(e);
  }
  // Streams: per chunk and direction rounds of one segment per lane; a
  // segment is up to `smax` outputs of one index i, padded to the round's
  // longest with the zero output.
  gc->tS = (int)t.size();
  t.resize(t.size() + 3 * rc.nchunks);
  const int lb2 = rc.lb + 2, lc2 = rc.lc + 2, ld1 = rc.ld + 1;
  auto comps = [](int l) {
    std::vector<std::array<int, 3>> v;
    for (int x = l; x >= 0; --x)
      for (int y = l - x; y >= 0; --y) v.push_back({x, y, l - x - y});
    return v;
  };
  const auto ca = comps(rc.la), cb = comps(rc.lb), cc = comps(rc.lc), cd = comps(rc.ld);
  for (int ch = 0; ch < rc.nchunks; ++ch) {
    const int r0 = ch * rc.rpc, r1 = std::min(r0 + rc.rpc, rc.na * rc.nb), ncd = rc.nc * rc.nd;
    const uint32_t none = (uint32_t)((r1 - r0) * ncd);  // Gamma = 0 there
    for (int dir = 0; dir < 3; ++dir) {
      struct Seg {
        uint32_t head;
        std::vector<uint32_t> e;
      };
      std::map<uint32_t, std::vector<uint32_t>> by;  // head -> outputs
      for (int row = r0; row < r1; ++row)
        for (int c = 0; c < rc.nc; ++c)
          for (int d = 0; d < rc.nd; ++d) {
            const auto &pa = ca[row / rc.nb], &pb = cb[row % rc.nb], &pc = cc[c], &pd = cd[d];
            auto off = [&](int x) { return ((pa[x] * lb2 + pb[x]) * lc2 + pc[x]) * ld1 + pd[x]; };
            const uint32_t out = (uint32_t)((row - r0) * ncd + c * rc.nd + d);
            by[(uint32_t)off(dir) | pa[dir] << 12 | pb[dir] << 15 | pc[dir] << 18].push_back(
                out | (uint32_t)off((dir + 1) % 3) << 10 | (uint32_t)off((dir + 2) % 3) << 21);
          }
      // the segment length with the fewest instructions: 2 per entry, 10 per round
      auto cut = [&](int smax) {
        std::vector<Seg> s;
        for (auto& kv : by) {
          const int n = (int)kv.second.size(), k = (n + smax - 1) / smax;
          for (int j = 0; j < k; ++j)
            s.push_back(Seg{kv.first, std::vector<uint32_t>(kv.second.begin() + j * n / k, kv.second.begin() + (j + 1) * n / k)});
        }
        std::stable_sort(s.begin(), s.end(), [](const Seg& a, const Seg& b) { return a.e.size() > b.e.size(); });
        return s;
      };
      int best = 1;
      long long cost = -1;
      for (int smax = 1; smax <= 96; smax += smax < 8 ? 1 : 4) {
        const std::vector<Seg> s = cut(smax);
        long long c = 0;
        for (size_t k = 0; k < s.size(); k += g) c += 2 * (long long)s[k].e.size() + 10;
        if (cost < 0 || c < cost) {
          cost = c;
          best = smax;
        }
      }
      const std::vector<Seg> s = cut(best);
      t[gc->tS + 3 * ch + dir] = (uint32_t)t.size();
      t.push_back((uint32_t)((s.size() + g - 1) / g));
      for (size_t k = 0; k < s.size(); k += g) {
        const size_t len = s[k].e.size();
        t.push_back((uint32_t)len);
        for (int lane = 0; lane < g; ++lane) t.push_back(k + lane < s.size() ? s[k + lane].head : s[k].head);
        for (size_t j = 0; j < len; ++j)
          for (int lane = 0; lane < g; ++lane)
            t.push_back(k + lane < s.size() && j < s[k + lane].e.size() ? s[k + lane].e[j] : none);
      }
    }
  }
  return t;
}

// sum_k C(n, k) X^(n - k) f[k stride]
__device__ __forceinline__ double move_power(const double* f, int stride, int n, double X) {
  double v = f[0];
  for (int k = 1; k < n; ++k) v = fma(v, X, kBin.b[n][k] * f[k * stride]);
  return n > 0 ? fma(v, X, f[n * stride]) : v;
}

__global__ void __launch_bounds__(128) rys_grad_kernel(const JKWork w, const PairSet ps, const KernelCommon kc,
                                                       const double* __restrict__ D,
                                                       const int* __restrict__ bf_atom, int nbf,
                                                       double* __restrict__ grad, const GradClass gc,
                                                       const uint32_t* __restrict__ tab) {
  extern __shared__ __align__(16) double rsm[];
  const RysClass& rc = gc.base;
  const int lane = threadIdx.x & 31;
  const int sub = lane & (gc.g - 1), grp = lane >> gc.lg, ngrp = 32 >> gc.lg;
  const int NB = rc.nb, NC = rc.nc, ND = rc.nd, NCD = NC * ND;
  // the warp's slice: AB and CD, Gamma of the chunk's outputs and a zero, the groups' tables
  const int ngam = rc.rpc * NCD + 1;
  double* const hd = rsm + (size_t)(threadIdx.x >> 5) * (6 + ngam + ngrp * gc.ws);
  double* const gam = hd + 6;
  double* const tb = gam + ngam + grp * gc.ws;
  const int M1 = gc.MG + 1, L1 = gc.NG + 1;
  const int sC = rc.ld + 1, sB = (rc.lc + 2) * sC, sA = (rc.lb + 2) * sB;
  const bool wide = 3 * L1 <= gc.g;  // one lane per (direction, n) in the G recursion
  const bool gl = sub < 3 * L1;
  const int gdir = wide && gl ? sub / L1 : 0, gn = wide && gl ? sub - gdir * L1 : 0;
  for (;;) {
    int t = 0;
    if (lane == 0) t = atomicAdd(w.counter, 1);
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t >= w.nitems) break;
    ItemRange it;
    rys_item(w, t, &it);
    const int bp = __ldg(w.bra + it.bi);
    if (!HF_BCHECK(kc, bp >= 0 && bp < ps.npairs, HF_BC_PAIR, bp)) continue;
    const PairInfo bra = ps.info[bp];
    for (int kidx = it.k0; kidx < it.k1; ++kidx) {
      const int kp = __ldg(w.ket + kidx);
      if (!HF_BCHECK(kc, kp >= 0 && kp < ps.npairs, HF_BC_PAIR, kp)) continue;
      const PairInfo ket = ps.info[kp];
      int q_lo, q_hi, c_lo, c_hi;
      rys_part(rc, w, bra, ket, it.part, it.nsp, &q_lo, &q_hi, &c_lo, &c_hi);
      if (q_hi <= q_lo) continue;
      __syncwarp();
      if (lane < 3) {
        hd[lane] = lane == 0 ? bra.AB[0] : lane == 1 ? bra.AB[1] : bra.AB[2];
        hd[3 + lane] = lane == 0 ? ket.AB[0] : lane == 1 ? ket.AB[1] : ket.AB[2];
      }
      double wdeg = 8.0;
      if (bra.same) wdeg *= 0.5;
      if (ket.same) wdeg *= 0.5;
      if (bp == kp) wdeg *= 0.5;
      const int a0 = bra.bfA, b0 = bra.bfB, c0 = ket.bfA, d0 = ket.bfB, nk = ket.nprim;
      const int ntask = (q_hi - q_lo) * gc.n;
      double g[9];  // dE/dA, dE/dB, dE/dC (x, y, z each)
#pragma unroll
      for (int k = 0; k < 9; ++k) g[k] = 0.0;
      for (int ch = c_lo; ch < c_hi; ++ch) {
        const int r0 = ch * rc.rpc, r1 = min(r0 + rc.rpc, rc.na * NB), nout = (r1 - r0) * NCD;
        __syncwarp();
        for (int e = lane; e <= nout; e += 32) {
          double v = 0.0;
          if (e < nout) {
            const int rl = e / NCD, cd = e - rl * NCD;
            const int row = r0 + rl, a = row / NB, b = row - a * NB;
            const int c = cd / ND, d = cd - c * ND;
            auto Dv = [&](int i, int j) { return __ldg(D + (size_t)i * nbf + j); };
            const int ia = a0 + a, ib = b0 + b, ic = c0 + c, id = d0 + d;
            v = wdeg * kBin.sc[rc.la][a] * kBin.sc[rc.lb][b] * kBin.sc[rc.lc][c] * kBin.sc[rc.ld][d] *
                (2.0 * Dv(ia, ib) * Dv(ic, id) - 0.5 * (Dv(ia, ic) * Dv(ib, id) + Dv(ia, id) * Dv(ib, ic)));
          }
          gam[e] = v;
        }
        __syncwarp();
        for (int t0 = 0; t0 < ntask; t0 += ngrp) {
          const bool live = t0 + grp < ntask;  // the last round's spare groups repeat a task with weight 0
          const int task = live ? t0 + grp : ntask - 1;
          const int qq = q_lo + task / gc.n, root = task - (qq - q_lo) * gc.n;
          const int ibp = qq / nk, ikp = qq - ibp * nk;
          const double* rb = ps.prim64 + (size_t)(bra.prim0 + ibp) * PRIM64_STRIDE;
          const double* rk = ps.prim64 + (size_t)(ket.prim0 + ikp) * PRIM64_STRIDE;
          const double p = __ldg(rb + 8), q = __ldg(rk + 8), s = p + q;
          const double PQ[3] = {__ldg(rb + 1) - __ldg(rk + 1), __ldg(rb + 2) - __ldg(rk + 2),
                                __ldg(rb + 3) - __ldg(rk + 3)};
          const double rs = hfk::hf_rsqrt(s);
          double ipq = rs * rs;
          ipq = fma(ipq, fma(-s, ipq, 1.0), ipq);
          const double qf = q * ipq, pf = p * ipq;
          double u, wt;
          rys_rule_root(kc.rys, gc.n, root, p * qf * fma(PQ[0], PQ[0], fma(PQ[1], PQ[1], PQ[2] * PQ[2])), &u, &wt);
          const double g0z = live ? wt * (__ldg(rb + 9) * __ldg(rk + 9) * rs) : 0.0;
          const double B00 = 0.5 * u * ipq, B10 = __ldg(rb) * (1.0 - u * qf), B01 = __ldg(rk) * (1.0 - u * pf);
          const double uq = u * qf, up = u * pf;
          if (wide) {  // G(gn, 0 .. MG) of direction gdir on this lane, G(gn - 1, m) from the lane below
            const double PQg = gdir == 0 ? PQ[0] : (gdir == 1 ? PQ[1] : PQ[2]);
            const double c00 = __ldg(rb + 4 + gdir) - uq * PQg, d00 = __ldg(rk + 4 + gdir) + up * PQg;
            double gg = gdir == 2 ? g0z : 1.0, gp = 0.0;
            for (int k = 0; k < gn; ++k) {
              const double tt = fma(c00, gg, kBin.k[k] * B10 * gp);
              gp = gg;
              gg = tt;
            }
            double* const Gd = tb + gdir * gc.SG + gn * M1;
            if (gl) Gd[0] = gg;
            const double nB00 = kBin.k[gn] * B00;
            double gm = 0.0;
            for (int m = 0; m < gc.MG; ++m) {
              const double left = __shfl_up_sync(0xffffffffu, gg, 1);
              const double tt = fma(d00, gg, fma(kBin.k[m] * B01, gm, gn > 0 ? nB00 * left : 0.0));
              gm = gg;
              gg = tt;
              if (gl) Gd[m + 1] = gg;
            }
          } else {  // one lane per direction, or one lane for all
            for (int dir = sub; dir < 3; dir += gc.g) {
              const double PQg = dir == 0 ? PQ[0] : (dir == 1 ? PQ[1] : PQ[2]);
              const double c00 = __ldg(rb + 4 + dir) - uq * PQg, d00 = __ldg(rk + 4 + dir) + up * PQg;
              double* const Gd = tb + dir * gc.SG;
              double gg = dir == 2 ? g0z : 1.0, gp = 0.0;
              Gd[0] = gg;
              for (int k = 0; k < gc.NG; ++k) {
                const double tt = fma(c00, gg, kBin.k[k] * B10 * gp);
                gp = gg;
                gg = tt;
                Gd[(k + 1) * M1] = gg;
              }
              for (int m = 0; m < gc.MG; ++m) {
                const double mB = kBin.k[m] * B01;
                double left = 0.0;  // G(n - 1, m)
                for (int n = 0; n <= gc.NG; ++n) {
                  double* const Gn = Gd + n * M1 + m;
                  const double here = Gn[0];
                  double v = d00 * here;
                  if (m > 0) v = fma(mB, Gn[-1], v);
                  if (n > 0) v = fma(kBin.k[n] * B00, left, v);
                  Gn[1] = v;
                  left = here;
                }
              }
            }
          }
          __syncwarp();
          for (int e = sub; e < gc.nH; e += gc.g) {  // H(ia, ib, m), ia <= la + 1, ib <= lb + 1
            const uint32_t d = __ldg(tab + gc.tH + e);
            tb[gc.oH + (d & 4095u)] = move_power(tb + ((d >> 12) & 2047u), M1, (d >> 23) & 7u, hd[d >> 26]);
          }
          __syncwarp();
          if (rc.ld > 0) {  // I(ia, ib, ic, id), ic <= lc + 1, id <= ld
            for (int e = sub; e < gc.nI; e += gc.g) {
              const uint32_t d = __ldg(tab + gc.tI + e);
              tb[gc.oI + (d & 4095u)] = move_power(tb + gc.oH + ((d >> 12) & 2047u), 1, (d >> 23) & 7u, hd[3 + (d >> 26)]);
            }
            __syncwarp();
          }
          const double za2 = 2.0 * __ldg(rb + 10), zb2 = 2.0 * (p - __ldg(rb + 10)), zc2 = 2.0 * __ldg(rk + 10);
#pragma unroll
          for (int dir = 0; dir < 3; ++dir) {
            const double* const X = tb + gc.oI + dir * gc.SI;
            const double* const Y = tb + gc.oI + ((dir + 1) % 3) * gc.SI;
            const double* const Z = tb + gc.oI + ((dir + 2) % 3) * gc.SI;
            const uint32_t* st = tab + __ldg(tab + gc.tS + 3 * ch + dir);
            int nr = (int)__ldg(st++);
            for (; nr > 0; --nr) {
              const int len = (int)__ldg(st);
              const uint32_t head = __ldg(st + 1 + sub);
              st += 1 + gc.g;
              double W = 0.0;
              for (int k = 0; k < len; ++k, st += gc.g) {
                const uint32_t e = __ldg(st + sub);
                W = fma(gam[e & 1023u], Y[(e >> 10) & 2047u] * Z[e >> 21], W);
              }
              const double* const x = X + (head & 4095u);
              const int na = (head >> 12) & 7u, nb = (head >> 15) & 7u, nc = (head >> 18) & 7u;
              // a spare lane of the round repeats the first segment's head with W = 0
              g[dir] = fma(fma(za2, x[sA], -kBin.k[na] * x[na > 0 ? -sA : 0]), W, g[dir]);
              g[3 + dir] = fma(fma(zb2, x[sB], -kBin.k[nb] * x[nb > 0 ? -sB : 0]), W, g[3 + dir]);
              g[6 + dir] = fma(fma(zc2, x[sC], -kBin.k[nc] * x[nc > 0 ? -sC : 0]), W, g[6 + dir]);
            }
          }
          __syncwarp();
        }
      }
#pragma unroll
      for (int k = 0; k < 9; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) g[k] += __shfl_xor_sync(0xffffffffu, g[k], o);
      if (lane < 3) {
        const double gA = lane == 0 ? g[0] : lane == 1 ? g[1] : g[2], gB = lane == 0 ? g[3] : lane == 1 ? g[4] : g[5],
                     gC = lane == 0 ? g[6] : lane == 1 ? g[7] : g[8];
        atomicAdd(grad + 3 * __ldg(bf_atom + a0) + lane, gA);
        atomicAdd(grad + 3 * __ldg(bf_atom + b0) + lane, gB);
        atomicAdd(grad + 3 * __ldg(bf_atom + c0) + lane, gC);
        atomicAdd(grad + 3 * __ldg(bf_atom + d0) + lane, -(gA + gB + gC));
      }
    }
  }
}

}  // namespace hfr

// A class's table on the device, built on first use and kept for the context.
struct HfGradTab {
  hfr::GradClass gc;
  DevArray<uint32_t> tab;
};
struct HfGradTabs {
  std::map<int, HfGradTab> m;  // class * 8 + log2(lanes per task)
};
void hf_grad_tabs_free(HfGradTabs* t) { delete t; }

// Derivative ERIs of class cls over its Rys work list w, contracted into grad
// (natom x 3, accumulated).  avg_pq: primitive quartets per work item on
// average.  Lanes per task: as few as let the warp's tables fit 14 KB, but no
// more tasks side by side than an average item has.
int hf_grad_launch(hf_ctx* ctx, int cls, const JKWork& w, const PairSet& ps, const KernelCommon& kc, const double* D,
                   const int* bf_atom, int nbf, double* grad, double avg_pq, cudaStream_t st) {
  using namespace hfr;
  const RysClass rc = rys_class_of(cls);
  int g = 32;
  while (g > 1) {
    const GradClass c = grad_class(rc, g / 2);
    if (64 / g * (long long)c.ws > 1792 || 64 / g > std::max(1.0, avg_pq * c.n)) break;
    g /= 2;
  }
  if (!ctx->grad_tabs) ctx->grad_tabs = new HfGradTabs();
  GradClass probe = grad_class(rc, g);
  HfGradTab& e = ctx->grad_tabs->m[cls * 8 + probe.lg];
  if (e.tab.n == 0) {
    const std::vector<uint32_t> t = grad_table(&probe);
    e.gc = probe;
    HF_CHECK(e.tab.alloc(ctx, t.size()));
    // allocated and filled on the context's stream; st may be a side stream
    cudaError_t err = cudaMemcpyAsync(e.tab.ptr, t.data(), t.size() * sizeof(uint32_t), cudaMemcpyHostToDevice, ctx->stream);
    if (err == cudaSuccess) err = cudaStreamSynchronize(ctx->stream);
    if (err != cudaSuccess) {
      e.tab.release();
      return hf_fail(HF_ERR_CUDA, "gradient table upload: %s", cudaGetErrorString(err));
    }
  }
  static PerDevice limit;
  if (hf_smem_limit(limit, rys_grad_kernel, 227 * 1024) < 0)
    return hf_fail(HF_ERR_CUDA, "gradient kernel's shared memory: %s", cudaGetErrorString(cudaGetLastError()));
  const size_t per_warp = (6 + (size_t)rc.rpc * rc.nc * rc.nd + 1 + (size_t)(32 / g) * e.gc.ws) * sizeof(double);
  int warps = 4;
  while (warps > 1 && warps * per_warp > 200 * 1024) warps /= 2;
  const int resident = std::max(1, std::min(4, (int)(220 * 1024 / (warps * per_warp))));
  const int grid = std::max(1, std::min(resident * ctx->num_sms, (w.nitems + warps - 1) / warps));
  rys_grad_kernel<<<grid, 32 * warps, warps * per_warp, st>>>(w, ps, kc, D, bf_atom, nbf, grad, e.gc, e.tab.ptr);
  return HF_OK;
}
