// rys_class.cuh -- what the Rys kernels of rys.cu and rys_grad.cu share: the
// shape of a class (roots, components, output chunks) and the reading of a work
// item.
#pragma once
#include <algorithm>

#include "eri.cuh"
#include "hf_device.h"
#include "rys.cuh"

namespace hfr {

// Binomials, small integers and the component scales s(l, c) = sqrt((2l-1)!! /
// ((2x-1)!! (2y-1)!! (2z-1)!!)) of the axial-normalised basis.
struct BinTable {
  double b[6][6];  // C(n, k)
  double k[16];    // k as a double
  double sc[5][15];
};
constexpr BinTable make_bin() {
  BinTable t{};
  for (int n = 0; n < 6; ++n)
    for (int k = 0; k <= n; ++k) t.b[n][k] = hfk::binom_c(n, k);
  for (int k = 0; k < 16; ++k) t.k[k] = k;
  for (int l = 0; l < 5; ++l)
    for (int c = 0; c < (l + 1) * (l + 2) / 2; ++c) t.sc[l][c] = hfk::comp_scale(l, c);
  return t;
}
static __constant__ BinTable kBin = make_bin();

// Fixed part of a warp's shared slice of the J/K kernels (doubles).
constexpr int kHead = 234;

// Outputs of one chunk: at most 32 per lane.
constexpr int kMaxChunk = 1024;

// Work of one class.  The output block (ab|cd) is split into chunks of
// whole rows (a, b) (all c, d), at most kMaxChunk outputs each; a chunk is
// evaluated over the quartet's primitive quartets with its outputs in
// registers (KM per lane).  For the f/g classes every chunk of every
// quartet is its own work item ("native": part = chunk); when HF_JK_RYS
// sends the s/p/d classes here, their lists are split along the primitive
// loop instead and an item walks all chunks.
struct RysClass {
  int la, lb, lc, ld;
  int n;                    // roots
  int na, nb, nc, nd;       // Cartesian components
  int nmax, mmax;           // la + lb, lc + ld
  int SG, SH, SI;           // per-direction sizes of G, bra-transferred H, I
  int oG, oH, oI, oBlk;     // offsets in the warp slice (doubles); the block reuses the tables
  int rpc, nchunks;         // rows (a, b) per chunk, chunks per quartet
  int km;                   // outputs per lane (template of the kernel)
  int native;               // work-item parts are chunks
  int ws;                   // doubles per warp
};

inline RysClass rys_class(int la, int lb, int lc, int ld) {
  RysClass r{};
  r.la = la; r.lb = lb; r.lc = lc; r.ld = ld;
  r.n = (la + lb + lc + ld) / 2 + 1;
  auto nc_ = [](int l) { return (l + 1) * (l + 2) / 2; };
  r.na = nc_(la); r.nb = nc_(lb); r.nc = nc_(lc); r.nd = nc_(ld);
  r.nmax = la + lb;
  r.mmax = lc + ld;
  r.SG = (r.nmax + 1) * (r.mmax + 1);
  r.SH = (la + 1) * (lb + 1) * (r.mmax + 1);
  r.SI = (la + 1) * (lb + 1) * (lc + 1) * (ld + 1);
  r.oG = kHead;
  int end = r.oG + 3 * r.SG;
  r.oH = lb == 0 ? r.oG : end;  // lb = 0: H is G
  if (lb > 0) end = r.oH + 3 * r.SH;
  r.oI = ld == 0 ? r.oH : end;  // ld = 0: I is H
  if (ld > 0) end = r.oI + 3 * r.SI;
  const int ncd = r.nc * r.nd, rows = r.na * r.nb;
  // as few chunks as fit, of even size: cutting off kMaxChunk at a time left
  // (fd|dp), 60 rows of 18, a second chunk of 4 rows with tables of its own
  const int most = std::max(1, std::min(rows, kMaxChunk / ncd));
  const int least = (rows + most - 1) / most;
  r.rpc = (rows + least - 1) / least;
  r.nchunks = (rows + r.rpc - 1) / r.rpc;
  const int per_lane = (r.rpc * ncd + 31) / 32;
  r.km = per_lane <= 4 ? 4 : per_lane <= 8 ? 8 : (per_lane + 3) / 4 * 4;
  r.native = std::max(std::max(la, lb), std::max(lc, ld)) > 2;
  r.oBlk = kHead;
  r.ws = (std::max(end, r.oBlk + r.rpc * ncd) + 1) & ~1;
  return r;
}

// class index -> (la, lb, lc, ld)
inline RysClass rys_class_of(int cls) {
  int X = 0;
  while ((X + 1) * (X + 2) / 2 <= cls) ++X;
  const int Y = cls - X * (X + 1) / 2;
  int la, lb, lc, ld;
  pair_ls(X, &la, &lb);
  pair_ls(Y, &lc, &ld);
  return rys_class(la, lb, lc, ld);
}

// Work item t -> entry bi, the kets of the item and its part.  Items hold
// w.chunk kets (1 for the Rys classes and the warp-cooperative lists, 32
// for the thread-per-quartet lists).
struct ItemRange {
  int bi, k0, k1, part, nsp;
};
__device__ __forceinline__ void rys_item(const JKWork& w, int t, ItemRange* it) {
  int lo = 0, hi = w.nbra;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (__ldg(w.ioff + mid) <= t) lo = mid; else hi = mid;
  }
  it->bi = lo;
  it->nsp = w.nsplit ? __ldg(w.nsplit + lo) : 1;
  const int rr = t - __ldg(w.ioff + lo);
  const int blk = rr / it->nsp;
  it->part = rr - blk * it->nsp;
  it->k0 = __ldg(w.kbeg + lo) + blk * w.chunk;
  it->k1 = min(it->k0 + w.chunk, __ldg(w.kend + lo));
}
// Primitive quartets and chunks of one item's part.  Rys lists (nchunk >
// 0): part = range * nchunk + chunk, the range one of nsp / nchunk equal
// slices of the primitive quartets.  Lists built for the Obara-Saika
// kernels (HF_JK_RYS with lists of another shape): every chunk, over a range
// of primitive quartets (chunk 1) or of bra primitive pairs (chunk 32).
__device__ __forceinline__ void rys_part(const RysClass& rc, const JKWork& w, const PairInfo& bra,
                                         const PairInfo& ket, int part, int nsp, int* q_lo, int* q_hi, int* c_lo,
                                         int* c_hi) {
  const int nq = bra.nprim * ket.nprim;
  if (w.nchunk > 0) {
    const int nr = max(1, nsp / w.nchunk), ch = part % w.nchunk, pr = part / w.nchunk;
    *q_lo = pr * nq / nr;
    *q_hi = (pr + 1) * nq / nr;
    *c_lo = ch;
    *c_hi = ch + 1;
  } else {
    *c_lo = 0;
    *c_hi = rc.nchunks;
    if (w.chunk == 1) {
      *q_lo = part * nq / nsp;
      *q_hi = (part + 1) * nq / nsp;
    } else {
      *q_lo = (part * bra.nprim / nsp) * ket.nprim;
      *q_hi = ((part + 1) * bra.nprim / nsp) * ket.nprim;
    }
  }
}

}  // namespace hfr
