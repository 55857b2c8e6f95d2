// tensor.cu -- the dense integral tensor (ij|kl) of small bases.
//
// The class kernels write each unique quartet's block once, at (i j | k l) in
// the order of its shell pairs; mirror_tensor then copies it to the other
// index permutations.  Every element is the same to the last bit on every call:
// a quartet that several work items share (ket units, parts of the bra's
// primitive loop) has a slot for each, and sum_slots adds the slots up in
// order.  Added into the tensor atomically they gave sums in the order the GPU
// happened to run them.
//
// The lists are the tensor's own.  Thread-per-quartet classes take ket units as
// the J/K build does, in the order of the pair list inside a bucket (all
// quartets are kept, so nothing is sorted by Schwarz factor), and one split per
// bra for every unit: the slots of (bra, ket) are then consecutive, at the
// ket's running unit number.  Whole kets instead of units, which need no slots
// without a split, cost an 11-atom s+p+d molecule 9.2 ms against 7.7; they
// are taken where a class's slots would pass kSlotMax (large molecules, whose
// lists fill the lanes anyway).
#include <algorithm>
#include <vector>

#include "hf_internal.h"

namespace {

constexpr int kCap = 12;                  // primitives of a unit, as in the J/K build
constexpr long long kSlotMax = 1LL << 25;  // doubles of a class's slots (256 MB)
constexpr size_t kKeep = 1 << 25;          // doubles of scratch the context keeps (256 MB)

// One thread per element of the quartets with slots: the slots added in order,
// their reads consecutive over the threads.  The FP64 additions bound it (80 % of
// the pipe): 0.12 ms for the 0.24 GB of slots of an 11-atom s+p+d molecule, with 16
// reads in flight; 32 saved 5 us on 2 hydrogens and cost that molecule 0.15 ms.
__global__ void __launch_bounds__(128) sum_slots(const HfSlotEntry* __restrict__ entries, int nentry, long long nelement,
                                                 const int* __restrict__ ketlist, const int* __restrict__ ints,
                                                 const PairInfo* __restrict__ info, const double* __restrict__ part,
                                                 double* __restrict__ G, int nbf) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= nelement) return;
  int lo = 0, hi = nentry;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (entries[mid].first <= t) lo = mid; else hi = mid;
  }
  const HfSlotEntry e = entries[lo];
  const int ncd = e.nc * e.nd, nout = e.na * e.nb * ncd;
  const int r = (int)(t - e.first), q = r / nout, o = r - q * nout;
  // the ket's first unit and their count (lists of one ket an item: no units)
  const int u0 = e.unit0 >= 0 ? ints[e.unit0 + q] : q, nu = e.unit0 >= 0 ? ints[e.unit0 + q + 1] - u0 : 1;
  const double* p = part + e.slot + (long long)u0 * e.nsplit * nout + o;
  double v = 0.0;
  for (int s = nu * e.nsplit; s > 0; s -= 16, p += 16 * nout) {  // 16 reads in flight
    double x[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = k < s ? p[k * nout] : 0.0;
#pragma unroll
    for (int k = 0; k < 16; ++k) v += x[k];
  }
  const PairInfo bra = info[e.bra], ket = info[ketlist[e.ket0 + q]];
  const int ab = o / ncd, cd = o - ab * ncd;
  const size_t n = (size_t)nbf;
  const size_t i = bra.bfA + ab / e.nb, j = bra.bfB + ab % e.nb, k = ket.bfA + cd / e.nd, l = ket.bfB + cd % e.nd;
  G[((i * n + j) * n + k) * n + l] = v;
}

// The kernels leave each unique quartet's block at (i j | k l) with the shells
// of i, j and of k, l in the order of their pairs and the bra pair's rank not
// below the ket's; every other element is the copy of one of those.  Inside a
// block that holds two images of an integral (i and j of one shell, or bra and
// ket the same pair) the one with the larger index first is copied to the
// other.  One block per row (i, j), a thread per (k, l), writes coalesced; the
// reads are of the element's image, so HBM (one tensor read and written) bounds
// it.  key[A * ns + B] (pair of shells A, B in its own order) is the pair's
// rank + 1, zero for the reversed order of two different shells.
__global__ void mirror_tensor(double* __restrict__ G, int n, const int* __restrict__ bf_shell,
                              const int* __restrict__ key, int ns) {
  const int ij = blockIdx.x, i = ij / n, j = ij - i * n;
  const int si = bf_shell[i], sj = bf_shell[j];
  int kij = key[(size_t)si * ns + sj];
  const bool rij = kij == 0 || (si == sj && i < j);
  if (kij == 0) kij = key[(size_t)sj * ns + si];
  const size_t nn = (size_t)n * n, bra = rij ? (size_t)j * n + i : (size_t)ij;
  for (int kl = blockIdx.y * blockDim.x + threadIdx.x; kl < (int)nn; kl += gridDim.y * blockDim.x) {
    const int k = kl / n, l = kl - k * n;
    const int sk = bf_shell[k], sl = bf_shell[l];
    int kkl = key[(size_t)sk * ns + sl];
    const bool rkl = kkl == 0 || (sk == sl && k < l);
    if (kkl == 0) kkl = key[(size_t)sl * ns + sk];
    const size_t ket = rkl ? (size_t)l * n + k : (size_t)kl;
    const bool sw = kij < kkl || (kij == kkl && bra < ket);
    if (!(rij || rkl || sw)) continue;  // the element itself was written
    G[(size_t)ij * nn + kl] = sw ? G[ket * nn + bra] : G[bra * nn + ket];
  }
}

int ncart(int l) { return (l + 1) * (l + 2) / 2; }

// Ket units of one pair class: {pair, first << 16 | count, running number, more
// than one unit}, in buckets of like size, by place in the pair list inside one.
struct Units {
  std::vector<int4> u;
  std::vector<int> place;      // of each unit's ket
  std::vector<int> buckets;    // boundaries
  std::vector<int> size;       // largest unit of each bucket
  std::vector<int> unit0;      // first running number of each ket, and the total
  int most = 0, multi = 0;     // largest unit; kets of more than one unit (the first of the list)
};

Units make_units(const hf_basis* b, int X, int cap) {
  const int s0 = b->class_begin[X], np = b->class_begin[X + 1] - s0;
  Units r;
  r.unit0.push_back(0);
  std::vector<long long> count(cap + 1, 0);
  auto size_of = [&](int k) { return b->nprim_sig_h[b->ketlist_h[s0 + k]]; };
  for (int k = 0; k < np; ++k) {
    const int n = size_of(k), nu = std::max(1, (n + cap - 1) / cap);
    for (int u = 0; u < nu; ++u) {
      const int c = (u + 1) * n / nu - u * n / nu;
      ++count[c];
      r.most = std::max(r.most, c);
    }
    r.multi += nu > 1;
    r.unit0.push_back(r.unit0.back() + nu);
  }
  const std::vector<int> cut = hf_lane_time_cuts(count.data(), r.most + 1);
  r.buckets.push_back(0);
  for (size_t c = 0; c + 1 < cut.size(); ++c) {
    for (int k = 0; k < np; ++k) {
      const int n = size_of(k), nu = r.unit0[k + 1] - r.unit0[k];
      for (int u = 0; u < nu; ++u) {
        const int k0 = u * n / nu, k1 = (u + 1) * n / nu;
        if (k1 - k0 < cut[c + 1] || k1 - k0 >= cut[c]) continue;
        r.u.push_back(make_int4(b->ketlist_h[s0 + k], k0 << 16 | (k1 - k0), r.unit0[k] + u, nu > 1));
        r.place.push_back(k);
      }
    }
    if ((int)r.u.size() > r.buckets.back()) {
      r.size.push_back(0);
      for (size_t v = r.buckets.back(); v < r.u.size(); ++v) r.size.back() = std::max(r.size.back(), r.u[v].y & 0xffff);
      r.buckets.push_back((int)r.u.size());
    }
  }
  return r;
}

// The lists of every class, built once per basis (they depend on nothing else).
int tensor_plan(hf_basis* b) {
  HfTensorPlan& p = b->tensor;
  if (p.ready) return HF_OK;
  hf_ctx* ctx = b->ctx;
  cudaStream_t st = ctx->stream;
  const int ns = b->nshell;
  // one host vector per device array: key, shells of the functions, then the lists
  std::vector<int> h;
  std::vector<int4> hu;
  std::vector<long long> hs;
  std::vector<HfSlotEntry> he;
  auto add = [&](const std::vector<int>& v) {
    const size_t at = h.size();
    h.insert(h.end(), v.begin(), v.end());
    return at;
  };
  h.assign((size_t)ns * ns, 0);
  for (int X = 0; X < HF_NPAIRCLASS; ++X)  // rank: by class, then the place in the class's list
    for (int k = b->class_begin[X]; k < b->class_begin[X + 1]; ++k) {
      const int pr = b->ketlist_h[k];
      h[(size_t)b->pair_A[pr] * ns + b->pair_B[pr]] = k + 1;
    }
  const size_t o_shell = h.size();
  for (int s = 0; s < ns; ++s) h.insert(h.end(), b->sh_bf[s + 1] - b->sh_bf[s], s);
  struct Span {
    size_t bra, kbeg, kend, ioff, nsplit, slot, unit;
  };
  Span span[HF_NCLASS];
  p.scratch = 0;
  p.nelement = 0;
  for (int Y = 0; Y < HF_NPAIRCLASS; ++Y) {
    if (b->class_begin[Y] == b->class_begin[Y + 1]) continue;
    const int yb = b->class_begin[Y];
    // units, and whole kets where a class's slots would be too many; uploaded at first use
    Units kind[2] = {make_units(b, Y, kCap), make_units(b, Y, HF_MAX_NPRIM * HF_MAX_NPRIM)};
    size_t o_unit[2] = {0, 0};
    int o_unit0[2] = {-1, -1};
    for (int X = Y; X < HF_NPAIRCLASS; ++X) {
      const int cls = X * (X + 1) / 2 + Y, xb = b->class_begin[X], xe = b->class_begin[X + 1];
      if (xb == xe) continue;
      const EriClassOps& op = ctx->ops[cls];
      const bool wide = !op.rys_native && op.chunk == 32;
      const int chunk = wide ? 32 : 1, nchunk = op.rys_native ? op.rys_nchunks : 0;
      int la, lb, lc, ld;
      pair_ls(X, &la, &lb);
      pair_ls(Y, &lc, &ld);
      HfSlotEntry proto{};
      proto.na = (unsigned char)ncart(la);
      proto.nb = (unsigned char)ncart(lb);
      proto.nc = (unsigned char)ncart(lc);
      proto.nd = (unsigned char)ncart(ld);
      const int nout = proto.na * proto.nb * proto.nc * proto.nd;
      auto slot_entry = [&](int pair, int ket0, int nsplit, long long at, long long quartet) {
        HfSlotEntry v = proto;
        v.bra = pair;
        v.ket0 = ket0;
        v.nsplit = nsplit;
        v.slot = at;
        v.first = quartet * nout;
        return v;
      };
      std::vector<int> bra, kb, ke, io, sp;
      std::vector<long long> slot;
      std::vector<HfSlotEntry> ent;
      long long used = 0, nquartet = 0;
      int which = 0;
      for (;; which = 1) {
        const Units& U = kind[which];
        const std::vector<int>& bk = wide ? U.buckets : b->buckets[Y];
        bra.clear(); kb.clear(); ke.clear(); sp.clear(); slot.clear(); ent.clear();
        io.assign(1, 0);
        used = nquartet = 0;
        std::vector<long long> len;  // primitive quartets of an item (its longest lane's)
        std::vector<int> bra_at;     // place of the entry's bra
        long long work = 0;
        for (int i = xb; i < xe; ++i) {
          const long long nbp = b->nprim_sig_h[b->ketlist_h[i]];
          for (size_t u = 0; u + 1 < bk.size(); ++u) {
            const int k0 = bk[u];
            int k1 = bk[u + 1];
            if (X == Y)  // kets up to the bra's own place: a prefix of the bucket
              k1 = wide ? (int)(std::upper_bound(U.place.begin() + k0, U.place.begin() + k1, i - xb) - U.place.begin())
                        : std::min(k1, i - xb + 1);
            const long long l = nbp * (wide ? std::max(1, U.size[u]) : b->nprim_sig_h[b->ketlist_h[yb + k0]]);
            // a pair without significant primitives: the zeroed tensor's blocks (as a
            // unit it is evaluated, since its slot is read)
            if (k0 >= k1 || l == 0) continue;
            bra.push_back(b->ketlist_h[i]);
            bra_at.push_back(i - xb);
            kb.push_back(k0);
            ke.push_back(k1);
            len.push_back(l);
            work += l * ((k1 - k0 + chunk - 1) / chunk) * std::max(1, nchunk);
          }
        }
        // split as the J/K lists are (hf_basis_prepare_work), but alike for all units of a bra
        const long long target =
            std::max<long long>(op.rys_native ? 16 : wide ? 9 : 64, work / (16LL * ctx->num_sms));
        for (size_t e = 0; e < bra.size(); ++e) {
          const long long nbp = b->nprim_sig_h[bra[e]], l = wide ? nbp * std::max(1, U.most) : len[e];
          const long long most = op.rys_native ? l : wide ? nbp : (l + 31) / 32;
          const int parts = (int)std::max(1LL, std::min((l + target - 1) / target, most));
          sp.push_back(parts * std::max(1, nchunk));
          const long long next = (long long)io.back() + (long long)((ke[e] - kb[e] + chunk - 1) / chunk) * sp[e];
          if (next > (1 << 30)) return hf_fail(HF_ERR_TOO_LARGE, "class %d: too many work items", cls);
          io.push_back((int)next);
          if (!wide) {
            slot.push_back(parts > 1 ? used : -1);
            if (parts > 1) {
              ent.push_back(slot_entry(bra[e], yb + kb[e], parts, used, nquartet));
              used += (long long)(ke[e] - kb[e]) * parts * nout;
              nquartet += ke[e] - kb[e];
            }
          } else if (e > 0 && bra[e] == bra[e - 1]) {
            slot.push_back(slot.back());
          } else {  // the kets of this bra that have slots: all of them, or those of several units
            const int kets = X == Y ? bra_at[e] + 1 : (int)U.unit0.size() - 1;
            const int have = parts > 1 ? kets : std::min(kets, U.multi);
            slot.push_back(used);
            if (have > 0) {
              ent.push_back(slot_entry(bra[e], yb, parts, used, nquartet));
              used += (long long)U.unit0[have] * parts * nout;
              nquartet += have;
            }
          }
        }
        if (!wide || which == 1 || used <= kSlotMax) break;
      }
      if (wide && o_unit0[which] < 0) {
        o_unit[which] = hu.size();
        hu.insert(hu.end(), kind[which].u.begin(), kind[which].u.end());
        o_unit0[which] = (int)add(kind[which].unit0);
      }
      for (long long& v : slot)
        if (v >= 0) v += (long long)p.scratch;
      for (HfSlotEntry& v : ent) {
        v.slot += (long long)p.scratch;
        v.first += p.nelement;
        v.unit0 = wide ? o_unit0[which] : -1;
      }
      p.scratch += (size_t)used;
      p.nelement += nquartet * nout;
      he.insert(he.end(), ent.begin(), ent.end());
      span[cls] = Span{add(bra), add(kb), add(ke), add(io), add(sp), hs.size(), o_unit[which]};
      hs.insert(hs.end(), slot.begin(), slot.end());
      JKWork& w = p.w[cls];
      w = JKWork{};
      w.nbra = (int)bra.size();
      w.nitems = io.back();
      w.chunk = chunk;
      w.nchunk = nchunk;
      w.ket = b->ketlist.ptr + yb;
      w.counter = b->counters.ptr + 2 * cls;
    }
  }
  HF_CHECK(p.ints.alloc(ctx, h.size()));
  HF_CHECK(p.units.alloc(ctx, std::max<size_t>(1, hu.size())));
  HF_CHECK(p.slots.alloc(ctx, std::max<size_t>(1, hs.size())));
  HF_CHECK(p.entries.alloc(ctx, std::max<size_t>(1, he.size())));
  HF_CUDA(cudaMemcpyAsync(p.ints.ptr, h.data(), sizeof(int) * h.size(), cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaMemcpyAsync(p.units.ptr, hu.data(), sizeof(int4) * hu.size(), cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaMemcpyAsync(p.slots.ptr, hs.data(), sizeof(long long) * hs.size(), cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaMemcpyAsync(p.entries.ptr, he.data(), sizeof(HfSlotEntry) * he.size(), cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaStreamSynchronize(st));  // the host vectors go
  for (int c = 0; c < HF_NCLASS; ++c) {
    JKWork& w = p.w[c];
    if (w.nitems == 0) continue;
    w.bra = p.ints.ptr + span[c].bra;
    w.kbeg = p.ints.ptr + span[c].kbeg;
    w.kend = p.ints.ptr + span[c].kend;
    w.ioff = p.ints.ptr + span[c].ioff;
    w.nsplit = p.ints.ptr + span[c].nsplit;
    p.slot[c] = p.slots.ptr + span[c].slot;
    p.unit[c] = w.chunk == 32 ? p.units.ptr + span[c].unit : nullptr;
  }
  p.key = p.ints.ptr;
  p.bf_shell = p.ints.ptr + o_shell;
  p.nentry = (int)he.size();
  p.ready = true;
  return HF_OK;
}

}  // namespace

int hf_eri_tensor_device(hf_basis* b, double* G) {
  hf_ctx* ctx = b->ctx;
  cudaStream_t st = ctx->stream;
  HF_CHECK(tensor_plan(b));
  const HfTensorPlan& p = b->tensor;
  const int n = b->nbf;
  const size_t nn = (size_t)n * n;
  // the slots: up to kKeep doubles stay with the context (one allocation that
  // grows; every user is ordered on its stream), larger ones go with the call
  DevArray<double> own;
  double* part = ctx->slots;
  if (p.scratch > kKeep) {
    HF_CHECK(own.alloc(ctx, p.scratch));
    part = own.ptr;
  } else if (p.scratch > ctx->nslots) {
    hf_dev_free(ctx, ctx->slots, ctx->nslots * sizeof(double));
    ctx->slots = nullptr;
    ctx->nslots = 0;
    void* v = nullptr;
    HF_CHECK(hf_dev_alloc(ctx, &v, p.scratch * sizeof(double)));
    part = ctx->slots = static_cast<double*>(v);
    ctx->nslots = p.scratch;
  }
  HF_CUDA(cudaMemsetAsync(G, 0, nn * nn * sizeof(double), st));
  HF_CUDA(cudaMemsetAsync(b->counters.ptr, 0, sizeof(int) * 2 * HF_NCLASS, st));
  const PairSet ps = hf_pairset(b);
  const KernelCommon kc = hf_kernel_common(ctx, 0);
  // heaviest classes first, forked onto the side streams as in hf_jk_run
  HF_CUDA(cudaEventRecord(ctx->fork_ev, st));
  for (int k = 0; k < hf_ctx::kSide; ++k) HF_CUDA(cudaStreamWaitEvent(ctx->side[k], ctx->fork_ev, 0));
  int nside = 0;
  for (int c = HF_NCLASS - 1; c >= 0; --c) {
    const JKWork& w = p.w[c];
    if (w.nitems <= 0) continue;
    ctx->ops[c].store(w, ps, kc, StoreOut{G, part, p.slot[c], p.unit[c], n}, hf_launch_grid(ctx, 4, w.nitems),
                      ctx->side[nside++ % hf_ctx::kSide]);
  }
  const cudaError_t launched = cudaGetLastError();
  for (int k = 0; k < hf_ctx::kSide; ++k) {
    HF_CUDA(cudaEventRecord(ctx->join_ev[k], ctx->side[k]));
    HF_CUDA(cudaStreamWaitEvent(st, ctx->join_ev[k], 0));
  }
  HF_CUDA(launched);
  if (p.nelement > 0)
    sum_slots<<<(unsigned)((p.nelement + 127) / 128), 128, 0, st>>>(p.entries.ptr, p.nentry, p.nelement, b->ketlist.ptr,
                                                                    p.ints.ptr, b->pinfo.ptr, part, G, n);
  const unsigned chunks = (unsigned)std::min<size_t>(std::max<size_t>(1, nn / 1024), 16);
  mirror_tensor<<<dim3((unsigned)nn, chunks), 256, 0, st>>>(G, n, p.bf_shell, p.key, b->nshell);
  HF_CUDA(cudaGetLastError());
  return HF_OK;
}

extern "C" int hf_eri_tensor(hf_basis* b, double* G) {
  if (!b || !G) return hf_fail(HF_ERR_INVALID, "hf_eri_tensor: null argument");
  if (b->nbf > HF_STORED_NBF_MAX)
    return hf_fail(HF_ERR_INVALID, "hf_eri_tensor: nbf %d above %d", b->nbf, HF_STORED_NBF_MAX);
  hf_ctx* ctx = b->ctx;
  std::lock_guard<std::mutex> lk(ctx->mu);
  cudaSetDevice(ctx->device);
  HF_CHECK(hf_eri_tensor_device(b, G));
  HF_CUDA(cudaStreamSynchronize(ctx->stream));
  return HF_OK;
}
