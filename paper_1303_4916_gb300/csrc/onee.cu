// onee.cu -- one-electron matrices S, T, V of Eqs. 2-4 by the Obara-Saika
// recurrences (setup work, O(nbf^2) per molecule).
//
//   overlap, per axis:  S_{i+1,j} = PA S_ij + (i S_{i-1,j} + j S_{i,j-1}) / (2p)
//                       S_{i,j+1} = PB S_ij + (i S_{i-1,j} + j S_{i,j-1}) / (2p)
//                       S_00 = sqrt(pi/p) exp(-ab/p AB_x^2)
//   kinetic, per axis (Laplacian on the ket):
//                       T_ij = -1/2 [ j(j-1) S_{i,j-2} - 2b(2j+1) S_ij + 4b^2 S_{i,j+2} ]
//                       T = Tx Sy Sz + Sx Ty Sz + Sx Sy Tz
//   nuclear attraction of nucleus C by Rys quadrature: with n = (la+lb)/2 + 1
//   roots u of the rule at T = p |PC|^2, (a|1/r_C|b) = 2 pi / p
//   exp(-ab/p |AB|^2) sum_u w_u Ix Iy Iz, the one-dimensional factors from
//                       I(i+1, 0) = (PA - u PC) I(i, 0) + i (1 - u) / (2p) I(i-1, 0),
//                       I(0, 0) = 1,  I(i, j+1) = I(i+1, j) + AB I(i, j).
#include <cmath>

#include "hf_internal.h"
#include "rys.cuh"

namespace {

__device__ __forceinline__ void cart_pow(int l, int c, int* p) {
  int k = 0;
  for (int x = l; x >= 0; --x)
    for (int y = l - x; y >= 0; --y) {
      if (k == c) { p[0] = x; p[1] = y; p[2] = l - x - y; return; }
      ++k;
    }
}

// scale of Cartesian component c of an axial-normalised shell of angular
// momentum l: sqrt((2l-1)!! / ((2x-1)!! (2y-1)!! (2z-1)!!))
__device__ double comp_scale_any(int l, int c) {
  int p[3];
  cart_pow(l, c, p);
  auto df = [](int x) {
    double r = 1.0;
    for (int k = 2 * x - 1; k > 1; k -= 2) r *= k;
    return r;
  };
  return sqrt(df(l) / (df(p[0]) * df(p[1]) * df(p[2])));
}

__device__ __forceinline__ double warp_add(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One warp per pair i >= j of basis functions (V, S and T are symmetric),
// its lanes over the primitive pairs for S and T and over (primitive pair,
// nucleus) for V.  FP64 issue bounds it; a thread per (i, j), the form
// before, walked all primitives and nuclei in series with the whole
// recursion array of an Obara-Saika attraction in local memory: 2.9 ms at 42
// functions of 7 atoms.
__global__ void __launch_bounds__(128) one_electron_kernel(
    int nbf, const int* __restrict__ bf_shell, const int* __restrict__ sh_l, const int* __restrict__ sh_bf,
    const int* __restrict__ sh_nprim, const int* __restrict__ sh_prim, const double* __restrict__ sh_xyz,
    const double* __restrict__ exps, const double* __restrict__ coefs, int natom,
    const double* __restrict__ atom_xyz, const int* __restrict__ atom_Z, const double* __restrict__ rys,
    double* __restrict__ S, double* __restrict__ T, double* __restrict__ V) {
  const long long t = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (t >= (long long)nbf * (nbf + 1) / 2) return;
  int i = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);  // t = i (i + 1) / 2 + j, corrected below
  while ((long long)i * (i + 1) / 2 > t) --i;
  while ((long long)(i + 1) * (i + 2) / 2 <= t) ++i;
  const int j = (int)(t - (long long)i * (i + 1) / 2);
  const int sa = bf_shell[i], sb = bf_shell[j];
  const int la = sh_l[sa], lb = sh_l[sb];
  int pa[3], pb[3];
  cart_pow(la, i - sh_bf[sa], pa);
  cart_pow(lb, j - sh_bf[sb], pb);
  const double* A = sh_xyz + 3 * sa;
  const double* B = sh_xyz + 3 * sb;
  const double scale = comp_scale_any(la, i - sh_bf[sa]) * comp_scale_any(lb, j - sh_bf[sb]);
  double AB[3], r2 = 0.0;
  for (int x = 0; x < 3; ++x) {
    AB[x] = A[x] - B[x];
    r2 += AB[x] * AB[x];
  }
  const int nb = sh_nprim[sb], np = sh_nprim[sa] * nb;
  double s_sum = 0.0, t_sum = 0.0, v_sum = 0.0;
  for (int k = lane; k < np; k += 32) {
    const int ka = k / nb, kb = k - ka * nb;
    const double a = exps[sh_prim[sa] + ka], b = exps[sh_prim[sb] + kb];
    const double c = coefs[sh_prim[sa] + ka] * coefs[sh_prim[sb] + kb];
    const double p = a + b, o2p = 0.5 / p, mu = a * b / p;
    double st[3], tk[3];
    for (int x = 0; x < 3; ++x) {
      const double P = (a * A[x] + b * B[x]) / p, PA = P - A[x], PB = P - B[x];
      double s[5][7];  // 1D overlaps, i <= la, j <= lb + 2
      s[0][0] = sqrt(3.14159265358979323846 / p) * exp(-mu * AB[x] * AB[x]);
      for (int ii = 0; ii < pa[x]; ++ii) s[ii + 1][0] = PA * s[ii][0] + (ii > 0 ? ii * o2p * s[ii - 1][0] : 0.0);
      for (int ii = 0; ii <= pa[x]; ++ii)
        for (int jj = 0; jj < pb[x] + 2; ++jj)
          s[ii][jj + 1] = PB * s[ii][jj] + ((ii > 0 ? ii * s[ii - 1][jj] : 0.0) + (jj > 0 ? jj * s[ii][jj - 1] : 0.0)) * o2p;
      const int jj = pb[x];
      double v = -2.0 * b * (2 * jj + 1) * s[pa[x]][jj] + 4.0 * b * b * s[pa[x]][jj + 2];
      if (jj >= 2) v += jj * (jj - 1) * s[pa[x]][jj - 2];
      st[x] = s[pa[x]][jj];
      tk[x] = -0.5 * v;
    }
    s_sum += c * st[0] * st[1] * st[2];
    t_sum += c * (tk[0] * st[1] * st[2] + st[0] * tk[1] * st[2] + st[0] * st[1] * tk[2]);
  }
  const int nr = (la + lb) / 2 + 1;
  for (long long q = lane; q < (long long)np * natom; q += 32) {
    const int at = (int)(q / np), k = (int)(q - (long long)at * np);
    if (atom_Z[at] == 0) continue;
    const int ka = k / nb, kb = k - ka * nb;
    const double a = exps[sh_prim[sa] + ka], b = exps[sh_prim[sb] + kb];
    const double c = coefs[sh_prim[sa] + ka] * coefs[sh_prim[sb] + kb];
    const double ip = 1.0 / (a + b), p = a + b, o2p = 0.5 * ip;
    const double pre = 2.0 * 3.14159265358979323846 * ip * exp(-(a * b * ip) * r2);
    double PA[3], PC[3];
    for (int x = 0; x < 3; ++x) {
      const double P = (a * A[x] + b * B[x]) * ip;
      PA[x] = P - A[x];
      PC[x] = P - atom_xyz[3 * at + x];
    }
    const double Tn = p * (PC[0] * PC[0] + PC[1] * PC[1] + PC[2] * PC[2]);
    double vr = 0.0;
    for (int r = 0; r < nr; ++r) {
      double u, prod;
      rys_rule_root(rys, nr, r, Tn, &u, &prod);
      for (int x = 0; x < 3; ++x) {
        double g[9];
        g[0] = 1.0;
        const double c00 = PA[x] - u * PC[x], b10 = (1.0 - u) * o2p;
        const int top = pa[x] + pb[x];
        for (int m = 0; m < top; ++m) g[m + 1] = c00 * g[m] + (m > 0 ? m * b10 * g[m - 1] : 0.0);
        for (int m = 1; m <= pb[x]; ++m)
          for (int e = pa[x]; e <= top - m; ++e) g[e] = g[e + 1] + AB[x] * g[e];
        prod *= g[pa[x]];
      }
      vr += prod;
    }
    v_sum -= c * atom_Z[at] * pre * vr;
  }
  s_sum = warp_add(s_sum);
  t_sum = warp_add(t_sum);
  v_sum = warp_add(v_sum);
  if (lane == 0) {
    const size_t ij = (size_t)i * nbf + j, ji = (size_t)j * nbf + i;
    S[ij] = S[ji] = s_sum * scale;
    T[ij] = T[ji] = t_sum * scale;
    V[ij] = V[ji] = v_sum * scale;
  }
}

}  // namespace

int hf_basis_one_electron(hf_basis* b) {
  if (b->have_one) return HF_OK;
  hf_ctx* ctx = b->ctx;
  cudaStream_t st = ctx->stream;
  const int n = b->nbf, ns = b->nshell;
  std::vector<int> bf_shell(n);
  for (int s = 0; s < ns; ++s)
    for (int k = b->sh_bf[s]; k < b->sh_bf[s + 1]; ++k) bf_shell[k] = s;
  std::vector<double> sh_xyz(3 * ns), at_xyz(3 * b->natom);
  std::vector<int> Z(b->natom);
  for (int s = 0; s < ns; ++s)
    for (int x = 0; x < 3; ++x) sh_xyz[3 * s + x] = b->atoms[b->sh_atom[s]].xyz[x];
  for (int a = 0; a < b->natom; ++a) {
    Z[a] = b->atoms[a].Z;
    for (int x = 0; x < 3; ++x) at_xyz[3 * a + x] = b->atoms[a].xyz[x];
  }
  DevArray<int> dbs, dl, dbf, dn, dp, dZ;
  DevArray<double> dsx, dex, dco, dax;
  HF_CHECK(dbs.alloc(ctx, n));
  HF_CHECK(dl.alloc(ctx, ns));
  HF_CHECK(dbf.alloc(ctx, ns + 1));
  HF_CHECK(dn.alloc(ctx, ns));
  HF_CHECK(dp.alloc(ctx, ns));
  HF_CHECK(dZ.alloc(ctx, b->natom));
  HF_CHECK(dsx.alloc(ctx, 3 * ns));
  HF_CHECK(dex.alloc(ctx, b->nprim));
  HF_CHECK(dco.alloc(ctx, b->nprim));
  HF_CHECK(dax.alloc(ctx, 3 * b->natom));
  HF_CHECK(b->S.alloc(ctx, (size_t)n * n));
  HF_CHECK(b->T.alloc(ctx, (size_t)n * n));
  HF_CHECK(b->V.alloc(ctx, (size_t)n * n));
  HF_CUDA(cudaMemcpyAsync(dbs.ptr, bf_shell.data(), sizeof(int) * n, cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaMemcpyAsync(dl.ptr, b->sh_l.data(), sizeof(int) * ns, cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaMemcpyAsync(dbf.ptr, b->sh_bf.data(), sizeof(int) * (ns + 1), cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaMemcpyAsync(dn.ptr, b->sh_nprim.data(), sizeof(int) * ns, cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaMemcpyAsync(dp.ptr, b->sh_prim.data(), sizeof(int) * ns, cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaMemcpyAsync(dZ.ptr, Z.data(), sizeof(int) * b->natom, cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaMemcpyAsync(dsx.ptr, sh_xyz.data(), sizeof(double) * 3 * ns, cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaMemcpyAsync(dex.ptr, b->exps.data(), sizeof(double) * b->nprim, cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaMemcpyAsync(dco.ptr, b->coefs.data(), sizeof(double) * b->nprim, cudaMemcpyHostToDevice, st));
  HF_CUDA(cudaMemcpyAsync(dax.ptr, at_xyz.data(), sizeof(double) * 3 * b->natom, cudaMemcpyHostToDevice, st));
  const long long warps = (long long)n * (n + 1) / 2;
  one_electron_kernel<<<(unsigned)((warps + 3) / 4), 128, 0, st>>>(n, dbs.ptr, dl.ptr, dbf.ptr, dn.ptr, dp.ptr, dsx.ptr,
                                                                  dex.ptr, dco.ptr, b->natom, dax.ptr, dZ.ptr,
                                                                  ctx->rys, b->S.ptr, b->T.ptr, b->V.ptr);
  HF_CUDA(cudaGetLastError());
  HF_CUDA(cudaStreamSynchronize(st));
  b->have_one = true;
  return HF_OK;
}

extern "C" int hf_one_electron(hf_basis* b, double* S, double* T, double* V, double* e_nuc) {
  if (!b) return hf_fail(HF_ERR_INVALID, "null basis");
  hf_ctx* ctx = b->ctx;
  std::lock_guard<std::mutex> lk(ctx->mu);
  cudaSetDevice(ctx->device);
  HF_CHECK(hf_basis_one_electron(b));
  const size_t nn = (size_t)b->nbf * b->nbf * sizeof(double);
  if (S) HF_CUDA(cudaMemcpyAsync(S, b->S.ptr, nn, cudaMemcpyDeviceToDevice, ctx->stream));
  if (T) HF_CUDA(cudaMemcpyAsync(T, b->T.ptr, nn, cudaMemcpyDeviceToDevice, ctx->stream));
  if (V) HF_CUDA(cudaMemcpyAsync(V, b->V.ptr, nn, cudaMemcpyDeviceToDevice, ctx->stream));
  HF_CUDA(cudaStreamSynchronize(ctx->stream));
  if (e_nuc) *e_nuc = b->e_nuc;
  return HF_OK;
}
