// eig.cu -- eigen-decomposition of small symmetric matrices (the orthogonalised
// Fock matrices of an SCF), one thread block per matrix, several matrices per
// launch.
//
// A library divide-and-conquer solve of a 42 x 42 matrix is some forty small
// launches and 1.6 ms on GB300, most of it latency, and a batch of molecules
// pays it once per molecule.  Here one block does the whole solve in shared
// memory by cyclic Jacobi rotations (Golub and Van Loan, Matrix Computations,
// 8.5), in two precisions: the FP64 pipe of one SM does two multiply-adds per
// clock, the FP32 pipe 128, so
//   1. Jacobi in FP32 gives X0, the eigenvectors to about 1e-6;
//   2. two Newton-Schulz steps X (3 I - X^T X) / 2 make it orthonormal to FP64;
//   3. S = X^T A X is diagonal to about 1e-6, and Jacobi in FP64 on S, rotating
//      X along, finishes in two sweeps or so (quadratic convergence) where a
//      start from A takes eight.
// The result is that of a FP64 Jacobi solve, whatever the FP32 stage left: the
// FP64 sweeps run until one finds no off-diagonal element above 2^-55 of the
// largest element of A, 16 at most.  Sixteen are reached where rounding itself
// keeps elements of a degenerate cluster above that; what is left is then
// checked to be of rounding size.  A matrix with an element that is not finite,
// or one that failed this check, gets NaN for all its eigenvalues and vectors,
// so that no caller goes on with numbers that mean nothing.
// GB300: 0.74 ms for a 42 x 42 Fock matrix (library 1.6 ms in 45 launches); ten RHF
// iterations of a 7-atom molecule from set-up 28.3 -> 17.8 ms, of six molecules of 4
// to 9 atoms in a batch 115 -> 44.6 ms, the overlap matrices' solves included.
#include <algorithm>

#include "herm.cuh"
#include "hf_internal.h"
#include "per_device.h"
#include "scf_internal.h"

namespace {

constexpr int kThreads = 512;

struct EigBatch {
  EigJob j[HF_EIG_BATCH];
};

// Pair k of round r of the round-robin schedule of m (even) indices.
__device__ __forceinline__ void jacobi_pair(int m, int r, int k, int* p, int* q) {
  int a = m - 1, b = r;
  if (k > 0) {
    a = r + k;
    if (a >= m - 1) a -= m - 1;
    b = r - k;
    if (b < 0) b += m - 1;
  }
  *p = min(a, b);
  *q = max(a, b);
}

// Cosine and sine of the rotation that removes a[p][q]: t = tan from the
// smaller root in FP32 (an angle is good enough to 1e-7, the next sweep takes
// the rest), c = 1 / sqrt(1 + t^2) and s = t c in the working precision.
__device__ __forceinline__ float jacobi_t(float app, float aqq, float apq) {
  const float th = (aqq - app) / (2.0f * apq);
  const float t = 1.0f / (fabsf(th) + sqrtf(fmaf(th, th, 1.0f)));  // th = +-inf: t = 0
  return th >= 0.0f ? t : -t;
}
__device__ __forceinline__ void rotation(float app, float aqq, float apq, float* c, float* s) {
  const float t = jacobi_t(app, aqq, apq);
  *c = 1.0f / sqrtf(fmaf(t, t, 1.0f));
  *s = t * *c;
}
__device__ __forceinline__ void rotation(double app, double aqq, double apq, double* c, double* s) {
  // the difference is formed in FP64; the matrix is scaled to elements of at
  // most 1, so FP32 holds what is worth rotating (above 2^-55)
  const double t = (double)jacobi_t(0.0f, (float)(aqq - app), (float)apq);
  *c = hfk::hf_rsqrt(fma(t, t, 1.0));
  *s = t * *c;
}

// Jacobi sweeps on the symmetric m x m matrix a (row stride ld, m even, padded
// with a zero row and column if need be), rotating the columns of v along,
// until a sweep finds no off-diagonal element above thr (true), max_sweeps at
// most (false).
// c, s: m / 2 values each.  One round rotates m / 2 disjoint pairs: each 2 x 2
// block (pair I, pair J) of a is transformed by itself, I <= J (the mirror
// image is written too), so a round takes one pass and two barriers.
template <typename R>
__device__ bool jacobi(R* a, R* v, int m, int ld, R* c, R* s, R thr, int max_sweeps) {
  const int N = m / 2, tid = threadIdx.x, nblk = N * (N + 1) / 2, ntask = nblk + N * m;
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    int any = 0;
    for (int r = 0; r < m - 1; ++r) {
      int mine = 0;
      if (tid < N) {
        int p, q;
        jacobi_pair(m, r, tid, &p, &q);
        const R apq = a[p * ld + q];
        R cc = (R)1, ss = (R)0;
        if (apq > thr || apq < -thr) {
          rotation(a[p * ld + p], a[q * ld + q], apq, &cc, &ss);
          mine = 1;
        }
        c[tid] = cc;
        s[tid] = ss;
      }
      if (!__syncthreads_or(mine)) continue;  // nothing to rotate in this round
      any = 1;
      for (int t = tid; t < ntask; t += kThreads) {
        if (t < nblk) {
          int I = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);  // t = I (I + 1) / 2 + J, J <= I
          while (I * (I + 1) / 2 > t) --I;
          while ((I + 1) * (I + 2) / 2 <= t) ++I;
          const int J = t - I * (I + 1) / 2;
          const R c1 = c[I], s1 = s[I], c2 = c[J], s2 = s[J];
          if (s1 == (R)0 && s2 == (R)0) continue;
          int p1, q1, p2, q2;
          jacobi_pair(m, r, I, &p1, &q1);
          jacobi_pair(m, r, J, &p2, &q2);
          const R x00 = a[p1 * ld + p2], x01 = a[p1 * ld + q2], x10 = a[q1 * ld + p2], x11 = a[q1 * ld + q2];
          const R y00 = c2 * x00 - s2 * x01, y01 = s2 * x00 + c2 * x01;
          const R y10 = c2 * x10 - s2 * x11, y11 = s2 * x10 + c2 * x11;
          const R z00 = c1 * y00 - s1 * y10, z01 = c1 * y01 - s1 * y11;
          const R z10 = s1 * y00 + c1 * y10, z11 = s1 * y01 + c1 * y11;
          a[p1 * ld + p2] = z00;
          a[p2 * ld + p1] = z00;
          a[p1 * ld + q2] = z01;
          a[q2 * ld + p1] = z01;
          a[q1 * ld + q2] = z11;
          a[q2 * ld + q1] = z11;
          if (I != J) {  // on the diagonal z10 = z01
            a[q1 * ld + p2] = z10;
            a[p2 * ld + q1] = z10;
          }
        } else {
          const int k = (t - nblk) / m, i = (t - nblk) - k * m;
          const R c2 = c[k], s2 = s[k];
          if (s2 == (R)0) continue;
          int p, q;
          jacobi_pair(m, r, k, &p, &q);
          const R x = v[i * ld + p], y = v[i * ld + q];
          v[i * ld + p] = c2 * x - s2 * y;
          v[i * ld + q] = s2 * x + c2 * y;
        }
      }
      __syncthreads();
    }
    if (!any) return true;
  }
  return false;
}

// out(i, j) = f(sum_k A B, i, j) over 2 x 2 tiles, A(i, k) at A[i * ai + k *
// ak] and B(k, j) at B[k * ld + j]; sym: i <= j only, mirrored.
template <class F>
__device__ void small_gemm(const double* A, int ai, int ak, const double* B, double* out, int m, int ld, bool sym, F f) {
  const int N = m / 2;
  for (int t = threadIdx.x; t < N * N; t += kThreads) {
    const int I = t / N, J = t - I * N;
    if (sym && I > J) continue;
    double s00 = 0.0, s01 = 0.0, s10 = 0.0, s11 = 0.0;
    const double *a0 = A + 2 * I * ai, *a1 = a0 + ai, *b = B + 2 * J;
    for (int k = 0; k < m; ++k) {
      const double x0 = a0[k * ak], x1 = a1[k * ak], y0 = b[k * ld], y1 = b[k * ld + 1];
      s00 = fma(x0, y0, s00);
      s01 = fma(x0, y1, s01);
      s10 = fma(x1, y0, s10);
      s11 = fma(x1, y1, s11);
    }
    const int i = 2 * I, j = 2 * J;
    double* o = out + i * ld + j;
    o[0] = f(s00, i, j);
    o[1] = f(s01, i, j + 1);
    o[ld] = sym && I == J ? o[1] : f(s10, i + 1, j);
    o[ld + 1] = f(s11, i + 1, j + 1);
    if (sym && I != J) {
      out[j * ld + i] = o[0];
      out[(j + 1) * ld + i] = o[1];
      out[j * ld + i + 1] = o[ld];
      out[(j + 1) * ld + i + 1] = o[ld + 1];
    }
  }
}

__global__ void __launch_bounds__(kThreads) eig_kernel(const EigBatch batch) {
  const EigJob job = batch.j[blockIdx.x];
  const int n = job.n, m = (n + 1) & ~1, ld = m + 1, tid = threadIdx.x;
  extern __shared__ __align__(16) double sm[];
  double* S0 = sm;
  double* S1 = S0 + m * ld;
  double* S2 = S1 + m * ld;
  double* cs = S2 + m * ld;  // rotations: m doubles
  double* red = cs + m;      // 32 doubles
  float* B = reinterpret_cast<float*>(S0);
  float* V = B + m * ld;
  const double* __restrict__ A = job.A;  // column-major, the lower triangle is read
  auto no_result = [&]() {
    for (int t = tid; t < n * n; t += kThreads) job.A[t] = nan("");
    for (int i = tid; i < n; i += kThreads) job.w[i] = nan("");
  };
  // largest element, infinite if one is not finite (tests and powers of two on
  // the exponent bits: a solve waits for every FP64 instruction here)
  auto expo = [](double x) { return (__double2hiint(x) >> 20) & 0x7ff; };
  double mx = 0.0;
  for (int t = tid; t < n * n; t += kThreads) {
    const double v = A[t];
    mx = expo(v) == 0x7ff ? INFINITY : fmax(mx, fabs(v));
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((tid & 31) == 0) red[tid >> 5] = mx;
  __syncthreads();
  mx = red[0];
  for (int k = 1; k < kThreads / 32; ++k) mx = fmax(mx, red[k]);
  if (expo(mx) == 0x7ff) {  // the same in every thread
    no_result();
    return;
  }
  // scaled by a power of two (exactly) to elements in [-1, 1], a little above at the ends of the range
  const int ex = mx > 0.0 ? max(-1022, min(1022, expo(mx) - 1022)) : 0;
  const double down = __hiloint2double((1023 - ex) << 20, 0), up = __hiloint2double((1023 + ex) << 20, 0);
  auto el = [&](int i, int j) -> double {
    return i < n && j < n ? A[(size_t)min(i, j) * n + max(i, j)] * down : 0.0;
  };
  for (int t = tid; t < m * m; t += kThreads) {
    const int i = t / m, j = t - i * m;
    B[i * ld + j] = (float)el(i, j);
    V[i * ld + j] = i == j ? 1.0f : 0.0f;
  }
  __syncthreads();
  float* cf = reinterpret_cast<float*>(cs);
  jacobi<float>(B, V, m, ld, cf, cf + m / 2, 1e-6f, 12);
  for (int t = tid; t < m * m; t += kThreads) {
    const int i = t / m, j = t - i * m;
    S1[i * ld + j] = (double)V[i * ld + j];
  }
  __syncthreads();
  // X <- X (3 I - X^T X) / 2, twice: S1 -> S0 -> S1
  for (int it = 0; it < 2; ++it) {
    double* X = it ? S0 : S1;
    double* Y = it ? S1 : S0;
    small_gemm(X, 1, ld, X, S2, m, ld, true, [](double v, int i, int j) { return i == j ? 1.5 - 0.5 * v : -0.5 * v; });
    __syncthreads();
    small_gemm(X, ld, 1, S2, Y, m, ld, false, [](double v, int, int) { return v; });
    __syncthreads();
  }
  // S = X^T A X into S0
  for (int t = tid; t < m * m; t += kThreads) {
    const int i = t / m, j = t - i * m;
    S0[i * ld + j] = el(i, j);
  }
  __syncthreads();
  small_gemm(S0, ld, 1, S1, S2, m, ld, false, [](double v, int, int) { return v; });
  __syncthreads();
  small_gemm(S1, 1, ld, S2, S0, m, ld, true, [](double v, int, int) { return v; });
  __syncthreads();
  if (!jacobi<double>(S0, S1, m, ld, cs, cs + m / 2, 0x1p-55, 16)) {
    int left = 0;
    for (int t = tid; t < m * m; t += kThreads) {
      const int i = t / m, j = t - i * m;
      left |= i != j && !(fabs(S0[i * ld + j]) <= m * 0x1p-50);
    }
    if (__syncthreads_or(left)) {
      no_result();
      return;
    }
  }
  // ascending order; the pad (a zero row, never rotated into the others) goes last
  for (int i = tid; i < n; i += kThreads) {
    const double w = S0[i * ld + i];
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      const double x = S0[j * ld + j];
      rank += x < w || (x == w && j < i);
    }
    job.w[rank] = w * up;
    cs[i] = (double)rank;
  }
  __syncthreads();
  for (int t = tid; t < n * n; t += kThreads) {
    const int i = t / n, k = t - i * n;  // eigenvector i, row k
    job.A[(size_t)(int)cs[i] * n + k] = S1[k * ld + i];
  }
}

size_t eig_smem(int n) {
  const size_t m = (n + 1) & ~1;
  return (3 * m * (m + 1) + m + 32) * sizeof(double);
}

}  // namespace

int hf_eig_small(hf_ctx* ctx, const EigJob* jobs, int count) {
  static PerDevice limit;
  if (hf_smem_limit(limit, eig_kernel, eig_smem(HF_EIG_NMAX)) < 0)
    return hf_fail(HF_ERR_CUDA, "eigensolver's shared memory: %s", cudaGetErrorString(cudaGetLastError()));
  for (int c0 = 0; c0 < count; c0 += HF_EIG_BATCH) {
    EigBatch b{};
    const int k = std::min(HF_EIG_BATCH, count - c0);
    int nmax = 0;
    for (int i = 0; i < k; ++i) {
      b.j[i] = jobs[c0 + i];
      nmax = std::max(nmax, jobs[c0 + i].n);
    }
    eig_kernel<<<k, kThreads, eig_smem(nmax), ctx->stream>>>(b);
  }
  HF_CUDA(cudaGetLastError());
  return HF_OK;
}
