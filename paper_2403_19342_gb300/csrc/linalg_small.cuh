// Small dense linear algebra inside one CTA (shared memory), FP64: parallel
// cyclic Jacobi eigensolver, stable ranking of a diagonal, Gauss-Jordan
// inverse.  Used by the local eigenproblems, Rayleigh-Ritz steps and the
// per-parent smoother inverses.
#pragma once
#include "msmg_internal.cuh"
#include "reduce.cuh"
#include <cmath>

namespace msmg {

// ------------------------------------------------------------------ Jacobi
// Parallel cyclic Jacobi (round-robin pairing) on the n x n symmetric matrix A
// in shared memory; V receives the eigenvectors (columns).  On return the
// diagonal of A holds the eigenvalues.
__device__ inline void jacobi_eig(double* A, double* V, int n, double* cs, int* pr, double* red, int max_sweeps,
                           double rtol) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int npad = n + (n & 1);
  const int half = npad / 2;
  for (int i = tid; i < n * n; i += nthr) V[i] = (i / n == i % n) ? 1.0 : 0.0;
  __syncthreads();
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    double v[2] = {0.0, 0.0};
    for (int i = tid; i < n * n; i += nthr) {
      const double a = A[i];
      v[1] += a * a;
      if (i / n != i % n) v[0] += a * a;
    }
    block_sum<2>(v, red + 2);
    if (tid == 0) { red[0] = v[0]; red[1] = v[1]; }
    __syncthreads();
    const bool conv = red[0] <= rtol * rtol * red[1];
    __syncthreads();
    if (conv) break;
    for (int r = 0; r < npad - 1; ++r) {
      for (int i = tid; i < half; i += nthr) {
        int pa = (i == 0) ? 0 : 1 + ((i - 1 + r) % (npad - 1));
        const int j = npad - 1 - i;
        int pb = 1 + ((j - 1 + r) % (npad - 1));
        if (pa > pb) { int t = pa; pa = pb; pb = t; }
        double c = 1.0, s = 0.0;
        if (pb < n) {
          const double apq = A[pa * n + pb];
          if (fabs(apq) > 1e-300) {
            const double theta = (A[pb * n + pb] - A[pa * n + pa]) / (2.0 * apq);
            const double t = (theta >= 0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
            c = 1.0 / sqrt(t * t + 1.0);
            s = t * c;
          }
        }
        cs[2 * i] = c;
        cs[2 * i + 1] = s;
        pr[2 * i] = pa;
        pr[2 * i + 1] = pb;
      }
      __syncthreads();
      for (int idx = tid; idx < half * n; idx += nthr) {     // rows: A <- J^T A
        const int i = idx / n, col = idx % n;
        const int p = pr[2 * i], q = pr[2 * i + 1];
        if (q >= n) continue;
        const double c = cs[2 * i], s = cs[2 * i + 1];
        const double ap = A[p * n + col], aq = A[q * n + col];
        A[p * n + col] = c * ap - s * aq;
        A[q * n + col] = s * ap + c * aq;
      }
      __syncthreads();
      for (int idx = tid; idx < half * n; idx += nthr) {     // columns: A <- A J, V <- V J
        const int i = idx / n, row = idx % n;
        const int p = pr[2 * i], q = pr[2 * i + 1];
        if (q >= n) continue;
        const double c = cs[2 * i], s = cs[2 * i + 1];
        const double ap = A[row * n + p], aq = A[row * n + q];
        A[row * n + p] = c * ap - s * aq;
        A[row * n + q] = s * ap + c * aq;
        const double vp = V[row * n + p], vq = V[row * n + q];
        V[row * n + p] = c * vp - s * vq;
        V[row * n + q] = s * vp + c * vq;
      }
      __syncthreads();
    }
  }
}

// order[k] = index of the k-th smallest diagonal entry of A (stable).  NaN
// entries sort as +infinity, so the ranks always form a permutation of 0..n-1.
__device__ __forceinline__ double sort_key(double v) { return isnan(v) ? INFINITY : v; }
__device__ inline void sort_diag(const double* A, int n, int* order) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double di = sort_key(A[i * n + i]);
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      const double dj = sort_key(A[j * n + j]);
      rank += (dj < di) || (dj == di && j < i);
    }
    order[rank] = i;
  }
  __syncthreads();
}

// In-place Gauss-Jordan inverse of an SPD n x n matrix in shared memory: one division per
// row and pivot, one FMA per entry (a division per entry made it as slow as the
// eigensolve beside it).
__device__ inline void gj_inverse(double* A, int n, double* rowk, double* colk) {
  for (int k = 0; k < n; ++k) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      rowk[i] = A[k * n + i];
      colk[i] = A[i * n + k] / A[k * n + k];
    }
    __syncthreads();
    const double piv = rowk[k];
    for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) {
      const int i = idx / n, j = idx - i * n;
      double v;
      if (i == k) v = j == k ? 1.0 / piv : rowk[j] / piv;
      else if (j == k) v = -colk[i];
      else v = fma(-colk[i], rowk[j], A[idx]);
      A[idx] = v;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ tridiagonal eigensolver
// The nc smallest eigenpairs of the symmetric n x n matrix A (shared memory, overwritten):
// Householder tridiagonalisation, bisection on the Sturm sequence (32 points per pass and
// warp), inverse iteration with partial pivoting, Gram-Schmidt over all vectors, back
// transformation (Golub and Van Loan, chapter 8; Barth, Martin and Wilkinson 1967 for the
// bisection; Peters and Wilkinson 1971 for the inverse iteration).  Returns whether every
// pair has residual ||T y - lambda y|| <= 1e-13 ||T|| (the same answer in every thread); the
// caller falls back to Jacobi otherwise.
// Work space w (tri_doubles(n, nc) doubles): eigenvalues at w[0 .. nc), vectors at
// w + tri_vectors(n) as nc rows of n.
constexpr int kTriBatch = 4;                         // inverse iterations at a time
__host__ __device__ inline int tri_vectors(int n) { return 5 * n + 16; }
__host__ __device__ inline int tri_doubles(int n, int nc) { return tri_vectors(n) + nc * n + 5 * kTriBatch * n + 8; }

// eigenvalues of T (diagonal d, squared off-diagonals e2) below x: sign changes of the
// leading minors' ratio-free recurrence, rescaled by powers of two
__device__ inline int sturm_count(const double* d, const double* e2, int n, double x) {
  int cnt = 0;
  double p0 = 1.0, p1 = d[0] - x;
  if (p1 == 0.0) p1 = -0x1p-200;
  if (p1 < 0.0) ++cnt;
  bool neg = p1 < 0.0;
  for (int k = 1; k < n; ++k) {
    const double p2 = fma(d[k] - x, p1, -e2[k - 1] * p0);
    p0 = p1;
    p1 = p2;
    // a zero minor becomes a tiny one of the sign opposite to its predecessor's
    if (p1 == 0.0) p1 = (neg ? 0x1p-200 : -0x1p-200) * fabs(p0);
    const bool ng = p1 < 0.0;
    if (ng != neg) ++cnt;
    neg = ng;
    const int e = (int)((__double_as_longlong(p1) >> 52) & 0x7ff), f = (int)((__double_as_longlong(p0) >> 52) & 0x7ff);
    const int m = e > f ? e : f;
    if (m > 1023 + 200) { p0 *= 0x1p-300; p1 *= 0x1p-300; }
    else if (m < 1023 - 200) { p0 *= 0x1p+300; p1 *= 0x1p+300; }
  }
  return cnt;
}

__device__ inline bool tridiag_eig(double* A, int n, int nc, double* w) {
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
  double *lam = w, *d = w + n, *e = d + n, *tau = e + n, *v = tau + n, *sc = v + n;   // sc: 16 scalars
  double* Z = w + tri_vectors(n);
  double* lu = Z + nc * n;                           // [5][n][kTriBatch]
  // ---- tridiagonalisation: column k's reflector v (v_0 first) stays below the diagonal
  for (int k = 0; k + 2 < n; ++k) {
    const int m = n - k - 1;
    if (warp == 0) {
      double s = 0.0;
      for (int i = lane + 1; i < m; i += 32) { const double x = A[(k + 1 + i) * n + k]; s = fma(x, x, s); }
      s = warp_sum(s);
      if (lane == 0) {
        const double x0 = A[(k + 1) * n + k];
        double t = 0.0, beta = x0, v0 = 1.0;
        if (s > 0.0) {
          beta = x0 <= 0.0 ? sqrt(fma(x0, x0, s)) : -sqrt(fma(x0, x0, s));
          v0 = x0 - beta;
          t = 2.0 / fma(v0, v0, s);                  // H = I - t v v^T
        }
        e[k] = beta;
        tau[k] = t;
        A[(k + 1) * n + k] = v0;
      }
    }
    __syncthreads();
    const double t = tau[k];
    if (t != 0.0) {
      // p = t A22 v: four threads per row, column reads (A22 is symmetric)
      const int part = tid & 3;
      for (int i = tid >> 2; i < (m + 7) / 8 * 8; i += nthr >> 2) {
        double s = 0.0;
        if (i < m)
          for (int j = part; j < m; j += 4) s = fma(A[(k + 1 + j) * n + k + 1 + i], A[(k + 1 + j) * n + k], s);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (part == 0 && i < m) v[i] = t * s;
      }
      __syncthreads();
      if (warp == 0) {
        double s = 0.0;
        for (int i = lane; i < m; i += 32) s = fma(v[i], A[(k + 1 + i) * n + k], s);
        s = warp_sum(s) * 0.5 * t;
        for (int i = lane; i < m; i += 32) v[i] = fma(-s, A[(k + 1 + i) * n + k], v[i]);   // w = p - (t p.v / 2) v
      }
      __syncthreads();
      for (int idx = tid; idx < m * m; idx += nthr) {
        const int i = idx / m, j = idx - i * m;
        const double vi = A[(k + 1 + i) * n + k], vj = A[(k + 1 + j) * n + k];
        const int at = (k + 1 + i) * n + k + 1 + j;
        A[at] = fma(-vi, v[j], fma(-v[i], vj, A[at]));
      }
    }
    __syncthreads();
  }
  for (int i = tid; i < n; i += nthr) d[i] = A[i * n + i];
  if (tid == 0 && n > 1) e[n - 2] = A[(n - 1) * n + n - 2];
  __syncthreads();
  // ---- Gershgorin interval; e2 in v
  if (warp == 0) {
    double lo = 1e300, hi = -1e300;
    for (int i = lane; i < n; i += 32) {
      const double r = (i > 0 ? fabs(e[i - 1]) : 0.0) + (i + 1 < n ? fabs(e[i]) : 0.0);
      lo = fmin(lo, d[i] - r);
      hi = fmax(hi, d[i] + r);
      if (i + 1 < n) v[i] = e[i] * e[i];
    }
    for (int o = 16; o > 0; o >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) { sc[0] = lo; sc[1] = hi; }
  }
  __syncthreads();
  const double nrm = fmax(fabs(sc[0]), fabs(sc[1]));
  if (!(nrm < 1e300)) return false;                  // not finite
  const double eps = 2.2e-16 * fmax(nrm, 1e-290);
  for (int j = warp; j < nc; j += nwarp) {
    double lo = sc[0] - 4.0 * eps, hi = sc[1] + 4.0 * eps;
    for (int pass = 0; pass < 14 && hi - lo > eps; ++pass) {
      const double h = (hi - lo) * (1.0 / 33.0), x = fma(h, (double)(lane + 1), lo);
      const unsigned above = __ballot_sync(0xffffffffu, sturm_count(d, v, n, x) > j);
      const int f = above ? __ffs(above) - 1 : 32;   // first point with more than j eigenvalues below it
      const double nlo = f > 0 ? fma(h, (double)f, lo) : lo;
      hi = f < 32 ? fma(h, (double)(f + 1), lo) : hi;
      lo = nlo;
    }
    if (lane == 0) lam[j] = 0.5 * (lo + hi);
  }
  __syncthreads();
  // ---- inverse iteration, kTriBatch vectors at a time, a thread each; then Gram-Schmidt
  // over all of them; a last iteration and Gram-Schmidt again
  double *u0 = lu, *u1 = u0 + kTriBatch * n, *u2 = u1 + kTriBatch * n, *ml = u2 + kTriBatch * n, *y = ml + kTriBatch * n;
  for (int round = 0; round < 2; ++round) {
    for (int j0 = 0; j0 < nc; j0 += kTriBatch) {
      const int j = j0 + tid;
      if (tid < kTriBatch && j < nc) {
        // T - lambda I = P L U: u0 (as reciprocals), u1, u2; ml the multiplier, its row swap in sw
        const double x = lam[j];
        unsigned sw[3] = {0u, 0u, 0u};
        double a = d[0] - x, b = n > 1 ? e[0] : 0.0;
        for (int k = 0; k + 1 < n; ++k) {
          const double c = e[k], dn = d[k + 1] - x, en = k + 2 < n ? e[k + 1] : 0.0;
          double p0 = a, p1 = b, p2 = 0.0, q0 = c, q1 = dn, q2 = en;
          if (fabs(c) > fabs(a)) {
            sw[k >> 5] |= 1u << (k & 31);
            p0 = c; p1 = dn; p2 = en; q0 = a; q1 = b; q2 = 0.0;
          }
          if (fabs(p0) < eps) p0 = p0 < 0.0 ? -eps : eps;
          const double r = 1.0 / p0, f = q0 * r;
          u0[k * kTriBatch + tid] = r;
          u1[k * kTriBatch + tid] = p1;
          u2[k * kTriBatch + tid] = p2;
          ml[k * kTriBatch + tid] = f;
          a = fma(-f, p1, q1);
          b = fma(-f, p2, q2);
        }
        if (fabs(a) < eps) a = a < 0.0 ? -eps : eps;
        u0[(n - 1) * kTriBatch + tid] = 1.0 / a;
        for (int it = 0; it < 2; ++it) {
          if (round == 0 && it == 0) {
            unsigned h = 0x9E3779B1u * (unsigned)(j + 1);
            for (int k = 0; k < n; ++k) {
              h ^= h << 13; h ^= h >> 17; h ^= h << 5;
              y[k * kTriBatch + tid] = (double)(int)h * 0x1p-31;
            }
          } else {
            if (it == 0)
              for (int k = 0; k < n; ++k) y[k * kTriBatch + tid] = Z[j * n + k];
            double t = y[tid];
            for (int k = 0; k + 1 < n; ++k) {        // L
              double s = y[(k + 1) * kTriBatch + tid];
              if ((sw[k >> 5] >> (k & 31)) & 1u) { const double z = t; t = s; s = z; }
              y[k * kTriBatch + tid] = t;
              t = fma(-ml[k * kTriBatch + tid], t, s);
            }
            y[(n - 1) * kTriBatch + tid] = t;
          }
          double z1 = 0.0, z2 = 0.0, top = 0.0;
          for (int k = n - 1; k >= 0; --k) {         // U
            double t = y[k * kTriBatch + tid];
            if (k + 1 < n) t = fma(-u1[k * kTriBatch + tid], z1, t);
            if (k + 2 < n) t = fma(-u2[k * kTriBatch + tid], z2, t);
            t *= u0[k * kTriBatch + tid];
            y[k * kTriBatch + tid] = t;
            z2 = z1;
            z1 = t;
            top = fmax(top, fabs(t));
          }
          const double f = 1.0 / top;
          for (int k = 0; k < n; ++k) y[k * kTriBatch + tid] *= f;
        }
        for (int k = 0; k < n; ++k) Z[j * n + k] = y[k * kTriBatch + tid];
      }
      __syncthreads();
    }
    if (warp == 0) {
      for (int j = 0; j < nc; ++j) {
        double* zj = Z + j * n;
        for (int pass = 0; pass < 2; ++pass) {
          for (int i = 0; i < j; ++i) {
            const double* zi = Z + i * n;
            double s = 0.0;
            for (int k = lane; k < n; k += 32) s = fma(zi[k], zj[k], s);
            s = warp_sum(s);
            for (int k = lane; k < n; k += 32) zj[k] = fma(-s, zi[k], zj[k]);
          }
          double s = 0.0;
          for (int k = lane; k < n; k += 32) s = fma(zj[k], zj[k], s);
          s = 1.0 / sqrt(warp_sum(s));
          for (int k = lane; k < n; k += 32) zj[k] *= s;
        }
      }
    }
    __syncthreads();
  }
  // ---- residuals, then Z <- H_0 .. H_{n-3} Z, a warp per vector
  double bad = 0.0;
  for (int j = warp; j < nc; j += nwarp) {
    double* zj = Z + j * n;
    double s = 0.0;
    for (int k = lane; k < n; k += 32) {
      double r = (d[k] - lam[j]) * zj[k];
      if (k > 0) r = fma(e[k - 1], zj[k - 1], r);
      if (k + 1 < n) r = fma(e[k], zj[k + 1], r);
      s = fma(r, r, s);
    }
    s = warp_sum(s);
    if (!(s <= 1e-26 * nrm * nrm)) bad = 1.0;
    __syncwarp();
    for (int k = n - 3; k >= 0; --k) {
      const int m = n - k - 1;
      double q = 0.0;
      for (int i = lane; i < m; i += 32) q = fma(A[(k + 1 + i) * n + k], zj[k + 1 + i], q);
      q = warp_sum(q) * tau[k];
      for (int i = lane; i < m; i += 32) zj[k + 1 + i] = fma(-q, A[(k + 1 + i) * n + k], zj[k + 1 + i]);
      __syncwarp();
    }
  }
  return __syncthreads_or(bad != 0.0) == 0;
}

// Positive double values order like their bit patterns: atomic max via int64.
__device__ __forceinline__ void atomic_max_pos(double* addr, double v) {
  atomicMax(reinterpret_cast<unsigned long long*>(addr), (unsigned long long)__double_as_longlong(v));
}

}  // namespace msmg
