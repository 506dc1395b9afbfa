// Level-1 local eigensolver for large elements (Eq. (spepb)): Chebyshev-
// filtered subspace iteration (the filtered Rayleigh-Ritz scheme of Zhou,
// Saad, Tiago and Chelikowsky, 2006), one CTA per element, everything in
// shared memory.  The FP64 form iterates in FP64 throughout; the mixed form
// first iterates in FP32 (vectors, filter, orthonormalisation, Rayleigh-Ritz
// projections; only the K x K eigensolve in FP64) to a residual near FP32's
// reach and then polishes the whole block in FP64 to the requested tolerance,
// so the bases it keeps are the FP64 form's to within that tolerance.
//
// The generalised problem A_K phi = lambda S_K phi is solved in its symmetric
// form A~ y = lambda y, A~ = S^{-1/2} A_K S^{-1/2}, phi = S^{-1/2} y.  A~ is the
// element's 7-point operator with diagonal g_c = (sum of in-element face
// coefficients) / s_c and off-diagonals -T / sqrt(s_c s_c').  Its spectrum lies
// in [0, 8] and S^{1/2} 1 spans its kernel exactly, so that vector seeds the
// block and stays in it.
//
// One outer iteration: filter the K-vector block with a Chebyshev polynomial that
// damps [theta_{K-1}, b] (b a Gershgorin bound, theta the current Ritz values);
// Rayleigh-Ritz on the filtered block as it is: G = X^T X and H = X^T A~ X, G's Cholesky
// factor, the K x K eigenproblem of L^-1 H L^-T, one rotation of X that orthonormalises
// and diagonalises at once; stop when the L wanted Ritz pairs have residual
// ||A~ y - theta y||_2 <= tol.  Columns too close to dependent for a Cholesky factor (a
// pivot of the unit-diagonal G below kPivot) are first orthonormalised by two-pass
// Gram-Schmidt.  K - L guard vectors keep the convergence rate set by the gap to
// theta_{K-1}, not by clusters at the L-th eigenvalue.  The degree follows from the
// reduction still needed: m = acosh(residual / tol) / acosh(t_L), 1 / T_m(t_L) being what
// the filter leaves of the unwanted part of the L-th vector, and varies where the residual
// does not fall (an unwanted eigenvalue at an extremum of T_m is not damped at all).
//
// Bound by the FP64 pipe (2 lanes per clock and SM).  Per cell and iteration, K = 10:
// filter 7 K per degree, A~ X 70, G and H 55 each with 14 of reduction, rotation and
// residuals 175.  Up to four cells per thread, so a sum over the element costs a lane's exchange
// tree (block_sums) once per four cells.  With a cell per thread, five shuffle-adds per product and thread, and the
// Gram-Schmidt passes of every iteration, the 4096 elements of a 128^3 lognormal field
// (L = 6, tolerance 1e-8) took 18.7 ms in FP32 and 45.5 ms in FP64; now 6.9 and 13.4.
//
// Starting block: the constant S^{1/2} 1 and separable cosine modes ranked by
// frequency, or, with a learned warm start, the network's guesses for
// eigenvectors 1 .. L-1 in place of the first cosines (the guard vectors stay
// cosines).  The stopping test is the same either way.
//
// One translation unit per arithmetic (eig_chfsi_f32.cu, eig_chfsi_f64.cu) instantiates the
// kernel; eig_chfsi_f64.cu holds the launcher.
#pragma once
#include "msmg_internal.cuh"
#include "reduce.cuh"
#include "linalg_small.cuh"
#include <type_traits>

namespace msmg {

constexpr int kKMax = 16;

// Threads of an element: four cells per thread above 128 cells, one below.  Four cells
// share a lane's reduction work; a small element takes a cell per thread all the same,
// because its slowest elements set the time (a warp issues one FP64 instruction per 64
// clocks: with all of an 80-cell element in one warp an iteration took 410 us alone).
__host__ __device__ constexpr int eig_cpt(int nb) { return nb > 128 ? 4 : 1; }
constexpr int kEigThreads = 128;
constexpr int kScrPer = 64;             // reduced values per warp in the exchange area

// One exchange step of block_sums: N values per lane become (N + 1) / 2, then the next step
// with half the lane distance D.
template <int N, int D, int NV, typename A>
__device__ __forceinline__ void exchange_sums(A (&v)[NV], int lane) {
  if constexpr (D > 0) {
    constexpr int h = (N + 1) / 2;
    const bool up = lane & D;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const A lo = v[k], hi = k + h < N ? v[k + h < NV ? k + h : 0] : (A)0;
      v[k] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, D);
    }
    exchange_sums<h, D / 2, NV>(v, lane);
  }
}
// values a lane holds after the five steps, and which value slot k of a lane is (-1: none)
__host__ __device__ constexpr int exchange_left(int n) {
  for (int d = 16; d > 0; d /= 2) n = (n + 1) / 2;
  return n;
}
template <int N, int D>
__device__ __forceinline__ int exchange_index(int k, int lane) {
  if constexpr (D == 0) {
    return k;
  } else {
    constexpr int h = (N + 1) / 2;
    const int below = exchange_index<h, D / 2>(k, lane);
    const int idx = below < 0 ? -1 : below + ((lane & D) ? h : 0);
    return idx < N ? idx : -1;
  }
}
// Sums over the CTA of NV (<= 64) values per thread, to out[0 .. NV) (shared, FP64; valid
// for every thread on return).  Within a warp the values are exchanged in halves: a lane
// keeps one half of its values and hands the other to its partner, so NV values cost about
// NV additions per lane instead of 5 NV.
template <int NV, typename A>
__device__ __forceinline__ void block_sums(A (&v)[NV], double* out, double* scr) {
  static_assert(NV <= kScrPer, "one slot per value");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  exchange_sums<NV, 16, NV>(v, lane);
#pragma unroll
  for (int k = 0; k < exchange_left(NV); ++k) {
    const int idx = exchange_index<NV, 16>(k, lane);
    if (idx >= 0) scr[warp * kScrPer + idx] = (double)v[k];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < NV; i += blockDim.x) {
    double acc = scr[i];
    for (int w = 1; w < nwarp; ++w) acc += scr[w * kScrPer + i];
    out[i] = acc;
  }
  __syncthreads();
}

// Rows I0 .. I0 + 3 (within KT) of the symmetric X^T B, both triangles of O (K x K).
template <typename R, int KT, int I0>
__device__ __noinline__ void gram_pass(const R* X, const R* B, double* O, int K, int nb, double* sums, double* scr) {
  if (I0 >= K) return;
  constexpr int NR = KT - I0 < 4 ? KT - I0 : 4;
  constexpr int NV = NR * (KT - I0) - NR * (NR - 1) / 2;     // upper-triangle entries of these rows
  R acc[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) acc[k] = (R)0;
  for (int c = threadIdx.x; c < nb; c += blockDim.x) {
    R a[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) a[r] = I0 + r < K ? X[(I0 + r) * nb + c] : (R)0;
#pragma unroll
    for (int j = I0; j < KT; ++j) {
      if (j >= K) continue;
      const R b = B[j * nb + c];
#pragma unroll
      for (int r = 0; r < NR; ++r)
        if (j >= I0 + r) {
          const int at = r * (KT - I0) - r * (r - 1) / 2 + j - I0 - r;
          acc[at] = fma(a[r], b, acc[at]);
        }
    }
  }
  block_sums<NV>(acc, sums, scr);
  for (int o = threadIdx.x; o < NR * KT; o += blockDim.x) {
    const int r = o / KT, j = o % KT, ii = I0 + r;
    if (ii < K && j >= ii && j < K) {
      const double v = sums[r * (KT - I0) - r * (r - 1) / 2 + j - ii];
      O[ii * K + j] = v;
      O[j * K + ii] = v;
    }
  }
  __syncthreads();
}

// The rotation (c, s) that annihilates a_pq of a symmetric 2 x 2 block.  The tangent is
// formed in FP32 (it only steers the iteration: a rotation by a slightly other angle leaves
// 1e-7 of a_pq for the next sweep); c = 1 / sqrt(1 + t^2) by Newton's iteration in FP64, so
// that c^2 + s^2 = 1 to FP64 rounding.  A chain of 11 FP64 instructions instead of two
// divisions and two square roots (about 2500 clocks of latency each round).
__device__ __forceinline__ void jacobi_rotation(double app, double aqq, double apq, double* c, double* s) {
  const float off = f32_of_f64_rn(apq), dif = f32_of_f64_rn(aqq - app);
  *c = 1.0;
  *s = 0.0;
  if (off == 0.f) return;
  const float th = dif / (2.f * off);
  const float tf = copysignf(1.f, th) / (fabsf(th) + sqrtf(fmaf(th, th, 1.f)));
  if (!(fabsf(tf) > 0.f)) return;
  const double t = f64_of_f32(tf), y = fma(t, t, 1.0);
  double r = f64_of_f32(rsqrtf(fmaf(tf, tf, 1.f)));
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double e = fma(-y * r, r, 1.0);
    r = fma(0.5 * r, e, r);
  }
  *c = r;
  *s = t * r;
}

// Cyclic Jacobi (round-robin pairs) on the n x n symmetric A (n <= 16) by one warp; V
// receives the eigenvectors (columns), A's diagonal the eigenvalues.  Half-warps take the
// pairs of a round in turn, a lane per column.
static __device__ __noinline__ void warp_jacobi(double* A, double* V, int n, double* cs, int* pq, int max_sweeps, double rtol) {
  const int lane = threadIdx.x & 31, col = lane & 15, par = lane >> 4;
  const int npad = n + (n & 1), half = npad / 2;
  const bool in = col < n;
  for (int r = par; r < n; r += 2)
    if (in) V[r * n + col] = r == col ? 1.0 : 0.0;
  __syncwarp();
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    double off = 0.0, all = 0.0;
    for (int r = par; r < n; r += 2) {
      const double a = in ? A[r * n + col] : 0.0;
      all = fma(a, a, all);
      if (r != col) off = fma(a, a, off);
    }
    off = warp_sum(off);
    all = warp_sum(all);
    if (off <= rtol * rtol * all) break;
    for (int r = 0; r < npad - 1; ++r) {
      if (lane < half) {
        // pair i of the round: (0, 1 + (npad - 2 + r) mod (npad - 1)), then folding inwards
        int pa = 0, pb = npad - 2 - lane + r;
        if (lane > 0) pa = 1 + (lane - 1 + r >= npad - 1 ? lane - 1 + r - (npad - 1) : lane - 1 + r);
        pb = 1 + (pb >= npad - 1 ? pb - (npad - 1) : pb);
        const int p = pa < pb ? pa : pb, q = pa < pb ? pb : pa;
        double c = 1.0, s = 0.0;
        if (q < n) jacobi_rotation(A[p * n + p], A[q * n + q], A[p * n + q], &c, &s);
        cs[2 * lane] = c;
        cs[2 * lane + 1] = s;
        pq[lane] = p | (q << 8);
      }
      __syncwarp();
      for (int i = par; i < half; i += 2) {                  // rows
        const int p = pq[i] & 255, q = pq[i] >> 8;
        if (q >= n || !in) continue;
        const double c = cs[2 * i], s = cs[2 * i + 1];
        const double ap = A[p * n + col], aq = A[q * n + col];
        A[p * n + col] = c * ap - s * aq;
        A[q * n + col] = s * ap + c * aq;
      }
      __syncwarp();
      for (int i = par; i < half; i += 2) {                  // columns of A and V
        const int p = pq[i] & 255, q = pq[i] >> 8;
        if (q >= n || !in) continue;
        const double c = cs[2 * i], s = cs[2 * i + 1];
        const double ap = A[col * n + p], aq = A[col * n + q];
        A[col * n + p] = c * ap - s * aq;
        A[col * n + q] = s * ap + c * aq;
        const double vp = V[col * n + p], vq = V[col * n + q];
        V[col * n + p] = c * vp - s * vq;
        V[col * n + q] = s * vp + c * vq;
      }
      __syncwarp();
    }
  }
}

// The K x K part of a Rayleigh-Ritz step, one warp: G (Gram matrix) and H (projected
// operator) in, the rotation Q (K x K, columns in ascending Ritz order) and theta out.
// Returns false, with nothing changed that the caller needs, when a pivot of the
// unit-diagonal G's Cholesky factor is below piv_min.  W1, W2: K x K scratch.
static __device__ __noinline__ bool ritz_warp(double* G, double* H, double* W1, double* W2, double* Q, double* theta, double* dsc,
                          double* cs, int* pq, int K, double piv_min) {
  const int lane = threadIdx.x & 31, col = lane & 15, par = lane >> 4;
  if (lane < K) dsc[lane] = 1.0 / sqrt(G[lane * K + lane]);
  __syncwarp();
  bool ok = true;
  for (int i = lane; i < K; i += 32) ok = ok && dsc[i] < 1e150 && dsc[i] > 0.0;
  if (!__all_sync(0xffffffffu, ok)) return false;
  if (col < K)
    for (int r = par; r < K; r += 2) {
      const double f = dsc[r] * dsc[col];
      G[r * K + col] *= f;
      H[r * K + col] *= f;
    }
  __syncwarp();
  for (int k = 0; k < K; ++k) {                       // G = C C^T, C in the lower triangle
    const double piv = G[k * K + k];
    if (!(piv >= piv_min)) return false;
    const double d = 1.0 / sqrt(piv);                 // the factor keeps 1 / c_kk on its diagonal
    __syncwarp();
    if (lane == k) G[k * K + k] = d;
    if (lane > k && lane < K) G[lane * K + k] *= d;
    __syncwarp();
    if (col > k && col < K)
      for (int r = k + 1 + par; r < K; r += 2)
        if (col <= r) G[r * K + col] = fma(-G[r * K + k], G[col * K + k], G[r * K + col]);
    __syncwarp();
  }
  // W1 = C^-1 H, then W2 = W1 C^-T (a lane per column, then per row), symmetrised
  if (lane < K)
    for (int r = 0; r < K; ++r) {
      double v = H[r * K + lane];
      for (int c = 0; c < r; ++c) v = fma(-G[r * K + c], W1[c * K + lane], v);
      W1[r * K + lane] = v * G[r * K + r];
    }
  __syncwarp();
  if (lane < K)
    for (int c = 0; c < K; ++c) {
      double v = W1[lane * K + c];
      for (int j = 0; j < c; ++j) v = fma(-G[c * K + j], W2[lane * K + j], v);
      W2[lane * K + c] = v * G[c * K + c];
    }
  __syncwarp();
  if (col < K)
    for (int r = par; r < K; r += 2) H[r * K + col] = 0.5 * (W2[r * K + col] + W2[col * K + r]);
  __syncwarp();
  warp_jacobi(H, W1, K, cs, pq, 30, 1e-15);
  // ranks (stable, NaN last), then Q = D C^-T V in Ritz order: a lane per column
  if (lane < K) {
    const double di = sort_key(H[lane * K + lane]);
    int rank = 0;
    for (int j = 0; j < K; ++j) {
      const double dj = sort_key(H[j * K + j]);
      rank += (dj < di) || (dj == di && j < lane);
    }
    theta[rank] = H[lane * K + lane];
    for (int r = K - 1; r >= 0; --r) {
      double v = W1[r * K + lane];
      for (int c = r + 1; c < K; ++c) v = fma(-G[c * K + r], W2[c * K + lane], v);
      v *= G[r * K + r];
      W2[r * K + lane] = v;                           // the solution before scaling
      Q[r * K + rank] = v * dsc[r];
    }
  }
  __syncwarp();
  return true;
}

__device__ __forceinline__ double hash_unit(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t h = a * 0x9E3779B1u ^ (b + 0x7F4A7C15u) * 0x85EBCA77u ^ (c + 0x165667B1u) * 0xC2B2AE3Du;
  h ^= h >> 15; h *= 0x2C1B3C6Du; h ^= h >> 12; h *= 0x297A2D39u; h ^= h >> 15;
  return (double)h * (1.0 / 4294967296.0) - 0.5;
}

// Two-pass Gram-Schmidt of the block's columns (nearly dependent ones), a collapsed column
// reseeded from its hash.  Each thread works on its own cells.
template <typename R>
__device__ __noinline__ void gram_schmidt(R* X, int K, int nb, const double* S, int it, double* sums, double* scr) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  for (int j = 0; j < K; ++j) {
    R* xj = X + (size_t)j * nb;
    for (int tries = 0; tries < 3; ++tries) {
      for (int pass = 0; pass < 2 && j > 0; ++pass) {
        R v[kKMax];
#pragma unroll
        for (int i = 0; i < kKMax; ++i) {
          v[i] = (R)0;
          if (i < j)
            for (int c = tid; c < nb; c += nthr) v[i] = fma(X[i * nb + c], xj[c], v[i]);
        }
        block_sums<kKMax>(v, sums, scr);
        for (int c = tid; c < nb; c += nthr) {
          R x = xj[c];
          for (int i = 0; i < j; ++i) x = fma(-(R)sums[i], X[i * nb + c], x);
          xj[c] = x;
        }
        __syncthreads();
      }
      R v[1] = {(R)0};
      for (int c = tid; c < nb; c += nthr) v[0] = fma(xj[c], xj[c], v[0]);
      block_sums<1>(v, sums, scr);
      const double nrm2 = sums[0];
      __syncthreads();
      if (nrm2 > (sizeof(R) == 4 ? 1e-12 : 1e-24)) {
        const R f = (R)(1.0 / sqrt(nrm2));
        for (int c = tid; c < nb; c += nthr) xj[c] *= f;
        __syncthreads();
        break;
      }
      for (int c = tid; c < nb; c += nthr)
        xj[c] = (R)(sqrt(S[c]) * hash_unit((uint32_t)c, (uint32_t)j, (uint32_t)(it * 4 + tries)));
      __syncthreads();
    }
  }
}

// Shared memory: (4 + 2K) nb values of R, then the FP64 Rayleigh-Ritz work.
__host__ __device__ inline size_t chfsi_r_bytes(int nb, int K, size_t rsize) {
  return ((size_t)(4 + 2 * K) * nb * rsize + 15) / 16 * 16;
}
__host__ __device__ inline int chfsi_threads(int nb) {
  return ((nb + eig_cpt(nb) - 1) / eig_cpt(nb) + 31) / 32 * 32;
}
__host__ __device__ inline size_t chfsi_smem(int nb, int K, size_t rsize) {
  return chfsi_r_bytes(nb, K, rsize) +
         ((size_t)5 * K * K + 3 * kKMax + 2 * kKMax + kScrPer * (chfsi_threads(nb) / 32) + 64 + 8 + kKMax * kKMax) *
             sizeof(double) +
         (size_t)(4 * kKMax + 2) * sizeof(int) + 64;
}

// R: arithmetic of the filter, orthonormalisation and residuals (FP64, or FP32
// for the first phase of the mixed form); the K x K Rayleigh-Ritz eigensolve is
// FP64 either way.
//   guess, guess_vecs   starting vectors (symmetric form, FP32): guess_vecs == L - 1
//                       fills slots 1 .. L-1 (learned warm start), == K fills every slot
//                       (the block a first phase left), 0: none
//   block_out           first phase: the K vectors of the final block (symmetric form,
//                       FP32) are written here and Phi, lam and the convergence flag
//                       are left to the second phase
//   kCpt                cells per thread (eig_cpt)
//   KT                  K rounded up to 8, 12 or 16 (register arrays; columns beyond K are skipped)
template <typename R, int KT, int kCpt>
__global__ void __launch_bounds__(kEigThreads) k_eig_l1_chfsi(const double* __restrict__ T, const double* __restrict__ S,
                                                      int64_t n, int bx, int by, int bz, int64_t m, int L, int K,
                                                      int max_iter, double tol,
                                                      const float* __restrict__ guess, int guess_vecs,
                                                      float* __restrict__ block_out, double* __restrict__ Phi,
                                                      double* __restrict__ lam, double* stats, int* flags,
                                                      const double* __restrict__ Wd) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int nb = bx * by * bz, bxy = bx * by;
  R* g = reinterpret_cast<R*>(smraw);
  R* wx = g + nb;
  R* wy = wx + nb;
  R* wz = wy + nb;
  R* X = wz + nb;                    // [K][nb]
  R* Y = X + K * nb;                 // [K][nb]
  double* G = reinterpret_cast<double*>(smraw + chfsi_r_bytes(nb, K, sizeof(R)));   // [K][K]
  double* H = G + K * K;
  double* W1 = H + K * K;
  double* W2 = W1 + K * K;
  double* Q = W2 + K * K;
  double* theta = Q + K * K;         // [kKMax]
  double* dsc = theta + kKMax;       // [kKMax]
  double* cs = dsc + kKMax;          // [kKMax] + [2 kKMax]
  double* scr = cs + 3 * kKMax;      // [warps][kScrPer]
  double* sums = scr + kScrPer * (blockDim.x / 32);   // [64]
  double* misc = sums + 64;          // [8]
  R* Qr = reinterpret_cast<R*>(misc + 8);             // [K][K] in R
  int* modes = reinterpret_cast<int*>(misc + 8 + kKMax * kKMax);   // [K][3]
  int* pq = modes + 3 * kKMax;                        // [kKMax] pairs of a Jacobi round
  constexpr double kPivot = sizeof(R) == 4 ? 3e-3 : 1e-3;

  const int64_t e = blockIdx.x;
  const int tid = threadIdx.x, nthr = blockDim.x;
  const double* Te = T + e * nb;
  // the thread's cells; a missing neighbour is the cell itself with coefficient 0
  int cell[kCpt], off[kCpt][6];
  bool act[kCpt], has[kCpt][6];
  // 1 / sqrt(s) staged in the (not yet used) Y, on an 8-byte boundary: K >= 5 vectors of R
  // hold nb doubles
  double* isq_s = reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(Y) + 7) & ~uintptr_t(7));
#pragma unroll
  for (int i = 0; i < kCpt; ++i) {
    const int c = tid + nthr * i;
    act[i] = c < nb;
    cell[i] = act[i] ? c : 0;
    const int lx = cell[i] % bx, ly = (cell[i] / bx) % by, lz = cell[i] / bxy;
    const bool h[6] = {lx > 0, lx + 1 < bx, ly > 0, ly + 1 < by, lz > 0, lz + 1 < bz};
    const int st[6] = {-1, 1, -bx, bx, -bxy, bxy};
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      has[i][f] = act[i] && h[f];
      off[i][f] = has[i][f] ? cell[i] + st[f] : cell[i];
    }
    if (act[i]) isq_s[c] = 1.0 / sqrt(S[e * nb + c]);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kCpt; ++i) {
    if (!act[i]) continue;
    const int c = cell[i];
    const double isq = isq_s[c];
    double diag = 0.0, w[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (has[i][2 * d + 1]) { const double t = Te[d * n + c]; diag += t; w[d] = t * isq * isq_s[off[i][2 * d + 1]]; }
      if (has[i][2 * d]) diag += Te[d * n + off[i][2 * d]];
    }
    if (Wd) diag += Wd[e * nb + c];   // cell term (wells), added to the left-hand form (Section 6)
    g[c] = (R)(diag * isq * isq);
    wx[c] = (R)w[0]; wy[c] = (R)w[1]; wz[c] = (R)w[2];
  }
  __syncthreads();                    // isq_s (in Y) is free from here
  // the cell's row of A~: diagonal, then the negated couplings to the six neighbours
  auto row = [&](int i, R (&a)[7], R scale, R shift) {
    const int c = cell[i];
    const R* const w[3] = {wx, wy, wz};
    a[0] = act[i] ? scale * (g[c] - shift) : (R)0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      a[1 + 2 * d] = has[i][2 * d] ? -scale * w[d][off[i][2 * d]] : (R)0;
      a[2 + 2 * d] = has[i][2 * d + 1] ? -scale * w[d][c] : (R)0;
    }
  };
  auto apply = [&](int i, const R (&a)[7], const R* v, R acc) {
    acc = fma(a[0], v[cell[i]], acc);
#pragma unroll
    for (int f = 0; f < 6; ++f) acc = fma(a[1 + f], v[off[i][f]], acc);
    return acc;
  };
  const bool all_given = guess && guess_vecs == K;
  if (!all_given) {
    // starting modes: separable cosines ranked by sum (k_d / b_d)^2 (mode 0 = constant)
    const int cx = bx < 4 ? bx : 4, cy = by < 4 ? by : 4, cz = bz < 4 ? bz : 4;
    const int ncand = cx * cy * cz;
    for (int c = tid; c < ncand; c += nthr) {
      const int kx = c % cx, ky = (c / cx) % cy, kz = c / (cx * cy);
      const double key = (double)(kx * kx) / (bx * bx) + (double)(ky * ky) / (by * by) + (double)(kz * kz) / (bz * bz);
      int rank = 0;
      for (int j = 0; j < ncand; ++j) {
        const int jx = j % cx, jy = (j / cx) % cy, jz = j / (cx * cy);
        const double kj = (double)(jx * jx) / (bx * bx) + (double)(jy * jy) / (by * by) + (double)(jz * jz) / (bz * bz);
        rank += (kj < key) || (kj == key && j < c);
      }
      if (rank < K) { modes[3 * rank] = kx; modes[3 * rank + 1] = ky; modes[3 * rank + 2] = kz; }
    }
    // cosine tables [4][b] per direction, in Y (4 (bx + by + bz) <= K nb values)
    const double PI = 3.141592653589793238462643383279502884;
    const int len = bx + by + bz;
    for (int i = tid; i < 4 * len; i += nthr) {
      const int k = i / len, r = i % len;
      const int b = r < bx ? bx : (r < bx + by ? by : bz), l = r < bx ? r : (r < bx + by ? r - bx : r - bx - by);
      Y[i] = (R)cos(PI * k * (l + 0.5) / b);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kCpt; ++i) {
      if (!act[i]) continue;
      const int c = cell[i], lx = c % bx, ly = (c / bx) % by, lz = c / bxy;
      const R sq = (R)sqrt(S[e * nb + c]);
      for (int q = 0; q < K; ++q)
        X[q * nb + c] = sq * (Y[modes[3 * q] * len + lx] * Y[modes[3 * q + 1] * len + bx + ly] *
                              Y[modes[3 * q + 2] * len + bx + by + lz]);
    }
  }
  if (guess) {
#pragma unroll
    for (int i = 0; i < kCpt; ++i) {
      if (!act[i]) continue;
      for (int q = 0; q < K; ++q) {
        if (!((guess_vecs == K) || (guess_vecs == L - 1 && q >= 1 && q < L))) continue;
        const int slot = guess_vecs == K ? q : q - 1;
        X[q * nb + cell[i]] = (R)guess[((size_t)e * guess_vecs + slot) * nb + cell[i]];
      }
    }
  }
  // Gershgorin upper bound of the spectrum
  {
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < kCpt; ++i) {
      R a[7];
      row(i, a, (R)1, (R)0);
      double r = (double)a[0];
#pragma unroll
      for (int f = 1; f < 7; ++f) r -= (double)a[f];
      t = fmax(t, r);
    }
    for (int o = 16; o > 0; o >>= 1) t = fmax(t, __shfl_xor_sync(0xffffffffu, t, o));
    if ((tid & 31) == 0) scr[tid >> 5] = t;
    __syncthreads();
    if (tid == 0) {
      double mx = 0.0;
      for (int w = 0; w < nthr / 32; ++w) mx = fmax(mx, scr[w]);
      misc[0] = mx;
    }
    __syncthreads();
  }
  const double bup = misc[0];

  int it = 0, stall = 0, slow = 0;
  double rmax = 0.0, rbest = 1e300, rprev = 1e300;
  for (;; ++it) {
    for (int attempt = 0; attempt < 2; ++attempt) {
      // ---- Y = A~ X
#pragma unroll
      for (int i = 0; i < kCpt; ++i) {
        R a[7];
        row(i, a, (R)1, (R)0);
        if (act[i])
          for (int q = 0; q < K; ++q) Y[q * nb + cell[i]] = apply(i, a, X + q * nb, (R)0);
      }
      // ---- G = X^T X, H = X^T Y: four rows of the upper triangle per pass
      gram_pass<R, KT, 0>(X, X, G, K, nb, sums, scr);
      gram_pass<R, KT, 0>(X, Y, H, K, nb, sums, scr);
      gram_pass<R, KT, 4>(X, X, G, K, nb, sums, scr);
      gram_pass<R, KT, 4>(X, Y, H, K, nb, sums, scr);
      if constexpr (KT > 8) {
        gram_pass<R, KT, 8>(X, X, G, K, nb, sums, scr);
        gram_pass<R, KT, 8>(X, Y, H, K, nb, sums, scr);
      }
      if constexpr (KT > 12) {
        gram_pass<R, KT, 12>(X, X, G, K, nb, sums, scr);
        gram_pass<R, KT, 12>(X, Y, H, K, nb, sums, scr);
      }
      // ---- K x K
      if (tid < 32) {
        const bool ok = ritz_warp(G, H, W1, W2, Q, theta, dsc, cs, pq, K, attempt == 0 ? kPivot : 0.0);
        if (tid == 0) misc[1] = ok ? 1.0 : 0.0;
        if (ok)
          for (int t = tid; t < K * K; t += 32) Qr[t] = (R)Q[t];
      }
      __syncthreads();
      const bool ok = misc[1] != 0.0;
      __syncthreads();
      if (ok || attempt == 1) break;
      gram_schmidt(X, K, nb, S + e * nb, it, sums, scr);
    }
    // ---- X <- X Q, and the residuals Y q_j - theta_j x_j of the wanted pairs (each
    // thread's own cells only)
    R res[kKMax];
#pragma unroll
    for (int j = 0; j < kKMax; ++j) res[j] = (R)0;
    for (int i = 0; i < kCpt; ++i) {
      const int c = tid + nthr * i;
      if (c >= nb) break;
      R v[KT];
#pragma unroll
      for (int q = 0; q < KT; ++q) v[q] = q < K ? X[q * nb + c] : (R)0;
      for (int j = 0; j < K; ++j) {
        R acc = (R)0;
#pragma unroll
        for (int q = 0; q < KT; ++q)
          if (q < K) acc = fma(v[q], Qr[q * K + j], acc);
        X[j * nb + c] = acc;
      }
#pragma unroll
      for (int q = 0; q < KT; ++q) v[q] = q < K ? Y[q * nb + c] : (R)0;
#pragma unroll
      for (int j = 0; j < kKMax; ++j) {
        if (j >= L) continue;
        R acc = (R)0;
#pragma unroll
        for (int q = 0; q < KT; ++q)
          if (q < K) acc = fma(v[q], Qr[q * K + j], acc);
        acc = fma(-(R)theta[j], X[j * nb + c], acc);
        res[j] = fma(acc, acc, res[j]);
      }
    }
    block_sums<kKMax>(res, sums, scr);
    rmax = 0.0;
    for (int j = 0; j < L; ++j) rmax = fmax(rmax, sums[j] >= 0.0 ? sqrt(sums[j]) : INFINITY);   // (a NaN is not converged)
    if (rmax <= tol || it >= max_iter) break;
    // a first phase stops where its arithmetic stops making progress (three
    // iterations without a 10% gain): the second phase takes over from there
    if (block_out) {
      stall = rmax < 0.9 * rbest ? 0 : stall + 1;
      rbest = fmin(rbest, rmax);
      if (stall >= 3) break;
    }
    // ---- Chebyshev filter on [a, bup]: T_0 = X, T_1 = t(A~) X, T_{j+1} = 2 t(A~) T_j - T_{j-1},
    // t(x) = (x - c) / e; the rows of 2 t(A~) are formed once, so a degree costs seven FMAs.
    // Degree: what the L-th pair still needs, kept where T_m(t_0) / T_m(t_L) (digits the
    // wanted vectors lose to the constant) stays moderate; ten where that says less.
    double a0 = theta[K - 1];
    if (!(a0 < 0.95 * bup)) a0 = 0.5 * bup;
    const double c0 = 0.5 * (a0 + bup), e0 = 0.5 * (bup - a0);
    if (tid == 0) {
      int deg = 10;
      const double tl = (c0 - theta[L - 1]) / e0, t0 = c0 / e0;
      if (tl > 1.0 && t0 >= tl) {
        const double al = acosh(tl), am = acosh(t0), need = log(6.0 * fmax(rmax / tol, 1.0));
        const double top = it == 0 && !all_given ? 12.0 : 24.0, keep = (sizeof(R) == 4 ? 4.6 : 7.0) / fmax(am - al, 1e-9);
        const double d = fmin(ceil(need / al), fmin(top, fmax(keep, 10.0)));
        deg = d >= 4.0 ? (int)d : 4;
      }
      // Where an iteration leaves more than half of the residual, every second one takes
      // 1, 3 or 5 degrees less.  On a cluster at the cutoff the interval and so the degree
      // settle, and an unwanted eigenvalue inside the interval at an extremum of that T_m
      // keeps its part of the block from one iteration to the next: a four-layer element
      // below a channel of 4.7e7 (L = 12) took 260 iterations, 1000 and more from some
      // starting blocks; with the degree varied 16 and 61.  Elements without such a
      // cluster halve their residual every time and are not touched.
      if (rmax > 0.5 * rprev && (++slow & 1)) deg = deg - slow % 6 > 4 ? deg - slow % 6 : 4;
      rprev = rmax;
      misc[2] = (double)deg;
    }
    __syncthreads();
    const int mdeg = (int)misc[2];
    R rw[kCpt][7];
#pragma unroll
    for (int i = 0; i < kCpt; ++i) row(i, rw[i], (R)(2.0 / e0), (R)c0);
    R* Yc = Y;   // current  (degree j)
    R* Xp = X;   // previous (degree j-1)
#pragma unroll
    for (int i = 0; i < kCpt; ++i)
      if (act[i])
        for (int q = 0; q < K; ++q) Yc[q * nb + cell[i]] = (R)0.5 * apply(i, rw[i], Xp + q * nb, (R)0);
    __syncthreads();
    for (int step = 2; step <= mdeg; ++step) {
      for (int q = 0; q < K; ++q) {
#pragma unroll
        for (int i = 0; i < kCpt; ++i)
          if (act[i]) Xp[q * nb + cell[i]] = apply(i, rw[i], Yc + q * nb, -Xp[q * nb + cell[i]]);
      }
      __syncthreads();
      R* t = Yc; Yc = Xp; Xp = t;
    }
    X = Yc;
    Y = Xp;
  }
  if (block_out) {
    // first phase: hand the whole block to the second
#pragma unroll
    for (int i = 0; i < kCpt; ++i)
      if (act[i])
        for (int q = 0; q < K; ++q) block_out[((size_t)e * K + q) * nb + cell[i]] = (float)X[q * nb + cell[i]];
    if (tid == 0) {
      atomicMax(&flags[3], it);
      atomicAdd(&flags[4], it);
    }
    return;
  }
  // ---- output: Phi = S^{-1/2} y for the L smallest
#pragma unroll
  for (int i = 0; i < kCpt; ++i) {
    if (!act[i]) continue;
    const double isq = 1.0 / sqrt(S[e * nb + cell[i]]);
    for (int k = 0; k < L; ++k) Phi[(e * L + k) * nb + cell[i]] = (double)X[k * nb + cell[i]] * isq;
  }
  if (tid < L) lam[e * L + tid] = theta[tid];
  if (tid == 0) {
    atomic_max_pos(&stats[0], rmax);
    atomicMax(&flags[3], it);
    atomicAdd(&flags[4], it);
    if (!(rmax <= tol)) atomicExch(&flags[2], 1);
  }
}

// One phase over every element of the context (R: its arithmetic).  gs / gv: starting vectors
// and how many per element (0: none); out: the block a first phase hands over, or null.
struct EigPhase {
  int L, K, max_iter;
  double tol;
  const float* guess;
  int guess_vecs;
  float* block_out;
};
template <typename R>
void launch_eig_phase(msmg_ctx* c, const EigPhase& p, cudaStream_t s) {
  const FineLevel& f = c->fine;
  auto run = [&](auto kt, auto ct) {
    constexpr int KT = decltype(kt)::value, CPT = decltype(ct)::value;
    const size_t sm = chfsi_smem(f.nb, p.K, sizeof(R));
    smem_at_least(k_eig_l1_chfsi<R, KT, CPT>, sm);
    k_eig_l1_chfsi<R, KT, CPT><<<(unsigned)f.m, (unsigned)chfsi_threads(f.nb), sm, s>>>(
        f.T, f.S, c->n, f.bx, f.by, f.bz, f.m, p.L, p.K, p.max_iter, p.tol, p.guess, p.guess_vecs, p.block_out,
        p.block_out ? nullptr : f.Phi, p.block_out ? nullptr : f.lam, c->dtmp, c->flags, f.Wd);
  };
  auto with_c = [&](auto kt) {
    if (eig_cpt(f.nb) == 4) run(kt, std::integral_constant<int, 4>{});
    else run(kt, std::integral_constant<int, 1>{});
  };
  if (p.K <= 8) with_c(std::integral_constant<int, 8>{});
  else if (p.K <= 12) with_c(std::integral_constant<int, 12>{});
  else with_c(std::integral_constant<int, 16>{});
}

}  // namespace msmg
