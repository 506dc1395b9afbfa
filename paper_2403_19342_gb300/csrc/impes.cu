// Two-phase flow by the improved IMPES scheme (Section 6): the pieces that run
// on the GPU around the pressure solve.
//
// Fluid model (Section 6): S* = (S - s_wc) / (1 - s_wc - s_or) clipped to
// [0, 1], relative permeabilities k_rw = S*^2 and k_ro = (1 - S*)^2, total
// mobility lambda = k_rw / mu_w + k_ro / mu_o, water fractional flow
// f_w = (k_rw / mu_w) / lambda.
//
// Pressure step, Eq. (IMP): div(-lambda(S^n) K grad p) = q(p).  Its two-point
// discretisation is the pressure system of this library with the permeability
// lambda(S^n) kappa (face coefficients harmonic averages of it), plus the
// producers' well terms: at a cell a producer crosses, q = W (p_BH - p) with
// W = WI kappa^x lambda, WI the well index.  So the system is (A + W) p = b,
// b = q_inj + W p_BH, W the library's cell term (options.cell_diag).
//
// Saturation sub-steps, Eq. (ES): phi (S^{m+1} - S^m) / dt + div(f_w(S^m) v) =
// q_w with the face flux f_w(S_up) v of the upstream cell (the cell the flow
// leaves) and q_w = q_inj at the injector, f_w(S) W (p_BH - p) at a producer;
// dt = DS_max / max |dS/dt| so that no cell changes by more than DS_max.
#include "msmg_internal.cuh"
#include <cmath>

namespace msmg {

struct Fluid {
  double mu_w, mu_o, s_wc, s_or;
};
__device__ __forceinline__ void fluid_eval(const Fluid& F, double S, double* lam, double* fw) {
  double s = (S - F.s_wc) / (1.0 - F.s_wc - F.s_or);
  s = s < 0.0 ? 0.0 : (s > 1.0 ? 1.0 : s);
  const double mw = s * s / F.mu_w, mo = (1.0 - s) * (1.0 - s) / F.mu_o;
  *lam = mw + mo;
  *fw = mw / (mw + mo);
}

__global__ void k_pressure_terms(int64_t n, Fluid F, const double* __restrict__ S, const double* __restrict__ kappa,
                                 const double* __restrict__ wi, const double* __restrict__ q_inj, double p_bh,
                                 double* __restrict__ kappa_eff, double* __restrict__ w, double* __restrict__ b) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double lam, fw;
  fluid_eval(F, S[i], &lam, &fw);
  for (int d = 0; d < 3; ++d) kappa_eff[(int64_t)d * n + i] = lam * kappa[(int64_t)d * n + i];
  const double wc = wi[i] * kappa[i] * lam;
  w[i] = wc;
  b[i] = q_inj[i] + wc * p_bh;
}

// ------------------------------------------------------------------ saturation sub-steps
// Every kernel here is bound by the FP64 pipe (two lanes per clock and SM: one FP64
// instruction per cell costs 1.9 us on 1.1 M cells, where the 70 bytes per cell, in
// L2, cost about 9), so the sub-step is arranged for few FP64 instructions:
//   * what stays fixed over the sub-steps is formed once per call (k_transport_terms):
//     v_d / h_d, w (p_BH - p) and 1 / phi, so a face costs one FMA and no division;
//   * f_w = s^2 mu_o / (s^2 mu_o + (1 - s)^2 mu_w): one division instead of three;
//   * comparisons (clipping, upstream side, the largest rate) on the integer pipes.
// 24 FP64 instructions per cell and sub-step, the FP64 pipe 81% busy in both kernels:
// 66 us on 60 x 220 x 85 cells, where the divisions in place (three by h_d, one by phi,
// four in the fluid model) and a serial maximum over the CTAs took 318 us.

__device__ __forceinline__ bool finite_bits(double v) {   // on the integer pipes
  return (((uint64_t)__double_as_longlong(v) >> 52) & 0x7ff) != 0x7ff;
}
// a / b by Newton's iteration from an FP32 reciprocal and Markstein's final
// correction (P. Markstein, IBM J. Res. Dev. 34, 1990: with r = a - b q exact in one
// FMA, q + r y rounds to a / b for y close enough to 1 / b): five FP64 instructions;
// the FP32 seed is converted on the integer pipes.  b outside FP32's normal range
// takes the ordinary division.
__device__ __forceinline__ double div_newton(double a, double b) {
  const int e = (int)(((uint64_t)__double_as_longlong(b) >> 52) & 0x7ff);
  if (e < 1023 - 120 || e > 1023 + 120) return a / b;
  const double y0 = f64_of_f32(__frcp_rn(f32_of_f64_rn(b)));
  const double y = fma(y0, fma(-b, y0, 1.0), y0);
  const double q = a * y;
  return fma(fma(-b, q, a), y, q);
}

struct Frac {        // f_w's constants: s* = (S - s_wc) / c, c = 1 - s_wc - s_or, y = 1 / c
  double s_wc, c, y, mu_w, mu_o;
};
__device__ __forceinline__ double frac_flow(const Frac& F, double S) {
  const double d = S - F.s_wc;
  double s = d * F.y;
  if (finite_bits(s)) s = fma(fma(-F.c, s, d), F.y, s);   // (S - s_wc) / c, Markstein's correction
  // clip to [0, 1]; NaN stays NaN
  const long long u = __double_as_longlong(s), one = 0x3ff0000000000000ll, inf = 0x7ff0000000000000ll;
  if (u < 0 && (u & 0x7fffffffffffffffll) <= inf) s = 0.0;
  if (u > one && u <= inf) s = 1.0;
  const double t = 1.0 - s, a = s * s * F.mu_o;
  return div_newton(a, fma(t * t, F.mu_w, a));
}

// The terms that stay fixed over a call's sub-steps: vh[d] = v_d / h_d on interior
// +d faces and 0 on the boundary, wq = w (p_BH - p), rphi = 1 / phi.
__global__ void k_transport_terms(int nx, int ny, int nz, double hx, double hy, double hz,
                                  const double* __restrict__ v, const double* __restrict__ p,
                                  const double* __restrict__ w, double p_bh, const double* __restrict__ phi,
                                  double* __restrict__ vh0, double* __restrict__ vh1, double* __restrict__ vh2,
                                  double* __restrict__ wq, double* __restrict__ rphi) {
  const unsigned n = (unsigned)nx * ny * nz;
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const unsigned row = i / (unsigned)nx;
  const int x = (int)(i - row * nx), y = (int)(row % (unsigned)ny), z = (int)(row / (unsigned)ny);
  vh0[i] = x + 1 < nx ? v[i] / hx : 0.0;
  vh1[i] = y + 1 < ny ? v[(size_t)n + i] / hy : 0.0;
  vh2[i] = z + 1 < nz ? v[2 * (size_t)n + i] / hz : 0.0;
  wq[i] = w[i] * (p_bh - p[i]);
  rphi[i] = 1.0 / phi[i];
}

// S += dt rate of the sub-step before (UPDATE; dt = DS_max / max |dS/dt|, the maximum
// in mx_old as bits), its dt added to sc[1]; then f_w of the new saturation (FRAC);
// mx_new is cleared for the rates that follow.
template <bool UPDATE, bool FRAC>
__global__ void __launch_bounds__(256) k_sat_step(unsigned n, Frac F, double* __restrict__ S,
                                                  const double* __restrict__ rate, double* __restrict__ fw,
                                                  const unsigned long long* mx_old, unsigned long long* mx_new,
                                                  double ds_max, double* sc) {
  __shared__ double s_dt;
  if (threadIdx.x == 0) {
    if (UPDATE) {
      const double m = __longlong_as_double((long long)*mx_old);
      s_dt = m > 0.0 ? ds_max / m : 0.0;
      if (blockIdx.x == 0) sc[1] += s_dt;
    }
    if (FRAC && blockIdx.x == 0) *mx_new = 0ull;
  }
  __syncthreads();
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double Si = S[i];
  if (UPDATE) {
    Si = fma(s_dt, rate[i], Si);
    S[i] = Si;
  }
  if (FRAC) fw[i] = frac_flow(F, Si);
}

// dS/dt of every cell (natural order) and the largest |dS/dt|, as bits, into mx (one
// atomic maximum per CTA: the same result in any order).  A face's water flux is
// f_w vh of the cell the flow leaves.
__global__ void __launch_bounds__(256) k_sat_rate(unsigned n, unsigned nx, unsigned ny, unsigned nz,
                                                  const double* __restrict__ vh0, const double* __restrict__ vh1,
                                                  const double* __restrict__ vh2, const double* __restrict__ wq,
                                                  const double* __restrict__ q_inj, const double* __restrict__ rphi,
                                                  const double* __restrict__ fw, double* __restrict__ rate,
                                                  unsigned long long* mx) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long top = 0ull;
  if (i < n) {
    const unsigned row = i / nx;
    const unsigned x = i - row * nx, y = row % ny, z = row / ny, nxy = nx * ny;
    const double f0 = fw[i];
    double acc = fma(f0, wq[i], q_inj[i]);
    // (a boundary face has vh = 0: its flux is 0 with this cell's f_w)
    const bool hi[3] = {x + 1 < nx, y + 1 < ny, z + 1 < nz}, lo[3] = {x > 0, y > 0, z > 0};
    const unsigned st[3] = {1u, nx, nxy};
    const double* const vh[3] = {vh0, vh1, vh2};
    double vp[3], vm[3], fp[3], fm[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      vp[d] = vh[d][i];
      vm[d] = lo[d] ? vh[d][i - st[d]] : 0.0;
      fp[d] = hi[d] ? fw[i + st[d]] : f0;
      fm[d] = lo[d] ? fw[i - st[d]] : f0;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      // upstream of a +d face is this cell unless vp < 0; of a -d face the neighbour unless vm < 0
      const bool bp = __double_as_longlong(vp[d]) < 0, bm = __double_as_longlong(vm[d]) < 0;
      acc = fma(-(bp ? fp[d] : f0), vp[d], acc);
      acc = fma(bm ? f0 : fm[d], vm[d], acc);
    }
    const double r = acc * rphi[i];
    rate[i] = r;
    const unsigned long long u = (unsigned long long)__double_as_longlong(r) & 0x7fffffffffffffffull;
    if (u <= 0x7ff0000000000000ull) top = u;      // a NaN rate does not set the step
  }
  // largest magnitude: non-negative doubles order like their bit patterns
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_xor_sync(0xffffffffu, top, o);
    top = t > top ? t : top;
  }
  __shared__ unsigned long long sh[8];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = top;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 1; k < 8; ++k) top = sh[k] > top ? sh[k] : top;
    if (top) atomicMax(mx, top);
  }
}

}  // namespace msmg

using namespace msmg;

extern "C" {

int msmg_impes_pressure_terms(int64_t n, const msmg_fluid* fluid, const double* S, const double* kappa,
                              const double* wi, const double* q_inj, double p_bh, double* kappa_eff, double* w,
                              double* b, msmg_stream stream) {
  if (n < 1 || !fluid || !S || !kappa || !wi || !q_inj || !kappa_eff || !w || !b) return MSMG_ERR_INVALID_ARG;
  if (!(fluid->mu_w > 0) || !(fluid->mu_o > 0) || !(fluid->s_wc >= 0) || !(fluid->s_or >= 0) ||
      !(fluid->s_wc + fluid->s_or < 1))
    return MSMG_ERR_INVALID_ARG;
  const Fluid F{fluid->mu_w, fluid->mu_o, fluid->s_wc, fluid->s_or};
  k_pressure_terms<<<(unsigned)((n + 255) / 256), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
      n, F, S, kappa, wi, q_inj, p_bh, kappa_eff, w, b);
  MSMG_CUDA_TRY(cudaGetLastError());
  return 0;
}

int msmg_impes_transport(msmg_ctx* c, const msmg_fluid* fluid, const double* v, const double* p, const double* w,
                         double p_bh, const double* q_inj, const double* phi, double* S, int M, double ds_max,
                         double* dt_host, msmg_stream stream) {
  if (!c || !fluid || !v || !p || !w || !q_inj || !phi || !S || M < 0 || !(ds_max > 0)) return MSMG_ERR_INVALID_ARG;
  if (!(fluid->mu_w > 0) || !(fluid->mu_o > 0) || !(fluid->s_wc >= 0) || !(fluid->s_or >= 0) ||
      !(fluid->s_wc + fluid->s_or < 1))
    return MSMG_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  Frac F{fluid->s_wc, 1.0 - fluid->s_wc - fluid->s_or, 0.0, fluid->mu_w, fluid->mu_o};
  F.y = 1.0 / F.c;
  const unsigned n = (unsigned)c->n;   // at most 2^31 - 1 cells
  // scratch: the solve buffers are free between solves
  const SolveBuffers& B = c->sb;
  double *rate = B.z, *fw = B.q, *vh0 = B.p0, *vh1 = B.p1, *vh2 = B.r, *wq = B.x, *rphi = B.b;
  double* sc = c->dtmp + 12;          // [1] sum of the sub-steps' dt
  unsigned long long* mx = reinterpret_cast<unsigned long long*>(c->dtmp + 14);   // two maxima in turn
  const unsigned grid = (n + 255u) / 256u;
  MSMG_CUDA_TRY(cudaMemsetAsync(sc, 0, 4 * sizeof(double), s));
  if (M > 0) {
    k_transport_terms<<<grid, 256, 0, s>>>(c->grid.nx, c->grid.ny, c->grid.nz, c->grid.hx, c->grid.hy, c->grid.hz, v,
                                           p, w, p_bh, phi, vh0, vh1, vh2, wq, rphi);
    k_sat_step<false, true><<<grid, 256, 0, s>>>(n, F, S, rate, fw, mx + 1, mx, ds_max, sc);
    for (int m = 0; m < M; ++m) {
      k_sat_rate<<<grid, 256, 0, s>>>(n, (unsigned)c->grid.nx, (unsigned)c->grid.ny, (unsigned)c->grid.nz, vh0, vh1,
                                      vh2, wq, q_inj, rphi, fw, rate, mx + (m & 1));
      if (m + 1 < M)
        k_sat_step<true, true><<<grid, 256, 0, s>>>(n, F, S, rate, fw, mx + (m & 1), mx + ((m + 1) & 1), ds_max, sc);
      else
        k_sat_step<true, false><<<grid, 256, 0, s>>>(n, F, S, rate, fw, mx + (m & 1), mx, ds_max, sc);
    }
  }
  MSMG_CUDA_TRY(cudaGetLastError());
  if (dt_host) {
    MSMG_CUDA_TRY(cudaMemcpyAsync(dt_host, sc + 1, sizeof(double), cudaMemcpyDeviceToHost, s));
    MSMG_CUDA_TRY(cudaStreamSynchronize(s));
  }
  return 0;
}

}  // extern "C"
