// The FP64 phase of the level-1 subspace eigensolve (eig_chfsi.cuh) and its launcher.
#include "eig_chfsi.cuh"

namespace msmg {

extern template void launch_eig_phase<float>(msmg_ctx*, const EigPhase&, cudaStream_t);

// Mixed form: a first FP32 phase to residual kMixedPhase1Tol (on the symmetric
// form, whose spectrum lies in [0, 8]: FP32 resolves residuals down to ~1e-6),
// then an FP64 phase from that block to eig_tol.  The FP64 form runs the FP64
// phase alone.  block is scratch for the FP32 block (m K nb floats) or null.
constexpr double kMixedPhase1Tol = 2e-5;

int launch_level1_chfsi(msmg_ctx* c, cudaStream_t s, const float* guess, float* block) {
  FineLevel& f = c->fine;
  const int L = f.L;
  int guard = L / 2 > 4 ? L / 2 : 4;
  int K = L + guard;
  if (K > kKMax) K = kKMax;
  if (K > f.nb) K = f.nb;
  const int cx = f.bx < 4 ? f.bx : 4, cy = f.by < 4 ? f.by : 4, cz = f.bz < 4 ? f.bz : 4;
  if (L >= kKMax || K > cx * cy * cz || f.nb > 512) return MSMG_ERR_UNSUPPORTED;
  // the cap only matters for rare elements with clustered eigenvalues at the
  // cutoff: on 512^3 layered channels (262,144 elements, L = 12) one element of
  // the mixed form needs ~500 iterations; an element that iterates longer costs
  // its own CTA's time, not the launch's
  const int max_iter = c->opts.eig_max_iter > 0 ? c->opts.eig_max_iter : 1000;
  const double tol = c->opts.eig_tol > 0 ? c->opts.eig_tol : 1e-12;
  const int guess_vecs = guess ? L - 1 : 0;
  if (block)
    launch_eig_phase<float>(c, EigPhase{L, K, max_iter, tol > kMixedPhase1Tol ? tol : kMixedPhase1Tol, guess, guess_vecs, block}, s);
  launch_eig_phase<double>(c, EigPhase{L, K, max_iter, tol, block ? block : guess, block ? K : guess_vecs, nullptr}, s);
  return 0;
}

}  // namespace msmg
