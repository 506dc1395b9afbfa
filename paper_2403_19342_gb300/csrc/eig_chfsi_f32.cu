// The FP32 phase of the mixed form's level-1 eigensolve (eig_chfsi.cuh).
#include "eig_chfsi.cuh"

namespace msmg {
template void launch_eig_phase<float>(msmg_ctx*, const EigPhase&, cudaStream_t);
}
