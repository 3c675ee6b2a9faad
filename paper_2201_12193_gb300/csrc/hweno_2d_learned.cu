// FP64 stage of handles with the learned indicator (2D Euler): the pipeline in
// plain double (fx64.cuh says why).
#include "hweno_2d_kernels.cuh"

namespace hw {

void run_stage_2d_learned(const Prob& P, const HostTabs& T, const Bufs& B, const StageCall& S, cudaStream_t st) {
  stage_t<double, 4>(P, T, T.wl, T.b2l, B, S, st);
}

}  // namespace hw
