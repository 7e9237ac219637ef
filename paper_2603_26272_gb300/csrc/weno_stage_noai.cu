// weno_stage_noai.cu -- sixth-order stage launches: weights without the affine-invariant descaler.
#include "weno_tiles.cuh"

namespace weno {

cudaError_t launch_stage_noai(const StageArgs &a, cudaStream_t s) {
  return a.p == 1.0 ? launch_stage_t<kNoAi, true, 0, 3>(a, s)
                    : launch_stage_t<kNoAi, false, 0, 3>(a, s);
}

}  // namespace weno
