// weno_stage_ai.cu -- sixth-order stage launches: affine-invariant weights with p != 1 or a
// sensitivity term that counts.
#include "weno_tiles.cuh"

namespace weno {

cudaError_t launch_stage_ai(const StageArgs &a, cudaStream_t s) {
  return a.p == 1.0 ? launch_stage_t<kAi, true, 0, 3>(a, s)
                    : launch_stage_t<kAi, false, 0, 3>(a, s);
}

}  // namespace weno
