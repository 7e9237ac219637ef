// weno_stage_fp32.cu -- sixth-order stage launches: FP32 reconstruction (affine-invariant weights).
#include "weno_tiles.cuh"

namespace weno {

cudaError_t launch_stage_fp32(const StageArgs &a, cudaStream_t s) {
  return a.p == 1.0 ? launch_stage_t<kAi, true, 1, 3>(a, s)
                    : launch_stage_t<kAi, false, 1, 3>(a, s);
}

}  // namespace weno
