// weno_stage_tiny.cu -- sixth-order stage launches: the default weights (Ai, p = 1, a sensitivity
// term below the integer path's resolution).
#include "weno_tiles.cuh"

namespace weno {

cudaError_t launch_stage_tiny(const StageArgs &a, cudaStream_t s) {
  return launch_stage_t<kAiTiny, true, 0, 3>(a, s);
}

}  // namespace weno
