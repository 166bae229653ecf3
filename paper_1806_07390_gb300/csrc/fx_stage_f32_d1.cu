// Stage kernel instantiations: state float, group arithmetic float, Newton/bookkeeping float
// (interaction kernel of its own), 1-d.
#define FX_LAUNCH_DEFINE
#include "fx_launch.h"

namespace fx {
template cudaError_t launch_stage<float, 1, float, false>(const StageArgs<float>&, cudaStream_t, cudaEvent_t,
                                                  cudaEvent_t);
template cudaError_t stage_regs<float, 1, float, false>(int, int*);
}  // namespace fx
