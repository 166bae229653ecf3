// Stage kernel instantiations: state float, group arithmetic float, Newton/bookkeeping double
// (interaction kernel of its own), 3-d.
#define FX_LAUNCH_DEFINE
#include "fx_launch.h"

namespace fx {
template cudaError_t launch_stage<float, 3, double, false>(const StageArgs<float>&, cudaStream_t, cudaEvent_t,
                                                  cudaEvent_t);
template cudaError_t stage_regs<float, 3, double, false>(int, int*);
}  // namespace fx
