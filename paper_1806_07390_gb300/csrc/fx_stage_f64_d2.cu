// Stage kernel instantiations: state double, group arithmetic double, Newton/bookkeeping double, 2-d Cartesian.
#define FX_LAUNCH_DEFINE
#include "fx_launch.h"

namespace fx {
template cudaError_t launch_stage<double, 2, double, false>(const StageArgs<double>&, cudaStream_t, cudaEvent_t,
                                                  cudaEvent_t);
template cudaError_t stage_regs<double, 2, double, false>(int, int*);
}  // namespace fx
