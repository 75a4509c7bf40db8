// Order 3 of the two-frame fused beamforming kernel.
#include "pa_bf_pipe.cuh"

PA_DEFINE_PIPE(3)
