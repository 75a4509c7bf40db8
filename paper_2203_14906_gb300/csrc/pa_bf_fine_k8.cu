// Order 8 of the fine-grained fused beamforming kernel.
#include "pa_bf_fine.cuh"

PA_DEFINE_FINE(8)
