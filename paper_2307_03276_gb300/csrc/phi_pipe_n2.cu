// FP64 Phi on FP64 rows with the divisor on the FP32 pipe, two gathered modes.
#define PIPE_NM1 2
#define PIPE_FN launch_phi_pipe_n2
#include "phi_pipe.cuh"
