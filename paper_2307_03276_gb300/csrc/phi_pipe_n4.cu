// FP64 Phi on FP64 rows with the divisor on the FP32 pipe, four gathered modes.
#define PIPE_NM1 4
#define PIPE_FN launch_phi_pipe_n4
#include "phi_pipe.cuh"
