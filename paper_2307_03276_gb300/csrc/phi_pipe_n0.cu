// FP64 Phi on FP64 rows with the divisor on the FP32 pipe, a runtime number of gathered modes.
#define PIPE_NM1 0
#define PIPE_FN launch_phi_pipe_n0
#include "phi_pipe.cuh"
