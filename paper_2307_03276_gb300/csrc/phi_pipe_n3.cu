// FP64 Phi on FP64 rows with the divisor on the FP32 pipe, three gathered modes.
#define PIPE_NM1 3
#define PIPE_FN launch_phi_pipe_n3
#include "phi_pipe.cuh"
