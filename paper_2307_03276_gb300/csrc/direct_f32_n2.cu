// FP32 Phi and MTTKRP with the Khatri-Rao rows formed in place: 2 gathered modes.
#define DIRECT_NM1 2
#define DIRECT_FN launch_direct_f32_n2
#include "direct_inst.cuh"
