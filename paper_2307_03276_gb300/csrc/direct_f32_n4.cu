// FP32 Phi and MTTKRP with the Khatri-Rao rows formed in place: 4 gathered modes.
#define DIRECT_NM1 4
#define DIRECT_FN launch_direct_f32_n4
#include "direct_inst.cuh"
