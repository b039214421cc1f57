// FP32 Phi and MTTKRP with the Khatri-Rao rows formed in place: 3 gathered modes.
#define DIRECT_NM1 3
#define DIRECT_FN launch_direct_f32_n3
#include "direct_inst.cuh"
