// FP32 Phi and MTTKRP with the Khatri-Rao rows formed in place: any number of gathered modes (runtime count).
#define DIRECT_NM1 0
#define DIRECT_FN launch_direct_f32_n0
#include "direct_inst.cuh"
