// FP32 Phi over materialised Khatri-Rao rows.
#define DIRECT_PI 1
#define DIRECT_FN launch_direct_f32_pi
#include "direct_inst.cuh"
