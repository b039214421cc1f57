// FP64 Phi over float-pair Khatri-Rao rows formed in place: 4 gathered modes.
#define DF_NM1 4
#define DF_FN launch_phi_df_n4
#include "phi_df.cuh"
