// FP64 Phi over float-pair Khatri-Rao rows formed in place: 3 gathered modes.
#define DF_NM1 3
#define DF_FN launch_phi_df_n3
#include "phi_df.cuh"
