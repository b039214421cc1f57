// FP64 Phi over float-pair Khatri-Rao rows formed in place: 2 gathered modes.
#define DF_NM1 2
#define DF_FN launch_phi_df_n2
#include "phi_df.cuh"
