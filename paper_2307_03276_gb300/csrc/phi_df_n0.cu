// FP64 Phi over float-pair Khatri-Rao rows formed in place: any number of gathered modes (runtime count).
#define DF_NM1 0
#define DF_FN launch_phi_df_n0
#include "phi_df.cuh"
