// Register-resident stages of length 256, FP64.
#include "wf_reg_impl.cuh"
WF_RG_INSTANTIATE(double, 256)
WF_DBG_READER(reg_f64_256)
