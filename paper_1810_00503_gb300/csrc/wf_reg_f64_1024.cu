// Register-resident stages of length 1024, FP64.
#include "wf_reg_impl.cuh"
WF_RG_INSTANTIATE(double, 1024)
WF_DBG_READER(reg_f64_1024)
