// Register-resident stages of lengths 8 to 128, FP64.
#include "wf_reg_impl.cuh"
WF_RG_INSTANTIATE(double, 8)
WF_RG_INSTANTIATE(double, 16)
WF_RG_INSTANTIATE(double, 32)
WF_RG_INSTANTIATE(double, 64)
WF_RG_INSTANTIATE(double, 128)
WF_DBG_READER(reg_f64_small)
