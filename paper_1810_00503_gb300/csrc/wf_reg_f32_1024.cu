// Register-resident stages of length 1024, FP32.
#include "wf_reg_impl.cuh"
WF_RG_INSTANTIATE(float, 1024)
WF_DBG_READER(reg_f32_1024)
