// Register-resident stages of length 256, FP32.
#include "wf_reg_impl.cuh"
WF_RG_INSTANTIATE(float, 256)
WF_DBG_READER(reg_f32_256)
