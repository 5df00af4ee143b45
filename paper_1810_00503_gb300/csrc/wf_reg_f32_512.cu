// Register-resident stages of length 512, FP32.
#include "wf_reg_impl.cuh"
WF_RG_INSTANTIATE(float, 512)
WF_DBG_READER(reg_f32_512)
