// Register-resident stages of lengths 8 to 128, FP32.
#include "wf_reg_impl.cuh"
WF_RG_INSTANTIATE(float, 8)
WF_RG_INSTANTIATE(float, 16)
WF_RG_INSTANTIATE(float, 32)
WF_RG_INSTANTIATE(float, 64)
WF_RG_INSTANTIATE(float, 128)
WF_DBG_READER(reg_f32_small)
