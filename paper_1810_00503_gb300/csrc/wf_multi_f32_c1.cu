// Shared FFT-stage launches, FP32, 1 channel.
#include "wf_multi_fft.cuh"
template cudaError_t wf_launch_multi_fft<float, 1>(const WfMultiArgs&, int, cudaStream_t);
WF_DBG_READER(multi_f32_c1)
