// Shared FFT-stage launches, FP64, 1 channel.
#include "wf_multi_fft.cuh"
template cudaError_t wf_launch_multi_fft<double, 1>(const WfMultiArgs&, int, cudaStream_t);
WF_DBG_READER(multi_f64_c1)
