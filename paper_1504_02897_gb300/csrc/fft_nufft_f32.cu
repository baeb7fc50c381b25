// The NUFFT's fine-grid FFT passes in FP32 (fft_nufft.cuh).
#include "fft_nufft.cuh"

namespace ddi {
template int nufft_forward_fft<float>(Plan&, const float*, cudaStream_t);
template int nufft_inverse_fft<float>(Plan&, float*, cudaStream_t, bool);
template int split_smooth_part<float>(Plan&, const float*, float*, cudaStream_t);
}  // namespace ddi
