// The NUFFT's fine-grid FFT passes in FP64 (fft_nufft.cuh).
#include "fft_nufft.cuh"

namespace ddi {
template int nufft_forward_fft<double>(Plan&, const double*, cudaStream_t);
template int nufft_inverse_fft<double>(Plan&, double*, cudaStream_t, bool);
template int split_smooth_part<double>(Plan&, const double*, double*, cudaStream_t);
}  // namespace ddi
