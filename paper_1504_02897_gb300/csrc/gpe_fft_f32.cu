// The GPE's Fourier passes in FP32 (gpe_fft.cuh).
#include "gpe_fft.cuh"

namespace ddi {
template int gpe_forward<float>(Plan&, const cx_t<float>*, cx_t<float>*, cudaStream_t);
template int gpe_kinetic<float>(Plan&, const cx_t<float>*, cx_t<float>*, const cx_t<float>*, float*, cudaStream_t);
template int gpe_gf_sweep<float>(Plan&, const GfSweep<float>&, cudaStream_t);
}  // namespace ddi
