// The GPE's Fourier passes in FP64 (gpe_fft.cuh).
#include "gpe_fft.cuh"

namespace ddi {
template int gpe_forward<double>(Plan&, const cx_t<double>*, cx_t<double>*, cudaStream_t);
template int gpe_kinetic<double>(Plan&, const cx_t<double>*, cx_t<double>*, const cx_t<double>*, double*, cudaStream_t);
template int gpe_gf_sweep<double>(Plan&, const GfSweep<double>&, cudaStream_t);
}  // namespace ddi
