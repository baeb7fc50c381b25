// The FP64-built twiddle tables of the Stockham FFTs (fft_core.cuh).
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>

#include "common.cuh"

namespace ddi {

int prepare_kernel(const void* fn, size_t smem) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, size_t> done;  // (device, kernel) -> limit set
  int dev = 0;
  DDI_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  auto it = done.find({dev, fn});
  if (it != done.end() && it->second >= smem) return DDI_OK;
  if (smem > 48 * 1024) DDI_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  done[{dev, fn}] = smem;
  return DDI_OK;
}

int make_twiddles(Plan& p, int n) {
  if (twiddles(p, n)) return DDI_OK;
  int b = 0;
  while (b < 8 && p.tw_n[b] != 0) ++b;
  if (b == 8) {
    set_error("too many distinct FFT lengths in one plan");
    return DDI_ERR_ARG;
  }
  // FP64: e^{-2 pi i k / n} from FP64 libm.  FP32: head and tail of each component,
  // [n] heads then [n] tails, so that a stage multiplies by the twiddle to FP64 accuracy:
  // a rounded twiddle has |w| != 1 by up to 6e-8, and the same table in every transform
  // would scale the data's norm by the same amount every time (a steady mass drift in
  // long time-splitting runs)
  const size_t es = p.cx_size();
  const size_t count = p.prec == DDI_FP64 ? (size_t)n : 2 * (size_t)n;
  std::vector<unsigned char> host(es * count);
  for (int k = 0; k < n; ++k) {
    const double ang = (-2.0 * M_PI * (double)k) / (double)n;
    const double c = std::cos(ang), sn = std::sin(ang);
    if (p.prec == DDI_FP64) {
      double2 v = make_double2(c, sn);
      memcpy(host.data() + es * k, &v, es);
    } else {
      const float ch = (float)c, sh = (float)sn;
      float2 hi = make_float2(ch, sh);
      float2 lo = make_float2((float)(c - (double)ch), (float)(sn - (double)sh));
      memcpy(host.data() + es * k, &hi, es);
      memcpy(host.data() + es * (n + (size_t)k), &lo, es);
    }
  }
  void* d = nullptr;
  if (cudaMalloc(&d, es * count) != cudaSuccess) {
    set_error("cudaMalloc of a twiddle table failed");
    return DDI_ERR_OOM;
  }
  p.bytes += es * count;
  DDI_CUDA(cudaMemcpy(d, host.data(), es * count, cudaMemcpyHostToDevice));
  p.d_tw[b] = d;
  p.tw_n[b] = n;
  return DDI_OK;
}

}  // namespace ddi
