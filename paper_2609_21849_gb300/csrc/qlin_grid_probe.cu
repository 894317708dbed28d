// Probes of the dynamic quantizers' grid-wide maximum (qlin_grid_probe.h), on
// the kernels of qlin_quant.cu, which the probe library links too.
#include "qlin_grid_probe.h"

#include "qlin_internal.h"

namespace qlin {
namespace {

constexpr int kHoldSmem = 227 * 1024;

// Waits on nothing but the clock.
__global__ void __launch_bounds__(32) hold_kernel(unsigned long long ns) {
  const uint64_t t0 = global_timer_ns();
  while (global_timer_ns() - t0 < ns) __nanosleep(200);
}

// The current device (no SMs: none that can be used).
Device device() {
  Device d{0, 0};
  if (cudaGetDevice(&d.index) != cudaSuccess || d.index >= kMaxDevices ||
      cudaDeviceGetAttribute(&d.num_sms, cudaDevAttrMultiProcessorCount, d.index) != cudaSuccess)
    return {0, 0};
  return d;
}

bool aligned(const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

}  // namespace
}  // namespace qlin

using namespace qlin;

extern "C" int qlin_probe_grid_max(int fmt, const void* x, long long M, long long K, void* out,
                                   unsigned* sync, unsigned long long help_ns,
                                   unsigned long long stop_ns, unsigned* counts, void* stream) {
  if ((fmt != 1 && fmt != 2) || x == nullptr || out == nullptr || sync == nullptr ||
      counts == nullptr || M < 1 || K < 64 || K % 64 != 0 || help_ns > 1000000 ||
      stop_ns > 1000000 || !aligned(x, 16) || !aligned(sync, 8))
    return 1;
  const GridWait wait{help_ns, stop_ns};
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e;
  if (fmt == 1) {
    const qlin_nvfp4_t& o = *static_cast<const qlin_nvfp4_t*>(out);
    if (o.codes == nullptr || o.scales == nullptr || o.tensor_scale == nullptr || o.rows != M ||
        o.K != K || !aligned(o.codes, 16))
      return 1;
    const Device dev = device();
    if (dev.num_sms == 0) return 4;
    e = launch_quant_nvfp4_dynamic(x, M, K, o, sync, false, s, dev, wait);
  } else {
    const qlin_fp8_t& o = *static_cast<const qlin_fp8_t*>(out);
    if (o.codes == nullptr || o.scale == nullptr || o.per_channel || o.rows != M || o.K != K ||
        !aligned(o.codes, 16))
      return 1;
    const Device dev = device();
    if (dev.num_sms == 0) return 4;
    e = launch_quant_fp8_dynamic(x, M, K, o, sync, false, s, dev, wait);
  }
  unsigned got[3] = {};
  if (e == cudaSuccess) e = take_grid_counts(got);
  for (int i = 0; i < 3; ++i) counts[i] = got[i];
  return e == cudaSuccess ? 0 : 4;
}

extern "C" int qlin_probe_hold_sms(int ctas, unsigned long long ns, void* stream) {
  if (ctas < 1 || ns > 5000000) return 1;
  if (ctas > device().num_sms) return 1;
  if (cudaFuncSetAttribute(hold_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kHoldSmem) !=
      cudaSuccess)
    return 4;
  hold_kernel<<<ctas, 32, kHoldSmem, static_cast<cudaStream_t>(stream)>>>(ns);
  return cudaGetLastError() == cudaSuccess ? 0 : 4;
}
