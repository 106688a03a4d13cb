// What a launch asks of the runtime before it: function attributes, occupancy
// and the SM count.  Each query takes 0.3-1 us of host time, which a small
// tensor's call (8 us of kernel, four launches for an encode) cannot hide, so the
// answers are kept per device.  They depend on the kernel, its CTA size and
// its shared memory only.
#include <algorithm>
#include <mutex>
#include <vector>

#include "host_internal.h"

namespace zipnn {

namespace {

constexpr int kMaxDevices = 64;
constexpr size_t kMaxOccupancies = 256;  // kept per device, the oldest makes room

struct KernelSetup {
  const void* kern;
  int smem;  // the most dynamic shared memory it was given room for
};
struct Occupancy {
  const void* kern;
  int smem, threads, ctas;
};
struct DeviceSetup {
  int sms = 0;
  std::vector<KernelSetup> kernels;
  std::vector<Occupancy> occupancies;
  size_t oldest = 0;
};

std::mutex g_mu;
DeviceSetup g_dev[kMaxDevices];

cudaError_t set_room(const void* kern, int smem) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  return e;
}

cudaError_t occupancy(const void* kern, int threads, int smem, int* ctas) {
  *ctas = 0;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, kern, threads, smem);
  *ctas = std::max(*ctas, 1);
  return e;
}

int query_sms(int dev) {
  int sms = 0;
  return cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess ? sms : 0;
}

}  // namespace

int device_sms() {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= kMaxDevices) return query_sms(dev);
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_dev[dev].sms) g_dev[dev].sms = query_sms(dev);
  return g_dev[dev].sms;
}

// The room of a kernel only grows: another thread may be about to launch it with
// the larger size.
cudaError_t prepare_kernel(const void* kern, int smem, int threads, int* ctas_per_sm) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) {
    e = set_room(kern, smem);
    if (e == cudaSuccess && ctas_per_sm) e = occupancy(kern, threads, smem, ctas_per_sm);
    return e;
  }
  std::lock_guard<std::mutex> lk(g_mu);
  DeviceSetup& d = g_dev[dev];
  auto k = std::find_if(d.kernels.begin(), d.kernels.end(),
                        [&](const KernelSetup& s) { return s.kern == kern; });
  if (k == d.kernels.end() || k->smem < smem) {
    e = set_room(kern, smem);
    if (e != cudaSuccess) return e;
    if (k == d.kernels.end()) d.kernels.push_back({kern, smem});
    else k->smem = smem;
  }
  if (!ctas_per_sm) return cudaSuccess;
  for (const Occupancy& o : d.occupancies)
    if (o.kern == kern && o.smem == smem && o.threads == threads) {
      *ctas_per_sm = o.ctas;
      return cudaSuccess;
    }
  e = occupancy(kern, threads, smem, ctas_per_sm);
  if (e != cudaSuccess) return cudaSuccess;  // (one CTA per SM; asked again next time)
  const Occupancy o{kern, smem, threads, *ctas_per_sm};
  if (d.occupancies.size() < kMaxOccupancies) d.occupancies.push_back(o);
  else d.occupancies[d.oldest++ % kMaxOccupancies] = o;
  return cudaSuccess;
}

}  // namespace zipnn
