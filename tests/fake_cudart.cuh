// The CUDA runtime calls that the launchers make, faked for the host: two or more devices, what is
// set on a kernel kept per device, launches recorded and not made.  Include it before a csrc/*.cu file.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <map>
#include <set>
#include <tuple>
#include <vector>

namespace fake {

struct Launch {
  int device;
  unsigned grid, block, cluster;
  size_t smem;
};
inline int device = 0;
inline int sms[4] = {152, 80, 40, 20};
inline int room[4][17] = {};                              // clusters of each size that a device runs at once
inline int failing_queries = 0;                           // so many occupancy queries fail first
inline std::map<std::pair<const void*, int>, int> limit;  // (kernel, device) -> dynamic shared memory allowed
inline std::set<std::pair<const void*, int>> wide;        // (kernel, device) -> clusters of more than 8 allowed
inline std::vector<Launch> launches;
inline int attribute_calls = 0;

inline cudaError_t last_error() { return cudaSuccess; }
inline cudaError_t get_device(int* d) {
  *d = device;
  return cudaSuccess;
}
inline cudaError_t device_attribute(int* v, cudaDeviceAttr a, int d) {
  *v = a == cudaDevAttrMultiProcessorCount ? sms[d] : 227 * 1024;
  return cudaSuccess;
}
template <class K>
cudaError_t set_attribute(K k, cudaFuncAttribute a, int v) {
  ++attribute_calls;
  const std::pair<const void*, int> key(reinterpret_cast<const void*>(k), device);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limit[key] = v;
  if (a == cudaFuncAttributeNonPortableClusterSizeAllowed) wide.insert(key);
  return cudaSuccess;
}
inline unsigned cluster_of(const cudaLaunchConfig_t* c) {
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return c->attrs[i].val.clusterDim.x;
  return 1;
}
template <class K>
cudaError_t max_clusters(int* n, K, const cudaLaunchConfig_t* c) {
  if (failing_queries > 0) {
    --failing_queries;
    return cudaErrorUnknown;
  }
  *n = room[device][cluster_of(c)];
  return cudaSuccess;
}
// A launch is refused where the real one would be: shared memory or a cluster beyond what this
// device was told to allow.
template <class... P, class... A>
cudaError_t launch(const cudaLaunchConfig_t* c, void (*k)(P...), A&&...) {
  const std::pair<const void*, int> key(reinterpret_cast<const void*>(k), device);
  const Launch l{device, c->gridDim.x, c->blockDim.x, cluster_of(c), c->dynamicSmemBytes};
  if (l.smem > 48 * 1024 && (!limit.count(key) || limit[key] < (int)l.smem)) return cudaErrorInvalidValue;
  if (l.cluster > 8 && !wide.count(key)) return cudaErrorInvalidValue;
  if (l.grid % l.cluster) return cudaErrorInvalidValue;
  launches.push_back(l);
  return cudaSuccess;
}
inline CUresult CUDAAPI encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                               const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                               CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}
inline cudaError_t entry_point(const char*, void** p, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q) {
  *p = reinterpret_cast<void*>(&encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

}  // namespace fake

#define cudaGetDevice fake::get_device
#define cudaDeviceGetAttribute fake::device_attribute
#define cudaFuncSetAttribute fake::set_attribute
#define cudaOccupancyMaxActiveClusters fake::max_clusters
#define cudaLaunchKernelEx fake::launch
#define cudaGetDriverEntryPointByVersion fake::entry_point
#define cudaGetLastError fake::last_error
