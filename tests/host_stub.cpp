// The CUDA runtime and the kernels' launch wrappers as csrc/apc_host.cpp uses
// them, on the CPU: pointer queries are answered from a fixed map of fake
// addresses and counted, launches are recorded and run nothing
// (tests/test_host_plans.py).
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "apc_internal.h"
#include "apc_launch.cuh"

namespace {

constexpr uint64_t kAllocation = 1ull << 30;  // an ordinary allocation spans each aligned GB

uint64_t g_ordinary_from;                // addresses below are virtual-memory mappings
long g_runtime_queries, g_range_queries;
cudaError_t g_pending, g_refuse;         // the runtime's pending error; what launches answer
struct Launch {
  int64_t count, grid, more, chained;
};
std::vector<Launch> g_launches;
float g_limit;                           // the last commit plan's

cudaError_t launched() {
  g_pending = g_refuse ? g_refuse : g_pending;
  return g_refuse;
}

template <class Plan>
void no_kernel(Plan, unsigned long long *) {}

template <class Plan>
int record(const Plan &plan, unsigned grid, unsigned long long *out) {
  g_launches.push_back({plan.count, grid, plan.more, plan.chained});
  return apc::launch_plan(no_kernel<Plan>, plan, plan.chained, grid, 32u, 0u, nullptr, out);
}

CUresult range_query(unsigned n, CUpointer_attribute *names, void **values, CUdeviceptr p) {
  ++g_range_queries;
  for (unsigned i = 0; i < n; ++i) {
    const bool ordinary = p >= g_ordinary_from;
    if (names[i] == CU_POINTER_ATTRIBUTE_IS_LEGACY_CUDA_IPC_CAPABLE) *(unsigned *)values[i] = ordinary;
    else if (names[i] == CU_POINTER_ATTRIBUTE_RANGE_START_ADDR) *(CUdeviceptr *)values[i] = p / kAllocation * kAllocation;
    else if (names[i] == CU_POINTER_ATTRIBUTE_RANGE_SIZE) *(size_t *)values[i] = kAllocation;
    else return CUDA_ERROR_INVALID_VALUE;
  }
  return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

// Addresses from `ordinary_from` on are cudaMalloc's; launches answer `refuse`.
__attribute__((visibility("default"))) void stub_reset(uint64_t ordinary_from, int refuse) {
  g_ordinary_from = ordinary_from;
  g_refuse = (cudaError_t)refuse;
  g_pending = cudaSuccess;
  g_runtime_queries = g_range_queries = 0;
  g_launches.clear();
}
__attribute__((visibility("default"))) long stub_runtime_queries() { return g_runtime_queries; }
__attribute__((visibility("default"))) long stub_range_queries() { return g_range_queries; }
__attribute__((visibility("default"))) float stub_limit() { return g_limit; }
__attribute__((visibility("default"))) int stub_pending() { return (int)g_pending; }
__attribute__((visibility("default"))) long stub_launches(int64_t *out, long cap) {
  for (long i = 0; i < (long)g_launches.size() && i < cap; ++i) {
    const Launch &l = g_launches[(size_t)i];
    out[4 * i] = l.count, out[4 * i + 1] = l.grid, out[4 * i + 2] = l.more, out[4 * i + 3] = l.chained;
  }
  return (long)g_launches.size();
}

const char *cudaGetErrorString(cudaError_t) { return "stub"; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_pending;
  g_pending = cudaSuccess;
  return e;
}
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *st) {
  *fn = (void *)range_query;
  *st = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
  ++g_runtime_queries;
  *a = {};
  a->type = cudaMemoryTypeDevice;
  a->devicePointer = const_cast<void *>(p);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) { return launched(); }

}  // extern "C"

namespace apc {

template <int MAXE>
int launch_commit(const CommitPlan<MAXE> &plan, int, bool, unsigned grid, void *, unsigned long long *out) {
  g_limit = plan.limit;
  return record(plan, grid, out);
}
template int launch_commit(const CommitPlan<kCommitSmall> &, int, bool, unsigned, void *, unsigned long long *);
template int launch_commit(const CommitPlan<kCommitMid> &, int, bool, unsigned, void *, unsigned long long *);
template int launch_commit(const CommitPlan<kCommitLarge> &, int, bool, unsigned, void *, unsigned long long *);

template <int MAXE>
int launch_digest(const DigestPlan<MAXE> &plan, int, unsigned grid, void *, unsigned long long *out) {
  return record(plan, grid, out);
}
template int launch_digest(const DigestPlan<kDigestSmall> &, int, unsigned, void *, unsigned long long *);
template int launch_digest(const DigestPlan<kDigestMid> &, int, unsigned, void *, unsigned long long *);
template int launch_digest(const DigestPlan<kDigestLarge> &, int, unsigned, void *, unsigned long long *);

template <int MAXE>
int launch_count(const DigestPlan<MAXE> &plan, unsigned grid, void *, unsigned long long *out) {
  return record(plan, grid, out);
}
template int launch_count(const DigestPlan<kDigestSmall> &, unsigned, void *, unsigned long long *);
template int launch_count(const DigestPlan<kDigestMid> &, unsigned, void *, unsigned long long *);
template int launch_count(const DigestPlan<kDigestLarge> &, unsigned, void *, unsigned long long *);

int launch_upload(const UploadPlan<kUploadMax> &, unsigned, void *) { return (int)launched(); }
int commit_blocks_per_sm(int *out) { return *out = 1, 0; }
int digest_blocks_per_sm(int *out) { return *out = 1, 0; }
int count_blocks_per_sm(int *out) { return *out = 2, 0; }
int read_commit_status(unsigned *out) { return *out = 0, 0; }
int launch_wait_timeout(uint64_t, void *) { return (int)launched(); }

}  // namespace apc
