// Test-only: the resident recurrence's wait for packets that nobody publishes, many to a thread.
#include "resident.cu"

namespace tbpm {
namespace {
__global__ void k_packet_wait(const ulonglong2* packets, int units, uint64_t budget_ns, int* expired) {
  bool failed = false;
  float sum = 0.f;
  for (int u = 0; u < units; ++u) sum += receive_or_zero<float, 2>(packets + 2 * u, 1u, budget_ns, failed).v[0];
  if (failed && sum == 0.f) atomicAdd(expired, 1);
}
}  // namespace
}  // namespace tbpm

// Threads of one warp whose wait expired (each waits for `units` packets of a zeroed buffer), or -1.
extern "C" int packet_wait(int units, double budget_s) {
  void* p = nullptr;
  int* e = nullptr;
  int n = -1;
  const size_t bytes = sizeof(ulonglong2) * 2 * (size_t)units;
  if (cudaMalloc(&p, bytes) == cudaSuccess && cudaMalloc((void**)&e, sizeof(int)) == cudaSuccess &&
      cudaMemset(p, 0, bytes) == cudaSuccess && cudaMemset(e, 0, sizeof(int)) == cudaSuccess) {
    tbpm::k_packet_wait<<<1, 32>>>((const ulonglong2*)p, units, (uint64_t)(budget_s * 1e9), e);
    if (cudaDeviceSynchronize() != cudaSuccess || cudaMemcpy(&n, e, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
      n = -1;
  }
  cudaFree(p);
  cudaFree(e);
  return n;
}
