// Makes a bounded wait of an index's flag run out: a barrier that nothing arrives on (about a second), as a kernel of
// the index's calls would, and returns what the wait reported.
#include "../../paper_1604_01879_gb300/csrc/tc_common.cuh"

namespace {
__global__ void k_wait(int* err, int* ok) {
  __shared__ uint64_t bar;
  const uint32_t b = gift::tc::smem_u32(&bar);
  gift::tc::mbar_init(b, 1);
  gift::tc::fence_barrier_init();
  *ok = gift::tc::mbar_wait(b, 0, err, gift::tc::kErrMma) ? 1 : 0;
  if (!*ok) gift::report_wait(err);
}
}  // namespace

extern "C" __attribute__((visibility("default"))) int wait_probe(void* index) {
  gift::Index& ix = *static_cast<gift::Index*>(index);
  int* ok = nullptr;
  int h = -1;
  if (cudaMalloc(&ok, 4) != cudaSuccess) return -1;
  k_wait<<<1, 1>>>(ix.d_err, ok);
  if (cudaMemcpy(&h, ok, 4, cudaMemcpyDeviceToHost) != cudaSuccess) h = -1;
  cudaFree(ok);
  return h;  // 0: gave up
}
