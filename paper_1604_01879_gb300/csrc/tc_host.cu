// Host helpers of the tcgen05 kernels: TMA tensor maps and device queries.
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "tc_common.cuh"

namespace gift {

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// the driver entry point is fetched through the runtime, so the library does
// not link against the driver library and still loads on GPU-less hosts
EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    GIFT_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q));
    if (q != cudaDriverEntryPointSuccess || !p) fail(GIFT_ECUDA, "cuTensorMapEncodeTiled is not available");
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

}  // namespace

CUtensorMap make_tmap_bf16(const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows, uint64_t pitch) {
  if (pitch == 0) pitch = cols;
  GIFT_REQUIRE(reinterpret_cast<uintptr_t>(base) % 16 == 0, "tensor map base must be 16-byte aligned");
  GIFT_REQUIRE((pitch * 2) % 16 == 0 && pitch >= cols, "tensor map row pitch must be >= cols and a multiple of 16 bytes");
  GIFT_REQUIRE(box_rows >= 1 && box_rows <= 256, "tensor map box rows must be in [1, 256]");
  // callers pad every source by one box, so a tile never leaves the allocation
  GIFT_REQUIRE(rows >= box_rows, "tensor map extent must cover at least one box");
  CUtensorMap m;
  const cuuint64_t dims[2] = {cols, rows > 0 ? rows : 1};
  const cuuint64_t strides[1] = {pitch * 2};
  const cuuint32_t box[2] = {64u, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                                 box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) fail(GIFT_ECUDA, "cuTensorMapEncodeTiled failed with " + std::to_string((int)r));
  return m;
}

CUtensorMap make_tmap_u8(const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows, uint64_t pitch) {
  if (pitch == 0) pitch = cols;
  GIFT_REQUIRE(reinterpret_cast<uintptr_t>(base) % 16 == 0, "tensor map base must be 16-byte aligned");
  GIFT_REQUIRE(pitch % 16 == 0 && pitch >= cols, "tensor map row pitch must be >= cols and a multiple of 16 bytes");
  GIFT_REQUIRE(box_rows >= 1 && box_rows <= 256, "tensor map box rows must be in [1, 256]");
  GIFT_REQUIRE(rows >= box_rows, "tensor map extent must cover at least one box");
  CUtensorMap m;
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {pitch};
  const cuuint32_t box[2] = {128u, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box,
                                 estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) fail(GIFT_ECUDA, "cuTensorMapEncodeTiled failed with " + std::to_string((int)r));
  return m;
}

CUtensorMap make_tmap_f32(const void* base, uint64_t rows, uint64_t cols, uint32_t box_cols, uint32_t box_rows) {
  GIFT_REQUIRE(reinterpret_cast<uintptr_t>(base) % 16 == 0, "tensor map base must be 16-byte aligned");
  GIFT_REQUIRE(cols % 4 == 0 && rows >= 1, "tensor map rows must be multiples of 16 bytes");
  GIFT_REQUIRE(box_rows >= 1 && box_rows <= 256 && box_cols % 4 == 0 && box_cols <= 256, "tensor map box out of range");
  CUtensorMap m;
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols * 4};
  const cuuint32_t box[2] = {box_cols, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides, box,
                                 estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) fail(GIFT_ECUDA, "cuTensorMapEncodeTiled failed with " + std::to_string((int)r));
  return m;
}

// Words of bounded waits, in blocks of a page or four that are registered with CUDA and kept for the life of the process
// (ordinary memory, so that the host's reads need no context). Words given back are taken again, so there are as many
// blocks as the most indices at a time need, usually one; threads have 1,024 words of their own (with more threads than
// that, one may be told of another's).
namespace {
constexpr int kBlockWords = 4096, kThreadWords = 1024;
std::mutex g_words_mu;
std::vector<int*> g_free_words;
int* g_thread_words = nullptr;
int* new_words(int n) {
  void* p = aligned_alloc(4096, n * sizeof(int));
  if (p) memset(p, 0, n * sizeof(int));
  if (!p || cudaHostRegister(p, n * sizeof(int), cudaHostRegisterPortable | cudaHostRegisterMapped) != cudaSuccess) {
    cudaGetLastError();
    free(p);
    fail(GIFT_ENOMEM, "host memory for the wait words could not be registered");
  }
  return static_cast<int*>(p);
}
}  // namespace

int* take_wait_word() {
  std::lock_guard<std::mutex> lock(g_words_mu);
  if (g_free_words.empty()) {
    g_free_words.reserve(kBlockWords);
    int* w = new_words(kBlockWords);
    for (int i = 0; i < kBlockWords; ++i) g_free_words.push_back(w + i);
  }
  int* w = g_free_words.back();
  g_free_words.pop_back();
  __atomic_store_n(w, 0, __ATOMIC_RELAXED);
  return w;
}

void give_wait_word(int* word) {
  if (!word) return;
  std::lock_guard<std::mutex> lock(g_words_mu);
  g_free_words.push_back(word);
}

int* thread_wait_word() {
  static std::atomic<unsigned> next{0};
  thread_local int* mine = nullptr;
  if (!mine) {
    std::lock_guard<std::mutex> lock(g_words_mu);
    if (!g_thread_words) g_thread_words = new_words(kThreadWords);
    mine = g_thread_words + next.fetch_add(1) % kThreadWords;
  }
  return mine;
}

void check_wait_word(int* word, int* flag, cudaStream_t s) {
  if (__atomic_load_n(word, __ATOMIC_ACQUIRE) == 0) return;
  const int site = __atomic_exchange_n(word, 0, __ATOMIC_ACQ_REL);
  if (site == 0) return;
  if (flag) GIFT_CUDA(cudaMemsetAsync(flag, 0, sizeof(int), s));
  fail(GIFT_ETIMEOUT, "a kernel's wait gave up (site " + std::to_string(site) +
                          "): the results of this call, or of the calls before it that were not waited for, are not valid");
}

int device_sm_count() {
  constexpr int kDevices = 64;
  static std::atomic<int> known[kDevices];  // a property of the device, asked once
  int dev = 0, n = 0;
  GIFT_CUDA(cudaGetDevice(&dev));
  if (dev < kDevices && (n = known[dev].load()) > 0) return n;
  GIFT_CUDA(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
  if (dev < kDevices) known[dev].store(n);
  return n;
}

}  // namespace gift
