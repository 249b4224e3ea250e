// Off-line vocabulary on the GPU: Lloyd's k-means (Sec. 2.3 trains the
// codebook of the first inverted file with k-means and gives no details).
//
// Iteration: every row goes to its nearest centre through the exact
// quantiser (tensor-core coarse scores + two-float refine, ties to the lowest
// index); rows are grouped by centre with a stable sort, and each centre
// becomes the mean of its rows, summed in two-float (compensated FP32)
// arithmetic in ascending row order (so the result does not depend on
// scheduling; no FP64 on the GPU). A centre left without rows takes
// the row farthest from the centre it was assigned to (distance desc, index
// asc), the empty centres served in ascending order.
#include "gift_internal.cuh"

namespace gift {

namespace {

// Mean of each centre's rows (perm[off[c] .. off[c+1]) ascending), two-float sums. A block
// takes one centre and 4 * kMeanT columns, one float4 of them per thread, and keeps
// kMeanRows row loads in flight per thread: the kernel is bound by reading X once
// (16,384 x 4096 FP32, 1,024 centres: 268 MB), and a loop with one dependent
// 4-byte load per row and thread left that read latency-bound (1,174 us against 75).
// Every column still adds its rows in ascending order, so the sums are the same.
constexpr int kMeanT = 128, kMeanRows = 8;
__global__ __launch_bounds__(kMeanT) void k_km_mean(const float* __restrict__ X, int D,
                                                    const int32_t* __restrict__ perm,
                                                    const int64_t* __restrict__ off, const float* __restrict__ C_old,
                                                    float* __restrict__ C_new) {
  dep_begin();
  const int c = blockIdx.x;
  const int d = (blockIdx.y * kMeanT + threadIdx.x) * 4;
  if (d >= D) return;
  const int64_t r0 = off[c], r1 = off[c + 1];
  float4 out;
  if (r1 == r0) {  // empty: keep the old centre until it is re-seeded
    out = *reinterpret_cast<const float4*>(C_old + (int64_t)c * D + d);
  } else {
    F2 s[4];
    for (int64_t e = r0; e < r1; e += kMeanRows) {
      float4 x[kMeanRows];
#pragma unroll
      for (int k = 0; k < kMeanRows; ++k)
        if (e + k < r1) x[k] = __ldcs(reinterpret_cast<const float4*>(X + (int64_t)perm[e + k] * D + d));
#pragma unroll
      for (int k = 0; k < kMeanRows; ++k)
        if (e + k < r1) {
          f2_add(s[0], x[k].x);
          f2_add(s[1], x[k].y);
          f2_add(s[2], x[k].z);
          f2_add(s[3], x[k].w);
        }
    }
    // (hi + lo) / n: the quotient of the two-float sum, rounded once more
    const float n = (float)(r1 - r0);
    float m[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float q = __fdiv_rn(s[k].hi, n);
      const float rem = __fmaf_rn(-q, n, s[k].hi);  // s.hi - q n exactly (n < 2^24)
      m[k] = q + __fdiv_rn(rem + s[k].lo, n);
    }
    out = make_float4(m[0], m[1], m[2], m[3]);
  }
  *reinterpret_cast<float4*>(C_new + (int64_t)c * D + d) = out;
}

// squared distance of every row to its assigned centre (warp per row, two-float):
// t = x - c exactly as th + tl (TwoSum), t^2 = th^2 + 2 th tl + tl^2 with the
// rounding error of th^2 recovered by an FMA
__global__ void k_km_dist(const float* __restrict__ X, int64_t n, int D, const float* __restrict__ C,
                          const int32_t* __restrict__ lab, float* __restrict__ dist) {
  const int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= n) return;
  const float* x = X + r * D;
  const float* c = C + (int64_t)lab[r] * D;
  F2 s;
  for (int d = lane; d < D; d += 32) {
    float th, tl;
    two_sum(x[d], -c[d], th, tl);
    const float p = th * th;
    const float pe = __fmaf_rn(th, th, -p);
    f2_add(s, p);
    s.lo += pe + tl * (2.f * th + tl);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s = f2_merge(s, f2_shfl_xor(s, o));
  if (lane == 0) dist[r] = f2_value(s);
}

__global__ void k_km_rows(const float* __restrict__ X, int D, const int32_t* __restrict__ rows,
                          int64_t n_rows, float* __restrict__ out) {
  const int64_t i = blockIdx.x;
  if (i >= n_rows) return;
  for (int d = threadIdx.x; d < D; d += blockDim.x) out[i * D + d] = X[(int64_t)rows[i] * D + d];
}

}  // namespace

void kmeans(const float* X, int64_t n, int D, int K, const std::vector<int32_t>& init_rows, int iters, float* C_out,
            Scratch& sc, cudaStream_t s) {
  Index tmp;  // the quantiser's view of the current centres
  tmp.prm.n_codewords = K;
  tmp.prm.dim = D;
  GIFT_CUDA(cudaGetDevice(&tmp.device));
  tmp.codebook = tmp.alloc<float>((size_t)K * D);
  tmp.make_wait_flag(s);
  int32_t* d_init = sc.get<int32_t>(K);
  GIFT_CUDA(cudaMemcpyAsync(d_init, init_rows.data(), (size_t)K * 4, cudaMemcpyHostToDevice, s));
  k_km_rows<<<(unsigned)K, 256, 0, s>>>(X, D, d_init, K, tmp.codebook);
  GIFT_LAUNCHED("k_km_rows");
  float* x_inv = sc.get<float>(n);
  float* C_new = sc.get<float>((size_t)K * D);
  int32_t* lab = sc.get<int32_t>(n);
  int32_t* perm = sc.get<int32_t>(n);
  int32_t* skeys = sc.get<int32_t>(n);
  int64_t* off = sc.get<int64_t>((size_t)K + 1);
  float* dist = sc.get<float>(n);
  std::vector<int64_t> h_off((size_t)K + 1);
  // rows of one quantiser pass: their two-part copy is the same in every iteration
  SplitRows parts;
  if (iters > 0 && n <= kAssignChunk) parts = split_for_assign(X, n, D, x_inv, sc, s);
  else launch_row_invnorm(X, n, D, x_inv, s);
  for (int it = 0; it < iters; ++it) {
    Scratch isc(s);
    const float* cb_max = prepare_codebook_async(tmp, isc, s);
    assign_codes(tmp, X, n, 1, lab, isc, s, x_inv, nullptr, parts.hi ? &parts : nullptr, cb_max);
    stable_sort_by_key(lab, n, K, perm, skeys, isc, s);
    bin_offsets(skeys, n, K, off, s);
    launch_dep(k_km_mean, dim3((unsigned)K, (unsigned)cdiv(D, 4 * kMeanT)), dim3(kMeanT), 0, s, X, D, perm, off,
               tmp.codebook, C_new);
    GIFT_LAUNCHED("k_km_mean");
    GIFT_CUDA(cudaMemcpyAsync(h_off.data(), off, ((size_t)K + 1) * 8, cudaMemcpyDeviceToHost, s));
    GIFT_CUDA(cudaStreamSynchronize(s));
    tmp.check_waits(s);
    std::vector<int32_t> empty;
    for (int c = 0; c < K; ++c)
      if (h_off[c + 1] == h_off[c]) empty.push_back(c);
    if (!empty.empty()) {
      const int E = (int)empty.size();
      k_km_dist<<<(unsigned)cdiv(n, 8), 256, 0, s>>>(X, n, D, tmp.codebook, lab, dist);
      GIFT_LAUNCHED("k_km_dist");
      int32_t* far = isc.get<int32_t>(E);
      topk_rows_f32(dist, 1, n, E, far, nullptr, s);  // distance desc, index asc
      std::vector<int32_t> h_far(E);
      GIFT_CUDA(cudaMemcpyAsync(h_far.data(), far, (size_t)E * 4, cudaMemcpyDeviceToHost, s));
      GIFT_CUDA(cudaStreamSynchronize(s));
      for (int e = 0; e < E; ++e)
        GIFT_CUDA(cudaMemcpyAsync(C_new + (int64_t)empty[e] * D, X + (int64_t)h_far[e] * D, (size_t)D * 4,
                                  cudaMemcpyDeviceToDevice, s));
    }
    std::swap(tmp.codebook, C_new);  // both live until the end of the call
  }
  GIFT_CUDA(cudaMemcpyAsync(C_out, tmp.codebook, (size_t)K * D * 4, cudaMemcpyDefault, s));
  GIFT_CUDA(cudaStreamSynchronize(s));
}

}  // namespace gift
