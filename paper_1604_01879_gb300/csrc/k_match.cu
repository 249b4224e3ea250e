// Matching score of Eq. 3 after a learned linear view projection u = W q,
// and its gradient through the argmax view pair: products on the tensor
// cores, the gradient's one-hot gathers on the CUDA cores.
//
// Forward: U = Q W^T and V = P W^T (engine GEMMs; BF16 inputs multiply
// exactly in one product, FP32 inputs in the two-part split), then the
// segmented-max contraction of U and V (two-part split, FP32-level) gives
// S and the first argmax j* of every (query view, shape).
// Backward, with c = grad_S[b, p] / |V(x_b)| and s = u_i.v_j*/(|u_i||v_j*|):
//   dU_i  = (1/|u_i|)  ( g_i - (g_i . u_i/|u_i|) u_i/|u_i| ),  g_i = sum_p c v_j*/|v_j*|
//   dV_r  = (1/|v_r|)  ( h_r - (h_r . v_r/|v_r|) v_r/|v_r| ),  h_r = sum_{(i,p): j*=r} c u_i/|u_i|
// (the projections use s = g-weighted cosines: sum_p c s = g_i . u_i/|u_i|).
// G = A V and H = A^T U, with the one-hot matrix A[i, r] = c / |v_r| (c / |u_i| for
// H) where r is the argmax view of (i, shape(r)), are gathers on the CUDA cores: N_v
// times fewer multiply-adds than the dense products, FP32 sums in a fixed order. A
// block stages slices of V (of U for H) and of the shape-major argmax in shared
// memory and adds one staged row per (query view, shape) entry. Then
//   dW = dU^T Q + dV^T P,  dQ = dU W,  dP = dV W
// as engine GEMMs on transposed two-part operands.
#include <cstring>

#include "gift_internal.cuh"
#include "segmax.cuh"
#include "tc_gemm.cuh"

namespace gift {

namespace {

// element of an input in FP32 or BF16
template <typename T>
__device__ __forceinline__ float ld_f(const T* p, int64_t i);
template <>
__device__ __forceinline__ float ld_f<float>(const float* p, int64_t i) { return p[i]; }
template <>
__device__ __forceinline__ float ld_f<__nv_bfloat16>(const __nv_bfloat16* p, int64_t i) {
  return __bfloat162float(p[i]);
}

// two-part BF16 copy of a row-major [rows, cols] matrix (lo may be null)
template <typename T>
__global__ void k_split_any(const T* __restrict__ in, int64_t n, __nv_bfloat16* __restrict__ hi,
                            __nv_bfloat16* __restrict__ lo) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float v = ld_f<T>(in, i);
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  hi[i] = h;
  if (lo) lo[i] = __float2bfloat16_rn(v - __bfloat162float(h));
}

// the same for FP32 inputs, four elements per thread (sizes multiples of four, 16-byte aligned inputs, 8-byte aligned
// outputs): up to three matrices in one launch, of which a small step would otherwise notice the launches
struct Split4 {
  const float4* in;
  uint2* hi;
  uint2* lo;
  int64_t end;  // elements / 4 of this matrix and those before it
};
struct Split4s {
  int n = 0;
  Split4 m[3];
};
__global__ void k_split4(const Split4s a) {
  const int64_t total = a.m[a.n - 1].end;
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total; g += (int64_t)gridDim.x * blockDim.x) {
    int k = 0;
    while (g >= a.m[k].end) ++k;
    const int64_t i = k ? g - a.m[k - 1].end : g;
    const float4 v = a.m[k].in[i];
    const __nv_bfloat162 h01 = __floats2bfloat162_rn(v.x, v.y), h23 = __floats2bfloat162_rn(v.z, v.w);
    const float2 f01 = __bfloat1622float2(h01), f23 = __bfloat1622float2(h23);
    const __nv_bfloat162 l01 = __floats2bfloat162_rn(v.x - f01.x, v.y - f01.y);
    const __nv_bfloat162 l23 = __floats2bfloat162_rn(v.z - f23.x, v.w - f23.y);
    a.m[k].hi[i] = make_uint2(*reinterpret_cast<const uint32_t*>(&h01), *reinterpret_cast<const uint32_t*>(&h23));
    if (a.m[k].lo)
      a.m[k].lo[i] = make_uint2(*reinterpret_cast<const uint32_t*>(&l01), *reinterpret_cast<const uint32_t*>(&l23));
  }
}

template <typename T>
__global__ void k_to_float(const T* __restrict__ in, int64_t n, float* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = ld_f<T>(in, i);
}

// Transposes: out[c, r] (row pitch ld) = in[r, c] for r < rows, zero for rows <= r < ld; several matrices of one kind
// in one launch, a block per tile of any of them.
struct Turn {
  const void* in;
  int64_t rows, cols, ld;
  __nv_bfloat16* hi;
  __nv_bfloat16* lo;  // two-part output; null: one part
  int64_t tiles_x, end;  // tiles across, and tiles of this matrix and those before it
};
constexpr int kTurns = 5;
struct Turns {
  int n = 0;
  Turn m[kTurns];
};
__device__ __forceinline__ const Turn& turn_of(const Turns& a, int64_t tile, int64_t& tx, int64_t& ty) {
  int k = 0;
  while (tile >= a.m[k].end) ++k;
  const uint32_t t = (uint32_t)(k ? tile - a.m[k - 1].end : tile), w = (uint32_t)a.m[k].tiles_x;  // (below 2^31)
  tx = t % w;
  ty = t / w;
  return a.m[k];
}

// two-part BF16 from FP32 or one-part from BF16, 32 x 32 tiles
template <typename T>
__global__ void k_transpose_split(const Turns a) {
  __shared__ float t[32][33];
  int64_t tx, ty;
  const Turn& m = turn_of(a, blockIdx.x, tx, ty);
  const T* in = static_cast<const T*>(m.in);
  const int64_t r0 = ty * 32, c0 = tx * 32;
  for (int y = threadIdx.y; y < 32; y += 8) {
    const int64_t r = r0 + y, c = c0 + threadIdx.x;
    t[y][threadIdx.x] = (r < m.rows && c < m.cols) ? ld_f<T>(in, r * m.cols + c) : 0.f;
  }
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += 8) {
    const int64_t c = c0 + y, r = r0 + threadIdx.x;
    if (c < m.cols && r < m.ld) {
      const float v = t[threadIdx.x][y];
      const __nv_bfloat16 h = __float2bfloat16_rn(v);
      m.hi[c * m.ld + r] = h;
      if (m.lo) m.lo[c * m.ld + r] = __float2bfloat16_rn(v - __bfloat162float(h));
    }
  }
}

// The same in 16-byte pieces, read and written in whole 128-byte lines (aligned rows; cols a multiple of a piece,
// ld of 64). A tile lies in shared memory as rows of 4-byte words whose index is exclusive-ored with four times the
// row's octet, so that the eight octets of an output line are read from different banks, and pieces stay whole.
__device__ __forceinline__ int turn_word(int row, int word) { return word ^ (((row >> 3) & 7) * 4); }

// BF16 in one part, 128 x 64 tiles: a thread turns eight rows of two columns.
// Bound by memory: 278,528 x 4,096 values (4.56 GB moved) in 668 us, 6.8 TB/s; 1,240 in 64 x 64 tiles read one value
// at a time (eight-way bank conflicts).
__global__ __launch_bounds__(256) void k_transpose_bf16(const Turns a) {
  __shared__ __align__(16) uint32_t t[128][32];
  int64_t tx, ty;
  const Turn& m = turn_of(a, blockIdx.x, tx, ty);
  const __nv_bfloat16* in = static_cast<const __nv_bfloat16*>(m.in);
  const int64_t r0 = ty * 128, c0 = tx * 64;
  const int tid = threadIdx.x, part = tid & 7;
  uint4 v[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t r = r0 + (tid >> 3) + 32 * i, c = c0 + part * 8;
    v[i] = make_uint4(0u, 0u, 0u, 0u);
    if (r < m.rows && c < m.cols) v[i] = __ldcs(reinterpret_cast<const uint4*>(in + r * m.cols + c));
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = (tid >> 3) + 32 * i;
    *reinterpret_cast<uint4*>(&t[row][turn_word(row, part * 4)]) = v[i];
  }
  __syncthreads();
  const int pair = tid >> 3;
  const int64_t c = c0 + 2 * pair;
  if (c >= m.cols) return;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int row = part * 8 + 64 * i;
    const int64_t r = r0 + row;
    if (r >= m.ld) return;
    uint32_t w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) w[k] = t[row + k][turn_word(row, pair)];
    uint4 x, y;  // columns c and c + 1
    x = make_uint4(__byte_perm(w[0], w[1], 0x5410), __byte_perm(w[2], w[3], 0x5410),
                   __byte_perm(w[4], w[5], 0x5410), __byte_perm(w[6], w[7], 0x5410));
    y = make_uint4(__byte_perm(w[0], w[1], 0x7632), __byte_perm(w[2], w[3], 0x7632),
                   __byte_perm(w[4], w[5], 0x7632), __byte_perm(w[6], w[7], 0x7632));
    *reinterpret_cast<uint4*>(m.hi + c * m.ld + r) = x;
    *reinterpret_cast<uint4*>(m.hi + (c + 1) * m.ld + r) = y;
  }
}

// FP32 in two parts, 64 x 64 tiles: a thread turns eight rows of a column, twice.
// Bound by memory: 278,528 x 512 values (1.14 GB moved) in 166 us, 6.9 TB/s; 480 in 32 x 32 tiles with
// two-byte stores, which rows off 16 bytes keep.
__global__ __launch_bounds__(256) void k_transpose_f32(const Turns a) {
  __shared__ __align__(16) float t[64][64];
  int64_t tx, ty;
  const Turn& m = turn_of(a, blockIdx.x, tx, ty);
  const float* in = static_cast<const float*>(m.in);
  const int64_t r0 = ty * 64, c0 = tx * 64;
  const int tid = threadIdx.x;
  float4 v[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t r = r0 + (tid >> 4) + 16 * i, c = c0 + (tid & 15) * 4;
    v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < m.rows && c < m.cols) v[i] = *reinterpret_cast<const float4*>(in + r * m.cols + c);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = (tid >> 4) + 16 * i;
    *reinterpret_cast<float4*>(&t[row][turn_word(row, (tid & 15) * 4)]) = v[i];
  }
  __syncthreads();
  const int row = (tid & 7) * 8;
  const int64_t r = r0 + row;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int col = (tid >> 3) + 32 * i;
    const int64_t c = c0 + col;
    if (c >= m.cols) return;
    __align__(16) __nv_bfloat16 h[8], l[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float x = t[row + k][turn_word(row, col)];
      h[k] = __float2bfloat16_rn(x);
      l[k] = __float2bfloat16_rn(x - __bfloat162float(h[k]));
    }
    *reinterpret_cast<uint4*>(m.hi + c * m.ld + r) = *reinterpret_cast<const uint4*>(h);
    *reinterpret_cast<uint4*>(m.lo + c * m.ld + r) = *reinterpret_cast<const uint4*>(l);
  }
}

// ---------------------------------------------------------------- staged copies
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// ---------------------------------------------------------------- G = A V on the CUDA cores
// G[i] = sum_p wU[p, i] V[p N_v + j(i, p)]: every (query view, shape) entry adds one
// row of V, so the product has N_v times fewer multiply-adds than the dense one-hot
// GEMM. A block owns 256 query views x 128 columns (16 warps of 16 views, 4 columns
// per lane, accumulators in registers) and walks the shapes in ascending order. A
// step stages, in shared memory, the rows of up to 64 database views restricted to the
// block's columns together with the entry records of the block's query views in those
// shapes: a row of V leaves L2 once per block instead of once per entry, and each entry
// is one broadcast record read, one 512-byte shared-memory read and four multiply-adds.
// The stages are a ring of four to six, filled by one thread of a 17th warp (a TMA tile of
// V and a bulk copy per shape's records) and freed warp by warp, so the warps drift apart
// and none issues copies: what is left is the 512-byte reads (137 GB at full size, 16,384 x 4,096
// entries of 512 columns: 3.4 ms at shared memory's rate), the records' and the copies' share of
// it, and their issue: 7.41 ms with copies by every thread and a barrier per step, 5.75 now.
// A step is up to kGShapes whole shapes of at most 64 views together, or one 64-view piece of a larger shape. The
// steps may be split into parts (blockIdx.z) whose partial sums k_tangent adds in
// part order: the result does not depend on the launch.
constexpr int kGWarps = 16, kGT = 32 * (kGWarps + 1), kGRows = 256, kGCols = 128, kGViews = 64, kGShapes = 8;
constexpr int kGRecOff = (kGViews + 1) * kGCols * 4;  // 33,280: V rows + one zero row, then records [shapes][kGRows]
constexpr int kGSmem = 227 * 1024;
static_assert(kGRecOff % 128 == 0, "stage alignment");
// bytes of a stage and stages of the ring for steps of `shapes` record rows
__host__ __device__ constexpr int g_stage_bytes(int shapes) { return kGRecOff + shapes * kGRows * 8; }
__host__ __device__ constexpr int g_stages(int shapes) { return (kGSmem - 1024) / g_stage_bytes(shapes); }
constexpr int kGStages = g_stages(1);  // the most: barriers a constant apart (5.75 ms; 6.35 with 8 * ring)

struct GatherSteps {
  int spc;  // whole shapes per step (N_v <= 64); 0: 64-view pieces of one shape
  int nch;  // pieces per shape (N_v > 64)
  int n;    // steps
};

// entry record of (query view i, shape p) for the gather: the weight wU and
//  - whole-shape steps (spc > 0): the staged row of the argmax view in float4
//    units, ((p mod spc) N_v + j) * 32, or the zero row kGViews * 32 (weight 0)
//    when the entry has no argmax;
//  - 64-view pieces (spc = 0): the argmax view j, or -1.
__device__ __forceinline__ float2 g_record(int spc, int64_t p, int nv, int j, float wu) {
  if (spc > 0) return make_float2(wu, __int_as_float(j >= 0 ? ((int)(p % spc) * nv + j) * 32 : kGViews * 32));
  return make_float2(wu, __int_as_float(j));
}

// shapes [p0, p0 + nps) and database views [vb, vb + nvs) of step s
__device__ __forceinline__ void g_step(const GatherSteps& st, int s, int nv, int Np, int& p0, int& nps, int64_t& vb,
                                       int& nvs) {
  if (st.spc > 0) {
    p0 = s * st.spc;
    nps = min(st.spc, Np - p0);
    vb = (int64_t)p0 * nv;
    nvs = nps * nv;
  } else {
    p0 = s / st.nch;
    const int ch = s - p0 * st.nch;
    nps = 1;
    vb = (int64_t)p0 * nv + ch * kGViews;
    nvs = min(kGViews, nv - ch * kGViews);
  }
}

// one entry: acc += w * staged row
__device__ __forceinline__ void g_add(float (&acc)[4], float w, const float4 x) {
  acc[0] = fmaf(w, x.x, acc[0]);
  acc[1] = fmaf(w, x.y, acc[1]);
  acc[2] = fmaf(w, x.z, acc[2]);
  acc[3] = fmaf(w, x.w, acc[3]);
}

// tmV: V [nr, dout] in boxes of 64 rows x 128 columns; gR: [Np, ldq] entry records (ldq a multiple of kGRows; no
// entry past nq); Gp: [parts, nq, dout]; every wait is bounded, and gives up once err is set
__global__ __launch_bounds__(kGT, 1) void k_gather_views(const __grid_constant__ CUtensorMap tmV,
                                                         const float2* __restrict__ gR, int64_t nq, int64_t ldq, int Np,
                                                         int nv, int dout, GatherSteps st, float* __restrict__ Gp,
                                                         int* err) {
  extern __shared__ __align__(128) uint8_t g_raw[];
  uint8_t* g_sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(g_raw) + 127) & ~uintptr_t(127));
  const int shapes = st.spc > 0 ? st.spc : 1;
  const int bytes = g_stage_bytes(shapes), ring = g_stages(shapes);
  uint64_t* bars = reinterpret_cast<uint64_t*>(g_sm + (size_t)ring * bytes);
  const uint32_t full0 = tc::smem_u32(bars), empty0 = full0 + 8 * kGStages;
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int64_t i0 = (int64_t)blockIdx.x * kGRows;
  const int c0 = blockIdx.y * kGCols;
  const int part = blockIdx.z, parts = gridDim.z;
  const int s0 = (int)((int64_t)st.n * part / parts), s1 = (int)((int64_t)st.n * (part + 1) / parts);
  for (int t = tid; t < ring * 32; t += kGT)  // the zero row of every stage (never a copy target)
    *reinterpret_cast<float4*>(g_sm + (size_t)(t >> 5) * bytes + kGViews * kGCols * 4 + (t & 31) * 16) =
        make_float4(0.f, 0.f, 0.f, 0.f);
  if (tid == 0) {
    for (int k = 0; k < ring; ++k) {
      tc::mbar_init(full0 + 8 * k, 1);
      tc::mbar_init(empty0 + 8 * k, kGWarps);
    }
    tc::fence_barrier_init();
  }
  __syncthreads();
  int stage = 0;
  uint32_t phase = 0;
  if (w == kGWarps) {
    if (lane == 0) {
      tc::prefetch_tmap(&tmV);
      bool ok = true;
      int issued = 0;
      for (int s = s0; s < s1; ++s) {
        if (!tc::mbar_wait(empty0 + 8 * stage, phase ^ 1, err, tc::kErrProducer)) {
          ok = false;
          break;
        }
        int p0, nps, nvs;
        int64_t vb;
        g_step(st, s, nv, Np, p0, nps, vb, nvs);
        const uint32_t buf = tc::smem_u32(g_sm + (size_t)stage * bytes), bar = full0 + 8 * stage;
        tc::mbar_expect_tx(bar, kGViews * kGCols * 4 + nps * kGRows * 8);
        tc::tma_load_2d(buf, &tmV, c0, (int)vb, bar);  // (rows past the step's are staged and not read)
        for (int ps = 0; ps < nps; ++ps)
          tc::bulk_load(buf + kGRecOff + ps * kGRows * 8, gR + (int64_t)(p0 + ps) * ldq + i0, kGRows * 8, bar);
        ++issued;
        if (++stage == ring) {
          stage = 0;
          phase ^= 1;
        }
      }
      if (!ok && issued) {  // let issued copies land before exiting (bounded)
        const long long t0 = clock64();
        while (clock64() - t0 < tc::kWaitCycles / 4) {
        }
      }
    }
    return;
  }
  float acc[16][4];
#pragma unroll
  for (int k = 0; k < 16; ++k)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[k][q] = 0.f;
  bool whole = true;
  for (int s = s0; s < s1; ++s) {
    if (!tc::mbar_wait(full0 + 8 * stage, phase, err, tc::kErrEpilogue)) {
      whole = false;
      break;
    }
    const uint8_t* buf = g_sm + (size_t)stage * bytes;
    const float4* vs = reinterpret_cast<const float4*>(buf) + lane;
    int p0, nps, nvs;
    int64_t vb;
    g_step(st, s, nv, Np, p0, nps, vb, nvs);
    for (int ps = 0; ps < nps; ++ps) {
      // the warp's 16 records, two per 16-byte broadcast read
      const float4* rp = reinterpret_cast<const float4*>(buf + kGRecOff + (ps * kGRows + 16 * w) * 8);
      if (st.spc > 0) {  // the record holds the staged row: no test
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 r = rp[q];
          g_add(acc[2 * q], r.x, vs[__float_as_int(r.y)]);
          g_add(acc[2 * q + 1], r.z, vs[__float_as_int(r.w)]);
        }
      } else {  // 64-view piece of a shape: the argmax view must fall inside it
        const int base = (int)((int64_t)p0 * nv - vb);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float4 r = rp[q];
          const int l0 = base + __float_as_int(r.y), l1 = base + __float_as_int(r.w);
          if ((unsigned)l0 < (unsigned)nvs) g_add(acc[2 * q], r.x, vs[l0 * 32]);
          if ((unsigned)l1 < (unsigned)nvs) g_add(acc[2 * q + 1], r.z, vs[l1 * 32]);
        }
      }
    }
    __syncwarp();
    if (lane == 0) tc::mbar_arrive(empty0 + 8 * stage);
    if (++stage == ring) {
      stage = 0;
      phase ^= 1;
    }
  }
  if (!whole && lane == 0) report_wait(err);
  const int c = c0 + 4 * lane;
  if (c >= dout) return;
  if (!whole) {  // partial sums do not pass for whole ones
    for (int64_t i = i0 + 16 * w; i < min(nq, i0 + 16 * w + 16); ++i)
      *reinterpret_cast<float4*>(Gp + ((int64_t)part * nq + i) * dout + c) = make_float4(NAN, NAN, NAN, NAN);
    return;
  }
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int64_t i = i0 + 16 * w + k;
    if (i < nq)
      *reinterpret_cast<float4*>(Gp + ((int64_t)part * nq + i) * dout + c) =
          make_float4(acc[k][0], acc[k][1], acc[k][2], acc[k][3]);
  }
}

// shape-major argmax and one-hot weights, rows padded to ldq: for every (query view i,
// shape p), j = argmax[i, p], the gather record of wU = c / |v_{p nv + j}| (g_record)
// and wV = c / |u_i|, with c = grad_S[b, p] / |V(x_b)|; j = -1 (no entry, zero
// weights) for an argmax outside [0, N_v) and for the padding views nq <= i < ldq
__global__ void k_onehot_prep(const int16_t* __restrict__ argmax, int64_t nq, int64_t ldq, int Np, int nv, int spc,
                              const int32_t* __restrict__ vquery, const float* __restrict__ vcoef,
                              const float* __restrict__ gS, const float* __restrict__ vinv,
                              const float* __restrict__ uinv, int16_t* __restrict__ amT, float2* __restrict__ gR,
                              float* __restrict__ wV) {
  __shared__ int16_t t[32][33];
  const int64_t p0 = (int64_t)blockIdx.x * 32, i0 = (int64_t)blockIdx.y * 32;
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int64_t i = i0 + k, p = p0 + threadIdx.x;
    if (i < nq && p < Np) t[k][threadIdx.x] = argmax[i * Np + p];
  }
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int64_t p = p0 + k, i = i0 + threadIdx.x;
    if (i >= ldq || p >= Np) continue;
    const int j = i < nq ? (int)t[threadIdx.x][k] : -1;
    const int64_t e = p * ldq + i;
    if (j < 0 || j >= nv) {
      amT[e] = -1;
      gR[e] = g_record(spc, p, nv, -1, 0.f);
      wV[e] = 0.f;
      continue;
    }
    const float c = gS[(int64_t)vquery[i] * Np + p] * vcoef[i];
    amT[e] = (int16_t)j;
    gR[e] = g_record(spc, p, nv, j, c * vinv[p * nv + j]);
    wV[e] = c * uinv[i];
  }
}

// out_r = inv_r (g_r - (g_r . x_r inv_r) x_r inv_r): the gradient through x / |x| (warp per
// row), for the rows of U and V in one launch; g_r is the sum of `parts` partial rows
// G[s pstride + r dout], added in part order. hi / lo (optional): the result's two-part copy.
struct Tangent {
  const float* x;
  const float* inv;
  const float* g;
  int parts;
  int64_t pstride, n;
  float* out;
  __nv_bfloat16* hi;
  __nv_bfloat16* lo;
};
struct Tangents {
  Tangent m[2];
};
// VW: elements per read, 4 where every row is 16-byte aligned
template <int VW>
struct VecOf;
template <>
struct VecOf<1> {
  typedef float F;
  typedef __nv_bfloat16 H;
};
template <>
struct VecOf<4> {
  typedef float4 F;
  typedef uint2 H;
};
template <int VW>
__global__ __launch_bounds__(256) void k_tangent(const Tangents a, int dout) {
  typedef typename VecOf<VW>::F F;
  typedef typename VecOf<VW>::H H;
  int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const bool second = r >= a.m[0].n;
  const Tangent m = second ? a.m[1] : a.m[0];
  if (second) r -= a.m[0].n;
  if (r >= m.n) return;
  const float iv = m.inv[r];
  const F* x = reinterpret_cast<const F*>(m.x + r * dout);
  const F* g = reinterpret_cast<const F*>(m.g + r * dout);
  const int64_t ps = m.pstride / VW;
  const int n = dout / VW;
  auto load = [&](const F* p, float (&v)[VW]) {
    const F f = *p;
#pragma unroll
    for (int c = 0; c < VW; ++c) v[c] = reinterpret_cast<const float*>(&f)[c];
  };
  auto g_at = [&](int i, float (&v)[VW]) {
    load(g + i, v);
    for (int s = 1; s < m.parts; ++s) {
      float w[VW];
      load(g + s * ps + i, w);
#pragma unroll
      for (int c = 0; c < VW; ++c) v[c] += w[c];
    }
  };
  constexpr int kHeld = 16 / VW;  // reads held per lane: dout up to 512 reads everything once
  float held[kHeld][VW], xs[kHeld][VW];
  float dot = 0.f;
#pragma unroll
  for (int k = 0; k < kHeld; ++k)
    if (lane + 32 * k < n) {
      g_at(lane + 32 * k, held[k]);
      load(x + lane + 32 * k, xs[k]);
    }
#pragma unroll
  for (int k = 0; k < kHeld; ++k)
    if (lane + 32 * k < n)
#pragma unroll
      for (int c = 0; c < VW; ++c) dot = fmaf(xs[k][c], held[k][c], dot);
  for (int i = lane + 32 * kHeld; i < n; i += 32) {
    float gv[VW], xv[VW];
    g_at(i, gv);
    load(x + i, xv);
#pragma unroll
    for (int c = 0; c < VW; ++c) dot = fmaf(xv[c], gv[c], dot);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
  const float t = dot * iv * iv;
  auto put = [&](int i, const float (&gv)[VW], const float (&xv)[VW]) {
    F f;
    H hv, lv;
#pragma unroll
    for (int c = 0; c < VW; ++c) {
      const float v = iv * (gv[c] - t * xv[c]);
      reinterpret_cast<float*>(&f)[c] = v;
      const __nv_bfloat16 h = __float2bfloat16_rn(v);
      reinterpret_cast<__nv_bfloat16*>(&hv)[c] = h;
      reinterpret_cast<__nv_bfloat16*>(&lv)[c] = __float2bfloat16_rn(v - __bfloat162float(h));
    }
    reinterpret_cast<F*>(m.out + r * dout)[i] = f;
    if (m.hi) {
      reinterpret_cast<H*>(m.hi + r * dout)[i] = hv;
      reinterpret_cast<H*>(m.lo + r * dout)[i] = lv;
    }
  };
#pragma unroll
  for (int k = 0; k < kHeld; ++k)
    if (lane + 32 * k < n) put(lane + 32 * k, held[k], xs[k]);
  for (int i = lane + 32 * kHeld; i < n; i += 32) {
    float gv[VW], xv[VW];
    g_at(i, gv);
    load(x + i, xv);
    put(i, gv, xv);
  }
}

// query of each view and 1 / |V(x_b)|
__global__ void k_view_query(const int32_t* __restrict__ qoff, int32_t* __restrict__ vq, float* __restrict__ coef) {
  const int b = blockIdx.x;
  const int v0 = qoff[b], v1 = qoff[b + 1];
  for (int v = v0 + threadIdx.x; v < v1; v += blockDim.x) {
    vq[v] = b;
    coef[v] = 1.f / (float)(v1 - v0);
  }
}

// ---------------------------------------------------------------- H = A^T U on the CUDA cores
// Every database view's row of H is the weighted sum of the query views whose
// argmax in its shape is that view:
//   H[p N_v + j] = sum_{i : j(i, p) = j} wV[p, i] U[i]
// (N_v times fewer multiply-adds than the dense one-hot GEMM), summed in ascending
// query view order: a result that does not depend on the launch.
//
// Shapes of up to 1,024 views: the entries of each shape are grouped by their argmax
// view (a counting sort per shape in shared memory), then one warp per database view
// sums its entries' rows of U, gathered from L2 (U is L2-resident).
// Larger shapes (the sort's per-warp counts would not fit in shared memory): a block
// owns 256 database views (flattened; at most kHShapes shapes, N_v >= 16) x 128
// columns, warp w the 16 views from 16 w on, 4 columns per lane with the accumulators
// in registers. A step stages 64 query views' rows of U (the column slice) and the
// argmax and weight of those query views in the block's shapes (cp.async, three
// stages); a warp finds the query views of each of its database views with two
// ballots over the staged argmax and adds their staged rows.
constexpr int kHT = 512, kHRows = 256, kHQ = 64, kHStages = 3, kHShapes = 18;
constexpr int kHMinNv = 16;                                  // kHRows / kHMinNv + 2 <= kHShapes
constexpr int kHAmOff = kHQ * kGCols * 4;                    // 32,768: argmax [kHShapes][kHQ] int16
constexpr int kHWOff = kHAmOff + kHShapes * kHQ * 2;         // 35,072: weight [kHShapes][kHQ] float
constexpr int kHStageBytes = kHWOff + kHShapes * kHQ * 4;    // 39,680
static_assert(kHStageBytes % 16 == 0 && kHWOff % 16 == 0, "stage alignment");
static_assert(kHRows / kHMinNv + 2 <= kHShapes, "shapes of one block");

// amT, wV: [Np, ldq] (ldq a multiple of kHQ; argmax -1 past nq); U: [nq, dout]
// (16-byte aligned, dout % 4 == 0); H: [nr, dout]
__global__ __launch_bounds__(kHT, 1) void k_gather_entries(const float* __restrict__ U, const int16_t* __restrict__ amT,
                                                           const float* __restrict__ wV, int64_t nq, int64_t ldq,
                                                           int64_t nr, int nv, int dout, float* __restrict__ H) {
  extern __shared__ __align__(16) uint8_t h_sm[];
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int64_t r0 = (int64_t)blockIdx.x * kHRows;
  const int c0 = blockIdx.y * kGCols;
  const int64_t ps0 = r0 / nv;
  const int ns = (int)((min(r0 + kHRows, nr) - 1) / nv - ps0 + 1);  // shapes of the block (<= kHShapes)
  const int nsteps = (int)cdiv(nq, (int64_t)kHQ);
  auto issue = [&](int s) {
    if (s < nsteps) {
      uint8_t* buf = h_sm + (s % kHStages) * kHStageBytes;
      const int64_t i0 = (int64_t)s * kHQ;
      for (int t = tid; t < kHQ * 32; t += kHT) {  // rows of U, 16-byte pieces of the column slice
        const int row = t >> 5, q = t & 31, c = c0 + 4 * q;
        if (c < dout && i0 + row < nq) cp_async16(buf + (row * kGCols + 4 * q) * 4, U + (i0 + row) * dout + c);
      }
      for (int t = tid; t < ns * 24; t += kHT) {  // per shape: 8 pieces of argmax, 16 of weight
        const int ps = t / 24, q = t - ps * 24;
        const int64_t e = (ps0 + ps) * ldq + i0;
        if (q < 8)
          cp_async16(buf + kHAmOff + (ps * kHQ + 8 * q) * 2, amT + e + 8 * q);
        else
          cp_async16(buf + kHWOff + (ps * kHQ + 4 * (q - 8)) * 4, wV + e + 4 * (q - 8));
      }
    }
    cp_async_commit();  // empty groups past the last step keep the wait count uniform
  };
  // shape and view of the warp's first database view
  const int64_t rw = r0 + 16 * w;
  const int pw0 = (int)(rw / nv - ps0), jw0 = (int)(rw % nv);
  float acc[16][4];
#pragma unroll
  for (int k = 0; k < 16; ++k)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[k][q] = 0.f;
#pragma unroll
  for (int k = 0; k < kHStages - 1; ++k) issue(k);
  for (int s = 0; s < nsteps; ++s) {
    cp_async_wait<kHStages - 2>();  // this step's copies have landed ...
    __syncthreads();                // ... for every thread, and the step before is done with its buffer
    issue(s + kHStages - 1);
    const uint8_t* buf = h_sm + (s % kHStages) * kHStageBytes;
    const float4* us = reinterpret_cast<const float4*>(buf);
    const int16_t* as = reinterpret_cast<const int16_t*>(buf + kHAmOff);
    const float* ws = reinterpret_cast<const float*>(buf + kHWOff);
    int ps = pw0, j = jw0, cur = -1;
    int ja = -1, jb = -1;
    float wa = 0.f, wb = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      if (rw + k < nr) {  // uniform over the warp
        if (ps != cur) {  // lane l holds query views l and l + 32 of the step
          cur = ps;
          ja = as[ps * kHQ + lane];
          jb = as[ps * kHQ + 32 + lane];
          wa = ws[ps * kHQ + lane];
          wb = ws[ps * kHQ + 32 + lane];
        }
        unsigned m = __ballot_sync(0xffffffffu, ja == j);
        while (m) {
          const int l = __ffs(m) - 1;
          m &= m - 1;
          const float wk = __shfl_sync(0xffffffffu, wa, l);
          const float4 x = us[l * 32 + lane];
          acc[k][0] = fmaf(wk, x.x, acc[k][0]);
          acc[k][1] = fmaf(wk, x.y, acc[k][1]);
          acc[k][2] = fmaf(wk, x.z, acc[k][2]);
          acc[k][3] = fmaf(wk, x.w, acc[k][3]);
        }
        m = __ballot_sync(0xffffffffu, jb == j);
        while (m) {
          const int l = __ffs(m) - 1;
          m &= m - 1;
          const float wk = __shfl_sync(0xffffffffu, wb, l);
          const float4 x = us[(l + 32) * 32 + lane];
          acc[k][0] = fmaf(wk, x.x, acc[k][0]);
          acc[k][1] = fmaf(wk, x.y, acc[k][1]);
          acc[k][2] = fmaf(wk, x.z, acc[k][2]);
          acc[k][3] = fmaf(wk, x.w, acc[k][3]);
        }
      }
      if (++j == nv) {
        j = 0;
        ++ps;
      }
    }
  }
  cp_async_wait<0>();
  const int c = c0 + 4 * lane;
  if (c >= dout) return;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int64_t r = rw + k;
    if (r < nr)
      *reinterpret_cast<float4*>(H + r * dout + c) = make_float4(acc[k][0], acc[k][1], acc[k][2], acc[k][3]);
  }
}

// The entries of shape p grouped by their argmax view j, ascending query view within a
// group (a stable counting sort, one block per shape): perm[p ld + ...] holds the entry
// indices e = p ld + i, beg[p N_v + j] the first position of view j's group and
// cnt[p N_v + j] its size; entries without an argmax (j = -1) are left out. Shared
// memory: 32 x N_v per-warp counts and N_v running group ends.
constexpr int kCsrT = 1024;
constexpr int kCsrMaxNv = 1024;  // 33 x 1024 ints of shared memory
static_assert(kCsrMaxNv >= kHMinNv, "the staged gather takes the larger shapes");
__global__ __launch_bounds__(kCsrT) void k_onehot_csr(const int16_t* __restrict__ amT, int64_t nq, int64_t ld,
                                                      int nv,
                                                      int32_t* __restrict__ perm, int64_t* __restrict__ beg,
                                                      int32_t* __restrict__ cnt) {
  extern __shared__ int csr_sm[];
  int* wc = csr_sm;            // [32][nv]
  int* base = csr_sm + 32 * nv;  // [nv]
  const int p = blockIdx.x, t = threadIdx.x, w = t >> 5, lane = t & 31;
  const int16_t* a = amT + (int64_t)p * ld;
  const int64_t e0 = (int64_t)p * ld;
  for (int j = t; j < nv; j += kCsrT) base[j] = 0;
  __syncthreads();
  for (int64_t i = t; i < nq; i += kCsrT) {
    const int j = a[i];
    if (j >= 0 && j < nv) atomicAdd(&base[j], 1);
  }
  __syncthreads();
  if (t == 0) {  // exclusive prefix over the views (N_v steps)
    int run = 0;
    for (int j = 0; j < nv; ++j) {
      const int c = base[j];
      cnt[(int64_t)p * nv + j] = c;
      beg[(int64_t)p * nv + j] = e0 + run;
      base[j] = run;
      run += c;
    }
  }
  __syncthreads();
  for (int64_t c0 = 0; c0 < nq; c0 += kCsrT) {
    const int64_t i = c0 + t;
    int j = -1;
    if (i < nq) {
      j = a[i];
      if (j < 0 || j >= nv) j = -1;
    }
    for (int k = t; k < 32 * nv; k += kCsrT) wc[k] = 0;
    __syncthreads();
    const unsigned peers = __match_any_sync(0xffffffffu, j);
    const int rank = __popc(peers & ((1u << lane) - 1u));  // earlier lanes of this warp with view j
    if (j >= 0 && rank == 0) wc[w * nv + j] = __popc(peers);
    __syncthreads();
    for (int v = t; v < nv; v += kCsrT) {  // per view: the warps' starts, in warp order
      int run = base[v];
      for (int w2 = 0; w2 < 32; ++w2) {
        const int c = wc[w2 * nv + v];
        wc[w2 * nv + v] = run;
        run += c;
      }
      base[v] = run;
    }
    __syncthreads();
    if (j >= 0) perm[e0 + wc[w * nv + j] + rank] = (int32_t)(e0 + i);
    __syncthreads();  // before the counts are cleared for the next chunk
  }
}

// H[r] = sum of wV[e] U[e mod ld] over the entries e of row r (perm[beg[r]] ..
// perm[beg[r] + cnt[r]]), in ascending e: one warp per database view, lane c owns columns
// 4 c + 128 t, up to kHCols columns per pass (dout % 4 == 0)
template <int kHCols, int kAhead>
__global__ __launch_bounds__(256) void k_segment_rows_sum(const float* __restrict__ U, const int32_t* __restrict__ perm,
                                                          const int64_t* __restrict__ beg,
                                                          const int32_t* __restrict__ cnt,
                                                          const float* __restrict__ wT, int64_t ld, int64_t nr,
                                                          int dout, float* __restrict__ H) {
  const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= nr) return;
  constexpr int kT = kHCols / 128;  // float4 pieces per lane and pass
  const int64_t e0 = beg[r], e1 = e0 + cnt[r];
  for (int cb = 0; cb < dout; cb += kHCols) {
    float acc[kT][4];
#pragma unroll
    for (int t = 0; t < kT; ++t)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[t][q] = 0.f;
    for (int64_t eb = e0; eb < e1; eb += 32) {
      const int n = (int)min((int64_t)32, e1 - eb);
      int64_t src = 0;
      float wl = 0.f;
      if (lane < n) {
        const int32_t e = perm[eb + lane];
        src = (int64_t)(e % ld) * dout;
        wl = wT[e];
      }
#pragma unroll(kAhead)
      for (int k = 0; k < n; ++k) {  // unrolled: several entries' row loads in flight
        const int64_t sk = __shfl_sync(0xffffffffu, src, k);
        const float wk = __shfl_sync(0xffffffffu, wl, k);
        const float* u = U + sk + cb;
#pragma unroll
        for (int t = 0; t < kT; ++t) {
          const int c = 4 * lane + 128 * t;
          if (cb + c < dout) {
            const float4 x = *reinterpret_cast<const float4*>(u + c);
            acc[t][0] = fmaf(wk, x.x, acc[t][0]);
            acc[t][1] = fmaf(wk, x.y, acc[t][1]);
            acc[t][2] = fmaf(wk, x.z, acc[t][2]);
            acc[t][3] = fmaf(wk, x.w, acc[t][3]);
          }
        }
      }
    }
#pragma unroll
    for (int t = 0; t < kT; ++t) {
      const int c = 4 * lane + 128 * t;
      if (cb + c < dout)
        *reinterpret_cast<float4*>(H + r * dout + cb + c) = make_float4(acc[t][0], acc[t][1], acc[t][2], acc[t][3]);
    }
  }
}

// two-part BF16 operand with one TMA box of padding rows
struct Operand {
  __nv_bfloat16* hi = nullptr;
  __nv_bfloat16* lo = nullptr;  // null: one-part (exact BF16 input)
  int64_t rows_alloc = 0;
};

// several: matrices whose split is left to be launched together (launch_splits)
Operand make_operand(const void* x, int dtype, int64_t rows, int cols, Split4s& several, Scratch& sc, cudaStream_t s) {
  Operand o;
  if (dtype != GIFT_F32 && rows >= tc::kTM && reinterpret_cast<uintptr_t>(x) % 16 == 0) {
    // a BF16 input is its own one-part operand: the tensor map covers its rows
    o.hi = const_cast<__nv_bfloat16*>(static_cast<const __nv_bfloat16*>(x));
    o.rows_alloc = rows;
    return o;
  }
  o.rows_alloc = rows + 128;
  const int64_t n = rows * cols;
  o.hi = sc.get<__nv_bfloat16>((size_t)o.rows_alloc * cols);
  if (dtype == GIFT_F32) o.lo = sc.get<__nv_bfloat16>((size_t)o.rows_alloc * cols);
  const bool vec = dtype == GIFT_F32 && n % 4 == 0 && reinterpret_cast<uintptr_t>(x) % 16 == 0 &&
                   reinterpret_cast<uintptr_t>(o.hi) % 8 == 0 && reinterpret_cast<uintptr_t>(o.lo) % 8 == 0;
  if (vec) {
    several.m[several.n] = Split4{static_cast<const float4*>(x), reinterpret_cast<uint2*>(o.hi),
                                  reinterpret_cast<uint2*>(o.lo),
                                  n / 4 + (several.n ? several.m[several.n - 1].end : 0)};
    ++several.n;
    return o;
  }
  if (dtype == GIFT_F32)
    k_split_any<float><<<(unsigned)cdiv(n, 256), 256, 0, s>>>(static_cast<const float*>(x), n, o.hi, o.lo);
  else
    k_split_any<__nv_bfloat16><<<(unsigned)cdiv(n, 256), 256, 0, s>>>(static_cast<const __nv_bfloat16*>(x), n,
                                                                        o.hi, o.lo);
  GIFT_LAUNCHED("k_split_any");
  return o;
}

void launch_splits(const Split4s& several, cudaStream_t s) {
  if (!several.n) return;
  const int64_t n4 = several.m[several.n - 1].end;
  const unsigned grid = (unsigned)std::min<int64_t>(cdiv(n4, 256), (int64_t)device_sm_count() * 16);
  k_split4<<<grid, 256, 0, s>>>(several);
  GIFT_LAUNCHED("k_split4");
}

// transposed operands: out [cols, ld] with ld = rows rounded up to 64; two-part
// for FP32 input, one-part (lo null) for BF16 input, which BF16 holds exactly
struct Transposes {
  Turns f32, bf16, wide_f32, wide;  // FP32 inputs, BF16 inputs, both in 16-byte pieces
  Operand add(const void* x, int dtype, int64_t rows, int64_t cols, int64_t& ld, Scratch& sc) {
    Operand o;
    ld = cdiv(rows, 64) * 64;
    o.rows_alloc = cols + 128;
    o.hi = sc.get<__nv_bfloat16>((size_t)o.rows_alloc * ld);
    if (dtype == GIFT_F32) o.lo = sc.get<__nv_bfloat16>((size_t)o.rows_alloc * ld);
    const bool one = dtype != GIFT_F32;
    const bool pieces = cols % (one ? 8 : 4) == 0 && reinterpret_cast<uintptr_t>(x) % 16 == 0 &&
                        reinterpret_cast<uintptr_t>(o.hi) % 16 == 0 && reinterpret_cast<uintptr_t>(o.lo) % 16 == 0;
    Turns& t = pieces ? (one ? wide : wide_f32) : one ? bf16 : f32;
    const int64_t tx = cdiv(cols, pieces ? 64 : 32), ty = cdiv(ld, !pieces ? 32 : one ? 128 : 64);
    t.m[t.n] = Turn{x, rows, cols, ld, o.hi, o.lo, tx, tx * ty + (t.n ? t.m[t.n - 1].end : 0)};
    ++t.n;
    return o;
  }
  static unsigned blocks(const Turns& t) {
    const int64_t n = t.m[t.n - 1].end;
    GIFT_REQUIRE(n < (int64_t)INT32_MAX, "too many views for the weight gradient");
    return (unsigned)n;
  }
  void launch(cudaStream_t s) const {
    if (f32.n) {
      k_transpose_split<float><<<blocks(f32), dim3(32, 8), 0, s>>>(f32);
      GIFT_LAUNCHED("k_transpose_split");
    }
    if (bf16.n) {
      k_transpose_split<__nv_bfloat16><<<blocks(bf16), dim3(32, 8), 0, s>>>(bf16);
      GIFT_LAUNCHED("k_transpose_split");
    }
    if (wide_f32.n) {
      k_transpose_f32<<<blocks(wide_f32), 256, 0, s>>>(wide_f32);
      GIFT_LAUNCHED("k_transpose_f32");
    }
    if (wide.n) {
      k_transpose_bf16<<<blocks(wide), 256, 0, s>>>(wide);
      GIFT_LAUNCHED("k_transpose_bf16");
    }
  }
};

float* as_float(const void* x, int dtype, int64_t n, Scratch& sc, cudaStream_t s) {
  if (dtype == GIFT_F32) return const_cast<float*>(static_cast<const float*>(x));
  float* f = sc.get<float>((size_t)n);
  k_to_float<__nv_bfloat16><<<(unsigned)cdiv(n, 256), 256, 0, s>>>(static_cast<const __nv_bfloat16*>(x), n, f);
  GIFT_LAUNCHED("k_to_float");
  return f;
}

struct Proj {
  float* U;
  float* V;
  float* uinv;
  float* vinv;
  Operand Uo, Vo;  // two-part copies (forward)
};

// inverse norms of the rows of U and V, and their two-part copies where hi is given; warp per row, both matrices in one
// launch (sums as k_row_invnorm's)
struct NormRows {
  const float* x[2];
  int64_t n[2];
  float* inv[2];
  __nv_bfloat16* hi[2];
  __nv_bfloat16* lo[2];
};
template <bool PARTS>
__global__ __launch_bounds__(256) void k_norm_rows(const NormRows a, int D) {
  int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const int m = row >= a.n[0] ? 1 : 0;
  if (m) row -= a.n[0];
  if (row >= a.n[m]) return;
  const float4* p = reinterpret_cast<const float4*>(a.x[m] + row * (int64_t)D);
  uint2* h = reinterpret_cast<uint2*>(a.hi[m] + row * (int64_t)D);
  uint2* l = reinterpret_cast<uint2*>(a.lo[m] + row * (int64_t)D);
  float acc = 0.f;
#pragma unroll 4
  for (int i = lane; i < (D >> 2); i += 32) {
    const float4 v = p[i];
    acc = fmaf(v.x, v.x, acc);
    acc = fmaf(v.y, v.y, acc);
    acc = fmaf(v.z, v.z, acc);
    acc = fmaf(v.w, v.w, acc);
    if (!PARTS) continue;
    const __nv_bfloat162 a2 = __floats2bfloat162_rn(v.x, v.y), b2 = __floats2bfloat162_rn(v.z, v.w);
    const float2 fa = __bfloat1622float2(a2), fb = __bfloat1622float2(b2);
    const __nv_bfloat162 c2 = __floats2bfloat162_rn(v.x - fa.x, v.y - fa.y);
    const __nv_bfloat162 d2 = __floats2bfloat162_rn(v.z - fb.x, v.w - fb.y);
    h[i] = make_uint2(*reinterpret_cast<const uint32_t*>(&a2), *reinterpret_cast<const uint32_t*>(&b2));
    l[i] = make_uint2(*reinterpret_cast<const uint32_t*>(&c2), *reinterpret_cast<const uint32_t*>(&d2));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) a.inv[m][row] = acc > 0.f ? 1.0f / sqrtf(acc) : 0.f;
}

Proj project(const void* q, int64_t nq, const void* p, int64_t nr, const void* W, int din, int dout, int dtype,
             bool parts, int* err, Scratch& sc, cudaStream_t s) {
  Proj P;
  if (W) {
    Split4s several;
    const Operand Qo = make_operand(q, dtype, nq, din, several, sc, s);
    const Operand Po = make_operand(p, dtype, nr, din, several, sc, s);
    const Operand Wo = make_operand(W, dtype, dout, din, several, sc, s);
    launch_splits(several, s);
    P.U = sc.get<float>((size_t)nq * dout);
    P.V = sc.get<float>((size_t)nr * dout);
    gemm_tc(Qo.hi, Qo.lo, nq, Qo.rows_alloc, 0, Wo.hi, Wo.lo, dout, Wo.rows_alloc, 0, din, P.U, dout, 0, err, s);
    gemm_tc(Po.hi, Po.lo, nr, Po.rows_alloc, 0, Wo.hi, Wo.lo, dout, Wo.rows_alloc, 0, din, P.V, dout, 0, err, s);
  } else {
    P.U = as_float(q, dtype, nq * din, sc, s);
    P.V = as_float(p, dtype, nr * din, sc, s);
  }
  P.uinv = sc.get<float>(nq);
  P.vinv = sc.get<float>(nr);
  NormRows nr2{{P.U, P.V}, {nq, nr}, {P.uinv, P.vinv}, {nullptr, nullptr}, {nullptr, nullptr}};
  if (parts) {
    Operand* o[2] = {&P.Uo, &P.Vo};
    for (int m = 0; m < 2; ++m) {
      o[m]->rows_alloc = nr2.n[m] + 128;
      o[m]->hi = nr2.hi[m] = sc.get<__nv_bfloat16>((size_t)o[m]->rows_alloc * dout);
      o[m]->lo = nr2.lo[m] = sc.get<__nv_bfloat16>((size_t)o[m]->rows_alloc * dout);
    }
  }
  if (parts)
    k_norm_rows<true><<<(unsigned)cdiv(nq + nr, 8), 256, 0, s>>>(nr2, dout);
  else
    k_norm_rows<false><<<(unsigned)cdiv(nq + nr, 8), 256, 0, s>>>(nr2, dout);
  GIFT_LAUNCHED("k_norm_rows");
  return P;
}

// the call's wait flag and its offsets behind it, in one copy
int* device_head(const std::vector<int32_t>& h_qoff, int32_t*& d_qoff, Scratch& sc, cudaStream_t s) {
  const WaitFlag f{0, 0, thread_wait_word()};
  constexpr size_t n = sizeof(WaitFlag) / 4;
  std::vector<int32_t> h(n + h_qoff.size());
  memcpy(h.data(), &f, sizeof(f));
  std::copy(h_qoff.begin(), h_qoff.end(), h.begin() + n);
  int32_t* d = sc.get<int32_t>(h.size());
  GIFT_CUDA(cudaMemcpyAsync(d, h.data(), h.size() * 4, cudaMemcpyHostToDevice, s));  // (pageable: taken before the return)
  d_qoff = d + n;
  return d;
}

}  // namespace

void match_forward(const void* q, const std::vector<int32_t>& h_qoff, int32_t Bq, const void* p, int32_t Np,
                   int32_t nv, const void* W, int32_t din, int32_t dout, int32_t dtype, float* S, int16_t* argmax,
                   Scratch& sc, cudaStream_t s) {
  const int64_t nq = h_qoff[Bq];
  const int64_t nr = (int64_t)Np * nv;
  int32_t* d_qoff = nullptr;
  int* err = device_head(h_qoff, d_qoff, sc, s);
  const Proj P = project(q, nq, p, nr, W, din, dout, dtype, true, err, sc, s);
  segmax_tc(P.Uo.hi, P.Uo.lo, P.Uo.rows_alloc, P.uinv, P.Vo.hi, P.Vo.lo, P.Vo.rows_alloc, P.vinv, nr, nv, dout, d_qoff, h_qoff,
            Bq, S, argmax, err, sc, s);
}

void match_backward(const void* q, const std::vector<int32_t>& h_qoff, int32_t Bq, const void* p, int32_t Np,
                    int32_t nv, const void* W, int32_t din, int32_t dout, int32_t dtype, const float* gS,
                    const int16_t* argmax, float* dW, float* dQ, float* dP, Scratch& sc, cudaStream_t s) {
  const int64_t nq = h_qoff[Bq];
  const int64_t nr = (int64_t)Np * nv;
  int32_t* d_qoff = nullptr;
  int* err = device_head(h_qoff, d_qoff, sc, s);
  const Proj P = project(q, nq, p, nr, W, din, dout, dtype, false, err, sc, s);
  int32_t* vquery = sc.get<int32_t>(nq);
  float* vcoef = sc.get<float>(nq);
  k_view_query<<<(unsigned)Bq, 128, 0, s>>>(d_qoff, vquery, vcoef);
  GIFT_LAUNCHED("k_view_query");
  // gradients w.r.t. the projected views (without a projection these are dQ, dP)
  float* dU = (W || !dQ) ? sc.get<float>((size_t)nq * dout) : dQ;
  float* dV = (W || !dP) ? sc.get<float>((size_t)nr * dout) : dP;
  // steps of the query-side gather
  GatherSteps st;
  if (nv <= kGViews) {
    st.spc = std::min(kGShapes, kGViews / nv);
    st.nch = 1;
    st.n = (int)cdiv((int64_t)Np, (int64_t)st.spc);
  } else {
    st.spc = 0;
    st.nch = (int)cdiv((int64_t)nv, (int64_t)kGViews);
    GIFT_REQUIRE((int64_t)Np * st.nch < INT32_MAX, "too many database views for the gradient");
    st.n = Np * st.nch;
  }
  // shape-major argmax, gather records and weights, query views padded to a multiple of the gather blocks
  const int64_t ldq = cdiv(nq, (int64_t)kGRows) * kGRows;
  int16_t* amT = sc.get<int16_t>((size_t)ldq * Np);
  float2* gR = sc.get<float2>((size_t)ldq * Np);
  float* wV = sc.get<float>((size_t)ldq * Np);
  k_onehot_prep<<<dim3((unsigned)cdiv(Np, 32), (unsigned)cdiv(ldq, 32)), dim3(32, 8), 0, s>>>(
      argmax, nq, ldq, Np, nv, st.spc, vquery, vcoef, gS, P.vinv, P.uinv, amT, gR, wV);
  GIFT_LAUNCHED("k_onehot_prep");
  GIFT_REQUIRE(dout % 4 == 0, "projected width must be a multiple of 4");
  // the staged copies read 16-byte pieces of the rows of U and V
  auto aligned16 = [&](float* x, int64_t n) {
    if (reinterpret_cast<uintptr_t>(x) % 16 == 0) return x;
    float* y = sc.get<float>((size_t)n);
    GIFT_CUDA(cudaMemcpyAsync(y, x, (size_t)n * sizeof(float), cudaMemcpyDeviceToDevice, s));
    return y;
  };
  const float* U16 = aligned16(P.U, nq * dout);
  const float* V16 = aligned16(P.V, nr * dout);
  const int sms = device_sm_count();
  Tangents tg;
  {  // G = A V
    // parts of the step range: a block's time is ~ steps / parts, the launch takes
    // ceil(blocks x parts / SMs) rounds of one block per SM; partial rows cost a little
    const int64_t units = cdiv(nq, (int64_t)kGRows) * cdiv((int64_t)dout, (int64_t)kGCols);
    // (in microseconds: 1.1 a step, and a part's row written and read twice at 4 TB/s, or its reads' latency)
    int parts = 1;
    double best = 1e30;
    const double part_us = std::max(1.0, (double)nq * dout * 12 / 4e6);
    for (int pc = 1; pc <= 64 && pc <= st.n; ++pc) {
      const double cost = 1.1 * (double)cdiv(units * pc, (int64_t)sms) * st.n / pc + part_us * pc;
      if (cost < best - 1e-9) {
        best = cost;
        parts = pc;
      }
    }
    float* Gp = sc.get<float>((size_t)parts * nq * dout);
    GIFT_CUDA(cudaFuncSetAttribute(k_gather_views, cudaFuncAttributeMaxDynamicSharedMemorySize, kGSmem));
    const dim3 grid((unsigned)cdiv(nq, (int64_t)kGRows), (unsigned)cdiv((int64_t)dout, (int64_t)kGCols),
                    (unsigned)parts);
    const CUtensorMap tmV = make_tmap_f32(V16, nr, dout, kGCols, kGViews);
    k_gather_views<<<grid, kGT, kGSmem, s>>>(tmV, gR, nq, ldq, Np, nv, dout, st, Gp, err);
    GIFT_LAUNCHED("k_gather_views");
    tg.m[0] = Tangent{P.U, P.uinv, Gp, parts, nq * dout, nq, dU, nullptr, nullptr};
  }
  {  // H = A^T U
    float* H = sc.get<float>((size_t)nr * dout);
    if (nv <= kCsrMaxNv) {  // entries grouped per shape, then one warp per database view
      const int64_t ne = ldq * (int64_t)Np;
      GIFT_REQUIRE(ne < (int64_t)INT32_MAX, "query views x database shapes must stay below 2^31 for the gradient");
      int32_t* perm = sc.get<int32_t>((size_t)ne);
      int64_t* beg = sc.get<int64_t>((size_t)nr);
      int32_t* cnt = sc.get<int32_t>((size_t)nr);
      const size_t smem = (size_t)33 * nv * sizeof(int);
      GIFT_CUDA(cudaFuncSetAttribute(k_onehot_csr, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      k_onehot_csr<<<(unsigned)Np, kCsrT, smem, s>>>(amT, nq, ldq, nv, perm, beg, cnt);
      GIFT_LAUNCHED("k_onehot_csr");
      // (a view that many query views prefer is one warp's chain of reads: narrow rows keep more of them in flight)
      if (dout <= 128)
        k_segment_rows_sum<128, 16><<<(unsigned)cdiv(nr, (int64_t)8), 256, 0, s>>>(U16, perm, beg, cnt, wV, ldq, nr, dout, H);
      else
        k_segment_rows_sum<512, 4><<<(unsigned)cdiv(nr, (int64_t)8), 256, 0, s>>>(U16, perm, beg, cnt, wV, ldq, nr, dout, H);
      GIFT_LAUNCHED("k_segment_rows_sum");
    } else {  // larger shapes: the staged gather
      const size_t smem = (size_t)kHStages * kHStageBytes;
      GIFT_CUDA(cudaFuncSetAttribute(k_gather_entries, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      const dim3 grid((unsigned)cdiv(nr, (int64_t)kHRows), (unsigned)cdiv((int64_t)dout, (int64_t)kGCols));
      k_gather_entries<<<grid, kHT, smem, s>>>(U16, amT, wV, nq, ldq, nr, nv, dout, H);
      GIFT_LAUNCHED("k_gather_entries");
    }
    tg.m[1] = Tangent{P.V, P.vinv, H, 1, 0, nr, dV, nullptr, nullptr};
  }
  // through the normalisation; the gradients that dQ and dP multiply leave as two parts too
  Operand dUo, dVo;
  auto two_parts = [&](Operand& o, Tangent& t) {
    o.rows_alloc = t.n + 128;
    o.hi = t.hi = sc.get<__nv_bfloat16>((size_t)o.rows_alloc * dout);
    o.lo = t.lo = sc.get<__nv_bfloat16>((size_t)o.rows_alloc * dout);
  };
  if (W && dQ) two_parts(dUo, tg.m[0]);
  if (W && dP) two_parts(dVo, tg.m[1]);
  bool wide = true;  // (d_out is a multiple of 16)
  for (const Tangent& t : tg.m)
    for (const void* ptr : {(const void*)t.x, (const void*)t.g, (const void*)t.out})
      wide = wide && reinterpret_cast<uintptr_t>(ptr) % 16 == 0;
  if (wide)
    k_tangent<4><<<(unsigned)cdiv(nq + nr, 8), 256, 0, s>>>(tg, dout);
  else
    k_tangent<1><<<(unsigned)cdiv(nq + nr, 8), 256, 0, s>>>(tg, dout);
  GIFT_LAUNCHED("k_tangent");
  if (!W) return;
  Transposes turns;
  int64_t ldt = 0, ldr = 0, ldo = 0;
  Operand dUt, Qt, dVt, Pt, Wt;
  if (dW) {
    dUt = turns.add(dU, GIFT_F32, nq, dout, ldt, sc);
    Qt = turns.add(q, dtype, nq, din, ldt, sc);
    dVt = turns.add(dV, GIFT_F32, nr, dout, ldr, sc);
    Pt = turns.add(p, dtype, nr, din, ldr, sc);
  }
  if (dQ || dP) Wt = turns.add(W, dtype, dout, din, ldo, sc);  // [din, ldo], K = dout
  turns.launch(s);
  if (dW) {
    gemm_tc(dUt.hi, dUt.lo, dout, dUt.rows_alloc, ldt, Qt.hi, Qt.lo, din, Qt.rows_alloc, ldt, (int)ldt, dW, din, 0,
            err, s, &sc);
    gemm_tc(dVt.hi, dVt.lo, dout, dVt.rows_alloc, ldr, Pt.hi, Pt.lo, din, Pt.rows_alloc, ldr, (int)ldr, dW, din, 1,
            err, s, &sc);
  }
  if (dQ)
    gemm_tc(dUo.hi, dUo.lo, nq, dUo.rows_alloc, dout, Wt.hi, Wt.lo, din, Wt.rows_alloc, ldo, dout, dQ, din, 0, err, s);
  if (dP)
    gemm_tc(dVo.hi, dVo.lo, nr, dVo.rows_alloc, dout, Wt.hi, Wt.lo, din, Wt.rows_alloc, ldo, dout, dP, din, 0, err, s);
}

}  // namespace gift
