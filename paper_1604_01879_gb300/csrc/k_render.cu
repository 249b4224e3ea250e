// Projection front end (Sec. 2.1): scale and translation normalisation of
// every mesh, then N_v = n_az * n_el depth-buffer views from cameras on the
// unit sphere, each looking at the origin.
//
// Normalisation: the area-weighted centroid of the surface goes to the origin
// (two-float FP32 sums, one block per mesh) and the largest vertex distance
// from it becomes 1. Views: orthographic along the camera's forward axis f, image axes
// r = f x z / |f x z| and u = r x f, the image spanning [-1, 1]^2 (the unit
// sphere's silhouette); depth = p . f + 1 in [0, 2], 2 where nothing is seen.
// A triangle is projected, the pixel centres of its bounding box are tested, those
// with all three edge functions >= 0 (orientation made positive; degenerate
// triangles cover nothing) are kept, and the interpolated depth is written with
// atomicMin on the float bits (non-negative floats order like their bit patterns):
// in shared memory, band by band of the image, or in global memory (band_plan).
#include <cmath>
#include <cstring>

#include "gift_internal.cuh"
#include "tc_common.cuh"

namespace gift {

namespace {

constexpr int kRenderT = 256;

__device__ __forceinline__ int find_mesh(const int64_t* __restrict__ off, int M, int64_t t) {
  int lo = 0, hi = M;  // off[lo] <= t < off[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (off[mid] <= t) lo = mid; else hi = mid;
  }
  return lo;
}

// per mesh: (cx, cy, cz) = sum(area * centroid) / sum(area); per-triangle terms
// in FP32, sums in two-float arithmetic (no FP64 on the GPU)
__global__ __launch_bounds__(kRenderT) void k_mesh_centre(const float* __restrict__ V, const int32_t* __restrict__ T,
                                                          const int64_t* __restrict__ voff,
                                                          const int64_t* __restrict__ toff, float* __restrict__ centre) {
  const int m = blockIdx.x;
  const float* Vm = V + voff[m] * 3;
  F2 acc[4];
  for (int64_t t = toff[m] + threadIdx.x; t < toff[m + 1]; t += blockDim.x) {
    const int32_t* tr = T + t * 3;
    float a[3], b[3], c[3];
    for (int d = 0; d < 3; ++d) {
      a[d] = Vm[(int64_t)tr[0] * 3 + d];
      b[d] = Vm[(int64_t)tr[1] * 3 + d];
      c[d] = Vm[(int64_t)tr[2] * 3 + d];
    }
    const float e1[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
    const float e2[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
    const float cx = e1[1] * e2[2] - e1[2] * e2[1];
    const float cy = e1[2] * e2[0] - e1[0] * e2[2];
    const float cz = e1[0] * e2[1] - e1[1] * e2[0];
    const float area = 0.5f * sqrtf(cx * cx + cy * cy + cz * cz);
    for (int d = 0; d < 3; ++d) f2_add(acc[d], area * ((a[d] + b[d] + c[d]) * (1.f / 3.f)));
    f2_add(acc[3], area);
  }
  __shared__ F2 red[4][kRenderT / 32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int k = 0; k < 4; ++k) {
    F2 x = acc[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = f2_merge(x, f2_shfl_xor(x, o));
    if (lane == 0) red[k][w] = x;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    F2 tot[4];
    for (int k = 0; k < 4; ++k)
      for (int i = 0; i < kRenderT / 32; ++i) tot[k] = f2_merge(tot[k], red[k][i]);
    const float A = f2_value(tot[3]);
    for (int d = 0; d < 3; ++d) centre[m * 4 + d] = A > 0.f ? __fdiv_rn(f2_value(tot[d]), A) : 0.f;
  }
}

// per mesh: scale = 1 / max_v |v - centre|
__global__ __launch_bounds__(kRenderT) void k_mesh_scale(const float* __restrict__ V, const int64_t* __restrict__ voff,
                                                         float* __restrict__ centre) {
  const int m = blockIdx.x;
  const float c0 = centre[m * 4], c1 = centre[m * 4 + 1], c2 = centre[m * 4 + 2];
  float mx = 0.f;
  for (int64_t v = voff[m] + threadIdx.x; v < voff[m + 1]; v += blockDim.x) {
    const float dx = V[v * 3] - c0, dy = V[v * 3 + 1] - c1, dz = V[v * 3 + 2] - c2;
    mx = fmaxf(mx, dx * dx + dy * dy + dz * dz);
  }
  __shared__ float red[kRenderT / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    float r = 0.f;
    for (int i = 0; i < kRenderT / 32; ++i) r = fmaxf(r, red[i]);
    centre[m * 4 + 3] = r > 0.f ? 1.f / sqrtf(r) : 1.f;
  }
}

// host: the float of an f2key (0: -infinity)
inline float key_value(uint32_t k) {
  const uint32_t u = k & 0x80000000u ? k & 0x7fffffffu : ~k;
  float f;
  memcpy(&f, &u, 4);
  return k ? f : -INFINITY;
}

// A mesh's triangles, as the host needs them to choose how to draw it (all zero: none). The box of a triangle
// shows, on average over all directions, a third of dx dy + dy dz + dz dx.
struct MeshFacts {
  float boxes;                // the triangles' sum
  float largest;              // and their largest
  uint32_t high[3], low[3];   // f2key of the largest coordinates, and of the largest of the negated ones
};

// every vertex index must address its own mesh's vertices; facts [M] (zeroed)
__global__ __launch_bounds__(kRenderT) void k_check_tris(const float* __restrict__ V, const int32_t* __restrict__ T,
                                                         const int64_t* __restrict__ voff,
                                                         const int64_t* __restrict__ toff, int M,
                                                         MeshFacts* __restrict__ facts, int* __restrict__ bad) {
  __shared__ MeshFacts part[kRenderT / 32];
  __shared__ int s_first;
  const int64_t t = (int64_t)blockIdx.x * kRenderT + threadIdx.x;
  const int m = t < toff[M] ? find_mesh(toff, M, t) : -1;
  MeshFacts f{};
  if (m >= 0) {
    const int64_t nv = voff[m + 1] - voff[m];
    const float* Vm = V + voff[m] * 3;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    bool ok = true;
    for (int k = 0; k < 3; ++k) {
      const int32_t i = T[t * 3 + k];
      if (i < 0 || i >= nv) {
        ok = false;
        continue;
      }
      for (int d = 0; d < 3; ++d) {
        const float x = Vm[(int64_t)i * 3 + d];
        lo[d] = fminf(lo[d], x);
        hi[d] = fmaxf(hi[d], x);
      }
    }
    if (ok) {
      const float d0 = hi[0] - lo[0], d1 = hi[1] - lo[1], d2 = hi[2] - lo[2];
      f.boxes = f.largest = d0 * d1 + d1 * d2 + d2 * d0;
      for (int d = 0; d < 3; ++d) {
        f.high[d] = f2key(hi[d]);
        f.low[d] = f2key(-lo[d]);
      }
    } else {
      atomicExch(bad, 1);
    }
  }
  auto add = [&](MeshFacts& to) {
    atomicAdd(&to.boxes, f.boxes);
    atomicMax(reinterpret_cast<int*>(&to.largest), __float_as_int(f.largest));  // (not negative)
    for (int d = 0; d < 3; ++d) {
      atomicMax(&to.high[d], f.high[d]);
      atomicMax(&to.low[d], f.low[d]);
    }
  };
  auto join = [&](const MeshFacts& o) {
    f.boxes += o.boxes;
    f.largest = fmaxf(f.largest, o.largest);
    for (int d = 0; d < 3; ++d) {
      f.high[d] = max(f.high[d], o.high[d]);
      f.low[d] = max(f.low[d], o.low[d]);
    }
  };
  // one thread adds for a block whose triangles are all of one mesh, else one for each such warp
  const int lane = threadIdx.x & 31;
  const bool warp_one = __all_sync(0xffffffffu, m == __shfl_sync(0xffffffffu, m, 0) || m < 0);
  if (warp_one) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      MeshFacts y;
      y.boxes = __shfl_xor_sync(0xffffffffu, f.boxes, o);
      y.largest = __shfl_xor_sync(0xffffffffu, f.largest, o);
      for (int d = 0; d < 3; ++d) {
        y.high[d] = __shfl_xor_sync(0xffffffffu, f.high[d], o);
        y.low[d] = __shfl_xor_sync(0xffffffffu, f.low[d], o);
      }
      join(y);
    }
    if (lane == 0) part[threadIdx.x >> 5] = f;
  }
  if (threadIdx.x == 0) s_first = m;
  __syncthreads();
  if (!__syncthreads_and(m == s_first || m < 0)) {
    if (m >= 0 && (lane == 0 || !warp_one)) add(facts[m]);
  } else if (threadIdx.x == 0) {
    for (int i = 1; i < kRenderT / 32; ++i) join(part[i]);
    add(facts[m]);
  }
}

__global__ void k_fill_depth(float* __restrict__ p, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = 2.f;
}

// One triangle seen from one view: projected corners (x, y image coordinates, z depth), oriented to a
// positive area; the same arithmetic whichever kernel draws it
struct Tri {
  float x[3], y[3], z[3], area;
};
__device__ __forceinline__ float tri_coord(const float (&p)[3], const float* fr) {
  return p[0] * fr[0] + p[1] * fr[1] + p[2] * fr[2];
}
__device__ __forceinline__ bool tri_orient(Tri& t) {
  t.area = (t.x[1] - t.x[0]) * (t.y[2] - t.y[0]) - (t.y[1] - t.y[0]) * (t.x[2] - t.x[0]);
  if (t.area == 0.f) return false;
  if (t.area < 0.f) {
    const float tx = t.x[1], ty = t.y[1], tz = t.z[1];
    t.x[1] = t.x[2];
    t.y[1] = t.y[2];
    t.z[1] = t.z[2];
    t.x[2] = tx;
    t.y[2] = ty;
    t.z[2] = tz;
    t.area = -t.area;
  }
  return true;
}
// corners of triangle tr of mesh Vm, centred and scaled (frame-independent)
__device__ __forceinline__ void tri_corners(const float* __restrict__ Vm, const int32_t* __restrict__ tr, float c0,
                                            float c1, float c2, float sc, float (&p)[3][3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int64_t vi = tr[k];
    p[k][0] = (Vm[vi * 3] - c0) * sc;
    p[k][1] = (Vm[vi * 3 + 1] - c1) * sc;
    p[k][2] = (Vm[vi * 3 + 2] - c2) * sc;
  }
}
// pixel columns (rows) that may lie in [lo, hi]: centres x_j = -1 + (2j + 1) / n
__device__ __forceinline__ int px_first(float lo, int n) { return max(0, (int)ceilf((lo + 1.f) * 0.5f * n - 0.5f) - 1); }
__device__ __forceinline__ int px_last(float hi, int n) {
  return min(n - 1, (int)floorf((hi + 1.f) * 0.5f * n - 0.5f) + 1);
}
__device__ __forceinline__ int py_first(float hi, int n) { return max(0, (int)ceilf((1.f - hi) * 0.5f * n - 0.5f) - 1); }
__device__ __forceinline__ int py_last(float lo, int n) {
  return min(n - 1, (int)floorf((1.f - lo) * 0.5f * n - 0.5f) + 1);
}
// an edge function dx (py - y) - dy (px - x) from the first product (the same along a row), rounded by itself
__device__ __forceinline__ float edge(float row, float dy, float px, float x) { return __fmaf_rn(-dy, px - x, row); }
// two FP32 values in one 64-bit register: add, multiply and fused multiply-add of both by one instruction
// each, rounded as the scalar ones are
typedef unsigned long long f2x;
__device__ __forceinline__ f2x f2_pack(float a, float b) {
  f2x r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_unpack(f2x v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2x f2x_add(f2x a, f2x b) {
  f2x r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2x f2x_mul(f2x a, f2x b) {
  f2x r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2x f2x_fma(f2x a, f2x b, f2x c) {
  f2x r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Every triangle's corners, centred and scaled, as nine planes of one float per triangle: the blocks of a mesh's
// images read them in whole lines, instead of three indices and nine gathered coordinates per triangle and band
__global__ __launch_bounds__(kRenderT) void k_tri_planes(const float* __restrict__ V, const int32_t* __restrict__ T,
                                                         const int64_t* __restrict__ voff,
                                                         const int64_t* __restrict__ toff, int M,
                                                         const float* __restrict__ cs, float* __restrict__ C) {
  const int64_t total = toff[M], t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= total) return;
  const int m = find_mesh(toff, M, t);
  float p[3][3];
  tri_corners(V + voff[m] * 3, T + t * 3, cs[m * 4], cs[m * 4 + 1], cs[m * 4 + 2], cs[m * 4 + 3], p);
#pragma unroll
  for (int k = 0; k < 9; ++k) C[k * total + t] = p[k / 3][k % 3];
}

// Images by bands in shared memory: a block takes some rows of one (mesh, view) image, draws every triangle of
// the mesh that meets them with shared-memory minima, and writes the band once, background included. Triangles
// are set up one per thread and queued; once the queue is filled, the pixels of their boxes are dealt out in
// units of kUnit horizontal pairs, so triangles of any size load all threads alike, and warps take their next
// 32 units from a counter. What bounds it is the issue of the edge tests (a box has about three pixels per covered one)
// and the block's barriers between set-ups and pixels, not memory, so a pair is tested with two-wide FP32 instructions:
// counters of 8 such meshes in 32 views, 67% of the issue slots taken with 22 of 32 lanes active, 30% of shared memory's
// wavefronts, a fifth of a warp's stalls at barriers. 64 meshes of 2,208 triangles,
// 64 views of 224 x 224: 1,395 us where a thread per triangle with minima in global memory took 1,865 and a separate
// fill 405; 1,549 with corners gathered per band and a ten-step search per unit. Units of whole rows, clipped to
// the columns between the edges, halve the tested pairs but take 1,484: a warp waits for its longest row. Two
// blocks of 512 threads share an SM, so one's set-up and write-out overlap the other's pixels; the price is that
// each of an image's bands (three at 224 x 224) sets up the mesh again, up to the first test of its y range.
constexpr int kBandT = 512, kUnit = 8;
constexpr int kQueue = 768, kQueueRun = 256;  // the queue is drawn once it holds more than kQueueRun
constexpr int kBandSmem = 112 * 1024;         // two blocks per SM
constexpr int kMostBands = 16;
constexpr int kStep = kQueue / 32;            // a queue's search: 32 parts of kStep, then one of kStep
struct BandQueue {
  float x[3][kQueue], y[3][kQueue], z[3][kQueue], inv[kQueue];
  int box[kQueue];   // first column and width, 16 bits each
  int rows[kQueue];  // first row within the band, and rows
  int pre[kQueue];   // units before this triangle's
  uint32_t wsum[kBandT / 32];
  int next;
};
static_assert(kQueueRun + kBandT <= kQueue, "a round of set-ups fits");
static_assert(kStep * 32 == kQueue && kStep <= 32, "the search ends in two steps");

// row pitch in shared memory: 16-byte rows, an odd multiple of four apart in the 32 banks, so that pixels below one
// another fall in different banks (224 is a multiple of 32)
__host__ __device__ constexpr int band_pitch(int W) { return (W + 3) / 4 * 4 + ((W + 3) / 4 % 2 ? 0 : 4); }
// shared memory of a band of `rows` rows
__host__ __device__ constexpr size_t band_bytes(int rows, int W) {
  return sizeof(BandQueue) + (size_t)(band_pitch(W) + rows + 4) * 4 + (size_t)rows * band_pitch(W) * 4;
}

__global__ __launch_bounds__(kBandT, 2) void k_render_bands(const float* __restrict__ C, const int64_t* __restrict__ toff,
                                                            int M, const float* __restrict__ frames, int Nv, int H,
                                                            int W, int band_rows, int bands,
                                                            float* __restrict__ depth) {
  extern __shared__ __align__(16) uint8_t band_sm[];
  const int pitch = band_pitch(W);
  int* img = reinterpret_cast<int*>(band_sm);                          // [band_rows][pitch], 16-byte rows
  BandQueue& q = *reinterpret_cast<BandQueue*>(img + (size_t)band_rows * pitch);
  float* pxs = reinterpret_cast<float*>(&q + 1);                       // pixel centres (with room past the last)
  float* pys = pxs + pitch;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int band = blockIdx.x % bands;
  const int64_t mv = blockIdx.x / bands;
  const int v = (int)(mv % Nv), m = (int)(mv / Nv);
  const int r0 = band * band_rows, r1 = min(H, r0 + band_rows);
  const int far = __float_as_int(2.f);
  for (int i = tid; i < (r1 - r0) * pitch / 4; i += kBandT)  // whole 16-byte pieces
    reinterpret_cast<int4*>(img)[i] = make_int4(far, far, far, far);
  for (int j = tid; j < W; j += kBandT) pxs[j] = -1.f + (float)(2 * j + 1) / (float)W;
  for (int i = r0 + tid; i < r1; i += kBandT) pys[i - r0] = 1.f - (float)(2 * i + 1) / (float)H;
  const float* fr = frames + v * 9;
  float f[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) f[k] = fr[k];
  const int64_t t1 = toff[m + 1], plane = toff[M];
  int kept = 0, total = 0;  // queued triangles and their units (the same in every thread)
  if (tid == 0) q.next = 0;
  __syncthreads();
  for (int64_t t0 = toff[m]; t0 < t1; t0 += kBandT) {
    Tri t;
    int i0 = 0, i1 = -1, j0 = 0, j1 = -1;
    if (t0 + tid < t1) {
      float p[3][3];
#pragma unroll
      for (int k = 0; k < 9; ++k) p[k / 3][k % 3] = C[k * plane + t0 + tid];
#pragma unroll
      for (int k = 0; k < 3; ++k) t.y[k] = tri_coord(p[k], f + 3);
      const float ymin = fminf(t.y[0], fminf(t.y[1], t.y[2])), ymax = fmaxf(t.y[0], fmaxf(t.y[1], t.y[2]));
      i0 = max(r0, py_first(ymax, H));
      i1 = min(r1 - 1, py_last(ymin, H));
      while (i0 <= i1 && pys[i0 - r0] > ymax) ++i0;
      while (i0 <= i1 && pys[i1 - r0] < ymin) --i1;
      if (i0 <= i1) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          t.x[k] = tri_coord(p[k], f);
          t.z[k] = p[k][0] * f[6] + p[k][1] * f[7] + p[k][2] * f[8] + 1.f;
        }
        if (tri_orient(t)) {
          const float xmin = fminf(t.x[0], fminf(t.x[1], t.x[2])), xmax = fmaxf(t.x[0], fmaxf(t.x[1], t.x[2]));
          j0 = px_first(xmin, W);
          j1 = px_last(xmax, W);
          while (j0 <= j1 && pxs[j0] < xmin) ++j0;
          while (j0 <= j1 && pxs[j1] > xmax) --j1;
        }
      }
    }
    const int width = j1 - j0 + 1, high = i1 - i0 + 1;
    const bool keep = width > 0 && high > 0;
    const uint32_t units = keep ? (uint32_t)(((width + 1) / 2 * high + kUnit - 1) / kUnit) : 0u;
    // kept triangles (high 10 bits: 512 at most) and units (low 22) before this thread's
    const uint32_t own = keep ? (1u << 22) | units : 0u;
    uint32_t x = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) q.wsum[w] = x;
    __syncthreads();
    uint32_t before = 0u, all = 0u;
#pragma unroll
    for (int k = 0; k < kBandT / 32; ++k) {
      const uint32_t s = q.wsum[k];
      if (k < w) before += s;
      all += s;
    }
    if (keep) {
      const uint32_t e = before + x - own;
      const int at = kept + (int)(e >> 22);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        q.x[k][at] = t.x[k];
        q.y[k][at] = t.y[k];
        q.z[k][at] = t.z[k];
      }
      q.inv[at] = 1.f / t.area;
      q.box[at] = j0 | (width << 16);
      q.rows[at] = (i0 - r0) | (high << 16);
      q.pre[at] = total + (int)(e & 0x3fffffu);
    }
    kept += (int)(all >> 22);
    total += (int)(all & 0x3fffffu);
    __syncthreads();
    if (kept <= kQueueRun && t0 + kBandT < t1) continue;
    while (true) {
      int u = 0;
      if (lane == 0) u = atomicAdd(&q.next, 32);
      u = __shfl_sync(0xffffffffu, u, 0);
      if (u >= total) break;
      // the triangle of each of the warp's 32 units: u's by two 32-way steps, then the others' by a bit at each
      // unit that begins a triangle (every queued triangle has one, so 32 of them reach past the last unit)
      int at = lane * kStep;
      uint32_t have = __ballot_sync(0xffffffffu, at < kept && q.pre[at] <= u);
      const int part = (__popc(have) - 1) * kStep;
      at = part + lane;
      have = __ballot_sync(0xffffffffu, lane < kStep && at < kept && q.pre[at] <= u);
      int lo = part + __popc(have) - 1;
      at = lo + 1 + lane;
      const int begins = at < kept ? q.pre[at] - u : 32;
      const uint32_t marks = __reduce_or_sync(0xffffffffu, begins < 32 ? 1u << begins : 0u);
      lo += __popc(marks & (0xffffffffu >> (31 - lane)));
      u += lane;
      if (u >= total) continue;
      const int box = q.box[lo], rw = q.rows[lo];
      const int wd = box >> 16, jf = box & 0xffff, jl = jf + wd - 1, wp = (wd + 1) >> 1;
      const int first = (u - q.pre[lo]) * kUnit;
      const int n = min(kUnit, wp * (rw >> 16) - first);
      // first / wp: both are below 2^15 (a band's pixels), so half a pair keeps the quotient off whole numbers by
      // far more than its error
      const int di = (int)__fdividef((float)first + 0.5f, (float)wp);
      int i = (rw & 0xffff) + di, j = jf + 2 * (first - di * wp);
      const float x0 = q.x[0][lo], x1 = q.x[1][lo], x2 = q.x[2][lo];
      const float y0 = q.y[0][lo], y1 = q.y[1][lo], y2 = q.y[2][lo];
      const f2x nxa = f2_pack(-x1, -x1), nxb = f2_pack(-x2, -x2), nxc = f2_pack(-x0, -x0);
      const f2x nda = f2_pack(y1 - y2, y1 - y2), ndb = f2_pack(y2 - y0, y2 - y0), ndc = f2_pack(y0 - y1, y0 - y1);
      const float ax = x2 - x1, bx = x0 - x2, cx = x1 - x0;
      const float z0 = q.z[0][lo], z1 = q.z[1][lo], z2 = q.z[2][lo], inv = q.inv[lo];
      // the row's products are formed for every pair: lanes change rows at different pairs, so a branch for
      // them would be taken in nearly every step of the warp
      for (int k = 0; k < n; ++k) {
        const f2x px = f2_pack(pxs[j], pxs[j + 1]);
        const float py = pys[i];
        const float ra = __fmul_rn(ax, py - y1), rb = __fmul_rn(bx, py - y2), rc = __fmul_rn(cx, py - y0);
        const f2x ea = f2x_fma(nda, f2x_add(px, nxa), f2_pack(ra, ra));
        const f2x eb = f2x_fma(ndb, f2x_add(px, nxb), f2_pack(rb, rb));
        const f2x ec = f2x_fma(ndc, f2x_add(px, nxc), f2_pack(rc, rc));
        const f2x zz = f2x_mul(f2x_fma(ec, f2_pack(z2, z2), f2x_fma(ea, f2_pack(z0, z0), f2x_mul(eb, f2_pack(z1, z1)))),
                               f2_pack(inv, inv));
        float a0, a1, b0, b1, d0, d1, s0, s1;
        f2_unpack(ea, a0, a1);
        f2_unpack(eb, b0, b1);
        f2_unpack(ec, d0, d1);
        f2_unpack(zz, s0, s1);
        int* at = img + i * pitch + j;
        if (!(fminf(a0, fminf(b0, d0)) < 0.f)) atomicMin(at, __float_as_int(fminf(fmaxf(s0, 0.f), 2.f)));
        if (j < jl && !(fminf(a1, fminf(b1, d1)) < 0.f))
          atomicMin(at + 1, __float_as_int(fminf(fmaxf(s1, 0.f), 2.f)));
        j += 2;
        const bool wrap = j > jl;
        j = wrap ? jf : j;
        i += wrap ? 1 : 0;  // (one past the band after its last pair: pys has room)
      }
    }
    __syncthreads();
    kept = total = 0;
    if (tid == 0) q.next = 0;  // before the next fill's barriers
  }
  __syncthreads();
  float* out = depth + (mv * H + r0) * W;
  if (reinterpret_cast<uintptr_t>(depth) % 16 == 0 && W % 4 == 0) {
    const int w4 = W / 4;
    for (int i = tid; i < (r1 - r0) * w4; i += kBandT)
      __stcs(reinterpret_cast<int4*>(out) + i, *reinterpret_cast<int4*>(img + i / w4 * pitch + i % w4 * 4));
  } else {
    for (int i = tid; i < (r1 - r0) * W; i += kBandT) out[i] = __int_as_float(img[i / W * pitch + i % W]);
  }
}

// thread per (triangle, view); frames [Nv, 9] = (r, u, f): minima in the images in global memory
__global__ __launch_bounds__(kRenderT) void k_render(const float* __restrict__ V, const int32_t* __restrict__ T,
                                                     const int64_t* __restrict__ voff,
                                                     const int64_t* __restrict__ toff, int M,
                                                     const float* __restrict__ cs, const float* __restrict__ frames,
                                                     int Nv, int H, int W, float* __restrict__ depth) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t total = toff[M] * Nv;
  if (idx >= total) return;
  const int v = (int)(idx % Nv);
  const int64_t t = idx / Nv;
  const int m = find_mesh(toff, M, t);
  const float* fr = frames + v * 9;
  Tri tr;
  float p[3][3];
  tri_corners(V + voff[m] * 3, T + t * 3, cs[m * 4], cs[m * 4 + 1], cs[m * 4 + 2], cs[m * 4 + 3], p);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    tr.x[k] = tri_coord(p[k], fr);
    tr.y[k] = tri_coord(p[k], fr + 3);
    tr.z[k] = p[k][0] * fr[6] + p[k][1] * fr[7] + p[k][2] * fr[8] + 1.f;
  }
  if (!tri_orient(tr)) return;
  const float xmin = fminf(tr.x[0], fminf(tr.x[1], tr.x[2])), xmax = fmaxf(tr.x[0], fmaxf(tr.x[1], tr.x[2]));
  const float ymin = fminf(tr.y[0], fminf(tr.y[1], tr.y[2])), ymax = fmaxf(tr.y[0], fmaxf(tr.y[1], tr.y[2]));
  const int j0 = px_first(xmin, W), j1 = px_last(xmax, W), i0 = py_first(ymax, H), i1 = py_last(ymin, H);
  float* img = depth + ((int64_t)m * Nv + v) * H * W;
  const float inv_area = 1.f / tr.area;
  for (int i = i0; i <= i1; ++i) {
    const float py = 1.f - (float)(2 * i + 1) / (float)H;
    if (py < ymin || py > ymax) continue;
    const float ra = __fmul_rn(tr.x[2] - tr.x[1], py - tr.y[1]);
    const float rb = __fmul_rn(tr.x[0] - tr.x[2], py - tr.y[2]);
    const float rc = __fmul_rn(tr.x[1] - tr.x[0], py - tr.y[0]);
    for (int j = j0; j <= j1; ++j) {
      const float px = -1.f + (float)(2 * j + 1) / (float)W;
      if (px < xmin || px > xmax) continue;
      const float ea = edge(ra, tr.y[2] - tr.y[1], px, tr.x[1]);
      const float eb = edge(rb, tr.y[0] - tr.y[2], px, tr.x[2]);
      const float ec = edge(rc, tr.y[1] - tr.y[0], px, tr.x[0]);
      if (ea < 0.f || eb < 0.f || ec < 0.f) continue;
      const float z = fminf(fmaxf((ea * tr.z[0] + eb * tr.z[1] + ec * tr.z[2]) * inv_area, 0.f), 2.f);
      atomicMin(reinterpret_cast<int*>(img + (int64_t)i * W + j), __float_as_int(z));
    }
  }
}

// Rows of a band and bands of an image: as many rows as shared memory holds, fewer where the images would not
// give every SM two blocks (but at least 16). False: the images are drawn in global memory. That is for images of more
// than kMostBands bands, and for meshes of many small triangles, which every band sets up anew: 13 ps a triangle,
// image and band, or a block's 2.9 us per 512 triangles where few blocks run, against 26 ps a triangle and image. Global
// memory costs 1.7 ps more per pixel of a triangle's box (beyond the first few), 80 ns a pixel for the largest one's
// thread, and the fill. Measured, closed surfaces, whole calls in us (bands, global): 512 images of 224 x 224 in
// 3 bands, 1,680 triangles 451 and 609, 9,408: 707 and 728, 28,560: 1,250 and 999; of 512 x 512 in 14 bands, 9,408:
// 1,789 and 1,955, 98,000: 8,868 and 3,458; 64 of 224 x 224, 1,680: 304 and 323, 9,408: 381 and 326, 397,000: 3,220 and
// 1,375.
bool band_plan(const std::vector<int64_t>& toff, int M, int Nv, int H, int W, const std::vector<MeshFacts>& facts,
               int& rows, int& bands) {
  const int64_t sms = device_sm_count(), images = (int64_t)M * Nv;
  int fit = 0;
  while (fit < H && band_bytes(fit + 1, W) <= (size_t)kBandSmem) ++fit;
  if (fit == 0) return false;
  bands = (int)cdiv(H, fit);
  if (bands > kMostBands) return false;
  const int64_t want = std::min<int64_t>(cdiv(2 * sms, images), std::max(1, H / 16));
  bands = std::max(bands, (int)std::min<int64_t>(want, kMostBands));
  rows = (int)cdiv(H, bands);
  bands = (int)cdiv(H, rows);
  if (images * bands >= INT32_MAX) return false;
  int64_t most = 0;  // triangles of the largest mesh
  double boxes = 0., largest = 0.;  // of meshes scaled to radius 1
  for (int m = 0; m < M; ++m) {
    most = std::max(most, toff[m + 1] - toff[m]);
    double r2 = 0.;  // the radius squared: a third of this for a ball's extents, all of it for a box's or a rod's
    for (int d = 0; d < 3; ++d) {
      const double e = key_value(facts[m].high[d]) + key_value(facts[m].low[d]);
      r2 += e * e / 4;
    }
    r2 *= 0.4;
    if (toff[m + 1] == toff[m] || r2 <= 0.) continue;
    boxes += facts[m].boxes / r2;
    largest = std::max(largest, facts[m].largest / r2);
  }
  const double seen = (double)toff[M] * Nv, image = (double)H * W;  // (the image spans 2 x 2)
  const double tested = boxes / 3 / std::max<int64_t>(toff[M], 1) * image / 4;
  const double band_us = std::max(13e-6 * bands * seen, 2.9 / 512 * most);
  const double global_us = 26e-6 * seen +
                           std::max(1.7e-6 * seen * std::max(0., tested - 5), 80e-3 * largest / 3 * image / 4) +
                           1.35e-6 * images * image + 2;
  return band_us < global_us;
}

}  // namespace

void render_views(const float* V, const int32_t* T, const std::vector<int64_t>& h_voff,
                  const std::vector<int64_t>& h_toff, int M, int n_az, int n_el, int H, int W, float* depth,
                  Scratch& sc, cudaStream_t s) {
  const int Nv = n_az * n_el;
  // camera frames in float64 on the host: r, u, f per view (view = el_index * n_az + az_index)
  std::vector<float> fr((size_t)Nv * 9);
  for (int je = 0; je < n_el; ++je)
    for (int ia = 0; ia < n_az; ++ia) {
      const double az = 2.0 * M_PI * ia / n_az;
      const double el = M_PI * ((je + 0.5) / n_el - 0.5);
      const double f[3] = {-cos(el) * cos(az), -cos(el) * sin(az), -sin(el)};
      double r[3] = {f[1], -f[0], 0.0};  // f x (0, 0, 1)
      const double rn = sqrt(r[0] * r[0] + r[1] * r[1]);
      r[0] /= rn;
      r[1] /= rn;
      const double u[3] = {r[1] * f[2] - r[2] * f[1], r[2] * f[0] - r[0] * f[2], r[0] * f[1] - r[1] * f[0]};
      float* o = fr.data() + (size_t)(je * n_az + ia) * 9;
      for (int d = 0; d < 3; ++d) {
        o[d] = (float)r[d];
        o[3 + d] = (float)u[d];
        o[6 + d] = (float)f[d];
      }
    }
  // frames and offsets in one copy
  const size_t n_off = (size_t)M + 1;
  std::vector<int64_t> head(2 * n_off + (fr.size() + 1) / 2);
  std::copy(h_voff.begin(), h_voff.end(), head.begin());
  std::copy(h_toff.begin(), h_toff.end(), head.begin() + n_off);
  std::copy(fr.begin(), fr.end(), reinterpret_cast<float*>(head.data() + 2 * n_off));
  int64_t* voff = sc.get<int64_t>(head.size());
  GIFT_CUDA(cudaMemcpyAsync(voff, head.data(), head.size() * 8, cudaMemcpyHostToDevice, s));
  const int64_t* toff = voff + n_off;
  const float* d_fr = reinterpret_cast<const float*>(voff + 2 * n_off);
  std::vector<MeshFacts> h_facts((size_t)M + 1);  // the last one's first word: an index was out of range
  if (h_toff[M] > 0) {
    MeshFacts* facts = sc.get<MeshFacts>(h_facts.size());
    GIFT_CUDA(cudaMemsetAsync(facts, 0, h_facts.size() * sizeof(MeshFacts), s));
    k_check_tris<<<(unsigned)cdiv(h_toff[M], kRenderT), kRenderT, 0, s>>>(V, T, voff, toff, M, facts,
                                                                          reinterpret_cast<int*>(facts + M));
    GIFT_LAUNCHED("k_check_tris");
    GIFT_CUDA(cudaMemcpyAsync(h_facts.data(), facts, h_facts.size() * sizeof(MeshFacts), cudaMemcpyDeviceToHost, s));
    GIFT_CUDA(cudaStreamSynchronize(s));
    int bad;
    memcpy(&bad, &h_facts[M], sizeof(int));
    if (bad) fail(GIFT_EINVAL, "a triangle addresses a vertex outside its mesh");
  }
  float* cs = sc.get<float>((size_t)M * 4);
  k_mesh_centre<<<(unsigned)M, kRenderT, 0, s>>>(V, T, voff, toff, cs);
  GIFT_LAUNCHED("k_mesh_centre");
  k_mesh_scale<<<(unsigned)M, kRenderT, 0, s>>>(V, voff, cs);
  GIFT_LAUNCHED("k_mesh_scale");
  const int64_t images = (int64_t)M * Nv;
  int rows = 0, bands = 0;
  if (band_plan(h_toff, M, Nv, H, W, h_facts, rows, bands)) {
    GIFT_CUDA(cudaFuncSetAttribute(k_render_bands, cudaFuncAttributeMaxDynamicSharedMemorySize, kBandSmem));
    float* corners = sc.get<float>((size_t)h_toff[M] * 9);
    if (h_toff[M] > 0) {
      k_tri_planes<<<(unsigned)cdiv(h_toff[M], kRenderT), kRenderT, 0, s>>>(V, T, voff, toff, M, cs, corners);
      GIFT_LAUNCHED("k_tri_planes");
    }
    k_render_bands<<<(unsigned)(images * bands), kBandT, band_bytes(rows, W), s>>>(corners, toff, M, d_fr, Nv, H, W, rows,
                                                                                  bands, depth);
    GIFT_LAUNCHED("k_render_bands");
    return;
  }
  const int64_t npix = images * H * W;
  k_fill_depth<<<(unsigned)cdiv(npix, 256), 256, 0, s>>>(depth, npix);
  GIFT_LAUNCHED("k_fill_depth");
  const int64_t work = h_toff[M] * Nv;
  if (work > 0) {
    k_render<<<(unsigned)cdiv(work, kRenderT), kRenderT, 0, s>>>(V, T, voff, toff, M, cs, d_fr, Nv, H, W, depth);
    GIFT_LAUNCHED("k_render");
  }
}

}  // namespace gift
