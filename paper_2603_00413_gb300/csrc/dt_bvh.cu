// Geometry kernels: vertex normals (DiffTrans Sec. 3.4, Eq. 13) and their
// backward, and the LBVH (Morton codes, a stable LSD radix sort, the Karras
// 2012 hierarchy, bottom-up bounds, and from them the nodes that the traversal
// reads), with a binned SAH builder beside it.
#include <cuda_runtime.h>
#include <stdint.h>

#include "dt_internal.cuh"
#include "dt_shade.cuh"

namespace dt {

extern dt_tuning g_tuning;

// ---------------------------------------------------------------------------
// Eq. 13: N_v = (1/3) sum_{f containing v} unit((v1 - v0) x (v2 - v0)).
// One thread per face adds its unit normal, in 2^-40 fixed point, to its
// three vertices with 64-bit integer atomics: integer addition is
// associative, so the sums -- and every ray that depends on them -- are the
// same bits on every run whatever order the atomics land in.  A second pass
// converts to float and applies the 1/3.  Both conversions are FP32: the
// scale is a power of two, so u * 2^40 is exact in float (|u| <= 1) and the
// integer is u's value rounded to 2^-40; the finish rounds the sum to float
// once and divides by 3 with IEEE rounding.
// ---------------------------------------------------------------------------
constexpr float kNormalFix = 0x1p40f;
constexpr float kNormalUnfix = 0x1p-40f;

__global__ void k_face_normals_scatter(const float* __restrict__ V, const int32_t* __restrict__ F, int32_t nf,
                                       unsigned long long* __restrict__ acc) {
  for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += gridDim.x * blockDim.x) {
    const int i0 = F[3 * f], i1 = F[3 * f + 1], i2 = F[3 * f + 2];
    const float3 v0 = load3(V + 3 * i0), v1 = load3(V + 3 * i1), v2 = load3(V + 3 * i2);
    const float3 c = cross_rn(v1 - v0, v2 - v0);
    const float lc = len(c);
    if (!(lc > 0.0f)) continue;  // a zero-area face has no unit normal and adds nothing
    const float3 u = mk(c.x / lc, c.y / lc, c.z / lc);
    const long long q[3] = {__float2ll_rn(u.x * kNormalFix), __float2ll_rn(u.y * kNormalFix),
                            __float2ll_rn(u.z * kNormalFix)};
    const int idx[3] = {i0, i1, i2};
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int c = 0; c < 3; ++c) atomicAdd(acc + 3 * (size_t)idx[k] + c, (unsigned long long)q[c]);
  }
}

__global__ void k_normals_finish(const unsigned long long* acc, int64_t n3, float* __restrict__ N) {
  chain_begin();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n3; i += (int64_t)gridDim.x * blockDim.x)
    N[i] = __fdiv_rn(__ll2float_rn((long long)acc[i]) * kNormalUnfix, 3.0f);
}

__global__ void k_face_normals_backward(const float* __restrict__ V, const int32_t* __restrict__ F, int32_t nf,
                                        const float* __restrict__ dN, float* __restrict__ dV) {
  for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += gridDim.x * blockDim.x)
    face_normal_backward_one(V, F, f, dN, dV);
}

size_t normals_scratch_bytes(int32_t nv) { return align_up((size_t)nv * 3 * sizeof(unsigned long long), 256); }

void launch_vertex_normals(const float* V, int32_t nv, const int32_t* F, int32_t nf, float* N, void* scratch,
                           cudaStream_t s) {
  ProfScope ps("k_vertex_normals", s);
  unsigned long long* acc = (unsigned long long*)scratch;
  cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * 3 * (size_t)nv, s);
  const int blocks = (int)((nf + 255) / 256) < 4 * num_sms() ? (int)((nf + 255) / 256) : 4 * num_sms();
  k_face_normals_scatter<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(V, F, nf, acc);
  const int64_t n3 = 3 * (int64_t)nv;
  const int b2 = (int)((n3 + 255) / 256) < 4 * num_sms() ? (int)((n3 + 255) / 256) : 4 * num_sms();
  launch_chained(k_normals_finish, b2 > 0 ? b2 : 1, 256, 0, s, acc, n3, N);
}

void launch_vertex_normals_backward(const float* V, int32_t nv, const int32_t* F, int32_t nf, const float* dN,
                                    float* dV, cudaStream_t s) {
  (void)nv;
  ProfScope ps("k_face_normals_backward", s);
  const int blocks = (int)((nf + 255) / 256) < 4 * num_sms() ? (int)((nf + 255) / 256) : 4 * num_sms();
  k_face_normals_backward<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(V, F, nf, dN, dV);
}

// ---------------------------------------------------------------------------
// LBVH build
// ---------------------------------------------------------------------------
// float <-> order-preserving unsigned, for atomicMin/Max on floats
__device__ __forceinline__ uint32_t f2ord(float f) {
  uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float ord2f(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

__device__ __forceinline__ float3 centroid_of(const float* V, const int32_t* F, int f) {
  const float3 v0 = load3(V + 3 * F[3 * f]), v1 = load3(V + 3 * F[3 * f + 1]), v2 = load3(V + 3 * F[3 * f + 2]);
  return (v0 + v1 + v2) * (1.0f / 3.0f);
}

__global__ void k_centroid_bounds(const float* __restrict__ V, const int32_t* __restrict__ F, int32_t nf,
                                  uint32_t* __restrict__ b) {
  float3 lo = mk(INFINITY, INFINITY, INFINITY), hi = mk(-INFINITY, -INFINITY, -INFINITY);
  for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += gridDim.x * blockDim.x) {
    const float3 c = centroid_of(V, F, f);
    lo = mk(fminf(lo.x, c.x), fminf(lo.y, c.y), fminf(lo.z, c.z));
    hi = mk(fmaxf(hi.x, c.x), fmaxf(hi.y, c.y), fmaxf(hi.z, c.z));
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo.x = fminf(lo.x, __shfl_xor_sync(kFull, lo.x, o));
    lo.y = fminf(lo.y, __shfl_xor_sync(kFull, lo.y, o));
    lo.z = fminf(lo.z, __shfl_xor_sync(kFull, lo.z, o));
    hi.x = fmaxf(hi.x, __shfl_xor_sync(kFull, hi.x, o));
    hi.y = fmaxf(hi.y, __shfl_xor_sync(kFull, hi.y, o));
    hi.z = fmaxf(hi.z, __shfl_xor_sync(kFull, hi.z, o));
  }
  if ((threadIdx.x & 31) == 0 && lo.x <= hi.x) {
    atomicMin(b + 0, f2ord(lo.x)); atomicMin(b + 1, f2ord(lo.y)); atomicMin(b + 2, f2ord(lo.z));
    atomicMax(b + 3, f2ord(hi.x)); atomicMax(b + 4, f2ord(hi.y)); atomicMax(b + 5, f2ord(hi.z));
  }
}

// 10 bits per axis interleaved into a 30-bit Morton code
__device__ __forceinline__ uint32_t spread10(uint32_t v) {
  v = (v | (v << 16)) & 0x030000FFu;
  v = (v | (v << 8)) & 0x0300F00Fu;
  v = (v | (v << 4)) & 0x030C30C3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}

__global__ void k_morton(const float* __restrict__ V, const int32_t* __restrict__ F, int32_t nf,
                         const uint32_t* __restrict__ b, uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  const float3 lo = mk(ord2f(b[0]), ord2f(b[1]), ord2f(b[2]));
  const float3 hi = mk(ord2f(b[3]), ord2f(b[4]), ord2f(b[5]));
  const float3 ext = mk(fmaxf(hi.x - lo.x, 1e-30f), fmaxf(hi.y - lo.y, 1e-30f), fmaxf(hi.z - lo.z, 1e-30f));
  for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += gridDim.x * blockDim.x) {
    const float3 c = centroid_of(V, F, f);
    const uint32_t x = (uint32_t)fminf(fmaxf((c.x - lo.x) / ext.x * 1024.0f, 0.0f), 1023.0f);
    const uint32_t y = (uint32_t)fminf(fmaxf((c.y - lo.y) / ext.y * 1024.0f, 0.0f), 1023.0f);
    const uint32_t z = (uint32_t)fminf(fmaxf((c.z - lo.z) / ext.z * 1024.0f, 0.0f), 1023.0f);
    keys[f] = (spread10(x) << 2) | (spread10(y) << 1) | spread10(z);
    vals[f] = (uint32_t)f;
  }
}

// ---- stable LSD radix sort, 8 bits per pass -------------------------------
constexpr int kSortThreads = 256;
constexpr int kSortIpt = 4;
constexpr int kSortTile = kSortThreads * kSortIpt;
constexpr int kSortWarps = kSortThreads / 32;

// hist is digit-major: hist[d * nblocks + block]
__global__ void k_radix_hist(const uint32_t* __restrict__ keys, int32_t n, int shift, uint32_t* __restrict__ hist) {
  __shared__ uint32_t cnt[256];
  cnt[threadIdx.x] = 0;
  __syncthreads();
  const int base = blockIdx.x * kSortTile;
  for (int j = 0; j < kSortIpt; ++j) {
    const int i = base + j * kSortThreads + threadIdx.x;
    if (i < n) atomicAdd(&cnt[(keys[i] >> shift) & 0xffu], 1u);
  }
  __syncthreads();
  hist[threadIdx.x * gridDim.x + blockIdx.x] = cnt[threadIdx.x];
}

// ---- exclusive scan -----------------------------------------------------------
// At most kScanBlocks CTAs have a contiguous span each: one launch sums the
// spans, the second adds up the spans before its own and scans its span tile
// by tile (eight entries per thread, two 16-byte loads).  An array of one tile
// needs the second launch only.  A scan of one CTA, each thread walking its
// own thousandth of the array, took 1.0 ms for 1.08M entries and 103 us for
// 120k; this takes 8 us for 120k and 18
// us for 1.08M.
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

// inclusive sum over the CTA's threads before this one (exclusive), and the total
__device__ __forceinline__ uint32_t cta_exclusive_sum(uint32_t v, uint32_t* s_warp, uint32_t& total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();  // the previous use of s_warp is over
  if (lane == 31) s_warp[wid] = x;
  __syncthreads();
  uint32_t before = 0, all = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    const uint32_t t = s_warp[w];
    if (w < wid) before += t;
    all += t;
  }
  total = all;
  return before + x - v;
}

// entries i .. i + 7 of a[0, m) (zeros past the end); i is a multiple of 8 and a 16-byte aligned
__device__ __forceinline__ void scan_load(const uint32_t* a, int64_t i, int64_t m, uint32_t (&v)[kScanItems]) {
  if (i + kScanItems <= m) {
    const uint4 x = *reinterpret_cast<const uint4*>(a + i), y = *reinterpret_cast<const uint4*>(a + i + 4);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
  } else {
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) v[k] = i + k < m ? a[i + k] : 0u;
  }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_totals(const uint32_t* a, int64_t m, int64_t span,
                                                              uint32_t* totals) {
  chain_begin();
  __shared__ uint32_t s_warp[kScanThreads / 32];
  const int64_t lo = blockIdx.x * span, hi = min(lo + span, m);
  uint32_t sum = 0, total;
  for (int64_t i = lo + threadIdx.x * kScanItems; i < hi; i += kScanTile) {
    uint32_t v[kScanItems];
    scan_load(a, i, hi, v);
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) sum += v[k];
  }
  cta_exclusive_sum(sum, s_warp, total);
  if (threadIdx.x == 0) totals[blockIdx.x] = total;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_apply(const uint32_t* src, uint32_t* dst, int64_t m, int64_t span,
                                                             const uint32_t* totals) {
  chain_begin();
  __shared__ uint32_t s_warp[kScanThreads / 32];
  const int64_t lo = blockIdx.x * span, hi = min(lo + span, m);
  uint32_t carry = 0, total;
  if (gridDim.x > 1) {
    uint32_t sum = 0;
    for (uint32_t b = threadIdx.x; b < blockIdx.x; b += blockDim.x) sum += totals[b];
    cta_exclusive_sum(sum, s_warp, carry);
  }
  for (int64_t t = lo; t < hi; t += kScanTile) {
    const int64_t i = t + threadIdx.x * kScanItems;
    uint32_t v[kScanItems], sum = 0;
    scan_load(src, i, hi, v);
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
      const uint32_t x = v[k];
      v[k] = sum;
      sum += x;
    }
    const uint32_t base = carry + cta_exclusive_sum(sum, s_warp, total);
    carry += total;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) v[k] += base;
    if (i + kScanItems <= hi) {
      *reinterpret_cast<uint4*>(dst + i) = make_uint4(v[0], v[1], v[2], v[3]);
      *reinterpret_cast<uint4*>(dst + i + 4) = make_uint4(v[4], v[5], v[6], v[7]);
    } else {
#pragma unroll
      for (int k = 0; k < kScanItems; ++k)
        if (i + k < hi) dst[i + k] = v[k];
    }
  }
}

// Scatter a tile keeping the input order among equal digits: items are taken
// in order j (stride kSortThreads), then warp, then lane; within a warp the
// rank among equal digits comes from __match_any_sync, across warps from a
// per-step prefix over per-warp digit counts.
__global__ void k_radix_scatter(const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin, int32_t n,
                                int shift, const uint32_t* __restrict__ hist, uint32_t* __restrict__ kout,
                                uint32_t* __restrict__ vout) {
  __shared__ uint32_t off[256];
  __shared__ uint32_t wcnt[kSortWarps][256];
  __shared__ uint32_t step_total[256];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  off[tid] = hist[tid * gridDim.x + blockIdx.x];
  const int base = blockIdx.x * kSortTile;
  const unsigned lanemask_lt = (1u << lane) - 1u;
  for (int j = 0; j < kSortIpt; ++j) {
    for (int w = 0; w < kSortWarps; ++w) wcnt[w][tid] = 0;
    __syncthreads();
    const int i = base + j * kSortThreads + tid;
    const bool valid = i < n;
    uint32_t key = 0, val = 0, dg = 256;
    if (valid) {
      key = kin[i];
      val = vin[i];
      dg = (key >> shift) & 0xffu;
    }
    const unsigned peers = __match_any_sync(kFull, dg);
    const uint32_t rank = __popc(peers & lanemask_lt);
    if (valid && rank == 0) wcnt[warp][dg] = __popc(peers);
    __syncthreads();
    {  // thread tid owns digit tid: prefix over warps
      uint32_t run = 0;
      for (int w = 0; w < kSortWarps; ++w) {
        const uint32_t c = wcnt[w][tid];
        wcnt[w][tid] = run;
        run += c;
      }
      step_total[tid] = run;
    }
    __syncthreads();
    if (valid) {
      const uint32_t pos = off[dg] + wcnt[warp][dg] + rank;
      if (pos < (uint32_t)n) {
        kout[pos] = key;
        vout[pos] = val;
      }
    }
    __syncthreads();
    off[tid] += step_total[tid];
  }
}

// ---- Karras (2012) hierarchy ------------------------------------------------
// delta(a, b): length of the common prefix of keys a and b, with the index
// appended to break ties between equal keys; -1 outside [0, n).
__device__ __forceinline__ int lcp(const uint32_t* keys, int n, int a, int b) {
  if (b < 0 || b >= n) return -1;
  const uint32_t ka = keys[a], kb = keys[b];
  if (ka == kb) return 32 + __clz((uint32_t)a ^ (uint32_t)b);
  return __clz(ka ^ kb);
}

__global__ void k_karras(const uint32_t* __restrict__ keys, int32_t n, int2* __restrict__ bin_child,
                         int32_t* __restrict__ parent) {
  const int n_int = n - 1;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_int; i += gridDim.x * blockDim.x) {
    const int d = (lcp(keys, n, i, i + 1) - lcp(keys, n, i, i - 1)) >= 0 ? 1 : -1;
    const int dmin = lcp(keys, n, i, i - d);
    int lmax = 2;
    while (lcp(keys, n, i, i + lmax * d) > dmin) lmax *= 2;
    int l = 0;
    for (int t = lmax / 2; t >= 1; t /= 2)
      if (lcp(keys, n, i, i + (l + t) * d) > dmin) l += t;
    const int j = i + l * d;
    const int dnode = lcp(keys, n, i, j);
    int s = 0;
    for (int div = 2;; div *= 2) {
      const int t = (l + div - 1) / div;
      if (lcp(keys, n, i, i + (s + t) * d) > dnode) s += t;
      if (t <= 1) break;
    }
    const int gamma = i + s * d + (d < 0 ? -1 : 0);
    const int lo = min(i, j), hi = max(i, j);
    const int left = (lo == gamma) ? ~gamma : gamma;
    const int right = (hi == gamma + 1) ? ~(gamma + 1) : gamma + 1;
    bin_child[i] = make_int2(left, right);
    parent[left < 0 ? n_int + gamma : gamma] = i;
    parent[right < 0 ? n_int + gamma + 1 : gamma + 1] = i;
    if (i == 0) parent[0] = -1;
  }
}

// one triangle: a single internal node whose two children are both leaf 0
__global__ void k_single_leaf(int2* bin_child, int32_t* parent) {
  bin_child[0] = make_int2(~0, ~0);
  parent[0] = -1;
  parent[1] = 0;
}

__global__ void k_gather_leaf_tri(const uint32_t* __restrict__ vals, int32_t n, int32_t* __restrict__ leaf_tri) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) leaf_tri[i] = (int32_t)vals[i];
}

// ---- bottom-up bounds of the binary tree -----------------------------------
__device__ __forceinline__ void store_box(float4* box, float3 lo, float3 hi) {
  volatile float* b = reinterpret_cast<volatile float*>(box);
  b[0] = lo.x; b[1] = lo.y; b[2] = lo.z; b[3] = 0.f;
  b[4] = hi.x; b[5] = hi.y; b[6] = hi.z; b[7] = 0.f;
}

__device__ __forceinline__ void load_box(const float4* box, float3& lo, float3& hi) {
  const volatile float* b = reinterpret_cast<const volatile float*>(box);
  lo = mk(b[0], b[1], b[2]);
  hi = mk(b[4], b[5], b[6]);
}

// Each leaf writes its triangle record and box, then climbs: the first of two
// children to reach a node stops, the second merges both boxes, stores the
// node's box and goes on.  Through global memory a step of the climb is a fence,
// an atomic and a read, two microseconds in a chain as long as the tree is deep.
// A node is numbered by a position inside its range of leaves (but the root), so
// a CTA takes kRefitLeaves leaves in a row, and the nodes numbered alike climb in
// shared memory first; where only one child came that way, it goes on to the
// second climb, through global memory, as do the nodes numbered outside the CTA's
// leaves: every node has its two arrivals in one of the two.  (With
// the nodes' boxes: 120k triangles 67 -> 56 us, 5k 47 -> 37, of which the climb
// through global memory is still most.)  A path to the root has at most n_int nodes; the bounds guard a
// corrupt tree.
constexpr int kRefitLeaves = 512;

// A node of the climb with its links; those of the next one are read while the
// arrival at this one is awaited.
struct ClimbNode {
  int node, up;
  int2 child;
};
__device__ __forceinline__ ClimbNode climb_node(const BvhView& B, int node, int n_int) {
  ClimbNode c{node, -1, make_int2(kNoChild, kNoChild)};
  if (node >= 0 && node < n_int) {
    c.up = B.parent[node];
    c.child = B.bin_child[node];
  }
  return c;
}

__global__ void __launch_bounds__(kRefitLeaves) k_refit(const float* __restrict__ V, const int32_t* __restrict__ F,
                                                        int32_t nf, BvhView B, uint32_t* arrive) {
  chain_begin();
  __shared__ int s_arrive[kRefitLeaves];
  __shared__ float s_box[2][6][kRefitLeaves];  // of the left and the right child
  if (B.hdr->corrupt) return;  // a tree that failed validation: its leaves may be unset
  const int n_int = B.hdr->n_int, tid = threadIdx.x;
  if (blockIdx.x == 0 && tid == 0) B.hdr->coarse = 0;  // counted by k_node_boxes
  for (int64_t tile = (int64_t)blockIdx.x * kRefitLeaves; tile < nf; tile += (int64_t)gridDim.x * kRefitLeaves) {
    __syncthreads();
    s_arrive[tid] = 0;
    __syncthreads();
    const int first = (int)tile, i = first + min(tid, nf - 1 - first);
    const bool on = tile + tid < nf;
    float3 lo = mk(0.f, 0.f, 0.f), hi = lo;
    int me = ~i;
    ClimbNode at{-1, -1, make_int2(kNoChild, kNoChild)};
    bool parked = false;
    if (on) {
      const int tri = B.leaf_tri[i];
      const float3 v0 = load3(V + 3 * F[3 * tri]), v1 = load3(V + 3 * F[3 * tri + 1]), v2 = load3(V + 3 * F[3 * tri + 2]);
      B.tris[3 * i + 0] = make_float4(v0.x, v0.y, v0.z, __int_as_float(tri));
      const float3 e1 = v1 - v0, e2 = v2 - v0;
      B.tris[3 * i + 1] = make_float4(e1.x, e1.y, e1.z, 0.f);
      B.tris[3 * i + 2] = make_float4(e2.x, e2.y, e2.z, 0.f);
      lo = mk(fminf(v0.x, fminf(v1.x, v2.x)), fminf(v0.y, fminf(v1.y, v2.y)), fminf(v0.z, fminf(v1.z, v2.z)));
      hi = mk(fmaxf(v0.x, fmaxf(v1.x, v2.x)), fmaxf(v0.y, fmaxf(v1.y, v2.y)), fmaxf(v0.z, fmaxf(v1.z, v2.z)));
      store_box(B.box_leaf + 2 * i, lo, hi);
      at = climb_node(B, B.parent[n_int + i], n_int);
      for (int hops = 0; at.node >= first && at.node < n_int && at.node - first < kRefitLeaves && hops < kRefitLeaves;
           ++hops) {
        const int side = at.child.x == me ? 0 : 1, slot = at.node - first;
        if ((side ? at.child.x : at.child.y) == kNoChild) break;  // the root of a single leaf
        const ClimbNode next = climb_node(B, at.up, n_int);
        s_box[side][0][slot] = lo.x;
        s_box[side][1][slot] = lo.y;
        s_box[side][2][slot] = lo.z;
        s_box[side][3][slot] = hi.x;
        s_box[side][4][slot] = hi.y;
        s_box[side][5][slot] = hi.z;
        __threadfence_block();
        parked = atomicAdd(&s_arrive[slot], 1) == 0;
        if (parked) break;  // the sibling is still on its way, or comes from another CTA
        __threadfence_block();
        const float(*o)[kRefitLeaves] = s_box[1 - side];
        lo = mk(fminf(lo.x, o[0][slot]), fminf(lo.y, o[1][slot]), fminf(lo.z, o[2][slot]));
        hi = mk(fmaxf(hi.x, o[3][slot]), fmaxf(hi.y, o[4][slot]), fmaxf(hi.z, o[5][slot]));
        store_box(B.box_int + 2 * at.node, lo, hi);
        me = at.node;
        at = next;
      }
    }
    __syncthreads();
    if (!on || (parked && s_arrive[at.node - first] > 1)) continue;
    for (int hops = 0; at.node >= 0 && at.node < n_int && hops <= n_int; ++hops) {
      const ClimbNode next = climb_node(B, at.up, n_int);
      const int sib = (at.child.x == me) ? at.child.y : at.child.x;
      if (sib != kNoChild) {
        __threadfence();
        const uint32_t prev = atomicAdd(arrive + at.node, 1u);
        if (prev == 0) break;  // the sibling is still on its way
        __threadfence();
        float3 olo, ohi;
        load_box(sib >= 0 ? B.box_int + 2 * sib : B.box_leaf + 2 * (~sib), olo, ohi);
        lo = mk(fminf(lo.x, olo.x), fminf(lo.y, olo.y), fminf(lo.z, olo.z));
        hi = mk(fmaxf(hi.x, ohi.x), fmaxf(hi.y, ohi.y), fmaxf(hi.z, ohi.z));
      }
      store_box(B.box_int + 2 * at.node, lo, hi);
      me = at.node;
      at = next;
    }
  }
}

// ---- binned SAH build (top-down) ---------------------------------------------
// A second builder of the same binary layout.  Top-down: each task is a
// contiguous range of a primitive permutation; its split is the bin boundary
// (of 32 centroid bins per axis; 16 in the small builder) with the least
// surface area cost area(left box) * left count + area(right box) * right
// count, and the range
// is partitioned stably into [left | right].  Tasks larger than kSahSmall
// are split level by level in one cooperative launch (k_sah_levels), in
// chunks of kSahChunk positions so that the few huge tasks near the root use
// the whole GPU: each chunk's bins are summed in shared memory and added to its
// task's, and the CTA that adds the last chunk of a task chooses the split;
// after a barrier of the grid each chunk is scattered, stably, past the left
// counts of the task's chunks before it (from their own bin counts).  A task
// of one chunk is binned, split and scattered by its CTA at once.  (As four
// launches per level, and as many levels as a tree could have, the host not
// knowing how many there are, this took 1.18 ms for 120k triangles and 0.67
// ms for 5k, most of it launches; now 212
// and 89 us.)  Smaller tasks are built
// down to their leaves by one CTA each, in shared memory.  An internal node
// is numbered by its split position s (the last position of its left child),
// which is unique in [0, nf - 2]; the root's number is swapped with 0 so the
// root is node 0.  Splits deeper than kSahFreeDepth (large tasks) or
// kSahSmallFreeDepth (small ones) take the median, which bounds the depth
// (see launch_sah_topology).  Every decision is a deterministic function of
// the geometry: bins are integer sums, minima and maxima, and partitions are
// stable.
constexpr int kSahBins = 32;       // bins per axis of the large-task levels
constexpr int kSahSmallBins = 16;  // of the small builder
constexpr int kSahTiny = 4;        // ranges up to this size split at the centroid median
constexpr int kSahSmall = 128;
constexpr int kSahFreeDepth = 24;
constexpr int kSahSmallFreeDepth = 56;
constexpr int kSahMaxLevels = 64;
constexpr int kSahChunk = 1024;
constexpr int kSahThreads = 256;
constexpr int kSahBlocksPerSm = 3;  // resident CTAs of the level kernel
constexpr int kSahSmallWarps = 4;

struct SahTask {
  int a, n, parent, sd;       // range, parent node, side | depth << 1
  int chunk0, axis, bin, nl;  // first chunk of the level; the split (axis < 0: median)
  float4 lo, hi;              // binning bounds (xyz), a superset of the centroids; lo.w: bits of the chunks binned
};
template <int kB>
struct SahBinsT {  // order-preserving uints for the float bounds
  uint32_t cnt[3][kB];
  uint32_t lo[3][kB][3];
  uint32_t hi[3][kB][3];
};
using SahBins = SahBinsT<kSahBins>;
using SahSmallBins = SahBinsT<kSahSmallBins>;
struct SahState {
  unsigned long long packed[kSahMaxLevels + 2];  // per level: tasks << 32 | chunks
  int n_small;
  int sroot;
  uint32_t barrier[kBarrierWords];
};
struct SahView {
  float4* cen;
  float4* pbox;
  uint32_t* idx[2];
  SahTask* tasks[2];
  SahBins* bins[2];
  int* chunk_task[2];   // [max_chunks]: the task of each chunk of a level
  uint32_t* chunk_cnt;  // [max_chunks][3][kSahBins]: bin counts of a chunk of a task of several
  int4* small;  // (a, n, parent, side | depth << 1 | buffer << 30)
  SahState* st;
  int max_large, max_small, max_chunks;
};

template <int kB = kSahBins>
__device__ __forceinline__ int sah_bin(float c, float lo, float scale) {
  const int b = (int)__fmul_rn(__fsub_rn(c, lo), scale);
  return min(kB - 1, max(0, b));
}
template <int kB = kSahBins>
__device__ __forceinline__ float sah_scale(float lo, float hi) {
  const float ext = __fsub_rn(hi, lo);
  return ext > 0.0f ? __fdiv_rn((float)kB, ext) : 0.0f;
}
__device__ __forceinline__ float sah_area(float3 lo, float3 hi) {
  const float3 d = hi - lo;
  return d.x * d.y + d.y * d.z + d.z * d.x;
}
__device__ __forceinline__ int sah_split_id(int s, int sroot) { return s == sroot ? 0 : (s == 0 ? sroot : s); }
__device__ __forceinline__ void sah_set_child(BvhView& B, int node, int side, int ref) {
  reinterpret_cast<int*>(B.bin_child + node)[side] = ref;
}
__device__ __forceinline__ float comp(const float4& v, int k) { return k == 0 ? v.x : (k == 1 ? v.y : v.z); }
__device__ __forceinline__ float comp3(const float3& v, int k) { return k == 0 ? v.x : (k == 1 ? v.y : v.z); }

// Primitive boxes and centroids, the bounds of the centroids, the identity
// permutation, bin_child cleared to kNoChild and internal parents to -1
// (validation catches any link a build leaves unset, and the depth walks stop
// at an unset parent).
__global__ void __launch_bounds__(256) k_sah_prims(const float* __restrict__ V, const int32_t* __restrict__ F, int32_t nf,
                                                   uint32_t* bounds, SahView S, BvhView B) {
  chain_begin();
  __shared__ uint32_t s_b[6];
  if (threadIdx.x < 6) s_b[threadIdx.x] = threadIdx.x < 3 ? 0xffffffffu : 0u;
  __syncthreads();
  const int n_int = nf - 1;
  float3 lo = mk(INFINITY, INFINITY, INFINITY), hi = mk(-INFINITY, -INFINITY, -INFINITY);
  for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += gridDim.x * blockDim.x) {
    const float3 v0 = load3(V + 3 * F[3 * f]), v1 = load3(V + 3 * F[3 * f + 1]), v2 = load3(V + 3 * F[3 * f + 2]);
    const float3 c = (v0 + v1 + v2) * (1.0f / 3.0f);
    lo = mk(fminf(lo.x, c.x), fminf(lo.y, c.y), fminf(lo.z, c.z));
    hi = mk(fmaxf(hi.x, c.x), fmaxf(hi.y, c.y), fmaxf(hi.z, c.z));
    S.cen[f] = make_float4(c.x, c.y, c.z, 0.f);
    S.pbox[2 * f] =
        make_float4(fminf(v0.x, fminf(v1.x, v2.x)), fminf(v0.y, fminf(v1.y, v2.y)), fminf(v0.z, fminf(v1.z, v2.z)), 0.f);
    S.pbox[2 * f + 1] =
        make_float4(fmaxf(v0.x, fmaxf(v1.x, v2.x)), fmaxf(v0.y, fmaxf(v1.y, v2.y)), fmaxf(v0.z, fmaxf(v1.z, v2.z)), 0.f);
    S.idx[0][f] = (uint32_t)f;
    if (f < n_int) {
      B.bin_child[f] = make_int2(kNoChild, kNoChild);
      B.parent[f] = -1;
    }
  }
  const uint32_t m[6] = {__reduce_min_sync(kFull, f2ord(lo.x)), __reduce_min_sync(kFull, f2ord(lo.y)),
                         __reduce_min_sync(kFull, f2ord(lo.z)), __reduce_max_sync(kFull, f2ord(hi.x)),
                         __reduce_max_sync(kFull, f2ord(hi.y)), __reduce_max_sync(kFull, f2ord(hi.z))};
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      atomicMin(&s_b[k], m[k]);
      atomicMax(&s_b[3 + k], m[3 + k]);
    }
  }
  __syncthreads();
  if (threadIdx.x < 3) atomicMin(bounds + threadIdx.x, s_b[threadIdx.x]);
  else if (threadIdx.x < 6) atomicMax(bounds + threadIdx.x, s_b[threadIdx.x]);
}

__device__ __forceinline__ int sah_chunks(int n) { return (n + kSahChunk - 1) / kSahChunk; }

// empty bins: zero counts, inverted bounds (threads i0, i0 + stride, ...)
template <int kB>
__device__ __forceinline__ void sah_zero_bins(SahBinsT<kB>* g, int i0, int stride) {
  uint32_t* cnt = &g->cnt[0][0];
  uint32_t* lo = &g->lo[0][0][0];
  uint32_t* hi = &g->hi[0][0][0];
  for (int i = i0; i < 3 * kB; i += stride) {
    cnt[i] = 0u;
    for (int q = 0; q < 3; ++q) {
      lo[3 * i + q] = 0xffffffffu;
      hi[3 * i + q] = 0u;
    }
  }
}

// the root task: large (level 0) or, for at most kSahSmall triangles, small
// (one CTA; the state starts out zero)
__device__ void sah_root(int32_t nf, const uint32_t* bounds, const SahView& S) {
  if (nf > kSahSmall) {
    sah_zero_bins(&S.bins[0][0], threadIdx.x, blockDim.x);
    for (int c = threadIdx.x; c < sah_chunks(nf); c += blockDim.x) S.chunk_task[0][c] = 0;
  }
  if (threadIdx.x == 0) {
    S.st->sroot = -1;
    if (nf > kSahSmall) {
      SahTask t;
      t.a = 0; t.n = nf; t.parent = -1; t.sd = 0;
      t.chunk0 = 0; t.axis = -1; t.bin = -1; t.nl = 0;
      t.lo = make_float4(ord2f(bounds[0]), ord2f(bounds[1]), ord2f(bounds[2]), 0.f);
      t.hi = make_float4(ord2f(bounds[3]), ord2f(bounds[4]), ord2f(bounds[5]), 0.f);
      S.tasks[0][0] = t;
      S.st->packed[0] = (1ull << 32) | (unsigned long long)sah_chunks(nf);
    } else {
      S.small[0] = make_int4(0, nf, -1, 0);
      S.st->n_small = 1;
    }
  }
}

template <int kB>
__device__ __forceinline__ void sah_flush(SahBinsT<kB>& sb, int k, int b, uint32_t n, float3 lo, float3 hi) {
  atomicAdd(&sb.cnt[k][b], n);
  atomicMin(&sb.lo[k][b][0], f2ord(lo.x)); atomicMin(&sb.lo[k][b][1], f2ord(lo.y)); atomicMin(&sb.lo[k][b][2], f2ord(lo.z));
  atomicMax(&sb.hi[k][b][0], f2ord(hi.x)); atomicMax(&sb.hi[k][b][1], f2ord(hi.y)); atomicMax(&sb.hi[k][b][2], f2ord(hi.z));
}

// Everything below is read after another CTA of the same launch wrote it, so
// the loads are plain ones (never the read-only path).
struct SahLevel {
  int ntask, nchunk;
};
__device__ __forceinline__ SahLevel sah_level(const SahView& S, int level) {
  const unsigned long long pk = S.st->packed[level];
  SahLevel l;
  l.ntask = min((int)(pk >> 32), S.max_large);
  l.nchunk = min((int)(pk & 0xffffffffull), S.max_chunks);
  return l;
}

__device__ __forceinline__ bool sah_free(const SahTask& T, float sc[3]) {
  sc[0] = sah_scale(T.lo.x, T.hi.x);
  sc[1] = sah_scale(T.lo.y, T.hi.y);
  sc[2] = sah_scale(T.lo.z, T.hi.z);
  return (T.sd >> 1) < kSahFreeDepth && (sc[0] > 0.f || sc[1] > 0.f || sc[2] > 0.f);
}

// A task's split, and what its children need.
struct SahChoice {
  int axis, bin, nl;
  float3 llo, lhi, rlo, rhi;
};

// The split of a task from its bins in shared memory, by the whole CTA: warp k
// has axis k and lane i bin i.  Boundary i puts bins 0..i left; the boxes
// and counts left of every boundary are an inclusive scan over the lanes, those
// right of it one from the other end.  The least cost wins, ties to the
// lower boundary and then to the lower axis.
__device__ __forceinline__ void sah_choose(const SahBins& sb, const SahTask& T, const float sc[3], bool free,
                                           SahChoice* s_axis, float* s_cost, SahChoice& out) {
  static_assert(kSahBins == 32, "a lane per bin");
  const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
  if (k < 3) {
    float best = INFINITY;
    SahChoice c;
    c.axis = k; c.bin = -1; c.nl = T.n / 2;
    c.llo = c.rlo = mk(T.lo.x, T.lo.y, T.lo.z);
    c.lhi = c.rhi = mk(T.hi.x, T.hi.y, T.hi.z);
    if (free && sc[k] > 0.f) {
      const uint32_t cnt = sb.cnt[k][lane];
      float3 ll = mk(INFINITY, INFINITY, INFINITY), lh = mk(-INFINITY, -INFINITY, -INFINITY);
      if (cnt) {
        ll = mk(ord2f(sb.lo[k][lane][0]), ord2f(sb.lo[k][lane][1]), ord2f(sb.lo[k][lane][2]));
        lh = mk(ord2f(sb.hi[k][lane][0]), ord2f(sb.hi[k][lane][1]), ord2f(sb.hi[k][lane][2]));
      }
      float3 rl = ll, rh = lh;
      uint32_t lc = cnt, rc = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t a = __shfl_up_sync(kFull, lc, o), b = __shfl_down_sync(kFull, rc, o);
        const float3 al = mk(__shfl_up_sync(kFull, ll.x, o), __shfl_up_sync(kFull, ll.y, o), __shfl_up_sync(kFull, ll.z, o));
        const float3 ah = mk(__shfl_up_sync(kFull, lh.x, o), __shfl_up_sync(kFull, lh.y, o), __shfl_up_sync(kFull, lh.z, o));
        const float3 bl = mk(__shfl_down_sync(kFull, rl.x, o), __shfl_down_sync(kFull, rl.y, o), __shfl_down_sync(kFull, rl.z, o));
        const float3 bh = mk(__shfl_down_sync(kFull, rh.x, o), __shfl_down_sync(kFull, rh.y, o), __shfl_down_sync(kFull, rh.z, o));
        if (lane >= o) {
          lc += a;
          ll = mk(fminf(ll.x, al.x), fminf(ll.y, al.y), fminf(ll.z, al.z));
          lh = mk(fmaxf(lh.x, ah.x), fmaxf(lh.y, ah.y), fmaxf(lh.z, ah.z));
        }
        if (lane + o < 32) {
          rc += b;
          rl = mk(fminf(rl.x, bl.x), fminf(rl.y, bl.y), fminf(rl.z, bl.z));
          rh = mk(fmaxf(rh.x, bh.x), fmaxf(rh.y, bh.y), fmaxf(rh.z, bh.z));
        }
      }
      // right of boundary `lane` begins at the next lane
      rc = __shfl_down_sync(kFull, rc, 1);
      rl = mk(__shfl_down_sync(kFull, rl.x, 1), __shfl_down_sync(kFull, rl.y, 1), __shfl_down_sync(kFull, rl.z, 1));
      rh = mk(__shfl_down_sync(kFull, rh.x, 1), __shfl_down_sync(kFull, rh.y, 1), __shfl_down_sync(kFull, rh.z, 1));
      const bool cut = lane < 31 && lc > 0 && rc > 0;
      const float cost = cut ? sah_area(ll, lh) * (float)lc + sah_area(rl, rh) * (float)rc : INFINITY;
      // (costs are not negative: their bits order like the numbers; a NaN never wins)
      const uint32_t key = cut && cost < INFINITY ? __float_as_uint(cost) : 0x7f800000u;
      const uint32_t least = __reduce_min_sync(kFull, key);
      if (least < 0x7f800000u) {
        const int at = __ffs(__ballot_sync(kFull, key == least)) - 1;
        best = __uint_as_float(least);
        c.bin = at;
        c.nl = (int)__shfl_sync(kFull, lc, at);
        c.llo = mk(__shfl_sync(kFull, ll.x, at), __shfl_sync(kFull, ll.y, at), __shfl_sync(kFull, ll.z, at));
        c.lhi = mk(__shfl_sync(kFull, lh.x, at), __shfl_sync(kFull, lh.y, at), __shfl_sync(kFull, lh.z, at));
        c.rlo = mk(__shfl_sync(kFull, rl.x, at), __shfl_sync(kFull, rl.y, at), __shfl_sync(kFull, rl.z, at));
        c.rhi = mk(__shfl_sync(kFull, rh.x, at), __shfl_sync(kFull, rh.y, at), __shfl_sync(kFull, rh.z, at));
      }
    }
    if (lane == 0) {
      s_axis[k] = c;
      s_cost[k] = best;
    }
  }
  __syncthreads();
  int k0 = -1;
  float least = INFINITY;
  for (int a = 0; a < 3; ++a)
    if (s_axis[a].bin >= 0 && s_cost[a] < least) {
      least = s_cost[a];
      k0 = a;
    }
  if (k0 >= 0) {
    out = s_axis[k0];
  } else {  // the median
    out.axis = out.bin = -1;
    out.nl = T.n / 2;
    out.llo = out.rlo = mk(T.lo.x, T.lo.y, T.lo.z);
    out.lhi = out.rhi = mk(T.hi.x, T.hi.y, T.hi.z);
  }
}

// Numbers the split's node, links it to its parent and queues the children:
// large ones for the next level (with cleared bins where several CTAs will add
// to them), the rest for the small builder.  By the whole CTA, a warp per child
// (each waits on an atomic).
__device__ __forceinline__ void sah_emit(int level, const SahTask& T, const SahChoice& c, int sroot, const SahView& S,
                                         BvhView& B) {
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q >= 2) return;
  const int depth = T.sd >> 1;
  const int s = T.a + c.nl - 1;
  if (T.parent < 0) sroot = s;
  const int id = sah_split_id(s, sroot);
  const int ca = q ? T.a + c.nl : T.a, cn = q ? T.n - c.nl : c.nl, nc = sah_chunks(cn);
  if (threadIdx.x == 0) {
    if (T.parent < 0) S.st->sroot = s;
    B.parent[id] = T.parent;
    if (T.parent >= 0) sah_set_child(B, T.parent, T.sd & 1, id);
  }
  if (cn <= kSahSmall) {  // (one triangle: the small builder writes the leaf)
    if (lane == 0) {
      const int slot = atomicAdd(&S.st->n_small, 1);
      if (slot < S.max_small) S.small[slot] = make_int4(ca, cn, id, q | ((depth + 1) << 1) | (((level + 1) & 1) << 30));
      else atomicExch(&B.hdr->corrupt, 1);  // more tasks than disjoint ranges: never expected
    }
    return;
  }
  unsigned long long old = 0;
  if (lane == 0) old = atomicAdd(&S.st->packed[level + 1], (1ull << 32) | (unsigned long long)nc);
  old = __shfl_sync(kFull, old, 0);
  const int slot = (int)(old >> 32), chunk0 = (int)(old & 0xffffffffull);
  if (slot >= S.max_large || chunk0 + nc > S.max_chunks) {
    if (lane == 0) atomicExch(&B.hdr->corrupt, 1);
    return;
  }
  if (lane == 0) {
    SahTask ct;
    ct.a = ca; ct.n = cn; ct.parent = id; ct.sd = q | ((depth + 1) << 1);
    ct.chunk0 = chunk0; ct.axis = -1; ct.bin = -1; ct.nl = 0;
    const float3 lo = q ? c.rlo : c.llo, hi = q ? c.rhi : c.lhi;
    ct.lo = make_float4(lo.x, lo.y, lo.z, 0.f);
    ct.hi = make_float4(hi.x, hi.y, hi.z, 0.f);
    S.tasks[(level + 1) & 1][slot] = ct;
  }
  for (int i = lane; i < nc; i += 32) S.chunk_task[(level + 1) & 1][chunk0 + i] = slot;
  if (nc > 1) sah_zero_bins(&S.bins[(level + 1) & 1][slot], lane, 32);
}

// A chunk's positions, kSahPer consecutive ones per thread: the primitive
// and, packed five bits each, its bins along the three axes.
constexpr int kSahPer = kSahChunk / kSahThreads;
struct SahItems {
  uint32_t p[kSahPer], bins[kSahPer];
};

// Stable scatter of a chunk's items to [left | right] of its task, i0 the
// chunk's first position in the task and `before` the left ones of the
// chunks before it.
__device__ __forceinline__ void sah_scatter(const SahTask& T, const SahItems& it, uint32_t* out, int i0, int before,
                                            BvhView& B, uint32_t* s_warp) {
  const int i = i0 + (int)threadIdx.x * kSahPer;
  const int i1 = min(T.n, i0 + kSahChunk);
  bool left[kSahPer];
  uint32_t nleft = 0, total;
#pragma unroll
  for (int j = 0; j < kSahPer; ++j) {
    left[j] = i + j < i1 && (T.axis < 0 ? i + j < T.nl : (int)((it.bins[j] >> (5 * T.axis)) & 31u) <= T.bin);
    nleft += left[j] ? 1u : 0u;
  }
  int l = before + (int)cta_exclusive_sum(nleft, s_warp, total);
#pragma unroll
  for (int j = 0; j < kSahPer; ++j) {
    if (i + j >= i1) break;
    // a right one follows the task's left ones and the right ones before it; positions stay
    // inside the task even if bins and partition disagreed
    const int q = left[j] ? l : T.nl + (i + j - l);
    if (q < T.n) out[T.a + q] = it.p[j];
    l += left[j] ? 1 : 0;
  }
  if (threadIdx.x == 0 && i1 == T.n && before + (int)total != T.nl) atomicExch(&B.hdr->corrupt, 1);  // never expected
}

__global__ void __launch_bounds__(kSahThreads, kSahBlocksPerSm) k_sah_levels(int32_t nf, int levels,
                                                                             const uint32_t* __restrict__ bounds,
                                                                             SahView S, BvhView B) {
  __shared__ SahBins sb;
  __shared__ SahChoice s_axis[3];
  __shared__ float s_cost[3];
  __shared__ int s_last, s_before;
  __shared__ uint32_t s_warp[kSahThreads / 32];
  const int tid = threadIdx.x;
  GridBarrier bar{S.st->barrier, 0u, false};
  if (blockIdx.x == 0) sah_root(nf, bounds, S);
  grid_barrier(bar);
  for (int level = 0; level < levels && !bar.failed; ++level) {
    const SahLevel L = sah_level(S, level);
    if (L.ntask == 0) break;  // the same in every CTA
    SahTask* tasks = S.tasks[level & 1];
    const uint32_t* in = S.idx[level & 1];
    uint32_t* out = S.idx[(level + 1) & 1];
    const int sroot = S.st->sroot;  // (level 0 sets it)
    // bins, splits, and the scatter of tasks of one chunk
    for (int c = blockIdx.x; c < L.nchunk; c += gridDim.x) {
      const int t = S.chunk_task[level & 1][c];
      SahTask T = tasks[t];
      const int nc = sah_chunks(T.n), i0 = (c - T.chunk0) * kSahChunk, i1 = min(T.n, i0 + kSahChunk);
      float sc[3];
      const bool free = sah_free(T, sc);  // uniform over the CTA
      SahItems it;
      const int i = i0 + tid * kSahPer;
#pragma unroll
      for (int j = 0; j < kSahPer; ++j) {
        it.p[j] = i + j < i1 ? in[T.a + i + j] : 0u;
        it.bins[j] = 0u;
      }
      sah_zero_bins(&sb, tid, blockDim.x);
      __syncthreads();
      if (free && i < i1) {
        float4 c4[kSahPer], lo[kSahPer], hi[kSahPer];
#pragma unroll
        for (int j = 0; j < kSahPer; ++j) {
          c4[j] = S.cen[it.p[j]];
          lo[j] = S.pbox[2 * it.p[j]];
          hi[j] = S.pbox[2 * it.p[j] + 1];
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          if (sc[k] <= 0.f) continue;
          // a run of equal bins is added at once
          int cb = -1;
          uint32_t cn = 0u;
          float3 clo, chi;
#pragma unroll
          for (int j = 0; j < kSahPer; ++j) {
            if (i + j >= i1) break;
            const int b = sah_bin(comp(c4[j], k), comp(T.lo, k), sc[k]);
            it.bins[j] |= (uint32_t)b << (5 * k);
            if (b != cb) {
              if (cb >= 0) sah_flush(sb, k, cb, cn, clo, chi);
              cb = b;
              cn = 0u;
              clo = mk(INFINITY, INFINITY, INFINITY);
              chi = mk(-INFINITY, -INFINITY, -INFINITY);
            }
            ++cn;
            clo = mk(fminf(clo.x, lo[j].x), fminf(clo.y, lo[j].y), fminf(clo.z, lo[j].z));
            chi = mk(fmaxf(chi.x, hi[j].x), fmaxf(chi.y, hi[j].y), fmaxf(chi.z, hi[j].z));
          }
          if (cb >= 0) sah_flush(sb, k, cb, cn, clo, chi);
        }
      }
      __syncthreads();
      bool last = true;
      if (nc > 1) {  // into the task's bins; the CTA that completes them goes on
        SahBins& G = S.bins[level & 1][t];
        for (int i = tid; i < 3 * kSahBins; i += blockDim.x) {
          const int k = i / kSahBins, b = i % kSahBins;
          const uint32_t n = sb.cnt[k][b];
          S.chunk_cnt[(size_t)c * (3 * kSahBins) + i] = n;
          if (!n) continue;
          atomicAdd(&G.cnt[k][b], n);
          for (int q = 0; q < 3; ++q) {
            atomicMin(&G.lo[k][b][q], sb.lo[k][b][q]);
            atomicMax(&G.hi[k][b][q], sb.hi[k][b][q]);
          }
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) s_last = atomicAdd(reinterpret_cast<uint32_t*>(&tasks[t].lo.w), 1u) == (uint32_t)nc - 1u;
        __syncthreads();
        last = s_last != 0;
        if (last) {
          __threadfence();
          for (int i = tid; i < 3 * kSahBins; i += blockDim.x) {
            const int k = i / kSahBins, b = i % kSahBins;
            sb.cnt[k][b] = __ldcg(&G.cnt[k][b]);
            for (int q = 0; q < 3; ++q) {
              sb.lo[k][b][q] = __ldcg(&G.lo[k][b][q]);
              sb.hi[k][b][q] = __ldcg(&G.hi[k][b][q]);
            }
          }
          __syncthreads();
        }
      }
      if (last) {
        SahChoice ch;
        sah_choose(sb, T, sc, free, s_axis, s_cost, ch);
        T.axis = ch.axis;
        T.bin = ch.bin;
        T.nl = ch.nl;
        if (nc > 1 && tid == 0) {
          tasks[t].axis = ch.axis;
          tasks[t].bin = ch.bin;
          tasks[t].nl = ch.nl;
        }
        sah_emit(level, T, ch, sroot, S, B);
        if (nc == 1) sah_scatter(T, it, out, 0, 0, B, s_warp);
      }
      __syncthreads();  // the shared arrays are used again
    }
    // the scatter of tasks of several chunks, once they are split
    if (L.nchunk > L.ntask) {
      grid_barrier(bar);
      if (bar.failed) break;
      for (int c = blockIdx.x; c < L.nchunk; c += gridDim.x) {
        const SahTask T = tasks[S.chunk_task[level & 1][c]];
        if (sah_chunks(T.n) == 1) continue;
        float sc[3];
        sah_free(T, sc);
        const int i0 = (c - T.chunk0) * kSahChunk, i1 = min(T.n, i0 + kSahChunk), i = i0 + tid * kSahPer;
        SahItems it;
#pragma unroll
        for (int j = 0; j < kSahPer; ++j) it.p[j] = i + j < i1 ? in[T.a + i + j] : 0u;
#pragma unroll
        for (int j = 0; j < kSahPer; ++j) {
          it.bins[j] = 0u;
          if (T.axis >= 0 && i + j < i1)
            it.bins[j] = (uint32_t)sah_bin(comp(S.cen[it.p[j]], T.axis), comp(T.lo, T.axis), sc[T.axis]) << (5 * T.axis);
        }
        if (tid == 0) s_before = 0;
        __syncthreads();
        if (T.axis < 0) {
          if (tid == 0) s_before = min(i0, T.nl);
        } else {
          uint32_t sum = 0;
          const int bins = T.bin + 1, n = (c - T.chunk0) * bins;
          for (int i = tid; i < n; i += blockDim.x)
            sum += S.chunk_cnt[(size_t)(T.chunk0 + i / bins) * (3 * kSahBins) + T.axis * kSahBins + i % bins];
          sum = __reduce_add_sync(kFull, sum);
          if ((tid & 31) == 0 && sum) atomicAdd(&s_before, (int)sum);
        }
        __syncthreads();
        sah_scatter(T, it, out, i0, s_before, B, s_warp);
        __syncthreads();
      }
    }
    grid_barrier(bar);
  }
  if (bar.failed && tid == 0) atomicExch(&B.hdr->corrupt, 1);  // not co-resident: never expected
}

// Small tasks: one CTA builds a whole subtree (at most kSahSmall triangles)
// with the same binned SAH, its triangles in shared memory, level by level: a
// warp splits a range, a group of four lanes a range of at most kSahTiny (most
// of the nodes).  What bounds it is the chain of splits of one task: a warp per
// task, one split after another and three lanes sweeping the bins, took 271 us
// for 5k triangles (1.40 ms for 1.08M); this takes 37 us (468 us).
struct SahRange {
  int a, n, parent, sd;  // positions within the task, parent node, side | depth << 1
};
struct SahSmallShared {
  float cen[3][kSahSmall], lo[3][kSahSmall], hi[3][kSahSmall];
  uint32_t prim[kSahSmall];
  uint8_t ids[kSahSmall];  // local triangles in position order
  SahRange big[2][kSahSmall / 4], tiny[2][kSahSmall / 2];
  int n_big[2], n_tiny[2], sroot;
  SahSmallBins bins[kSahSmallWarps];
};

// Node of a split range at its split position s: numbered, linked to its
// parent, its children queued for the next level or, single triangles, linked.
__device__ __forceinline__ void sah_small_node(SahSmallShared& sh, int cur, const SahRange& r, int nl, int a, int n_int,
                                               const SahView& S, BvhView& B) {
  const int s = a + r.a + nl - 1;
  int sroot = sh.sroot;
  if (r.parent < 0) {  // the whole tree is this one task
    sroot = sh.sroot = s;
    S.st->sroot = s;
  }
  const int id = sah_split_id(s, sroot);
  B.parent[id] = r.parent;
  if (r.parent >= 0) sah_set_child(B, r.parent, r.sd & 1, id);
  for (int c = 0; c < 2; ++c) {
    const SahRange ch{c ? r.a + nl : r.a, c ? r.n - nl : nl, id, c | (((r.sd >> 1) + 1) << 1)};
    if (ch.n == 1) {
      sah_set_child(B, id, c, ~(a + ch.a));
      B.parent[n_int + a + ch.a] = id;
    } else if (ch.n <= kSahTiny) {
      sh.tiny[cur ^ 1][atomicAdd(&sh.n_tiny[cur ^ 1], 1)] = ch;
    } else {
      sh.big[cur ^ 1][atomicAdd(&sh.n_big[cur ^ 1], 1)] = ch;
    }
  }
}

// The split of a range of more than kSahTiny triangles, by one warp.
__device__ __forceinline__ void sah_small_split(SahSmallShared& sh, SahSmallBins& sb, int cur, const SahRange& r, int a,
                                                int n_int, const SahView& S, BvhView& B) {
  static_assert(kSahSmallBins == 16 && kSahSmall == 128, "half a warp per axis; four triangles per lane");
  const int lane = threadIdx.x & 31;
  const int depth = r.sd >> 1;
  // the range's triangles, in position order, and their centroids' bounds
  int id[4];
  float lo[3], hi[3], sc[3];
#pragma unroll
  for (int q = 0; q < 4; ++q) id[q] = q * 32 + lane < r.n ? sh.ids[r.a + q * 32 + lane] : -1;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    uint32_t l = 0xffffffffu, h = 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (id[q] >= 0) {
        const uint32_t o = f2ord(sh.cen[k][id[q]]);
        l = min(l, o);
        h = max(h, o);
      }
    lo[k] = ord2f(__reduce_min_sync(kFull, l));
    hi[k] = ord2f(__reduce_max_sync(kFull, h));
    sc[k] = sah_scale<kSahSmallBins>(lo[k], hi[k]);
  }
  int axis = -1, bin = -1, nl = r.n / 2;
  if (depth < kSahSmallFreeDepth && (sc[0] > 0.f || sc[1] > 0.f || sc[2] > 0.f)) {
    sah_zero_bins(&sb, lane, 32);
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (id[q] < 0) continue;
      const float3 plo = mk(sh.lo[0][id[q]], sh.lo[1][id[q]], sh.lo[2][id[q]]);
      const float3 phi = mk(sh.hi[0][id[q]], sh.hi[1][id[q]], sh.hi[2][id[q]]);
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (sc[k] > 0.f) sah_flush(sb, k, sah_bin<kSahSmallBins>(sh.cen[k][id[q]], lo[k], sc[k]), 1u, plo, phi);
    }
    __syncwarp();
    // lanes 0..15 scan the bins upward (left of boundary i: lane i), lanes 16..31
    // downward (right of boundary i: bins i + 1.., lane 16 + 14 - i)
    float bc = INFINITY;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (!(sc[k] > 0.f)) continue;
      const int b = lane < 16 ? lane : 31 - lane;
      uint32_t c = sb.cnt[k][b];
      float3 l = mk(INFINITY, INFINITY, INFINITY), h = mk(-INFINITY, -INFINITY, -INFINITY);
      if (c) {
        l = mk(ord2f(sb.lo[k][b][0]), ord2f(sb.lo[k][b][1]), ord2f(sb.lo[k][b][2]));
        h = mk(ord2f(sb.hi[k][b][0]), ord2f(sb.hi[k][b][1]), ord2f(sb.hi[k][b][2]));
      }
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
        const uint32_t oc = __shfl_up_sync(kFull, c, o, 16);
        const float3 ol = mk(__shfl_up_sync(kFull, l.x, o, 16), __shfl_up_sync(kFull, l.y, o, 16), __shfl_up_sync(kFull, l.z, o, 16));
        const float3 oh = mk(__shfl_up_sync(kFull, h.x, o, 16), __shfl_up_sync(kFull, h.y, o, 16), __shfl_up_sync(kFull, h.z, o, 16));
        if ((lane & 15) >= o) {
          c += oc;
          l = mk(fminf(l.x, ol.x), fminf(l.y, ol.y), fminf(l.z, ol.z));
          h = mk(fmaxf(h.x, oh.x), fmaxf(h.y, oh.y), fmaxf(h.z, oh.z));
        }
      }
      const float area = c ? sah_area(l, h) : 0.f;
      const int from = lane < 15 ? 30 - lane : lane;
      const uint32_t rc = __shfl_sync(kFull, c, from);
      const float rarea = __shfl_sync(kFull, area, from);
      const bool cut = lane < 15 && c > 0 && rc > 0;
      const float cost = cut ? area * (float)c + rarea * (float)rc : INFINITY;
      const uint32_t key = cut && cost < INFINITY ? __float_as_uint(cost) : 0x7f800000u;
      const uint32_t least = __reduce_min_sync(kFull, key);
      if (least < 0x7f800000u && __uint_as_float(least) < bc) {
        bc = __uint_as_float(least);
        axis = k;
        bin = __ffs(__ballot_sync(kFull, key == least)) - 1;
        nl = (int)__shfl_sync(kFull, c, bin);
      }
    }
    __syncwarp();
  }
  // stable partition in place (every lane holds its triangles)
  int lbase = 0, rbase = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const bool valid = id[q] >= 0;
    bool left = false;
    if (valid) {
      if (axis < 0) left = q * 32 + lane < nl;
      else {
        const float c = axis == 0 ? sh.cen[0][id[q]] : (axis == 1 ? sh.cen[1][id[q]] : sh.cen[2][id[q]]);
        const float l = axis == 0 ? lo[0] : (axis == 1 ? lo[1] : lo[2]), s = axis == 0 ? sc[0] : (axis == 1 ? sc[1] : sc[2]);
        left = sah_bin<kSahSmallBins>(c, l, s) <= bin;
      }
    }
    const unsigned bl = __ballot_sync(kFull, left), bv = __ballot_sync(kFull, valid);
    const unsigned below = (1u << lane) - 1u;
    if (valid) {  // inside the range even if bins and partition disagreed
      const int p = left ? lbase + __popc(bl & below) : nl + rbase + __popc(bv & ~bl & below);
      if (p < r.n) sh.ids[r.a + p] = (uint8_t)id[q];
    }
    lbase += __popc(bl);
    rbase += __popc(bv & ~bl);
  }
  if (lane == 0) {
    if (lbase != nl) atomicExch(&B.hdr->corrupt, 1);
    sah_small_node(sh, cur, r, nl, a, n_int, S, B);
  }
}

// The split of a range of 2..kSahTiny triangles, by four lanes (`live`: the
// group has one; every lane of the warp calls): the median of the centroids
// along their longest extent (ties by position); binning would cost far more
// than it can gain on a handful of triangles.
__device__ __forceinline__ void sah_tiny_split(SahSmallShared& sh, int cur, bool live, const SahRange& r, int a,
                                               int n_int, const SahView& S, BvhView& B) {
  const int lane = threadIdx.x & 31, l4 = lane & 3;
  const bool mine = live && l4 < r.n;
  const int id = mine ? sh.ids[r.a + l4] : 0;
  float c[3], ext[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    c[k] = mine ? sh.cen[k][id] : 0.f;
    float lo = mine ? c[k] : INFINITY, hi = mine ? c[k] : -INFINITY;
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      lo = fminf(lo, __shfl_xor_sync(kFull, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(kFull, hi, o));
    }
    ext[k] = hi - lo;
  }
  const int la = (ext[0] >= ext[1] && ext[0] >= ext[2]) ? 0 : (ext[1] >= ext[2] ? 1 : 2);
  const float x = la == 0 ? c[0] : (la == 1 ? c[1] : c[2]);
  int rank = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float xj = __shfl_sync(kFull, x, j, 4);
    if (j < r.n) rank += (xj < x || (xj == x && j < l4)) ? 1 : 0;
  }
  const int nl = r.n / 2;
  const bool left = mine && rank < nl;
  const unsigned bl = (__ballot_sync(kFull, left) >> (lane & 28)) & 15u;
  const unsigned bv = (__ballot_sync(kFull, mine) >> (lane & 28)) & 15u;
  const unsigned below = (1u << l4) - 1u;
  if (mine) {
    const int p = left ? __popc(bl & below) : nl + __popc(bv & ~bl & below);
    if (p < r.n) sh.ids[r.a + p] = (uint8_t)id;
  }
  if (live && l4 == 0) {
    if (__popc(bl) != nl) atomicExch(&B.hdr->corrupt, 1);
    sah_small_node(sh, cur, r, nl, a, n_int, S, B);
  }
}

__global__ void __launch_bounds__(32 * kSahSmallWarps) k_sah_small(SahView S, BvhView B) {
  chain_begin();
  static_assert(kSahTiny == 4, "a tiny range has four lanes");
  __shared__ SahSmallShared sh;
  if (B.hdr->corrupt) return;  // the large levels gave up: their permutation is incomplete
  const int n_int = B.hdr->n_int;
  const int tid = threadIdx.x, w = tid >> 5;
  const int nsmall = min(S.st->n_small, S.max_small);
  for (int t = blockIdx.x; t < nsmall; t += gridDim.x) {
    const int4 T = S.small[t];
    const int a = T.x, n = T.y;
    const uint32_t* in = S.idx[(T.w >> 30) & 1];
    if (n == 1) {  // a one-triangle child of a large task
      if (tid == 0) {
        sah_set_child(B, T.z, T.w & 1, ~a);
        B.parent[n_int + a] = T.z;
        B.leaf_tri[a] = (int32_t)in[a];
      }
      continue;  // uniform over the CTA
    }
    for (int i = tid; i < n; i += blockDim.x) {
      const uint32_t p = in[a + i];
      const float4 c = S.cen[p], lo = S.pbox[2 * p], hi = S.pbox[2 * p + 1];
      sh.prim[i] = p;
      sh.ids[i] = (uint8_t)i;
      sh.cen[0][i] = c.x; sh.cen[1][i] = c.y; sh.cen[2][i] = c.z;
      sh.lo[0][i] = lo.x; sh.lo[1][i] = lo.y; sh.lo[2][i] = lo.z;
      sh.hi[0][i] = hi.x; sh.hi[1][i] = hi.y; sh.hi[2][i] = hi.z;
    }
    if (tid == 0) {
      const SahRange r{0, n, T.z, T.w & 0x3fffffff};
      sh.n_big[0] = n > kSahTiny;
      sh.n_tiny[0] = n <= kSahTiny;
      if (n > kSahTiny) sh.big[0][0] = r; else sh.tiny[0][0] = r;
      sh.n_big[1] = sh.n_tiny[1] = 0;
      sh.sroot = T.z < 0 ? -1 : S.st->sroot;
    }
    __syncthreads();
    for (int cur = 0;; cur ^= 1) {
      const int nb = sh.n_big[cur], nt = sh.n_tiny[cur];
      if (nb == 0 && nt == 0) break;  // uniform: read between two barriers
      for (int i = w; i < nb; i += kSahSmallWarps) sah_small_split(sh, sh.bins[w], cur, sh.big[cur][i], a, n_int, S, B);
      // (the warps take the tiny ranges from the other end, so that the big ones' do not wait)
      for (int i0 = (kSahSmallWarps - 1 - w) * 8; i0 < nt; i0 += kSahSmallWarps * 8) {
        const int i = i0 + ((tid & 31) >> 2);
        sah_tiny_split(sh, cur, i < nt, sh.tiny[cur][i < nt ? i : i0], a, n_int, S, B);
      }
      __syncthreads();
      if (tid == 0) sh.n_big[cur] = sh.n_tiny[cur] = 0;
      __syncthreads();
    }
    for (int i = tid; i < n; i += blockDim.x) B.leaf_tri[a + i] = (int32_t)sh.prim[sh.ids[i]];
    __syncthreads();
  }
}

// ---- the 4-wide BVH ----------------------------------------------------------
// flag[j] = 1 and bin_to4[j] = 0 when binary node j sits at even depth (walks up
// to the root), else 0 and -1; also clears the arrivals of the refit that follows
__global__ void k_even_depth(BvhView B, uint32_t* flag, uint32_t* arrive) {
  chain_begin();
  const int n_int = B.hdr->n_int;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n_int; j += gridDim.x * blockDim.x) {
    int d = 0, p = j;
    for (int hops = 0; hops <= n_int && p > 0; ++hops) {
      p = B.parent[p];
      ++d;
    }
    flag[j] = (d & 1) ? 0u : 1u;
    B.bin_to4[j] = (d & 1) ? -1 : 0;
    arrive[j] = 0u;
  }
}

// after an exclusive scan of the flags: node4 index per even-depth node, -1 else
__global__ void k_bin_to4(BvhView B, const uint32_t* scanned) {
  chain_begin();
  const int n_int = B.hdr->n_int;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n_int; j += gridDim.x * blockDim.x) {
    const bool even = B.bin_to4[j] >= 0;
    if (even) B.bin_to4[j] = (int)scanned[j];
    if (j == n_int - 1) B.hdr->n4 = (int)scanned[j] + (even ? 1 : 0);
  }
}

// children of 4-wide node bin_to4[j] = the grandchildren of binary node j (a
// leaf child stays as it is); refs in row 6, binary sources in row 7
__global__ void k_node4_topology(BvhView B) {
  chain_begin();
  const int n_int = B.hdr->n_int;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n_int; j += gridDim.x * blockDim.x) {
    const int m = B.bin_to4[j];
    if (m < 0) continue;
    int ref[4] = {kNoChild, kNoChild, kNoChild, kNoChild};
    int srcs[4] = {kNoChild, kNoChild, kNoChild, kNoChild};
    int k = 0;
    const int2 ch = B.bin_child[j];
    const int c2[2] = {ch.x, ch.y};
    for (int a = 0; a < 2; ++a) {
      const int c = c2[a];
      if (c == kNoChild) continue;
      if (c < 0) {
        ref[k] = c; srcs[k] = c; ++k;
        continue;
      }
      const int2 g = B.bin_child[c];
      const int gg[2] = {g.x, g.y};
      for (int b = 0; b < 2; ++b) {
        const int x = gg[b];
        if (x == kNoChild) continue;
        ref[k] = x < 0 ? x : B.bin_to4[x];
        srcs[k] = x;
        ++k;
      }
    }
    reinterpret_cast<int4*>(B.node4)[8 * m + 6] = make_int4(ref[0], ref[1], ref[2], ref[3]);
    reinterpret_cast<int4*>(B.node4)[8 * m + 7] = make_int4(srcs[0], srcs[1], srcs[2], srcs[3]);
  }
}

// 256-bit store of a whole sector (p 32-byte aligned).  With stores of 128 bits, which
// write each sector in halves, keeping the exact nodes cost a refit of 82k triangles
// 4.7 us of 49; it is 1.9 with every kind of node stored so.
__device__ __forceinline__ void st_v8(float4* p, float4 a, float4 b) {
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z), "f"(a.w), "f"(b.x),
               "f"(b.y), "f"(b.z), "f"(b.w)
               : "memory");
}

// child boxes of 4-wide node m from the binary boxes
__device__ __forceinline__ void node4_boxes(const BvhView& B, int m) {
  const int4 sv = reinterpret_cast<const int4*>(B.node4)[8 * m + 7];
  const int srcs[4] = {sv.x, sv.y, sv.z, sv.w};
  float r[6][4];
  for (int k = 0; k < 4; ++k) {
    float3 lo = mk(INFINITY, INFINITY, INFINITY), hi = mk(-INFINITY, -INFINITY, -INFINITY);
    const int x = srcs[k];
    if (x != kNoChild) {
      const float4* bx = x >= 0 ? B.box_int + 2 * x : B.box_leaf + 2 * (~x);
      const float4 a = bx[0], b = bx[1];
      lo = mk(a.x, a.y, a.z);
      hi = mk(b.x, b.y, b.z);
    }
    r[0][k] = lo.x; r[1][k] = hi.x; r[2][k] = lo.y; r[3][k] = hi.y; r[4][k] = lo.z; r[5][k] = hi.z;
  }
#pragma unroll
  for (int row = 0; row < 6; row += 2)
    st_v8(B.node4 + 8 * (size_t)m + row, make_float4(r[row][0], r[row][1], r[row][2], r[row][3]),
          make_float4(r[row + 1][0], r[row + 1][1], r[row + 1][2], r[row + 1][3]));
}

// The nodes' child boxes after each refit, from the binary boxes: the 4-wide
// nodes', and the binary nodes' for the 2-wide traversal: the grid over the scene's box (the union of the root's two child
// boxes) and every child box coded on it, rounded outward.  The 0.02 steps
// cover the rounding of (x - lo) inv, at most 65000 steps times 2^-23.
__device__ __forceinline__ uint32_t code_planes(float lo, float hi, float base, float inv) {
  const float a = floorf((lo - base) * inv + (kQOffset - 0.02f)), b = ceilf((hi - base) * inv + (kQOffset + 0.02f));
  return (uint32_t)fminf(fmaxf(a, 0.0f), 65535.0f) | ((uint32_t)fminf(fmaxf(b, 0.0f), 65535.0f) << 16);
}
__device__ __forceinline__ float longest_side(const float4* box) {
  const float4 a = box[0], b = box[1];
  return fmaxf(fmaxf(b.x - a.x, b.y - a.y), b.z - a.z);
}
__device__ __forceinline__ const float4* child_box(const BvhView& B, int c) {
  return c >= 0 ? B.box_int + 2 * c : B.box_leaf + 2 * (~c);
}

// A coded box is up to a step longer on every side, so a ray near a patch of
// triangles a few steps in size tests several that the exact boxes would spare it.
// Such patches are found by nodes whose kQCluster-th ancestor, a patch of some 16
// triangles, is shorter than kQPatch steps, which is where the edges are some ten
// steps: a sphere of 77k triangles filling the frame, in a scene of 2.5 units,
// traced with coded and exact boxes, took 1477 and 1614 us (edges of 15 steps),
// 1589 and 1623 (10), 1777 and 1609 (6), 2672 and 1606 (2.6), 14970 and 1458 (0.5);
// 200k queries of it 156 and 157, 168 and 155, 188 and 158, 283 and 156, 1189 and
// 160 us.  Meshes of 19k and 307k triangles cross at the same edge length.  A scene
// of few triangles has no such patches, and its rays would test all of a part that
// one grid step holds: there one node shorter than kQTinyNode steps decides (80
// triangles of unit size above a ground triangle of 1e4 and 1e5, a frame of 512x512:
// coded 861 and 1492 us, exact 372 and 374; float boxes of before 478).
constexpr int kQCluster = 4;
constexpr float kQPatch = 26.0f;
constexpr int kQTiny = 1024;  // nodes of a scene of few triangles
constexpr float kQTinyNode = 8.0f;

__global__ void k_node_boxes(BvhView B) {
  chain_begin();
  if (B.hdr->corrupt) return;
  const int n_int = B.hdr->n_int, n4 = B.hdr->n4;
  float3 rlo = mk(INFINITY, INFINITY, INFINITY), rhi = mk(-INFINITY, -INFINITY, -INFINITY);
  const int2 root = B.bin_child[0];
  for (int k = 0; k < 2; ++k) {
    const int c = k ? root.y : root.x;
    if (c == kNoChild) continue;
    const float4 a = child_box(B, c)[0], b = child_box(B, c)[1];
    rlo = mk(fminf(rlo.x, a.x), fminf(rlo.y, a.y), fminf(rlo.z, a.z));
    rhi = mk(fmaxf(rhi.x, b.x), fmaxf(rhi.y, b.y), fmaxf(rhi.z, b.z));
  }
  const float step = fmaxf(fmaxf(fmaxf(rhi.x - rlo.x, rhi.y - rlo.y), rhi.z - rlo.z), 1e-30f) * (1.0f / kQSteps);
  const float inv = 1.0f / step;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n_int; j += gridDim.x * blockDim.x) {
    if (j == 0) {
      B.hdr->q[0] = rlo.x; B.hdr->q[1] = rlo.y; B.hdr->q[2] = rlo.z; B.hdr->q[3] = step;
      B.hdr->hi[0] = rhi.x; B.hdr->hi[1] = rhi.y; B.hdr->hi[2] = rhi.z;
    }
    if (j < n4) node4_boxes(B, j);
    const int2 ch = B.bin_child[j];
    uint32_t w[6];
    float3 lo[2], hi[2];
    for (int k = 0; k < 2; ++k) {
      const int c = k ? ch.y : ch.x;
      w[3 * k] = w[3 * k + 1] = w[3 * k + 2] = 0x0000ffffu;
      lo[k] = mk(INFINITY, INFINITY, INFINITY);
      hi[k] = -lo[k];
      if (c == kNoChild) continue;
      const float4 a = child_box(B, c)[0], b = child_box(B, c)[1];
      lo[k] = xyz(a);
      hi[k] = xyz(b);
      w[3 * k] = code_planes(a.x, b.x, rlo.x, inv);
      w[3 * k + 1] = code_planes(a.y, b.y, rlo.y, inv);
      w[3 * k + 2] = code_planes(a.z, b.z, rlo.z, inv);
    }
    st_v8(reinterpret_cast<float4*>(B.node2) + 2 * (size_t)j,
          make_float4(__uint_as_float(w[0]), __uint_as_float(w[1]), __uint_as_float(w[2]), __uint_as_float(w[3])),
          make_float4(__uint_as_float(w[4]), __uint_as_float(w[5]), __int_as_float(ch.x), __int_as_float(ch.y)));
    float4* X = B.node2x + 4 * (size_t)j;
    st_v8(X, make_float4(lo[0].x, hi[0].x, lo[0].y, hi[0].y), make_float4(lo[1].x, hi[1].x, lo[1].y, hi[1].y));
    st_v8(X + 2, make_float4(lo[0].z, hi[0].z, lo[1].z, hi[1].z),
          make_float4(__int_as_float(ch.x), __int_as_float(ch.y), 0.f, 0.f));
    if (n_int <= kQTiny) {
      if (j > 0 && longest_side(B.box_int + 2 * j) < kQTinyNode * step) atomicAdd(&B.hdr->coarse, kQCoarse + 1);
    } else if (longest_side(B.box_int + 2 * j) < kQPatch * step) {
      int p = j;
      for (int l = 0; l < kQCluster && p > 0; ++l) p = B.parent[p];
      if (p > 0 && p < n_int && longest_side(B.box_int + 2 * p) < kQPatch * step) atomicAdd(&B.hdr->coarse, 1);
    }
  }
}

// Validation of the built hierarchy: every reference in range, every parent
// link consistent with the child lists.  The traversal reads `corrupt` once
// and refuses to run on a tree that failed.
__global__ void k_validate(BvhView B) {
  chain_begin();
  const int n_int = B.hdr->n_int, n4 = B.hdr->n4, nf = B.hdr->nf;
  bool bad = (n4 < 1 || n4 > n_int);
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n_int; j += gridDim.x * blockDim.x) {
    const int2 ch = B.bin_child[j];
    const int c2[2] = {ch.x, ch.y};
    for (int k = 0; k < 2; ++k) {
      const int c = c2[k];
      if (c >= 0) bad |= c >= n_int || B.parent[c] != j;
      else bad |= (uint32_t)(~c) >= (uint32_t)nf || (nf > 1 && B.parent[n_int + ~c] != j);
    }
    if (j < n4) {
      const int4 r = reinterpret_cast<const int4*>(B.node4)[8 * j + 6];
      const int rr[4] = {r.x, r.y, r.z, r.w};
      for (int k = 0; k < 4; ++k) {
        const int c = rr[k];
        if (c == kNoChild) continue;
        bad |= c >= 0 ? c >= n4 : (uint32_t)(~c) >= (uint32_t)nf;
      }
    }
  }
  if (bad) atomicExch(&B.hdr->corrupt, 1);
}

// the header, the (empty) centroid bounds and the SAH build's state
__global__ void k_bvh_header(BvhHeader* h, int32_t nf, uint32_t* bounds, SahState* st) {
  if (threadIdx.x < 6) bounds[threadIdx.x] = threadIdx.x < 3 ? 0xffffffffu : 0u;
  for (uint32_t i = threadIdx.x; i < sizeof(SahState) / 4; i += blockDim.x) reinterpret_cast<uint32_t*>(st)[i] = 0u;
  if (threadIdx.x) return;
  h->nf = nf;
  h->n_int = nf > 1 ? nf - 1 : 1;
  h->n4 = 0;
  h->corrupt = 0;
  h->coarse = 0;
}

// scratch layout for build/refit
struct BuildScratch {
  uint32_t *keys_a, *keys_b, *vals_a, *vals_b, *hist, *arrive, *bounds, *totals;
  SahView sah;
  size_t total;
  BuildScratch(void* base, int32_t nf) {
    const int nblocks = (nf + kSortTile - 1) / kSortTile;
    const size_t n_int = nf > 1 ? (size_t)nf - 1 : 1;
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + bytes, 256); return r; };
    const size_t ka = take(sizeof(uint32_t) * nf), kb = take(sizeof(uint32_t) * nf);
    const size_t va = take(sizeof(uint32_t) * nf), vb = take(sizeof(uint32_t) * nf);
    const size_t hi = take(sizeof(uint32_t) * 256 * (size_t)nblocks);
    const size_t ar = take(sizeof(uint32_t) * n_int);
    const size_t bo = take(sizeof(uint32_t) * 8);
    const size_t to = take(sizeof(uint32_t) * kScanBlocks);
    // binned SAH build: centroids, boxes, task lists and bins of two levels,
    // left counts per chunk, small tasks
    sah.max_large = nf / (kSahSmall + 1) + 1;
    sah.max_small = nf + 1;
    sah.max_chunks = nf / kSahChunk + sah.max_large + 1;
    const size_t ce = take(sizeof(float4) * nf), pb = take(sizeof(float4) * 2 * (size_t)nf);
    const size_t t0 = take(sizeof(SahTask) * sah.max_large), t1 = take(sizeof(SahTask) * sah.max_large);
    const size_t b0 = take(sizeof(SahBins) * sah.max_large), b1 = take(sizeof(SahBins) * sah.max_large);
    const size_t c0 = take(sizeof(int) * sah.max_chunks), c1 = take(sizeof(int) * sah.max_chunks);
    const size_t cl = take(sizeof(uint32_t) * 3 * kSahBins * (size_t)sah.max_chunks);
    const size_t sm = take(sizeof(int4) * sah.max_small), st = take(sizeof(SahState));
    total = o;
    char* b = (char*)base;
    keys_a = (uint32_t*)(b + ka); keys_b = (uint32_t*)(b + kb);
    vals_a = (uint32_t*)(b + va); vals_b = (uint32_t*)(b + vb);
    hist = (uint32_t*)(b + hi); arrive = (uint32_t*)(b + ar); bounds = (uint32_t*)(b + bo);
    totals = (uint32_t*)(b + to);
    sah.cen = (float4*)(b + ce);
    sah.pbox = (float4*)(b + pb);
    sah.idx[0] = vals_a;
    sah.idx[1] = vals_b;
    sah.tasks[0] = (SahTask*)(b + t0);
    sah.tasks[1] = (SahTask*)(b + t1);
    sah.bins[0] = (SahBins*)(b + b0);
    sah.bins[1] = (SahBins*)(b + b1);
    sah.chunk_task[0] = (int*)(b + c0);
    sah.chunk_task[1] = (int*)(b + c1);
    sah.chunk_cnt = (uint32_t*)(b + cl);
    sah.small = (int4*)(b + sm);
    sah.st = (SahState*)(b + st);
  }
};

size_t bvh_scratch_bytes(int32_t nf) { return BuildScratch(nullptr, nf).total; }

static int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  const int64_t cap = 8 * (int64_t)num_sms();
  if (b > cap) b = cap;
  return b < 1 ? 1 : (int)b;
}

// The boxes of a tree whose arrivals are cleared, by the kernel before on the stream.
static void launch_boxes(const float* V, const int32_t* F, int32_t nf, BvhView& B, BuildScratch& S, cudaStream_t s) {
  ProfScope ps("k_refit", s);
  launch_chained(k_refit, grid_for(nf, kRefitLeaves), kRefitLeaves, 0, s, V, F, nf, B, S.arrive);
  launch_chained(k_node_boxes, grid_for(nf, 256), 256, 0, s, B);
}

void launch_refit(const float* V, const int32_t* F, int32_t nf, void* bvh, void* scratch, cudaStream_t s) {
  BvhView B = bvh_view(bvh, nf);
  BuildScratch S(scratch, nf);
  cudaMemsetAsync(S.arrive, 0, sizeof(uint32_t) * (nf > 1 ? (size_t)nf - 1 : 1), s);
  launch_boxes(V, F, nf, B, S, s);
}

// Binned SAH topology (see above).  Large levels: kSahFreeDepth levels of
// free splits, then median splits, which halve a task per level, so after
// ceil(log2(nf / kSahSmall)) + 1 more levels every task is small; small
// tasks take free splits to depth kSahSmallFreeDepth, then at most
// log2(kSahSmall) median levels: the tree is at most 63 deep, within the
// traversal's 64-entry stack.
// False when it could not be launched: the tree is then marked corrupt.
static bool launch_sah_topology(const float* V, const int32_t* F, int32_t nf, BvhView& B, BuildScratch& S,
                                cudaStream_t s) {
  launch_chained(k_sah_prims, grid_for(nf, 256), 256, 0, s, V, F, nf, S.bounds, S.sah, B);
  int levels = 0;
  if (nf > kSahSmall) {
    int lg = 0;
    while (((int64_t)kSahSmall << lg) < (int64_t)nf) ++lg;
    levels = kSahFreeDepth + lg + 2;
    if (levels > kSahMaxLevels) levels = kSahMaxLevels;
  }
  {
    ProfScope ps("sah_large_levels", s);
    // one CTA per 512 triangles: enough for the tasks of the last levels, and
    // a small mesh's barriers stay cheap
    int blocks = (nf + 511) / 512;
    int most = kSahBlocksPerSm * num_sms();
    if (most > kBarrierBlocks) most = kBarrierBlocks;
    if (blocks > most) blocks = most;
    const uint32_t* bounds = S.bounds;
    void* args[] = {&nf, &levels, &bounds, &S.sah, &B};
    const bool launched = launch_cooperative(blocks, [&](int n) {
      return cudaLaunchCooperativeKernel((const void*)k_sah_levels, dim3(n), dim3(kSahThreads), args, 0, s);
    });
    if (!launched) {
      cudaMemsetAsync(&B.hdr->corrupt, 1, sizeof(B.hdr->corrupt), s);
      return false;
    }
  }
  ProfScope ps("sah_small", s);
  // at most one task per two triangles, a CTA each; about kSahSmall / 2 in practice
  launch_chained(k_sah_small, grid_for(nf / 32 + 1, 1), 32 * kSahSmallWarps, 0, s, S.sah, B);
  return true;
}

void launch_scan_exclusive(const uint32_t* src, uint32_t* dst, int32_t m, uint32_t* totals, cudaStream_t s) {
  const int64_t tiles = ((int64_t)m + kScanTile - 1) / kScanTile;
  const int64_t per = (tiles + kScanBlocks - 1) / kScanBlocks;  // tiles per span
  const int blocks = (int)((tiles + per - 1) / per);
  if (blocks > 1) launch_chained(k_scan_totals, blocks, kScanThreads, 0, s, src, m, per * kScanTile, totals);
  launch_chained(k_scan_apply, blocks, kScanThreads, 0, s, src, dst, m, per * kScanTile, totals);
}

void launch_build(const float* V, const int32_t* F, int32_t nf, void* bvh, void* scratch, cudaStream_t s) {
  BvhView B = bvh_view(bvh, nf);
  BuildScratch S(scratch, nf);
  const int n_int = nf > 1 ? nf - 1 : 1;
  const bool sah = g_tuning.bvh_builder == 1 && nf > 1;
  {
    ProfScope ps(sah ? "sah_build" : "lbvh_build", s);
    k_bvh_header<<<1, 256, 0, s>>>(B.hdr, nf, S.bounds, S.sah.st);
    if (sah) {
      if (!launch_sah_topology(V, F, nf, B, S, s)) return;
    } else {
      k_centroid_bounds<<<grid_for(nf, 256), 256, 0, s>>>(V, F, nf, S.bounds);
      k_morton<<<grid_for(nf, 256), 256, 0, s>>>(V, F, nf, S.bounds, S.keys_a, S.vals_a);
      const int nblocks = (nf + kSortTile - 1) / kSortTile;
      uint32_t *kin = S.keys_a, *vin = S.vals_a, *kout = S.keys_b, *vout = S.vals_b;
      for (int shift = 0; shift < 32; shift += 8) {
        k_radix_hist<<<nblocks, kSortThreads, 0, s>>>(kin, nf, shift, S.hist);
        launch_scan_exclusive(S.hist, S.hist, 256 * nblocks, S.totals, s);
        k_radix_scatter<<<nblocks, kSortThreads, 0, s>>>(kin, vin, nf, shift, S.hist, kout, vout);
        uint32_t* t = kin; kin = kout; kout = t;
        t = vin; vin = vout; vout = t;
      }
      // after an even number of passes the sorted data is back in keys_a/vals_a
      k_gather_leaf_tri<<<grid_for(nf, 256), 256, 0, s>>>(vin, nf, B.leaf_tri);
      if (nf > 1) {
        k_karras<<<grid_for(nf - 1, 256), 256, 0, s>>>(kin, nf, B.bin_child, B.parent);
      } else {
        k_single_leaf<<<1, 1, 0, s>>>(B.bin_child, B.parent);
      }
    }
    // 4-wide topology: even-depth nodes, numbered by a scan
    uint32_t* flag = S.keys_b;  // free after the sort (unused by the SAH build)
    launch_chained(k_even_depth, grid_for(n_int, 256), 256, 0, s, B, flag, S.arrive);
    launch_scan_exclusive(flag, flag, n_int, S.totals, s);
    launch_chained(k_bin_to4, grid_for(n_int, 256), 256, 0, s, B, flag);
    launch_chained(k_node4_topology, grid_for(n_int, 256), 256, 0, s, B);
    launch_chained(k_validate, grid_for(n_int, 256), 256, 0, s, B);
  }
  launch_boxes(V, F, nf, B, S, s);
}

}  // namespace dt
