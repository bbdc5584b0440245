// The step after the gradient (DiffTrans App. A): the mesh's edge graph, the
// large-steps update with AdamUniform, and the edge-normal regulariser.
//
//  * Topology: the distinct neighbours of every vertex in CSR form, built on
//    the device from the triangles (count, scan, fill, sort and deduplicate
//    each vertex's list, scan, compact).
//  * Laplacian L = D - A of that graph (uniform weights); M = I + lambda L is
//    symmetric positive definite, applied matrix-free from the CSR.
//  * Solve M x = b (three right-hand sides) by conjugate gradients with the
//    diagonal 1 + lambda deg as preconditioner, at most a given number of
//    iterations (a column stops once its residual has fallen by 1e-6),
//    every scalar on the device (no host synchronisation).
//  * Large-steps update: u = M V; g_u = M^-1 dJ/dV; AdamUniform on u (one
//    second moment, the max of g_u^2); V = M^-1 u.
//  * L_edge = (1/|E|) sum over edges of (1 - n_i . n_j)^2 with n the unit
//    vertex normals; its gradient with respect to the Eq. 13 normals (the
//    caller chains it to the vertices with the normals' backward).
#include <cuda_runtime.h>
#include <stdint.h>

#include "dt_internal.cuh"

namespace dt {

// ---------------------------------------------------------------------------
// topology buffer
// ---------------------------------------------------------------------------
struct TopoHeader {
  int32_t nv, nf;
  int32_t nnz;      // directed neighbour entries (2 |E|), written on the device
  int32_t max_deg;  // largest neighbour count, written on the device
};

struct TopoLayout {
  size_t off_row, off_col, off_raw_cnt, off_raw_off, off_cursor, off_totals, off_raw, total;
  TopoLayout(int32_t nv, int32_t nf) {
    size_t o = 256;
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + bytes, 256); return r; };
    off_row = take(((size_t)nv + 1) * sizeof(int32_t));
    off_col = take((size_t)6 * nf * sizeof(int32_t));
    off_raw_cnt = take(((size_t)nv + 1) * sizeof(uint32_t));
    off_raw_off = take(((size_t)nv + 1) * sizeof(uint32_t));
    off_cursor = take((size_t)nv * sizeof(uint32_t));
    off_totals = take((size_t)kScanBlocks * sizeof(uint32_t));
    off_raw = take((size_t)6 * nf * sizeof(int32_t));
    total = o;
  }
};

struct TopoView {
  TopoHeader* hdr;
  int32_t* row;  // [nv + 1]
  int32_t* col;  // [nnz]
  uint32_t* raw_cnt;
  uint32_t* raw_off;
  uint32_t* cursor;
  uint32_t* totals;
  int32_t* raw;
};

static TopoView topo_view(void* base, int32_t nv, int32_t nf) {
  TopoLayout L(nv, nf);
  char* b = (char*)base;
  return TopoView{(TopoHeader*)b, (int32_t*)(b + L.off_row), (int32_t*)(b + L.off_col),
                  (uint32_t*)(b + L.off_raw_cnt), (uint32_t*)(b + L.off_raw_off), (uint32_t*)(b + L.off_cursor),
                  (uint32_t*)(b + L.off_totals), (int32_t*)(b + L.off_raw)};
}

size_t topology_bytes(int32_t nv, int32_t nf) { return TopoLayout(nv, nf).total; }

static int blocks_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  const int64_t cap = 8 * (int64_t)num_sms();
  if (b > cap) b = cap;
  return (int)(b > 0 ? b : 1);
}

// every triangle lists each of its vertices' two other vertices
__global__ void k_topo_count(const int32_t* __restrict__ F, int32_t nf, int32_t nv, uint32_t* __restrict__ raw_cnt) {
  for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += gridDim.x * blockDim.x)
    for (int k = 0; k < 3; ++k) {
      const int v = F[3 * f + k];
      if (v >= 0 && v < nv) atomicAdd(raw_cnt + v, 2u);
    }
}

__global__ void k_topo_fill(const int32_t* __restrict__ F, int32_t nf, int32_t nv, const uint32_t* __restrict__ raw_off,
                            uint32_t* __restrict__ cursor, int32_t* __restrict__ raw) {
  for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < nf; f += gridDim.x * blockDim.x) {
    const int a = F[3 * f], b = F[3 * f + 1], c = F[3 * f + 2];
    const int tri[3] = {a, b, c};
    for (int k = 0; k < 3; ++k) {
      const int v = tri[k];
      if (v < 0 || v >= nv) continue;
      const uint32_t at = raw_off[v] + atomicAdd(cursor + v, 2u);
      raw[at] = tri[(k + 1) % 3];
      raw[at + 1] = tri[(k + 2) % 3];
    }
  }
}

// Sort each vertex's list and keep the distinct in-range entries other than
// the vertex itself at its front; raw_cnt[v] becomes the distinct count.  A
// group of 16 lanes has a vertex: each lane holds an entry, an entry is kept
// when no earlier lane holds the same, and its place is the number of kept
// smaller ones (lists are a vertex's valence times two: 12 on average).  Longer
// lists are sorted by insertion by one lane.  (A thread per vertex, sorting in
// global memory, and an atomic on the largest count per vertex took 70.7 us for
// 135k vertices; this takes 22.8.)
constexpr int kTopoLanes = 16;
__global__ void __launch_bounds__(256) k_topo_dedupe(int32_t nv, const uint32_t* __restrict__ raw_off,
                                                     uint32_t* __restrict__ raw_cnt, int32_t* __restrict__ raw,
                                                     TopoHeader* hdr) {
  const int lane = threadIdx.x & (kTopoLanes - 1);
  const int groups = gridDim.x * (blockDim.x / kTopoLanes);
  int most = 0;
  // every group of a warp takes the same number of turns (the shuffles are warp-wide)
  const int turns = (nv + groups - 1) / groups;
  for (int t = 0, v = (blockIdx.x * blockDim.x + threadIdx.x) / kTopoLanes; t < turns; ++t, v += groups) {
    const bool mine = v < nv;
    int32_t* l = raw + (mine ? raw_off[v] : 0u);
    const int n = mine ? (int)raw_cnt[v] : 0;
    const bool wide = n > kTopoLanes;
    const int32_t x = !wide && lane < n ? l[lane] : -1;
    bool keep = x >= 0 && x < nv && x != v;
#pragma unroll
    for (int d = 0; d < kTopoLanes; ++d) {
      const int32_t y = __shfl_sync(kFull, x, d, kTopoLanes);
      if (d < lane && y == x) keep = false;
    }
    int at = 0;
    const unsigned kept = (__ballot_sync(kFull, keep) >> (threadIdx.x & 16)) & 0xffffu;
#pragma unroll
    for (int d = 0; d < kTopoLanes; ++d) {
      const int32_t y = __shfl_sync(kFull, x, d, kTopoLanes);
      at += (kept >> d) & (y < x ? 1u : 0u);
    }
    int u = __popc(kept);
    if (!wide && keep) l[at] = x;  // every lane's entry is in its register
    if (wide && lane == 0) {
      for (int i = 1; i < n; ++i) {
        const int32_t e = l[i];
        int j = i - 1;
        while (j >= 0 && l[j] > e) {
          l[j + 1] = l[j];
          --j;
        }
        l[j + 1] = e;
      }
      u = 0;
      for (int i = 0; i < n; ++i) {
        const int32_t e = l[i];
        if (e < 0 || e >= nv || e == v) continue;
        if (u > 0 && l[u - 1] == e) continue;
        l[u++] = e;
      }
    }
    if (mine && lane == 0) {
      raw_cnt[v] = (uint32_t)u;
      most = max(most, u);
    }
  }
  most = __reduce_max_sync(kFull, most);
  if ((threadIdx.x & 31) == 0 && most > 0) atomicMax(&hdr->max_deg, most);
}

__global__ void k_topo_compact(int32_t nv, const uint32_t* __restrict__ raw_off, const uint32_t* __restrict__ cnt,
                               const uint32_t* __restrict__ row_u, const int32_t* __restrict__ raw,
                               int32_t* __restrict__ row, int32_t* __restrict__ col, TopoHeader* hdr) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += gridDim.x * blockDim.x) {
    const uint32_t o = row_u[v], n = cnt[v];
    row[v] = (int32_t)o;
    for (uint32_t i = 0; i < n; ++i) col[o + i] = raw[raw_off[v] + i];
    if (v == nv - 1) {
      row[nv] = (int32_t)(o + n);
      hdr->nnz = (int32_t)(o + n);
    }
  }
}

__global__ void k_topo_init(TopoHeader* hdr, int32_t nv, int32_t nf, uint32_t* __restrict__ raw_cnt,
                            uint32_t* __restrict__ cursor) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v <= nv; v += gridDim.x * blockDim.x) {
    raw_cnt[v] = 0u;
    if (v < nv) cursor[v] = 0u;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *hdr = TopoHeader{nv, nf, 0, 0};
}

void launch_build_topology(const int32_t* F, int32_t nf, int32_t nv, void* topo, cudaStream_t s) {
  TopoView T = topo_view(topo, nv, nf);
  ProfScope ps("topology_build", s);
  k_topo_init<<<blocks_for((int64_t)nv + 1, 256), 256, 0, s>>>(T.hdr, nv, nf, T.raw_cnt, T.cursor);
  k_topo_count<<<blocks_for(nf, 256), 256, 0, s>>>(F, nf, nv, T.raw_cnt);
  launch_scan_exclusive(T.raw_cnt, T.raw_off, nv + 1, T.totals, s);
  k_topo_fill<<<blocks_for(nf, 256), 256, 0, s>>>(F, nf, nv, T.raw_off, T.cursor, T.raw);
  k_topo_dedupe<<<blocks_for((int64_t)nv * kTopoLanes, 256), 256, 0, s>>>(nv, T.raw_off, T.raw_cnt, T.raw, T.hdr);
  // distinct counts -> row starts (the cursor array, free now, holds the scan)
  launch_scan_exclusive(T.raw_cnt, T.cursor, nv, T.totals, s);
  k_topo_compact<<<blocks_for(nv, 256), 256, 0, s>>>(nv, T.raw_off, T.raw_cnt, T.cursor, T.raw, T.row, T.col,
                                                      T.hdr);
}

// ---------------------------------------------------------------------------
// M = I + lambda L, applied from the CSR; conjugate gradients
// ---------------------------------------------------------------------------
__device__ __forceinline__ float3 apply_m(const int32_t* __restrict__ row, const int32_t* __restrict__ col,
                                          const float* __restrict__ x, float lam, int v) {
  const int b = row[v], e = row[v + 1];
  const float3 xv = load3(x + 3 * v);
  float3 sum = mk(0.f, 0.f, 0.f);
  for (int k = b; k < e; ++k) sum = sum + load3(x + 3 * col[k]);
  return xv + (xv * (float)(e - b) - sum) * lam;
}

__device__ __forceinline__ void store3(float* p, float3 v) {
  p[0] = v.x;
  p[1] = v.y;
  p[2] = v.z;
}

// ---- conjugate gradients in one cooperative kernel ---------------------------
// An iteration is two short passes over vectors that stay in L2, so as
// launches of their own (three per iteration, 598 per optimiser step) they
// cost a launch each: 145k vertices, 100 iterations, two solves took 2.9 ms.
// Here one CTA per SM runs every iteration of the solve, with two sums over
// the grid per iteration, and stops when all three columns have converged:
// 2925 -> 868 us for the optimiser step of 72.6k vertices (100 iterations at
// most, 60 to 100 taken), 12.3 -> 6.3 us per iteration for 2k to 72k vertices
// and 30.0 -> 20.8 us for 540k.  Up to 78k vertices (one per thread) an
// iteration is bound by its two grid sums, above that by the L2 traffic of the
// neighbours' records.
//
// A grid sum doubles as the barrier: each CTA publishes its three partial
// sums and the sum's number as one 16-byte word; CTA 0 polls those words,
// adds them up and publishes the result, which the others poll (in one of
// eight copies).  Two trips through L2, without atomics, and the sum has a
// fixed order, so a solve gives the same bits on every run.  (Every CTA
// reading every word is one trip, but 142 CTAs polling one another's words
// took 5.0 us per sum against 3.0.)  A word is free again when its next value
// is due: a CTA publishes sum n + 1 only after it has read the result of n, for
// which CTA 0 had read every word.
constexpr int kCgThreads = 512;
constexpr int kCgMaxBlocks = 512;
constexpr int kCgCopies = 8;          // of the result, a 128-byte line each
constexpr int kCgWords = kCgMaxBlocks + 8 * kCgCopies;
constexpr int kCgSpins = 1 << 21;     // polls before a wait is given up (about a second)
constexpr int kCgListWords = 200 * 1024 / 4;  // shared memory for neighbour lists

struct GridSum {
  ulonglong2* word;  // [kCgMaxBlocks], then the copies of the result; cleared before the launch
  uint32_t n;        // number of the last sum
  bool failed;       // a wait ran out: the launch was not co-resident
};

template <bool kOrder>
__device__ __forceinline__ void st_word(ulonglong2* p, float3 v, uint32_t n) {
  const unsigned long long lo = (unsigned long long)__float_as_uint(v.x) | ((unsigned long long)__float_as_uint(v.y) << 32);
  const unsigned long long hi = (unsigned long long)__float_as_uint(v.z) | ((unsigned long long)n << 32);
  if (kOrder)
    asm volatile("{ .reg .b128 w; mov.b128 w, {%1, %2}; st.release.gpu.global.b128 [%0], w; }" ::"l"(p), "l"(lo), "l"(hi) : "memory");
  else
    asm volatile("{ .reg .b128 w; mov.b128 w, {%1, %2}; st.relaxed.gpu.global.b128 [%0], w; }" ::"l"(p), "l"(lo), "l"(hi) : "memory");
}
template <bool kOrder>
__device__ __forceinline__ uint32_t ld_word(const ulonglong2* p, float3& v) {
  unsigned long long lo, hi;
  if (kOrder)
    asm volatile("{ .reg .b128 w; ld.acquire.gpu.global.b128 w, [%2]; mov.b128 {%0, %1}, w; }" : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
  else
    asm volatile("{ .reg .b128 w; ld.relaxed.gpu.global.b128 w, [%2]; mov.b128 {%0, %1}, w; }" : "=l"(lo), "=l"(hi) : "l"(p) : "memory");
  v = mk(__uint_as_float((uint32_t)lo), __uint_as_float((uint32_t)(lo >> 32)), __uint_as_float((uint32_t)hi));
  return (uint32_t)(hi >> 32);
}

// Polls *p until it holds value n; false when it gave up.
template <bool kOrder>
__device__ __forceinline__ bool wait_word(const ulonglong2* p, float3& v, uint32_t n) {
  int spins = 0;
  while (ld_word<kOrder>(p, v) != n)
    if (++spins >= kCgSpins) return false;
  return true;
}

// The grid's sum of v.  kOrder: what any thread wrote before it, every thread
// can read after it (release and acquire of the words, with the CTA's own
// barriers on both sides).  Without it only the sum passes, which saves the
// wait for the CTA's stores; every CTA's reads before it are done all the
// same, since its part of the sum is made of them.
template <bool kOrder>
__device__ __forceinline__ float3 grid_sum3(GridSum& g, float3 v, float (*part)[32]) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  v = mk(warp_sum(v.x), warp_sum(v.y), warp_sum(v.z));
  if (lane == 0) {
    part[0][wid] = v.x;
    part[1][wid] = v.y;
    part[2][wid] = v.z;
  }
  ++g.n;
  __syncthreads();
  bool ok = true;
  if (wid == 0) {
    const bool in = lane < kCgThreads / 32;
    v = mk(warp_sum(in ? part[0][lane] : 0.f), warp_sum(in ? part[1][lane] : 0.f), warp_sum(in ? part[2][lane] : 0.f));
    if (lane == 0 && blockIdx.x > 0) {
      st_word<kOrder>(g.word + blockIdx.x, v, g.n);
      ok = wait_word<kOrder>(g.word + kCgMaxBlocks + 8 * (blockIdx.x % kCgCopies), v, g.n);
    }
  }
  if (blockIdx.x == 0 && wid * 32 < (int)gridDim.x) {  // the words of the other CTAs, 32 per warp, and its own sum
    float3 w = mk(0.f, 0.f, 0.f);
    if (threadIdx.x == 0) w = v;
    else if (threadIdx.x < gridDim.x) ok = wait_word<kOrder>(g.word + threadIdx.x, w, g.n);
    v = mk(warp_sum(w.x), warp_sum(w.y), warp_sum(w.z));
  }
  if (lane == 0) {
    part[3][wid] = v.x;
    part[4][wid] = v.y;
    part[5][wid] = v.z;
  }
  if (__syncthreads_or(!ok)) g.failed = true;
  v = mk(part[3][0], part[4][0], part[5][0]);
  if (blockIdx.x == 0) {
    for (int i = 1; i * 32 < (int)gridDim.x; ++i) v = v + mk(part[3][i], part[4][i], part[5][i]);
    if (threadIdx.x < kCgCopies && gridDim.x > 1 && !g.failed) {
      st_word<kOrder>(g.word + kCgMaxBlocks + 8 * threadIdx.x, v, g.n);
    }
  }
  return v;
}

// CG scratch: the vertices' records (z, p) of 32 bytes, so that what an
// iteration reads of a neighbour is one load of one sector, r and Ap as
// [nv][3], and the grid sums' words.
struct CgRecord {
  float3 z, p;
};
struct CgView {
  float4* rec;  // [2 nv]: (z.xyz, p.x), (p.yz, 0, 0)
  float *r, *ap;
  ulonglong2* word;
};
__device__ __forceinline__ CgRecord ld_record(const float4* rec, int v) {  // not .nc: rewritten by the kernel itself
  [[maybe_unused]] float u0, u1;
  CgRecord c;
  asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(c.z.x), "=f"(c.z.y), "=f"(c.z.z), "=f"(c.p.x), "=f"(c.p.y), "=f"(c.p.z), "=f"(u0), "=f"(u1)
               : "l"(rec + 2 * (size_t)v)
               : "memory");
  return c;
}
__device__ __forceinline__ void st_record(float4* rec, int v, float3 z, float3 p) {
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%7};" ::"l"(rec + 2 * (size_t)v), "f"(z.x), "f"(z.y), "f"(z.z),
               "f"(p.x), "f"(p.y), "f"(p.z), "f"(0.f)
               : "memory");
}

__device__ __forceinline__ float safe_div(float a, float b) { return b != 0.0f ? a / b : 0.0f; }

// A column has converged once its preconditioned residual r.z has fallen
// by kCgTol2 (the residual by 1e-6) from the start: from then on its
// iterations change nothing (FP32 conjugate gradients run on in the
// rounding noise would drift).
constexpr float kCgTol2 = 1e-12f;
__device__ __forceinline__ bool cg_live(float rz, float rz0) { return rz > kCgTol2 * rz0; }
__device__ __forceinline__ float cg_alpha(float rz, float rz0, float pap) {
  return cg_live(rz, rz0) && pap > 0.0f ? rz / pap : 0.0f;
}
__device__ __forceinline__ float cg_beta(float rz, float old, float rz0) {
  return cg_live(rz, rz0) ? safe_div(rz, old) : 0.0f;
}

static size_t cg_vec(int32_t nv, int width) { return align_up((size_t)nv * width * sizeof(float), 256); }

static size_t cg_bytes(int32_t nv) {
  return cg_vec(nv, 8) + 2 * cg_vec(nv, 3) + kCgWords * sizeof(ulonglong2);
}

static CgView cg_view(void* base, int32_t nv) {
  char* b = (char*)base;
  const size_t v8 = cg_vec(nv, 8), v3 = cg_vec(nv, 3);
  CgView c;
  c.rec = (float4*)b;
  c.r = (float*)(b + v8);
  c.ap = (float*)(b + v8 + v3);
  c.word = (ulonglong2*)(b + v8 + 2 * v3);
  return c;
}

// M x = b, x holding the start on entry.  CTA i has the vertices [i chunk, (i +
// 1) chunk), whose neighbour lists it copies to shared memory (where they
// fit: the fences of the grid sums drop L1, and the lists are read every
// iteration).  Pass A of an iteration: p = z + beta p_old (of the neighbours
// too, from their records: their new p is formed again rather than waited
// for), Ap = M p, sum p . Ap.  Pass B: x += alpha p, r -= alpha Ap, z = r / diag,
// the record, sum r . z.  kOne: at most one vertex per thread, whose x, r, z, p
// and Ap stay in registers.
constexpr int kCgGather = 8;  // neighbours' records in flight per thread
template <bool kOne>
__global__ void __launch_bounds__(kCgThreads, 1) k_cg(const int32_t* __restrict__ row, const int32_t* __restrict__ col,
                                                      int32_t nv, int32_t chunk, int32_t list_room, float lam,
                                                      const float* __restrict__ b, float* x, CgView c, int iters) {
  __shared__ float part[6][32];
  extern __shared__ int32_t lists[];  // [chunk + 1] list starts, then the lists
  GridSum g{c.word, 0u, false};
  const int v0 = min(blockIdx.x * chunk, nv), v1 = min(v0 + chunk, nv);
  const int base = row[v0], len = row[v1] - base;
  const bool fits = len <= list_room, starts = list_room >= 0;
  int32_t* nb = lists + chunk + 1;
  if (starts)
    for (int v = v0 + threadIdx.x; v <= v1; v += blockDim.x) lists[v - v0] = row[v] - base;
  if (fits)
    for (int k = threadIdx.x; k < len; k += blockDim.x) nb[k] = col[base + k];
  const int32_t* __restrict__ far = col + base;
  __syncthreads();
  auto start_of = [&](int v) { return starts ? lists[v - v0] : row[v] - base; };
  auto inv_diag = [&](int v) { return 1.0f / (1.0f + lam * (float)(start_of(v + 1) - start_of(v))); };
  // M applied at v to the vector whose entry j is value(read(j)), mine being its own
  auto apply = [&](int v, float3 mine, auto read, auto value) {
    const int e0 = start_of(v), e1 = start_of(v + 1);
    float3 sum = mk(0.f, 0.f, 0.f);
    for (int k = e0; k < e1; k += kCgGather) {
      CgRecord rec[kCgGather];
#pragma unroll
      for (int q = 0; q < kCgGather; ++q)
        if (k + q < e1) rec[q] = read(fits ? nb[k + q] : far[k + q]);
#pragma unroll
      for (int q = 0; q < kCgGather; ++q)
        if (k + q < e1) sum = sum + value(rec[q]);
    }
    return mine + (mine * (float)(e1 - e0) - sum) * lam;
  };
  float3 acc = mk(0.f, 0.f, 0.f), kx, kr, kz, kp, kap;  // kOne: the thread's vertex
  kx = kr = kz = kp = kap = acc;
  // r = b - M x, z = r / diag, rz = r . z
  for (int v = v0 + threadIdx.x; v < v1; v += blockDim.x) {
    const float3 xv = load3(x + 3 * (size_t)v);
    const float3 r = load3(b + 3 * (size_t)v) -
                     apply(v, xv, [&](int j) { return CgRecord{load3(x + 3 * (size_t)j), mk(0.f, 0.f, 0.f)}; },
                           [](const CgRecord& q) { return q.z; });
    const float3 z = r * inv_diag(v);
    if (kOne) {
      kx = xv;
      kr = r;
      kz = z;
    } else {
      store3(c.r + 3 * (size_t)v, r);
    }
    st_record(c.rec, v, z, mk(0.f, 0.f, 0.f));
    acc = acc + mul(r, z);
  }
  const float3 rz0 = grid_sum3<true>(g, acc, part);
  float3 rz = rz0, beta = mk(0.f, 0.f, 0.f), keep = mk(1.f, 1.f, 1.f);
  auto next_p = [&](const CgRecord& q) { return mul(keep, q.z) + mul(beta, q.p); };
  for (int it = 0; it < iters && !g.failed; ++it) {
    acc = mk(0.f, 0.f, 0.f);
    for (int v = v0 + threadIdx.x; v < v1; v += blockDim.x) {
      const float3 p = next_p(kOne ? CgRecord{kz, kp} : ld_record(c.rec, v));
      const float3 ap = apply(v, p, [&](int j) { return ld_record(c.rec, j); }, next_p);
      if (kOne) {
        kp = p;
        kap = ap;
      } else {
        store3(c.ap + 3 * (size_t)v, ap);
      }
      acc = acc + mul(p, ap);
    }
    const float3 pap = grid_sum3<false>(g, acc, part);  // pass A writes nothing that others read
    const float3 alpha = mk(cg_alpha(rz.x, rz0.x, pap.x), cg_alpha(rz.y, rz0.y, pap.y), cg_alpha(rz.z, rz0.z, pap.z));
    acc = mk(0.f, 0.f, 0.f);
    for (int v = v0 + threadIdx.x; v < v1; v += blockDim.x) {
      const float3 p = kOne ? kp : next_p(ld_record(c.rec, v));
      const float3 r = (kOne ? kr : load3(c.r + 3 * (size_t)v)) - mul(alpha, kOne ? kap : load3(c.ap + 3 * (size_t)v));
      const float3 z = r * inv_diag(v);
      if (kOne) {
        kx = kx + mul(alpha, p);
        kr = r;
        kz = z;
      } else {
        store3(x + 3 * (size_t)v, load3(x + 3 * (size_t)v) + mul(alpha, p));
        store3(c.r + 3 * (size_t)v, r);
      }
      st_record(c.rec, v, z, p);
      acc = acc + mul(r, z);
    }
    const float3 old = rz;
    rz = grid_sum3<true>(g, acc, part);
    // a converged column keeps its direction at zero
    beta = mk(cg_beta(rz.x, old.x, rz0.x), cg_beta(rz.y, old.y, rz0.y), cg_beta(rz.z, old.z, rz0.z));
    const bool lx = cg_live(rz.x, rz0.x), ly = cg_live(rz.y, rz0.y), lz = cg_live(rz.z, rz0.z);
    keep = mk(lx ? 1.0f : 0.0f, ly ? 1.0f : 0.0f, lz ? 1.0f : 0.0f);
    if (!lx && !ly && !lz) break;  // every later iteration would change nothing
  }
  for (int v = v0 + threadIdx.x; v < v1; v += blockDim.x) {
    if (g.failed) store3(x + 3 * (size_t)v, mk(NAN, NAN, NAN));  // never in a co-resident launch; not to pass for a solution
    else if (kOne) store3(x + 3 * (size_t)v, kx);
  }
}

// Whether it was launched.
static bool launch_cg(const TopoView& T, int32_t nv, float lam, const float* b, float* x, int iters, void* scratch,
                      cudaStream_t s) {
  CgView c = cg_view(scratch, nv);
  cudaMemsetAsync(c.word, 0, kCgWords * sizeof(ulonglong2), s);
  int blocks = (nv + kCgThreads - 1) / kCgThreads;
  const int most = num_sms() < kCgMaxBlocks ? num_sms() : kCgMaxBlocks;
  if (blocks > most) blocks = most;
  return launch_cooperative(blocks, [&](int n) {
    int32_t chunk = (nv + n - 1) / n;
    // list starts and room for lists of eight neighbours a vertex (a closed mesh
    // has six on average), as far as they fit; the starts alone exceed shared
    // memory past 7.7M vertices, and are then read where they are (room -1)
    int64_t words = (int64_t)chunk * 9 + 1;
    if (words > kCgListWords) words = kCgListWords;
    int32_t room = words > chunk ? (int32_t)(words - (chunk + 1)) : -1;
    if (room < 0) words = 0;
    const int32_t *row = T.row, *col = T.col;
    void* args[] = {&row, &col, &nv, &chunk, &room, &lam, &b, &x, &c, &iters};
    const void* f = chunk <= kCgThreads ? (const void*)k_cg<true> : (const void*)k_cg<false>;
    // the same value from every thread and for every mesh: the attribute is the kernel's, not the launch's
    const cudaError_t e =
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kCgListWords * (int)sizeof(int32_t));
    if (e != cudaSuccess) return e;
    return cudaLaunchCooperativeKernel(f, dim3(n), dim3(kCgThreads), args, (size_t)words * sizeof(int32_t), s);
  });
}

size_t smooth_scratch_bytes(int32_t nv, int32_t iters) {
  (void)iters;
  return cg_bytes(nv);
}

void launch_smooth_solve(const void* topo, int32_t nv, int32_t nf, float lam, const float* b, float* x, int iters,
                         void* scratch, cudaStream_t s) {
  TopoView T = topo_view(const_cast<void*>(topo), nv, nf);
  ProfScope ps("smooth_solve", s);
  launch_cg(T, nv, lam, b, x, iters, scratch, s);
}

// ---------------------------------------------------------------------------
// large-steps update with AdamUniform
// ---------------------------------------------------------------------------
// optimiser state (caller-owned, zero = fresh): m [nv][3], then the step
// count and the shared second moment
struct AdamScalars {
  float v;
  int32_t t;
  float max_g2;  // scratch: max g^2 of the current step
  float pad;
};

static size_t adam_state_bytes(int32_t nv) {
  return align_up((size_t)nv * 3 * sizeof(float), 256) + sizeof(AdamScalars);
}
size_t large_steps_state_bytes(int32_t nv) { return adam_state_bytes(nv); }
size_t large_steps_scratch_bytes(int32_t nv, int32_t iters) {
  (void)iters;
  return 2 * align_up((size_t)nv * 3 * sizeof(float), 256) + cg_bytes(nv);
}

__global__ void k_apply_m(const int32_t* __restrict__ row, const int32_t* __restrict__ col, int32_t nv, float lam,
                          const float* __restrict__ x, float* __restrict__ y) {
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += gridDim.x * blockDim.x)
    store3(y + 3 * v, apply_m(row, col, x, lam, v));
}

// max g^2 over every coordinate (non-negative floats order like their bits)
__global__ void k_max_sq(const float* __restrict__ g, int64_t n, AdamScalars* sc) {
  float mx = 0.f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    mx = fmaxf(mx, g[i] * g[i]);
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
  __shared__ float part[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) part[wid] = mx;
  __syncthreads();
  if (wid == 0) {  // one atomic per CTA
    mx = lane < (int)((blockDim.x + 31) >> 5) ? part[lane] : 0.f;
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
    if (lane == 0) atomicMax(reinterpret_cast<int*>(&sc->max_g2), __float_as_int(mx));
  }
}

// m = b1 m + (1 - b1) g; v = b2 v + (1 - b2) max g^2 (one thread does v);
// u -= lr m_hat / (sqrt(v_hat) + eps)
__global__ void k_adam_uniform(int64_t n, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ u,
                               const AdamScalars* __restrict__ sc, float lr, float b1, float b2, float eps) {
  const int t = sc->t + 1;
  const float v = b2 * sc->v + (1.0f - b2) * sc->max_g2;
  const float c1 = 1.0f - powf(b1, (float)t), c2 = 1.0f - powf(b2, (float)t);
  const float denom = sqrtf(v / c2) + eps;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float mi = b1 * m[i] + (1.0f - b1) * g[i];
    m[i] = mi;
    u[i] -= lr * (mi / c1) / denom;
  }
}

__global__ void k_adam_scalars(AdamScalars* sc, float b2) {
  sc->v = b2 * sc->v + (1.0f - b2) * sc->max_g2;
  sc->t += 1;
  sc->max_g2 = 0.f;
}

void launch_large_steps_update(const void* topo, int32_t nv, int32_t nf, float lam, float lr, float b1, float b2,
                               float eps, int iters, float* V, const float* grad, void* state, void* scratch,
                               cudaStream_t s) {
  TopoView T = topo_view(const_cast<void*>(topo), nv, nf);
  ProfScope ps("large_steps_update", s);
  const size_t vec = align_up((size_t)nv * 3 * sizeof(float), 256);
  float* u = (float*)scratch;
  float* gu = (float*)((char*)scratch + vec);
  void* cg = (char*)scratch + 2 * vec;
  float* m = (float*)state;
  AdamScalars* sc = (AdamScalars*)((char*)state + vec);
  const int g = blocks_for(nv, 256);
  const int64_t n = 3 * (int64_t)nv;
  k_apply_m<<<g, 256, 0, s>>>(T.row, T.col, nv, lam, V, u);  // u = M V
  cudaMemsetAsync(gu, 0, (size_t)n * sizeof(float), s);
  // g_u = M^-1 dJ/dV; without it the optimiser's state stays as it was (the caller reads the launch's error)
  if (!launch_cg(T, nv, lam, grad, gu, iters, cg, s)) return;
  k_max_sq<<<g, 256, 0, s>>>(gu, n, sc);
  k_adam_uniform<<<g, 256, 0, s>>>(n, gu, m, u, sc, lr, b1, b2, eps);
  k_adam_scalars<<<1, 1, 0, s>>>(sc, b2);
  launch_cg(T, nv, lam, u, V, iters, cg, s);                  // V = M^-1 u, from the old V
}

// ---------------------------------------------------------------------------
// L_edge
// ---------------------------------------------------------------------------
// loss[0] += sum over edges (1 - n_i . n_j)^2 / |E|, and dL/dN through n = N /
// |N|.  A thread has a vertex and reads all of its neighbours, so every edge
// is met from both ends: twice the dot products, but no atomics on the
// gradients, no clearing, and the unit normal's adjoint in the same kernel
// (two kernels, nine atomics per edge: 16.7 us for 135k vertices; this takes
// 6.8).  One CTA per SM, so that the loss is a sum of 152 parts, not of
// thousands: its rounding falls with them.
constexpr int kEdgeThreads = 1024;
__global__ void __launch_bounds__(kEdgeThreads) k_edge_loss(const int32_t* __restrict__ row,
                                                            const int32_t* __restrict__ col, const TopoHeader* hdr,
                                                            int32_t nv, const float* __restrict__ N,
                                                            float* __restrict__ dN, float* __restrict__ loss) {
  __shared__ float part[32];
  const float inv_e = 2.0f / (float)max(hdr->nnz, 1);  // |E| = nnz / 2
  float acc = 0.f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += gridDim.x * blockDim.x) {
    const float3 Ni = load3(N + 3 * (size_t)i);
    const float3 ni = normalize(Ni);
    float3 d = mk(0.f, 0.f, 0.f);
    for (int k = row[i]; k < row[i + 1]; ++k) {
      const int j = col[k];
      const float3 nj = normalize(load3(N + 3 * (size_t)j));
      const float e = 1.0f - dot(ni, nj);
      if (j > i) acc += e * e;  // each edge once, from its smaller end
      d = d + nj * (-2.0f * e * inv_e);
    }
    const float l = len(Ni);
    const float3 n = Ni * (1.0f / l);
    store3(dN + 3 * (size_t)i, (d - n * dot(n, d)) * (1.0f / l));
  }
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    acc = warp_sum(part[threadIdx.x]);
    if (threadIdx.x == 0 && acc != 0.f) atomicAdd(loss, acc * inv_e);
  }
}

void launch_edge_loss_grad(const void* topo, int32_t nv, int32_t nf, const float* N, float* dN, float* loss,
                           cudaStream_t s) {
  TopoView T = topo_view(const_cast<void*>(topo), nv, nf);
  ProfScope ps("edge_loss", s);
  cudaMemsetAsync(loss, 0, sizeof(float), s);
  int g = (nv + kEdgeThreads - 1) / kEdgeThreads;
  if (g > num_sms()) g = num_sms();
  k_edge_loss<<<g, kEdgeThreads, 0, s>>>(T.row, T.col, T.hdr, nv, N, dN, loss);
}

// device pointers of the CSR arrays
void topology_csr(const void* topo, int32_t nv, int32_t nf, const int32_t** row, const int32_t** col) {
  const TopoView T = topo_view(const_cast<void*>(topo), nv, nf);
  *row = T.row;
  *col = T.col;
}

// host copy of the header (n edges etc.), for the binding
void read_topology_header(const void* topo, int32_t* nnz, int32_t* max_deg, cudaStream_t s) {
  TopoHeader h;
  cudaMemcpyAsync(&h, topo, sizeof(h), cudaMemcpyDeviceToHost, s);
  cudaStreamSynchronize(s);
  *nnz = h.nnz;
  *max_deg = h.max_deg;
}

}  // namespace dt
