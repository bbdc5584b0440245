// Spatially varying absorption (DiffTrans Eq. 11 with mu_t(x) = sigma +
// G(x)): G is a dense grid of per-channel rates at the nodes of an
// nx x ny x nz lattice over a box, read with trilinear interpolation at
// positions clamped to the box.  Over an interior segment o + s d, s in
// [0, t], the optical depth gains the sum of Eq. 11 over steps of length h
// from the segment's start: m = floor(t / h) full steps (at most
// kMaxMediumSteps) and a last one of length r = t - m h, each sampled at its
// midpoint and weighted by its length.  The sum is continuous in t (the
// partial step grows into the next full one), so only the partial step
// depends on t:
//   dS/dt = G(x_m) + (r / 2) dG/dx(x_m) d,
// and at fixed t every sample moves with o and d:
//   dS/do = sum_i w_i dG/dx(x_i),  dS/dd = sum_i w_i s_i dG/dx(x_i).
// The forward shading pass and the adjoint evaluate S and dS/dt; a separate
// pass over the interior segments of each level adds the o and d terms to
// their adjoint records and scatters dJ/dS w_i into the eight nodes of each
// sample's cell.
//
// G may instead be a multi-resolution hash texture (Sec. 3.3's 3D texture
// after Instant-NGP): the sum over up to 16 levels of the trilinear
// interpolation of a cubic lattice over the same box, whose corners are
// entries of the level's table slice, dense when the lattice fits it and
// otherwise at Instant-NGP's spatial hash.  Every sum above then runs level
// by level: the same steps, each level's cell and weights, its own scale.
#pragma once

#include <type_traits>

#include "dt_internal.cuh"

namespace dt {

constexpr int kMaxMediumSteps = 8192;

struct MediumView {
  const float4* mu;
  int nx, ny, nz;
  float3 lo, scale;
  float step;
  int levels;             // hash texture levels (0: the dense grid)
  const GridLevel* lev;   // their descriptors, in the workspace's copy of the scene entry
};

// E: the scene entry as the kernel reads it (a kernel parameter or the
// table); Eg: the same entry in the workspace table, whose level array is
// indexed at run time.
__device__ __forceinline__ MediumView medium_view(const SceneEntry& E, const SceneEntry* Eg) {
  return MediumView{E.mu, E.gnx, E.gny, E.gnz, mk(E.glo_x, E.glo_y, E.glo_z),
                    mk(E.gscale_x, E.gscale_y, E.gscale_z), E.gstep, E.glevels, Eg->glev};
}

// Number of full steps of a segment of length t.
__device__ __forceinline__ int medium_full_steps(float t, float h) {
  const float m = floorf(t / h);
  if (!(m > 0.0f)) return 0;  // also a NaN length
  return m >= (float)kMaxMediumSteps ? kMaxMediumSteps : (int)m;
}

// A segment's steps: sample i < m at the middle of full step i, sample m at the
// middle of the last one, of length r.  The roundings are written out (for the
// reason at Lattice below): r is t - m h rounded once for a hash texture and after
// the product for a dense grid.
struct MediumSteps {
  float h, r, mid;
  int m;
  __device__ __forceinline__ MediumSteps(float t, const MediumView& g, bool hash)
      : h(g.step), m(medium_full_steps(t, g.step)) {
    const float mh = __fmul_rn((float)m, h), rest = __fsub_rn(t, mh);
    r = hash ? __fmaf_rn(-(float)m, h, t) : rest;
    mid = __fmaf_rn(0.5f, rest, mh);
  }
  __device__ __forceinline__ float weight(int i) const { return i < m ? h : r; }
  __device__ __forceinline__ float full_place(int i) const { return __fmul_rn((float)i + 0.5f, h); }
  __device__ __forceinline__ float place(int i) const { return i < m ? full_place(i) : mid; }
};

// ---------------------------------------------------------------------------
// lattices
// ---------------------------------------------------------------------------
// Instant-NGP's spatial hash of a lattice point (Mueller et al. 2022, Eq. 4
// with d = 3): XOR of the coordinates times 1, 2654435761 and 805459861 in
// 32-bit arithmetic; the level keeps its low bits (tables are powers of two).
constexpr uint32_t kHashPrimeY = 2654435761u, kHashPrimeZ = 805459861u;

// (ordinary loads: the table is written by an earlier kernel of the chain)
__device__ __forceinline__ GridLevel load_level(const GridLevel* p) {
  GridLevel L;
  const int4 a = *reinterpret_cast<const int4*>(p);
  const int4 b = *(reinterpret_cast<const int4*>(p) + 1);
  L.n = a.x;
  L.mask = (uint32_t)a.y;
  L.off = (uint32_t)a.z;
  L.sx = __int_as_float(a.w);
  L.sy = __int_as_float(b.x);
  L.sz = __int_as_float(b.y);
  L.pad[0] = L.pad[1] = 0;
  return L;
}

// One lattice (the dense grid, or a level of the hash texture) along one
// segment.  The sample at s is at the lattice position u = ((o + s d) - lo)
// scale, rounded after each of the three operations and written out below, so
// that every pass puts it into the same cell.  The gradient of a table of
// unrelated entries jumps at the cells' faces, and dJ/dIoR is a sum that cancels
// to a thousandth of its terms: u0 + s du, one fused multiply-add, puts a few
// samples per million into the neighbouring cell, neither nearer to nor farther
// from exact positions, and moved that gradient by 1e-4.  (An add and a product
// more per axis and sample cost 2 %: the adjoint of 8 views of 360x360 with an
// 8-level hash texture 8.8 -> 9.0 ms, of 16 views of 384x384 with a 64^3 grid 2.20
// -> 2.31.)
struct Lattice {
  float3 scale, lo, o, d;
  int nx, ny, nz;
  uint32_t off, mask;  // first entry; hashed level: entries - 1 (0: dense index (k ny + j) nx + i)
};

template <bool kHash>
__device__ __forceinline__ Lattice lattice_of(const MediumView& g, int l, float3 o, float3 d) {
  Lattice T;
  if (kHash && g.levels) {
    const GridLevel L = load_level(g.lev + l);
    T.scale = mk(L.sx, L.sy, L.sz);
    T.nx = T.ny = T.nz = L.n;
    T.off = L.off;
    T.mask = L.mask;
  } else {
    T.scale = g.scale;
    T.nx = g.nx;
    T.ny = g.ny;
    T.nz = g.nz;
    T.off = T.mask = 0u;
  }
  T.lo = g.lo;
  T.o = o;
  T.d = d;
  return T;
}

// Whether the segment stays inside the lattice's box (an object's box usually
// holds it whole): its samples then need no clamping.  The margin, 1/64 of a
// cell or, where that is more, a millionth of the lattice and of the ends'
// coordinates, is above the rounding of a position (6e-8 of the coordinate, and
// twice that of the lattice).
__device__ __forceinline__ bool lattice_inside(const Lattice& T, float t) {
  auto in = [&](float o, float d, float lo, float scale, int n) {
    const float x1 = fmaf(t, d, o), u0 = (o - lo) * scale, u1 = (x1 - lo) * scale;
    const float e = fmaxf(0.015625f, 1e-6f * fmaf(fabsf(o) + fabsf(x1), scale, (float)n));
    return fminf(u0, u1) >= e && fmaxf(u0, u1) <= (float)(n - 1) - e;
  };
  return in(T.o.x, T.d.x, T.lo.x, T.scale.x, T.nx) && in(T.o.y, T.d.y, T.lo.y, T.scale.y, T.ny) &&
         in(T.o.z, T.d.z, T.lo.z, T.scale.z, T.nz);
}

// The cell of a sample: per axis u clamped to [0, n - 1], cell index
// min(floor(u), n - 2) and fraction u - index; `free` = the axis was not
// clamped (a clamped coordinate is constant, so it has no derivative).
// kInside: known to need no clamping.
struct LatticeCell {
  int i, j, k;
  float fx, fy, fz;
  bool free_x, free_y, free_z;
};

template <bool kInside>
__device__ __forceinline__ float lattice_axis(float s, float o, float d, float lo, float scale, int n, int& i, bool& free) {
  float u = __fmul_rn(__fsub_rn(__fmaf_rn(d, s, o), lo), scale);
  if (kInside) {
    const float f = floorf(u);
    i = (int)f;
    free = true;
    return u - f;
  }
  const float top = (float)(n - 1);
  free = u >= 0.0f && u <= top;
  u = fminf(fmaxf(u, 0.0f), top);
  i = min((int)u, n - 2);
  return u - (float)i;
}

template <bool kInside>
__device__ __forceinline__ LatticeCell lattice_cell(const Lattice& T, float s) {
  LatticeCell c;
  c.fx = lattice_axis<kInside>(s, T.o.x, T.d.x, T.lo.x, T.scale.x, T.nx, c.i, c.free_x);
  c.fy = lattice_axis<kInside>(s, T.o.y, T.d.y, T.lo.y, T.scale.y, T.ny, c.j, c.free_y);
  c.fz = lattice_axis<kInside>(s, T.o.z, T.d.z, T.lo.z, T.scale.z, T.nz, c.k, c.free_z);
  return c;
}

// The entries of the lattice points (x0 or x1, y0 or y1, z0 or z1), entry q
// taking x1 for bit 0 of q, y1 for bit 1, z1 for bit 2; the per-axis terms are
// formed once, so an entry is a three-way XOR, a mask and an add, or two adds.
__device__ __forceinline__ void lattice_entries(const Lattice& T, uint32_t x0, uint32_t x1, uint32_t y0, uint32_t y1,
                                                uint32_t z0, uint32_t z1, uint32_t (&e)[8]) {
  if (T.mask) {
    y0 *= kHashPrimeY; y1 *= kHashPrimeY;
    z0 *= kHashPrimeZ; z1 *= kHashPrimeZ;
    const uint32_t a = y0 ^ z0, b = y1 ^ z0, c = y0 ^ z1, d = y1 ^ z1;
    e[0] = T.off + ((x0 ^ a) & T.mask); e[1] = T.off + ((x1 ^ a) & T.mask);
    e[2] = T.off + ((x0 ^ b) & T.mask); e[3] = T.off + ((x1 ^ b) & T.mask);
    e[4] = T.off + ((x0 ^ c) & T.mask); e[5] = T.off + ((x1 ^ c) & T.mask);
    e[6] = T.off + ((x0 ^ d) & T.mask); e[7] = T.off + ((x1 ^ d) & T.mask);
  } else {
    const uint32_t nx = (uint32_t)T.nx, ny = (uint32_t)T.ny;
    const uint32_t a = T.off + (z0 * ny + y0) * nx, b = T.off + (z0 * ny + y1) * nx;
    const uint32_t c = T.off + (z1 * ny + y0) * nx, d = T.off + (z1 * ny + y1) * nx;
    e[0] = a + x0; e[1] = a + x1; e[2] = b + x0; e[3] = b + x1;
    e[4] = c + x0; e[5] = c + x1; e[6] = d + x0; e[7] = d + x1;
  }
}

// The eight corner values of a cell (xyz of the float4 entries).
struct CellNodes {
  float3 c000, c100, c010, c110, c001, c101, c011, c111;
};

__device__ __forceinline__ CellNodes cell_nodes(const float4* __restrict__ mu, const Lattice& T, const LatticeCell& c) {
  const uint32_t i = (uint32_t)c.i, j = (uint32_t)c.j, k = (uint32_t)c.k;
  uint32_t e[8];
  lattice_entries(T, i, i + 1u, j, j + 1u, k, k + 1u, e);
  CellNodes q;
  q.c000 = xyz(__ldg(mu + e[0]));
  q.c100 = xyz(__ldg(mu + e[1]));
  q.c010 = xyz(__ldg(mu + e[2]));
  q.c110 = xyz(__ldg(mu + e[3]));
  q.c001 = xyz(__ldg(mu + e[4]));
  q.c101 = xyz(__ldg(mu + e[5]));
  q.c011 = xyz(__ldg(mu + e[6]));
  q.c111 = xyz(__ldg(mu + e[7]));
  return q;
}

// G and its gradient (dG_c/dx_a for the three channels c: columns gx, gy, gz,
// zero along clamped axes), sharing the interpolation's intermediate values:
// the differences along x feed both the x interpolations and dG/dx, the
// differences of the x-interpolated values along y feed the y interpolations
// and dG/dy, and the difference of the two y-interpolated values along z gives
// G and dG/dz.
__device__ __forceinline__ float3 trilinear_value_grad(const CellNodes& q, const LatticeCell& c, float3 scale,
                                                       float3& gx, float3& gy, float3& gz) {
  const float3 a00 = q.c100 - q.c000, a10 = q.c110 - q.c010, a01 = q.c101 - q.c001, a11 = q.c111 - q.c011;
  const float3 x00 = q.c000 + a00 * c.fx, x10 = q.c010 + a10 * c.fx;
  const float3 x01 = q.c001 + a01 * c.fx, x11 = q.c011 + a11 * c.fx;
  const float3 b0 = x10 - x00, b1 = x11 - x01;
  const float3 y0 = x00 + b0 * c.fy, y1 = x01 + b1 * c.fy;
  const float3 e = y1 - y0;
  const float3 ax0 = a00 + (a10 - a00) * c.fy, ax1 = a01 + (a11 - a01) * c.fy;
  gx = (ax0 + (ax1 - ax0) * c.fz) * (c.free_x ? scale.x : 0.0f);
  gy = (b0 + (b1 - b0) * c.fz) * (c.free_y ? scale.y : 0.0f);
  gz = e * (c.free_z ? scale.z : 0.0f);
  return y0 + e * c.fz;
}

// ---------------------------------------------------------------------------
// optical depth
// ---------------------------------------------------------------------------
__device__ __forceinline__ float3 fma3(float3 a, float b, float3 c) {
  return mk(__fmaf_rn(a.x, b, c.x), __fmaf_rn(a.y, b, c.y), __fmaf_rn(a.z, b, c.z));
}
__device__ __forceinline__ float3 lerp3(float3 a, float3 b, float f) { return fma3(b - a, f, a); }

// G at a cell's position.
__device__ __forceinline__ float3 trilinear(const CellNodes& q, const LatticeCell& c) {
  const float3 x00 = lerp3(q.c000, q.c100, c.fx), x10 = lerp3(q.c010, q.c110, c.fx);
  const float3 x01 = lerp3(q.c001, q.c101, c.fx), x11 = lerp3(q.c011, q.c111, c.fx);
  return lerp3(lerp3(x00, x10, c.fy), lerp3(x01, x11, c.fy), c.fz);
}

// Optical depth over o + s d, s in [0, t]: the sum over the levels (of the hash
// texture; the dense grid is one) and their samples, in this order, of weight
// times G (kHash: the scene may hold a hash texture; without it that code is not
// compiled).
template <bool kHash>
__device__ __forceinline__ float3 medium_depth(const MediumView& g, float3 o, float3 d, float t) {
  const int levels = kHash && g.levels ? g.levels : 1;
  const MediumSteps st(t, g, kHash && g.levels);
  float3 sum = mk(0.f, 0.f, 0.f);
  for (int l = 0; l < levels; ++l) {
    const Lattice T = lattice_of<kHash>(g, l, o, d);
    for (int i = 0; i <= st.m; ++i) {
      const LatticeCell c = lattice_cell<false>(T, st.place(i));
      sum = fma3(trilinear(cell_nodes(g.mu, T, c), c), st.weight(i), sum);
    }
  }
  return sum;
}

// The steps of a warp's segments, kLanes lanes each, in groups of kLanes samples:
// body(i0, full) with i0 the group's first sample and `full` whether all of its
// samples are full steps of every segment of the warp (a segment of m full steps
// has the samples 0..m; m < 0: the lane has none, in either case).
template <int kLanes, class Body>
__device__ __forceinline__ void warp_steps(int m, const Body& body) {
  const int top = __reduce_max_sync(kFull, m), low = (int)__reduce_min_sync(kFull, (unsigned)m);
  int i0 = 0;
  for (; i0 + kLanes <= low; i0 += kLanes) body(i0, std::true_type());
  for (; i0 <= top; i0 += kLanes) body(i0, std::false_type());
}

// Columns <-> lanes: with x = 1, then 2, v[q] of lane p becomes v[p] of lane q.
__device__ __forceinline__ void swap_if(bool up, float& lo, float& hi, int x) {
  const float got = __shfl_xor_sync(kFull, up ? lo : hi, x);
  lo = up ? got : lo;
  hi = up ? hi : got;
}
__device__ __forceinline__ void swap_if(bool up, float3& lo, float3& hi, int x) {
  swap_if(up, lo.x, hi.x, x);
  swap_if(up, lo.y, hi.y, x);
  swap_if(up, lo.z, hi.z, x);
}
template <class T>
__device__ __forceinline__ void transpose4(T (&v)[4], int p) {
  swap_if(p & 1, v[0], v[1], 1);
  swap_if(p & 1, v[2], v[3], 1);
  swap_if(p & 2, v[0], v[2], 2);
  swap_if(p & 2, v[1], v[3], 2);
}

// medium_depth for a warp's segments, four lanes each (`on`: the lane has one;
// every lane of the warp calls): a lane has every fourth sample, the values of
// four samples change places so that lane c holds channel c of each, and it adds
// them in the samples' order: medium_depth bit for bit.  dJ/dIoR is so
// ill-conditioned near the critical angle that depths which differ in the last bit
// move it by up to 5e-5.  (The shading of 8 views of 360x360 with an 8-level hash
// texture takes 6.4 ms; 6.0 with each lane summing its own samples, 7.1 with every
// lane of a segment adding all three channels and no loop for full groups.)
constexpr int kDepthLanes = 4;
template <bool kInside>
__device__ __forceinline__ void depth_walk(const float4* __restrict__ mu, const Lattice& T, const MediumSteps& st, int m,
                                           float& sum) {
  const int p = threadIdx.x & (kDepthLanes - 1);
  warp_steps<kDepthLanes>(m, [&](int i0, auto full) {
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (i0 + p <= m) {
      const LatticeCell c = lattice_cell<kInside>(T, full ? st.full_place(i0 + p) : st.place(i0 + p));
      const float3 G = trilinear(cell_nodes(mu, T, c), c);
      v[0] = G.x;
      v[1] = G.y;
      v[2] = G.z;
    }
    transpose4(v, p);
#pragma unroll
    for (int q = 0; q < kDepthLanes; ++q)
      if (full || i0 + q <= m) sum = __fmaf_rn(v[q], full ? st.h : st.weight(i0 + q), sum);
  });
}
template <bool kHash>
__device__ __forceinline__ float3 medium_depth_warp(const MediumView& g, float3 o, float3 d, float t, bool on) {
  const int levels = !on ? 0 : kHash && g.levels ? g.levels : 1;
  const MediumSteps st(t, g, kHash && g.levels);
  const int most = kHash ? __reduce_max_sync(kFull, levels) : 1;
  float sum = 0.f;
  for (int l = 0; l < most; ++l) {
    const bool mine = l < levels;
    const Lattice T = lattice_of<kHash>(g, mine ? l : 0, o, d);
    // one copy of the loop for the warp, whichever its lanes need
    if (__all_sync(kFull, !mine || lattice_inside(T, t))) depth_walk<true>(g.mu, T, st, mine ? st.m : -1, sum);
    else depth_walk<false>(g.mu, T, st, mine ? st.m : -1, sum);
  }
  return mk(__shfl_sync(kFull, sum, 0, kDepthLanes), __shfl_sync(kFull, sum, 1, kDepthLanes),
            __shfl_sync(kFull, sum, 2, kDepthLanes));
}

// dG_c/dx_a over the three channels c: columns gx, gy, gz, zero along clamped axes.
__device__ __forceinline__ void trilinear_grad(const CellNodes& q, const LatticeCell& c, float3 scale, float3& gx,
                                               float3& gy, float3& gz) {
  const float ux = 1.0f - c.fx, uy = 1.0f - c.fy, uz = 1.0f - c.fz;
  gx = ((q.c100 - q.c000) * (uy * uz) + (q.c110 - q.c010) * (c.fy * uz) + (q.c101 - q.c001) * (uy * c.fz) +
        (q.c111 - q.c011) * (c.fy * c.fz)) * (c.free_x ? scale.x : 0.0f);
  gy = ((q.c010 - q.c000) * (ux * uz) + (q.c110 - q.c100) * (c.fx * uz) + (q.c011 - q.c001) * (ux * c.fz) +
        (q.c111 - q.c101) * (c.fx * c.fz)) * (c.free_y ? scale.y : 0.0f);
  gz = ((q.c001 - q.c000) * (ux * uy) + (q.c101 - q.c100) * (c.fx * uy) + (q.c011 - q.c010) * (ux * c.fy) +
        (q.c111 - q.c110) * (c.fx * c.fy)) * (c.free_z ? scale.z : 0.0f);
}

// dS/dt per channel (only the partial last step depends on t).
template <bool kHash>
__device__ __forceinline__ float3 medium_depth_dt(const MediumView& g, float3 o, float3 d, float t) {
  const MediumSteps st(t, g, kHash && g.levels);
  float3 sum = mk(0.f, 0.f, 0.f);
  const int levels = kHash && g.levels ? g.levels : 1;
  for (int l = 0; l < levels; ++l) {
    const Lattice T = lattice_of<kHash>(g, l, o, d);
    const LatticeCell c = lattice_cell<false>(T, st.mid);
    const CellNodes q = cell_nodes(g.mu, T, c);
    float3 gx, gy, gz;
    trilinear_grad(q, c, T.scale, gx, gy, gz);
    sum = sum + trilinear(q, c) + (gx * d.x + gy * d.y + gz * d.z) * (0.5f * st.r);
  }
  return sum;
}

// ---------------------------------------------------------------------------
// march tiles
// ---------------------------------------------------------------------------
// The segments of a level that march the medium are some of its segments, of
// lengths from nothing to the object's diameter: 32 neighbours marched by a
// warp as they come leave two thirds of its lanes idle.  A CTA therefore takes a
// tile of the level's positions, lists those that march in shared memory by
// falling number of steps (a counting sort), and its warps take units of
// listed segments of nearly equal length, the longest first: 32 segments on one
// level of the texture for the adjoint, whose walks run along a segment, or
// eight segments with four lanes each for the forward passes, whose samples are
// independent (neighbouring samples read the same cells, so the four lanes
// share their reads as well).
constexpr int kTileThreads = 256;
constexpr int kTileMax = 512;  // positions
constexpr int kTileKeys = 128;
constexpr int kPartSteps = 32;  // (16: the grid's adjoint 5 % slower, for the corners that two parts share)

struct MarchTile {
  uint32_t pos[kTileMax];
  int hist[kTileKeys];
  int n, levels, next;
  int parts;  // of the longest listed segment
};

// Key of a segment of m full steps: m itself below 64, then eight per octave.
__device__ __forceinline__ int march_key(int m) {
  if (m < 64) return m;
  const int e = 31 - __clz(m);  // >= 6; m <= 8192
  return min(kTileKeys - 1, 64 + 8 * (e - 6) + ((m >> (e - 3)) & 7));
}

// Positions per tile for a level of n: 512, or 256 where the level would not
// fill the CTAs four times over.
__device__ __forceinline__ uint32_t march_tile(uint32_t n, uint32_t ctas) {
  return n >= 4u * kTileMax * ctas ? (uint32_t)kTileMax : kTileMax / 2u;
}

// Lists the positions [first, first + size) with steps(i, levels) >= 0 (levels:
// the lattices the position marches) by falling key.  By the whole CTA; the
// list may be read on return.
template <class Steps>
__device__ __forceinline__ void march_list(MarchTile& T, uint32_t first, uint32_t size, const Steps& steps) {
  constexpr int kPer = kTileMax / kTileThreads;
  for (int i = threadIdx.x; i < kTileKeys; i += kTileThreads) T.hist[i] = 0;
  if (threadIdx.x == 0) T.levels = T.next = T.parts = 0;
  __syncthreads();
  int key[kPer], rank[kPer], most = 0, parts = 0;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    key[j] = -1;
    const uint32_t p = j * kTileThreads + threadIdx.x;
    if (p >= size) continue;
    int levels = 0;
    const int m = steps(first + p, levels);
    if (m < 0) continue;
    key[j] = march_key(m);
    rank[j] = atomicAdd(&T.hist[key[j]], 1);
    most = max(most, levels);
    parts = max(parts, m / kPartSteps + 1);
  }
  most = __reduce_max_sync(kFull, most);
  parts = __reduce_max_sync(kFull, parts);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&T.levels, most);
    atomicMax(&T.parts, parts);
  }
  __syncthreads();
  if (threadIdx.x < 32) {  // counts -> starts, from the longest down
    const int k0 = kTileKeys - 1 - 4 * (int)threadIdx.x;
    int c[4], sum = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      c[q] = T.hist[k0 - q];
      sum += c[q];
    }
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, x, o);
      if ((int)threadIdx.x >= o) x += y;
    }
    if (threadIdx.x == 31) T.n = x;
    x -= sum;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      T.hist[k0 - q] = x;
      x += c[q];
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kPer; ++j)
    if (key[j] >= 0) T.pos[T.hist[key[j]] + rank[j]] = first + j * kTileThreads + threadIdx.x;
  __syncthreads();
}

// The warp's next unit of the forward passes: a listed segment's index for each
// group of kLanes lanes (T.n and above: none); false when the list is done.
template <int kLanes>
__device__ __forceinline__ bool march_group(MarchTile& T, int& index) {
  int u = 0;
  if ((threadIdx.x & 31) == 0) u = atomicAdd(&T.next, 32 / kLanes);
  u = __shfl_sync(kFull, u, 0);
  index = u + (int)(threadIdx.x & 31) / kLanes;
  return u < T.n;
}
// The warp's next unit of the adjoint: a listed segment's index for each lane
// (T.n and above: none), a level and a part of the samples; false when the list
// is done.  With few levels a tile has about as many chunks of 32 segments as
// the CTA has warps, the longest many times the shortest, and the warps would
// wait for the longest: its walks are cut into parts of kPartSteps samples
// (each ends with its eight corners' atomics).
constexpr int kPartLevels = 2;  // levels up to which walks are cut
__device__ __forceinline__ bool march_unit(MarchTile& T, int& index, int& level, int& part) {
  int u = 0;
  if ((threadIdx.x & 31) == 0) u = atomicAdd(&T.next, 1);
  u = __shfl_sync(kFull, u, 0);
  const int levels = max(T.levels, 1), chunks = (T.n + 31) / 32;
  level = levels - 1 - u % levels;
  const int v = u / levels;
  part = 0;
  int chunk = v;
  if (levels <= kPartLevels && chunks > 0) {
    part = v / chunks;
    chunk = v % chunks;
    if (part >= T.parts) return false;
  }
  index = chunk * 32 + (int)(threadIdx.x & 31);
  return chunk < chunks;
}

// ---------------------------------------------------------------------------
// tape_mode 2: the medium's moments in the forward, its scatter in the backward
// ---------------------------------------------------------------------------
// Everything the backward needs of the optical depth S over o + s d, s in
// [0, t], at fixed t: S; dS/dt (the partial last step, as medium_depth_dt);
// and the motion of the samples with o and d, whose adjoint is linear in
// sbar = dJ/dS:
//   dJ/do = sum_c sbar_c Do[c],  Do[c] = sum_i w_i grad G_c(x_i),
//   dJ/dd = sum_c sbar_c Dd[c],  Dd[c] = sum_i w_i s_i grad G_c(x_i),
// so the forward, which reads the corner values of every sample anyway,
// keeps the two 3x3 sums and the backward needs no corner value at all.
// gx, gy, gz of trilinear_grad are the columns dG/dx_a over the channels.
//
// Four lanes have a segment of a hash texture, two one of a dense grid, each every
// fourth or second sample, and add the samples up in their order all the same (as
// the depth's, for the same reason): G and the gradient's columns of a group of
// samples change places, so that each lane has one or two of the four for all
// samples of the group and sums what belongs to them.  (A 64^3 grid, 16 views of
// 384x384: 1.66 ms, 1.87 with four lanes or with one, 1.53 with each of two lanes
// summing its own samples; an 8-level hash texture, 8 views of 360x360: 9.1 ms,
// 16.0 with one lane, 6.9 with each of four summing its own.)
template <bool kHash>
constexpr int kMomentLanes = kHash ? 4 : 2;
template <int kLanes>
struct MomentSums {  // column j of lane p is column (4 / kLanes) p + j: G, dG/dx, dG/dy, dG/dz
  float3 a[4 / kLanes];  // S for G, dS/do along the axis
  float3 b[4 / kLanes];  // dS/dd along the axis (of G: unused)
  float3 dt;             // of the lane that has the last sample
};

template <bool kInside, int kLanes>
__device__ __forceinline__ void moments_walk(MomentSums<kLanes>& M, const float4* __restrict__ mu, const Lattice& T,
                                             const MediumSteps& st, float3 d, int m) {
  constexpr int kCols = 4 / kLanes;
  const int p = threadIdx.x & (kLanes - 1);
  warp_steps<kLanes>(m, [&](int i0, auto full) {
    float3 v[4];
    v[0] = v[1] = v[2] = v[3] = mk(0.f, 0.f, 0.f);
    if (i0 + p <= m) {
      const LatticeCell c = lattice_cell<kInside>(T, full ? st.full_place(i0 + p) : st.place(i0 + p));
      v[0] = trilinear_value_grad(cell_nodes(mu, T, c), c, T.scale, v[1], v[2], v[3]);
      if (!full && i0 + p == m) M.dt = M.dt + v[0] + (v[1] * d.x + v[2] * d.y + v[3] * d.z) * (0.5f * st.r);
    }
    if (kLanes == 4) {
      transpose4(v, p);
    } else {  // v[2 q + j]: column 2 p + j of sample q
      swap_if(p, v[0], v[2], 1);
      swap_if(p, v[1], v[3], 1);
    }
#pragma unroll
    for (int q = 0; q < kLanes; ++q)
      if (full || i0 + q <= m) {
        const float w = full ? st.h : st.weight(i0 + q);
        const float ws = __fmul_rn(w, full ? st.full_place(i0 + q) : st.place(i0 + q));
#pragma unroll
        for (int j = 0; j < kCols; ++j) {
          M.a[j] = fma3(v[kCols * q + j], w, M.a[j]);
          M.b[j] = fma3(v[kCols * q + j], ws, M.b[j]);
        }
      }
  });
}

// The moments of a warp's segments (`on`: the lane has one; every lane of the warp
// calls).
template <bool kHash>
__device__ __forceinline__ MomentSums<kMomentLanes<kHash>> medium_moments(const MediumView& g, float3 o, float3 d, float t,
                                                                          bool on) {
  const int levels = !on ? 0 : kHash && g.levels ? g.levels : 1;
  const MediumSteps st(t, g, kHash && g.levels);
  const int most = kHash ? __reduce_max_sync(kFull, levels) : 1;
  MomentSums<kMomentLanes<kHash>> M;
#pragma unroll
  for (int j = 0; j < 4 / kMomentLanes<kHash>; ++j) M.a[j] = M.b[j] = mk(0.f, 0.f, 0.f);
  M.dt = mk(0.f, 0.f, 0.f);
  for (int l = 0; l < most; ++l) {
    const bool mine = l < levels;
    const Lattice T = lattice_of<kHash>(g, mine ? l : 0, o, d);
    if (__all_sync(kFull, !mine || lattice_inside(T, t))) moments_walk<true>(M, g.mu, T, st, d, mine ? st.m : -1);
    else moments_walk<false>(M, g.mu, T, st, d, mine ? st.m : -1);
  }
  return M;
}

// ---------------------------------------------------------------------------
// adjoint
// ---------------------------------------------------------------------------
// One 128-bit vector reduction per entry (w unused) where `on`: predicated, not
// branched around.
__device__ __forceinline__ void red4_if(bool on, float4* p, float3 v) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %0, 0; @q red.relaxed.gpu.global.add.v4.f32 [%1], {%2, %3, %4, %5}; }" ::"r"(
                   (uint32_t)on), "l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(0.f)
               : "memory");
}

// Adjoint of one lattice's share of the optical depth over the samples
// [i0, i1) of one segment at fixed t (sbar = dJ/dS per channel): dJ/dG into dmu
// (unless null) and, when `gather` is set (the forward kept no moments of this
// segment), the sums of dJ/du and s dJ/du (lattice units) added to ob and db,
// from sbar . G at the samples' corners.
//
// Consecutive samples share their cell, or step to a neighbouring one (at
// most one cell along each axis), which shares corners with it: the weight
// sums of shared corners are carried along, and only the corners left behind
// are added to their entries with an atomic (about 40 % fewer atomics than for
// whole cells; hashed corners that share an entry add).  The eight slots are
// the parities of the corners' lattice coordinates (bit a of a slot: the
// coordinate along axis a is odd), so a corner has the same slot in every cell
// that holds it and nothing moves on a step: a step's new corners take the
// slots of those it leaves.  Within a cell sbar . G is a polynomial in the odd
// coordinates' weights X, Y, Z, whose coefficients are formed once per cell: its
// gradient is then nine fused multiply-adds a sample.
//
// The lanes of a warp enter new cells at different samples, so a loop over
// samples would run the step to a new cell, three times a sample's
// instructions, at nearly every sample with a few lanes each.  Lanes therefore
// take steps together and then up to kCellSamples samples of their cell (8 views
// of 360x360 with an 8-level hash texture, 1 to 8 samples per cell: 9.9 -> 8.1
// ms; 2 samples: 8.6; 8: 8.1; all samples of the cell in a loop that is not
// unrolled: slower than a sample at a time).
constexpr int kCellSamples = 4;
template <bool kInside>
__device__ __forceinline__ void adjoint_walk(const float4* __restrict__ mu, float4* __restrict__ dmu, const Lattice& T,
                                             const MediumSteps& st, int i0, int i1, float3 sbar, bool gather, float3& ob,
                                             float3& db) {
  float acc[8];
  uint32_t e[8];
  float px = 0.f, py = 0.f, pz = 0.f, pxy = 0.f, pxz = 0.f, pyz = 0.f, pxyz = 0.f;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    acc[q] = 0.f;
    e[q] = 0u;
  }
  int pi = 0, pj = 0, pk = 0;
  for (int i = i0; i < i1;) {
    {
      const LatticeCell c = lattice_cell<kInside>(T, st.place(i));
      const int dx = c.i - pi, dy = c.j - pj, dz = c.k - pk;
      if ((dx | dy | dz) != 0 || i == i0) {
        // slots whose corner the cell before does not share
        unsigned fresh = 0xFFu;
        if (i > i0) {
          if (((dx + 1) | (dy + 1) | (dz + 1) | (1 - dx) | (1 - dy) | (1 - dz)) >= 0) {
            // the coordinate left behind along an axis: p for a step up, p + 1 for one down
            fresh = (dx ? (((pi + (dx < 0)) & 1) ? 0xAAu : 0x55u) : 0u) | (dy ? (((pj + (dy < 0)) & 1) ? 0xCCu : 0x33u) : 0u) |
                    (dz ? (((pk + (dz < 0)) & 1) ? 0xF0u : 0x0Fu) : 0u);
          }
          if (dmu) {
#pragma unroll
            for (int q = 0; q < 8; ++q) red4_if((fresh >> q) & 1u, dmu + e[q], sbar * acc[q]);
          }
        }
        lattice_entries(T, (uint32_t)((c.i + 1) & ~1), (uint32_t)(c.i | 1), (uint32_t)((c.j + 1) & ~1),
                        (uint32_t)(c.j | 1), (uint32_t)((c.k + 1) & ~1), (uint32_t)(c.k | 1), e);
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] = fresh & (1u << q) ? 0.f : acc[q];
        if (gather) {
          float v[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) v[q] = dot(sbar, xyz(__ldg(mu + e[q])));
          const float a0 = v[1] - v[0], a1 = v[3] - v[2], a2 = v[5] - v[4], a3 = v[7] - v[6];
          const float b0 = v[2] - v[0], b2 = v[6] - v[4];
          px = a0;
          py = b0;
          pz = v[4] - v[0];
          pxy = a1 - a0;
          pxz = a2 - a0;
          pyz = b2 - b0;
          pxyz = (a3 - a2) - (a1 - a0);
        }
        pi = c.i;
        pj = c.j;
        pk = c.k;
      }
    }
#pragma unroll
    for (int n = 0; n < kCellSamples; ++n) {
      if (i >= i1) break;
      const float w = st.weight(i), s = st.place(i);
      const LatticeCell c = lattice_cell<kInside>(T, s);
      if (n > 0 && ((c.i ^ pi) | (c.j ^ pj) | (c.k ^ pk)) != 0) break;
      // weights of the odd and the even coordinate along each axis
      const float X = c.i & 1 ? 1.0f - c.fx : c.fx, Y = c.j & 1 ? 1.0f - c.fy : c.fy, Z = c.k & 1 ? 1.0f - c.fz : c.fz;
      const float xe = 1.0f - X, ye = 1.0f - Y, wzo = w * Z, wze = w - wzo;
      const float w00 = xe * ye, w10 = X * ye, w01 = xe * Y, w11 = X * Y;
      acc[0] += w00 * wze;
      acc[1] += w10 * wze;
      acc[2] += w01 * wze;
      acc[3] += w11 * wze;
      acc[4] += w00 * wzo;
      acc[5] += w10 * wzo;
      acc[6] += w01 * wzo;
      acc[7] += w11 * wzo;
      if (gather) {
        const float gx = fmaf(Z, fmaf(pxyz, Y, pxz), fmaf(pxy, Y, px)) * w;
        const float gy = fmaf(Z, fmaf(pxyz, X, pyz), fmaf(pxy, X, py)) * w;
        const float gz = fmaf(Y, fmaf(pxyz, X, pyz), fmaf(pxz, X, pz)) * w;
        // (X grows with u where the lower coordinate is even)
        const float3 gp =
            mk(kInside || c.free_x ? (c.i & 1 ? -gx : gx) : 0.0f, kInside || c.free_y ? (c.j & 1 ? -gy : gy) : 0.0f,
               kInside || c.free_z ? (c.k & 1 ? -gz : gz) : 0.0f);
        ob = ob + gp;
        db = db + gp * s;
      }
      ++i;
    }
  }
  if (dmu && i1 > i0) {
#pragma unroll
    for (int q = 0; q < 8; ++q) red4_if(true, dmu + e[q], sbar * acc[q]);
  }
}

// adjoint_walk over part `part` of a segment's samples (kPartSteps of them, or
// all with `whole`) on level l of the hash texture, or on the dense grid (l =
// 0): adds dJ/do and dJ/dd.  Every lane of the warp calls (`on`: the lane has a
// segment on level l).
template <bool kHash>
__device__ __forceinline__ void medium_level_adjoint(const MediumView& g, float4* dmu, int l, int part, bool whole, bool on,
                                                     float3 o, float3 d, float t, float3 sbar, bool gather, float3& ob,
                                                     float3& db) {
  const MediumSteps st(t, g, kHash && g.levels);
  const int i0 = whole ? 0 : part * kPartSteps;
  const int i1 = !on ? i0 : whole ? st.m + 1 : min(i0 + kPartSteps, st.m + 1);
  const Lattice T = lattice_of<kHash>(g, l, o, d);
  float3 uo = mk(0.f, 0.f, 0.f), ud = uo;
  // one copy of the walk for the warp, whichever its lanes need
  if (__all_sync(kFull, i0 >= i1 || lattice_inside(T, t))) adjoint_walk<true>(g.mu, dmu, T, st, i0, i1, sbar, gather, uo, ud);
  else adjoint_walk<false>(g.mu, dmu, T, st, i0, i1, sbar, gather, uo, ud);
  ob = ob + mul(uo, T.scale);
  db = db + mul(ud, T.scale);
}

}  // namespace dt
