// The matrix-free FP32 Laplacian (stencil7.cuh) on units of consecutive floats.
//
// A block of k columns on a grid is one array of n k floats, its x lines n_x k floats long.  A
// unit is V of them (16, 8 or 4 bytes) whatever cells and columns they belong to, and a warp's
// lanes take consecutive units: every load and store is one contiguous piece, where one cell or
// a run of cells per thread reads k = 3 columns at a 12- or 48-byte stride (three times the cache
// wavefronts).  The neighbours along y and z are a line and a plane away, those along x k floats.
//
// Units: with k = 4 kp columns (kp a power of two) the V = 4 floats lie in one cell (KC = 0
// below); with k = KC in {1, 2, 3} they may span cells, V the widest of 4, 2, 1 that divides a
// line (every line then starts on a unit).
#pragma once

#include <algorithm>

#include "common.cuh"
#include "stencil7.cuh"

namespace rb {

// Division of n < 2^31 by a fixed 2 <= d < 2^31: with l = ceil(log2 d), m = ceil(2^(31 + l) / d)
// fits in 32 bits and floor(n / d) = floor(m n / 2^(31 + l)) (Granlund and Montgomery, as FastDiv,
// whose 32-bit dividends cost three instructions more)
struct FastDiv31 {
  uint32_t m = 0;
  int s = 0;
  __host__ void init(uint32_t d) {
    int l = 1;
    while (((uint64_t)1 << l) < d) ++l;
    m = (uint32_t)((((uint64_t)1 << (31 + l)) + d - 1) / d);
    s = l - 1;
  }
  __device__ __forceinline__ uint32_t div(uint32_t n) const { return __umulhi(m, n) >> s; }
};

struct Unit7 {
  int n[3], per[3];
  const float* w[3];
  const float* ic[3];
  float scale = 1.0f;
  int k = 1;
  uint32_t line = 0, plane = 0;  // floats per x line and per z plane
  FastDiv31 dline, dplane, dk;   // dk: by k
  __host__ void init(const Stencil7<float>& st, int columns) {
    for (int d = 0; d < 3; ++d) n[d] = st.n[d], per[d] = st.per[d], w[d] = st.w[d], ic[d] = st.ic[d];
    scale = st.scale;
    k = columns;
    line = (uint32_t)n[0] * (uint32_t)k;
    plane = line * (uint32_t)n[1];
    dline.init(line);
    dplane.init(plane);
    dk.init((uint32_t)std::max(k, 2));
  }
};

// The unit width for k columns of this grid; 0: the columns do not form units
inline int unit7_width(const int n[3], int k) {
  if ((int64_t)n[0] * n[1] * n[2] * k >= ((int64_t)1 << 31) || n[0] < 2) return 0;
  if (k % 4 == 0) return (k & (k - 1)) == 0 ? 4 : 0;
  if (k > 3) return 0;
  const int64_t line = (int64_t)n[0] * k;
  return line % 4 == 0 ? 4 : (line % 2 == 0 ? 2 : 1);
}

// What a unit needs of an axis position: the width and the two inverse distances, and (y, z, and x
// when a unit lies in one cell) the offsets of the two neighbours, 0 at a wall (whose inverse
// distance is 0: the unit's own values are read).  Kept in shared memory for the launch: one
// 16-byte and one 8-byte load per axis and no comparisons.  x cells, then y, then z.
constexpr int kUnitTab = 768;
struct UnitTab {
  float4 c[kUnitTab];
  int2 o[kUnitTab];
};
inline bool unit7_table_fits(const int n[3]) { return (int64_t)n[0] + n[1] + n[2] <= kUnitTab; }

__device__ __forceinline__ void unit7_table(const Unit7& m, UnitTab& tab) {
  int at = 0;
  const int str[3] = {m.k, (int)m.line, (int)m.plane};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int n = m.n[d];
    const int wrap = m.per[d] ? (n - 1) * str[d] : 0;
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
      tab.c[at + t] = make_float4(__ldg(m.w[d] + t), __ldg(m.ic[d] + t), __ldg(m.ic[d] + t + 1), 0.0f);
      tab.o[at + t] = make_int2(t > 0 ? -str[d] : wrap, t + 1 < n ? str[d] : -wrap);
    }
    at += n;
  }
}

// Where a unit lies: its first float, the line and plane, the float's place in the line
struct UnitPos {
  uint32_t F, f, iy, iz;
};
__device__ __forceinline__ UnitPos unit7_pos(const Unit7& m, uint32_t F) {
  UnitPos u;
  u.F = F;
  u.iz = m.dplane.div(F);
  const uint32_t rest = F - u.iz * m.plane;
  u.iy = m.dline.div(rest);
  u.f = rest - u.iy * m.line;
  return u;
}
template <int KC>
__device__ __forceinline__ uint32_t unit7_cell(const Unit7& m, uint32_t f) {
  if constexpr (KC == 0) return m.dk.div(f);
  else return f / KC;
}

// q = A p on the unit u, the centre values into x0.  Called by whole warps whose lanes hold
// consecutive units (`last`: the lane's right-hand neighbour holds another unit): the x neighbours
// come from the other lanes, except at the warp's and the line's ends.  Each axis' two terms are
// formed from differences, sum_f c_f (p_neighbour - p): the diagonal is never formed, and the
// factors fixed on a line (face areas and inverse distances along y and z) are products of table
// entries shared by the unit's floats.  p is read through L2 (other blocks of the launch write it
// between grid barriers).
template <int KC, int V>
__device__ __forceinline__ void unit7_apply(const Unit7& m, const UnitTab& tab, const float* p, const UnitPos& u,
                                            int last, Vec<float, V>& x0, Vec<float, V>& q) {
  constexpr bool kOne = KC == 0;
  constexpr int E = kOne ? 1 : V;
  const uint32_t iy = u.iy, iz = u.iz, f = u.f;
  const uint32_t i0 = unit7_cell<KC>(m, f);
  const int rem = (int)(f - i0 * (kOne ? (uint32_t)m.k : (uint32_t)KC));
  const int nx = m.n[0], ny = m.n[1], lane = threadIdx.x & 31;
  const int2 oy = tab.o[nx + iy], oz = tab.o[nx + ny + iz];
  auto at = [&](int off) { return ldv_cg<float, V>(p + (uint32_t)((int)u.F + off)); };
  x0 = at(0);
  const Vec<float, V> zm = at(oz.x), zp = at(oz.y), ym = at(oy.x), yp = at(oy.y);
  Vec<float, V> xl, xr;
  if constexpr (kOne) {
    const int kp = m.k / V;
#pragma unroll
    for (int e = 0; e < V; ++e) {
      xl.v[e] = __shfl_up_sync(0xffffffffu, x0.v[e], kp);
      xr.v[e] = __shfl_down_sync(0xffffffffu, x0.v[e], kp);
    }
    const int2 ox = tab.o[i0];
    if (lane < kp || ox.x >= 0) xl = at(ox.x);
    if (lane + kp > last || ox.y <= 0) xr = at(ox.y);
  } else if constexpr (V == 4) {  // the units next to this one hold them
    Vec<float, V> a, b;
#pragma unroll
    for (int e = 0; e < KC; ++e) {
      a.v[V - 1 - e] = __shfl_up_sync(0xffffffffu, x0.v[V - 1 - e], 1);
      b.v[e] = __shfl_down_sync(0xffffffffu, x0.v[e], 1);
    }
    const int wrap = m.per[0] ? (int)m.line - V : 0;
    if (lane == 0 || f == 0) a = at(f > 0 ? -V : wrap);
    if (lane == last || f + V == m.line) b = at(f + V < m.line ? V : -wrap);
#pragma unroll
    for (int e = 0; e < V; ++e) {
      xl.v[e] = e < KC ? a.v[(V + e - KC) & 3] : x0.v[(e - KC) & 3];
      xr.v[e] = e + KC < V ? x0.v[(e + KC) & 3] : b.v[(e + KC) & 3];
    }
  } else {
    // the float e - KC (e + KC) of this unit lies in the unit -dl (dr) lanes away
#pragma unroll
    for (int e = 0; e < V; ++e) {
      constexpr int B = 4 * V;  // keeps the divisions below non-negative
      const int dl = (B - 1 - (e - KC + B - V)) / V, el = (e - KC + B) % V;
      const int dr = (e + KC) / V, er = (e + KC) % V;
      xl.v[e] = dl == 0 ? x0.v[el] : __shfl_up_sync(0xffffffffu, x0.v[el], dl);
      xr.v[e] = dr == 0 ? x0.v[er] : __shfl_down_sync(0xffffffffu, x0.v[er], dr);
      if (dl > 0 || dr > 0) {
        const int2 ox = tab.o[i0 + (uint32_t)(rem + e) / (KC ? KC : 1)];
        if (dl > 0 && (lane < dl || ox.x >= 0)) xl.v[e] = __ldcg(p + (uint32_t)((int)u.F + e + ox.x));
        if (dr > 0 && (lane + dr > last || ox.y <= 0)) xr.v[e] = __ldcg(p + (uint32_t)((int)u.F + e + ox.y));
      }
    }
  }
  const float4 ty = tab.c[nx + iy], tz = tab.c[nx + ny + iz];
  const float wy = m.scale * ty.x, wz = m.scale * tz.x;
  const float ax = wy * tz.x;
  const float bym = wz * ty.y, byp = wz * ty.z, bzm = wy * tz.y, bzp = wy * tz.z;
  float icm[E], icp[E], wx[E];
  if constexpr (kOne || KC == 1 || (KC == 2 && V == 2)) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const float4 tx = tab.c[KC == 1 ? i0 + e : i0];
      wx[e] = tx.x, icm[e] = tx.y, icp[e] = tx.z;
    }
  } else {  // two cells at most
    const float4 t0 = tab.c[i0], t1 = tab.c[rem + V > KC ? i0 + 1 : i0];
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const bool second = rem + e >= KC;
      wx[e] = second ? t1.x : t0.x, icm[e] = second ? t1.y : t0.y, icp[e] = second ? t1.z : t0.z;
    }
  }
#pragma unroll
  for (int e = 0; e < V; ++e) {
    const int g = e < E ? e : 0;
    const float c0 = x0.v[e];
    const float w = fmaf(icp[g], xr.v[e] - c0, icm[g] * (xl.v[e] - c0));
    float v = bym * (ym.v[e] - c0);
    v = fmaf(byp, yp.v[e] - c0, v);
    v = fmaf(bzm, zm.v[e] - c0, v);
    v = fmaf(bzp, zp.v[e] - c0, v);
    q.v[e] = fmaf(ax, w, wx[g] * v);
  }
}

// Per-cell values d (ld = 1) of a unit's floats: cell0 its first cell, rem its first column
template <int KC, int V>
__device__ __forceinline__ Vec<float, V> unit7_cells(const float* __restrict__ d, uint32_t cell0, int rem) {
  Vec<float, V> r;
  if constexpr (KC == 0 || (KC == 2 && V == 2)) {
    const float v = __ldg(d + cell0);
#pragma unroll
    for (int e = 0; e < V; ++e) r.v[e] = v;
  } else if constexpr (KC == 1) {
    r = ldv<float, V>(d + cell0);
  } else if constexpr (KC == 2) {
    const Vec<float, 2> v = ldv<float, 2>(d + cell0);
    r.v[0] = r.v[1] = v.v[0], r.v[2] = r.v[3] = v.v[1];
  } else {
    const float a = __ldg(d + cell0), b = rem + V > 3 ? __ldg(d + cell0 + 1) : a;
#pragma unroll
    for (int e = 0; e < V; ++e) r.v[e] = rem + e < 3 ? a : b;
  }
  return r;
}

}  // namespace rb
