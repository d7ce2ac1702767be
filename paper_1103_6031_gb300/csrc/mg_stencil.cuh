// Finite-difference Laplacian of Table 1 (Hahn & Abel 2011, Sec. 3.2): the 3D
// operator is the sum over x, y, z of the 1D second difference of order n,
// i.e. 7, 13 or 19 points.  Weights below are the 1D weights on offsets
// 0, +-1, +-2, +-3 (units 1/h^2).
#pragma once

#include "mg_fixed.cuh"
#include "mg_internal.h"

namespace mgk {

template <int ORDER>
struct Lap;
template <>
struct Lap<2> {
  static constexpr double w0 = -2.0, w1 = 1.0, w2 = 0.0, w3 = 0.0;
};
template <>
struct Lap<4> {
  static constexpr double w0 = -30.0 / 12.0, w1 = 16.0 / 12.0, w2 = -1.0 / 12.0, w3 = 0.0;
};
template <>
struct Lap<6> {
  static constexpr double w0 = -490.0 / 180.0, w1 = 270.0 / 180.0, w2 = -27.0 / 180.0,
                          w3 = 2.0 / 180.0;
};

// The 6 neighbours at each distance 1 .. ORDER / 2 of element p: nb[6 (d - 1)] ..: -z, +z,
// -y, +y, -x, +x.
template <int ORDER, typename T>
__device__ __forceinline__ void load_neighbours(const T* u, long long p, int sy,
                                                int sx, T (&nb)[3 * ORDER]) {
  const T* c = u + p;
#pragma unroll
  for (int d = 1; d <= ORDER / 2; ++d) {
    T* o = nb + 6 * (d - 1);
    o[0] = c[-d];
    o[1] = c[d];
    o[2] = *(c - d * sy);
    o[3] = c[d * sy];
    o[4] = *(c - d * sx);
    o[5] = c[d * sx];
  }
}

template <typename T>
struct Vec2;
template <>
struct Vec2<double> {
  typedef double2 type;
};
template <>
struct Vec2<float> {
  typedef float2 type;
};

// The neighbours of the z-pair at p (an even cell of its row) and the pair itself, every row
// by 2-element loads.
template <int ORDER, typename T>
__device__ __forceinline__ void load_pair_neighbours(const T* u, long long p, int sy,
                                                     int sx, T (&n0)[3 * ORDER],
                                                     T (&n1)[3 * ORDER], T& c0, T& c1) {
  typedef typename Vec2<T>::type V2;
  constexpr int R = ORDER / 2, RZ = (R + 1) / 2 * 2;
  auto ld2 = [](const T* q) { return *reinterpret_cast<const V2*>(q); };
  const T* c = u + p;
  T z[2 * RZ + 2];
#pragma unroll
  for (int a = 0; a <= RZ; ++a) {
    const V2 v = ld2(c + 2 * a - RZ);
    z[2 * a] = v.x;
    z[2 * a + 1] = v.y;
  }
  c0 = z[RZ];
  c1 = z[RZ + 1];
#pragma unroll
  for (int d = 1; d <= R; ++d) {
    const V2 ym = ld2(c - d * sy), yp = ld2(c + d * sy);
    const V2 xm = ld2(c - d * sx), xp = ld2(c + d * sx);
    const T a[6] = {z[RZ - d], z[RZ + d], ym.x, yp.x, xm.x, xp.x};
    const T b[6] = {z[RZ + 1 - d], z[RZ + 1 + d], ym.y, yp.y, xm.y, xp.y};
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      n0[6 * (d - 1) + q] = a[q];
      n1[6 * (d - 1) + q] = b[q];
    }
  }
}

template <typename T>
__device__ __forceinline__ T sum6(const T* o) {
  return (o[0] + o[1]) + (o[2] + o[3]) + (o[4] + o[5]);
}

// The largest exponent of the neighbours, low bits set (the key of mg_fixed.cuh).
template <int ORDER>
__device__ __forceinline__ unsigned neighbour_key(const double (&nb)[3 * ORDER]) {
  unsigned m = 0;
#pragma unroll
  for (int q = 0; q < 3 * ORDER; ++q) m = max(m, fx_key(nb[q]));
  return m | 0x1fffffu;
}

// acc - (sum_off w nb) / w_centre: the value that solves the row of L u = f, with
// acc = (h^2 / w_centre) f.  float64 sums the neighbours on the integer pipe
// (mg_fixed.cuh): 3 FP64 instructions per update instead of 19.  Measured on GB300, order 6,
// warm L2, 128^3 nest: 41.7 -> 17.6 us per half-sweep, 16.0 with CVT (64^3: 6.9 -> 3.9,
// 32^3: 3.0 -> 2.2); order 4: 29.2 -> 12.8; order 2: 16.5 -> 8.7.  Plain instead of read-only
// loads (mg_launch.cuh) have added 2 to 4% since.
template <int ORDER, typename T, bool CVT = false>
__device__ __forceinline__ T relax(const T (&nb)[3 * ORDER], T acc) {
  constexpr double wc = 3.0 * Lap<ORDER>::w0;
  if constexpr (sizeof(T) == 8) {
    const unsigned key = neighbour_key<ORDER>(nb);
    if (fx_in_range(key))
      return fma(fx_scale(-FxUnit<ORDER>::v / wc, key), (double)fx_neighbours<ORDER, CVT>(nb, key), acc);
  }
  acc = fma(T(-Lap<ORDER>::w1 / wc), sum6(nb), acc);
  if constexpr (ORDER >= 4) acc = fma(T(-Lap<ORDER>::w2 / wc), sum6(nb + 6), acc);
  if constexpr (ORDER >= 6) acc = fma(T(-Lap<ORDER>::w3 / wc), sum6(nb + 12), acc);
  return acc;
}

// acc + scale h^2 L u from a cell's neighbours and its own value c.  float64 on the integer
// pipe as in relax (2 FP64 instructions instead of 20; scale * FxUnit is loop-invariant)
// unless FX is false.
template <int ORDER, typename T, bool FX = true>
__device__ __forceinline__ T add_lap_of(const T (&nb)[3 * ORDER], T c, T scale, T acc) {
  if constexpr (sizeof(T) == 8 && FX) {
    const unsigned key = max(neighbour_key<ORDER>(nb), fx_key(c)) | 0x1fffffu;
    const double k = scale * FxUnit<ORDER>::v;
    if (fx_in_range(key) && fx_scalable(k, key)) {
      const long long t = fx_neighbours<ORDER>(nb, key) + fx_centre<ORDER>(fx_align(c, key));
      return fma(fx_scale(k, key), (double)t, acc);
    }
  }
  T lu = T(3.0 * Lap<ORDER>::w0) * c;
  lu = fma(T(Lap<ORDER>::w1), sum6(nb), lu);
  if constexpr (ORDER >= 4) lu = fma(T(Lap<ORDER>::w2), sum6(nb + 6), lu);
  if constexpr (ORDER >= 6) lu = fma(T(Lap<ORDER>::w3), sum6(nb + 12), lu);
  return fma(scale, lu, acc);
}

// The same at element p, c = u[p].
template <int ORDER, typename T, bool FX = true>
__device__ __forceinline__ T add_lap_h2(const T* u, long long p, int sy, int sx, T c,
                                        T scale, T acc) {
  T nb[3 * ORDER];
  load_neighbours<ORDER, T>(u, p, sy, sx, nb);
  return add_lap_of<ORDER, T, FX>(nb, c, scale, acc);
}

// On a periodic level, every ghost cell is the image of one interior cell (all
// sides are >= g).  Along an axis of n cells with element stride st, index a has
// an image at a + n when a < g and at a - n when a >= n - g (both when n < 2g);
// ImgAxis holds the element offsets of those images, 0 for none.
struct ImgAxis {
  long long lo, hi;
};

__device__ __forceinline__ ImgAxis img_axis(int a, int n, int g, long long st) {
  return ImgAxis{a < g ? (long long)n * st : 0, a >= n - g ? -(long long)n * st : 0};
}

// Writes v to the images of interior cell (i, j, k): every combination of own
// or image index per axis except own on every axis.  Straight-line predicated
// stores (the loops unroll; no local memory); the cell itself is written by the
// caller.  Rows away from the x and y faces (the same for a whole warp) have z images only:
// they take two stores instead of the 26 predicated ones, which every warp that reaches a z
// face would execute.
template <typename T>
__device__ __forceinline__ void write_images(const Grid& G, T* u, int i, int j,
                                             int k, T v) {
  const int g = G.g;
  const bool in_xy = i >= g && i < G.n0 - g && j >= g && j < G.n1 - g;
  if (in_xy && k >= g && k < G.n2 - g) return;
  const long long sy = G.Zp, sx = (long long)G.Y * G.Zp;
  const ImgAxis az = img_axis(k, G.n2, g, 1);
  T* p = u + gidx(G, i, j, k);
  if (in_xy) {
    if (az.lo) p[az.lo] = v;
    if (az.hi) p[az.hi] = v;
    return;
  }
  const ImgAxis ax = img_axis(i, G.n0, g, sx), ay = img_axis(j, G.n1, g, sy);
  const long long ox[3] = {0, ax.lo, ax.hi}, oy[3] = {0, ay.lo, ay.hi}, oz[3] = {0, az.lo, az.hi};
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
      for (int c = 0; c < 3; ++c)
        if ((a | b | c) && (a == 0 || ox[a]) && (b == 0 || oy[b]) && (c == 0 || oz[c]))
          p[ox[a] + oy[b] + oz[c]] = v;
}

// Images of the z-pair (k, k+1), k even and k + 1 < n2, with values (va, vb): the
// x/y images of the pair as one vector store each (x and y offsets are multiples
// of the row pitch, so the alignment of the pair is kept), the z images of each
// cell scalar, at the cell's own row and at every x/y image row.
template <typename T>
__device__ __forceinline__ void write_pair_images(const Grid& G, T* u, int i, int j,
                                                  int k, T va, T vb) {
  const int g = G.g;
  const bool in_xy = i >= g && i < G.n0 - g && j >= g && j < G.n1 - g;
  if (in_xy && k >= g && k + 1 < G.n2 - g) return;
  typedef typename Vec2<T>::type V2;
  const long long sy = G.Zp, sx = (long long)G.Y * G.Zp;
  const ImgAxis z0 = img_axis(k, G.n2, g, 1), z1 = img_axis(k + 1, G.n2, g, 1);
  T* p = u + gidx(G, i, j, k);
  if (in_xy) {
    if (z0.lo) p[z0.lo] = va;
    if (z0.hi) p[z0.hi] = va;
    if (z1.lo) p[1 + z1.lo] = vb;
    if (z1.hi) p[1 + z1.hi] = vb;
    return;
  }
  const ImgAxis ax = img_axis(i, G.n0, g, sx), ay = img_axis(j, G.n1, g, sy);
  const long long ox[3] = {0, ax.lo, ax.hi}, oy[3] = {0, ay.lo, ay.hi};
  V2 pv;
  pv.x = va;
  pv.y = vb;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      if ((a != 0 && !ox[a]) || (b != 0 && !oy[b])) continue;
      T* q = p + ox[a] + oy[b];
      if (a | b) *reinterpret_cast<V2*>(q) = pv;
      if (z0.lo) q[z0.lo] = va;
      if (z0.hi) q[z0.hi] = va;
      if (z1.lo) q[1 + z1.lo] = vb;
      if (z1.hi) q[1 + z1.hi] = vb;
    }
}

}  // namespace mgk
