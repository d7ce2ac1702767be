// Tiles of aligned integers in shared memory for the float64 stencils that need every
// cell (mg_fixed.cuh): a block of 256 threads loads 8 x 8 x 32 cells with the halo of the
// star-shaped stencil, aligns every value once to the block's largest exponent, and the
// cells' sums read shared memory.  A value is aligned 2.7 times on average (halos) instead
// of once for each of the 19 cells whose stencil it is in.
//
// What it is bounded by: the alignment and the sums, about 140 integer and shared-memory
// instructions per cell; 63 KB of shared memory at order 6 let three blocks share an SM,
// so that one block's loads overlap the others' sums.  A half-sweep, which needs only
// every second cell's sum, gains nothing from it (17.8 against 17.6 us at 128^3).
//
// Accuracy: a unit is 2^-58 to 2^-59 of the BLOCK's largest value (halo included), not of the
// cell's own neighbours'.  A tile is summed as integers only if every cell's star holds a value
// of at least 2^52 units (2^51 at order 2) or nothing but zeros (tile_key); the rounding of a
// difference, at most 30 units (12), then stays below 2^-47 of the largest value in the cell's own
// star, and is far smaller where that is the block's largest too.  Other tiles (a strong cell
// among weak ones, a steep tail) are left to FP64 arithmetic.
#pragma once

#include "mg_fixed.cuh"
#include "mg_internal.h"
#include "mg_stencil.cuh"

namespace mgk {

constexpr int kTileX = 8, kTileY = 8, kTileZ = 32;
constexpr int kTileThreads = 256;

template <int ORDER>
struct FxTile {
  static constexpr int R = ORDER / 2;
  static constexpr int RZ = (R + 1) / 2 * 2;  // z halo rounded up to pairs
  static constexpr int SY = kTileY + 2 * R, SZ = kTileZ + 2 * RZ;
  static constexpr int px = SY * SZ, py = SZ;  // element strides along x and y
  static constexpr int elems = (kTileX + 2 * R) * px;
  static constexpr int bytes = elems * 8;
  // element of tile cell (x, y, z)
  static __device__ __forceinline__ int at(int x, int y, int z) {
    return (x + R) * px + (y + R) * py + z + RZ;
  }
};

inline dim3 tile_grid(const Grid& G) {
  return dim3((G.n2 + kTileZ - 1) / kTileZ, (G.n1 + kTileY - 1) / kTileY,
              (G.n0 + kTileX - 1) / kTileX);
}

// Levels that the tile kernels take: below, their blocks are too few to hide a block's load
// phase.  Float64 V-cycle of a base and two nests, order 6, without tiles and with: 32^3 179
// and 207 us, 48^3 229 and 245, 64^3 295 and 287, 80^3 493 and 448, 96^3 670 and 600.  Orders 2
// and 4 and a single periodic level cross between 48^3 (111 thousand cells) and 64^3 too.
constexpr long long kTileMinCells = 1ll << 17;

inline bool tile_pays(const Grid& G) {
  return (long long)G.n0 * G.n1 * G.n2 >= kTileMinCells;
}

// Which cells of the tile a thread works on: the z-pair 2 zz, 2 zz + 1 of row y in the
// planes 4 xh .. 4 xh + 3 (lanes 0-15 and 16-31 of a warp: two neighbouring rows).
struct TilePos {
  int zz, y, xh;
};

__device__ __forceinline__ TilePos tile_pos() {
  const int t = threadIdx.x;
  return TilePos{t & 15, (t >> 4) & 7, t >> 7};
}

// A level as a kernel reads it: padded, with its ghosts filled, or a dense periodic array
// whose ghosts are the cells one period away (sides at least the halo, even rows).  at(i, j, k):
// address of cell (i, j, k), of a pair for even k.
struct PaddedSource {
  const double* cell0;
  int sx, sy;
  __device__ __forceinline__ PaddedSource(const Grid& G, const double* u)
      : cell0(u + gidx(G, 0, 0, 0)), sx(G.Y * G.Zp), sy(G.Zp) {}
  __device__ __forceinline__ const double* at(int i, int j, int k) const {
    return cell0 + ((long long)i * sx + j * sy + k);
  }
};
struct DensePeriodicSource {
  const double* cell0;
  int n0, n1, n2;
  __device__ __forceinline__ DensePeriodicSource(const Grid& G, const double* u)
      : cell0(u), n0(G.n0), n1(G.n1), n2(G.n2) {}
  static __device__ __forceinline__ int wrap(int a, int n) {
    return a < 0 ? a + n : (a >= n ? a - n : a);
  }
  __device__ __forceinline__ const double* at(int i, int j, int k) const {
    return cell0 + ((long long)wrap(i, n0) * n1 + wrap(j, n1)) * n2 + wrap(k, n2);
  }
};

__device__ __forceinline__ unsigned block_max(unsigned m) {
  __shared__ unsigned red[kTileThreads / 32];
  m = __reduce_max_sync(~0u, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kTileThreads / 32; ++w) m = max(m, red[w]);
  return m;
}

// Exponents a cell's star may lie below the block's largest: the bits that an aligned value has
// beyond a mantissa's 53.  Tiles of a smooth field pass, also where it is zero on a surface:
// its star reaches ORDER / 2 cells to either side, a tile 32.  At order 2, whose unweighted sums
// lose half as many units, one more: 6 rejects 0.2 to 0.9% of the tiles of a potential (none at
// orders 4 and 6), and on a small level one tile in FP64 arithmetic is what the launch waits for
// (solve to 1e-10 of 64^3 886 us with 6, 842 with 7).
template <int ORDER>
constexpr int kTileRange = ORDER == 2 ? 7 : 6;

// Whether the star of one of a thread's cells (tile_pos: a z-pair in 4 planes; a and b their keys or
// magnitudes) can be low: the least of the largest values of windows along x of which every star
// holds one.
template <int ORDER>
__device__ __forceinline__ unsigned least_window(const unsigned (&a)[4], const unsigned (&b)[4]) {
  constexpr int W = ORDER / 2 < 3 ? ORDER / 2 + 1 : 4, STEP = W < 4 ? 4 - W : 1;
  unsigned least = ~0u;
#pragma unroll
  for (int q = 0; q + W <= 4; q += STEP) {
    unsigned ma = 0, mb = 0;
#pragma unroll
    for (int n = q; n < q + W; ++n) {
      ma = max(ma, a[n]);
      mb = max(mb, b[n]);
    }
    least = min(least, min(ma, mb));
  }
  return least;
}

// Ends the filling of a tile of ex x ey x ez cells at (i0, j0, k0) of src: its key, or 0 (out of
// range: FP64 arithmetic) where the star of a cell holds only values more than kTileRange exponents
// below the block's largest, and not only zeros (a star that the alignment leaves nothing of is
// looked up in src).  low: a star of the thread's cells can be (least_window).  The same answer in
// every thread.  Few tiles of a potential have to look: 4.4% in the steps of 192 x 160 x 224 and
// 3.4% of two levels of 128^3, 0.02% of which then go to FP64.  What the question costs, without /
// with, order 6, 192 x 160 x 224: the first cycle's restriction 50.1 / 52.8 us, the norm 83.8 /
// 82.9 (with f loaded ahead); tau of 256^3 705 / 721 us.  Asked after the sums it costs the norm 2
// and tau 4% more; with every cell of the thread told apart beforehand, the restriction 56.0.
template <int ORDER, typename Src>
__device__ __forceinline__ unsigned tile_key(unsigned key, const long long* S, const Src& src,
                                             int i0, int j0, int k0, int ex, int ey, int ez,
                                             bool low) {
  typedef FxTile<ORDER> L;
  constexpr long long kWeak = 1ll << (58 - kTileRange<ORDER>);
  auto mag = [](long long v) { return v ^ (v >> 63); };
  if (__builtin_expect(!__syncthreads_or(low), 1)) return key;
  bool wide = false;
#pragma unroll 1
  for (int e = low ? 0 : 8; e < 8; ++e) {
    const TilePos t = tile_pos();
    const int x = 4 * t.xh + (e >> 1), y = t.y, z = 2 * t.zz + (e & 1);
    if (x >= ex || y >= ey || z >= ez) continue;
    const long long* c = S + L::at(x, y, z);
    long long m = mag(c[0]);
#pragma unroll 1
    for (int d = 1; d <= L::R; ++d)
      m |= mag(c[d]) | mag(c[-d]) | mag(c[d * L::py]) | mag(c[-d * L::py]) | mag(c[d * L::px]) |
           mag(c[-d * L::px]);
    if (m >= kWeak) continue;
    wide |= m != 0;
    if (m == 0)
#pragma unroll 1
      for (int d = -L::R; d <= L::R; ++d)
        wide |= *src.at(i0 + x + d, j0 + y, k0 + z) != 0.0 ||
                *src.at(i0 + x, j0 + y + d, k0 + z) != 0.0 ||
                *src.at(i0 + x, j0 + y, k0 + z + d) != 0.0;
  }
  return __syncthreads_or(wide) ? 0u : key;
}

// Loads the tile at cell (i0, j0, k0) of u with its star halo into S, aligned to the
// returned key (low bits set).  Values outside the stencils' reach (beyond the ghosts,
// row padding, edge and corner ghosts) count as 0.  If the returned key is out of range
// (fx_in_range; 0 for a tile of too wide a range), S is not to be used.
template <int ORDER>
__device__ __forceinline__ unsigned tile_load(const Grid& G, const double* u, int i0,
                                              int j0, int k0, long long* S) {
  typedef FxTile<ORDER> L;
  constexpr int R = L::R, RZ = L::RZ;
  const TilePos t = tile_pos();
  const int sy = G.Zp, sx = G.Y * G.Zp;
  const double* base = u + gidx(G, i0, j0, k0);
  const int ex = min(kTileX, G.n0 - i0), ey = min(kTileY, G.n1 - j0), ez = min(kTileZ, G.n2 - k0);
  const int z = 2 * t.zz;
  // a pair at z >= ez is out along z; the first R cells there are ghosts
  const bool in0 = z < ez, in1 = z + 1 < ez;
  auto pair = [&](int x, int y, bool a, bool b) {
    double2 v = make_double2(0.0, 0.0);
    if (a || b) {
      v = *reinterpret_cast<const double2*>(base + (x * sx + y * sy + z));
      if (!a) v.x = 0.0;
      if (!b) v.y = 0.0;
    }
    return v;
  };
  double2 c[4], vx[R], vy[R], vz = make_double2(0.0, 0.0);
  int xs[R], ys[R];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int x = 4 * t.xh + q;
    const bool row = x < ex && t.y < ey;
    // a row that is out along one axis, by at most R, is a halo row for its interior z
    const bool halo = (x < ex && t.y < ey + R) || (x < ex + R && t.y < ey);
    c[q] = pair(x, t.y, row ? z < ez + R : halo && in0, row ? z + 1 < ez + R : halo && in1);
  }
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int s = t.xh + 2 * q;  // 0 .. 2 R - 1: the halo's layers
    xs[q] = s < R ? s - R : kTileX + s - R;
    ys[q] = s < R ? s - R : kTileY + s - R;
    const bool ox = xs[q] < ex + R && t.y < ey;
    vx[q] = pair(xs[q], t.y, ox && in0, ox && in1);
    // y layers: the thread's row index runs along x
    const bool oy = ys[q] < ey + R && t.y < ex;
    vy[q] = pair(t.y, ys[q], oy && in0, oy && in1);
  }
  // z halo: RZ pairs per row, half of them on either side, 64 rows
  const int zr = (int)threadIdx.x / RZ, ze = (int)threadIdx.x % RZ;
  const int zx = zr >> 3, zy = zr & 7;
  const int zo = ze < RZ / 2 ? 2 * ze - RZ : kTileZ + 2 * (ze - RZ / 2);
  const bool zact = zr < 64;
  if (zact && zx < ex && zy < ey) {
    const bool a = zo >= -R && zo < ez + R, b = zo + 1 < ez + R;
    if (a || b) {
      vz = *reinterpret_cast<const double2*>(base + (zx * sx + zy * sy + zo));
      if (!a) vz.x = 0.0;
      if (!b) vz.y = 0.0;
    }
  }
  unsigned m = max(fx_key(vz.x), fx_key(vz.y));
#pragma unroll
  for (int q = 0; q < 4; ++q) m = max(m, max(fx_key(c[q].x), fx_key(c[q].y)));
#pragma unroll
  for (int q = 0; q < R; ++q)
    m = max(m, max(max(fx_key(vx[q].x), fx_key(vx[q].y)), max(fx_key(vy[q].x), fx_key(vy[q].y))));
  m = block_max(m) | 0x1fffffu;
  if (fx_in_range(m)) {
    auto put = [&](int x, int y, int zq, double2 v) {
      longlong2 a;
      a.x = fx_align(v.x, m);
      a.y = fx_align(v.y, m);
      *reinterpret_cast<longlong2*>(S + L::at(x, y, zq)) = a;
    };
#pragma unroll
    for (int q = 0; q < 4; ++q) put(4 * t.xh + q, t.y, z, c[q]);
#pragma unroll
    for (int q = 0; q < R; ++q) {
      put(xs[q], t.y, z, vx[q]);
      put(t.y, ys[q], z, vy[q]);
    }
    if (zact) put(zx, zy, zo, vz);
  }
  unsigned a[4], b[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    a[q] = fx_key(c[q].x);
    b[q] = fx_key(c[q].y);
  }
  const bool low =
      fx_in_range(m) && least_window<ORDER>(a, b) <= m - ((kTileRange<ORDER> + 1u) << 21);
  return tile_key<ORDER>(m, S, PaddedSource(G, u), i0, j0, k0, ex, ey, ez, low);
}

// T (mg_fixed.cuh: h^2 L u = T FxUnit 2^(e - kFxBias)) of the thread's 8 cells and their
// aligned values: do_cell(q, T of the pair, values of the pair) for plane 4 xh + q.
template <int ORDER, typename F>
__device__ __forceinline__ void tile_laplacians(const long long* S, F do_pair) {
  typedef FxTile<ORDER> L;
  constexpr int R = L::R;
  const TilePos t = tile_pos();
  const long long* C = S + L::at(4 * t.xh, t.y, 2 * t.zz);
  longlong2 w[4 + 2 * R];
#pragma unroll
  for (int q = 0; q < 4 + 2 * R; ++q)
    w[q] = *reinterpret_cast<const longlong2*>(C + (q - R) * L::px);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const long long* c = C + q * L::px;
    const longlong2 own = w[q + R];
    // z window: elements -RZ .. RZ + 1
    long long z[2 * L::RZ + 2];
#pragma unroll
    for (int a = 0; a < L::RZ + 1; ++a) {
      const longlong2 v = 2 * a == L::RZ ? own
                                         : *reinterpret_cast<const longlong2*>(c + 2 * a - L::RZ);
      z[2 * a] = v.x;
      z[2 * a + 1] = v.y;
    }
    long long s0[3] = {0, 0, 0}, s1[3] = {0, 0, 0};
#pragma unroll
    for (int d = 1; d <= R; ++d) {
      const longlong2 ym = *reinterpret_cast<const longlong2*>(c - d * L::py);
      const longlong2 yp = *reinterpret_cast<const longlong2*>(c + d * L::py);
      s0[d - 1] = (z[L::RZ - d] + z[L::RZ + d]) + (ym.x + yp.x) + (w[q + R - d].x + w[q + R + d].x);
      s1[d - 1] =
          (z[L::RZ + 1 - d] + z[L::RZ + 1 + d]) + (ym.y + yp.y) + (w[q + R - d].y + w[q + R + d].y);
    }
    longlong2 T;
    T.x = fx_weighted<ORDER>(s0) + fx_centre<ORDER>(own.x);
    T.y = fx_weighted<ORDER>(s1) + fx_centre<ORDER>(own.y);
    do_pair(q, T, own);
  }
}

// T of the three first derivatives (fx_first) of the thread's 8 cells: do_pair(q, x, y, z
// pairs) for plane 4 xh + q.
template <int ORDER, typename F>
__device__ __forceinline__ void tile_gradients(const long long* S, F do_pair) {
  typedef FxTile<ORDER> L;
  constexpr int R = L::R;
  const TilePos t = tile_pos();
  const long long* C = S + L::at(4 * t.xh, t.y, 2 * t.zz);
  longlong2 w[4 + 2 * R];
#pragma unroll
  for (int q = 0; q < 4 + 2 * R; ++q)
    w[q] = *reinterpret_cast<const longlong2*>(C + (q - R) * L::px);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const long long* c = C + q * L::px;
    long long z[2 * L::RZ + 2];
#pragma unroll
    for (int a = 0; a < L::RZ + 1; ++a) {
      const longlong2 v = *reinterpret_cast<const longlong2*>(c + 2 * a - L::RZ);
      z[2 * a] = v.x;
      z[2 * a + 1] = v.y;
    }
    long long x0[3] = {0, 0, 0}, x1[3] = {0, 0, 0}, y0[3] = {0, 0, 0}, y1[3] = {0, 0, 0};
    long long z0[3] = {0, 0, 0}, z1[3] = {0, 0, 0};
#pragma unroll
    for (int d = 1; d <= R; ++d) {
      const longlong2 ym = *reinterpret_cast<const longlong2*>(c - d * L::py);
      const longlong2 yp = *reinterpret_cast<const longlong2*>(c + d * L::py);
      y0[d - 1] = yp.x - ym.x;
      y1[d - 1] = yp.y - ym.y;
      x0[d - 1] = w[q + R + d].x - w[q + R - d].x;
      x1[d - 1] = w[q + R + d].y - w[q + R - d].y;
      z0[d - 1] = z[L::RZ + d] - z[L::RZ - d];
      z1[d - 1] = z[L::RZ + 1 + d] - z[L::RZ + 1 - d];
    }
    do_pair(q, make_longlong2(fx_first<ORDER>(x0), fx_first<ORDER>(x1)),
            make_longlong2(fx_first<ORDER>(y0), fx_first<ORDER>(y1)),
            make_longlong2(fx_first<ORDER>(z0), fx_first<ORDER>(z1)));
  }
}

// The tile with the edges between two faces as well (mixed derivatives), in two passes:
// the values into shared memory with their largest exponent, then every value aligned in
// place.  Cells outside along more than two axes count as 0.
template <int ORDER, typename Src>
__device__ __forceinline__ unsigned tile_load_edges(const Grid& G, const Src& src, int i0, int j0,
                                                    int k0, long long* S) {
  typedef FxTile<ORDER> L;
  constexpr int R = L::R, RZ = L::RZ, ZP = L::SZ / 2;
  const int ex = min(kTileX, G.n0 - i0), ey = min(kTileY, G.n1 - j0), ez = min(kTileZ, G.n2 - k0);
  double2* D = reinterpret_cast<double2*>(S);
  unsigned m = 0;
#pragma unroll 4
  for (int e = threadIdx.x; e < L::elems / 2; e += kTileThreads) {
    const int z = 2 * (e % ZP) - RZ, r = e / ZP;
    const int y = r % L::SY - R, x = r / L::SY - R;
    const int out = (x < 0 || x >= ex) + (y < 0 || y >= ey);
    double2 v = make_double2(0.0, 0.0);
    if (x < ex + R && y < ey + R) {
      const bool all = out < 2;  // z ghosts belong to rows that are out along one axis at most
      const bool a = (z >= 0 && z < ez) || (all && z >= -R && z < ez + R);
      const bool b = (z + 1 >= 0 && z + 1 < ez) || (all && z + 1 >= -R && z + 1 < ez + R);
      if (a || b) {
        v = *reinterpret_cast<const double2*>(src.at(i0 + x, j0 + y, k0 + z));
        if (!a) v.x = 0.0;
        if (!b) v.y = 0.0;
      }
    }
    D[e] = v;
    m = max(m, max(fx_key(v.x), fx_key(v.y)));
  }
  m = block_max(m) | 0x1fffffu;
  if (fx_in_range(m)) {
    longlong2* A = reinterpret_cast<longlong2*>(S);
#pragma unroll 4
    for (int e = threadIdx.x; e < L::elems / 2; e += kTileThreads) {
      const double2 v = D[e];
      A[e] = make_longlong2(fx_align(v.x, m), fx_align(v.y, m));
    }
  }
  __syncthreads();
  if (!fx_in_range(m)) return m;
  const TilePos t = tile_pos();
  unsigned a[4], b[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const longlong2 v = *reinterpret_cast<const longlong2*>(S + L::at(4 * t.xh + q, t.y, 2 * t.zz));
    a[q] = (unsigned)((int)(v.x >> 32) ^ (int)(v.x >> 63));
    b[q] = (unsigned)((int)(v.y >> 32) ^ (int)(v.y >> 63));
  }
  const bool low = least_window<ORDER>(a, b) < 1u << (26 - kTileRange<ORDER>);
  return tile_key<ORDER>(m, S, src, i0, j0, k0, ex, ey, ez, low);
}

// The finite-difference Hessian of a column of 8 cells per thread (z = lane, y = warp) as
// integers: do_cell(x, d, m) with d = the second differences along x, y, z (fx_second) and
// m = G_x G_y, G_x G_z, G_y G_z (fx_first of fx_first).  The column's values and its first
// derivatives along y and z slide through registers (7 planes of each at order 6).
template <int ORDER, typename F>
__device__ __forceinline__ void tile_hessians(const long long* S, F do_cell) {
  typedef FxTile<ORDER> L;
  constexpr int R = L::R, N = kTileX + 2 * R;
  const long long* C = S + L::at(0, threadIdx.x >> 5, threadIdx.x & 31);
  // first derivative at p along the axis of stride st
  auto first = [](const long long* p, int st) {
    long long d[3] = {0, 0, 0};
#pragma unroll
    for (int q = 1; q <= R; ++q) d[q - 1] = p[q * st] - p[-q * st];
    return fx_first<ORDER>(d);
  };
  auto second = [](const long long* p, int st, long long c) {
    long long s[3] = {0, 0, 0};
#pragma unroll
    for (int q = 1; q <= R; ++q) s[q - 1] = p[q * st] + p[-q * st];
    return fx_second<ORDER>(s, c);
  };
  long long w[N], fy[N], fz[N];
#pragma unroll
  for (int n = 0; n < N; ++n) {
    const long long* e = C + (n - R) * L::px;
    w[n] = e[0];
    fy[n] = first(e, L::py);
    fz[n] = first(e, 1);
    if (n < 2 * R) continue;
    const int x = n - 2 * R;  // the window is complete for this plane
    const long long* c = C + x * L::px;
    long long s[3] = {0, 0, 0}, gy[3] = {0, 0, 0}, gz[3] = {0, 0, 0}, yz[3] = {0, 0, 0};
#pragma unroll
    for (int q = 1; q <= R; ++q) {
      s[q - 1] = w[x + R + q] + w[x + R - q];
      gy[q - 1] = fy[x + R + q] - fy[x + R - q];
      gz[q - 1] = fz[x + R + q] - fz[x + R - q];
      yz[q - 1] = first(c + q * L::py, 1) - first(c - q * L::py, 1);
    }
    const long long own = w[x + R];
    const long long d[3] = {fx_second<ORDER>(s, own), second(c, L::py, own), second(c, 1, own)};
    const long long m[3] = {fx_first<ORDER>(gy), fx_first<ORDER>(gz), fx_first<ORDER>(yz)};
    do_cell(x, d, m);
  }
}

}  // namespace mgk
