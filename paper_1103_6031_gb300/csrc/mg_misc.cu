// Coarsest-level solve, convergence norms, composite mean, packing between the
// caller's dense arrays and the padded level layout, the 2LPT source and the
// displacement gradient (Hahn & Abel 2011, Sec. 3.1, 3.2).
#include <type_traits>

#include "mg_internal.h"
#include "mg_launch.cuh"
#include "mg_stencil.cuh"
#include "mg_tile.cuh"
#include "mg_vbody.cuh"

namespace mgk {

namespace {

// Table 1 gradient: antisymmetric weights on offsets +1, +2, +3 (units 1/h).
template <int ORDER>
struct Grad;
template <>
struct Grad<2> {
  static constexpr double g1 = 0.5, g2 = 0.0, g3 = 0.0;
};
template <>
struct Grad<4> {
  static constexpr double g1 = 8.0 / 12.0, g2 = -1.0 / 12.0, g3 = 0.0;
};
template <>
struct Grad<6> {
  static constexpr double g1 = 45.0 / 60.0, g2 = -9.0 / 60.0, g3 = 1.0 / 60.0;
};

template <int ORDER>
__device__ __forceinline__ double grad_w(int s) {  // weight at offset s in [-3, 3]
  const int a = s < 0 ? -s : s;
  const double v = a == 1 ? Grad<ORDER>::g1 : (a == 2 ? Grad<ORDER>::g2 : (a == 3 ? Grad<ORDER>::g3 : 0.0));
  return s < 0 ? -v : v;
}

template <int ORDER>
__device__ __forceinline__ double lap_w(int s) {
  const int a = s < 0 ? -s : s;
  return a == 0 ? Lap<ORDER>::w0 : (a == 1 ? Lap<ORDER>::w1 : (a == 2 ? Lap<ORDER>::w2 : Lap<ORDER>::w3));
}

// Periodic pseudo-inverse of L on the coarsest level as a circular convolution:
// u(x) = sum_y K(x - y) f(y), K precomputed on the host from the DFT symbol.
// One block per output cell; the block's threads split the sum over y.  The
// result is also written to the cell's periodic ghost images.
constexpr int kCoarseBlock = kCoarseThreads;

template <typename T>
__global__ void __launch_bounds__(kCoarseBlock)
    k_coarsest(Grid G, const T* f, T* u,
               const double* kern) {
  grid_wait();
  coarsest_body<T>(G, f, u, kern, (int)blockIdx.x, (int)threadIdx.x);
}

template <int BLOCK>
__device__ __forceinline__ void block_sum2(double& a, double& b) {
  __shared__ double sa[BLOCK], sb[BLOCK];
  sa[threadIdx.x] = a;
  sb[threadIdx.x] = b;
  __syncthreads();
#pragma unroll
  for (int w = BLOCK / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      sa[threadIdx.x] += sa[threadIdx.x + w];
      sb[threadIdx.x] += sb[threadIdx.x + w];
    }
    __syncthreads();
  }
  a = sa[0];
  b = sb[0];
}

constexpr int kRedBlock = 256;

// One block per (x plane, 8 y rows); 32 lanes stride along z.  Block b writes
// its partial sums to slot b, so the reduction order is fixed.
// MIXED: the float64 residual of every uncovered interior cell is also stored in r32,
// rounded to float32, as the source of the correction equation; covered cells are skipped
// for both.  The stencil sums run on the integer pipe (mg_fixed.cuh) except in MIXED, where
// the last bits of r decide float32 roundings of the whole correction cycle: with them
// changed, displacements of the deepest nest of a 5-level hierarchy moved by 1.1e-9
// relative, so that mode keeps the FP64 operations one by one and sheds what does not touch
// them: the source's sum is left from the solve's first call (u = nullptr, the only one to
// form it), and r is rounded to float32 on the integer pipe (FP64-bound: 91 us per 128^3 level).
//
// r rounded to nearest even; results that are not normal floats by the conversion instruction.
__device__ __forceinline__ float to_float(double r) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(r);
  const unsigned long long m = b & 0x7fffffffffffffffull;
  const unsigned q = (unsigned)((m + 0x0fffffffull + ((m >> 29) & 1)) >> 29);  // exponent bias 1023
  const unsigned e = (unsigned)(b >> 52) & 0x7ffu;
  if (e - 897u >= 253u) return (float)r;
  return __uint_as_float((q - (896u << 23)) | ((unsigned)(b >> 32) & 0x80000000u));
}

template <int ORDER, bool MIXED>
__global__ void __launch_bounds__(kRedBlock)
    k_norm_partial(Grid G, const double* u, const double* f,
                   double invh2, double vol, Int3 clo, Int3 chi, double* __restrict__ partial,
                   float* __restrict__ r32) {
  grid_wait();
  const int sy = G.Zp, sx = G.Y * G.Zp;
  const int i = blockIdx.y;
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  double rr = 0.0, ff = 0.0;
  if (j < G.n1) {
    const bool row_cov = i >= clo.x && i < chi.x && j >= clo.y && j < chi.y;
    const long long row = gidx(G, i, j, 0);
#pragma unroll 1
    for (int k = lane; k < G.n2; k += 32) {
      // covered cells: no norm term, and no correction source either (the FAS
      // restriction overwrites a covered parent cell's source before the parent uses it)
      const bool cov = row_cov && k >= clo.z && k < chi.z;
      if (cov) continue;
      const long long p = row + k;
      const double fv = f[p];
      const double r = u ? add_lap_h2<ORDER, double, !MIXED>(u, p, sy, sx, u[p],
                                                                 -invh2, fv)
                         : fv;
      if (MIXED) r32[p] = to_float(r);
      rr = fma(r, r, rr);
      if (!MIXED || !u) ff = fma(fv, fv, ff);
    }
  }
  block_sum2<kRedBlock>(rr, ff);
  if (threadIdx.x == 0) {
    const int b = blockIdx.y * gridDim.x + blockIdx.x;
    partial[2 * b] = rr * vol;
    if (!MIXED || !u) partial[2 * b + 1] = ff * vol;
  }
}

// The norm sums of float64 levels on tiles of aligned integers (mg_tile.cuh): 4 FP64
// instructions per cell (the conversion, the residual, two squares).  Block b writes slot b,
// the first block zeros the slots that k_norm_partial would use beyond.
template <int ORDER>
__global__ void __launch_bounds__(kTileThreads, 3)
    k_norm_tile(Grid G, const double* u, const double* f, double invh2,
                double vol, Int3 clo, Int3 chi, double* __restrict__ partial, int slots) {
  grid_wait();
  extern __shared__ __align__(16) long long norm_smem[];
  const int i0 = blockIdx.z * kTileX, j0 = blockIdx.y * kTileY, k0 = blockIdx.x * kTileZ;
  const int b = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  const int blocks = gridDim.x * gridDim.y * gridDim.z;
  if (b == 0)
    for (int q = blocks + threadIdx.x; q < slots; q += kTileThreads)
      partial[2 * q] = partial[2 * q + 1] = 0.0;
  double rr = 0.0, ff = 0.0;
  // a block inside the covered region has no leaf cell
  const bool covered = i0 >= clo.x && min(i0 + kTileX, G.n0) <= chi.x && j0 >= clo.y &&
                       min(j0 + kTileY, G.n1) <= chi.y && k0 >= clo.z &&
                       min(k0 + kTileZ, G.n2) <= chi.z;
  if (!covered) {
    const TilePos t = tile_pos();
    const int i = i0 + 4 * t.xh, j = j0 + t.y, k = k0 + 2 * t.zz;
    const long long p = gidx(G, i, j, k);
    const int sx = G.Y * G.Zp;
    const double kr = -invh2 * FxUnit<ORDER>::v;
    double2 fv[4];  // under way while the tile is filled (86.3 us after it, 82.5 so)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      fv[q] = i + q < G.n0 && j < G.n1 && k < G.n2
                  ? *reinterpret_cast<const double2*>(f + p + q * sx) : make_double2(0.0, 0.0);
    const unsigned key = tile_load<ORDER>(G, u, i0, j0, k0, norm_smem);
    const bool fx = fx_in_range(key) && fx_scalable(kr, key);
    const double ks = fx_scale(kr, key);
    auto leaf = [&](int q, int dk) {
      return i + q < G.n0 && j < G.n1 && k + dk < G.n2 &&
             !(i + q >= clo.x && i + q < chi.x && j >= clo.y && j < chi.y && k + dk >= clo.z &&
               k + dk < chi.z);
    };
    auto add = [&](double r, double fv) {
      rr = fma(r, r, rr);
      ff = fma(fv, fv, ff);
    };
    if (fx) {
      tile_laplacians<ORDER>(norm_smem, [&](int q, longlong2 T, longlong2) {
        if (leaf(q, 0)) add(fma(ks, (double)T.x, fv[q].x), fv[q].x);
        if (leaf(q, 1)) add(fma(ks, (double)T.y, fv[q].y), fv[q].y);
      });
    } else {
#pragma unroll 1
      for (int q = 0; q < 8; ++q) {
        if (!leaf(q >> 1, q & 1)) continue;
        const long long e = p + (q >> 1) * sx + (q & 1);
        const double fv = f[e];
        add(add_lap_h2<ORDER, double, false>(u, e, G.Zp, sx, u[e], -invh2, fv), fv);
      }
    }
  }
  block_sum2<kTileThreads>(rr, ff);
  if (threadIdx.x == 0) {
    partial[2 * b] = rr * vol;
    partial[2 * b + 1] = ff * vol;
  }
}

__global__ void __launch_bounds__(kRedBlock)
    k_sum_partial(Grid G, const double* f, double vol, Int3 clo, Int3 chi,
                  double* partial) {
  grid_wait();
  const int i = blockIdx.y;
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  double s = 0.0, unused = 0.0;
  if (j < G.n1) {
    const bool row_cov = i >= clo.x && i < chi.x && j >= clo.y && j < chi.y;
    const long long row = gidx(G, i, j, 0);
    for (int k = lane; k < G.n2; k += 32) {
      if (row_cov && k >= clo.z && k < chi.z) continue;
      s += f[row + k];
    }
  }
  block_sum2<kRedBlock>(s, unused);
  if (threadIdx.x == 0) {
    const int b = blockIdx.y * gridDim.x + blockIdx.x;
    partial[2 * b] = s * vol;
    partial[2 * b + 1] = 0.0;
  }
}

// Sums `count` consecutive (a, b) pairs in a fixed order into out[0], out[1].
__global__ void __launch_bounds__(kRedBlock)
    k_reduce_partials(const double* partial, int count, double* out) {
  grid_wait();
  double a = 0.0, b = 0.0;
  for (int t = threadIdx.x; t < count; t += kRedBlock) {
    a += partial[2 * t];
    b += partial[2 * t + 1];
  }
  block_sum2<kRedBlock>(a, b);
  if (threadIdx.x == 0) {
    out[0] = a;
    out[1] = b;
  }
}

// Block 0: exactly k_reduce_partials over all `count` pairs into out[0], out[1].
// Block 1 + l: the pairs of leaf level l alone, [R.off[l], R.off[l] + R.cnt[l]), into
// out_levels[2 l], out_levels[2 l + 1] (the per-level residual and source sums).  With host
// (pinned host memory, laid out like the record that starts at out) the record's entries go
// there as well, so that no copy follows: out[2..4], left by earlier kernels, by block 0.
__global__ void __launch_bounds__(kRedBlock)
    k_reduce_levels(const double* partial, int count, LevelRanges R,
                    double* out, double* out_levels,
                    double* host) {
  grid_wait();
  int lo = 0, hi = count;
  if (blockIdx.x > 0) {
    lo = R.off[blockIdx.x - 1];
    hi = lo + R.cnt[blockIdx.x - 1];
  }
  double a = 0.0, b = 0.0;
  for (int t = lo + threadIdx.x; t < hi; t += kRedBlock) {
    a += partial[2 * t];
    b += partial[2 * t + 1];
  }
  block_sum2<kRedBlock>(a, b);
  if (threadIdx.x == 0) {
    double* o = blockIdx.x == 0 ? out : out_levels + 2 * (blockIdx.x - 1);
    o[0] = a;
    o[1] = b;
    if (host) {
      double* ho = host + (o - out);
      ho[0] = a;
      ho[1] = b;
      if (blockIdx.x == 0)
        for (int q = 2; q < 5; ++q) host[q] = out[q];
    }
  }
}

// Copies between dense and padded arrays: blocks of kCopyZ x kCopyY cells of a plane (no
// divisions per cell).
constexpr int kCopyZ = 64, kCopyY = 4;

inline dim3 copy_grid(const Grid& G) {
  return dim3((G.n2 + kCopyZ - 1) / kCopyZ, (G.n1 + kCopyY - 1) / kCopyY, G.n0);
}

__global__ void __launch_bounds__(256)
    k_pack(Grid G, const double* src, double* __restrict__ dst, double shift) {
  grid_wait();
  const int k = blockIdx.x * kCopyZ + threadIdx.x, j = blockIdx.y * kCopyY + threadIdx.y;
  const int i = blockIdx.z;
  if (k >= G.n2 || j >= G.n1) return;
  dst[gidx(G, i, j, k)] = src[((long long)i * G.n1 + j) * G.n2 + k] - shift;
}

__global__ void __launch_bounds__(256)
    k_unpack(Grid G, const double* src, double* __restrict__ dst, double add) {
  grid_wait();
  const int k = blockIdx.x * kCopyZ + threadIdx.x, j = blockIdx.y * kCopyY + threadIdx.y;
  const int i = blockIdx.z;
  if (k >= G.n2 || j >= G.n1) return;
  dst[((long long)i * G.n1 + j) * G.n2 + k] = src[gidx(G, i, j, k)] + add;
}

// f -= mean, f2 = f on the interior; mean = *mean_num * inv_volume (device-side).
__global__ void __launch_bounds__(256)
    k_shift_copy(Grid G, double* f, double* f2,
                 const double* mean_num, double inv_volume) {
  grid_wait();
  const int k = blockIdx.x * kCopyZ + threadIdx.x, j = blockIdx.y * kCopyY + threadIdx.y;
  const int i = blockIdx.z;
  if (k >= G.n2 || j >= G.n1) return;
  const long long p = gidx(G, i, j, k);
  const double v = f[p] - mean_num[0] * inv_volume;
  f[p] = v;
  if (f2) f2[p] = v;
}

// u += e on the interior (float64 += float32 correction); periodic levels also
// update their ghost images.  One thread per cell of a (32 x 4)-cell tile row.
__global__ void __launch_bounds__(128)
    k_add_correction(Grid G, double* u, const float* e, int periodic) {
  grid_wait();
  const int k = blockIdx.x * 32 + threadIdx.x;
  const int j = blockIdx.y * 4 + threadIdx.y;
  const int i = blockIdx.z;
  if (k >= G.n2 || j >= G.n1) return;
  const long long p = gidx(G, i, j, k);
  const double v = u[p] + (double)e[p];
  u[p] = v;
  if (periodic) write_images<double>(G, u, i, j, k, v);
}

// p = p - sum[0] * scale (+ add) over n elements (sum read on the device).
__global__ void __launch_bounds__(256)
    k_sub_mean(double* p, long long n, const double* sum, double scale,
               double add) {
  grid_wait();
  const long long t = blockIdx.x * 256LL + threadIdx.x;
  if (t >= n) return;
  const double v = p[t] - sum[0] * scale;
  p[t] = add != 0.0 ? v + add : v;
}

__global__ void __launch_bounds__(256) k_fill(double* p, long long n, double v) {
  grid_wait();
  const long long t = blockIdx.x * 256LL + threadIdx.x;
  if (t < n) p[t] = v;
}

// The 2LPT source in FP64 arithmetic, operation by operation, for the second solve of the
// mixed mode: its float32 cycles turn a changed last bit of the source into changes of
// 1e-9 of the result (measured: two cells whose source rounded differently to float32
// moved displacements of the finest nest by 1.7e-9).
//
// First derivatives D_b = G_b phi (Table 1 gradient, times h), b = y, z, on every cell whose
// b coordinate is interior and whose other two coordinates lie anywhere in the ghost-padded
// box (the mixed derivatives read D_b up to g cells outside the interior along the other
// axes).
template <int ORDER>
__global__ void __launch_bounds__(128)
    k_first_derivs(Grid G, const double* phi, double* __restrict__ dy,
                   double* __restrict__ dz) {
  grid_wait();
  constexpr int half = ORDER / 2;
  const int g = G.g;
  const int k = (int)(blockIdx.x * 32 + threadIdx.x) - g;
  const int j = (int)(blockIdx.y * 4 + threadIdx.y) - g;
  const int i = (int)blockIdx.z - g;
  if (k >= G.n2 + g || j >= G.n1 + g) return;
  const long long p = gidx(G, i, j, k);
  const int st[2] = {G.Zp, 1};
  const bool in[2] = {j >= 0 && j < G.n1, k >= 0 && k < G.n2};
  double* out[2] = {dy, dz};
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    if (!in[b]) continue;
    double acc = 0.0;
#pragma unroll
    for (int s = 1; s <= half; ++s)
      acc = fma(grad_w<ORDER>(s), phi[p + s * st[b]] - phi[p - s * st[b]], acc);
    out[b][p] = acc;
  }
}

// tau from phi and its first derivatives: phi_aa the 1D second difference along a, phi_xy =
// G_x D_y, phi_xz = G_x D_z, phi_yz = G_y D_z.
template <int ORDER>
__global__ void __launch_bounds__(128)
    k_lpt2_source(Grid G, const double* phi, const double* dy,
                  const double* dz, double invh2, double* __restrict__ tau) {
  grid_wait();
  constexpr int half = ORDER / 2;
  const int k = blockIdx.x * 32 + threadIdx.x;
  const int j = blockIdx.y * 4 + threadIdx.y;
  const int i = blockIdx.z;
  if (k >= G.n2 || j >= G.n1) return;
  const long long p = gidx(G, i, j, k);
  const int st[3] = {G.Y * G.Zp, G.Zp, 1};
  double d[3], m[3];
  const double c = phi[p];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double acc = Lap<ORDER>::w0 * c;
#pragma unroll
    for (int s = 1; s <= half; ++s)
      acc = fma(lap_w<ORDER>(s), phi[p + s * st[a]] + phi[p - s * st[a]], acc);
    d[a] = acc * invh2;
  }
  const double* src[3] = {dy, dz, dz};
  const int ax[3] = {0, 0, 1};
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    double acc = 0.0;
#pragma unroll
    for (int s = 1; s <= half; ++s)
      acc = fma(grad_w<ORDER>(s), src[q][p + s * st[ax[q]]] - src[q][p - s * st[ax[q]]],
                acc);
    m[q] = acc * invh2;
  }
  tau[p] = fma(d[0], d[1] + d[2], d[1] * d[2]) - fma(m[0], m[0], fma(m[1], m[1], m[2] * m[2]));
}

// Finite-difference Hessian at element p in FP64 arithmetic: d[a] = phi_aa h^2, m = (phi_xy,
// phi_xz, phi_yz) h^2 with phi_ab = G_a (G_b phi).
template <int ORDER, typename Src>
__device__ __forceinline__ void fd_hessian(const Src& src, int i, int j, int k, double (&d)[3],
                                           double (&m)[3]) {
  constexpr int half = ORDER / 2;
  // the cell at offset s along axis a and t along axis b
  auto at = [&](int a, int s, int b, int t) {
    return *src.at(i + (a == 0 ? s : 0) + (b == 0 ? t : 0), j + (a == 1 ? s : 0) + (b == 1 ? t : 0),
                        k + (a == 2 ? s : 0) + (b == 2 ? t : 0));
  };
  const double c = at(0, 0, 0, 0);
#pragma unroll 1
  for (int a = 0; a < 3; ++a) {
    double acc = Lap<ORDER>::w0 * c;
    for (int s = 1; s <= half; ++s)
      acc = fma(lap_w<ORDER>(s), at(a, s, a, 0) + at(a, -s, a, 0), acc);
    d[a] = acc;
  }
#pragma unroll 1
  for (int q = 0; q < 3; ++q) {
    const int a = q == 2 ? 1 : 0, b = q == 0 ? 1 : 2;
    double acc = 0.0;
    for (int s = -half; s <= half; ++s) {
      if (s == 0) continue;
      double g = 0.0;
      for (int t = 1; t <= half; ++t) g = fma(grad_w<ORDER>(t), at(a, s, b, t) - at(a, s, b, -t), g);
      acc = fma(grad_w<ORDER>(s), g, acc);
    }
    m[q] = acc;
  }
}

// What is made of the Hessian (second derivatives d, mixed m = xy, xz, yz).
// 2LPT source: tau = sum_{i<j} (phi_ii phi_jj - phi_ij^2) (Sec. 3.1.2).
// d and m in units of s2 and s1.
struct TauOp {
  double k2, k1;
  __device__ __forceinline__ TauOp(double s2, double s1) : k2(s2 * s2), k1(s1 * s1) {}
  __device__ __forceinline__ double operator()(const double (&d)[3], const double (&m)[3]) const {
    return fma(k2, fma(d[0], d[1] + d[2], d[1] * d[2]),
               -(k1 * fma(m[0], m[0], fma(m[1], m[1], m[2] * m[2]))));
  }
};

// Local Lagrangian density (Sec. 5.3): with H the Hessian of the combined potential Phi
// (L = -grad Phi), rho / rho_bar = 1 / det[I - H]; writes 1/det - 1 (the renormalisation and
// the +1 follow on the host side).  det[I - H] = a b c - a m_yz^2 - b m_xz^2 - c m_xy^2
// - 2 m_xy m_xz m_yz with a, b, c = 1 - phi_xx, 1 - phi_yy, 1 - phi_zz.
struct LlaOp {
  double s2, s1;
  __device__ __forceinline__ LlaOp(double s2_, double s1_) : s2(s2_), s1(s1_) {}
  __device__ __forceinline__ double operator()(const double (&d)[3], const double (&m_)[3]) const {
    const double a = fma(-s2, d[0], 1.0), b = fma(-s2, d[1], 1.0), c = fma(-s2, d[2], 1.0);
    const double m[3] = {s1 * m_[0], s1 * m_[1], s1 * m_[2]};
    const double w = fma(2.0, m[0] * m[2], b * m[1]);
    const double det = fma(a, fma(b, c, -(m[2] * m[2])), -fma(m[1], w, c * m[0] * m[0]));
    return 1.0 / det - 1.0;
  }
};

// A scale whose square is far from overflow and underflow.
__device__ __forceinline__ bool squarable(double s) {
  const int e = (__double2hiint(s) >> 20) & 0x7ff;
  return e > 600 && e < 1400;
}

// OP of the Hessian of phi (ghosts and edge ghosts filled), one launch and no work arrays:
// a tile of aligned integers with its edges (mg_tile.cuh), first derivatives and their
// derivatives as integer sums; FP64 instructions are left only for the 6 conversions and OP
// (14 per cell for tau, 65 when every sum ran on the FP64 pipe).  DENSE: phi and out are
// dense arrays of a periodic level, read and written without a padded copy (256^3, order 6:
// the copies and the ghost fill were 128 of 845 us).
template <int ORDER, typename OP, bool DENSE>
__global__ void __launch_bounds__(kTileThreads, 3)
    k_hessian_tile(Grid G, const double* phi, double invh2, double* __restrict__ out) {
  grid_wait();
  extern __shared__ __align__(16) long long hess_smem[];
  const int i0 = blockIdx.z * kTileX, j0 = blockIdx.y * kTileY, k0 = blockIdx.x * kTileZ;
  typedef typename std::conditional<DENSE, DensePeriodicSource, PaddedSource>::type Src;
  const Src src(G, phi);
  const unsigned key = tile_load_edges<ORDER>(G, src, i0, j0, k0, hess_smem);
  const int j = j0 + (threadIdx.x >> 5), k = k0 + (threadIdx.x & 31);
  if (j >= G.n1 || k >= G.n2) return;
  const long long p = DENSE ? ((long long)i0 * G.n1 + j) * G.n2 + k : gidx(G, i0, j, k);
  const int sx = DENSE ? G.n1 * G.n2 : G.Y * G.Zp;
  const int nx = min(kTileX, G.n0 - i0);
  const double k2 = invh2 * FxUnit<ORDER>::v;
  const double k1 = invh2 * (FxGradUnit<ORDER>::v * FxGradUnit<ORDER>::v);
  const double s2 = fx_scale(k2, key), s1 = fx_scale(k1, key);
  if (fx_in_range(key) && fx_scalable(k2, key) && fx_scalable(k1, key) && squarable(s2) &&
      squarable(s1)) {
    const OP op(s2, s1);
    tile_hessians<ORDER>(hess_smem, [&](int x, const long long (&di)[3], const long long (&mi)[3]) {
      if (x >= nx) return;
      const double d[3] = {(double)di[0], (double)di[1], (double)di[2]};
      const double m[3] = {(double)mi[0], (double)mi[1], (double)mi[2]};
      out[p + x * sx] = op(d, m);
    });
    return;
  }
  const OP op(1.0, 1.0);
#pragma unroll 1
  for (int x = 0; x < nx; ++x) {
    double d[3], m[3];
    fd_hessian<ORDER>(src, i0 + x, j, k, d, m);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      d[a] *= invh2;
      m[a] *= invh2;
    }
    out[p + x * sx] = op(d, m);
  }
}

// out[t] = a1 x1[t] + a2 x2[t] (x2 may be NULL) over n dense elements.
__global__ void __launch_bounds__(256)
    k_axpby(long long n, double a1, const double* __restrict__ x1, double a2,
            const double* __restrict__ x2, double* __restrict__ out) {
  const long long t = blockIdx.x * 256LL + threadIdx.x;
  if (t >= n) return;
  out[t] = x2 ? fma(a2, __ldg(x2 + t), a1 * __ldg(x1 + t)) : a1 * __ldg(x1 + t);
}

template <int ORDER>
__global__ void __launch_bounds__(128)
    k_gradient(Grid G, const double* phi, double invh, double* __restrict__ dx,
               double* __restrict__ dy, double* __restrict__ dz) {
  grid_wait();
  constexpr int half = ORDER / 2;
  const int k = blockIdx.x * 32 + threadIdx.x, j = blockIdx.y * 4 + threadIdx.y, i = blockIdx.z;
  if (k >= G.n2 || j >= G.n1) return;
  const long long t = ((long long)i * G.n1 + j) * G.n2 + k;
  const long long p = gidx(G, i, j, k);
  const long long st[3] = {(long long)G.Y * G.Zp, (long long)G.Zp, 1};
  double out[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double acc = 0.0;
#pragma unroll
    for (int s = 1; s <= half; ++s)
      acc = fma(grad_w<ORDER>(s), phi[p + s * st[a]] - phi[p - s * st[a]], acc);
    out[a] = -acc * invh;
  }
  dx[t] = out[0];
  dy[t] = out[1];
  dz[t] = out[2];
}

// The same on tiles of aligned integers (mg_tile.cuh): 6 FP64 instructions per cell instead
// of 21.
template <int ORDER>
__global__ void __launch_bounds__(kTileThreads, 3)
    k_gradient_tile(Grid G, const double* phi, double invh, double* __restrict__ dx,
                    double* __restrict__ dy, double* __restrict__ dz) {
  grid_wait();
  extern __shared__ __align__(16) long long grad_smem[];
  const int i0 = blockIdx.z * kTileX, j0 = blockIdx.y * kTileY, k0 = blockIdx.x * kTileZ;
  const unsigned key = tile_load<ORDER>(G, phi, i0, j0, k0, grad_smem);
  const TilePos t = tile_pos();
  const int i = i0 + 4 * t.xh, j = j0 + t.y, k = k0 + 2 * t.zz;
  if (j >= G.n1 || k >= G.n2) return;
  const long long o = ((long long)i * G.n1 + j) * G.n2 + k, ox = (long long)G.n1 * G.n2;
  const double kg = -invh * FxGradUnit<ORDER>::v;
  const bool two = k + 1 < G.n2;
  if (fx_in_range(key) && fx_scalable(kg, key)) {
    const double s = fx_scale(kg, key);
    const bool vec = (G.n2 & 1) == 0 &&
                     ((reinterpret_cast<size_t>(dx) | reinterpret_cast<size_t>(dy) |
                       reinterpret_cast<size_t>(dz)) & 15) == 0;
    tile_gradients<ORDER>(grad_smem, [&](int q, longlong2 x, longlong2 y, longlong2 z) {
      if (i + q >= G.n0) return;
      auto put = [&](double* dst, longlong2 v) {
        const double a = s * (double)v.x, b = s * (double)v.y;
        double* e = dst + o + q * ox;
        if (vec) {
          *reinterpret_cast<double2*>(e) = make_double2(a, b);
        } else {
          e[0] = a;
          if (two) e[1] = b;
        }
      };
      put(dx, x);
      put(dy, y);
      put(dz, z);
    });
    return;
  }
  const long long p = gidx(G, i, j, k);
  const int st[3] = {G.Y * G.Zp, G.Zp, 1};
  double* const out[3] = {dx, dy, dz};
#pragma unroll 1
  for (int q = 0; q < 8; ++q) {
    if (i + (q >> 1) >= G.n0 || k + (q & 1) >= G.n2) continue;
    const double* c = phi + p + (q >> 1) * st[0] + (q & 1);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      double acc = 0.0;
      for (int d = 1; d <= ORDER / 2; ++d)
        acc = fma(grad_w<ORDER>(d), c[d * st[a]] - c[-d * st[a]], acc);
      out[a][o + (q >> 1) * ox + (q & 1)] = -acc * invh;
    }
  }
}

inline unsigned blocks_for(long long n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

int norm_blocks(const Grid& G) { return ((G.n1 + 7) / 8) * G.n0; }

cudaError_t launch_coarsest(const Grid& G, const double* f, double* u, const double* kern,
                            cudaStream_t s) {
  const int n = G.n0 * G.n1 * G.n2;
  return launch_dep(k_coarsest<double>, n, kCoarseBlock, 0, s, G, f, u, kern);
}

cudaError_t launch_coarsest(const Grid& G, const float* f, float* u, const double* kern,
                            cudaStream_t s) {
  const int n = G.n0 * G.n1 * G.n2;
  return launch_dep(k_coarsest<float>, n, kCoarseBlock, 0, s, G, f, u, kern);
}

cudaError_t launch_norm_partial(int order, const Grid& G, const double* u, const double* f,
                                double invh2, double vol, Int3 clo, Int3 chi, double* partial,
                                int blocks, float* r32, cudaStream_t s) {
  const dim3 grid((G.n1 + 7) / 8, G.n0);
  if ((int)(grid.x * grid.y) != blocks) return cudaErrorInvalidValue;
  const dim3 tg = tile_grid(G);
  if (!r32 && u && tile_pays(G) && (long long)tg.x * tg.y * tg.z <= blocks) {
    switch (order) {
      case 2: return launch_dep(k_norm_tile<2>, tg, kTileThreads, FxTile<2>::bytes, s, G, u, f, invh2, vol, clo, chi, partial, blocks);
      case 4: return launch_dep(k_norm_tile<4>, tg, kTileThreads, FxTile<4>::bytes, s, G, u, f, invh2, vol, clo, chi, partial, blocks);
      case 6: return launch_dep(k_norm_tile<6>, tg, kTileThreads, FxTile<6>::bytes, s, G, u, f, invh2, vol, clo, chi, partial, blocks);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (order) {
    case 2:
      return r32 ? launch_dep(k_norm_partial<2, true>, grid, kRedBlock, 0, s, G, u, f, invh2, vol, clo, chi, partial, r32)
                 : launch_dep(k_norm_partial<2, false>, grid, kRedBlock, 0, s, G, u, f, invh2, vol, clo, chi, partial, r32);
    case 4:
      return r32 ? launch_dep(k_norm_partial<4, true>, grid, kRedBlock, 0, s, G, u, f, invh2, vol, clo, chi, partial, r32)
                 : launch_dep(k_norm_partial<4, false>, grid, kRedBlock, 0, s, G, u, f, invh2, vol, clo, chi, partial, r32);
    case 6:
      return r32 ? launch_dep(k_norm_partial<6, true>, grid, kRedBlock, 0, s, G, u, f, invh2, vol, clo, chi, partial, r32)
                 : launch_dep(k_norm_partial<6, false>, grid, kRedBlock, 0, s, G, u, f, invh2, vol, clo, chi, partial, r32);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t prepare_norm_tile() {
  const cudaError_t e = cudaFuncSetAttribute(
      k_norm_tile<6>, cudaFuncAttributeMaxDynamicSharedMemorySize, FxTile<6>::bytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_gradient_tile<6>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              FxTile<6>::bytes);
}

cudaError_t launch_sum_partial(const Grid& G, const double* f, double vol, Int3 clo, Int3 chi,
                               double* partial, int blocks, cudaStream_t s) {
  const dim3 grid((G.n1 + 7) / 8, G.n0);
  if ((int)(grid.x * grid.y) != blocks) return cudaErrorInvalidValue;
  return launch_dep(k_sum_partial, grid, kRedBlock, 0, s, G, f, vol, clo, chi, partial);
}

cudaError_t launch_reduce_partials(const double* partial, int count, int width, double* out,
                                   cudaStream_t s) {
  (void)width;
  return launch_dep(k_reduce_partials, 1, kRedBlock, 0, s, partial, count, out);
}

cudaError_t launch_reduce_levels(const double* partial, int count, const LevelRanges& R,
                                 double* out, double* out_levels, double* host, cudaStream_t s) {
  if (R.n < 0 || R.n > MG_MAX_LEVELS) return cudaErrorInvalidValue;
  for (int l = 0; l < R.n; ++l)
    if (R.off[l] < 0 || R.cnt[l] < 0 || R.off[l] + R.cnt[l] > count) return cudaErrorInvalidValue;
  return launch_dep(k_reduce_levels, 1 + R.n, kRedBlock, 0, s, partial, count, R, out, out_levels, host);
}

cudaError_t launch_pack(const Grid& G, const double* src, double* dst, double shift,
                        cudaStream_t s) {
  return launch_dep(k_pack, copy_grid(G), dim3(kCopyZ, kCopyY), 0, s, G, src, dst, shift);
}

cudaError_t launch_unpack(const Grid& G, const double* src, double* dst, cudaStream_t s,
                          double add) {
  return launch_dep(k_unpack, copy_grid(G), dim3(kCopyZ, kCopyY), 0, s, G, src, dst, add);
}

cudaError_t launch_shift_copy(const Grid& G, double* f, double* f2, const double* mean_num,
                              double inv_volume, cudaStream_t s) {
  return launch_dep(k_shift_copy, copy_grid(G), dim3(kCopyZ, kCopyY), 0, s, G, f, f2, mean_num, inv_volume);
}

cudaError_t launch_add_correction(const Grid& G, double* u, const float* e, int periodic,
                                  cudaStream_t s) {
  dim3 block(32, 4, 1);
  dim3 grid((G.n2 + 31) / 32, (G.n1 + 3) / 4, G.n0);
  return launch_dep(k_add_correction, grid, block, 0, s, G, u, e, periodic);
}

cudaError_t launch_sub_mean(double* p, long long n, const double* sum, double scale,
                            cudaStream_t s, double add) {
  if (n <= 0) return cudaSuccess;
  return launch_dep(k_sub_mean, blocks_for(n, 256), 256, 0, s, p, n, sum, scale, add);
}

cudaError_t launch_fill(double* p, long long n, double v, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  return launch_dep(k_fill, blocks_for(n, 256), 256, 0, s, p, n, v);
}

template <typename OP, bool DENSE>
static cudaError_t launch_hessian(int order, const Grid& G, const double* phi, double invh2,
                                  double* out, cudaStream_t s) {
  const dim3 tg = tile_grid(G);
  switch (order) {
    case 2: return launch_dep(k_hessian_tile<2, OP, DENSE>, tg, kTileThreads, FxTile<2>::bytes, s, G, phi, invh2, out);
    case 4: return launch_dep(k_hessian_tile<4, OP, DENSE>, tg, kTileThreads, FxTile<4>::bytes, s, G, phi, invh2, out);
    case 6: {
      // opted in here as well: callers without a hierarchy (mg_static.cu)
      const cudaError_t e =
          cudaFuncSetAttribute(k_hessian_tile<6, OP, DENSE>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, FxTile<6>::bytes);
      if (e != cudaSuccess) return e;
      return launch_dep(k_hessian_tile<6, OP, DENSE>, tg, kTileThreads, FxTile<6>::bytes, s, G, phi, invh2, out);
    }
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_lpt2_source(int order, const Grid& G, const double* phi, double invh2,
                               double* tau, cudaStream_t s) {
  return launch_hessian<TauOp, false>(order, G, phi, invh2, tau, s);
}

bool lpt2_source_dense_usable(const Grid& G, const double* phi, const double* tau) {
  const size_t a = reinterpret_cast<size_t>(phi), b = reinterpret_cast<size_t>(tau);
  const size_t bytes = (size_t)G.n0 * G.n1 * G.n2 * sizeof(double);
  return G.n2 % 2 == 0 && a % 16 == 0 && (a + bytes <= b || b + bytes <= a);
}

cudaError_t launch_lpt2_source_dense(int order, const Grid& G, const double* phi, double invh2,
                                     double* tau, cudaStream_t s) {
  return launch_hessian<TauOp, true>(order, G, phi, invh2, tau, s);
}

cudaError_t launch_lpt2_source_fp64(int order, const Grid& G, const double* phi, double invh2,
                                    double* tau, double* work, cudaStream_t s) {
  double* dy = work;
  double* dz = work + grid_elems(G);
  const dim3 block(32, 4, 1);
  const dim3 gpad((G.n2 + 2 * G.g + 31) / 32, (G.n1 + 2 * G.g + 3) / 4, G.n0 + 2 * G.g);
  const dim3 gin((G.n2 + 31) / 32, (G.n1 + 3) / 4, G.n0);
  cudaError_t e = cudaErrorInvalidValue;
  switch (order) {
    case 2:
      e = launch_dep(k_first_derivs<2>, gpad, block, 0, s, G, phi, dy, dz);
      return e != cudaSuccess ? e : launch_dep(k_lpt2_source<2>, gin, block, 0, s, G, phi, dy, dz, invh2, tau);
    case 4:
      e = launch_dep(k_first_derivs<4>, gpad, block, 0, s, G, phi, dy, dz);
      return e != cudaSuccess ? e : launch_dep(k_lpt2_source<4>, gin, block, 0, s, G, phi, dy, dz, invh2, tau);
    case 6:
      e = launch_dep(k_first_derivs<6>, gpad, block, 0, s, G, phi, dy, dz);
      return e != cudaSuccess ? e : launch_dep(k_lpt2_source<6>, gin, block, 0, s, G, phi, dy, dz, invh2, tau);
    default: return e;
  }
}

cudaError_t launch_lla(int order, const Grid& G, const double* phi, double invh2, double* out,
                       cudaStream_t s) {
  return launch_hessian<LlaOp, false>(order, G, phi, invh2, out, s);
}

cudaError_t launch_lla_dense(int order, const Grid& G, const double* phi, double invh2,
                             double* out, cudaStream_t s) {
  return launch_hessian<LlaOp, true>(order, G, phi, invh2, out, s);
}

cudaError_t launch_axpby(long long n, double a1, const double* x1, double a2, const double* x2,
                         double* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_axpby<<<blocks_for(n, 256), 256, 0, s>>>(n, a1, x1, a2, x2, out);
  return cudaGetLastError();
}

cudaError_t launch_gradient(int order, const Grid& G, const double* phi, double invh, double* dx,
                            double* dy, double* dz, cudaStream_t s) {
  if (tile_pays(G)) {
    const dim3 tg = tile_grid(G);
    switch (order) {
      case 2: return launch_dep(k_gradient_tile<2>, tg, kTileThreads, FxTile<2>::bytes, s, G, phi, invh, dx, dy, dz);
      case 4: return launch_dep(k_gradient_tile<4>, tg, kTileThreads, FxTile<4>::bytes, s, G, phi, invh, dx, dy, dz);
      case 6: return launch_dep(k_gradient_tile<6>, tg, kTileThreads, FxTile<6>::bytes, s, G, phi, invh, dx, dy, dz);
      default: return cudaErrorInvalidValue;
    }
  }
  const dim3 b((G.n2 + 31) / 32, (G.n1 + 3) / 4, G.n0), th(32, 4);
  switch (order) {
    case 2: return launch_dep(k_gradient<2>, b, th, 0, s, G, phi, invh, dx, dy, dz);
    case 4: return launch_dep(k_gradient<4>, b, th, 0, s, G, phi, invh, dx, dy, dz);
    case 6: return launch_dep(k_gradient<6>, b, th, 0, s, G, phi, invh, dx, dy, dz);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mgk
