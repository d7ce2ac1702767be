// Red-black Gauss-Seidel half-sweeps, residual + restriction, FAS source and
// prolongation-correction (Hahn & Abel 2011, Sec. 3.2 steps 2-9; Sec. 3.3).
//
// Smoother: one colour c = (i+j+k) mod 2 per launch.  Every cell of colour c
// takes the value that solves its own row of L u = f with all other values
// fixed at their pre-half-sweep values ("colour-Jacobi"; exact red-black GS for
// the 7-point stencil; for 13/19 points same-colour cells at distance 2 couple
// and this fixes their order).  The kernel reads buffer `uin` and writes every
// interior cell of `uout` (colour c updated, the other colour copied), so no
// thread ever reads a value another thread of the same launch writes.  k_smooth_faces is the
// half-sweep of a small nest with the coarse-fine ghosts of its result, k_smooth_fas the
// float32 half-sweep after a restriction with the FAS source.
#include "mg_internal.h"
#include "mg_launch.cuh"
#include "mg_stencil.cuh"
#include "mg_tile.cuh"
#include "mg_vbody.cuh"

namespace mgk {

namespace {

constexpr int kPairX = kVPairX;  // z-pairs per block row; blockDim.y = rows (1..8)
// At least 5 blocks of up to 256 threads per SM: caps the smoother at 48 registers
// (80 unbounded).  Measured on GB300 in CUDA graphs: float32 half-sweeps 15-20%
// faster at 128^3 (more warps in flight for the L1-bound loads).  float64 at order 6 holds
// its 18 neighbours while their largest exponent is found (mg_fixed.cuh) and spills at 48
// registers: 4 blocks give 17.6 us per 128^3 half-sweep, 5 blocks 21.9, 3 blocks 19.1; at
// order 4, 5 blocks give 12.8, 4 blocks 13.6.
template <int ORDER, typename T>
constexpr int smooth_min_blocks = sizeof(T) == 8 && ORDER == 6 ? 4 : 5;

template <int ORDER, typename T, bool CVT>
__global__ void __launch_bounds__(kPairX * 8, (smooth_min_blocks<ORDER, T>))
    k_smooth_half(Grid G, const T* uin, T* __restrict__ uout,
                  const T* f, T a_f, int colour, int periodic) {
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k0 = 2 * (blockIdx.x * kPairX + threadIdx.x);
  if (j >= G.n1 || k0 >= G.n2) return;
  grid_wait();
  smooth_pair_at<ORDER, T, CVT>(G, uin, uout, f, a_f, colour, periodic, blockIdx.z, j, k0);
}

// The first half-sweep of a level after a restriction into it, with the FAS source of the
// restricted cells (smooth_fas_pair_at): one launch instead of two.
template <int ORDER>
__global__ void __launch_bounds__(128, 8)
    k_smooth_fas(Grid G, const float* uin, float* __restrict__ uout,
                 float* f, float a_f, float invh2, FasBox box, int colour,
                 int periodic) {
  const int j = blockIdx.y * 4 + threadIdx.y;
  const int k0 = 2 * (blockIdx.x * 32 + threadIdx.x);
  if (j >= G.n1 || k0 >= G.n2) return;
  grid_wait();
  smooth_fas_pair_at<ORDER, float>(G, uin, uout, f, a_f, invh2, box, colour, periodic,
                                        blockIdx.z, j, k0);
}

// float32 rows whose length is a multiple of 4: one z-quad per thread (elements k0 ..
// k0 + 3, 16-byte aligned: the first interior element of a row sits at index 4 and the
// row pitch is a multiple of 8), updating the quad's two cells of colour c.  Every
// neighbour row along x and y is one 16-byte load serving both updates, and the z
// window k0 - 4 .. k0 + 7 three more; the two cells' sums and updates are those of
// smooth_half_body term by term, so the result is bit-identical to it.  The colour
// offset (0 or 1) is a run-time value shared by a row: it picks operands by select,
// never by a dynamic index into a register array.
__device__ __forceinline__ float4 ld4(const float* p) {
  return *reinterpret_cast<const float4*>(p);
}

template <int ORDER>
__device__ __forceinline__ void smooth_quad_at(const Grid& G, const float* uin,
                                               float* uout,
                                               const float* f, float a_f, int colour,
                                               int periodic, int i, int j, int k0) {
  constexpr int R = ORDER / 2;
  const long long sy = G.Zp;
  const long long sx = (long long)G.Y * G.Zp;
  const long long p0 = gidx(G, i, j, k0);
  // the quad's cells of colour c are k0 + o and k0 + o + 2
  const bool o = ((i + j) & 1) != colour;
  const float4 c = ld4(uin + p0);
  float w[12];  // z window: elements k0 - 4 .. k0 + 7
  {
    const float4 a = ld4(uin + p0 - 4), b = ld4(uin + p0 + 4);
    w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
    w[4] = c.x; w[5] = c.y; w[6] = c.z; w[7] = c.w;
    w[8] = b.x; w[9] = b.y; w[10] = b.z; w[11] = b.w;
  }
  // x and y neighbours at distance d of the two updated cells: [cell][d - 1]
  float xm[2][R], xp[2][R], ym[2][R], yp[2][R];
#pragma unroll
  for (int d = 1; d <= R; ++d) {
    const float4 a = ld4(uin + p0 - d * sx), b = ld4(uin + p0 + d * sx);
    const float4 e = ld4(uin + p0 - d * sy), g = ld4(uin + p0 + d * sy);
    xm[0][d - 1] = o ? a.y : a.x; xm[1][d - 1] = o ? a.w : a.z;
    xp[0][d - 1] = o ? b.y : b.x; xp[1][d - 1] = o ? b.w : b.z;
    ym[0][d - 1] = o ? e.y : e.x; ym[1][d - 1] = o ? e.w : e.z;
    yp[0][d - 1] = o ? g.y : g.x; yp[1][d - 1] = o ? g.w : g.z;
  }
  const float4 fv = ld4(f + p0);
  const float fc[2] = {o ? fv.y : fv.x, o ? fv.w : fv.z};
  constexpr double wc = 3.0 * Lap<ORDER>::w0;
  float v[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    // z neighbour at offset q of cell k0 + 2h + o: window index 4 + 2h + o + q
#define MGK_ZN(q) (o ? w[5 + 2 * h + (q)] : w[4 + 2 * h + (q)])
    const float s1 = (MGK_ZN(-1) + MGK_ZN(1)) + (ym[h][0] + yp[h][0]) + (xm[h][0] + xp[h][0]);
    float r = a_f * fc[h];
    r = fmaf(float(-Lap<ORDER>::w1 / wc), s1, r);
    if constexpr (ORDER >= 4) {
      const float s2 = (MGK_ZN(-2) + MGK_ZN(2)) + (ym[h][1] + yp[h][1]) + (xm[h][1] + xp[h][1]);
      r = fmaf(float(-Lap<ORDER>::w2 / wc), s2, r);
    }
    if constexpr (ORDER >= 6) {
      const float s3 = (MGK_ZN(-3) + MGK_ZN(3)) + (ym[h][2] + yp[h][2]) + (xm[h][2] + xp[h][2]);
      r = fmaf(float(-Lap<ORDER>::w3 / wc), s3, r);
    }
#undef MGK_ZN
    v[h] = r;
  }
  float4 out = c;
  if (o) {
    out.y = v[0];
    out.w = v[1];
  } else {
    out.x = v[0];
    out.z = v[1];
  }
  *reinterpret_cast<float4*>(uout + p0) = out;
  if (periodic) {
    write_pair_images<float>(G, uout, i, j, k0, out.x, out.y);
    write_pair_images<float>(G, uout, i, j, k0 + 2, out.z, out.w);
  }
}

template <int ORDER>
__global__ void __launch_bounds__(256, 4)
    k_smooth_quad(Grid G, const float* uin, float* __restrict__ uout,
                  const float* f, float a_f, int colour, int periodic) {
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (j >= G.n1 || k0 >= G.n2) return;
  grid_wait();
  smooth_quad_at<ORDER>(G, uin, uout, f, a_f, colour, periodic, blockIdx.z, j, k0);
}

// ---- half-sweep of a nest with its ghosts ----------------------------------------------
// The half-sweep of a nest and the coarse-fine ghosts of its result, which the next
// half-sweep or the residual reads, in one launch instead of two dependent ones.  The first
// face_blocks blocks work on 32 fine face columns each: of the ORDER cells nearest the face
// that a column's ghosts depend on, ORDER / 2 have the colour and are updated from uin once
// more, one warp per depth, and one warp writes the ghosts from the block's values in shared
// memory; the other blocks are those of the plain half-sweep.  No block reads what another
// writes, and every value is the same chain of operations as in the separate kernels.  The
// repeated updates cost 18 / n of a half-sweep's for order 6 and n^3 cells; the launch that
// goes away is nearly all latency on small levels (kFaceFusedMaxCells).
constexpr int kFacesThreads = 128;

// FAS (VEC = 2): the plain part is smooth_fas_pair_at, whose cells with a new f lie deeper
// than the face columns.
template <int ORDER, typename T, int VEC, bool FAS>
__global__ void __launch_bounds__(kFacesThreads,
                                  FAS ? 5 : ((smooth_min_blocks<ORDER, T>) < 5 || VEC == 4 ? 8 : 10))
    k_smooth_faces(Grid G, const T* uin, T* uout, T* f, T a_f, int colour,
                   int face_blocks, int gx, int gy, int qx, int by, T invh2, FasBox box,
                   FaceArgs<T> fa) {
  const int b = (int)blockIdx.x - face_blocks;
  if (b >= 0) {
    const int ty = (int)threadIdx.x / qx, tx = (int)threadIdx.x - ty * qx;
    const int j = b / gx % gy * by + ty;
    const int k0 = VEC * (b % gx * qx + tx);
    if (ty >= by || j >= G.n1 || k0 >= G.n2) return;
    grid_wait();
    if constexpr (FAS)
      smooth_fas_pair_at<ORDER, T>(G, uin, uout, f, a_f, invh2, box, colour, 0,
                                               b / (gx * gy), j, k0);
    else if constexpr (VEC == 4)
      smooth_quad_at<ORDER>(G, uin, uout, f, a_f, colour, 0, b / (gx * gy), j, k0);
    else
      smooth_pair_at<ORDER, T>(G, uin, uout, f, a_f, colour, 0, b / (gx * gy), j, k0);
    return;
  }
  __shared__ T cells[ORDER][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t = (int)blockIdx.x * 32 + lane;
  const bool in = t < 4 * (int)fa.fs.ebase[6];  // whole groups of 4, an element's columns
  FaceCol c;
  if (in) {
    const int e = t >> 2;
    const int fc = face_of(fa.fs, e, fa.fs.ebase);
    const unsigned loc = (unsigned)(e - (int)fa.fs.ebase[fc]), ne1 = fa.fs.nt[fc][1] / 2;
    c = face_col(G, fc, (int)(loc / ne1), (int)(loc % ne1), t & 3);
    // the cells at depths o, o + 2, .. have the colour (index along the normal: 0 or n - 1)
    const int na = (fc >> 1) == 0 ? G.n0 : ((fc >> 1) == 1 ? G.n1 : G.n2);
    const int o = ((((fc & 1) ? na - 1 : 0) + c.tj + c.tk) & 1) == colour ? 0 : 1;
    grid_wait();
    if (warp < ORDER / 2) {
      const int q = 2 * warp + o;
      const long long p = c.in0 + q * c.step;
      T nb[3 * ORDER];
      load_neighbours<ORDER, T>(uin, p, G.Zp, G.Y * G.Zp, nb);
      cells[q][lane] = relax<ORDER, T>(nb, a_f * f[p]);
    } else if (warp == kFacesThreads / 32 - 1) {
#pragma unroll
      for (int q = 0; q < ORDER / 2; ++q)
        cells[2 * q + 1 - o][lane] = uin[c.in0 + (2 * q + 1 - o) * c.step];
    }
  }
  __syncthreads();
  if (warp != 0 || !in) return;
  T v[ORDER];
#pragma unroll
  for (int q = 0; q < ORDER; ++q) v[q] = cells[q][lane];
  fa.template ghosts<ORDER>(uout, c, v, 0xfu << (lane & 28));
}

// r = f - L u at the 8 children of every covered parent cell; parent u := mean(u), ubar :=
// mean(u), parent f_fas := mean(r) (L ubar added later).  Four threads per parent (threadIdx.y:
// the child's x and y offset), each with the z-pair of children there: every neighbour row
// is one 2-element load for two children (17 loads instead of 38 at order 6), and a small
// level has four times the threads in flight of one thread per parent.  The sums run over
// the children in residual_restrict_body's order.  Blocks of lz x 4 x (32 / lz), lz lanes
// along z.
template <int ORDER, typename T>
__global__ void __launch_bounds__(128)
    k_residual_restrict(Grid F, const T* u, const T* f, T invh2, Grid P,
                        T* __restrict__ pu, T* __restrict__ pfas, T* __restrict__ ubar, Int3 off,
                        Int3 cn, int parent_periodic) {
  typedef typename Vec2<T>::type V2;
  __shared__ T sm[2][8][32];  // u and r by child and parent of the block
  const int kc = blockIdx.x * blockDim.x + threadIdx.x;
  const int jc = blockIdx.y * blockDim.z + threadIdx.z;
  const int ic = blockIdx.z;
  const int child = threadIdx.y, slot = threadIdx.z * blockDim.x + threadIdx.x;
  const bool in = kc < cn.z && jc < cn.y;
  grid_wait();
  if (in) {
    const long long p = gidx(F, 2 * ic + (child >> 1), 2 * jc + (child & 1), 2 * kc);
    T n0[3 * ORDER], n1[3 * ORDER], c0, c1;
    load_pair_neighbours<ORDER, T>(u, p, F.Zp, F.Y * F.Zp, n0, n1, c0, c1);
    const V2 fv = *reinterpret_cast<const V2*>(f + p);
    sm[0][2 * child][slot] = c0;
    sm[0][2 * child + 1][slot] = c1;
    sm[1][2 * child][slot] = add_lap_of<ORDER, T>(n0, c0, -invh2, fv.x);
    sm[1][2 * child + 1][slot] = add_lap_of<ORDER, T>(n1, c1, -invh2, fv.y);
  }
  __syncthreads();
  if (!in || child > 1) return;
  T s = T(0);
#pragma unroll
  for (int q = 0; q < 8; ++q) s += sm[child][q][slot];
  s *= T(0.125);
  const long long q = gidx(P, off.x + ic, off.y + jc, off.z + kc);
  if (child == 0) {
    pu[q] = s;
    if (parent_periodic) write_images<T>(P, pu, off.x + ic, off.y + jc, off.z + kc, s);
    ubar[((long long)ic * cn.y + jc) * cn.z + kc] = s;
  } else {
    pfas[q] = s;
  }
}

// The same on tiles of aligned integers (mg_tile.cuh), float64: the mean of a parent's 8
// children and of their T are integer sums (every T shifted by 3 first, so that the sum cannot
// overflow: up to 8 more units lost of a mean's 20, mg_tile.cuh), leaving about 12 FP64 instructions per
// parent cell, 7 of them the sum of f.  A thread holds 2 x 1 x 2 children of two parents;
// the row above or below is in the other half of its warp.
template <int ORDER>
__global__ void __launch_bounds__(kTileThreads, 3)
    k_residual_restrict_tile(Grid F, const double* u, const double* f,
                             double invh2, Grid P, double* __restrict__ pu,
                             double* __restrict__ pfas, double* __restrict__ ubar, Int3 off, Int3 cn,
                             int parent_periodic) {
  grid_wait();
  extern __shared__ __align__(16) long long tile_smem[];
  const int i0 = blockIdx.z * kTileX, j0 = blockIdx.y * kTileY, k0 = blockIdx.x * kTileZ;
  const unsigned key = tile_load<ORDER>(F, u, i0, j0, k0, tile_smem);
  const TilePos t = tile_pos();
  const int i = i0 + 4 * t.xh, j = j0 + t.y, k = k0 + 2 * t.zz;
  const long long p = gidx(F, i, j, k);
  const int sx = F.Y * F.Zp;
  const bool row = j < F.n1 && k < F.n2;
  const double kr = -invh2 * FxUnit<ORDER>::v;
  double mu[2] = {0.0, 0.0}, mr[2] = {0.0, 0.0};  // sums over the two planes of a parent
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (!(row && i + q < F.n0)) continue;
    const double2 fv = *reinterpret_cast<const double2*>(f + p + q * sx);
    mr[q >> 1] += fv.x + fv.y;
  }
  if (fx_in_range(key) && fx_scalable(kr, key)) {
    long long su[2] = {0, 0}, st[2] = {0, 0};
    tile_laplacians<ORDER>(tile_smem, [&](int q, longlong2 T, longlong2 c) {
      su[q >> 1] += c.x + c.y;
      st[q >> 1] += (T.x >> 3) + (T.y >> 3);
    });
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      mr[a] += __shfl_xor_sync(~0u, mr[a], 16);
      su[a] += __shfl_xor_sync(~0u, su[a], 16);
      st[a] += __shfl_xor_sync(~0u, st[a], 16);
      mr[a] = fma(fx_scale(kr, key), (double)st[a], 0.125 * mr[a]);
      mu[a] = fx_scale(0.125, key) * (double)su[a];
    }
  } else {
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
      if (!(row && i + q < F.n0)) continue;
      for (int dk = 0; dk < 2; ++dk) {
        const double c = u[p + q * sx + dk];
        const double r =
            add_lap_h2<ORDER, double, false>(u, p + q * sx + dk, F.Zp, sx, c, -invh2, 0.0);
        if (q < 2) {
          mu[0] += c;
          mr[0] += r;
        } else {
          mu[1] += c;
          mr[1] += r;
        }
      }
    }
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      mr[a] = 0.125 * (mr[a] + __shfl_xor_sync(~0u, mr[a], 16));
      mu[a] = 0.125 * (mu[a] + __shfl_xor_sync(~0u, mu[a], 16));
    }
  }
  // the lower row's thread writes the first parent, the upper row's the second
  const int a = t.y & 1;
  const int ic = (i >> 1) + a, jc = j >> 1, kc = k >> 1;
  if (!row || i + 2 * a >= F.n0) return;
  const double vu = a ? mu[1] : mu[0];
  const long long q = gidx(P, off.x + ic, off.y + jc, off.z + kc);
  pu[q] = vu;
  if (parent_periodic) write_images<double>(P, pu, off.x + ic, off.y + jc, off.z + kc, vu);
  pfas[q] = a ? mr[1] : mr[0];
  ubar[((long long)ic * cn.y + jc) * cn.z + kc] = vu;
}

// Covered parent cells: f_fas += L u (u = restricted fine solution there).
template <int ORDER, typename T>
__global__ void __launch_bounds__(128)
    k_fas_source(Grid P, const T* pu, T* pfas, T invH2, Int3 off,
                 Int3 cn) {
  grid_wait();
  fas_source_body<ORDER, T>(P, pu, pfas, invH2, off, cn,
                                 Blk{(int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z,
                                     (int)threadIdx.x, (int)threadIdx.y});
}

// u += inject(parent u - ubar) on the fine interior; one thread per z-pair.
template <typename T>
__global__ void __launch_bounds__(128)
    k_prolong(Grid F, T* u, Grid P, const T* pu,
              const T* ubar, Int3 off, Int3 cn, int periodic) {
  grid_wait();
  prolong_body<T>(F, u, P, pu, ubar, off, cn, periodic,
                       Blk{(int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z, (int)threadIdx.x,
                           (int)threadIdx.y});
}

// parent u := mean of children (covered region), one thread per parent cell.
template <typename T>
__global__ void __launch_bounds__(128)
    k_restrict_u(Grid F, const T* u, Grid P, T* __restrict__ pu, Int3 off, Int3 cn) {
  grid_wait();
  const int kc = blockIdx.x * blockDim.x + threadIdx.x;
  const int jc = blockIdx.y * blockDim.y + threadIdx.y;
  const int ic = blockIdx.z;
  if (kc >= cn.z || jc >= cn.y) return;
  T s = T(0);
#pragma unroll
  for (int di = 0; di < 2; ++di)
#pragma unroll
    for (int dj = 0; dj < 2; ++dj) {
      typedef typename Vec2<T>::type V2;
      const V2 v = *reinterpret_cast<const V2*>(u + gidx(F, 2 * ic + di, 2 * jc + dj, 2 * kc));
      s += v.x + v.y;
    }
  pu[gidx(P, off.x + ic, off.y + jc, off.z + kc)] = s * T(0.125);
}

dim3 coarse_grid(Int3 cn, dim3 block) {
  return dim3((cn.z + block.x - 1) / block.x, (cn.y + block.y - 1) / block.y, cn.x);
}

}  // namespace

// The z-quad kernel: as many threads per block as the pair kernel's (32 x rows), the
// block's x extent the row's quads up to 32.
cudaError_t launch_smooth_quad(int order, const Grid& G, const float* uin, float* uout,
                               const float* f, double a_f, int colour, int periodic, int rows,
                               cudaStream_t s) {
  const int quads = G.n2 / 4;
  const int qx = quads < 32 ? quads : 32;
  int by = 32 * rows / qx;
  if (by > G.n1) by = G.n1;
  dim3 block(qx, by, 1);
  dim3 grid((quads + qx - 1) / qx, (G.n1 + by - 1) / by, G.n0);
  switch (order) {
    case 2: return launch_dep(k_smooth_quad<2>, grid, block, 0, s, G, uin, uout, f, float(a_f), colour, periodic);
    case 4: return launch_dep(k_smooth_quad<4>, grid, block, 0, s, G, uin, uout, f, float(a_f), colour, periodic);
    case 6: return launch_dep(k_smooth_quad<6>, grid, block, 0, s, G, uin, uout, f, float(a_f), colour, periodic);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
cudaError_t launch_smooth_half(int order, const Grid& G, const T* uin, T* uout, const T* f,
                               double a_f, int colour, int periodic, int rows, bool quad,
                               cudaStream_t s) {
  if (rows < 1 || rows > 8) return cudaErrorInvalidValue;
  if constexpr (sizeof(T) == 4) {
    if (quad && G.n2 % 4 == 0 && G.n2 > 0 && G.n1 > 0)
      return launch_smooth_quad(order, G, uin, uout, f, a_f, colour, periodic, rows, s);
  }
  dim3 block(kPairX, rows, 1);
  const int pairs = (G.n2 + 1) / 2;
  dim3 grid((pairs + kPairX - 1) / kPairX, (G.n1 + rows - 1) / rows, G.n0);
  switch (order) {
    case 2: return launch_dep(k_smooth_half<2, T, false>, grid, block, 0, s, G, uin, uout, f, T(a_f), colour, periodic);
    case 4: return launch_dep(k_smooth_half<4, T, false>, grid, block, 0, s, G, uin, uout, f, T(a_f), colour, periodic);
    case 6:
      if constexpr (sizeof(T) == 8) {
        if ((long long)G.n0 * G.n1 * G.n2 > kFxCvtMinCells)
          return launch_dep(k_smooth_half<6, T, true>, grid, block, 0, s, G, uin, uout, f, T(a_f), colour, periodic);
      }
      return launch_dep(k_smooth_half<6, T, false>, grid, block, 0, s, G, uin, uout, f, T(a_f), colour, periodic);
    default: return cudaErrorInvalidValue;
  }
}

template <int ORDER, typename T, int VEC, bool FAS = false>
static cudaError_t launch_faces_vec(const Grid& G, const T* uin, T* uout, T* f, double a_f,
                                    int colour, double invh2, const FasBox& box,
                                    const FaceArgs<T>& fa, cudaStream_t s) {
  // blocks of qx groups of a row x by rows
  const int groups = (G.n2 + VEC - 1) / VEC;
  const int qx = groups < 32 ? groups : 32;
  const int by = kFacesThreads / qx < G.n1 ? kFacesThreads / qx : G.n1;
  const int gx = (groups + qx - 1) / qx, gy = (G.n1 + by - 1) / by;
  const int faces = (int)((4 * fa.fs.ebase[6] + 31) / 32);
  return launch_dep(k_smooth_faces<ORDER, T, VEC, FAS>, dim3(faces + gx * gy * G.n0), kFacesThreads,
                    0, s, G, uin, uout, f, T(a_f), colour, faces, gx, gy, qx, by, T(invh2), box, fa);
}

template <typename T>
cudaError_t launch_smooth_faces(int order, const Grid& G, const T* uin, T* uout, T* f, double a_f,
                                int colour, bool quad, const FaceSet& fs, const CfWeights& w,
                                const T* inter, const T* fc_unc, double h, double invH, bool fas,
                                double invh2, Int3 lo, Int3 hi, cudaStream_t s) {
  const FaceArgs<T> fa = make_face_args<T>(order, fs, w, inter, fc_unc, h, invH);
  const FasBox box{lo, hi};
  if constexpr (sizeof(T) == 4) {
    if (fas) {
      switch (order) {
        case 2: return launch_faces_vec<2, T, 2, true>(G, uin, uout, f, a_f, colour, invh2, box, fa, s);
        case 4: return launch_faces_vec<4, T, 2, true>(G, uin, uout, f, a_f, colour, invh2, box, fa, s);
        case 6: return launch_faces_vec<6, T, 2, true>(G, uin, uout, f, a_f, colour, invh2, box, fa, s);
        default: return cudaErrorInvalidValue;
      }
    }
    if (quad && G.n2 % 4 == 0) {
      switch (order) {
        case 2: return launch_faces_vec<2, T, 4>(G, uin, uout, f, a_f, colour, invh2, box, fa, s);
        case 4: return launch_faces_vec<4, T, 4>(G, uin, uout, f, a_f, colour, invh2, box, fa, s);
        case 6: return launch_faces_vec<6, T, 4>(G, uin, uout, f, a_f, colour, invh2, box, fa, s);
        default: return cudaErrorInvalidValue;
      }
    }
  }
  switch (order) {
    case 2: return launch_faces_vec<2, T, 2>(G, uin, uout, f, a_f, colour, invh2, box, fa, s);
    case 4: return launch_faces_vec<4, T, 2>(G, uin, uout, f, a_f, colour, invh2, box, fa, s);
    case 6: return launch_faces_vec<6, T, 2>(G, uin, uout, f, a_f, colour, invh2, box, fa, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_smooth_fas(int order, const Grid& G, const float* uin, float* uout, float* f,
                              double a_f, int colour, int periodic, double invh2, Int3 lo, Int3 hi,
                              cudaStream_t s) {
  if (G.n2 % 2) return cudaErrorInvalidValue;
  const dim3 block(32, 4, 1);
  const dim3 grid((G.n2 / 2 + 31) / 32, (G.n1 + 3) / 4, G.n0);
  const FasBox box{lo, hi};
  switch (order) {
    case 2: return launch_dep(k_smooth_fas<2>, grid, block, 0, s, G, uin, uout, f, float(a_f), float(invh2), box, colour, periodic);
    case 4: return launch_dep(k_smooth_fas<4>, grid, block, 0, s, G, uin, uout, f, float(a_f), float(invh2), box, colour, periodic);
    case 6: return launch_dep(k_smooth_fas<6>, grid, block, 0, s, G, uin, uout, f, float(a_f), float(invh2), box, colour, periodic);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
cudaError_t launch_residual_restrict(int order, const Grid& F, const T* u, const T* f,
                                     double invh2, const Grid& P, T* pu, T* pfas, T* ubar,
                                     Int3 off, Int3 cn, int parent_periodic, cudaStream_t s) {
  if constexpr (sizeof(T) == 8) {
    if (tile_pays(F)) {
      const dim3 tg = tile_grid(F);
      switch (order) {
        case 2: return launch_dep(k_residual_restrict_tile<2>, tg, kTileThreads, FxTile<2>::bytes, s, F, u, f, invh2, P, pu, pfas, ubar, off, cn, parent_periodic);
        case 4: return launch_dep(k_residual_restrict_tile<4>, tg, kTileThreads, FxTile<4>::bytes, s, F, u, f, invh2, P, pu, pfas, ubar, off, cn, parent_periodic);
        case 6: return launch_dep(k_residual_restrict_tile<6>, tg, kTileThreads, FxTile<6>::bytes, s, F, u, f, invh2, P, pu, pfas, ubar, off, cn, parent_periodic);
        default: return cudaErrorInvalidValue;
      }
    }
  }
  const int lz = cn.z > 16 ? 32 : (cn.z > 8 ? 16 : 8);
  const dim3 block(lz, 4, 32 / lz);
  const dim3 grid((cn.z + lz - 1) / lz, (cn.y + 32 / lz - 1) / (32 / lz), cn.x);
  switch (order) {
    case 2: return launch_dep(k_residual_restrict<2, T>, grid, block, 0, s, F, u, f, T(invh2), P, pu, pfas, ubar, off, cn, parent_periodic);
    case 4: return launch_dep(k_residual_restrict<4, T>, grid, block, 0, s, F, u, f, T(invh2), P, pu, pfas, ubar, off, cn, parent_periodic);
    case 6: return launch_dep(k_residual_restrict<6, T>, grid, block, 0, s, F, u, f, T(invh2), P, pu, pfas, ubar, off, cn, parent_periodic);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
cudaError_t launch_fas_source(int order, const Grid& P, const T* pu, T* pfas, double invH2,
                              Int3 off, Int3 cn, cudaStream_t s) {
  dim3 block(32, 4, 1);
  dim3 grid = coarse_grid(cn, block);
  switch (order) {
    case 2: return launch_dep(k_fas_source<2, T>, grid, block, 0, s, P, pu, pfas, T(invH2), off, cn);
    case 4: return launch_dep(k_fas_source<4, T>, grid, block, 0, s, P, pu, pfas, T(invH2), off, cn);
    case 6: return launch_dep(k_fas_source<6, T>, grid, block, 0, s, P, pu, pfas, T(invH2), off, cn);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
cudaError_t launch_prolong(const Grid& F, T* u, const Grid& P, const T* pu, const T* ubar,
                           Int3 off, Int3 cn, int periodic, cudaStream_t s) {
  dim3 block(32, 4, 1);
  const int pairs = F.n2 / 2;
  dim3 grid((pairs + 31) / 32, (F.n1 + 3) / 4, F.n0);
  return launch_dep(k_prolong<T>, grid, block, 0, s, F, u, P, pu, ubar, off, cn, periodic);
}

template <typename T>
cudaError_t launch_restrict_u(const Grid& F, const T* u, const Grid& P, T* pu, Int3 off, Int3 cn,
                              cudaStream_t s) {
  dim3 block(32, 4, 1);
  dim3 grid = coarse_grid(cn, block);
  return launch_dep(k_restrict_u<T>, grid, block, 0, s, F, u, P, pu, off, cn);
}

cudaError_t prepare_restrict_tile() {
  return cudaFuncSetAttribute(k_residual_restrict_tile<6>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, FxTile<6>::bytes);
}

#define MGK_INSTANTIATE(T)                                                                     \
  template cudaError_t launch_smooth_half<T>(int, const Grid&, const T*, T*, const T*, double, \
                                             int, int, int, bool, cudaStream_t);               \
  template cudaError_t launch_smooth_faces<T>(int, const Grid&, const T*, T*, T*, double, int, \
                                              bool, const FaceSet&, const CfWeights&,          \
                                              const T*, const T*, double, double, bool,        \
                                              double, Int3, Int3, cudaStream_t);               \
  template cudaError_t launch_residual_restrict<T>(int, const Grid&, const T*, const T*,       \
                                                   double, const Grid&, T*, T*, T*, Int3,      \
                                                   Int3, int, cudaStream_t);                   \
  template cudaError_t launch_fas_source<T>(int, const Grid&, const T*, T*, double, Int3,      \
                                            Int3, cudaStream_t);                               \
  template cudaError_t launch_prolong<T>(const Grid&, T*, const Grid&, const T*, const T*,     \
                                         Int3, Int3, int, cudaStream_t);                       \
  template cudaError_t launch_restrict_u<T>(const Grid&, const T*, const Grid&, T*, Int3,      \
                                            Int3, cudaStream_t);

MGK_INSTANTIATE(double)
MGK_INSTANTIATE(float)

}  // namespace mgk
