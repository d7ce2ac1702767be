// Ghost zones (Hahn & Abel 2011, Sec. 3.2 periodic boundaries; Sec. 3.3
// coarse-fine boundaries).
//
// Coarse-fine faces of a nest, in three steps (large nests and float64 leave the flux step
// its own launch; small ones run it with the half-sweep, k_smooth_faces in mg_smooth.cu):
//  * k_cf_tangential (once per parent state): for each face, each of the n/2
//    parent layers outside it and each fine tangential position, the degree-n
//    tensor Lagrange interpolant of the parent values parallel to the face
//    ("intermediate values"); and the part of the parent face flux (Table 2,
//    order n-1) that reads uncovered parent cells.
//  * k_cf_flux (before every half-sweep / residual): per parent face element,
//    the ghosts of its 4 fine columns from a degree-n polynomial normal to the
//    face through the n/2 intermediate values and n/2+1 fine interior values;
//    the parent flux with covered parent cells taken as the mean of their
//    current 8 children (two-way interface); the mean of the 4 fine fluxes;
//    and the difference added uniformly to the ghosts of each column so that
//    the fine fluxes average to the parent flux.  MG_FP64 folds everything linear into
//    per-layer weights and the interpolants (k_cf_flux_fold).
//  * k_cf_edges (before the 2LPT source only): edge and corner ghosts, which
//    only mixed derivatives read, by tensor degree-n interpolation of parent
//    values.
#include "mg_internal.h"
#include "mg_launch.cuh"
#include "mg_stencil.cuh"
#include "mg_vbody.cuh"

namespace mgk {

namespace {

template <typename T>
__global__ void __launch_bounds__(256) k_ghost_periodic(Grid G, T* u) {
  grid_wait();
  ghost_periodic_body<T>(G, u, blockIdx.x * (long long)blockDim.x + threadIdx.x);
}

// Parent face elements per block of the tangential kernel: kTangB along the face's first
// axis, kTangC along its second.
constexpr int kTangB = 8, kTangC = 16, kTangThreads = 256;

struct TangTiles {
  int nb[6], nc[6];  // tiles of every face along its axes
  int first[7];      // prefix sums of nb nc
};

TangTiles tang_tiles(const FaceSet& fs) {
  TangTiles t;
  t.first[0] = 0;
  for (int f = 0; f < 6; ++f) {
    t.nb[f] = (fs.nt[f][0] / 2 + kTangB - 1) / kTangB;
    t.nc[f] = (fs.nt[f][1] / 2 + kTangC - 1) / kTangC;
    t.first[f + 1] = t.first[f] + t.nb[f] * t.nc[f];
  }
  return t;
}

// Coarse parts of the folded flux step (k_cf_flux_fold): with fold, inter holds per ghost
// layer the parent values' part of the ghost, and fc_unc the parent values' part of the
// ghost shift.
struct TangFold {
  double ncoarse[3][3];
  double a[2];      // h / c_side
  double bg[2][3];  // b_side x the flux weight of ghost layer m
};

// Tangential interpolation of one tile of a face, all half layers: first each parent row
// (m, bb) of the tile is reduced along c for both parities (shared memory), then along b:
// a row serves the up to ORDER + 1 elements whose patch it is in, so an element of order 6
// costs 53 operations per layer (126 when every element reduces its own 7 rows).  Every
// value is the same chain of fmas either way.  FP64-bound in float64: 128^3 nest, order 6,
// cold, 23.2 us with an element per thread, 16.1 so, 19.5 with the folded coarse parts.
template <int ORDER, typename T, bool FOLD>
__device__ __forceinline__ void tangential_tile(const Grid& F, const Grid& P,
                                                const T* pu, Int3 off,
                                                const FaceSet& fs, const TangTiles& tt,
                                                const CfW<T>& w, const TangFold& fo, T invH,
                                                T* inter, T* fc_unc) {
  constexpr int half = ORDER / 2;
  constexpr int RB = kTangB + ORDER;
  typedef typename Vec2<T>::type V2;
  __shared__ V2 row[half][RB][kTangC];  // (parity 0, parity 1) along c
  int f = 0;
#pragma unroll
  for (int q = 1; q < 6; ++q)
    if ((int)blockIdx.x >= tt.first[q]) f = q;
  const int tile = (int)blockIdx.x - tt.first[f];
  const int jt = tile / tt.nc[f] * kTangB, kt = tile % tt.nc[f] * kTangC;
  const int a = f >> 1, side = f & 1;
  int b, c;
  face_axes(a, b, c);
  const int nt0 = fs.nt[f][0], nt1 = fs.nt[f][1];
  const int nb = min(kTangB, nt0 / 2 - jt), nc = min(kTangC, nt1 / 2 - kt);
  auto pick = [](int ax, int x, int y, int z) { return ax == 0 ? x : (ax == 1 ? y : z); };
  const int off_a = pick(a, off.x, off.y, off.z), nf_a = pick(a, F.n0, F.n1, F.n2);
  const int sxP = P.Y * P.Zp, syP = P.Zp;
  auto stride = [&](int ax) { return ax == 0 ? sxP : (ax == 1 ? syP : 1); };
  const int sa = stride(a), sb = stride(b), sc = stride(c);
  // parent cell (pface, b origin, c origin) of the tile; layers lie at pface -+ m
  const int p0a = side == 0 ? off_a - 1 : off_a + nf_a / 2;
  const int pb = pick(b, off.x, off.y, off.z) + jt, pc = pick(c, off.x, off.y, off.z) + kt;
  auto coord = [&](int ax, int va, int vb, int vc) { return ax == a ? va : (ax == b ? vb : vc); };
  const T* org = pu + gidx(P, coord(0, p0a, pb, pc), coord(1, p0a, pb, pc), coord(2, p0a, pb, pc));
  const int sm = side == 0 ? -sa : sa;
  const int rows = nb + ORDER;
  grid_wait();
  for (int q = threadIdx.x; q < half * RB * kTangC; q += kTangThreads) {
    const int kc = q % kTangC, r = q / kTangC % RB, m = q / (kTangC * RB);
    if (kc >= nc || r >= rows) continue;
    const T* v = org + (m * sm + (r - half) * sb + (kc - half) * sc);
    T r0 = T(0), r1 = T(0);
#pragma unroll
    for (int cc = 0; cc <= ORDER; ++cc) {
      const T x = v[cc * sc];
      r0 = fma(w.tang[0][cc], x, r0);
      r1 = fma(w.tang[1][cc], x, r1);
    }
    V2 o;
    o.x = r0;
    o.y = r1;
    row[m][r][kc] = o;
  }
  __syncthreads();
  if constexpr (!FOLD) {
    for (int q = threadIdx.x; q < half * kTangB * kTangC; q += kTangThreads) {
      const int kc = q % kTangC, jc = q / kTangC % kTangB, m = q / (kTangC * kTangB);
      if (kc >= nc || jc >= nb) continue;
#pragma unroll
      for (int pj = 0; pj < 2; ++pj) {
        V2 acc;
        acc.x = acc.y = T(0);
#pragma unroll
        for (int bb = 0; bb <= ORDER; ++bb) {
          const V2 r = row[m][jc + bb][kc];
          acc.x = fma(w.tang[pj][bb], r.x, acc.x);
          acc.y = fma(w.tang[pj][bb], r.y, acc.y);
        }
        // (tk, tk + 1) = (2 kc, 2 kc + 1): an even, hence 2-element aligned, pair
        const long long tj = 2 * (jt + jc) + pj;
        *reinterpret_cast<V2*>(inter + fs.base[f] + ((long long)m * nt0 + tj) * nt1 +
                               2 * (kt + kc)) = acc;
      }
    }
  }
  // with FOLD, the two fine rows pj of an element are neighbouring lanes
  constexpr int PJ = FOLD ? 2 : 1;
  static_assert(PJ * kTangB * kTangC % 32 == 0 && kTangThreads % 32 == 0, "whole warps");
  for (int q = threadIdx.x; q < PJ * kTangB * kTangC; q += kTangThreads) {
    const int pj = q % PJ, kc = q / PJ % kTangC, jc = q / (PJ * kTangC);
    const bool in = kc < nc && jc < nb;
    T fc = T(0);
    if (in) {
      // uncovered part of the parent face flux: parent cells outside the face, along a
      const T* v = org + (jc * sb + kc * sc);
      if (side == 0) {
#pragma unroll
        for (int s = 0; s < half; ++s) fc = fma(w.flux[s], v[(half - 1 - s) * sm], fc);
      } else {
#pragma unroll
        for (int s = half; s < ORDER; ++s) fc = fma(w.flux[s], v[(s - half) * sm], fc);
      }
      fc *= invH;
    }
    if constexpr (FOLD) {
      T sum = T(0);  // of b_side x the ghosts' coarse part of the fine fluxes of the columns
      if (in) {
        V2 t[half];
#pragma unroll
        for (int m = 0; m < half; ++m) {
          t[m].x = t[m].y = T(0);
#pragma unroll
          for (int bb = 0; bb <= ORDER; ++bb) {
            const V2 r = row[m][jc + bb][kc];
            t[m].x = fma(w.tang[pj][bb], r.x, t[m].x);
            t[m].y = fma(w.tang[pj][bb], r.y, t[m].y);
          }
        }
        const long long tj = 2 * (jt + jc) + pj;
#pragma unroll
        for (int m = 0; m < half; ++m) {
          V2 g;
          g.x = g.y = T(0);
#pragma unroll
          for (int n = 0; n < half; ++n) {
            g.x = fma(fo.ncoarse[m][n], t[n].x, g.x);
            g.y = fma(fo.ncoarse[m][n], t[n].y, g.y);
          }
          sum = fma(fo.bg[side][m], g.x + g.y, sum);
          *reinterpret_cast<V2*>(inter + fs.base[f] + ((long long)m * nt0 + tj) * nt1 +
                                 2 * (kt + kc)) = g;
        }
      }
      sum += __shfl_xor_sync(~0u, sum, 1);
      fc = fma(fc, fo.a[side], -sum);
    }
    if (in && pj == 0)
      fc_unc[fs.ebase[f] + (long long)(jt + jc) * (nt1 / 2) + kt + kc] = fc;
  }
}

template <int ORDER, typename T, bool FOLD>
__global__ void __launch_bounds__(kTangThreads)
    k_cf_tangential(Grid F, Grid P, const T* pu, Int3 off, FaceSet fs, TangTiles tt,
                    CfW<T> w, TangFold fo, T invH, T* inter,
                    T* fc_unc) {
  tangential_tile<ORDER, T, FOLD>(F, P, pu, off, fs, tt, w, fo, invH, inter, fc_unc);
}

// Tangential interpolation and prolongation of a nest, both from the parent's new values and
// independent of each other, in one launch: the tiles of the faces first, then blocks of 32
// z-pairs x 8 rows (gx x gy per plane).
template <int ORDER, typename T, bool FOLD>
__global__ void __launch_bounds__(kTangThreads)
    k_tangential_prolong(Grid F, Grid P, const T* pu, Int3 off, FaceSet fs,
                         TangTiles tt, CfW<T> w, TangFold fo, T invH, T* inter,
                         T* fc_unc, T* u, const T* ubar,
                         Int3 cn, int gx, int gy) {
  const int b = (int)blockIdx.x - tt.first[6];
  if (b < 0) {
    tangential_tile<ORDER, T, FOLD>(F, P, pu, off, fs, tt, w, fo, invH, inter, fc_unc);
    return;
  }
  grid_wait();
  prolong_at<T>(F, u, P, pu, ubar, off, cn, 0, b / (gx * gy),
                     b / gx % gy * (kTangThreads / 32) + (int)(threadIdx.x >> 5),
                     b % gx * 32 + (int)(threadIdx.x & 31));
}

template <int ORDER, typename T>
__global__ void __launch_bounds__(128)
    k_cf_flux(Grid F, T* u, FaceSet fs, CfW<T> w, const T* inter,
              const T* fc_unc, T fc_scale, T a0, T a1, T b0, T b1, int flux_fix) {
  const int t = blockIdx.x * 128 + threadIdx.x;
  if (t >= 4 * (int)fs.ebase[6]) return;
  const unsigned quad = __activemask();
  const int e = t >> 2;
  const int f = face_of(fs, e, fs.ebase);
  const unsigned loc = (unsigned)(e - (int)fs.ebase[f]), ne1 = fs.nt[f][1] / 2;
  const FaceCol c = face_col(F, f, (int)(loc / ne1), (int)(loc % ne1), t & 3);
  grid_wait();
  T v[ORDER];
  load_column<ORDER, T>(u, c, v);
  cf_flux_at<ORDER, T>(u, fs, w, inter, fc_unc, fc_scale, a0, a1, b0, b1, flux_fix, c, v, quad);
}

template <int ORDER>
__global__ void __launch_bounds__(128)
    k_cf_flux_fold(Grid F, double* u, FaceArgs<double> fa) {
  const int t = blockIdx.x * 128 + threadIdx.x;
  if (t >= 4 * (int)fa.fs.ebase[6]) return;
  const unsigned quad = __activemask();
  const int e = t >> 2;
  const int f = face_of(fa.fs, e, fa.fs.ebase);
  const unsigned loc = (unsigned)(e - (int)fa.fs.ebase[f]), ne1 = fa.fs.nt[f][1] / 2;
  const FaceCol c = face_col(F, f, (int)(loc / ne1), (int)(loc % ne1), t & 3);
  grid_wait();
  double v[ORDER];
  load_column<ORDER, double>(u, c, v);
  fa.ghosts<ORDER>(u, c, v, quad);
}

// Edge and corner ghosts of a level in a row: the edges along x, y and z, (2 g)^2 cells at
// every position along them, then the corners.
__host__ __device__ inline int edge_count(const Grid& F) {
  const int w = 2 * F.g;
  return w * w * (F.n0 + F.n1 + F.n2 + w);
}

__device__ __forceinline__ bool edge_cell(const Grid& F, int t, int& i, int& j, int& k) {
  const int g = F.g, w = 2 * g, ww = w * w;
  const int n[3] = {F.n0, F.n1, F.n2};
  auto ghost = [&](int q, int len) { return q < g ? q - g : len + q - g; };
  const int pos = t / ww, q = t % ww;
  const int a = q / w, b = q % w;
  if (pos < n[0]) {
    i = pos;
    j = ghost(a, n[1]);
    k = ghost(b, n[2]);
  } else if (pos < n[0] + n[1]) {
    i = ghost(a, n[0]);
    j = pos - n[0];
    k = ghost(b, n[2]);
  } else if (pos < n[0] + n[1] + n[2]) {
    i = ghost(a, n[0]);
    j = ghost(b, n[1]);
    k = pos - n[0] - n[1];
  } else {
    const int c = pos - n[0] - n[1] - n[2];
    if (c >= w) return false;
    i = ghost(c, n[0]);
    j = ghost(a, n[1]);
    k = ghost(b, n[2]);
  }
  return true;
}

template <int ORDER, typename T>
__global__ void __launch_bounds__(128)
    k_cf_edges(Grid F, T* u, Grid P, const T* pu, Int3 off,
               CfWeights w) {
  grid_wait();
  constexpr int half = ORDER / 2;
  int i, j, k;
  if (!edge_cell(F, blockIdx.x * 128 + (int)threadIdx.x, i, j, k)) return;
  const int pi = off.x + (i >> 1), pj = off.y + (j >> 1), pk = off.z + (k >> 1);
  const double* wi = w.tang[i & 1];
  const double* wj = w.tang[j & 1];
  const double* wk = w.tang[k & 1];
  T acc = T(0);
  for (int a = 0; a <= ORDER; ++a) {
    T pa = T(0);
    for (int bq = 0; bq <= ORDER; ++bq) {
      T row = T(0);
      for (int cq = 0; cq <= ORDER; ++cq)
        row = fma(T(wk[cq]), pu[gidx(P, pi + a - half, pj + bq - half, pk + cq - half)], row);
      pa = fma(T(wj[bq]), row, pa);
    }
    acc = fma(T(wi[a]), pa, acc);
  }
  u[gidx(F, i, j, k)] = acc;
}

}  // namespace

template <typename T>
cudaError_t launch_ghost_periodic(const Grid& G, T* u, cudaStream_t s) {
  const long long g = G.g;
  const long long X = G.n0 + 2 * g, Y = G.n1 + 2 * g;
  const long long total = X * Y * 2 * g + X * 2 * g * G.n2 + 2 * g * (long long)G.n1 * G.n2;
  const int block = 256;
  return launch_dep(k_ghost_periodic<T>, (unsigned)((total + block - 1) / block), block, 0, s, G, u);
}

template <int ORDER, typename T, bool FOLD>
static cudaError_t launch_tangential_as(const Grid& F, const Grid& P, const T* pu, Int3 off,
                                        const FaceSet& fs, const CfWeights& w, double h,
                                        double invH, T* inter, T* fc_unc, T* prolong_u,
                                        const T* ubar, Int3 cn, cudaStream_t s) {
  constexpr int half = ORDER / 2;
  const CfW<T> wt = cf_weights_as<T>(w);
  const TangTiles tt = tang_tiles(fs);
  TangFold fo{};
  if (FOLD) {
    for (int m = 0; m < half; ++m)
      for (int q = 0; q < half; ++q) fo.ncoarse[m][q] = w.ncoarse[m][q];
    for (int sd = 0; sd < 2; ++sd) {
      fo.a[sd] = h / w.ghost_coef[sd];
      for (int m = 0; m < half; ++m)
        fo.bg[sd][m] = 0.25 / w.ghost_coef[sd] * w.flux[sd == 0 ? half - 1 - m : half + m];
    }
  }
  if (!prolong_u)
    return launch_dep(k_cf_tangential<ORDER, T, FOLD>, tt.first[6], kTangThreads, 0, s, F, P, pu,
                      off, fs, tt, wt, fo, T(invH), inter, fc_unc);
  if constexpr (sizeof(T) == 4 || FOLD) {  // V-cycles run in float32, or in float64 folded
    const int gx = (F.n2 / 2 + 31) / 32, gy = (F.n1 + kTangThreads / 32 - 1) / (kTangThreads / 32);
    return launch_dep(k_tangential_prolong<ORDER, T, FOLD>, tt.first[6] + gx * gy * F.n0,
                      kTangThreads, 0, s, F, P, pu, off, fs, tt, wt, fo, T(invH), inter, fc_unc,
                      prolong_u, ubar, cn, gx, gy);
  }
  return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_cf_tangential(int order, const Grid& F, const Grid& P, const T* pu, Int3 off,
                                 const FaceSet& fs, const CfWeights& w, double h, double invH,
                                 bool fold, T* inter, T* fc_unc, cudaStream_t s, T* prolong_u,
                                 const T* ubar, Int3 cn) {
  if constexpr (sizeof(T) == 8) {
    if (fold) {
      switch (order) {
        case 2: return launch_tangential_as<2, T, true>(F, P, pu, off, fs, w, h, invH, inter, fc_unc, prolong_u, ubar, cn, s);
        case 4: return launch_tangential_as<4, T, true>(F, P, pu, off, fs, w, h, invH, inter, fc_unc, prolong_u, ubar, cn, s);
        case 6: return launch_tangential_as<6, T, true>(F, P, pu, off, fs, w, h, invH, inter, fc_unc, prolong_u, ubar, cn, s);
        default: return cudaErrorInvalidValue;
      }
    }
  }
  switch (order) {
    case 2: return launch_tangential_as<2, T, false>(F, P, pu, off, fs, w, h, invH, inter, fc_unc, prolong_u, ubar, cn, s);
    case 4: return launch_tangential_as<4, T, false>(F, P, pu, off, fs, w, h, invH, inter, fc_unc, prolong_u, ubar, cn, s);
    case 6: return launch_tangential_as<6, T, false>(F, P, pu, off, fs, w, h, invH, inter, fc_unc, prolong_u, ubar, cn, s);
    default: return cudaErrorInvalidValue;
  }
}

template <>
FaceArgs<double> make_face_args<double>(int order, const FaceSet& fs, const CfWeights& w,
                                        const double* inter, const double* fc_unc, double h,
                                        double invH) {
  const int half = order / 2;
  FaceArgs<double> o{};
  o.fs = fs;
  o.inter = inter;
  o.fc_unc = fc_unc;
  for (int m = 0; m < half; ++m)
    for (int q = 0; q <= half; ++q) o.w.nfine[m][q] = w.nfine[m][q];
  for (int sd = 0; sd < 2; ++sd) {
    const double c = w.ghost_coef[sd];
    for (int q = 0; q < 2 * half; ++q) {
      const int sp = sd == 0 ? half + q / 2 : half - 1 - q / 2;
      double fine = 0.0;  // of v_q in the fine flux, directly and through the ghosts
      if (q < half) fine += w.flux[sd == 0 ? half + q : half - 1 - q];
      if (q <= half)
        for (int m = 0; m < half; ++m)
          fine += w.flux[sd == 0 ? half - 1 - m : half + m] * w.nfine[m][q];
      o.w.d[sd][q] = (h / c) * (0.125 * invH) * w.flux[sp] - 0.25 / c * fine;
    }
  }
  return o;
}

template <>
FaceArgs<float> make_face_args<float>(int order, const FaceSet& fs, const CfWeights& w,
                                      const float* inter, const float* fc_unc, double h,
                                      double invH) {
  (void)order;
  const double invh = 1.0 / h;
  FaceArgs<float> o{};
  o.fs = fs;
  o.w = cf_weights_as<float>(w);
  o.inter = inter;
  o.fc_unc = fc_unc;
  o.fc_scale = float(0.125 * invH);
  o.a0 = float(h / w.ghost_coef[0]);
  o.a1 = float(h / w.ghost_coef[1]);
  o.b0 = float(0.25 * invh * h / w.ghost_coef[0]);
  o.b1 = float(0.25 * invh * h / w.ghost_coef[1]);
  return o;
}

cudaError_t launch_cf_flux_fold(int order, const Grid& F, double* u, const FaceSet& fs,
                                const CfWeights& w, const double* inter, const double* fc_unc,
                                double h, double invH, cudaStream_t s) {
  const FaceArgs<double> fa = make_face_args<double>(order, fs, w, inter, fc_unc, h, invH);
  const unsigned grid = (unsigned)((4 * fs.ebase[6] + 127) / 128);
  switch (order) {
    case 2: return launch_dep(k_cf_flux_fold<2>, grid, 128, 0, s, F, u, fa);
    case 4: return launch_dep(k_cf_flux_fold<4>, grid, 128, 0, s, F, u, fa);
    case 6: return launch_dep(k_cf_flux_fold<6>, grid, 128, 0, s, F, u, fa);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
cudaError_t launch_cf_flux(int order, const Grid& F, T* u, const FaceSet& fs, const CfWeights& w,
                           const T* inter, const T* fc_unc, double h, double invh, double invH,
                           int flux_fix, cudaStream_t s) {
  const int block = 128;
  const unsigned grid = (unsigned)((4 * fs.ebase[6] + block - 1) / block);
  const T fc_scale = T(0.125 * invH);
  const T a0 = T(h / w.ghost_coef[0]), a1 = T(h / w.ghost_coef[1]);
  const T b0 = T(0.25 * invh * h / w.ghost_coef[0]), b1 = T(0.25 * invh * h / w.ghost_coef[1]);
  const CfW<T> wt = cf_weights_as<T>(w);
  switch (order) {
    case 2: return launch_dep(k_cf_flux<2, T>, grid, block, 0, s, F, u, fs, wt, inter, fc_unc, fc_scale, a0, a1, b0, b1, flux_fix);
    case 4: return launch_dep(k_cf_flux<4, T>, grid, block, 0, s, F, u, fs, wt, inter, fc_unc, fc_scale, a0, a1, b0, b1, flux_fix);
    case 6: return launch_dep(k_cf_flux<6, T>, grid, block, 0, s, F, u, fs, wt, inter, fc_unc, fc_scale, a0, a1, b0, b1, flux_fix);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
cudaError_t launch_cf_edges(int order, const Grid& F, T* u, const Grid& P, const T* pu, Int3 off,
                            const CfWeights& w, cudaStream_t s) {
  const int block = 128;
  const unsigned grid = (unsigned)((edge_count(F) + block - 1) / block);
  switch (order) {
    case 2: return launch_dep(k_cf_edges<2, T>, grid, block, 0, s, F, u, P, pu, off, w);
    case 4: return launch_dep(k_cf_edges<4, T>, grid, block, 0, s, F, u, P, pu, off, w);
    case 6: return launch_dep(k_cf_edges<6, T>, grid, block, 0, s, F, u, P, pu, off, w);
    default: return cudaErrorInvalidValue;
  }
}

#define MGK_GHOST_INSTANTIATE(T)                                                              \
  template cudaError_t launch_ghost_periodic<T>(const Grid&, T*, cudaStream_t);               \
  template cudaError_t launch_cf_tangential<T>(int, const Grid&, const Grid&, const T*, Int3, \
                                               const FaceSet&, const CfWeights&, double,      \
                                               double, bool, T*, T*, cudaStream_t, T*,        \
                                               const T*, Int3);                               \
  template cudaError_t launch_cf_flux<T>(int, const Grid&, T*, const FaceSet&,                \
                                         const CfWeights&, const T*, const T*, double,        \
                                         double, double, int, cudaStream_t);                  \
  template cudaError_t launch_cf_edges<T>(int, const Grid&, T*, const Grid&, const T*, Int3,  \
                                          const CfWeights&, cudaStream_t);

MGK_GHOST_INSTANTIATE(double)
MGK_GHOST_INSTANTIATE(float)

}  // namespace mgk
