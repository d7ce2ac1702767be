// Bodies of the kernels of one float32/float64 V-cycle (Hahn & Abel 2011, Sec. 3.2
// steps 2-9; Sec. 3.3), run two ways: by stream kernels (block and thread indices from the
// hardware) and by the persistent batch kernel (mg_persist.cu), which runs any block of any
// level operation of any hierarchy as a work item of a 128-thread block.  Every body gets
// its block and thread indices as arguments and reads by plain loads: in the persistent kernel
// earlier items of the same launch wrote the data (ordered by release/acquire flags), in the
// stream kernels the predecessor that grid_wait waits for (mg_launch.cuh).  residual_restrict_body and
// cf_tangential_body serve the persistent kernel only: the stream kernels share a parent's
// or a tile's work between threads, with the operations of every value in the same order, so
// both ways give bit-identical results in float32, which is all the persistent kernel runs.
#pragma once

#include "mg_internal.h"
#include "mg_stencil.cuh"

namespace mgk {

// Block and thread indices of one block of a level operation.
struct Blk {
  int bx, by, bz;
  int tx, ty;
};

// Threads along z per block of the smoother and the transfer operations.
constexpr int kVPairX = 32;

// ---- smoother: one colour of red-black Gauss-Seidel, colour-Jacobi ----------------
// Every cell of colour c takes the value that solves its own row of L u = f with all
// other values fixed at their pre-half-sweep values.  Reads uin, writes every interior
// cell of uout (colour c updated, the other colour copied), one z-pair per thread;
// blocks of kVPairX x rows threads.
template <int ORDER, typename T, bool CVT = false>
__device__ __forceinline__ void smooth_pair_at(const Grid& G, const T* uin,
                                               T* uout, const T* f,
                                               T a_f, int colour, int periodic, int i, int j,
                                               int k0) {
  const int sy = G.Zp;
  const int sx = G.Y * G.Zp;
  const long long p0 = gidx(G, i, j, k0);
  const int upd = (((i + j + k0) & 1) == colour) ? 0 : 1;
  const bool pair = (k0 + 1) < G.n2;
  if (!pair && upd == 1) {
    const T c = uin[p0];
    uout[p0] = c;
    if (periodic) write_images<T>(G, uout, i, j, k0, c);
    return;
  }
  const long long p = p0 + upd;
  // u = (h^2 f - sum_off w u_nb) / w_centre
  T nb[3 * ORDER];
  load_neighbours<ORDER, T>(uin, p, sy, sx, nb);
  const T other = upd == 0 ? nb[1] : nb[0];  // the pair's cell of the other colour
  const T v = relax<ORDER, T, CVT>(nb, a_f * f[p]);
  if (pair) {
    typedef typename Vec2<T>::type V2;
    V2 out;
    out.x = upd == 0 ? v : other;
    out.y = upd == 0 ? other : v;
    *reinterpret_cast<V2*>(uout + p0) = out;
    if (periodic) write_pair_images<T>(G, uout, i, j, k0, out.x, out.y);
  } else {
    uout[p0] = v;
    if (periodic) write_images<T>(G, uout, i, j, k0, v);
  }
}

// FAS source of the cells [lo, hi) of a level and the level's first half-sweep after it: f of
// those cells (the restricted residual) gains L u of the restricted solution, whose neighbours
// the half-sweep reads anyway, before the pair's cell of the colour is updated.  Rows of even
// length (levels with a parent).
struct FasBox {
  Int3 lo, hi;
};

template <int ORDER, typename T>
__device__ __forceinline__ void smooth_fas_pair_at(const Grid& G, const T* uin,
                                                   T* uout, T* f,
                                                   T a_f, T invh2, const FasBox& box, int colour,
                                                   int periodic, int i, int j, int k0) {
  typedef typename Vec2<T>::type V2;
  const long long p = gidx(G, i, j, k0);
  T n0[3 * ORDER], n1[3 * ORDER], c0, c1;
  load_pair_neighbours<ORDER, T>(uin, p, G.Zp, G.Y * G.Zp, n0, n1, c0, c1);
  V2 fv = *reinterpret_cast<const V2*>(f + p);
  if (i >= box.lo.x && i < box.hi.x && j >= box.lo.y && j < box.hi.y) {
    const bool in0 = k0 >= box.lo.z && k0 < box.hi.z;
    const bool in1 = k0 + 1 >= box.lo.z && k0 + 1 < box.hi.z;
    if (in0) fv.x = add_lap_of<ORDER, T>(n0, c0, invh2, fv.x);
    if (in1) fv.y = add_lap_of<ORDER, T>(n1, c1, invh2, fv.y);
    if (in0 || in1) *reinterpret_cast<V2*>(f + p) = fv;
  }
  V2 out;
  out.x = c0;
  out.y = c1;
  if (((i + j + k0) & 1) == colour) out.x = relax<ORDER, T>(n0, a_f * fv.x);
  else out.y = relax<ORDER, T>(n1, a_f * fv.y);
  *reinterpret_cast<V2*>(uout + p) = out;
  if (periodic) write_pair_images<T>(G, uout, i, j, k0, out.x, out.y);
}

template <int ORDER, typename T, bool CVT = false>
__device__ __forceinline__ void smooth_half_body(const Grid& G, const T* uin,
                                                 T* uout, const T* f,
                                                 T a_f, int colour, int periodic, int rows, Blk b) {
  const int j = b.by * rows + b.ty;
  const int k0 = 2 * (b.bx * kVPairX + b.tx);
  if (j >= G.n1 || k0 >= G.n2) return;
  smooth_pair_at<ORDER, T, CVT>(G, uin, uout, f, a_f, colour, periodic, b.bz, j, k0);
}

// ---- residual + restriction: one thread per covered parent cell ---------------------
// r = f - L u at its 8 children; parent u := mean(u), ubar := mean(u), parent
// f_fas := mean(r) (L ubar is added by fas_source).  Blocks of 32 x 4 threads.
template <int ORDER, typename T>
__device__ __forceinline__ void residual_restrict_body(const Grid& F, const T* u,
                                                       const T* f, T invh2,
                                                       const Grid& P, T* pu,
                                                       T* pfas, T* ubar,
                                                       Int3 off, Int3 cn, int parent_periodic,
                                                       Blk b) {
  const int kc = b.bx * 32 + b.tx;
  const int jc = b.by * 4 + b.ty;
  const int ic = b.bz;
  if (kc >= cn.z || jc >= cn.y) return;
  const int sy = F.Zp;
  const int sx = F.Y * F.Zp;
  T su = T(0), sr = T(0);
#pragma unroll
  for (int di = 0; di < 2; ++di) {
#pragma unroll
    for (int dj = 0; dj < 2; ++dj) {
#pragma unroll
      for (int dk = 0; dk < 2; ++dk) {
        const long long p = gidx(F, 2 * ic + di, 2 * jc + dj, 2 * kc + dk);
        const T c = u[p];
        su += c;
        sr += add_lap_h2<ORDER, T>(u, p, sy, sx, c, -invh2, f[p]);
      }
    }
  }
  const long long q = gidx(P, off.x + ic, off.y + jc, off.z + kc);
  const T mu = su * T(0.125);
  pu[q] = mu;
  if (parent_periodic) write_images<T>(P, pu, off.x + ic, off.y + jc, off.z + kc, mu);
  pfas[q] = sr * T(0.125);
  ubar[((long long)ic * cn.y + jc) * cn.z + kc] = mu;
}

// ---- FAS source: covered parent cells f_fas += L u (u = restricted fine solution) ----
template <int ORDER, typename T>
__device__ __forceinline__ void fas_source_body(const Grid& P, const T* pu,
                                                T* pfas, T invH2, Int3 off, Int3 cn,
                                                Blk b) {
  const int kc = b.bx * 32 + b.tx;
  const int jc = b.by * 4 + b.ty;
  const int ic = b.bz;
  if (kc >= cn.z || jc >= cn.y) return;
  const long long q = gidx(P, off.x + ic, off.y + jc, off.z + kc);
  pfas[q] = add_lap_h2<ORDER, T>(pu, q, P.Zp, P.Y * P.Zp, pu[q], invH2, pfas[q]);
}

// ---- prolongation-correction: u += inject(parent u - ubar), one thread per z-pair ----
template <typename T>
__device__ __forceinline__ void prolong_at(const Grid& F, T* u, const Grid& P,
                                           const T* pu, const T* ubar,
                                           Int3 off, Int3 cn, int periodic, int i, int j, int t) {
  const int k0 = 2 * t;
  if (j >= F.n1 || k0 >= F.n2) return;
  const int ic = i >> 1, jc = j >> 1, kc = t;
  const T d = pu[gidx(P, off.x + ic, off.y + jc, off.z + kc)] -
              ubar[((long long)ic * cn.y + jc) * cn.z + kc];
  const long long p = gidx(F, i, j, k0);
  typedef typename Vec2<T>::type V2;
  V2 v = *reinterpret_cast<const V2*>(u + p);
  v.x += d;
  v.y += d;
  *reinterpret_cast<V2*>(u + p) = v;
  if (periodic) {
    if (k0 + 1 < F.n2) write_pair_images<T>(F, u, i, j, k0, v.x, v.y);
    else write_images<T>(F, u, i, j, k0, v.x);
  }
}

template <typename T>
__device__ __forceinline__ void prolong_body(const Grid& F, T* u, const Grid& P,
                                             const T* pu, const T* ubar,
                                             Int3 off, Int3 cn, int periodic, Blk b) {
  prolong_at<T>(F, u, P, pu, ubar, off, cn, periodic, b.bz, b.by * 4 + b.ty, b.bx * 32 + b.tx);
}

// ---- periodic ghost shell: element t of the shell takes its interior image ----------
// (ghost_shell_count(G) elements, mg_internal.h)

template <typename T>
__device__ __forceinline__ void ghost_periodic_body(const Grid& G, T* u, long long t) {
  const long long g = G.g;
  const long long X = G.n0 + 2 * g, Y = G.n1 + 2 * g;
  const long long cntA = X * Y * 2 * g;
  const long long cntB = X * 2 * g * G.n2;
  const long long cntC = 2 * g * (long long)G.n1 * G.n2;
  int i, j, k;
  if (t < cntA) {
    const int kk = (int)(t % (2 * g));
    t /= 2 * g;
    j = (int)(t % Y) - (int)g;
    i = (int)(t / Y) - (int)g;
    k = kk < g ? kk - (int)g : G.n2 + kk - (int)g;
  } else if (t < cntA + cntB) {
    t -= cntA;
    k = (int)(t % G.n2);
    t /= G.n2;
    const int jj = (int)(t % (2 * g));
    i = (int)(t / (2 * g)) - (int)g;
    j = jj < g ? jj - (int)g : G.n1 + jj - (int)g;
  } else if (t < cntA + cntB + cntC) {
    t -= cntA + cntB;
    k = (int)(t % G.n2);
    t /= G.n2;
    j = (int)(t % G.n1);
    const int ii = (int)(t / G.n1);
    i = ii < g ? ii - (int)g : G.n0 + ii - (int)g;
  } else {
    return;
  }
  const int si = ((i % G.n0) + G.n0) % G.n0;
  const int sj = ((j % G.n1) + G.n1) % G.n1;
  const int sk = ((k % G.n2) + G.n2) % G.n2;
  u[gidx(G, i, j, k)] = u[gidx(G, si, sj, sk)];
}

// ---- coarse-fine ghosts (Sec. 3.3) ---------------------------------------------------
// The interpolation and flux weights in the kernels' own precision.  The host rounds
// the float64 weights once (round to nearest, the rounding of the device's T(double)
// conversion), so results are bit-identical to converting each weight on the device,
// without the per-use conversions (double-to-float conversions issue on the FP64 pipe,
// which bounded the float32 ghost kernels).
template <typename T>
struct CfW {
  T tang[2][7];
  T ncoarse[3][3];
  T nfine[3][4];
  T flux[6];
};

template <typename T>
inline CfW<T> cf_weights_as(const CfWeights& w) {
  CfW<T> o;
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 7; ++b) o.tang[a][b] = T(w.tang[a][b]);
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b) o.ncoarse[a][b] = T(w.ncoarse[a][b]);
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 4; ++b) o.nfine[a][b] = T(w.nfine[a][b]);
  for (int a = 0; a < 6; ++a) o.flux[a] = T(w.flux[a]);
  return o;
}

__device__ __forceinline__ void face_axes(int a, int& b, int& c) {
  b = (a == 0) ? 1 : 0;
  c = (a == 2) ? 1 : 2;
}

__device__ __forceinline__ int face_of(const FaceSet& fs, long long t, const long long* base) {
  int f = 0;
#pragma unroll
  for (int q = 1; q < 6; ++q)
    if (t >= base[q]) f = q;
  return f;
}

// Tangential interpolation: thread t handles one parent face element (jc, kc) of a
// layer m: the 4 fine positions over it (tj = 2 jc + pj, tk = 2 kc + pk) interpolate
// the same (n+1) x (n+1) patch of parent values, so each row of the patch is reduced
// along c once per parity pk, then along b once per parity pj.
template <int ORDER, typename T>
__device__ __forceinline__ void cf_tangential_body(const Grid& F, const Grid& P,
                                                   const T* pu, Int3 off,
                                                   const FaceSet& fs, const CfW<T>& w, T invH,
                                                   T* inter, T* fc_unc,
                                                   long long t) {
  constexpr int half = ORDER / 2;
  if (t >= half * fs.ebase[6]) return;
  int f = 0;
#pragma unroll
  for (int q = 1; q < 6; ++q)
    if (t >= half * fs.ebase[q]) f = q;
  const int a = f >> 1, side = f & 1;
  int b, c;
  face_axes(a, b, c);
  const int nt0 = fs.nt[f][0], nt1 = fs.nt[f][1];
  const int ne1 = nt1 / 2;
  const long long ne = (long long)(nt0 / 2) * ne1;
  long long loc = t - half * fs.ebase[f];
  const int m = (int)(loc / ne);
  loc -= (long long)m * ne;
  const int jc = (int)(loc / ne1), kc = (int)(loc % ne1);
  auto pick = [](int ax, int x, int y, int z) { return ax == 0 ? x : (ax == 1 ? y : z); };
  const int off_a = pick(a, off.x, off.y, off.z), nf_a = pick(a, F.n0, F.n1, F.n2);
  const int pn = side == 0 ? off_a - 1 - m : off_a + nf_a / 2 + m;
  const int pb = pick(b, off.x, off.y, off.z) + jc, pc = pick(c, off.x, off.y, off.z) + kc;
  // parent element strides along a, b, c and the patch corner (pn, pb - half, pc - half)
  const long long sxP = (long long)P.Y * P.Zp, syP = P.Zp;
  auto stride = [&](int ax) { return ax == 0 ? sxP : (ax == 1 ? syP : 1LL); };
  const long long sa = stride(a), sb = stride(b), sc = stride(c);
  auto coord = [&](int ax, int va, int vb, int vc) { return ax == a ? va : (ax == b ? vb : vc); };
  const long long p0 = gidx(P, coord(0, pn, pb - half, pc - half), coord(1, pn, pb - half, pc - half),
                            coord(2, pn, pb - half, pc - half));
  T row[2][ORDER + 1];
#pragma unroll
  for (int bb = 0; bb <= ORDER; ++bb) {
    T r0 = T(0), r1 = T(0);
#pragma unroll
    for (int cc = 0; cc <= ORDER; ++cc) {
      const T v = pu[p0 + bb * sb + cc * sc];
      r0 = fma(w.tang[0][cc], v, r0);
      r1 = fma(w.tang[1][cc], v, r1);
    }
    row[0][bb] = r0;
    row[1][bb] = r1;
  }
  typedef typename Vec2<T>::type V2;
#pragma unroll
  for (int pj = 0; pj < 2; ++pj) {
    T acc0 = T(0), acc1 = T(0);
#pragma unroll
    for (int bb = 0; bb <= ORDER; ++bb) {
      acc0 = fma(w.tang[pj][bb], row[0][bb], acc0);
      acc1 = fma(w.tang[pj][bb], row[1][bb], acc1);
    }
    // (tk, tk + 1) = (2 kc, 2 kc + 1): an even, hence 2-element aligned, pair
    V2 out;
    out.x = acc0;
    out.y = acc1;
    *reinterpret_cast<V2*>(inter + fs.base[f] + ((long long)m * nt0 + 2 * jc + pj) * nt1 + 2 * kc) =
        out;
  }
  if (m == 0) {
    // uncovered part of the parent face flux for element (jc, kc): parent cells
    // pface - half + s along a, s0 <= s < s1, at (pb, pc)
    const int pface = side == 0 ? off_a : off_a + nf_a / 2;
    const long long q0 = p0 + half * sb + half * sc + (long long)(pface - half - pn) * sa;
    T fc = T(0);
    const int s0 = side == 0 ? 0 : half, s1 = side == 0 ? half : ORDER;
    for (int s = s0; s < s1; ++s) fc = fma(w.flux[s], pu[q0 + s * sa], fc);
    fc_unc[fs.ebase[f] + (long long)jc * ne1 + kc] = fc * invH;
  }
}

// Normal interpolation and flux matching: thread t handles one fine column of a face;
// the 4 columns under one parent face element are 4 consecutive lanes (a "quad"), which
// share the parent flux and the mean of their fine fluxes through warp shuffles.  Scale
// factors come precomputed: fc_scale = 1/(8 H) for the covered parent cells (mean of 8
// children, parent spacing H); the ghost shift (F_c - mean F_f) h / c_side is
// a_side F_c - b_side (sum of the 4 unscaled fine flux stencils), a_side = h / c_side,
// b_side = 1 / (4 c_side) (c_side: the sum of the flux weights on the ghost side).
// Reads and writes u with plain accesses (the ghosts it writes are not read by it).
// A fine column of face f: column col (0..3) of parent face element (jc, kc).
struct FaceCol {
  int f, jc, kc, col;
  int tj, tk;      // fine tangential position
  long long in0;   // element of the column's cell at the face
  int step;        // element stride inwards
};

__device__ __forceinline__ FaceCol face_col(const Grid& F, int f, int jc, int kc, int col) {
  FaceCol c;
  c.f = f;
  c.jc = jc;
  c.kc = kc;
  c.col = col;
  const int a = f >> 1, side = f & 1;
  c.tj = 2 * jc + (col >> 1);
  c.tk = 2 * kc + (col & 1);
  // strides along the normal (a) and the tangential axes (b, c) of this face
  const int sx = F.Y * F.Zp, sy = F.Zp;
  const int sa = a == 0 ? sx : (a == 1 ? sy : 1);
  const int sb = a == 0 ? sy : sx;
  const int sc = a == 2 ? sy : 1;
  const int na = a == 0 ? F.n0 : (a == 1 ? F.n1 : F.n2);
  // moving inwards is +sa (low face) or -sa (high)
  c.in0 = gidx(F, 0, 0, 0) + ((long long)c.tj * sb + c.tk * sc);
  if (side) c.in0 += (long long)(na - 1) * sa;
  c.step = side == 0 ? sa : -sa;
  return c;
}

// Writes the ghosts of column c into u from its ORDER cells nearest the face, v; quad: a
// mask of converged lanes that holds the element's four.
template <int ORDER, typename T>
__device__ __forceinline__ void cf_flux_at(T* u, const FaceSet& fs, const CfW<T>& w,
                                           const T* inter,
                                           const T* fc_unc, T fc_scale, T a0, T a1,
                                           T b0, T b1, int flux_fix, const FaceCol& fcol,
                                           const T (&v)[ORDER], unsigned quad) {
  constexpr int half = ORDER / 2;
  const int f = fcol.f, side = f & 1;
  const int nt0 = fs.nt[f][0], nt1 = fs.nt[f][1];
  const long long e = fs.ebase[f] + (long long)fcol.jc * (nt1 / 2) + fcol.kc;
  const int tj = fcol.tj, tk = fcol.tk;
  // parent flux: uncovered part + covered parent cells as the mean of their 8
  // children; each column holds 2 of the 8 (normal 2d, 2d+1)
  T cov = T(0);
#pragma unroll
  for (int d = 0; d < half; ++d) {
    const int s = side == 0 ? half + d : half - 1 - d;
    T pair = v[2 * d] + v[2 * d + 1];
    pair += __shfl_xor_sync(quad, pair, 1);
    pair += __shfl_xor_sync(quad, pair, 2);
    cov = fma(w.flux[s], pair, cov);
  }
  const T fc = fma(cov, fc_scale, fc_unc[e]);
  T cq[half];
#pragma unroll
  for (int q = 0; q < half; ++q) cq[q] = inter[fs.base[f] + ((long long)q * nt0 + tj) * nt1 + tk];
  T ghost[half];
#pragma unroll
  for (int m = 0; m < half; ++m) {
    T gv = T(0);
#pragma unroll
    for (int q = 0; q < half; ++q) gv = fma(w.ncoarse[m][q], cq[q], gv);
#pragma unroll
    for (int q = 0; q <= half; ++q) gv = fma(w.nfine[m][q], v[q], gv);
    ghost[m] = gv;
  }
  T ff = T(0);
#pragma unroll
  for (int s = 0; s < ORDER; ++s) {
    T x;
    if (side == 0) x = s < half ? ghost[half - 1 - s] : v[s - half];
    else x = s < half ? v[half - 1 - s] : ghost[s - half];
    ff = fma(w.flux[s], x, ff);
  }
  ff += __shfl_xor_sync(quad, ff, 1);
  ff += __shfl_xor_sync(quad, ff, 2);
  T shift = T(0);
  if (flux_fix) shift = fma(-(side ? b1 : b0), ff, fc * (side ? a1 : a0));
#pragma unroll
  for (int m = 0; m < half; ++m) u[fcol.in0 - (m + 1) * fcol.step] = ghost[m] + shift;
}

// The ORDER cells of a column nearest the face.
template <int ORDER, typename T>
__device__ __forceinline__ void load_column(const T* u, const FaceCol& c, T (&v)[ORDER]) {
#pragma unroll
  for (int q = 0; q < ORDER; ++q) v[q] = u[c.in0 + q * c.step];
}

template <int ORDER, typename T>
__device__ __forceinline__ void cf_flux_body(const Grid& F, T* u, const FaceSet& fs,
                                             const CfW<T>& w, const T* inter,
                                             const T* fc_unc, T fc_scale, T a0, T a1,
                                             T b0, T b1, int flux_fix, long long t) {
  if (t >= 4 * fs.ebase[6]) return;
  const unsigned quad = __activemask();
  const int e = (int)(t >> 2);
  const int f = face_of(fs, e, fs.ebase);
  const unsigned loc = (unsigned)(e - (int)fs.ebase[f]), ne1 = fs.nt[f][1] / 2;
  const FaceCol c = face_col(F, f, (int)(loc / ne1), (int)(loc % ne1), (int)(t & 3));
  T v[ORDER];
  load_column<ORDER, T>(u, c, v);
  cf_flux_at<ORDER, T>(u, fs, w, inter, fc_unc, fc_scale, a0, a1, b0, b1, flux_fix, c, v, quad);
}

// The flux step of float64 solves with everything that is linear folded on the host or into
// the tangential kernel: the ghost of layer m is G_m + sum_q nfine[m][q] v_q + shift, and
// shift = K + sum over the 4 columns of sum_q d[side][q] v_q, where G_m and K (inter and
// fc_unc of the folded tangential kernel) carry the parent values, and d the parent flux of
// the covered cells minus the fine fluxes.  24 FP64 instructions per column instead of 47.
struct FluxFold {
  double d[2][6];
  double nfine[3][4];
};

template <int ORDER>
__device__ __forceinline__ void cf_fold_at(double* u, const FaceSet& fs, const FluxFold& w,
                                           const double* inter,
                                           const double* fc_unc, const FaceCol& c,
                                           const double (&v)[ORDER], unsigned quad) {
  constexpr int half = ORDER / 2;
  const int side = c.f & 1;
  const int nt0 = fs.nt[c.f][0], nt1 = fs.nt[c.f][1];
  double g[half];
  const double* ip = inter + fs.base[c.f] + ((long long)c.tj * nt1 + c.tk);
#pragma unroll
  for (int m = 0; m < half; ++m) g[m] = ip[(long long)m * nt0 * nt1];
  const double k = fc_unc[fs.ebase[c.f] + (long long)c.jc * (nt1 / 2) + c.kc];
  double s = w.d[side][0] * v[0];
#pragma unroll
  for (int q = 1; q < 2 * half; ++q) s = fma(w.d[side][q], v[q], s);
  s += __shfl_xor_sync(quad, s, 1);
  s += __shfl_xor_sync(quad, s, 2);
  s += k;
#pragma unroll
  for (int m = 0; m < half; ++m) {
    double x = g[m] + s;
#pragma unroll
    for (int q = 0; q <= half; ++q) x = fma(w.nfine[m][q], v[q], x);
    u[c.in0 - (m + 1) * c.step] = x;
  }
}

// What a kernel needs to write a nest's ghosts: float as cf_flux_at, double folded.
template <typename T>
struct FaceArgs;
template <>
struct FaceArgs<float> {
  FaceSet fs;
  CfW<float> w;
  const float* inter;
  const float* fc_unc;
  float fc_scale, a0, a1, b0, b1;
  template <int ORDER>
  __device__ __forceinline__ void ghosts(float* u, const FaceCol& c, const float (&v)[ORDER],
                                         unsigned quad) const {
    cf_flux_at<ORDER, float>(u, fs, w, inter, fc_unc, fc_scale, a0, a1, b0, b1, 1, c, v, quad);
  }
};
template <>
struct FaceArgs<double> {
  FaceSet fs;
  FluxFold w;
  const double* inter;
  const double* fc_unc;
  template <int ORDER>
  __device__ __forceinline__ void ghosts(double* u, const FaceCol& c, const double (&v)[ORDER],
                                         unsigned quad) const {
    cf_fold_at<ORDER>(u, fs, w, inter, fc_unc, c, v, quad);
  }
};
template <typename T>
FaceArgs<T> make_face_args(int order, const FaceSet& fs, const CfWeights& w, const T* inter,
                           const T* fc_unc, double h, double invH);

// ---- coarsest level: periodic pseudo-inverse of L as a circular convolution --------
// u(x) = sum_y K(x - y) f(y), K precomputed on the host from the DFT symbol; block x
// computes output cell x, its kCoarseThreads threads split the sum over y (float64
// sums for either precision); the result also goes to the cell's periodic images.
// Every thread of the block must call it (block-wide reduction).
constexpr int kCoarseThreads = 128;

template <typename T>
__device__ __forceinline__ void coarsest_body(const Grid& G, const T* f,
                                              T* u, const double* kern,
                                              int x, int tid) {
  const int n12 = G.n1 * G.n2;
  const int n = G.n0 * n12;
  const int xk = x % G.n2, xj = (x / G.n2) % G.n1, xi = x / n12;
  double acc = 0.0;
  for (int y = tid; y < n; y += kCoarseThreads) {
    const int yk = y % G.n2, yj = (y / G.n2) % G.n1, yi = y / n12;
    int di = xi - yi, dj = xj - yj, dk = xk - yk;
    di += di < 0 ? G.n0 : 0;
    dj += dj < 0 ? G.n1 : 0;
    dk += dk < 0 ? G.n2 : 0;
    acc = fma(__ldg(kern + (di * G.n1 + dj) * G.n2 + dk), (double)f[gidx(G, yi, yj, yk)], acc);
  }
  __shared__ double red[kCoarseThreads];
  red[tid] = acc;
  __syncthreads();
#pragma unroll
  for (int w = kCoarseThreads / 2; w > 0; w >>= 1) {
    if (tid < w) red[tid] += red[tid + w];
    __syncthreads();
  }
  if (tid == 0) {
    const T v = (T)red[0];
    u[gidx(G, xi, xj, xk)] = v;
    write_images<T>(G, u, xi, xj, xk, v);
  }
  __syncthreads();  // red[] may be reused by the caller's next block
}

}  // namespace mgk
