// Hybrid Poisson solver correction (Hahn & Abel 2011, Sec. 3.5.2).
//
// The finite-difference solution loses small-scale power on the finest level; the
// paper replaces the finest level's own contribution by the exact k-space one:
// with f the level's source (zero outside the level, on a grid zero-padded to
// twice its size), the displacement correction is the difference between the
// exact gradient of the inverse Laplacian and the order-n finite-difference one,
//   d psi_j(k) = i [k_j / k^2 + g_j(k) / Lt(k)] f(k)
// for psi = -G phi, forward transform sum_x f(x) e^{-ik.x}, Lt = -sum_a lam_n(k_a h)
// / h^2 the Table 1 Laplacian symbol and i g_j = i g_n(k_j h) / h the Table 1
// gradient symbol (lam_2 = 2(1 - cos t), g_2 = sin t, and so on), 0 at k = 0 and,
// as the multiplier is odd in k_j, on the Nyquist plane of axis j.
// A single periodic level is corrected periodically, without padding.
//
// With t_a = k_a h, the multiplier of component j is h [t_j / t^2 - gamma_j / lambda],
// gamma_j = g_n(t_j), lambda = sum_a lam_n(t_a): two nearly equal fractions at small k.  It
// is formed as h [t_j (lambda - t^2) - (gamma_j - t_j) t^2] / (t^2 lambda) from per-axis tables
// of t, lam_n, lam_n - t^2 and g_n - t, the last two by their Taylor series at small t, so
// that nothing cancels.
//
// Steps: copy f into the rows of a real grid padded along y and z; 2D transforms of the
// level's own x planes (the padding planes are zero) and 1D transforms along x; per
// component j a kernel forms the multiplied half spectrum (with the 1/N of the inverse), 1D
// inverses along x and 2D inverses of the level's own planes, and a kernel adds the level's
// part of the result to psi_j.
#include <cufft.h>

#include <cmath>
#include <vector>

#include "mg_internal.h"
#include "mg_setup.h"

namespace mgk {

namespace {

// Per axis and index: t = k h, lam_n(t), lam_n(t) - t^2, g_n(t) - t.
struct AxisSymbol {
  double t, lam, dlam, dgam;
};

// lam_n(t) = sum_s w_s 2 (1 - cos s t), g_n(t) = sum_s g_s 2 sin s t with the Table 1 weights.
// Their Taylor coefficients vanish between t^2 (t) and t^(n + 2) (t^(n + 1)); the series
// from there on gives the differences below t = 1.5, where 30 terms reach rounding.
AxisSymbol axis_symbol(int order, double t) {
  const int half = order / 2;
  double l[7];
  laplacian_1d(order, l);
  const double g[4][3] = {{}, {0.5, 0, 0}, {8.0 / 12, -1.0 / 12, 0}, {45.0 / 60, -9.0 / 60, 1.0 / 60}};
  AxisSymbol a{t, 0.0, 0.0, 0.0};
  double gam = 0.0;
  for (int s = 1; s <= half; ++s) {
    const double si = std::sin(0.5 * s * t);
    a.lam += l[half + s] * 4.0 * si * si;
    gam += g[half][s - 1] * 2.0 * std::sin(s * t);
  }
  if (std::fabs(t) > 1.5) {
    a.dlam = a.lam - t * t;
    a.dgam = gam - t;
    return a;
  }
  for (int s = 1; s <= half; ++s) {
    const double x = s * t;
    double term = 1.0;  // x^p / p!
    for (int p = 1; p <= order + 60; ++p) {
      term *= x / p;
      const int q = p / 2;
      if (p % 2 == 0 && p >= order + 2) a.dlam += (q % 2 ? 2.0 : -2.0) * l[half + s] * term;
      if (p % 2 == 1 && p >= order + 1) a.dgam += (q % 2 ? -2.0 : 2.0) * g[half][s - 1] * term;
    }
  }
  return a;
}

// R (n0 x N1 x N2 dense) := f on [0, n) of every axis, 0 elsewhere.
__global__ void __launch_bounds__(256)
    k_pad(const double* __restrict__ f, int n0, int n1, int n2, double* __restrict__ R, int N1,
          int N2) {
  const long long total = (long long)n0 * N1 * N2;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(e % N2);
    const long long r = e / N2;
    const int j = (int)(r % N1);
    const int i = (int)(r / N1);
    R[e] = (j < n1 && k < n2) ? __ldg(f + ((long long)i * n1 + j) * n2 + k) : 0.0;
  }
}

// W = i c F / N over the half spectrum of the N grid, c the multiplier of component comp.
// tab: the tables of the three axes one after another.  About 22 FP64 instructions per mode
// (the FP64 pipe bounds it; nine sincos per mode took 4.28 ms at 256 x 192 x 224).
__global__ void __launch_bounds__(256)
    k_hybrid_multiply(const cufftDoubleComplex* __restrict__ F, cufftDoubleComplex* __restrict__ W,
                      int N0, int N1, int N2, const AxisSymbol* __restrict__ tab, double scale,
                      int comp) {
  const int N2h = N2 / 2 + 1;
  // blocks in one dimension, along m first: a side may pass the 65535 of the other dimensions
  const unsigned bm = (N2h + 255) / 256, row = blockIdx.x / bm;
  const int i = row / N1, j = row % N1;
  const int m = (blockIdx.x - row * bm) * 256 + threadIdx.x;
  if (m >= N2h) return;
  const AxisSymbol a[3] = {tab[i], tab[N0 + j], tab[N0 + N1 + m]};
  const int idx[3] = {i, j, m}, N[3] = {N0, N1, N2};
  const double tsq = fma(a[0].t, a[0].t, fma(a[1].t, a[1].t, a[2].t * a[2].t));
  const double lam = a[0].lam + a[1].lam + a[2].lam;
  const double dl = a[0].dlam + a[1].dlam + a[2].dlam;
  // the multiplier is odd in k_comp: 0 on the self-conjugate Nyquist plane of that axis
  // (even N), so the product stays Hermitian and its inverse real
  const bool nyq = (N[comp] & 1) == 0 && idx[comp] == N[comp] / 2;
  double c = 0.0;
  if ((i | j | m) != 0 && !nyq) {
    const AxisSymbol s = comp == 0 ? a[0] : (comp == 1 ? a[1] : a[2]);
    c = fma(s.t, dl, -(s.dgam * tsq)) * (scale / (tsq * lam));
  }
  const long long e = ((long long)i * N1 + j) * N2h + m;
  const cufftDoubleComplex v = F[e];
  W[e] = make_cuDoubleComplex(-v.y * c, v.x * c);  // i c v
}

// psi[x] += R[x] for x in the level's [0, n) block of the N grid.
__global__ void __launch_bounds__(256)
    k_crop_add(const double* __restrict__ R, int N1, int N2, double* __restrict__ psi, int n0,
               int n1, int n2) {
  const long long total = (long long)n0 * n1 * n2;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(e % n2);
    const long long r = e / n2;
    const int j = (int)(r % n1);
    const int i = (int)(r / n1);
    psi[e] += __ldg(R + ((long long)i * N1 + j) * N2 + k);
  }
}

unsigned blocks_cap(long long work) {
  const long long b = (work + 255) / 256;
  return (unsigned)(b < 1 ? 1 : (b > 152 * 16 ? 152 * 16 : b));
}

}  // namespace

struct HybridFFT {
  int n[3] = {0, 0, 0}, N[3] = {0, 0, 0};
  double h = 0.0;
  double* R = nullptr;              // n0 x N1 x N2
  cufftDoubleComplex* F = nullptr;  // N0 x N1 x (N2 / 2 + 1)
  cufftDoubleComplex* W = nullptr;
  AxisSymbol* tab = nullptr;
  void* work = nullptr;  // shared by the plans
  // planes (y, z) of the level's own x range; lines along x
  cufftHandle fwd_planes = 0, inv_planes = 0, lines = 0;
  int plans = 0;  // how many of the three exist
};

size_t hybrid_bytes(int n0, int n1, int n2, bool pad) {
  const long long f = pad ? 2 : 1;
  const long long N0 = f * n0, N1 = f * n1, N2 = f * n2;
  const long long real = n0 * N1 * N2 * 8;
  const long long spec = N0 * N1 * (N2 / 2 + 1) * 16;
  // real grid (the level's own planes), two half spectra, the axes' tables, and at most about one
  // half spectrum of cuFFT work area (0.03 to 0.13 of one at 128^3 and above, 0.36 at 60^3)
  return (size_t)(real + 3 * spec + (N0 + N1 + N2) * (long long)sizeof(AxisSymbol));
}

void hybrid_destroy(HybridFFT* hy) {
  if (!hy) return;
  cufftHandle* const h[3] = {&hy->fwd_planes, &hy->inv_planes, &hy->lines};
  for (int q = 0; q < hy->plans; ++q) cufftDestroy(*h[q]);
  cudaFree(hy->R);
  cudaFree(hy->F);
  cudaFree(hy->W);
  cudaFree(hy->tab);
  cudaFree(hy->work);
  delete hy;
}

cudaError_t hybrid_create(HybridFFT** out, int n0, int n1, int n2, double h, int order,
                          bool pad) {
  *out = nullptr;
  HybridFFT* hy = new HybridFFT();
  const int f = pad ? 2 : 1;
  hy->n[0] = n0;
  hy->n[1] = n1;
  hy->n[2] = n2;
  hy->N[0] = f * n0;
  hy->N[1] = f * n1;
  hy->N[2] = f * n2;
  hy->h = h;
  const int N2h = hy->N[2] / 2 + 1;
  const size_t real = (size_t)n0 * hy->N[1] * hy->N[2];
  const size_t spec = (size_t)hy->N[0] * hy->N[1] * N2h;
  std::vector<AxisSymbol> tab;
  for (int a = 0; a < 3; ++a)
    for (int q = 0; q < hy->N[a]; ++q) {
      const int idx = q <= hy->N[a] / 2 ? q : q - hy->N[a];
      tab.push_back(axis_symbol(order, 2.0 * M_PI * (double)idx / hy->N[a]));
    }
  cudaError_t e = cudaMalloc(&hy->R, real * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&hy->F, spec * sizeof(cufftDoubleComplex));
  if (e == cudaSuccess) e = cudaMalloc(&hy->W, spec * sizeof(cufftDoubleComplex));
  if (e == cudaSuccess) e = cudaMalloc(&hy->tab, tab.size() * sizeof(AxisSymbol));
  if (e == cudaSuccess)
    e = cudaMemcpy(hy->tab, tab.data(), tab.size() * sizeof(AxisSymbol), cudaMemcpyHostToDevice);
  // the plans run one after another: one work area of the largest size serves all
  size_t need = 0;
  auto plan = [&](cufftHandle* p, int rank, int* n, int* embed, int stride, int dist,
                  cufftType type, int batch) {
    if (e != cudaSuccess) return;
    size_t bytes = 0;
    if (cufftCreate(p) != CUFFT_SUCCESS) {
      e = cudaErrorMemoryAllocation;
      return;
    }
    hy->plans++;
    if (cufftSetAutoAllocation(*p, 0) != CUFFT_SUCCESS ||
        cufftMakePlanMany(*p, rank, n, embed, stride, dist, embed, stride, dist, type, batch,
                          &bytes) != CUFFT_SUCCESS)
      e = cudaErrorMemoryAllocation;
    if (bytes > need) need = bytes;
  };
  int n2d[2] = {hy->N[1], hy->N[2]}, n1d[1] = {hy->N[0]};
  plan(&hy->fwd_planes, 2, n2d, nullptr, 1, 0, CUFFT_D2Z, n0);
  plan(&hy->inv_planes, 2, n2d, nullptr, 1, 0, CUFFT_Z2D, n0);
  plan(&hy->lines, 1, n1d, n1d, hy->N[1] * N2h, 1, CUFFT_Z2Z, hy->N[1] * N2h);
  if (e == cudaSuccess && need) e = cudaMalloc(&hy->work, need);
  if (e == cudaSuccess && need)
    for (cufftHandle p : {hy->fwd_planes, hy->inv_planes, hy->lines})
      if (cufftSetWorkArea(p, hy->work) != CUFFT_SUCCESS) e = cudaErrorMemoryAllocation;
  if (e != cudaSuccess) {
    hybrid_destroy(hy);
    return e;
  }
  *out = hy;
  return cudaSuccess;
}

cudaError_t hybrid_apply(HybridFFT* hy, const double* f, double* const psi[3], cudaStream_t s) {
  for (cufftHandle p : {hy->fwd_planes, hy->inv_planes, hy->lines})
    if (cufftSetStream(p, s) != CUFFT_SUCCESS) return cudaErrorUnknown;
  const int n0 = hy->n[0], N0 = hy->N[0], N1 = hy->N[1], N2 = hy->N[2], N2h = N2 / 2 + 1;
  const long long real = (long long)n0 * N1 * N2, plane = (long long)N1 * N2h;
  const long long cells = (long long)n0 * hy->n[1] * hy->n[2];
  k_pad<<<blocks_cap(real), 256, 0, s>>>(f, n0, hy->n[1], hy->n[2], hy->R, N1, N2);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (cufftExecD2Z(hy->fwd_planes, hy->R, hy->F) != CUFFT_SUCCESS) return cudaErrorUnknown;
  if (N0 > n0 && (e = cudaMemsetAsync(hy->F + n0 * plane, 0,
                                      (size_t)(N0 - n0) * plane * sizeof(cufftDoubleComplex),
                                      s)) != cudaSuccess)
    return e;
  if (cufftExecZ2Z(hy->lines, hy->F, hy->F, CUFFT_FORWARD) != CUFFT_SUCCESS)
    return cudaErrorUnknown;
  const double scale = hy->h / ((double)N0 * N1 * N2);
  const unsigned grid = (unsigned)((N2h + 255) / 256) * N1 * N0;
  for (int c = 0; c < 3; ++c) {
    k_hybrid_multiply<<<grid, 256, 0, s>>>(hy->F, hy->W, N0, N1, N2, hy->tab, scale, c);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (cufftExecZ2Z(hy->lines, hy->W, hy->W, CUFFT_INVERSE) != CUFFT_SUCCESS ||
        cufftExecZ2D(hy->inv_planes, hy->W, hy->R) != CUFFT_SUCCESS)
      return cudaErrorUnknown;
    k_crop_add<<<blocks_cap(cells), 256, 0, s>>>(hy->R, N1, N2, psi[c], n0, hy->n[1], hy->n[2]);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace mgk
