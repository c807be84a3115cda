// Spectral bounds for the Chebyshev scaling chi_q, zeta_q of Sec. 4 (FP64 for SQ_FP64; for
// SQ_MIXED the Krylov vectors and H_q applications are FP32, the Gram-Schmidt coefficients,
// tridiagonal and Ritz values FP64 - the bounds are widened by 1 % of the width anyway).
//
// The paper takes chi_q and zeta_q from the extreme eigenvalues of H_q and does not say how
// they are obtained. Here: k-step Lanczos on the nodal Hamiltonian H_q of every node of a few
// sample tiles (one Lanczos column per node, all columns advanced together with the tile
// kernels), full reorthogonalisation by classical Gram-Schmidt applied twice, Ritz extremes
// of the tridiagonal matrix widened by their residual norms, the interval over all columns,
// then widened by 1 % of its width on each side. One interval serves every node (every H_q
// is a principal submatrix of the infinite-crystal H, so a shared interval is valid for all
// of them when it contains the sampled spectra with margin).
#include <algorithm>
#include <cmath>
#include <vector>

#include "sq_device.cuh"

namespace sq {

constexpr int kTileLz = 8;              // nodes per tile (columns per tile)
constexpr int kMaxLanczosVecs = 136;    // Krylov vectors held (k + 1, k <= 128 + 7)

// Start vector of the column of node q: 1 + (hash(i, node) mod 1009) / 1009 on the window
// (i = window-local index, C order z, y, x), zero elsewhere; normalised afterwards.
template <typename Real>
__global__ void k_lz_init(Geo g, Wave w, Real* __restrict__ V0) {
  const size_t per_tile = (size_t)g.Upts * g.B;
  const size_t total = per_tile * w.ntiles;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
    const int tl = int(idx / per_tile);
    const int r = int(idx % per_tile);
    const int q = r % g.B, pt = r / g.B;
    const int ux = pt % g.U[0], uy = (pt / g.U[0]) % g.U[1], uz = pt / (g.U[0] * g.U[1]);
    int o[3], qo[3];
    tile_origin(g, wave_tile(w, tl), o);
    node_offset(g, q, qo);
    double v = 0.0;
    if (node_valid(g, o, qo) && in_window(g, qo, ux, uy, uz)) {
      const int kx = ux - qo[0], ky = uy - qo[1], kz = uz - qo[2];
      const unsigned long long i = (unsigned long long)((kz * (2 * g.m[1] + 1) + ky) * (2 * g.m[0] + 1) + kx);
      const unsigned long long node =
          (unsigned long long)((o[0] + qo[0]) + g.n[0] * ((o[1] + qo[1]) + g.n[1] * (o[2] + qo[2])));
      const unsigned long long hsh = (i * 2654435761ull + node * 40503ull) & 0xFFFFFFFFull;
      v = 1.0 + double(hsh % 1009ull) / 1009.0;
    }
    V0[idx] = Real(v);
  }
}

// Start vector e_q: one at node q's own point of the union window, zero elsewhere (and an
// all-zero column for padding nodes, which the mark-empty pass then skips).
template <typename Real>
__global__ void k_lz_init_unit(Geo g, Wave w, Real* __restrict__ V0) {
  const size_t per_tile = (size_t)g.Upts * g.B;
  const size_t total = per_tile * w.ntiles;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
    const int tl = int(idx / per_tile);
    const int r = int(idx % per_tile);
    const int q = r % g.B, pt = r / g.B;
    int o[3], qo[3];
    tile_origin(g, wave_tile(w, tl), o);
    node_offset(g, q, qo);
    const int cpt = ((qo[2] + g.m[2]) * g.U[1] + (qo[1] + g.m[1])) * g.U[0] + (qo[0] + g.m[0]);
    V0[idx] = (node_valid(g, o, qo) && pt == cpt) ? Real(1) : Real(0);
  }
}

// ---- Gram-Schmidt on the Krylov vectors of a wave.
// One block per (chunk of a tile's points, tile), in rounds of 256 groups of four nodes. Update: a thread
// owns one group and walks the vectors. Products: the round's x sits in shared memory and the eight warps
// share out the vectors V_i, each taking all groups of its vectors, so x is read from memory once, a
// V chunk read by the update is still in cache for the products, and no product crosses warps. The
// four products of a lane are added over the warp by a reduce-scatter (5 exchanges in place of 16).
// Cross-thread sums: FP64 vectors add doubles, FP32 vectors add pairs of floats
// (two-sum; FP64 adds issue at 1.7 lanes per clock here and cost more than the products).
constexpr int kLzThreads = 256, kLzWarps = kLzThreads / 32;

template <typename Real> struct LzV4;
template <> struct LzV4<float> { using T = float4; };
template <> struct LzV4<double> { using T = double4_32a; };

// the four products of a lane (nodes 4 (lane & 1) ..), added over the warp into acc[8] (one warp per acc)
template <typename Real>
__device__ __forceinline__ void lz_warp_add(const Real d[4], typename LzAcc<Real>::T* acc) {
  int node;
  const auto s = lz_warp_sum<Real>(d, &node);
  if ((threadIdx.x & 31) < 8) acc[node] = lz_add(acc[node], s);
}

enum LzMode { kLzDots = 0, kLzUpdateDots = 1, kLzUpdateNorm = 2, kLzNorm = 3 };

// in, out[((tile nch + chunk) ld + i) 8 + node]: the chunk's share of <V_i, x>; norms, <x, x>, are packed
// (ld = 1, i = 0).
//   kLzDots        out = V^T x
//   kLzUpdateDots  x -= V (sum over chunks of in), then out = V^T x
//   kLzUpdateNorm  x -= V (sum over chunks of in), then out = x^T x
//   kLzNorm        out = x^T x
// The coefficient of the last vector goes to (kLzUpdateDots) or is added to (kLzUpdateNorm)
// alpha[col k + nvec - 1].
template <typename Real, int MODE>
__global__ void __launch_bounds__(kLzThreads)
k_lz_ortho(Geo g, const Real* __restrict__ V, int nvec, size_t vstride, Real* __restrict__ x,
           const double* __restrict__ in, double* __restrict__ out, int ld, int k, double* __restrict__ alpha) {
  using V4 = typename LzV4<Real>::T;
  using A = typename LzAcc<Real>::T;
  extern __shared__ __align__(16) unsigned char lz_smem[];
  constexpr bool kNorm = MODE == kLzUpdateNorm || MODE == kLzNorm;
  constexpr bool kUpdate = MODE == kLzUpdateDots || MODE == kLzUpdateNorm;
  const int nch = gridDim.x, c = blockIdx.x, tl = blockIdx.y, warp = threadIdx.x >> 5;
  V4* xs = reinterpret_cast<V4*>(lz_smem);                             // [kLzThreads] the round's x
  A* acc = reinterpret_cast<A*>(xs + kLzThreads);                      // products [nvec][8], norms [kLzWarps][8]
  Real* cf = reinterpret_cast<Real*>(acc + (kNorm ? kLzWarps : nvec) * kTileLz);   // [nvec][8]
  for (int i = threadIdx.x; i < (kNorm ? kLzWarps : nvec) * kTileLz; i += kLzThreads) acc[i] = LzAcc<Real>::make(Real(0));
  if constexpr (kUpdate) {
    for (int i = threadIdx.x; i < nvec * kTileLz; i += kLzThreads) {
      const double* p = in + (size_t)tl * nch * ld * kTileLz + i;
      double s = 0.0;
#pragma unroll 4
      for (int cc = 0; cc < nch; ++cc) s += p[(size_t)cc * ld * kTileLz];
      cf[i] = Real(s);
      if (c == 0 && i / kTileLz == nvec - 1) {
        double* al = alpha + (size_t)(tl * kTileLz + i % kTileLz) * k + nvec - 1;
        *al = (MODE == kLzUpdateDots) ? s : *al + s;
      }
    }
  }
  __syncthreads();
  const size_t n = (size_t)g.Upts * 2;                  // groups of four nodes of the tile
  const size_t g0 = (size_t)g.Upts * c / nch * 2, g1 = (size_t)g.Upts * (c + 1) / nch * 2;
  const V4* Vt = reinterpret_cast<const V4*>(V) + (size_t)tl * n;
  V4* xt = reinterpret_cast<V4*>(x) + (size_t)tl * n;
  const size_t vs = vstride / 4;
  const int lane = threadIdx.x & 31;
  for (size_t r0 = g0; r0 < g1; r0 += kLzThreads) {
    const size_t p = r0 + threadIdx.x;
    V4 xv;
    xv.x = xv.y = xv.z = xv.w = Real(0);
    if (p < g1) {
      xv = xt[p];
      if constexpr (kUpdate) {
        const Real* ci = cf + 4 * (threadIdx.x & 1);
        Real u[4] = {Real(0), Real(0), Real(0), Real(0)};
#pragma unroll 4
        for (int i = 0; i < nvec; ++i, ci += kTileLz) {
          const V4 t = Vt[i * vs + p];
          u[0] += ci[0] * t.x; u[1] += ci[1] * t.y; u[2] += ci[2] * t.z; u[3] += ci[3] * t.w;
        }
        xv.x -= u[0]; xv.y -= u[1]; xv.z -= u[2]; xv.w -= u[3];
        xt[p] = xv;
      }
    }
    if constexpr (kNorm) {
      if (r0 + 32 * warp < g1) {
        const Real d[4] = {xv.x * xv.x, xv.y * xv.y, xv.z * xv.z, xv.w * xv.w};
        lz_warp_add<Real>(d, acc + warp * kTileLz);
      }
    } else {
      xs[threadIdx.x] = xv;
      __syncthreads();
      const int ng = int(min((size_t)kLzThreads, g1 - r0));
      for (int i = warp; i < nvec; i += kLzWarps) {
        const V4* Vi = Vt + i * vs + r0;
        Real d[4] = {Real(0), Real(0), Real(0), Real(0)};
#pragma unroll
        for (int e = 0; e < kLzThreads; e += 32)
          if (e + lane < ng) {
            const V4 t = Vi[e + lane], xx = xs[e + lane];
            d[0] += xx.x * t.x; d[1] += xx.y * t.y; d[2] += xx.z * t.z; d[3] += xx.w * t.w;
          }
        lz_warp_add<Real>(d, acc + i * kTileLz);
      }
      __syncthreads();
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < (kNorm ? 1 : nvec) * kTileLz; i += kLzThreads) {
    double s = lz_double(acc[i]);
    if constexpr (kNorm)
      for (int w = 1; w < kLzWarps; ++w) s += lz_double(acc[w * kTileLz + i]);
    out[((size_t)tl * nch + c) * (kNorm ? 1 : ld) * kTileLz + i] = s;
  }
}

// End of step i: beta_i = ||x||; a column whose beta falls below 1e-12 max(1, |alpha_i|) or that took all
// kk steps stops with k_eff = i + 1 (keff < 0 while running). V_next = x / beta for running columns, zero
// otherwise (Vn null: no next vector). i < 0: normalises the start vector; a zero one marks an empty
// column (keff = 0). The blocks of a tile all form the same decision; the first one records it (a
// block that already reads the recorded keff comes to the same decision).
template <typename Real>
__global__ void __launch_bounds__(256)
k_lz_scale(Geo g, const Real* x, const double* __restrict__ nrm, int nch, int i, int kk, int k,
           const double* __restrict__ alpha, double* __restrict__ beta, int* keff, Real* Vn) {
  using V4 = typename LzV4<Real>::T;
  __shared__ Real bb_s[kTileLz], inv_s[kTileLz], low_s[kTileLz];   // beta, 1 / beta and its rounding error
  const int tl = blockIdx.y;
  if (threadIdx.x < kTileLz) {
    const size_t col = (size_t)tl * kTileLz + threadIdx.x;
    double s = 0.0;
    for (int c = 0; c < nch; ++c) s += nrm[((size_t)tl * nch + c) * kTileLz + threadIdx.x];
    const double b = sqrt(s);
    bool run;
    if (i < 0) {
      run = b > 0.0;
      if (blockIdx.x == 0) keff[col] = run ? -1 : 0;
    } else {
      const bool live = keff[col] < 0;
      const double a = alpha[col * k + i];
      const bool stop = i == kk - 1 || b <= 1e-12 * fmax(1.0, fabs(a));
      run = live && !stop;
      if (blockIdx.x == 0 && live) {
        beta[col * k + i] = b;
        if (stop) keff[col] = i + 1;
      }
    }
    const double r = run ? 1.0 / b : 0.0;
    bb_s[threadIdx.x] = run ? Real(b) : Real(0);
    inv_s[threadIdx.x] = Real(r);
    low_s[threadIdx.x] = Real(r - double(Real(r)));
  }
  __syncthreads();
  if (!Vn) return;
  const size_t n = (size_t)g.Upts * 2;
  const V4* xt = reinterpret_cast<const V4*>(x) + (size_t)tl * n;
  V4* vt = reinterpret_cast<V4*>(Vn) + (size_t)tl * n;
  const int h = 4 * (threadIdx.x & 1);
  Real bb[4], inv[4], low[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    bb[q] = bb_s[h + q];
    inv[q] = inv_s[h + q];
    low[q] = low_s[h + q];
  }
  // x / beta rounded once, without a division per element: FP64 corrects x (1 / beta) by its remainder,
  // FP32 takes 1 / beta as a pair of floats
  auto div = [&](Real v, int q) -> Real {
    if constexpr (sizeof(Real) == 8) {
      const Real t = v * inv[q];
      return fma(fma(-bb[q], t, v), inv[q], t);
    } else {
      return fmaf(v, inv[q], v * low[q]);
    }
  };
  for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < n; p += (size_t)gridDim.x * blockDim.x) {
    V4 t = xt[p];
    t.x = div(t.x, 0); t.y = div(t.y, 1); t.z = div(t.z, 2); t.w = div(t.w, 3);
    vt[p] = t;
  }
}

constexpr int kRitzWarps = 4;   // columns per block of the Ritz kernels

struct RitzBuf {
  double a[kMaxLanczos], b[kMaxLanczos], b2[kMaxLanczos];
  double y[2][kMaxLanczos], inv[2][kMaxLanczos];
};

// Number of eigenvalues of the tridiagonal (a, b) below x: the sign changes of the Sturm polynomials
// p_i = (a_i - x) p_{i-1} - b_{i-1}^2 p_{i-2}, rescaled by powers of two (three FP64 instructions a step;
// the ratio form needs a division, about 20).
__device__ __forceinline__ int sturm_count(const RitzBuf& r, int n, double x) {
  int cnt = 0;
  double p0 = 1.0, p1 = r.a[0] - x;
  if (p1 == 0.0) p1 = -1e-300;
  bool neg = p1 < 0.0;   // sign of p_i relative to p_{i-1}: a change is an eigenvalue below x
  cnt += neg;
  for (int i = 1; i < n; ++i) {
    double p2 = (r.a[i] - x) * p1 - r.b2[i - 1] * p0;
    if (p2 == 0.0) p2 = (p1 > 0.0) ? -1e-300 : 1e-300;   // a zero counts as a change, as in the ratio form
    cnt += (p2 < 0.0) != (p1 < 0.0);
    p0 = p1;
    p1 = p2;
    if ((i & 7) == 7) {
      const double m = fmax(fabs(p0), fabs(p1));
      if (m > 1e120) {
        p0 *= 0x1p-400;
        p1 *= 0x1p-400;
      } else if (m < 1e-120) {
        p0 *= 0x1p400;
        p1 *= 0x1p400;
      }
    }
  }
  return cnt;
}

// Extreme Ritz values of the tridiagonal of one column, widened by their residual norms
// |beta_last| |last component of the unit eigenvector|. One warp per column: lanes 0..15 bracket the
// smallest and lanes 16..31 the largest eigenvalue, 16 Sturm counts a round (a bisection by one
// thread, with a division per Sturm step, took 2.6 ms); then lanes 0 and 16 run three steps of inverse
// iteration with the shift just outside the spectrum (definite, so the unpivoted solve is stable).
__device__ void ritz_interval(RitzBuf& r, const double* __restrict__ a, const double* __restrict__ b, int n, double& lo,
                              double& hi) {
  const int lane = threadIdx.x & 31, half = lane >> 4, sub = lane & 15;
  const unsigned full = 0xffffffffu;
  __syncwarp();
  for (int i = lane; i < n; i += 32) {
    r.a[i] = a[i];
    r.b[i] = b[i];
    r.b2[i] = b[i] * b[i];
  }
  __syncwarp();
  double gl = INFINITY, gu = -INFINITY;   // Gershgorin interval
  for (int i = lane; i < n; i += 32) {
    const double w = (i > 0 ? fabs(r.b[i - 1]) : 0.0) + (i < n - 1 ? fabs(r.b[i]) : 0.0);
    gl = fmin(gl, r.a[i] - w);
    gu = fmax(gu, r.a[i] + w);
  }
  for (int d = 16; d > 0; d >>= 1) {
    gl = fmin(gl, __shfl_xor_sync(full, gl, d));
    gu = fmax(gu, __shfl_xor_sync(full, gu, d));
  }
  // a half's bracket (l, u]: the count at l is below the target, at u it is not
  const int target = half ? n : 1;
  double l = gl, u = gu;
  for (int it = 0; it < 64; ++it) {
    const double w = u - l;
    const bool open = w > 1e-15 * fmax(1.0, fmax(fabs(l), fabs(u)));
    if (!__any_sync(full, open)) break;
    const double x = l + w * (sub + 1) / 17.0;
    const unsigned m = (__ballot_sync(full, sturm_count(r, n, x) >= target) >> (16 * half)) & 0xffffu;
    const int first = m ? __ffs(m) - 1 : 16;   // first point of the half at or past the eigenvalue
    const double xu = __shfl_sync(full, x, 16 * half + min(first, 15));
    const double xl = __shfl_sync(full, x, 16 * half + max(first - 1, 0));
    if (open) {
      if (first < 16) u = xu;
      if (first > 0) l = xl;
    }
  }
  const double theta = 0.5 * (l + u);
  double res = fabs(r.b[n - 1]);
  if (n > 1 && sub == 0) {
    const double shift = half ? theta + 1e-10 * fmax(gu - gl, 1e-300) : theta - 1e-10 * fmax(gu - gl, 1e-300);
    double* y = r.y[half];
    double* inv = r.inv[half];
    inv[0] = 1.0 / (r.a[0] - shift);   // LDL^T of (T - shift I)
    y[0] = 1.0;
    for (int i = 1; i < n; ++i) {
      inv[i] = 1.0 / (r.a[i] - shift - r.b2[i - 1] * inv[i - 1]);
      y[i] = 1.0;
    }
    for (int it = 0; it < 3; ++it) {
      double t = y[0];
      for (int i = 1; i < n; ++i) {
        t = y[i] - r.b[i - 1] * inv[i - 1] * t;
        y[i] = t;
      }
      t = 0.0;
      double nr = 0.0;
      for (int i = n - 1; i >= 0; --i) {
        t = (i == n - 1) ? y[i] * inv[i] : (y[i] - r.b[i] * t) * inv[i];
        y[i] = t;
        nr += t * t;
      }
      nr = 1.0 / sqrt(nr);
      for (int i = 0; i < n; ++i) y[i] *= nr;
    }
    res *= fabs(y[n - 1]);
  }
  lo = __shfl_sync(full, theta, 0) - __shfl_sync(full, res, 0);
  hi = __shfl_sync(full, theta, 16) + __shfl_sync(full, res, 16);
}

// colb[2 col], colb[2 col + 1] = each column's widened Ritz extremes (an empty column: +inf, -inf)
__global__ void __launch_bounds__(32 * kRitzWarps)
k_lz_bounds(int ncols, int k, const double* __restrict__ alpha, const double* __restrict__ beta,
            const int* __restrict__ keff, double* __restrict__ colb) {
  __shared__ RitzBuf buf[kRitzWarps];
  const int col = blockIdx.x * kRitzWarps + (threadIdx.x >> 5);
  if (col >= ncols) return;
  double lo = INFINITY, hi = -INFINITY;
  if (keff[col] > 0)
    ritz_interval(buf[threadIdx.x >> 5], alpha + (size_t)col * k, beta + (size_t)col * k, keff[col], lo, hi);
  if ((threadIdx.x & 31) == 0) {
    colb[2 * col] = lo;
    colb[2 * col + 1] = hi;
  }
}

// min / max over the columns, widened by 1 % of the width; writes scal[8] = lo, scal[9] = hi.
__global__ void __launch_bounds__(256) k_lz_bounds_final(int ncols, const double* __restrict__ colb,
                                                         double* __restrict__ scal) {
  __shared__ double slo[256], shi[256];
  double lo = INFINITY, hi = -INFINITY;
  for (int col = threadIdx.x; col < ncols; col += blockDim.x) {
    lo = fmin(lo, colb[2 * col]);
    hi = fmax(hi, colb[2 * col + 1]);
  }
  slo[threadIdx.x] = lo;
  shi[threadIdx.x] = hi;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      slo[threadIdx.x] = fmin(slo[threadIdx.x], slo[threadIdx.x + s]);
      shi[threadIdx.x] = fmax(shi[threadIdx.x], shi[threadIdx.x + s]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double wdt = shi[0] - slo[0];
    scal[8] = slo[0] - 0.01 * wdt;
    scal[9] = shi[0] + 0.01 * wdt;
  }
}

// The per-node bounds mode: each column's own interval (Ritz extremes widened by their residual
// norms, then by 1 % of that column's width, as the shared interval is formed from all sample
// columns) and the step coefficients the recurrence of that node uses, with the scaling rules
// of set_bounds (SQ_MIXED: FP32-exact 2 / zeta and -2 chi / zeta; the diagonal coefficient
// rounded once; the stencil's constant-mode offset and that rounding folded into the centre).
__global__ void __launch_bounds__(32 * kRitzWarps)
k_lz_node_bounds(Geo g, Wave w, int k, const double* __restrict__ alpha, const double* __restrict__ beta,
                 const int* __restrict__ keff, int mixed, double lap_offset, double* __restrict__ nbnd,
                 double* __restrict__ ncoef) {
  __shared__ RitzBuf buf[kRitzWarps];
  const int col = blockIdx.x * kRitzWarps + (threadIdx.x >> 5);
  if (col >= w.ntiles * g.B) return;
  int o[3], qo[3];
  tile_origin(g, wave_tile(w, col / g.B), o);
  node_offset(g, col % g.B, qo);
  if (!node_valid(g, o, qo)) return;
  const int node = (o[0] + qo[0]) + g.n[0] * ((o[1] + qo[1]) + g.n[1] * (o[2] + qo[2]));
  const int n = keff[col];
  if (n <= 0) return;
  double lo, hi;
  ritz_interval(buf[threadIdx.x >> 5], alpha + (size_t)col * k, beta + (size_t)col * k, n, lo, hi);
  if ((threadIdx.x & 31) != 0) return;
  const double wdt = hi - lo;
  lo -= 0.01 * wdt;
  hi += 0.01 * wdt;
  // scaling of this node's recurrence (set_bounds, per node)
  double chi = 0.5 * (hi + lo), zeta = 0.5 * (hi - lo);
  double ca = 2.0 / zeta, cb = -2.0 * chi / zeta;
  if (mixed) {
    ca = double(float(ca));
    zeta = 2.0 / ca;
    cb = double(float(-2.0 * chi / zeta));
    chi = -cb * zeta / 2.0;
  }
  double cd = ca * g.lap0 + cb;
  if (mixed) cd = double(float(cd));
  const double eps = cd - (ca * g.lap0 + cb);
  chi -= lap_offset + eps / ca;
  nbnd[2 * node] = chi - zeta;
  nbnd[2 * node + 1] = chi + zeta;
  ncoef[2 * node] = ca;
  ncoef[2 * node + 1] = cd;
}

// k-step Lanczos (CGS2 reorthogonalisation) of every node column of the wave's tiles, from the
// hash start vector (start = 0, the spectral bounds) or from e_q (start = 1, Gauss SQ). V holds
// k + 1 vectors of the wave, W one, P the projections; C is (5 k + 8) doubles per column:
// cA, cB, nrm [ncols][k + 1], alpha, beta [ncols][k], keff (ints).
template <typename Real>
int lanczos_columns(sq_handle* h, const Wave& w, int start, int k, Real* V, Real* W, Real* P, double* C,
                    double* dots, WaveBufs* b) {
  const Geo& g = h->geo;
  cudaStream_t s = h->stream;
  const int nst = w.ntiles;
  // never more steps than the region has dimensions (the Krylov space is exhausted)
  const long long nc = (long long)(2 * g.m[0] + 1) * (2 * g.m[1] + 1) * (2 * g.m[2] + 1);
  const int kk = int(std::min<long long>(k, nc));
  const int ncols = nst * g.B;
  const int ld = k + 1;
  const size_t vstride = (size_t)nst * g.Upts * g.B;
  // dots holds the partial products of two passes and the norms; a wave of more tiles than it holds has
  // one chunk per tile, in C.
  const int nch = lz_chunks(nst, g.Upts);
  const bool small = nch * nst <= kLzChunkTiles;
  const size_t set = (size_t)nch * nst * ld * kTileLz;
  double* cA = small ? dots : C;
  double* cB = cA + set;
  double* nrm = cB + set;
  double* alpha = C + (size_t)3 * ncols * ld;
  double* beta = alpha + (size_t)ncols * k;
  int* keff = (int*)(beta + (size_t)ncols * k);
  const int eb = 1024;
  const dim3 og(nch, nst);
  const dim3 sg(std::max(1, std::min((2 * g.Upts + 255) / 256, 8 * 152 / std::max(1, nst) + 1)), nst);
  // the sample tiles' lists (their own buffers) only change with the atoms; a graph capture
  // records the build
  int rc = SQ_OK;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  SQ_CUDA_TRY(h, cudaStreamIsCapturing(s, &cap));
  if (b != &h->lzb || !h->keep_lists || h->lz_lists_epoch != h->atoms_epoch || cap != cudaStreamCaptureStatusNone) {
    rc = build_wave_entries(h, w, b);
    if (rc != SQ_OK) return rc;
    if (b == &h->lzb) h->lz_lists_epoch = h->atoms_epoch;
  }
  if (start == 0) k_lz_init<Real><<<eb, 256, 0, s>>>(g, w, V);
  else k_lz_init_unit<Real><<<eb, 256, 0, s>>>(g, w, V);
  SQ_LAUNCH_CHECK(h);
  const size_t xsb = 4 * sizeof(Real) * kLzThreads, acc1 = sizeof(double) * kTileLz;   // x of a round, sums per product
  k_lz_ortho<Real, kLzNorm><<<og, kLzThreads, xsb + acc1 * kLzWarps, s>>>(g, V, 0, vstride, V, nullptr, nrm, ld, k, nullptr);
  SQ_LAUNCH_CHECK(h);
  k_lz_scale<Real><<<sg, 256, 0, s>>>(g, V, nrm, nch, -1, kk, k, alpha, beta, keff, V);
  SQ_LAUNCH_CHECK(h);
  for (int i = 0; i < kk; ++i) {
    Real* Vi = V + (size_t)i * vstride;
    const int nv = i + 1;
    const size_t cfb = sizeof(Real) * nv * kTileLz;
    rc = launch_apply_h(h, w, Vi, W, P, *b);
    if (rc != SQ_OK) return rc;
    k_lz_ortho<Real, kLzDots><<<og, kLzThreads, xsb + acc1 * nv, s>>>(g, V, nv, vstride, W, nullptr, cA, ld, k, nullptr);
    SQ_LAUNCH_CHECK(h);
    k_lz_ortho<Real, kLzUpdateDots><<<og, kLzThreads, xsb + acc1 * nv + cfb, s>>>(g, V, nv, vstride, W, cA, cB, ld, k, alpha);
    SQ_LAUNCH_CHECK(h);
    k_lz_ortho<Real, kLzUpdateNorm><<<og, kLzThreads, xsb + acc1 * kLzWarps + cfb, s>>>(g, V, nv, vstride, W, cB, nrm, ld, k, alpha);
    SQ_LAUNCH_CHECK(h);
    k_lz_scale<Real><<<sg, 256, 0, s>>>(g, W, nrm, nch, i, kk, k, alpha, beta, keff,
                                        i < kk - 1 ? V + (size_t)(i + 1) * vstride : (Real*)nullptr);
    SQ_LAUNCH_CHECK(h);
  }
  return SQ_OK;
}

template int lanczos_columns<float>(sq_handle*, const Wave&, int, int, float*, float*, float*, double*, double*, WaveBufs*);
template int lanczos_columns<double>(sq_handle*, const Wave&, int, int, double*, double*, double*, double*, double*, WaveBufs*);

template <typename Real>
static int run_lanczos_t(sq_handle* h) {
  const int nst = int(h->lanczos_tiles.size());
  const int k = h->lanczos_k;
  const int ncols = nst * h->geo.B;
  const Wave w{0, nst, h->d.lz_tiles};
  // the sample tiles' lists go to their own buffers, so the sweep's lists (and W) stay valid
  int rc = lanczos_columns<Real>(h, w, 0, k, reinterpret_cast<Real*>(h->d.lzV), reinterpret_cast<Real*>(h->d.lzW),
                                 reinterpret_cast<Real*>(h->d.lzP), h->d.lzC, h->d.lzdot, &h->lzb);
  if (rc != SQ_OK) return rc;
  const double* alpha = h->d.lzC + (size_t)3 * ncols * (k + 1);
  const double* beta = alpha + (size_t)ncols * k;
  const int* keff = (const int*)(beta + (size_t)ncols * k);
  cudaStream_t s = h->stream;
  double* colb = h->d.lzC + (size_t)2 * ncols * (k + 1);   // the norms' slots, free after the last step
  k_lz_bounds<<<(ncols + kRitzWarps - 1) / kRitzWarps, 32 * kRitzWarps, 0, s>>>(ncols, k, alpha, beta, keff, colb);
  SQ_LAUNCH_CHECK(h);
  k_lz_bounds_final<<<1, 256, 0, s>>>(ncols, colb, h->d.scal);
  SQ_LAUNCH_CHECK(h);
  return set_bounds_device(h);   // no host round trip: the whole evaluation can be graph-captured
}

// set_bounds on the device, from the Lanczos interval scal[8], scal[9]: the step coefficients
// ca = 2 / zeta, cb = -2 chi / zeta, cd = ca lap0 + cb (SQ_MIXED: FP32-exact ca and cb, cd rounded
// once) and the effective interval the recurrence realises (centre moved by the stored
// stencil's constant-mode offset and cd's rounding) in scal[0], scal[1], scal[4..6]. Explicit
// rounding intrinsics keep every product and sum separately rounded, as in set_bounds.
__global__ void k_set_bounds(double* __restrict__ scal, double lap0, double lap_offset, int mixed, int* __restrict__ status) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double lo = scal[8], hi = scal[9];
  if (!(lo < hi) || !isfinite(lo) || !isfinite(hi)) {
    status[kStBadBounds] = 1;
    return;
  }
  status[kStBadBounds] = 0;
  double chi = __dmul_rn(0.5, __dadd_rn(hi, lo)), zeta = __dmul_rn(0.5, __dsub_rn(hi, lo));
  double ca = __ddiv_rn(2.0, zeta), cb = __ddiv_rn(__dmul_rn(-2.0, chi), zeta);
  if (mixed) {
    ca = double(__double2float_rn(ca));
    zeta = __ddiv_rn(2.0, ca);
    cb = double(__double2float_rn(__ddiv_rn(__dmul_rn(-2.0, chi), zeta)));
    chi = __ddiv_rn(__dmul_rn(-cb, zeta), 2.0);
  }
  const double exact = __dadd_rn(__dmul_rn(ca, lap0), cb);
  const double cd = mixed ? double(__double2float_rn(exact)) : exact;
  const double eps = __dsub_rn(cd, exact);
  chi = __dsub_rn(chi, __dadd_rn(lap_offset, __ddiv_rn(eps, ca)));
  scal[0] = __dsub_rn(chi, zeta);
  scal[1] = __dadd_rn(chi, zeta);
  scal[4] = ca;
  scal[5] = cb;
  scal[6] = cd;
}

int set_bounds_device(sq_handle* h) {
  k_set_bounds<<<1, 32, 0, h->stream>>>(h->d.scal, h->geo.lap0, h->lap_offset, h->precision == SQ_MIXED, h->d.status);
  SQ_LAUNCH_CHECK(h);
  return SQ_OK;
}

// Per-node bounds: every node column of the handle's tiles, in waves of nlz_wave tiles.
template <typename Real>
static int run_lanczos_nodes_t(sq_handle* h) {
  const Geo& g = h->geo;
  const int k = h->lanczos_k;
  for (int t0 = h->tile_begin; t0 < h->tile_end; t0 += h->nlz_wave) {
    const Wave w{t0, std::min(h->nlz_wave, h->tile_end - t0), nullptr};
    int rc = lanczos_columns<Real>(h, w, 0, k, reinterpret_cast<Real*>(h->d.nV), reinterpret_cast<Real*>(h->d.nW),
                                   reinterpret_cast<Real*>(h->d.nP), h->d.nC, h->d.lzdot, &h->wb);
    if (rc != SQ_OK) return rc;
    const int ncols = w.ntiles * g.B;
    const double* alpha = h->d.nC + (size_t)3 * ncols * (k + 1);
    const double* beta = alpha + (size_t)ncols * k;
    const int* keff = (const int*)(beta + (size_t)ncols * k);
    k_lz_node_bounds<<<(ncols + kRitzWarps - 1) / kRitzWarps, 32 * kRitzWarps, 0, h->stream>>>(g, w, k, alpha, beta, keff, h->precision == SQ_MIXED,
                                                               h->lap_offset, h->d.nbnd, h->d.ncoef);
    SQ_LAUNCH_CHECK(h);
  }
  // the extreme node bounds (sq_get_bounds)
  std::vector<double> b(2 * size_t(h->Nd));
  SQ_CUDA_TRY(h, cudaMemcpyAsync(b.data(), h->d.nbnd, sizeof(double) * b.size(), cudaMemcpyDeviceToHost, h->stream));
  SQ_CUDA_TRY(h, cudaStreamSynchronize(h->stream));
  double lo = INFINITY, hi = -INFINITY;
  for (int q = 0; q < h->Nd; ++q) {
    if (!(b[2 * q] < b[2 * q + 1]) || !std::isfinite(b[2 * q]) || !std::isfinite(b[2 * q + 1]))
      return fail(h, SQ_ERR_CUDA, "per-node Lanczos bounds are not finite");
    lo = std::min(lo, b[2 * q]);
    hi = std::max(hi, b[2 * q + 1]);
  }
  h->lam_lo = lo;
  h->lam_hi = hi;
  return SQ_OK;
}

int run_lanczos_nodes(sq_handle* h) {
  if (h->lanczos_k + 1 > kMaxLanczosVecs) return fail(h, SQ_ERR_INVALID_ARG, "lanczos_k too large");
  if (h->precision == SQ_MIXED) return run_lanczos_nodes_t<float>(h);
  return run_lanczos_nodes_t<double>(h);
}

int run_lanczos(sq_handle* h) {
  if (h->lanczos_k + 1 > kMaxLanczosVecs) return fail(h, SQ_ERR_INVALID_ARG, "lanczos_k too large");
  if (h->precision == SQ_MIXED) return run_lanczos_t<float>(h);
  return run_lanczos_t<double>(h);
}

}  // namespace sq
