// Device-side helpers shared by the SQ kernels.
#pragma once

#include <cooperative_groups.h>

#include "sq_internal.h"

namespace sq {

__device__ __forceinline__ int floor_div_d(int a, int b) { return (a >= 0) ? a / b : -((-a + b - 1) / b); }
__device__ __forceinline__ int ceil_div_d(int a, int b) { return -floor_div_d(-a, b); }

// Tile t (global index) -> origin of its first node in lattice coordinates.
__device__ __forceinline__ void tile_origin(const Geo& g, int t, int o[3]) {
  o[0] = (t % g.tiles[0]) * g.b;
  o[1] = ((t / g.tiles[0]) % g.tiles[1]) * g.b;
  o[2] = (t / (g.tiles[0] * g.tiles[1])) * g.b;
}

__device__ __forceinline__ int wave_tile(const Wave& w, int tl) { return w.ids ? w.ids[tl] : w.tile0 + tl; }

// Node slot q of a tile -> offsets inside the tile.
__device__ __forceinline__ void node_offset(const Geo& g, int q, int qo[3]) {
  qo[0] = q % g.b;
  qo[1] = (q / g.b) % g.b;
  qo[2] = q / (g.b * g.b);
}

__device__ __forceinline__ bool node_valid(const Geo& g, const int o[3], const int qo[3]) {
  return o[0] + qo[0] < g.n[0] && o[1] + qo[1] < g.n[1] && o[2] + qo[2] < g.n[2];
}

// Is U-local point (ux, uy, uz) inside the window of the node with offsets qo?
__device__ __forceinline__ bool in_window(const Geo& g, const int qo[3], int ux, int uy, int uz) {
  return (unsigned)(ux - qo[0]) <= (unsigned)(2 * g.m[0]) &&
         (unsigned)(uy - qo[1]) <= (unsigned)(2 * g.m[1]) &&
         (unsigned)(uz - qo[2]) <= (unsigned)(2 * g.m[2]);
}

// x = hi + lo with hi, lo TF32 values (11 significant bits each, held in FP32 registers): hi by Dekker's
// split (x rounded to 24 - 13 bits), lo, exact in 12 bits and a sign, rounded to 11 by half an ulp and a mask.
// Six cheap instructions; cvt.rna.tf32 expands to about a dozen integer ones on this part and made the
// splits the largest share of the projector kernels' instructions. A NaN stays one through hi.
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
  const float t = __fmul_rn(x, 8193.f), h = __fsub_rn(t, __fsub_rn(t, x));
  hi = __float_as_uint(h);
  lo = (__float_as_uint(__fsub_rn(x, h)) + 0x1000u) & 0xffffe000u;
}

// d (16 x 8, FP32) += a (16 x 8, TF32, row) * b (8 x 8, TF32, col); fragment of lane (g, t),
// g = lane / 4, t = lane % 4: a = {(g, t), (g + 8, t), (g, t + 4), (g + 8, t + 4)},
// b = {(t, g), (t + 4, g)}, d = {(g, 2t), (g, 2t + 1), (g + 8, 2t), (g + 8, 2t + 1)}
__device__ __forceinline__ void mma_tf32(float d[4], const uint32_t a[4], const uint32_t b[2]) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// d = a * b, the same fragments. Sums longer than a product add these in FP32: the tensor core truncates where it
// adds to an accumulator, and 24 products into one accumulator came 10 times as far from 64 bits.
__device__ __forceinline__ void mma_tf32_set(float d[4], const uint32_t a[4], const uint32_t b[2]) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%10, %10, %10, %10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(0.f));
}

// Linear index of an absolute lattice point inside an atom image's support box, or -1.
__device__ __forceinline__ int box_index(const AtomTab& at, const int s[3], const int n[3],
                                         int ax, int ay, int az) {
  int lx = ax - s[0] * n[0] - at.lo[0];
  int ly = ay - s[1] * n[1] - at.lo[1];
  int lz = az - s[2] * n[2] - at.lo[2];
  if ((unsigned)lx >= (unsigned)at.dim[0] || (unsigned)ly >= (unsigned)at.dim[1] ||
      (unsigned)lz >= (unsigned)at.dim[2])
    return -1;
  return (lz * at.dim[1] + ly) * at.dim[0] + lx;
}

// Pointer to the channel group of box point li of an atom's table.
template <typename Real>
__device__ __forceinline__ const Real* chi_row(const Real* chi, const AtomTab& at, int li) {
  return chi + at.off + (long long)li * at.nchp;
}

// Exclusive block-wide scan of one int per thread (blockDim.x a multiple of 32, <= 1024).
// Deterministic; returns the exclusive prefix and writes the block total to *total.
__device__ __forceinline__ int block_exclusive_scan(int v, int* total) {
  __shared__ int warp_sums[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int x = v;
  for (int d = 1; d < 32; d <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int w = (lane < nw) ? warp_sums[lane] : 0;
    for (int d = 1; d < 32; d <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= d) w += y;
    }
    warp_sums[lane] = w;   // inclusive
  }
  __syncthreads();
  int excl = x - v + (warp > 0 ? warp_sums[warp - 1] : 0);
  *total = warp_sums[nw - 1];
  __syncthreads();
  return excl;
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}


// Fermi-Dirac occupation 1 / (1 + e^x), evaluated without overflow for any x.
__device__ __forceinline__ double fermi_occ(double x) {
  const double ex = exp(-fabs(x));
  return (x > 0.0) ? ex / (1.0 + ex) : 1.0 / (1.0 + ex);
}

// Deterministic block sum (blockDim.x a power of two, sh holds blockDim.x doubles).
__device__ __forceinline__ double block_sum_d(double v, double* sh) {
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  const double r = sh[0];
  __syncthreads();
  return r;
}

// Root finder of the Fermi level. The result is that of bisection from the whole bracket (N(mid) < N_e takes the
// upper half, until it is < 1e-13 max(1, |mid|) wide or after 200 halvings; mu = the final midpoint), also where a
// truncated expansion makes N(mu) rise and fall and N = N_e has several roots: bisection itself until N is
// shown to rise on all of the bracket, then a few Newton steps to its one root there (on ln N far from it: concave
// where the electrons are dilute), and the bisection's last interval is the cell of its grid that holds the root.
// Shown by N' and D = (4/M) sum_k g (1 - g) |F_k| / kT at an end of the bracket: their half sum and half difference are
// the terms that rise and those that fall, and g (1 - g) changes by at most a factor e^s over s kT, so N' > 0 on a
// bracket s kT wide where e^(2 s) (D - N') < D + N'. About 11 evaluations in place of bisection's 46 (each M
// exponentials).
struct FermiRoot {
  double lo, hi;       // bracket: of the bisection, then of the Newton steps
  double a, w;         // the bisection's when Newton took over: lower end, width
  double n_e, kT, mu;
  int it, halved;
  bool rises;
  // rising: N is known to rise everywhere
  __host__ __device__ void init(double l, double u, double ne, double kt, bool rising = false) {
    lo = l;
    hi = u;
    n_e = ne;
    kT = kt;
    mu = 0.5 * (l + u);
    it = halved = 0;
    rises = rising;
    a = l;
    w = u - l;
  }
  // the midpoint of the bisection's last interval around the root r
  __host__ __device__ double cell(double r) const {
    const double am = fabs(r), tol = 1e-13 * (am > 1.0 ? am : 1.0);
    int k;
    frexp(w / tol, &k);
    if (k > 1 && ldexp(w, 1 - k) < tol) --k;
    k = k < 1 ? 1 : k;
    k = k > 200 - halved ? 200 - halved : k;
    const double s = ldexp(w, -k);
    return a + (floor((r - a) / s) + 0.5) * s;
  }
  // n, dn, ad: N, dN/dmu and D at mu; true when done (mu is then the result)
  __host__ __device__ bool update(double n, double dn, double ad) {
    ++it;
    const bool below = n < n_e;
    if (below) lo = mu;
    else hi = mu;
    const double am = fabs(mu), tol = 1e-13 * (am > 1.0 ? am : 1.0);
    if (!rises) {
      ++halved;
      if (hi - lo < tol || halved >= 200) {
        mu = 0.5 * (lo + hi);
        return true;
      }
      const double s = (hi - lo) / kT;
      const double down = (ad > dn ? ad - dn : 0.0) + 1e-13 * ad;   // (with the sums' rounding)
      if (!(dn > 0.0 && s < 20.0 && double(expf(2.0f * float(s))) * 1.00001 * down < ad + dn)) {
        mu = 0.5 * (lo + hi);
        return false;
      }
      rises = true;
      a = lo;
      w = hi - lo;
    }
    if (hi - lo < 0.02 * tol || it >= 200) {
      mu = cell(0.5 * (lo + hi));
      return true;
    }
    double next = lo;   // outside the open bracket: midpoint
    if (it < 64 && dn > 0.0) {
      const double miss = n_e - n, step = (fabs(miss) < 0.05 * n_e || n <= 0.0) ? miss / dn : log(n_e / n) * n / dn;
      next = mu + step;
      // the step's own error is below step^2 D / (kT N') for short steps
      if (fabs(step) < 0.1 * kT && step * step * ad < 0.01 * tol * kT * dn && next >= a && next <= a + w) {
        mu = cell(next);
        return true;
      }
    }
    mu = (next > lo && next < hi) ? next : 0.5 * (lo + hi);
    return false;
  }
};

// N(mu) = 2 sum'_j c^j(mu) R^j = (4/M) sum_k g((chi + zeta cos theta_k - mu) / kT) F_k with
// F_k = sum'_j cos(j theta_k) R^j, theta_k = pi (k + 1/2) / M (the M-point Chebyshev-Gauss rule
// for the coefficient integral of Sec. 4), and its root N(mu) = N_e on
// [lam_lo - 40 kT, lam_hi + 40 kT]. One cluster of kFermiCluster blocks: M FP64 exponentials per
// evaluation are bound by the 1.7 FP64 lanes per clock of an SM (one block: 43 us at M = 2048), so the
// points are spread over 8 SMs and the blocks' sums meet in distributed shared memory, two barriers'
// worth of slots so that one cluster barrier per evaluation suffices. Every thread adds the same
// numbers in the same order, so all blocks take the same steps. Returns false (and leaves *mu alone)
// when N(mu) - N_e has no sign change on the bracket.
constexpr int kFermiCluster = 8, kFermiThreads = 256;

__device__ __forceinline__ bool fermi_cluster_search(const double* __restrict__ F, int M, double lam_lo, double lam_hi,
                                                    double kT, double n_e, double* mu) {
  namespace cg = cooperative_groups;
  const cg::cluster_group cl = cg::this_cluster();
  const int rank = int(cl.block_rank());
  const double chi_q = 0.5 * (lam_hi + lam_lo), zeta_q = 0.5 * (lam_hi - lam_lo);
  constexpr int kWarps = kFermiThreads / 32;
  constexpr int kPts = SQ_NOALLOC_MAX_M / (kFermiCluster * kFermiThreads);   // most points per thread
  __shared__ double sums[2][3][kWarps];   // [slot][N, dN/dmu, D][warp]
  double lam[kPts], f[kPts];
  int np = 0;
#pragma unroll
  for (int i = 0; i < kPts; ++i) {
    const int k = (i * kFermiCluster + rank) * kFermiThreads + threadIdx.x;
    lam[i] = f[i] = 0.0;
    if (k < M) {
      lam[i] = chi_q + zeta_q * cospi((k + 0.5) / M);
      f[i] = F[k];
      np = i + 1;
    }
  }
  int slot = 0;
  auto count = [&](double x, double& n, double& dn, double& ad) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
#pragma unroll
    for (int i = 0; i < kPts; ++i)
      if (i < np) {
        const double g = fermi_occ((lam[i] - x) / kT), gf = g * f[i];
        s0 += gf;
        const double d = gf * (1.0 - g);
        s1 += d;
        s2 += fabs(d);
      }
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
    s2 = warp_sum(s2);
    if ((threadIdx.x & 31) == 0) {
      sums[slot][0][threadIdx.x >> 5] = s0;
      sums[slot][1][threadIdx.x >> 5] = s1;
      sums[slot][2][threadIdx.x >> 5] = s2;
    }
    cl.sync();
    const int lane = threadIdx.x & 31;   // lanes: 8 blocks x 4 warps each, then the other 4 warps
    static_assert(kFermiCluster == 8 && kWarps == 8, "one lane per block and half of its warps");
    const double* r = cl.map_shared_rank(&sums[slot][0][0], lane >> 2);
    const int w = lane & 3;
    n = 4.0 / M * warp_sum(r[w] + r[w + 4]);
    dn = 4.0 / M / kT * warp_sum(r[kWarps + w] + r[kWarps + w + 4]);
    ad = 4.0 / M / kT * warp_sum(r[2 * kWarps + w] + r[2 * kWarps + w + 4]);
    slot ^= 1;
  };
  const double lo = lam_lo - 40.0 * kT, hi = lam_hi + 40.0 * kT;
  double n0, n1, dn, ad;
  count(lo, n0, dn, ad);
  count(hi, n1, dn, ad);
  bool ok = n0 < n_e && n_e < n1;
  if (ok) {
    FermiRoot r;
    r.init(lo, hi, n_e, kT);
    do count(r.mu, n0, dn, ad);
    while (!r.update(n0, dn, ad));
    *mu = r.mu;
  }
  cl.sync();   // no block leaves while another still reads its sums
  return ok;
}

// ---- cross-thread sums: doubles for FP64 vectors, pairs of floats (two-sum, about 2^-47 relative, on terms rounded
// to 2^-24) for FP32 ones; FP64 adds issue at 1.7 lanes per clock and SM and cost more than the products they sum.
struct FloatPair { float h, l; };

__device__ __forceinline__ FloatPair lz_add(FloatPair a, FloatPair b) {   // Knuth's two-sum, tails added
  const float s = __fadd_rn(a.h, b.h), z = __fsub_rn(s, a.h);
  const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, z)), __fsub_rn(b.h, z));
  const float t = __fadd_rn(e, __fadd_rn(a.l, b.l)), h = __fadd_rn(s, t);
  return {h, __fsub_rn(t, __fsub_rn(h, s))};
}
__device__ __forceinline__ double lz_add(double a, double b) { return a + b; }
__device__ __forceinline__ FloatPair lz_shfl(FloatPair a, int m) {
  return {__shfl_xor_sync(0xffffffffu, a.h, m), __shfl_xor_sync(0xffffffffu, a.l, m)};
}
__device__ __forceinline__ double lz_shfl(double a, int m) { return __shfl_xor_sync(0xffffffffu, a, m); }
__device__ __forceinline__ double lz_double(FloatPair a) { return double(a.h) + double(a.l); }
__device__ __forceinline__ double lz_double(double a) { return a; }
template <typename Real> struct LzAcc;
template <> struct LzAcc<float> {
  using T = FloatPair;
  static __device__ __forceinline__ T make(float x) { return {x, 0.f}; }
};
template <> struct LzAcc<double> {
  using T = double;
  static __device__ __forceinline__ T make(double x) { return x; }
};

// the four values of a lane (nodes 4 (lane & 1) .. + 3) added over the warp's 16 lanes of that parity by a
// reduce-scatter (5 exchanges in place of 16); lanes 0 .. 7 return node *node's sum
template <typename Real>
__device__ __forceinline__ typename LzAcc<Real>::T lz_warp_sum(const Real d[4], int* node) {
  using A = typename LzAcc<Real>::T;
  const int lane = threadIdx.x & 31, s0 = (lane >> 1) & 1, s1 = (lane >> 2) & 1;
  const A v0 = LzAcc<Real>::make(d[0]), v1 = LzAcc<Real>::make(d[1]), v2 = LzAcc<Real>::make(d[2]), v3 = LzAcc<Real>::make(d[3]);
  const A k0 = lz_add(s0 ? v2 : v0, lz_shfl(s0 ? v0 : v2, 2));
  const A k1 = lz_add(s0 ? v3 : v1, lz_shfl(s0 ? v1 : v3, 2));
  A k = lz_add(s1 ? k1 : k0, lz_shfl(s1 ? k0 : k1, 4));
  k = lz_add(k, lz_shfl(k, 8));
  k = lz_add(k, lz_shfl(k, 16));
  *node = 4 * (lane & 1) + 2 * s0 + s1;
  return k;
}

}  // namespace sq
