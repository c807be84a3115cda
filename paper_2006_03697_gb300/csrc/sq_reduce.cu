// Fermi level and contraction kernels (FP64).
//
//   R^j      = sum_q rho_q^j                                    (node sums, fixed order)
//   F_k      = sum'_j cos(j theta_k) R^j,  theta_k = pi (k + 1/2) / M
//   N(mu)    = 2 sum'_j c^j(mu) R^j = (4/M) sum_k g((chi + zeta cos theta_k - mu)/kT) F_k
// because c^j = (2/M) sum_k g(cos theta_k) cos(j theta_k) is the M-point Chebyshev-Gauss
// rule for the Clenshaw-Curtis coefficient integral of Sec. 4; bisection on N(mu) = N_e (FermiRoot).
// The contraction evaluates c^j, d^j (coefficients of r g(r), App. A) and s^j (entropy
// function) at mu and forms rho_q, E_band, E_s, E_nl and sigma (Sec. 4 stress sums).
#include <algorithm>
#include <cmath>

#include "sq_device.cuh"

namespace sq {

// g ln g + (1 - g) ln(1 - g) at g = fermi(x), stable form -[ln(1+e^-|x|) + |x| e^-|x|/(1+e^-|x|)]
__device__ __forceinline__ double entropy_d(double x) {
  const double ax = fabs(x), ex = exp(-ax);
  return -(log1p(ex) + ax * ex / (1.0 + ex));
}

__global__ void k_rsum(const double* __restrict__ mom, int Nd, int n_pl, double* __restrict__ R) {
  __shared__ double sh[256];
  const int j = blockIdx.x;
  double s = 0.0;
  for (int q = threadIdx.x; q < Nd; q += blockDim.x) s += mom[((size_t)q * (n_pl + 1) + j) * SQ_N_MOMENTS];
  s = block_sum_d(s, sh);
  if (threadIdx.x == 0) R[j] = s;
}

// F_k = sum'_j cos(j theta_k) R^j. Eight lanes per k split the j range (one lane per k left most of
// the FP64 pipes idle: 2048 threads on 8 SMs). tab (or null): cos(pi t / (2 M)), so that
// cos(j theta_k) = tab[j (2 k + 1) mod 4 M]; without it the cosines are evaluated here.
__global__ void __launch_bounds__(128) k_cosF(const double* __restrict__ R, int n_pl, int M, const double* __restrict__ tab,
                                              double* __restrict__ F) {
  const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 3, sub = threadIdx.x & 7;
  double s = 0.0;
  if (k < M) {
    const int odd = 2 * k + 1, M4 = 4 * M;
    for (int j = sub; j <= n_pl; j += 8) {
      const int t = int((long long)j * odd % M4);
      s += (j == 0) ? 0.5 * R[0] : (tab ? tab[t] : cospi(double(t) / (2.0 * M))) * R[j];
    }
  }
  for (int d = 4; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
  if (k < M && sub == 0) F[k] = s;
}

// scal[0], scal[1]: bounds; writes scal[2] = mu, status[kStNoBracket].
__global__ void __cluster_dims__(kFermiCluster, 1, 1) __launch_bounds__(kFermiThreads)
k_fermi(const double* __restrict__ F, int M, double kT, double n_e, double* __restrict__ scal, int* __restrict__ status) {
  double mu = 0.0;
  const bool ok = fermi_cluster_search(F, M, scal[0], scal[1], kT, n_e, &mu);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    scal[2] = ok ? mu : NAN;
    status[kStNoBracket] = ok ? 0 : 1;
  }
}

// The coefficients c, d (r g(r)) and s (entropy function) at mu, in two launches. One kernel with a
// block per function took 2.26 ms (M = 2048, n_pl = 60): FP64 issues 1.7 lanes per clock and SM
// here, and three SMs evaluated M (n_pl + 1) cosines each. Now the cosines come from the handle's
// table, k_fvals spreads the M exponentials over M / 64 blocks and k_coef takes one block per j: a
// density and a pressure call on a 5 x 4 x 6 cell together took 4.5 ms less.
//   k_fvals: fv[3][M] = g, r g, entropy at the Chebyshev-Gauss points; mu from scal[2] (from_scal) or
//            the argument, left in scal[3]
__global__ void __launch_bounds__(64) k_fvals(double* __restrict__ scal, double mu_arg, int from_scal, double kT, int M,
                                              const double* __restrict__ tab, double* __restrict__ fv) {
  const double lam_lo = scal[0], lam_hi = scal[1], mu = from_scal ? scal[2] : mu_arg;
  const double chi_q = 0.5 * (lam_hi + lam_lo), zeta_q = 0.5 * (lam_hi - lam_lo);
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k == 0) scal[3] = mu;
  if (k >= M) return;
  const double r = tab[2 * k + 1];
  const double x = (chi_q + zeta_q * r - mu) / kT;
  const double f = fermi_occ(x);
  fv[k] = f;
  fv[M + k] = r * f;
  fv[2 * M + k] = entropy_d(x);
}

// coef[w][j] = (2/M) sum_k fv[w][k] cos(j theta_k), one block per j
__global__ void __launch_bounds__(128) k_coef(const double* __restrict__ fv, int n_pl, int M,
                                              const double* __restrict__ tab, double* __restrict__ coef) {
  __shared__ double sh[3][4];
  const int j = blockIdx.x, M4 = 4 * M;
  double a[3] = {0.0, 0.0, 0.0};
  int t = int((long long)j * (2 * threadIdx.x + 1) % M4);              // j (2 k + 1) mod 4 M
  const int step = int((long long)j * (2 * int(blockDim.x)) % M4);
  for (int k = threadIdx.x; k < M; k += blockDim.x) {
    const double cs = tab[t];
    for (int w = 0; w < 3; ++w) a[w] += fv[w * M + k] * cs;
    t += step;
    if (t >= M4) t -= M4;
  }
  for (int w = 0; w < 3; ++w) {
    a[w] = warp_sum(a[w]);
    if ((threadIdx.x & 31) == 0) sh[w][threadIdx.x >> 5] = a[w];
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    const double* r = sh[threadIdx.x];
    coef[threadIdx.x * (n_pl + 1) + j] = 2.0 / M * ((r[0] + r[1]) + (r[2] + r[3]));
  }
}

constexpr int kNPart = 20;
constexpr int kContractThreads = 256;
constexpr int kContractGroups = kContractThreads / SQ_N_MOMENTS;   // j values in flight per node

// The contraction terms of nodes [q0, q1) with coefficients c, d, sc ([n_pl + 1] each) and one interval,
// left in part[kNPart] (whole block; red: kContractGroups * kNPart + 8 doubles of shared memory). A
// thread owns one moment slot and walks j, so a block reads whole contiguous moment rows (one
// thread per node read 136-byte strides on a few blocks: 80-114 us at 1,728-32,768 nodes).
__device__ void contract_block(const double* __restrict__ mom, const double* c, const double* d, const double* sc,
                               double chi_q, double zeta_q, const double* __restrict__ v, int q0, int q1, int n_pl,
                               double dV, double* __restrict__ rho, double* red, double* __restrict__ part) {
  const int slot = threadIdx.x % SQ_N_MOMENTS, grp = threadIdx.x / SQ_N_MOMENTS;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0;
  if (grp < kContractGroups) {
    for (int j = grp; j <= n_pl; j += kContractGroups) {
      const double* m = mom + ((size_t)q0 * (n_pl + 1) + j) * SQ_N_MOMENTS + slot;
      double s = 0.0;
#pragma unroll 4
      for (int q = q0; q < q1; ++q, m += (size_t)(n_pl + 1) * SQ_N_MOMENTS) s += *m;
      const double wp = (j == 0) ? 0.5 : 1.0;
      a0 += wp * c[j] * s;
      if (slot == 0) {
        a1 += wp * (chi_q * c[j] + zeta_q * d[j]) * s;
        a2 += wp * sc[j] * s;
      }
    }
    // slots: 0 E_band, 1 E_s, 2 N, 3..8 K, 9..17 S, 18 rho (19: V rho, below)
    double* r = red + grp * kNPart;
    if (slot == 0) {
      r[0] = a1;
      r[1] = a2;
      r[18] = a0;
    } else if (slot == 7) {
      r[2] = a0;
    } else {
      r[slot < 7 ? 2 + slot : slot + 1] = a0;
    }
  }
  // rho per node: one warp per node
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double ev = 0.0;
  for (int q = q0 + warp; q < q1; q += kContractThreads / 32) {
    double r = 0.0;
    for (int j = lane; j <= n_pl; j += 32)
      r += (j == 0 ? 0.5 : 1.0) * c[j] * mom[((size_t)q * (n_pl + 1) + j) * SQ_N_MOMENTS];
    r = warp_sum(r);
    if (lane == 0) {
      if (rho) rho[q] = 2.0 / dV * r;
      ev += v[q] * r;   // |dOmega| V_q rho_q / 2
    }
  }
  if (lane == 0) red[kContractGroups * kNPart + warp] = ev;
  __syncthreads();
  if (threadIdx.x < kNPart) {
    double t = 0.0;
    if (threadIdx.x == kNPart - 1)
      for (int w = 0; w < kContractThreads / 32; ++w) t += red[kContractGroups * kNPart + w];
    else
      for (int w = 0; w < kContractGroups; ++w) t += red[w * kNPart + threadIdx.x];
    part[threadIdx.x] = t;
  }
}

// block b: nodes [Nd b / nblk, Nd (b + 1) / nblk)
__global__ void __launch_bounds__(kContractThreads)
k_contract(const double* __restrict__ mom, const double* __restrict__ coef, const double* __restrict__ scal,
           const double* __restrict__ v, int Nd, int n_pl, double dV, double* __restrict__ rho, double* __restrict__ part) {
  __shared__ double red[kContractGroups * kNPart + kContractThreads / 32];
  const double lam_lo = scal[0], lam_hi = scal[1];
  const int q0 = int((long long)Nd * blockIdx.x / gridDim.x), q1 = int((long long)Nd * (blockIdx.x + 1) / gridDim.x);
  contract_block(mom, coef, coef + (n_pl + 1), coef + 2 * (n_pl + 1), 0.5 * (lam_hi + lam_lo), 0.5 * (lam_hi - lam_lo),
                 v, q0, q1, n_pl, dV, rho, red, part + (size_t)blockIdx.x * kNPart);
}

// rows of kNPart terms added up in a fixed order to gridDim.x rows (one warp per term)
__global__ void __launch_bounds__(32 * kNPart) k_sum_rows(const double* __restrict__ rows, int n, double* __restrict__ out) {
  const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
  const int r0 = int((long long)n * blockIdx.x / gridDim.x), r1 = int((long long)n * (blockIdx.x + 1) / gridDim.x);
  double s = 0.0;
  for (int r = r0 + lane; r < r1; r += 32) s += rows[(size_t)r * kNPart + k];
  s = warp_sum(s);
  if (lane == 0) out[blockIdx.x * kNPart + k] = s;
}

// out (scal + 16): [E_band, E_s, E_nl, N_check, sigma(9, row-major), E_pot, P]
// E_pot = |dOmega| sum_q V_q rho_q; P = the App. A pressure restricted to the kinetic and
// nonlocal terms: -(1/(3|Omega|)) [-2 (E_band - E_pot) - E_nl - 4 sum_q sum' c^j tr S^j_q]
// (the V_eff part of -4 tr(D H) goes with the exchange-correlation / electrostatic terms)
// One warp per term adds the nblk rows (one thread took 19-170 us, 2.2 ms for per-node rows).
__global__ void __launch_bounds__(32 * kNPart) k_contract_final(const double* __restrict__ part, int nblk, double kT,
                                                                double vol, double* __restrict__ scal) {
  __shared__ double tot[kNPart];
  {
    const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
    double s = 0.0;
    for (int b = lane; b < nblk; b += 32) s += part[b * kNPart + k];
    s = warp_sum(s);
    if (lane == 0) tot[k] = s;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  double* out = scal + 16;
  out[0] = 2.0 * tot[0];
  out[1] = 2.0 * kT * tot[1];
  const double E_nl = 2.0 * tot[2];
  out[2] = E_nl;
  out[3] = 2.0 * tot[18];   // |dOmega| sum_q rho_q = 2 sum_q sum' c rho^j
  const int ka[6] = {0, 1, 2, 1, 0, 0}, kb[6] = {0, 1, 2, 2, 2, 1};
  double sig[9];
  for (int k = 0; k < 9; ++k) sig[k] = 0.0;
  for (int k = 0; k < 6; ++k) {
    sig[3 * ka[k] + kb[k]] += 2.0 * tot[3 + k];
    if (ka[k] != kb[k]) sig[3 * kb[k] + ka[k]] += 2.0 * tot[3 + k];
  }
  for (int a = 0; a < 3; ++a)
    for (int b = 0; b < 3; ++b)
      sig[3 * a + b] += -2.0 * ((a == b ? 0.5 * E_nl : 0.0) + 2.0 * tot[9 + 3 * a + b]);
  for (int k = 0; k < 9; ++k) out[4 + k] = sig[k] / vol;
  const double E_pot = 2.0 * tot[19];
  out[13] = E_pot;
  out[14] = -(-2.0 * (out[0] - E_pot) - E_nl - 4.0 * (tot[9] + tot[13] + tot[17])) / (3.0 * vol);
}

// Fermi search on the node sums already in d.R (the whole cell's, or the caller's allreduced ones)
static int fermi_from_R(sq_handle* h, double* mu_out) {
  const Geo& g = h->geo;
  cudaStream_t s = h->stream;
  k_cosF<<<(h->M + 15) / 16, 128, 0, s>>>(h->d.R, g.n_pl, h->M, h->d.costab, h->d.cosF);
  SQ_LAUNCH_CHECK(h);
  k_fermi<<<kFermiCluster, kFermiThreads, 0, s>>>(h->d.cosF, h->M, h->kT, h->n_e, h->d.scal, h->d.status);
  SQ_LAUNCH_CHECK(h);
  double mu = 0.0;
  int st[kStCount];
  SQ_CUDA_TRY(h, cudaMemcpyAsync(&mu, h->d.scal + 2, sizeof(double), cudaMemcpyDeviceToHost, s));
  SQ_CUDA_TRY(h, cudaMemcpyAsync(st, h->d.status, sizeof(st), cudaMemcpyDeviceToHost, s));
  SQ_CUDA_TRY(h, cudaStreamSynchronize(s));
  if (st[kStBadBounds]) return fail(h, SQ_ERR_CUDA, "spectral bounds are not finite or empty");
  if (st[kStOverflow]) return fail(h, SQ_ERR_CUDA, "internal list capacity exceeded");
  if (st[kStNoBracket]) return fail(h, SQ_ERR_NO_BRACKET, "N(mu) - N_e has no sign change on the bisection bracket");
  if (mu_out) *mu_out = mu;
  return SQ_OK;
}

int run_fermi(sq_handle* h, double* mu_out) {
  k_rsum<<<h->geo.n_pl + 1, 256, 0, h->stream>>>(h->d.mom, h->Nd, h->geo.n_pl, h->d.R);
  SQ_LAUNCH_CHECK(h);
  return fermi_from_R(h, mu_out);
}

int run_node_sums(sq_handle* h, double* R_out) {
  cudaStream_t s = h->stream;
  k_rsum<<<h->geo.n_pl + 1, 256, 0, s>>>(h->d.mom, h->Nd, h->geo.n_pl, h->d.R);
  SQ_LAUNCH_CHECK(h);
  SQ_CUDA_TRY(h, cudaMemcpyAsync(R_out, h->d.R, sizeof(double) * (h->geo.n_pl + 1), cudaMemcpyDeviceToHost, s));
  SQ_CUDA_TRY(h, cudaStreamSynchronize(s));
  return SQ_OK;
}

int run_fermi_sums(sq_handle* h, const double* R_host, double* mu_out) {
  SQ_CUDA_TRY(h, cudaMemcpyAsync(h->d.R, R_host, sizeof(double) * (h->geo.n_pl + 1), cudaMemcpyHostToDevice,
                                 h->stream));
  return fermi_from_R(h, mu_out);
}

// Coefficients and contraction at mu (from_scal: the Fermi level in scal[2]); outputs in scal[16 ..].
static int contract_launches(sq_handle* h, double mu, int from_scal, double* rho_dev) {
  const Geo& g = h->geo;
  cudaStream_t s = h->stream;
  k_fvals<<<(h->M + 63) / 64, 64, 0, s>>>(h->d.scal, mu, from_scal, h->kT, h->M, h->d.costab, h->d.fvals);
  SQ_LAUNCH_CHECK(h);
  k_coef<<<g.n_pl + 1, 128, 0, s>>>(h->d.fvals, g.n_pl, h->M, h->d.costab, h->d.coef);
  SQ_LAUNCH_CHECK(h);
  // four blocks per SM, at least two nodes each (d.part holds 4096 * 32 doubles)
  const int nblk = std::max(1, std::min(4 * 152, (h->Nd + 1) / 2));
  k_contract<<<nblk, kContractThreads, 0, s>>>(h->d.mom, h->d.coef, h->d.scal, h->d.v64, h->Nd, g.n_pl, g.dV, rho_dev,
                                               h->d.part);
  SQ_LAUNCH_CHECK(h);
  k_contract_final<<<1, 32 * kNPart, 0, s>>>(h->d.part, nblk, h->kT, h->vol, h->d.scal);
  SQ_LAUNCH_CHECK(h);
  return SQ_OK;
}

// The Fermi level and the contraction with nothing crossing to the host (graph capture): mu
// stays in scal[2] (NaN and the no-bracket status word when there is no sign change), the
// contraction takes it from there and leaves its outputs in scal[16 ..].
int run_fermi_contraction_device(sq_handle* h) {
  const Geo& g = h->geo;
  cudaStream_t s = h->stream;
  k_rsum<<<g.n_pl + 1, 256, 0, s>>>(h->d.mom, h->Nd, g.n_pl, h->d.R);
  SQ_LAUNCH_CHECK(h);
  k_cosF<<<(h->M + 15) / 16, 128, 0, s>>>(h->d.R, g.n_pl, h->M, h->d.costab, h->d.cosF);
  SQ_LAUNCH_CHECK(h);
  k_fermi<<<kFermiCluster, kFermiThreads, 0, s>>>(h->d.cosF, h->M, h->kT, h->n_e, h->d.scal, h->d.status);
  SQ_LAUNCH_CHECK(h);
  return contract_launches(h, 0.0, 1, h->d.rho);
}

int run_contraction(sq_handle* h, double mu, double* rho_dev, double* out_host) {
  cudaStream_t s = h->stream;
  const int rc = contract_launches(h, mu, 0, rho_dev);
  if (rc != SQ_OK) return rc;
  if (out_host) {
    SQ_CUDA_TRY(h, cudaMemcpyAsync(out_host, h->d.scal + 16, 15 * sizeof(double), cudaMemcpyDeviceToHost, s));
    SQ_CUDA_TRY(h, cudaStreamSynchronize(s));
  }
  return SQ_OK;
}


// ---------------------------------------------------------------- per-node bounds mode
// Every node q has its own interval (chi_q, zeta_q) and so its own coefficients
// c_q^j(mu) = (2/M) sum_k g((chi_q + zeta_q cos theta_k - mu)/kT) cos(j theta_k), and
//   N(mu) = 2 sum_q sum'_j c_q^j rho_q^j = (4/M) sum_q sum_k g(...) F_q(k),
//   F_q(k) = sum'_j cos(j theta_k) rho_q^j      (one table of N_d x M, formed once per search).
// tab[t] = cos(pi t / (2 M)), so cos(j theta_k) = tab[j (2 k + 1) mod 4 M].

// F_q(k) for k and M - 1 - k together: cos(j theta_{M-1-k}) = (-1)^j cos(j theta_k), so the even and the odd
// part are summed once (half the FP64 multiply-adds).
__global__ void __launch_bounds__(256) k_cosF_nodes(const double* __restrict__ mom, int Nd, int n_pl, int M,
                                                    const double* __restrict__ tab, double* __restrict__ F) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x, q = blockIdx.y;
  if (k >= (M + 1) / 2 || q >= Nd) return;
  const double* m = mom + (size_t)q * (n_pl + 1) * SQ_N_MOMENTS;
  const int M4 = 4 * M, odd = 2 * k + 1;
  double s[2] = {0.5 * m[0], 0.0};
  int t = 0;
  for (int j = 1; j <= n_pl; j += 2) {
    t += odd;
    if (t >= M4) t -= M4;
    s[1] += tab[t] * m[(size_t)j * SQ_N_MOMENTS];
    if (j == n_pl) break;
    t += odd;
    if (t >= M4) t -= M4;
    s[0] += tab[t] * m[(size_t)(j + 1) * SQ_N_MOMENTS];
  }
  F[(size_t)q * M + k] = s[0] + s[1];
  F[(size_t)q * M + M - 1 - k] = s[0] - s[1];   // k = M - 1 - k: the odd part is zero there
}

// part[3 block ..] = N, dN/dmu and D (FermiRoot) of the block's nodes: (4/M) sum_q sum_k
// g((chi_q + zeta_q cos theta_k - mu)/kT) F_q(k), g (1 - g) / kT in place of g, and that with |F_q(k)|
__global__ void __launch_bounds__(256) k_count_nodes(const double* __restrict__ F, const double* __restrict__ nbnd, int Nd,
                                                     int M, const double* __restrict__ tab, double kT, double mu,
                                                     double* __restrict__ part) {
  __shared__ double sh[256];
  double a0 = 0.0, a1 = 0.0, a2 = 0.0;
  for (int q = blockIdx.x; q < Nd; q += gridDim.x) {
    const double lo = nbnd[2 * q], hi = nbnd[2 * q + 1];
    const double chi_q = 0.5 * (hi + lo), zeta_q = 0.5 * (hi - lo);
    const double* Fq = F + (size_t)q * M;
    for (int k = threadIdx.x; k < M; k += blockDim.x) {
      const double g = fermi_occ((chi_q + zeta_q * tab[2 * k + 1] - mu) / kT), gf = g * Fq[k];
      a0 += gf;
      const double d = gf * (1.0 - g);
      a1 += d;
      a2 += fabs(d);
    }
  }
  a0 = block_sum_d(a0, sh);
  a1 = block_sum_d(a1, sh);
  a2 = block_sum_d(a2, sh);
  if (threadIdx.x == 0) {
    part[3 * blockIdx.x] = 4.0 / M * a0;
    part[3 * blockIdx.x + 1] = 4.0 / M / kT * a1;
    part[3 * blockIdx.x + 2] = 4.0 / M / kT * a2;
  }
}

// part[3 block], part[3 block + 1] = the block's shares of (4/M) sum F and (4/M) sum |F| over all nodes and points
__global__ void __launch_bounds__(256) k_F_sums(const double* __restrict__ F, size_t n, int M, double* __restrict__ part) {
  __shared__ double sh[256];
  double a0 = 0.0, a1 = 0.0;
  for (size_t i = blockIdx.x * (size_t)256 + threadIdx.x; i < n; i += (size_t)gridDim.x * 256) {
    a0 += F[i];
    a1 += fabs(F[i]);
  }
  a0 = block_sum_d(a0, sh);
  a1 = block_sum_d(a1, sh);
  if (threadIdx.x == 0) {
    part[3 * blockIdx.x] = 4.0 / M * a0;
    part[3 * blockIdx.x + 1] = 4.0 / M * a1;
    part[3 * blockIdx.x + 2] = 0.0;
  }
}

// out[0 .. 2] = sums of the (N, dN/dmu, D) triples, fixed order; with nbnd: out[3] = min lo_q,
// out[4] = max hi_q. One block of 256.
__global__ void __launch_bounds__(256) k_sum_parts(const double* __restrict__ part, int n, const double* __restrict__ nbnd,
                                                   int Nd, double* __restrict__ out) {
  __shared__ double sh[256], slo[256], shi[256];
  for (int c = 0; c < 3; ++c) {
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += part[3 * i + c];
    s = block_sum_d(s, sh);
    if (threadIdx.x == 0) out[c] = s;
  }
  if (!nbnd) return;
  double lo = INFINITY, hi = -INFINITY;
  for (int q = threadIdx.x; q < Nd; q += blockDim.x) {
    lo = fmin(lo, nbnd[2 * q]);
    hi = fmax(hi, nbnd[2 * q + 1]);
  }
  slo[threadIdx.x] = lo;
  shi[threadIdx.x] = hi;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      slo[threadIdx.x] = fmin(slo[threadIdx.x], slo[threadIdx.x + w]);
      shi[threadIdx.x] = fmax(shi[threadIdx.x], shi[threadIdx.x + w]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[3] = slo[0];
    out[4] = shi[0];
  }
}

// Blocks of k_count_nodes, three per SM: it is bound by the SMs' FP64 units, and 512 blocks left some SMs a third
// more of them than others (1728 nodes: 332 -> 285 us). d.npart holds a triple per block.
constexpr int kCountBlocks = 3 * 152;
static_assert(3 * kCountBlocks <= kNodeParts, "d.npart");

int run_fermi_nodes(sq_handle* h, double* mu_out) {
  const Geo& g = h->geo;
  cudaStream_t s = h->stream;
  const int M = h->M;
  k_cosF_nodes<<<dim3(((M + 1) / 2 + 255) / 256, h->Nd), 256, 0, s>>>(h->d.mom, h->Nd, g.n_pl, M, h->d.costab, h->d.nF);
  SQ_LAUNCH_CHECK(h);
  double* out = h->d.scal + 40;   // [N, dN/dmu, D, min lo, max hi]
  // ext: (4/M) sum F and sum |F| and the interval of all nodes (an evaluation is bound by its N_d M FP64
  // exponentials: 0.28 ms at 12^3)
  auto count = [&](double mu, double* res, bool ext) -> int {
    if (ext) k_F_sums<<<kCountBlocks, 256, 0, s>>>(h->d.nF, (size_t)h->Nd * M, M, h->d.npart);
    else k_count_nodes<<<kCountBlocks, 256, 0, s>>>(h->d.nF, h->d.nbnd, h->Nd, M, h->d.costab, h->kT, mu, h->d.npart);
    SQ_LAUNCH_CHECK(h);
    k_sum_parts<<<1, 256, 0, s>>>(h->d.npart, kCountBlocks, ext ? h->d.nbnd : nullptr, h->Nd, out);
    SQ_LAUNCH_CHECK(h);
    SQ_CUDA_TRY(h, cudaMemcpyAsync(res, out, (ext ? 5 : 3) * sizeof(double), cudaMemcpyDeviceToHost, s));
    SQ_CUDA_TRY(h, cudaStreamSynchronize(s));
    return SQ_OK;
  };
  // the shared mode's rule on [min lo_q - 40 kT, max hi_q + 40 kT]
  double e[5], nlo[3], nhi[3];
  int rc = count(0.0, e, true);
  if (rc != SQ_OK) return rc;
  const double lo = e[3] - 40.0 * h->kT, hi = e[4] + 40.0 * h->kT;
  // 40 kT outside every interval g is below 5e-18 or that close to one: the sums of F and |F| tell which side of N_e
  // the ends lie on, unless they come that close to it
  const double tail = 5e-18 * e[1];
  if (tail < 0.5 * h->n_e && e[0] - tail > h->n_e * (1.0 + 1e-10)) {
    nlo[0] = 0.0;
    nhi[0] = e[0];
  } else if ((rc = count(lo, nlo, false)) != SQ_OK || (rc = count(hi, nhi, false)) != SQ_OK) {
    return rc;
  }
  if (!(nlo[0] < h->n_e && h->n_e < nhi[0]))
    return fail(h, SQ_ERR_NO_BRACKET, "N(mu) - N_e has no sign change on the bisection bracket");
  FermiRoot r;
  r.init(lo, hi, h->n_e, h->kT);
  do {
    if ((rc = count(r.mu, e, false)) != SQ_OK) return rc;
  } while (!r.update(e[0], e[1], e[2]));
  if (mu_out) *mu_out = r.mu;
  return SQ_OK;
}

// One block per node: its coefficients c, d, s at mu (M-point Chebyshev-Gauss rule, as k_coef) and
// its contraction terms, rho_q. FP64 bound: M exponentials and logarithms, then the cosine sums.
// cos(j theta_{M-1-k}) = (-1)^j cos(j theta_k) folds the sums to M / 2 points, and r cos(j theta) =
// (cos((j-1) theta) + cos((j+1) theta)) / 2 gives d^j = (c^{|j-1|} + c^{j+1}) / 2 from c up to n_pl + 1, so a
// coefficient pair costs M multiply-adds instead of 3 M.
__global__ void __launch_bounds__(kContractThreads)
k_contract_nodes(const double* __restrict__ mom, const double* __restrict__ nbnd, const double* __restrict__ v, int Nd,
                 int n_pl, int M, const double* __restrict__ tab, double kT, double mu, double dV,
                 double* __restrict__ rho, double* __restrict__ rows) {
  extern __shared__ double sm[];
  __shared__ double red[kContractGroups * kNPart + kContractThreads / 32];
  const int Mh = (M + 1) / 2;
  double* fv = sm;                       // [2][2][Mh]: g, entropy; even and odd folds
  double* cf = sm + 4 * (size_t)Mh;      // c [n_pl + 2], s [n_pl + 2], d [n_pl + 1]
  const int q = blockIdx.x;
  const double lo = nbnd[2 * q], hi = nbnd[2 * q + 1];
  const double chi_q = 0.5 * (hi + lo), zeta_q = 0.5 * (hi - lo);
  for (int k = threadIdx.x; k < Mh; k += blockDim.x) {
    const int k2 = M - 1 - k;
    const double x1 = (chi_q + zeta_q * tab[2 * k + 1] - mu) / kT;
    const double g1 = fermi_occ(x1), s1 = entropy_d(x1);
    double g2 = 0.0, s2 = 0.0;
    if (k2 != k) {
      const double x2 = (chi_q + zeta_q * tab[2 * k2 + 1] - mu) / kT;
      g2 = fermi_occ(x2);
      s2 = entropy_d(x2);
    }
    fv[k] = g1 + g2;
    fv[Mh + k] = g1 - g2;
    fv[2 * Mh + k] = s1 + s2;
    fv[3 * Mh + k] = s1 - s2;
  }
  __syncthreads();
  const int M4 = 4 * M, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int j = warp; j <= n_pl + 1; j += kContractThreads / 32) {   // one warp per j
    const double* fg = fv + (j & 1) * Mh;
    const double* fs = fv + (2 + (j & 1)) * Mh;
    double ac = 0.0, as = 0.0;
    int t = int((long long)j * (2 * lane + 1) % M4);
    const int step = int((long long)j * 64 % M4);
    for (int k = lane; k < Mh; k += 32) {
      const double cs = tab[t];
      ac += fg[k] * cs;
      as += fs[k] * cs;
      t += step;
      if (t >= M4) t -= M4;
    }
    ac = warp_sum(ac);
    as = warp_sum(as);
    if (lane == 0) {
      cf[j] = 2.0 / M * ac;
      cf[n_pl + 2 + j] = 2.0 / M * as;
    }
  }
  __syncthreads();
  double* d = cf + 2 * (n_pl + 2);
  for (int j = threadIdx.x; j <= n_pl; j += blockDim.x) d[j] = 0.5 * (cf[j == 0 ? 1 : j - 1] + cf[j + 1]);
  __syncthreads();
  contract_block(mom, cf, d, cf + n_pl + 2, chi_q, zeta_q, v, q, q + 1, n_pl, dV, rho, red, rows + (size_t)q * kNPart);
}

int run_contraction_nodes(sq_handle* h, double mu, double* rho_dev, double* out_host) {
  const Geo& g = h->geo;
  cudaStream_t s = h->stream;
  const size_t smem = sizeof(double) * (4 * size_t((h->M + 1) / 2) + 3 * size_t(g.n_pl + 2));
  // the attribute belongs to the function and handles on other host threads launch it too: every caller sets the
  // size of the largest M and n_pl sq_setup accepts (192 KB), never its own
  constexpr int kMaxM = 6144, kMaxNpl = 4096;
  constexpr int smem_max = int(sizeof(double)) * (4 * (kMaxM / 2) + 3 * (kMaxNpl + 2));
  SQ_CUDA_TRY(h, cudaFuncSetAttribute(k_contract_nodes, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
  k_contract_nodes<<<h->Nd, 256, smem, s>>>(h->d.mom, h->d.nbnd, h->d.v64, h->Nd, g.n_pl, h->M, h->d.costab, h->kT,
                                            mu, g.dV, rho_dev, h->d.nrow);
  SQ_LAUNCH_CHECK(h);
  const double* rows = h->d.nrow;
  int n_rows = h->Nd;
  if (n_rows > 2048) {   // two stages: one block over tens of thousands of rows is a serial chain
    k_sum_rows<<<4 * 152, 32 * kNPart, 0, s>>>(rows, n_rows, h->d.part);
    SQ_LAUNCH_CHECK(h);
    rows = h->d.part;
    n_rows = 4 * 152;
  }
  k_contract_final<<<1, 32 * kNPart, 0, s>>>(rows, n_rows, h->kT, h->vol, h->d.scal);
  SQ_LAUNCH_CHECK(h);
  if (out_host) {
    SQ_CUDA_TRY(h, cudaMemcpyAsync(out_host, h->d.scal + 16, 15 * sizeof(double), cudaMemcpyDeviceToHost, s));
    SQ_CUDA_TRY(h, cudaStreamSynchronize(s));
  }
  return SQ_OK;
}

}  // namespace sq
