// The Chebyshev sweep of Sec. 4 over node tiles: for j = 0..n_pl
//     t^{j+1} = 2 Hhat_q t^j - t^{j-1}     (t^1 = Hhat_q t^0),   Hhat_q = (H_q - chi I) / zeta
// with H_q t = -1/2 sum_a (D2_a / h_a^2) t + V_eff t + sum_rows gamma |dOmega| chi (chi^T t),
// and the per-node moments rho^j, K^j_ab, N^j, S^j_ab of each column.
//
// Kernels (Real = double for SQ_FP64, float for SQ_MIXED; node sums always FP64):
//   k_step      SQ_FP64, and SQ_MIXED with more than 4 projector channels per atom (SQ_MIXED otherwise
//               takes the split step of sq_step_mixed.cu). One block per (y-row of bricks, tile), 4..8
//               warps; each warp walks whole 4^3 bricks, so the atom-image records of a brick (table
//               offset, 64-bit mask of the points inside the support sphere) are warp-uniform. Per brick:
//               A  the nonlocal apply sum_rows chi_row(u) Pg^j (Pg^j staged in shared memory),
//                  record-major;
//               B  Laplacian + V + the apply, the window mask, the recurrence update and the
//                  nonlocal-stress partial sum_u W_b (grad_a t^j) (the gradient taps reuse the
//                  Laplacian loads; SQ_FP64: sum_u G_ab t^j, G = -grad_a W_b formed once per sweep);
//               C  fused, the projections gamma |dOmega| chi^T t^{j+1} of the new column (register
//                  sums and a reduce-scatter over the point lanes), one shared-memory FP64 add per
//                  (image, channel, node), one global add per row and node per slab.
//   k_moments   one block per tile: rho^j, K^j (restricted grad_a grad_b at the node),
//               N^j = sum_rows chi(x_q) Pg^j, S^j = sum of the slab partials; FP64 table
//               row; then (k_step) clears Pg^j, which accumulates the projections of step j + 1.
//   k_apply_h / k_project   plain H_q v for the Lanczos bounds (sweep precision).
#include <algorithm>
#include <type_traits>

#include "sq_device.cuh"

namespace sq {

// ------------------------------------------------------------------------------ Lanczos apply
template <typename Real> struct V4;
template <> struct V4<float> { using T = float4; };
template <> struct V4<double> { using T = double4_32a; };

template <typename Real>
__device__ __forceinline__ void load4(const Real* p, Real out[4]) {
  const typename V4<Real>::T x = *reinterpret_cast<const typename V4<Real>::T*>(p);
  out[0] = x.x;
  out[1] = x.y;
  out[2] = x.z;
  out[3] = x.w;
}

// P[row][q] = gamma |dOmega| chi_row^T v: one block per atom image of a tile (images in a stride of
// gridDim.x). A thread owns an (x, y) column of the image's box and half of the nodes: one projector load
// per point serves four nodes, and the column only walks the z-chord of the support sphere (FP32 with a
// 1e-5 margin; points past it hold zeros). Per thread in the vectors' precision, across threads as
// doubles (FP64) or float pairs, fixed order. NCH as in k_step. Bound by load latency (FP32) and the FP64
// units (FP64). 216 tiles of a 12^3 cell, one channel: 278 us with the block's partial products summed in FP64 through
// shared memory and channels padded to four -> 85 us; its 10 sample tiles 21 -> 12 us.
constexpr int kProjThreads = 128, kProjWarps = kProjThreads / 32;
template <typename Real, int NCH>
__global__ void __launch_bounds__(kProjThreads)
k_project(Geo g, Wave w, const Real* __restrict__ Tn, const Real* __restrict__ chi, const AtomTab* __restrict__ atoms,
          const double* __restrict__ rcmax, const double* __restrict__ chs, const TileEntry* __restrict__ entries,
          const int* __restrict__ n_entries, Real* __restrict__ P) {
  const int tl = blockIdx.y, t = wave_tile(w, tl), B = 8;
  int o[3];
  tile_origin(g, t, o);
  const Real* T = Tn + (size_t)tl * g.Upts * B;
  Real* Pt = P + (size_t)tl * g.r_cap * B;
  const int half = threadIdx.x & 1, lane = threadIdx.x >> 1;
  __shared__ typename LzAcc<Real>::T red[kProjWarps][NCH * 8];   // [warp][channel][node]
  for (int eidx = blockIdx.x; eidx < n_entries[tl]; eidx += gridDim.x) {
    const TileEntry te = entries[(size_t)tl * g.e_cap + eidx];
    const AtomTab& at = atoms[te.atom];
    const float rc = float(rcmax[te.atom]), rc2 = rc * rc * (1.f + 1e-5f) + 1e-10f;
    int lo[3], hi[3], bl[3];
    for (int a = 0; a < 3; ++a) {
      bl[a] = at.lo[a] + te.s[a] * g.n[a] - (o[a] - g.m[a]);   // box corner in U-local coords
      lo[a] = max(0, bl[a]);
      hi[a] = min(g.U[a], bl[a] + at.dim[a]);
    }
    const int nx = max(0, hi[0] - lo[0]), ny = max(0, hi[1] - lo[1]);
    const float hx = float(g.h[0]), hy = float(g.h[1]), hz = float(g.h[2]);
    const int dx = at.dim[0], dxy = at.dim[0] * at.dim[1], nchp = at.nchp;
    for (int c0 = 0; c0 < at.nch; c0 += NCH) {
      Real acc[NCH][4];
#pragma unroll
      for (int c = 0; c < NCH; ++c)
        for (int q = 0; q < 4; ++q) acc[c][q] = Real(0);
      for (int col = lane; col < nx * ny; col += kProjThreads / 2) {
        const int lx = lo[0] + col % nx, ly = lo[1] + col / nx;
        const float px = float(lx - bl[0]) * hx + at.dlo[0], py = float(ly - bl[1]) * hy + at.dlo[1];
        const float r2 = rc2 - px * px - py * py;
        if (r2 < 0.f) continue;
        const float zc = sqrtf(r2) * (1.f + 1e-6f);
        const int z0 = max(lo[2], bl[2] + int(ceilf((-zc - at.dlo[2]) / hz - 1e-3f)));
        const int z1 = min(hi[2] - 1, bl[2] + int(floorf((zc - at.dlo[2]) / hz + 1e-3f)));
        const Real* tp = T + ((size_t)(z0 * g.U[1] + ly) * g.U[0] + lx) * B + 4 * half;
        const Real* cp = chi + at.off + ((long long)(z0 - bl[2]) * dxy + (ly - bl[1]) * dx + (lx - bl[0])) * nchp + c0;
        const size_t ts = (size_t)g.U[1] * g.U[0] * B, cs = (size_t)dxy * nchp;
#pragma unroll 4
        for (int z = z0; z <= z1; ++z, tp += ts, cp += cs) {
          Real tv[4], cv[NCH];
          load4(tp, tv);
          if constexpr (NCH == 1) cv[0] = *cp;
          else load4(cp, cv);
#pragma unroll
          for (int c = 0; c < NCH; ++c)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[c][q] += cv[c] * tv[q];
        }
      }
      __syncthreads();   // red free
#pragma unroll
      for (int c = 0; c < NCH; ++c) {
        int node;
        const auto s = lz_warp_sum<Real>(acc[c], &node);
        if ((threadIdx.x & 31) < 8) red[threadIdx.x >> 5][8 * c + node] = s;
      }
      __syncthreads();
      if (threadIdx.x < NCH * 8 && c0 + int(threadIdx.x >> 3) < at.nch) {
        const int c = c0 + (threadIdx.x >> 3);
        double s = lz_double(red[0][threadIdx.x]);
        for (int i = 1; i < kProjWarps; ++i) s += lz_double(red[i][threadIdx.x]);
        Pt[(size_t)(te.row0 + c) * B + (threadIdx.x & 7)] = Real(s * chs[6 * (at.ch0 + c)]);
      }
    }
  }
}

// out = H_q v on every node window of the wave (zero outside the windows); P from k_project. One block
// per (4^3 brick of the window, tile): a warp is one z-plane of the brick, a thread one point and four of
// its nodes, so the brick's image records (table offset, 64-bit sphere mask) are warp-uniform and a
// projector load serves four nodes. Bound by load latency: with one channel per atom four images are read
// at once (105 -> 73 us for the 216 tiles of a 12^3 cell, 15 -> 12 us for its 10 sample tiles). One thread per
// (point, node) that looked every image of its brick up in the atom tables took 410 and 78 us.
constexpr int kApplyThreads = 128;
template <typename Real, int NCH>
__global__ void __launch_bounds__(kApplyThreads)
k_apply_h(Geo g, Wave w, const Real* __restrict__ Tc, Real* __restrict__ Tn, const Real* __restrict__ P,
          const Real* __restrict__ chi, const int4* __restrict__ brec, const int* __restrict__ bn, const Real* __restrict__ v) {
  const int br = blockIdx.x, tl = blockIdx.y, t = wave_tile(w, tl), B = 8;
  int o[3];
  tile_origin(g, t, o);
  const int bx = br % g.nbr[0], by = (br / g.nbr[0]) % g.nbr[1], bz = br / (g.nbr[0] * g.nbr[1]);
  const int half = threadIdx.x & 1, pa = (threadIdx.x >> 1) & 3, pb = (threadIdx.x >> 3) & 3, pc = threadIdx.x >> 5;
  const int u[3] = {bx * kBrick + pa, by * kBrick + pb, bz * kBrick + pc};
  const int Ux = g.U[0], Uy = g.U[1], Uz = g.U[2];
  if (u[1] >= Uy || u[2] >= Uz) return;
  const size_t tbase = (size_t)tl * g.Upts * B;
  const Real* T = Tc + tbase;
  const Real* Pt = P + (size_t)tl * g.r_cap * B + 4 * half;
  const size_t e = (size_t)((u[2] * Uy + u[1]) * Ux + u[0]) * B + 4 * half;
  bool in[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int qo[3] = {q & 1, q >> 1, half};
    in[q] = node_valid(g, o, qo) && in_window(g, qo, u[0], u[1], u[2]);
  }
  const int st[3] = {B, Ux * B, Ux * Uy * B};
  const int Ua[3] = {Ux, Uy, Uz};
  Real tc[4], y[4];
  load4(T + e, tc);
  int wr[3];
  for (int a = 0; a < 3; ++a) {
    wr[a] = (o[a] - g.m[a] + u[a]) % g.n[a];
    if (wr[a] < 0) wr[a] += g.n[a];
  }
  const Real diag = Real(g.lap0) + v[(wr[2] * g.n[1] + wr[1]) * g.n[0] + wr[0]];
#pragma unroll
  for (int q = 0; q < 4; ++q) y[q] = diag * tc[q];
#pragma unroll
  for (int a = 0; a < 3; ++a)
    for (int pp = 1; pp <= g.n_o; ++pp) {
      Real fp[4] = {Real(0), Real(0), Real(0), Real(0)}, fm[4] = {Real(0), Real(0), Real(0), Real(0)};
      if (u[a] + pp < Ua[a]) load4(T + e + (size_t)pp * st[a], fp);
      if (u[a] - pp >= 0) load4(T + e - (size_t)pp * st[a], fm);
      const Real wl = Real(g.lap[a][pp]);
#pragma unroll
      for (int q = 0; q < 4; ++q) y[q] += wl * (fp[q] + fm[q]);
    }
  const int4* rb = brec + ((size_t)tl * g.nbricks + br) * g.br_cap * 2;
  const int nb = bn[(size_t)tl * g.nbricks + br];
  const int bit = pa + 4 * pb + 16 * (pc & 1);
  if constexpr (NCH == 1) {
#pragma unroll 4
    for (int k = 0; k < nb; ++k) {
      const int4 r0 = rb[2 * k], r1 = rb[2 * k + 1];
      Real pv[4];
      load4(Pt + (size_t)r0.y * B, pv);
      if ((unsigned(pc < 2 ? r1.z : r1.w) >> bit) & 1u) {
        const Real cv = chi[r0.x + ((pc * r1.y + pb) * r1.x + pa) * ((r0.w >> 8) & 0xff)];
#pragma unroll
        for (int q = 0; q < 4; ++q) y[q] += cv * pv[q];
      }
    }
  } else {
    for (int k = 0; k < nb; ++k) {
      const int4 r0 = rb[2 * k], r1 = rb[2 * k + 1];
      if (!((unsigned(pc < 2 ? r1.z : r1.w) >> bit) & 1u)) continue;
      const int nch = r0.w & 0xff, nchp = (r0.w >> 8) & 0xff;
      const Real* cp = chi + r0.x + ((pc * r1.y + pb) * r1.x + pa) * nchp;
      for (int c0 = 0; c0 < nch; c0 += 4) {
        Real cv[4];
        load4(cp + c0, cv);
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (c0 + c < nch) {
            Real pv[4];
            load4(Pt + (size_t)(r0.y + c0 + c) * B, pv);
#pragma unroll
            for (int q = 0; q < 4; ++q) y[q] += cv[c] * pv[q];
          }
      }
    }
  }
  typename V4<Real>::T out;
  out.x = in[0] ? y[0] : Real(0);
  out.y = in[1] ? y[1] : Real(0);
  out.z = in[2] ? y[2] : Real(0);
  out.w = in[3] ? y[3] : Real(0);
  *reinterpret_cast<typename V4<Real>::T*>(Tn + tbase + e) = out;
}

// ------------------------------------------------------------------------------ sweep step
// stencil weights of the sweep's precision, read straight from the kernel parameters
template <typename Real> struct Coef;
template <> struct Coef<float> {
  static __device__ __forceinline__ float lap(const Geo& g, int a, int p) { return g.lapf[a][p]; }
  static __device__ __forceinline__ float grd(const Geo& g, int a, int p) { return g.grdf[a][p]; }
};
template <> struct Coef<double> {
  static __device__ __forceinline__ double lap(const Geo& g, int a, int p) { return g.lap[a][p]; }
  static __device__ __forceinline__ double grd(const Geo& g, int a, int p) { return g.grd[a][p]; }
};

constexpr int kTileB = 8;   // nodes per tile (2 x 2 x 2); one warp = 4 points x 8 nodes

// mode 0: t^1 = Hhat t^0;  mode 1: t^{j+1} = 2 Hhat t^j - t^{j-1};  mode 2: moments only.
// Each warp walks whole 4^3 bricks of the slab: iteration it covers brick points
// (a, b, c) = (lane >> 3, it & 3, it >> 2) for node q = lane & 7, so the 4 x-points of an
// iteration are contiguous in memory and every image record is warp-uniform.
// kSmemP: stage Pg^j and accumulate the slab's projections in shared memory (false when a
// tile has too many projector rows; Pg^j is then read and Pg^{j+1} accumulated in global memory)
constexpr int kStepThreads = 256;   // most threads of a k_step block (its warps walk the slab's bricks)

// Warps per k_step block: 4..8, the count that leaves the fewest idle warp-turns over the
// slab's bricks (49 bricks -> 7 warps, 16 -> 8, 36 -> 6); ties go to more warps.
static int step_warps(int bricks_per_slab) {
  int best = kStepThreads / 32, idle_best = 1 << 30;
  for (int w = kStepThreads / 32; w >= 4; --w) {
    const int idle = (bricks_per_slab + w - 1) / w * w - bricks_per_slab;
    if (idle < idle_best) {
      idle_best = idle;
      best = w;
    }
  }
  return best;
}

// FP64 sweeps with at most one brick per SM quarter (of small cells, or a short last wave) give each brick a
// block of its own and each of its four z-planes a warp: the FP64 unit of a quarter takes one warp
// instruction in 75 clocks, so a brick's time is its longest warp's, and one warp per brick leaves most quarters
// idle. 18 tiles of a 5 x 4 x 6 cell, 144 bricks: 210 -> 68 us a step (a block per brick with
// one warp: 232 us). Returns the blocks per slab; 1: whole bricks per warp, all of the slab's in one block.
int step_parts(const Geo& g, int ntiles, bool fp64) {
  const int bricks = g.nbr[0] * g.nbr[2];
  return fp64 && (long long)bricks * g.nslab * ntiles <= kStepFill ? bricks : 1;
}

// NCH: every atom has one channel (1: a table value per point in place of a padded group of four) or any number (4).
// kParts: a block per brick, a warp per z-plane of it (step_parts)
template <typename Real, int NO, bool kSmemP, int NCH, bool kParts>
__global__ void __launch_bounds__(kStepThreads, sizeof(Real) == 4 ? 4 : 2)
k_step(Geo g, Wave w, const Real* __restrict__ Tc, const Real* __restrict__ Tp, Real* __restrict__ Tn,
       const double* __restrict__ Pg, double* __restrict__ Pg_next, const Real* __restrict__ Wt,
       const Real* __restrict__ chi, const Real* __restrict__ gdv,
       const int4* __restrict__ brec, const int* __restrict__ slab_n, const int* __restrict__ slab_map, const int* __restrict__ bn,
       const Real* __restrict__ v, const double* __restrict__ scal, int mode, double* __restrict__ Spart,
       int rows_smem, const double* __restrict__ ncoef, int* __restrict__ status) {
  // dynamic shared memory: [Ps: rows_smem x 8 FP64][red: nw x 8 x 9 FP64][Pstage: rows_smem x 8]
  // [tn_sm: nw x 16 x 32] (Ps and Pstage only with kSmemP; rows_smem = 0 otherwise)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // wrapped V_eff index contributions of the slab's x, y and z positions (cell is periodic)
  __shared__ int wrx[kMaxU], wry[kBrick], wrz[kMaxU];
  const int slab = blockIdx.x, tl = blockIdx.y, t = wave_tile(w, tl);
  double* Pn = Pg_next + (size_t)tl * g.r_cap * kTileB;
  // projections of t^{j+1}, summed in FP64 ([slab rows][8]); Pg^j staged in the sweep precision.
  // In shared memory only the rows of the images that meet this slab are held (slab-local
  // numbering, smap: slab row -> tile row); without it records index the tile rows directly.
  double* Ps = kSmemP ? reinterpret_cast<double*>(smem_raw) : Pn;
  const int nsr = kSmemP ? slab_n[(size_t)tl * g.nslab + slab] : 0;
  if (kSmemP && nsr > rows_smem) {   // a launch sized for another layout (e.g. a stale graph): refuse
    if (threadIdx.x == 0) atomicOr(status + kStOverflow, 4);
    return;
  }
  const int* smap = slab_map + ((size_t)tl * g.nslab + slab) * g.r_cap;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double* red = reinterpret_cast<double*>(smem_raw) + (size_t)rows_smem * kTileB;        // S partials [nw][8][9]
  Real* Pstage = reinterpret_cast<Real*>(red + nw * kTileB * 9);
  Real* tn_sm = Pstage + (size_t)rows_smem * kTileB;                                      // [nw][16][32]
  int o[3];
  tile_origin(g, t, o);
  const double f = (mode == 0) ? 0.5 : 1.0;
  // step coefficients: off-diagonal ca = 2/zeta, diagonal cd = ca lap0 + cb (cb = -2 chi/zeta)
  const Real ca = Real(f * scal[4]), cd = Real(f * scal[6]), cc = Real(mode == 0 ? 0.0 : 1.0);
  const int Ux = g.U[0], Uy = g.U[1], Uz = g.U[2];
  const size_t tbase = (size_t)tl * g.Upts * kTileB;
  const Real* T = Tc + tbase;
  const double* Pt = Pg + (size_t)tl * g.r_cap * kTileB;
  const bool project = (mode != 2);
  const int st[3] = {kTileB, Ux * kTileB, Ux * Uy * kTileB};
  const int Ua[3] = {Ux, Uy, Uz};
  for (int i = threadIdx.x; i < g.U[0] + kBrick + g.U[2]; i += blockDim.x) {
    int a, u;
    if (i < g.U[0]) { a = 0; u = i; }
    else if (i < g.U[0] + kBrick) { a = 1; u = slab * kBrick + i - g.U[0]; }
    else { a = 2; u = i - g.U[0] - kBrick; }
    int wv = (o[a] - g.m[a] + u) % g.n[a];
    if (wv < 0) wv += g.n[a];
    if (a == 0) wrx[u] = wv;
    else if (a == 1) wry[u - slab * kBrick] = wv * g.n[0];
    else wrz[u] = wv * g.n[0] * g.n[1];
  }
  if (kSmemP) {
    for (int i = threadIdx.x; i < nsr * kTileB; i += blockDim.x) {
      Pstage[i] = Real(Pt[smap[i >> 3] * kTileB + (i & 7)]);
      if (project) Ps[i] = 0.0;
    }
  }
  __syncthreads();
  // without shared memory the apply reads Pg^j from global memory (FP64) directly
  auto pg = [&](int idx) -> Real { return kSmemP ? Pstage[idx] : Real(Pt[idx]); };

  const int q = lane & 7, pa = lane >> 3;
  int qo[3];
  qo[0] = q & 1;
  qo[1] = (q >> 1) & 1;
  qo[2] = q >> 2;
  const bool valid = node_valid(g, o, qo);
  // step coefficients of the lane's node: the block's (shared bounds) or the node's own
  // (per-node bounds)
  Real caA = ca, cdA = cd;
  if (ncoef && valid) {
    const int node = (o[0] + qo[0]) + g.n[0] * ((o[1] + qo[1]) + g.n[1] * (o[2] + qo[2]));
    caA = Real(f * ncoef[2 * node]);
    cdA = Real(f * ncoef[2 * node + 1]);
  }
  constexpr bool kG = sizeof(Real) == 8;   // S^j from G_ab t^j (k_gtable) in place of W_b grad_a t^j
  const Real* Wq = Wt + (size_t)tl * (kG ? 9 : 3) * g.Upts * kTileB;
  const size_t wstr = (size_t)g.Upts * kTileB;
  // S partial sums, per lane across bricks
  Real sacc[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) sacc[k] = Real(0);
  const int nbx = g.nbr[0], nby = g.nbr[1], nbz = g.nbr[2];

  // a warp's units of work: whole bricks, or one z-plane of a brick (step_parts); FP64 takes a plane's four
  // points per lane at a time, FP32 two planes'
  constexpr int kGrp = kG ? 1 : 2;   // planes per group
  const int bps = nbx * nbz, step = kParts ? gridDim.z * nw : nw;
  for (int un = kParts ? blockIdx.z + gridDim.z * warp : warp; un < (kParts ? 4 * bps : bps); un += step) {
    const int bi = kParts ? un % bps : un, pl0 = kParts ? un / bps : 0, pl1 = kParts ? pl0 + 1 : 4;   // planes [pl0, pl1)
    const int bx = bi % nbx, bz = bi / nbx, by = slab;
    const int br = (bz * nby + by) * nbx + bx;
    const int4* rb = brec + ((size_t)tl * g.nbricks + br) * g.br_cap * 2;
    const int nb = bn[(size_t)tl * g.nbricks + br];
    Real* tnv = tn_sm + warp * 16 * 32 + lane;   // per lane and brick point: V_nl t^j, then t^{j+1}
    {
      // phase A: nonlocal apply, record-major: sum_rows chi_row(u) Pg^j[row][q] for the lane's
      // points; the table loads of one record are independent of each other
#pragma unroll 1
      for (int pl = pl0; pl < pl1; pl += kGrp) {   // a few points at a time keep the accumulators in registers
        Real ynl[4 * kGrp];
#pragma unroll
        for (int i = 0; i < 4 * kGrp; ++i) ynl[i] = Real(0);
        for (int k = 0; k < nb; ++k) {
          const int4 r0 = rb[2 * k], r1 = rb[2 * k + 1];
          const int nch = r0.w & 0xff, nchp = (r0.w >> 8) & 0xff;
          const int prow = kSmemP ? (int(unsigned(r0.w) >> 16)) : r0.y;
          const unsigned mk = unsigned(pl < 2 ? r1.z : r1.w) >> (pa + 16 * (pl & 1));   // bits 4 i of this group
          if (!(mk & (kGrp == 1 ? 0x1111u : 0x11111111u))) continue;
          if constexpr (NCH == 1) {
            const Real pv = pg(prow * kTileB + q);
#pragma unroll
            for (int i = 0; i < 4 * kGrp; ++i)
              if ((mk >> (4 * i)) & 1u) {
                const int it = 4 * pl + i;
                ynl[i] += chi[r0.x + (((it >> 2) * r1.y + (it & 3)) * r1.x + pa) * nchp] * pv;
              }
            continue;
          }
          for (int c0 = 0; c0 < nch; c0 += 4) {
            Real pv[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) pv[c] = (c0 + c < nch) ? pg((prow + c0 + c) * kTileB + q) : Real(0);
#pragma unroll
            for (int i = 0; i < 4 * kGrp; ++i) {
              if ((mk >> (4 * i)) & 1u) {
                const int it = 4 * pl + i;
                Real cv[4];
                load4(chi + r0.x + (((it >> 2) * r1.y + (it & 3)) * r1.x + pa) * nchp + c0, cv);
                ynl[i] += cv[0] * pv[0] + cv[1] * pv[1] + cv[2] * pv[2] + cv[3] * pv[3];
              }
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 4 * kGrp; ++i) tnv[(4 * pl + i) * 32] = ynl[i];
      }
    }
    __syncwarp();
    {
#pragma unroll 1
      for (int it = 4 * pl0; it < 4 * pl1; ++it) {
        const int pb = it & 3, pc = it >> 2;
        const int ux = bx * kBrick + pa, uy = by * kBrick + pb, uz = bz * kBrick + pc;
        const bool inU = (uy < Uy) && (uz < Uz);
        const size_t e = (size_t)((uz * Uy + uy) * Ux + ux) * kTileB + q;
        const bool inwin = inU && valid && in_window(g, qo, ux, uy, uz);
        Real tn = Real(0);
        if (inwin) {
          // loads that do not depend on the stencil, issued first
          const Real w0 = Wq[e], w1 = Wq[wstr + e], w2 = Wq[2 * wstr + e];
          Real wv[kG ? 6 : 1];
          if constexpr (kG) {
#pragma unroll
            for (int k = 0; k < 6; ++k) wv[k] = Wq[(3 + k) * wstr + e];
          }
          const Real tp = (mode == 1) ? Tp[tbase + e] : Real(0);
          const Real tc = T[e];
          Real y = Real(0);                           // off-diagonal part of H t^j
          Real gr[3];
          const int u[3] = {ux, uy, uz};
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            gr[a] = Real(0);
#pragma unroll
            for (int pp = 1; pp <= NO; ++pp) {
              const Real fp = (u[a] + pp < Ua[a]) ? T[e + (size_t)pp * st[a]] : Real(0);
              const Real fm = (u[a] - pp >= 0) ? T[e - (size_t)pp * st[a]] : Real(0);
              y += Coef<Real>::lap(g, a, pp) * (fp + fm);
              if constexpr (!kG) gr[a] += Coef<Real>::grd(g, a, pp) * (fp - fm);
            }
          }
          const Real vloc = v[wrz[uz] + wry[pb] + wrx[ux]];   // V_eff at the wrapped node
          y += tnv[it * 32];                          // nonlocal part from phase A
          if (mode != 2) {
            tn = caA * y + (cdA + caA * vloc) * tc - cc * tp;
            Tn[tbase + e] = tn;
          }
          if constexpr (kG) {
            sacc[0] += w0 * tc;
            sacc[1] += w1 * tc;
            sacc[2] += w2 * tc;
#pragma unroll
            for (int k = 0; k < 6; ++k) sacc[3 + k] += wv[k] * tc;
          } else {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              sacc[3 * a + 0] += gr[a] * w0;
              sacc[3 * a + 1] += gr[a] * w1;
              sacc[3 * a + 2] += gr[a] * w2;
            }
          }
        } else if (inU && mode != 2) {
          Tn[tbase + e] = Real(0);
        }
        tnv[it * 32] = tn;
      }
    }
    __syncwarp();
    // projections of t^{j+1} over this brick: each lane sums its 16 points in registers, a
    // reduce-scatter over the 4 x-point lanes (xor 8, then xor 16) leaves lane (pa, q) with the
    // brick sum of channel c0 + pa for node q, so one FP64 conversion and one shared add per
    // lane cover 4 channels x 8 nodes (FP64 instructions are narrow on this part)
    {
      if (project) {
        const bool b0 = (pa & 1) != 0, b1 = (pa & 2) != 0;
        for (int k = 0; k < nb; ++k) {
          const int4 r0 = rb[2 * k], r1 = rb[2 * k + 1];
          const int nch = r0.w & 0xff, nchp = (r0.w >> 8) & 0xff;
          const int prow = kSmemP ? (int(unsigned(r0.w) >> 16)) : r0.y;
          const unsigned mlo = unsigned(r1.z) >> pa, mhi = unsigned(r1.w) >> pa;
          if (kParts && !((unsigned(pl0 < 2 ? r1.z : r1.w) >> (16 * (pl0 & 1))) & 0xffffu)) continue;
          if constexpr (NCH == 1) {
            Real acc = Real(0);
#pragma unroll 8
            for (int it = 4 * pl0; it < 4 * pl1; ++it)
              if (((it < 8 ? mlo : mhi) >> (4 * (it & 7))) & 1u)
                acc += chi[r0.x + (((it >> 2) * r1.y + (it & 3)) * r1.x + pa) * nchp] * tnv[it * 32];
            acc += __shfl_xor_sync(0xffffffffu, acc, 8);
            acc += __shfl_xor_sync(0xffffffffu, acc, 16);
            if (pa == 0 && acc != Real(0)) atomicAdd(&Ps[prow * kTileB + q], double(acc * gdv[r0.z]));
            continue;
          }
          for (int c0 = 0; c0 < nch; c0 += 4) {
            Real acc[4] = {Real(0), Real(0), Real(0), Real(0)};
#pragma unroll 4
            for (int it = 4 * pl0; it < 4 * pl1; ++it) {
              const unsigned bit = ((it < 8 ? mlo : mhi) >> (4 * (it & 7))) & 1u;
              if (bit) {
                const Real tv = tnv[it * 32];
                Real cv[4];
                load4(chi + r0.x + (((it >> 2) * r1.y + (it & 3)) * r1.x + pa) * nchp + c0, cv);
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[c] += cv[c] * tv;
              }
            }
            // step 1 (pa bit 0): keep channels {b0, 2 + b0}, hand the other two to the partner
            Real k0 = b0 ? acc[1] : acc[0], k1 = b0 ? acc[3] : acc[2];
            const Real g0 = b0 ? acc[0] : acc[1], g1 = b0 ? acc[2] : acc[3];
            k0 += __shfl_xor_sync(0xffffffffu, g0, 8);
            k1 += __shfl_xor_sync(0xffffffffu, g1, 8);
            // step 2 (pa bit 1): keep channel b0 + 2 b1 = pa
            Real s = b1 ? k1 : k0;
            s += __shfl_xor_sync(0xffffffffu, b1 ? k0 : k1, 16);
            const int c = c0 + pa;
            if (c < nch && s != Real(0)) atomicAdd(&Ps[(prow + c) * kTileB + q], double(s * gdv[r0.z + c]));
          }
        }
      }
    }
  }
  // S partials: fixed-order reduction per node (the point lanes by shuffles, then warps)
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    double sv = double(sacc[k]);
    sv += __shfl_xor_sync(0xffffffffu, sv, 8);
    sv += __shfl_xor_sync(0xffffffffu, sv, 16);
    if (lane < kTileB) red[(warp * kTileB + lane) * 9 + k] = sv;
  }
  __syncthreads();
  for (int k2 = threadIdx.x; k2 < kTileB * 9; k2 += blockDim.x) {
    const int qq = k2 / 9, k = k2 % 9;
    double sv = 0.0;
    for (int wv = 0; wv < nw; ++wv) sv += red[(wv * kTileB + qq) * 9 + k];
    Spart[((((size_t)tl * g.nslab + slab) * gridDim.z + blockIdx.z) * kTileB + qq) * 9 + k] = sv;
  }
  if (kSmemP && project) {
    for (int i = threadIdx.x; i < nsr * kTileB; i += blockDim.x) {
      const double s = Ps[i];
      if (s != 0.0) atomicAdd(&Pn[smap[i >> 3] * kTileB + (i & 7)], s);
    }
  }
}

// Moments of t^j per node (one warp per node), then Pg^j := 0 (the accumulator of step j + 1). kPair: the
// split mixed step, which keeps the projections as pairs of floats and rewrites them each step.
// nslab: S^j partials per tile.
template <typename Real, bool kPair>
__global__ void __launch_bounds__(kThreads)
k_moments(Geo g, Wave w, int j, const Real* __restrict__ Tj, const Real* __restrict__ A, double* __restrict__ Pg,
          const int* __restrict__ n_rows, const double* __restrict__ Spart, int nslab, double* __restrict__ mom) {
  const int tl = blockIdx.x, t = wave_tile(w, tl);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int o[3];
  tile_origin(g, t, o);
  const int B = g.B;
  const Real* T = Tj + (size_t)tl * g.Upts * B;
  const Real* At = A + (size_t)tl * g.r_cap * B;
  double* Pt = Pg + (size_t)tl * g.r_cap * B;
  const int nr = n_rows[tl];
  for (int q = warp; q < B; q += kThreads / 32) {
    int qo[3];
    node_offset(g, q, qo);
    if (!node_valid(g, o, qo)) continue;
    const int node = (o[0] + qo[0]) + g.n[0] * ((o[1] + qo[1]) + g.n[1] * (o[2] + qo[2]));
    const int c[3] = {qo[0] + g.m[0], qo[1] + g.m[1], qo[2] + g.m[2]};
    // FP64 arithmetic on the stored values: the restricted grad_a grad_a at the node cancels
    // strongly, and an FP32 version measured 4x the sigma^I error on the 216-atom instance
    auto tval = [&](int x, int y, int z) -> double {
      if ((unsigned)x >= (unsigned)g.U[0] || (unsigned)y >= (unsigned)g.U[1] || (unsigned)z >= (unsigned)g.U[2]) return 0.0;
      return double(T[((size_t)(z * g.U[1] + y) * g.U[0] + x) * B + q]);
    };
    // K^j_ab = [grad_a,q grad_b,q t^j]_q with both factors restricted to the window (columns are zero outside
    // it). FP64 issues 1.7 lanes per clock and SM, so the sums are arranged for few FP64 instructions: the
    // diagonal pairs are one 4 n_o + 1 point stencil, the others the quadruples t(i,j) - t(-i,j) - t(i,-j) +
    // t(-i,-j), and the seven totals share one reduce-scatter (200 -> 60 instructions per node at n_o = 6).
    double val[8];
    val[7] = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int d = lane - 2 * g.n_o;
      val[a] = (lane <= 4 * g.n_o)
                   ? g.grd2[a][abs(d)] * tval(c[0] + (a == 0 ? d : 0), c[1] + (a == 1 ? d : 0), c[2] + (a == 2 ? d : 0)) : 0.0;
    }
#pragma unroll
    for (int pr = 3; pr < 6; ++pr) {
      const int a = (pr == 3) ? 1 : 0, b = (pr == 5) ? 1 : 2;   // yz, xz, xy
      double s = 0.0;
      for (int e = lane; e < g.n_o * g.n_o; e += 32) {
        const int i = e / g.n_o + 1, j = e - (i - 1) * g.n_o + 1;
        auto at = [&](int si, int sj) {
          return tval(c[0] + (a == 0 ? si : 0), c[1] + (a == 1 ? si : b == 1 ? sj : 0), c[2] + (b == 2 ? sj : 0));
        };
        s += g.grd[a][i] * g.grd[b][j] * ((at(i, j) - at(-i, j)) - (at(i, -j) - at(-i, -j)));
      }
      val[pr] = s;
    }
    // N^j = w_q^T V_nl,q t^j = sum_rows chi_row(x_q) (gamma |dOmega| chi_row^T t^j)
    if constexpr (kPair) {   // float pairs: products and sums with their rounding errors (about 2^-47 relative)
      float nh = 0.f, nl = 0.f;
      for (int r = lane; r < nr; r += 32) {
        const size_t k = (size_t)r * B + q;
        const float2 x = reinterpret_cast<const float2*>(Pt)[k];
        const float ak = At[k], p = __fmul_rn(ak, x.x), pe = fmaf(ak, x.x, -p) + ak * x.y;
        const float sm = __fadd_rn(nh, p), z = __fsub_rn(sm, nh);
        nl = __fadd_rn(nl, __fadd_rn(__fadd_rn(__fsub_rn(nh, __fsub_rn(sm, z)), __fsub_rn(p, z)), pe));
        nh = sm;
      }
      val[6] = double(nh) + double(nl);
    } else {
      double nacc = 0.0;
      for (int r = lane; r < nr; r += 32) nacc += double(At[(size_t)r * B + q]) * Pt[(size_t)r * B + q];
      val[6] = nacc;
    }
    auto halve = [&](int n, int d) {   // keep n of 2 n values, hand the others to the partner lane
      const bool up = (lane & d) != 0;
#pragma unroll
      for (int k = 0; k < n; ++k) {
        const double give = up ? val[k] : val[k + n], keep = up ? val[k + n] : val[k];
        val[k] = keep + __shfl_xor_sync(0xffffffffu, give, d);
      }
    };
    halve(4, 16);
    halve(2, 8);
    halve(1, 4);
    val[0] += __shfl_xor_sync(0xffffffffu, val[0], 2);
    val[0] += __shfl_xor_sync(0xffffffffu, val[0], 1);
    double* row = mom + ((size_t)node * (g.n_pl + 1) + j) * SQ_N_MOMENTS;
    const int slot = 1 + (lane >> 4) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
    if ((lane & 3) == 0 && slot < 8) row[slot] = val[0];
    if (lane == 1) row[0] = tval(c[0], c[1], c[2]);
    if (lane < 9) {
      double sv = 0.0;
      for (int sl = 0; sl < nslab; ++sl) sv += Spart[(((size_t)tl * nslab + sl) * B + q) * 9 + lane];
      row[8 + lane] = sv;
    }
  }
  if constexpr (!kPair) {
    __syncthreads();
    for (int i = threadIdx.x; i < nr * B; i += kThreads) Pt[i] = 0.0;
  }
}

// dynamic shared memory of k_step: staged projections (at most kStepRowsSmemMax, else they stay
// in global memory) + the per-warp arrays
constexpr int kStepRowsSmemMax = 160 * 1024;
constexpr int kStepSmemMax = kStepRowsSmemMax + (kStepThreads / 32) * (kTileB * 9 * 8 + 16 * 32 * 8);

// largest projector-row count a step block stages in shared memory (more rows: global memory)
int step_rows_smem_max(int precision) {
  return int(kStepRowsSmemMax / (kTileB * (sizeof(double) + (precision == SQ_FP64 ? sizeof(double) : sizeof(float)))));
}

template <typename Real, int NO>
static int launch_step(sq_handle* h, const Wave& w, dim3 grid, size_t smem, const Real* Tc, const Real* Tp, Real* Tn,
                       const double* Pg, double* Pgn, const Real* W, const Real* chi, const Real* gdv, const Real* v,
                       int mode) {
  const int rows_smem = int(smem / (kTileB * (sizeof(double) + sizeof(Real))));
  const double* ncoef = (h->bounds_mode == SQ_BOUNDS_PER_NODE) ? h->d.ncoef : nullptr;
  grid.z = step_parts(h->geo, w.ntiles, sizeof(Real) == 8);
  const int nw = h->step_warps > 0 ? h->step_warps : grid.z > 1 ? 4 : step_warps(h->geo.nbr[0] * h->geo.nbr[2]);
  const int nthr = 32 * nw;
  const size_t smem_warps = size_t(nw) * (kTileB * 9 * sizeof(double) + 16 * 32 * sizeof(Real));
  // The dynamic-size attribute belongs to the function, not the launch, and handles on other
  // host threads launch the same kernel, so every caller sets the same value (the largest
  // dynamic size this kernel uses)
  const bool staged = rows_smem <= h->step_rows_cap, one = h->max_nch == 1;
  h->step_variant[staged ? 1 : 2]++;
  auto go = [&](auto kernel, size_t bytes, int rows) -> int {
    SQ_CUDA_TRY(h, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kStepSmemMax));
    kernel<<<grid, nthr, bytes, h->stream>>>(h->geo, w, Tc, Tp, Tn, Pg, Pgn, W, chi, gdv, h->wb.brick_rec, h->wb.slab_n,
                                             h->wb.slab_map, h->wb.brick_n, v, h->d.scal, mode, h->wb.Spart, rows, ncoef,
                                             h->d.status);
    return SQ_OK;
  };
  int rc = SQ_OK;
  auto pick = [&](auto parts) {
    constexpr bool kP = decltype(parts)::value;
    if (staged) rc = one ? go(k_step<Real, NO, true, 1, kP>, smem + smem_warps, rows_smem)
                         : go(k_step<Real, NO, true, 4, kP>, smem + smem_warps, rows_smem);
    else rc = one ? go(k_step<Real, NO, false, 1, kP>, smem_warps, 0) : go(k_step<Real, NO, false, 4, kP>, smem_warps, 0);
  };
  if constexpr (sizeof(Real) == 8) {
    if (grid.z > 1) pick(std::true_type{});
    else pick(std::false_type{});
  } else {
    pick(std::false_type{});
  }
  if (rc != SQ_OK) return rc;
  SQ_LAUNCH_CHECK(h);
  return SQ_OK;
}

template <typename Real>
static int dispatch_step(sq_handle* h, const Wave& w, dim3 grid, size_t smem, const Real* Tc, const Real* Tp, Real* Tn,
                         const double* Pg, double* Pgn, const Real* W, const Real* chi, const Real* gdv, const Real* v,
                         int mode) {
  switch (h->geo.n_o) {
    case 1: return launch_step<Real, 1>(h, w, grid, smem, Tc, Tp, Tn, Pg, Pgn, W, chi, gdv, v, mode);
    case 2: return launch_step<Real, 2>(h, w, grid, smem, Tc, Tp, Tn, Pg, Pgn, W, chi, gdv, v, mode);
    case 3: return launch_step<Real, 3>(h, w, grid, smem, Tc, Tp, Tn, Pg, Pgn, W, chi, gdv, v, mode);
    case 4: return launch_step<Real, 4>(h, w, grid, smem, Tc, Tp, Tn, Pg, Pgn, W, chi, gdv, v, mode);
    case 5: return launch_step<Real, 5>(h, w, grid, smem, Tc, Tp, Tn, Pg, Pgn, W, chi, gdv, v, mode);
    default: return launch_step<Real, 6>(h, w, grid, smem, Tc, Tp, Tn, Pg, Pgn, W, chi, gdv, v, mode);
  }
}

// images one stage of the TMA-staged step holds in wave wi: the wave's fullest brick, at most
// kStepTmaRecs (a brick with more takes them in chunks)
static int stage_recs(const sq_handle* h, size_t wi) {
  return std::max(1, std::min(h->wave_recs[wi], h->stage_recs_cap));
}

// The TMA-staged step (sq_step_tma.cu), when selected (SQ_STEP_KERNEL=staged), runs a mixed sweep
// wave when its maps exist and the slab's projections and one stage fit in shared memory.
static bool use_tma(const sq_handle* h, size_t wi) {
  if (!h->tma_ok || !h->step_staged || h->precision != SQ_MIXED) return false;
  if (wi >= h->wave_rows.size() || wi >= h->wave_recs.size()) return false;
  const int rows = std::max(1, h->wave_rows[wi]);
  if (rows > h->step_rows_cap) return false;   // the global-memory projection path
  return step_tma_smem_bytes(rows, stage_recs(h, wi)) <= kStepTmaSmemMax;
}

// The split mixed step: SQ_MIXED with at most 4 channels per atom, unless the staged step was asked for, or
// SQ_STEP_SMEM_ROWS asks for the global-memory projections of k_step.
bool want_split(const sq_handle* h, size_t wi) {
  if (!h->split_able || use_tma(h, wi)) return false;
  return !(h->step_rows_env && wi < h->wave_rows.size() && std::max(1, h->wave_rows[wi]) > h->step_rows_cap);
}
bool use_split(const sq_handle* h, size_t wi) { return want_split(h, wi) && nl_fits(h, wi); }

template <typename Real>
static int sweep_t(sq_handle* h, const Real* chi, const Real* v, const Real* gdv) {
  const Geo& g = h->geo;
  cudaStream_t s = h->stream;
  Real* T[3] = {(Real*)h->wb.T[0], (Real*)h->wb.T[1], (Real*)h->wb.T[2]};
  double* Pg[2] = {(double*)h->wb.Pg[0], (double*)h->wb.Pg[1]};
  Real* A = (Real*)h->wb.A;
  Real* W = (Real*)h->wb.W;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  SQ_CUDA_TRY(h, cudaStreamIsCapturing(s, &cap));
  const bool capturing = cap != cudaStreamCaptureStatusNone;
  if (h->wave_rows.size() != h->waves.size() || h->wave_recs.size() != h->waves.size()) {
    if (capturing) return fail(h, SQ_ERR_STATE, "wave layout not measured before capture");
    int rc = measure_wave_rows(h);
    if (rc != SQ_OK) return rc;
  }
  for (size_t wi = 0; wi < h->waves.size(); ++wi) {
    NvtxRange nvtx("sweep wave");
    const Wave& w = h->waves[wi];
    // a captured graph must rebuild the lists itself (the atoms may move before it runs again)
    int rc = build_wave_lists(h, wi, !capturing);
    const bool split = use_split(h, wi);
    if (rc != SQ_OK) return rc;
    // largest slab projector-row count of the wave (measured once per layout) sizes the
    // per-slab shared accumulator
    const int rmax = h->wave_rows[wi];
    const size_t smem = std::max<size_t>(1, size_t(rmax)) * kTileB * (sizeof(double) + sizeof(Real));

    const dim3 gstencil(g.nslab, w.ntiles);
    const int parts = step_parts(g, w.ntiles, sizeof(Real) == 8);   // k_step's blocks per slab
    // algorithmic bytes of one stencil launch: node columns x region points x vectors moved
    long long nodes = 0;
    for (int tl = 0; tl < w.ntiles; ++tl) {
      const int t = w.tile0 + tl;
      const int o[3] = {(t % g.tiles[0]) * g.b, ((t / g.tiles[0]) % g.tiles[1]) * g.b,
                        (t / (g.tiles[0] * g.tiles[1])) * g.b};
      nodes += (long long)std::min(g.b, g.n[0] - o[0]) * std::min(g.b, g.n[1] - o[1]) * std::min(g.b, g.n[2] - o[2]);
    }
    const double col_bytes = double(nodes) * (2 * g.m[0] + 1) * (2 * g.m[1] + 1) * (2 * g.m[2] + 1) * sizeof(Real);
    for (int j = 0; j <= g.n_pl; ++j) {
      Real* Tc = T[j % 3];
      Real* Tn = T[(j + 1) % 3];
      Real* Tp = T[(j + 2) % 3];
      const int mode = (j == g.n_pl) ? 2 : (j == 0 ? 0 : 1);
      const double vecs = (mode == 0) ? 2.0 : (mode == 1) ? 3.0 : 1.0;   // reads t^j (t^{j-1}), writes t^{j+1}
      cudaEvent_t ev = capturing ? nullptr : timing_begin(h, SQ_K_STENCIL, vecs * col_bytes);
      if (split)
        rc = launch_step_mixed(h, wi, (const float*)Tc, (const float*)Tp, (float*)Tn, mode);
      else if (sizeof(Real) == 4 && use_tma(h, wi))
        rc = launch_step_tma(h, w, gstencil, j % 3, (j + 2) % 3, (float*)Tn, Pg[j % 2], Pg[(j + 1) % 2], mode,
                             std::max(1, rmax), stage_recs(h, wi));
      else
        rc = dispatch_step<Real>(h, w, gstencil, smem, Tc, Tp, Tn, Pg[j % 2], Pg[(j + 1) % 2], W, chi, gdv, v, mode);
      if (rc != SQ_OK) return rc;
      timing_end(h, ev);
      ev = capturing ? nullptr : timing_begin(h, SQ_K_MOMENTS, 0.0);
      if (split)
        k_moments<float, true><<<w.ntiles, kThreads, 0, s>>>(g, w, j, (const float*)Tc, (const float*)A, Pg[0],
                                                             h->wb.n_rows, h->wb.Spart, stencil_chunks(g), h->d.mom);
      else
        k_moments<Real, false><<<w.ntiles, kThreads, 0, s>>>(g, w, j, Tc, A, Pg[j % 2], h->wb.n_rows, h->wb.Spart,
                                                             g.nslab * parts, h->d.mom);
      timing_end(h, ev);
      SQ_LAUNCH_CHECK(h);
      if (split && mode != 2) {
        ev = capturing ? nullptr : timing_begin(h, SQ_K_PROJECT, 0.0);
        rc = launch_project_mixed(h, wi, (const float*)Tn);
        if (rc != SQ_OK) return rc;
        timing_end(h, ev);
      }
    }
  }
  if (capturing) return SQ_OK;   // the status words are read after the graph runs
  {
    int rc = timing_collect(h);
    if (rc != SQ_OK) return rc;
  }
  int st[kStCount];
  SQ_CUDA_TRY(h, cudaMemcpyAsync(st, h->d.status, sizeof(st), cudaMemcpyDeviceToHost, s));
  SQ_CUDA_TRY(h, cudaStreamSynchronize(s));
  if (st[kStOverflow]) return fail(h, SQ_ERR_CUDA, "internal list capacity exceeded");
  if (st[kStBadBounds]) return fail(h, SQ_ERR_CUDA, "spectral bounds are not finite or empty");
  if (st[kStTimeout]) return fail(h, SQ_ERR_TIMEOUT, "a staged step block's copy wait ran out");
  return SQ_OK;
}

template <typename Real>
static int time_step_t(sq_handle* h, int reps, double* ms_out, const Real* chi, const Real* v, const Real* gdv) {
  const Geo& g = h->geo;
  cudaStream_t s = h->stream;
  if (h->waves.empty()) {
    *ms_out = 0.0;
    return SQ_OK;
  }
  if (h->wave_rows.size() != h->waves.size() || h->wave_recs.size() != h->waves.size()) {
    int rc = measure_wave_rows(h);
    if (rc != SQ_OK) return rc;
  }
  const Wave& w = h->waves[0];
  cudaEvent_t e0, e1;
  SQ_CUDA_TRY(h, cudaEventCreate(&e0));
  SQ_CUDA_TRY(h, cudaEventCreate(&e1));
  // a sweep rebuilds each wave's lists and W table (unless sq_keep_lists holds them for one wave):
  // that cost, spread over the sweep's n_pl + 1 steps, belongs to the step time the tuner compares
  const bool rebuilt = h->waves.size() > 1 || !h->keep_lists;
  cudaEventRecord(e0, s);
  int rc = build_wave_lists(h, 0, !rebuilt);
  cudaEventRecord(e1, s);
  float ms_lists = 0.f;
  if (rc == SQ_OK && rebuilt && cudaEventSynchronize(e1) == cudaSuccess) cudaEventElapsedTime(&ms_lists, e0, e1);
  if (rc != SQ_OK) {
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return rc;
  }
  Real* T[3] = {(Real*)h->wb.T[0], (Real*)h->wb.T[1], (Real*)h->wb.T[2]};
  double* Pg[2] = {(double*)h->wb.Pg[0], (double*)h->wb.Pg[1]};
  const size_t smem = std::max<size_t>(1, size_t(h->wave_rows[0])) * kTileB * (sizeof(double) + sizeof(Real));
  const dim3 grid(g.nslab, w.ntiles);
  const bool tma = sizeof(Real) == 4 && use_tma(h, 0), split = use_split(h, 0);
  const int rows = std::max(1, h->wave_rows[0]), recs = stage_recs(h, 0);
  auto step = [&](int c, int p, int n, int mode) -> int {
    if (split) {
      const int r = launch_step_mixed(h, 0, (const float*)T[c], (const float*)T[p], (float*)T[n], mode);
      return r != SQ_OK ? r : launch_project_mixed(h, 0, (const float*)T[n]);
    }
    if (tma) return launch_step_tma(h, w, grid, c, p, (float*)T[n], Pg[c], Pg[1 - c], mode, rows, recs);
    return dispatch_step<Real>(h, w, grid, smem, T[c], T[p], T[n], Pg[c], Pg[1 - c], (Real*)h->wb.W, chi, gdv, v, mode);
  };
  // the first launch (mode 0) forms t^1 from t^0, so the timed launches read defined values
  rc = step(0, 2, 1, 0);
  if (rc != SQ_OK) {
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return rc;
  }
  cudaEventRecord(e0, s);
  for (int r = 0; r < reps && rc == SQ_OK; ++r) rc = step(1, 0, 2, 1);
  cudaEventRecord(e1, s);
  float ms = 0.f;
  const cudaError_t e = cudaEventSynchronize(e1);
  if (e == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc != SQ_OK) return rc;
  if (e != cudaSuccess) return fail(h, SQ_ERR_CUDA, std::string("step timing: ") + cudaGetErrorString(e));
  *ms_out = double(ms) / std::max(1, reps) + double(ms_lists) / (g.n_pl + 1);
  return SQ_OK;
}

int time_step_launch(sq_handle* h, int reps, double* ms_out) {
  if (h->precision == SQ_FP64) return time_step_t<double>(h, reps, ms_out, h->d.chi64, h->d.v64, h->d.gdv64);
  return time_step_t<float>(h, reps, ms_out, h->d.chi32, h->d.v32, h->d.gdv32);
}

// out[0]: most projector rows of a slab, [1]: most images of a brick, [2], [3]: most (brick, row) and (brick, image)
// pairs of a tile. One block per tile of the wave.
__global__ void __launch_bounds__(kThreads)
k_wave_measure(Geo g, const int* __restrict__ slab_n, const int* __restrict__ bn, const int4* __restrict__ brec,
               int* __restrict__ out) {
  const int tl = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int slab = 0, most = 0, rows = 0, imgs = 0;
  for (int i = threadIdx.x; i < g.nslab; i += kThreads) slab = max(slab, slab_n[(size_t)tl * g.nslab + i]);
  for (int br = warp; br < g.nbricks; br += kThreads / 32) {
    const size_t tb = (size_t)tl * g.nbricks + br;
    const int nb = bn[tb];
    for (int k = lane; k < nb; k += 32) rows += brec[(tb * g.br_cap + k) * 2].w & 0xff;
    most = max(most, nb);
    if (lane == 0) imgs += nb;
  }
  int tot_rows, tot_imgs;
  block_exclusive_scan(rows, &tot_rows);
  block_exclusive_scan(imgs, &tot_imgs);
  slab = __reduce_max_sync(0xffffffffu, slab);
  if (lane == 0) {
    atomicMax(out, slab);
    atomicMax(out + 1, most);
  }
  if (threadIdx.x == 0) {
    atomicMax(out + 2, tot_rows);
    atomicMax(out + 3, tot_imgs);
  }
}

int measure_wave_rows(sq_handle* h) {
  const Geo& g = h->geo;
  cudaStream_t s = h->stream;
  h->wave_rows.assign(h->waves.size(), 0);
  h->wave_recs.assign(h->waves.size(), 0);
  h->wave_nl.assign(h->waves.size(), NlNeed());
  for (size_t wi = 0; wi < h->waves.size(); ++wi) {
    const Wave& w = h->waves[wi];
    int rc = build_wave_entries(h, w);
    if (rc != SQ_OK) return rc;
    int* out = h->wb.nl_cnt + 2;   // slab rows, brick images, tile rows, tile images; table rows, images
    SQ_CUDA_TRY(h, cudaMemsetAsync(out, 0, 6 * sizeof(int), s));
    k_wave_measure<<<w.ntiles, kThreads, 0, s>>>(g, h->wb.slab_n, h->wb.brick_n, h->wb.brick_rec, out);
    SQ_LAUNCH_CHECK(h);
    if (h->split_able) rc = count_nl_tables(h, wi, out + 4);
    if (rc != SQ_OK) return rc;
    int r[6];
    SQ_CUDA_TRY(h, cudaMemcpyAsync(r, out, sizeof(r), cudaMemcpyDeviceToHost, s));
    SQ_CUDA_TRY(h, cudaStreamSynchronize(s));
    h->wave_rows[wi] = r[0];
    h->wave_recs[wi] = r[1];
    NlNeed& n = h->wave_nl[wi];
    n.tile_rows = r[2];
    n.tile_imgs = r[3];
    n.x_rows = r[4];
    n.imgs = r[5];
  }
  bool split = false;
  for (size_t wi = 0; wi < h->waves.size(); ++wi) split = split || want_split(h, wi);
  return split ? ensure_nl_buffers(h) : SQ_OK;
}

template <typename Real>
static int apply_h_t(sq_handle* h, const Wave& w, const Real* v, Real* out, Real* P, const Real* chi, const Real* vpot,
                     const WaveBufs& b) {
  const Geo& g = h->geo;
  cudaStream_t s = h->stream;
  const bool one = h->max_nch == 1;
  (one ? k_project<Real, 1> : k_project<Real, 4>)<<<dim3(std::min(g.e_cap, 256), w.ntiles), kProjThreads, 0, s>>>(
      g, w, v, chi, h->d.atoms, h->d.rcmax, h->d.gdv, b.entries, b.n_entries, P);
  SQ_LAUNCH_CHECK(h);
  (one ? k_apply_h<Real, 1> : k_apply_h<Real, 4>)<<<dim3(g.nbricks, w.ntiles), kApplyThreads, 0, s>>>(
      g, w, v, out, P, chi, b.brick_rec, b.brick_n, vpot);
  SQ_LAUNCH_CHECK(h);
  return SQ_OK;
}

int launch_apply_h(sq_handle* h, const Wave& w, const double* v, double* out, double* P, const WaveBufs& b) {
  return apply_h_t<double>(h, w, v, out, P, h->d.chi64, h->d.v64, b);
}

int launch_apply_h(sq_handle* h, const Wave& w, const float* v, float* out, float* P, const WaveBufs& b) {
  return apply_h_t<float>(h, w, v, out, P, h->d.chi32, h->d.v32, b);
}

int run_sweep(sq_handle* h) {
  if (h->precision == SQ_FP64) return sweep_t<double>(h, h->d.chi64, h->d.v64, h->d.gdv64);
  return sweep_t<float>(h, h->d.chi32, h->d.v32, h->d.gdv32);
}

}  // namespace sq
