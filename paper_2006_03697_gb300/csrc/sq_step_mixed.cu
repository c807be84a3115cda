// The FP32 recurrence step of SQ_MIXED (at most 4 projector channels per atom), split so that every
// part has the data reuse it needs:
//
//   k_nl_apply    Y = sum_rows chi_row P^j[row] of every tile, on tensor cores (3-term TF32 split)
//   k_stencil     t^{j+1} = 2 Hhat t^j - t^{j-1} from t^j, Y, V_eff, and the S^j sums
//   k_nl_project  partial projections chi_row^T t^{j+1} per (brick, tile), on tensor cores
//   k_nl_reduce   P^{j+1}[row] = gamma |dOmega| sum over the bricks of the row's image
//
// One kernel over the bricks of a slab used to do all of it and gathered the projector values of every
// image from L2 for each tile (eight columns per value): 2.4 M warp instructions per tile and step,
// issue and latency bound. Here a block of the projector kernels owns one 4^3 brick of absolute
// lattice points and walks the tiles whose window holds that brick (up to prod(2 m + 2) / 64 of them; tiles
// whose origins agree modulo 4 share their bricks), with the brick's values as MMA fragments in
// registers; the stencil owns rows of a tile, keeps the z-neighbours in registers and the x-y plane in
// shared memory. Y lives in the buffer that receives t^{j+1}.
#include <algorithm>

#include "sq_device.cuh"

namespace sq {

constexpr int kNlThreads = 256;   // k_nl_apply: 8 warps
constexpr int kPrThreads = 256;   // k_nl_project: 8 warps over 1 .. 4 row tiles
constexpr int kNlRows = 64;       // projector rows of a brick per pass (eight K-steps of 8)
constexpr int kNlList = 352;      // (tile, brick) pairs per list
constexpr int kApG = 8;           // tiles per staged group of k_nl_apply (one per warp)
constexpr int kPrG = 8;           // of k_nl_project
__device__ __forceinline__ void cp16(unsigned dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src));
}

__device__ __forceinline__ float2 ld2g(const float* p) { return *reinterpret_cast<const float2*>(p); }

// The absolute bricks of a wave. Tile (tx, ty, tz) = 2 i + kappa has its window at 4 i + 2 kappa - m, so the tiles
// of one parity class kappa share the bricks beta = i + b, b the tile's brick. A grid over (beta_x, beta_y,
// 8 beta_z + class) needs no division to find its brick.
struct NlGrid {
  int tlo[3], thi[3];   // range of the wave's tiles per axis
  int nb[3];            // most bricks of a class per axis
  int z0, nz;           // brick layers of the launch (those the tiles of a chunk reach)
};

// of a wave, for a launch over its tiles [c0, c0 + cn)
static NlGrid nl_grid(const Geo& g, const Wave& w, int c0, int cn) {
  NlGrid r;
  const int t1 = w.tile0 + w.ntiles - 1, n01 = g.tiles[0] * g.tiles[1];
  const int lo[3] = {0, 0, w.tile0 / n01}, hi[3] = {g.tiles[0] - 1, g.tiles[1] - 1, t1 / n01};
  for (int a = 0; a < 3; ++a) {
    r.tlo[a] = lo[a];
    r.thi[a] = hi[a];
  }
  if (lo[2] == hi[2]) {
    r.tlo[1] = w.tile0 / g.tiles[0] % g.tiles[1];
    r.thi[1] = t1 / g.tiles[0] % g.tiles[1];
  }
  for (int a = 0; a < 3; ++a) r.nb[a] = (r.thi[a] - r.tlo[a] + 2) / 2 + g.nbr[a] - 1;
  const int z0 = (w.tile0 + c0) / n01, z1 = (w.tile0 + c0 + cn - 1) / n01;
  int f0 = r.nb[2], f1 = 0;
  for (int k = 0; k < 2; ++k) {   // tile layers of parity k
    const int base = std::max(0, (r.tlo[2] - k + 1) >> 1), ilo = std::max(0, (z0 - k + 1) >> 1), ihi = (z1 - k) >> 1;
    if (ihi < ilo) continue;
    f0 = std::min(f0, ilo - base);
    f1 = std::max(f1, ihi - base + g.nbr[2]);
  }
  r.z0 = f0;
  r.nz = f1 - f0;
  return r;
}
static NlGrid nl_grid(const Geo& g, const Wave& w) { return nl_grid(g, w, 0, w.ntiles); }

size_t nl_bricks_max(const Geo& g, int wave_cap) {   // of any wave of up to wave_cap contiguous tiles
  const long long n01 = (long long)g.tiles[0] * g.tiles[1];
  const int tz = int(std::min<long long>(g.tiles[2], (wave_cap + n01 - 1) / n01 + 1));
  const int t[3] = {g.tiles[0], g.tiles[1], tz};
  size_t n = 8;
  for (int a = 0; a < 3; ++a) n *= size_t((t[a] + 1) / 2 + g.nbr[a]);
  return n;
}

struct NlBrick {
  int beta[3], lo[3], cnt[3], kap[3];
  int index;   // of the brick's table entry
};

__device__ __forceinline__ bool nl_brick(const Geo& g, const NlGrid& n, NlBrick& r) {
  const int f[3] = {int(blockIdx.x), int(blockIdx.y), int(blockIdx.z >> 3) + n.z0}, cls = blockIdx.z & 7;
  for (int a = 0; a < 3; ++a) {
    r.kap[a] = (cls >> a) & 1;
    const int ilo = max(0, (n.tlo[a] - r.kap[a] + 1) >> 1), ihi = (n.thi[a] - r.kap[a]) >> 1;   // ihi < ilo: no tile
    if (ihi < ilo || f[a] >= ihi - ilo + g.nbr[a]) return false;
    r.beta[a] = ilo + f[a];
    r.lo[a] = max(ilo, r.beta[a] - g.nbr[a] + 1);
    r.cnt[a] = min(ihi, r.beta[a]) - r.lo[a] + 1;
  }
  r.index = ((8 * f[2] + cls) * n.nb[1] + f[1]) * n.nb[0] + f[0];
  return true;
}

// table entry of brick br of global tile t
__device__ __forceinline__ int nl_index(const Geo& g, const NlGrid& n, int t, int br) {
  const int tc[3] = {t % g.tiles[0], t / g.tiles[0] % g.tiles[1], t / (g.tiles[0] * g.tiles[1])};
  const int b[3] = {br % g.nbr[0], br / g.nbr[0] % g.nbr[1], br / (g.nbr[0] * g.nbr[1])};
  int f[3], cls = 0;
  for (int a = 0; a < 3; ++a) {
    const int k = tc[a] & 1;
    f[a] = (tc[a] >> 1) + b[a] - max(0, (n.tlo[a] - k + 1) >> 1);
    cls |= k << a;
  }
  return ((8 * f[2] + cls) * n.nb[1] + f[1]) * n.nb[0] + f[0];
}

// Where the partial projections of a chunk's tiles go: off[tile of the wave][brick] = the brick's first row among
// the tile's (-1: the tile is left out), rows of Part per tile
struct NlPart {
  const int* off;
  int rows;
};

struct NlShared {
  // tile of the chunk, tile * nbricks + brick (apply) or first row in Part (project), first point of the brick in
  // the tile's window, points of the brick inside the window in y | in z << 4
  int4 list[kNlList];
  int img[32];                   // first row (of the pass) << 4 | channels of the images of the pass
  int n, nb, nrows, nimg, row0;
  int x0;                        // the brick's first row in X
};

// the brick's tiles among tiles [c0, c0 + cn) of the wave, entries [i0, i0 + kNlList) of the class box, by
// threads first, first + 1, ... of the block (between barriers; sh.n starts at 0)
__device__ __forceinline__ void nl_list(const Geo& g, const Wave& w, int c0, int cn, const NlBrick& b, int i0, int first,
                                        const NlPart& part, NlShared& sh) {
  const int total = b.cnt[0] * b.cnt[1] * b.cnt[2], n = min(kNlList, total - i0);
  for (int i = int(threadIdx.x) - first; i >= 0 && i < n; i += blockDim.x - first) {
    const int f = i0 + i, f1 = f / b.cnt[0], f2 = f1 / b.cnt[1];
    const int i3[3] = {b.lo[0] + f - f1 * b.cnt[0], b.lo[1] + f1 - f2 * b.cnt[1], b.lo[2] + f2};
    const int tl = 2 * i3[0] + b.kap[0] + g.tiles[0] * (2 * i3[1] + b.kap[1] + g.tiles[1] * (2 * i3[2] + b.kap[2])) -
                   w.tile0 - c0;
    if (tl < 0 || tl >= cn) continue;
    const int bx = b.beta[0] - i3[0], by = b.beta[1] - i3[1], bz = b.beta[2] - i3[2];
    int y = tl * g.nbricks + (bz * g.nbr[1] + by) * g.nbr[0] + bx;
    if (part.off) {
      const int o = __ldg(part.off + (size_t)c0 * g.nbricks + y);
      if (o < 0) continue;
      y = tl * part.rows + o;
    }
    sh.list[atomicAdd(&sh.n, 1)] = make_int4(tl, y, kBrick * ((bz * g.U[1] + by) * g.U[0] + bx),
                                             min(kBrick, g.U[1] - kBrick * by) | min(kBrick, g.U[2] - kBrick * bz) << 4);
  }
}

// Table of the wave's bricks, built with its lists and read by every step. head [brick] = {images, rows, first row
// in X, c}: c >= 0: every image has c channels, else its image list (first row << 4 | channels) starts at
// img[-1 - c]; X [rows][64 points] = the image's channel at the brick's points as a TF32 (hi, lo) pair, zero
// outside the support sphere. The records of all tiles that share a brick list the same images in the same
// order, so any of them will do. Rows are handed out by a counter, a brick taking what it needs: the sum over the
// bricks hardly depends on where the atoms are, while the fullest brick of a cluster holds several times the mean
// (a fixed number of rows per brick had to be 2.5 times the mean and sent clusters to the scalar step: 48 H in a
// 3.9 bohr sphere of a 16 bohr cell, 257 ms an evaluation with the step before the split one, 506 with the scalar one).
// cnt [2] = rows, images needed; X null: counts only.
__global__ void __launch_bounds__(128)
k_nl_table(Geo g, Wave w, NlGrid grid, const float* __restrict__ chis, const int4* __restrict__ brec,
           const int* __restrict__ bn, long long rows_cap, long long img_cap, int* __restrict__ cnt, int4* __restrict__ head,
           int* __restrict__ img, float2* __restrict__ X, int* __restrict__ status) {
  __shared__ NlShared sh;
  __shared__ int row_of[32], wsum[4], wlo[4], whi[4];
  __shared__ int4 hd_s;
  NlBrick b;
  if (!nl_brick(g, grid, b)) return;
  const int total = b.cnt[0] * b.cnt[1] * b.cnt[2], lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i0 = 0; i0 < total; i0 += kNlList) {
    __syncthreads();
    if (threadIdx.x == 0) sh.n = 0;
    __syncthreads();
    nl_list(g, w, 0, w.ntiles, b, i0, 0, NlPart{nullptr, 0}, sh);
    __syncthreads();
    if (sh.n == 0) continue;
    const size_t tb = sh.list[0].y;
    const int4* rec = brec + tb * g.br_cap * 2;
    const int nb = bn[tb];
    int sum = 0, lo = kMaxCh, hi = 0;   // rows; fewest and most channels of an image
    for (int k = threadIdx.x; k < nb; k += blockDim.x) {
      const int nch = rec[2 * k].w & 0xff;
      sum += nch;
      lo = min(lo, nch);
      hi = max(hi, nch);
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
      wsum[warp] = sum;
      wlo[warp] = lo;
      whi[warp] = hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      const int rows = wsum[0] + wsum[1] + wsum[2] + wsum[3];
      const int l = min(min(wlo[0], wlo[1]), min(wlo[2], wlo[3])), h = max(max(whi[0], whi[1]), max(whi[2], whi[3]));
      const bool list = nb > 0 && l != h;
      int4 hd = make_int4(nb, rows, atomicAdd(cnt, rows), nb > 0 ? h : 0);
      if (list) hd.w = -1 - atomicAdd(cnt + 1, nb);
      if (X && (hd.z + (long long)rows > rows_cap || (list && -1ll - hd.w + nb > img_cap))) {
        atomicOr(status + kStOverflow, 8);   // a launch sized for another layout (a stale graph): refuse
        hd = make_int4(0, 0, 0, 0);
      }
      hd_s = hd;
      if (X) head[b.index] = hd;
    }
    __syncthreads();
    const int4 hd = hd_s;
    if (!X || hd.x == 0) return;
    float2* Xb = X + (size_t)hd.z * 64;
    int row = 0;
    for (int k0 = 0; k0 < nb; k0 += 32) {
      const int k = k0 + lane, nch = k < nb ? rec[2 * k].w & 0xff : 0;
      int incl = nch;
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += v;
      }
      __syncthreads();
      if (warp == 0) {
        row_of[lane] = row + incl - nch;
        if (hd.w < 0 && k < nb) img[-1 - hd.w + k] = (row + incl - nch) << 4 | nch;
      }
      row += __shfl_sync(0xffffffffu, incl, 31);
      __syncthreads();
      for (int i = warp; i < min(32, nb - k0); i += 4) {
        const int4 r0 = rec[2 * (k0 + i)], r1 = rec[2 * (k0 + i) + 1];
        for (int h = 0; h < 2; ++h) {   // points lane and lane + 32
          const bool in = (unsigned(h ? r1.w : r1.z) >> lane) & 1u;
          const float* c0 = chis + 2 * (r0.x + (((2 * h + (lane >> 4)) * r1.y + ((lane >> 2) & 3)) * r1.x + (lane & 3)) * 4);
          for (int ch = 0; ch < (r0.w & 0xff); ++ch)
            Xb[(row_of[i] + ch) * 64 + 32 * h + lane] = in ? ld2g(c0 + 2 * ch) : make_float2(0.f, 0.f);
        }
      }
    }
    return;
  }
  if (threadIdx.x == 0 && X) head[b.index] = make_int4(0, 0, 0, 0);
}

// The next pass over the brick's images (from image k0 on, as many as fit 32 images, one per lane, and
// kNlRows rows): sh.nimg, sh.nrows, their rows, and sh.row0, the pass's first row of the brick. One warp.
__device__ __forceinline__ void nl_pass(const int4* __restrict__ hd_p, const int* __restrict__ img, int k0, NlShared& sh) {
  const int4 hd = __ldg(hd_p);
  const int lane = threadIdx.x & 31, nb = hd.x, k = k0 + lane;
  const int x = k < nb ? (hd.w >= 0 ? (k * hd.w) << 4 | hd.w : __ldg(img - 1 - hd.w + k)) : 0;
  const int first = __shfl_sync(0xffffffffu, x >> 4, 0), end = (x >> 4) + (x & 15) - first;
  const bool fits = k < nb && end <= kNlRows;
  sh.img[lane] = ((x >> 4) - first) << 4 | (x & 15);
  const unsigned m = __ballot_sync(0xffffffffu, fits);
  if (lane == 0) {
    sh.nb = nb;
    sh.nimg = __popc(m);
    sh.row0 = first;
    sh.x0 = hd.z;
    if (!m) sh.nrows = 0;
  }
  if (m && lane == 31 - __clz(m)) sh.nrows = end;
}

// Tiles i0 .. of the brick and the first pass of its images, side by side: warp 0 reads the brick's
// table entry while the others list its tiles.
__device__ __forceinline__ void nl_begin(const Geo& g, const Wave& w, int c0, int cn, const NlBrick& b, int i0,
                                         const NlPart& part, const int4* __restrict__ hd, const int* __restrict__ img,
                                         NlShared& sh) {
  __syncthreads();
  if (threadIdx.x == 0) sh.n = 0;
  __syncthreads();
  if (threadIdx.x < 32) nl_pass(hd, img, 0, sh);
  else nl_list(g, w, c0, cn, b, i0, 32, part, sh);
  __syncthreads();
}

__device__ __forceinline__ void nl_next(const int4* __restrict__ hd, const int* __restrict__ img, int k0, NlShared& sh) {
  __syncthreads();
  if (threadIdx.x < 32) nl_pass(hd, img, k0, sh);
  __syncthreads();
}

// Y[64 points][8 nodes] = X[64][rows] P^j[rows][8] of every tile that holds the brick. P^j is kept split as TF32
// hi and lo planes; per group of kApG tiles its rows are copied to shared memory once (cp.async; a warp
// copies one tile, its row numbers read a group ahead) and serve the four z-planes of the brick: a warp
// owns a z-plane (M = 16 points; A fragments of up to 64 rows in registers) and every second tile. Planes of
// hi and lo keep each B register a load of its own: pairs loaded as (hi, lo) had to be moved apart again.
template <int NKS>
__device__ __forceinline__ void nl_apply_pass(const Geo& g, NlShared& sh, float* Bs, int k0, int max_nch,
                                              const float2* __restrict__ X, const float* __restrict__ P, size_t lo_plane,
                                              const int4* __restrict__ brec, float* __restrict__ Y) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g8 = lane >> 2, t4 = lane & 3;
  const int mt = warp & 3, p = 16 * mt + g8, n = sh.n, nimg = sh.nimg, nrows = sh.nrows;
  constexpr int kPlane = 8 * NKS * 8, kTile = 2 * kPlane;   // floats of one plane, one staged tile
  const unsigned bs = (unsigned)__cvta_generic_to_shared(Bs) + warp * kTile * 4;
  // lane = image: first row << 4 | channels, and its first projector row in the warp's tile of a group
  const int img = sh.img[lane];
  const int* recy = reinterpret_cast<const int*>(brec) + 8 * (k0 + min(lane, max(nimg - 1, 0))) + 1;
  auto look_up = [&](int j) { return j < n ? __ldg(recy + (unsigned long long)(unsigned)sh.list[j].y * (unsigned)(8 * g.br_cap)) : 0; };
  int r0v = look_up(warp);
  uint32_t ah[NKS + 1][4], al[NKS + 1][4];   // (one spare: no zero-size arrays)
#pragma unroll
  for (int ks = 0; ks < NKS; ++ks) {
    const float2* xr = X + (8 * ks + t4) * 64 + p;
    const bool in0 = 8 * ks + t4 < nrows, in1 = 8 * ks + t4 + 4 < nrows;   // (another pass's or brick's rows follow)
    const float2 zero = make_float2(0.f, 0.f);
    const float2 x0 = in0 ? __ldg(xr) : zero, x1 = in0 ? __ldg(xr + 8) : zero;
    const float2 x2 = in1 ? __ldg(xr + 256) : zero, x3 = in1 ? __ldg(xr + 264) : zero;
    ah[ks][0] = __float_as_uint(x0.x); al[ks][0] = __float_as_uint(x0.y);
    ah[ks][1] = __float_as_uint(x1.x); al[ks][1] = __float_as_uint(x1.y);
    ah[ks][2] = __float_as_uint(x2.x); al[ks][2] = __float_as_uint(x2.y);
    ah[ks][3] = __float_as_uint(x3.x); al[ks][3] = __float_as_uint(x3.y);
  }
  // an image's rows are 32 nch contiguous bytes in each plane; a lane copies 16 bytes, 32 / (4 max_nch) images
  // at a time (lanes: image, plane, piece)
  const int lpi = max_nch == 3 ? 16 : 4 * max_nch, ips = 32 / lpi, half = lpi / 2;
  const int sub = lane / lpi, pl = lane % lpi / half, pc = lane % half;
  const size_t src0 = pl * lo_plane + 4 * pc;
  const int dst0 = (pl * kPlane + 4 * pc) * 4;
  auto copy = [&](int j, int buf) {
    if (j < n) {
      const float* Pt = P + (unsigned long long)(unsigned)sh.list[j].x * (unsigned)(g.r_cap * 8) + src0;
      const unsigned d = bs + buf * (kApG * kTile * 4) + dst0;
      for (int i = sub; i < nimg + sub; i += ips) {   // (all lanes take part in the shuffles)
        const int im = __shfl_sync(0xffffffffu, img, i), r0 = __shfl_sync(0xffffffffu, r0v, i);
        if (i < nimg && pc < 2 * (im & 15)) cp16(d + (im >> 4) * 32, Pt + r0 * 8);
      }
    }
    asm volatile("cp.async.commit_group;");
  };
  // rows past the last one multiply zero A values: clear them once (stale bits could be NaN)
  for (int i = threadIdx.x; i < 2 * kApG * kTile / 4; i += kNlThreads) reinterpret_cast<float4*>(Bs)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  const int poff = (mt * g.U[0] * g.U[1] + (g8 >> 2) * g.U[0] + (g8 & 3)) * 8 + 2 * t4;
  __syncthreads();
  copy(warp, 0);
  r0v = look_up(kApG + warp);
  int buf = 0;
  for (int j0 = 0; j0 < n; j0 += kApG, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;");
    __syncthreads();   // the group has landed; the other buffer is free
    if (j0 + kApG < n) {
      copy(j0 + kApG + warp, buf ^ 1);
      r0v = look_up(j0 + 2 * kApG + warp);
    }
    for (int tt = warp >> 2; tt < kApG && j0 + tt < n; tt += 2) {
      const int4 cur = sh.list[j0 + tt];
      const float* bt = Bs + (buf * kApG + tt) * kTile + t4 * 8 + g8;
      float* y0 = Y + (unsigned long long)(unsigned)cur.x * (unsigned)(g.Upts * 8) + (cur.z * 8 + poff);
      float* y1 = y0 + 16 * g.U[0];
      const int ny = cur.w & 15;
      const bool inz = mt < (cur.w >> 4), s0 = inz && (g8 >> 2) < ny, s1 = inz && (g8 >> 2) + 2 < ny;
      float dh[4] = {0.f, 0.f, 0.f, 0.f}, dl[4] = {0.f, 0.f, 0.f, 0.f};
      if (k0 > 0) {
        const float2 a = s0 ? ld2g(y0) : make_float2(0.f, 0.f), c = s1 ? ld2g(y1) : make_float2(0.f, 0.f);
        dh[0] = a.x; dh[1] = a.y; dh[2] = c.x; dh[3] = c.y;
      }
#pragma unroll
      for (int ks = 0; ks < NKS; ++ks) {
        const uint32_t bh[2] = {__float_as_uint(bt[64 * ks]), __float_as_uint(bt[64 * ks + 32])};
        const uint32_t bl[2] = {__float_as_uint(bt[kPlane + 64 * ks]), __float_as_uint(bt[kPlane + 64 * ks + 32])};
        mma_tf32(dl, al[ks], bh);   // small terms in their own sum (a third one cost more moves than it hid)
        mma_tf32(dl, ah[ks], bl);
        float d[4];
        mma_tf32_set(d, ah[ks], bh);
#pragma unroll
        for (int i = 0; i < 4; ++i) dh[i] += d[i];
      }
      if (s0) *reinterpret_cast<float2*>(y0) = make_float2(dh[0] + dl[0], dh[1] + dl[1]);
      if (s1) *reinterpret_cast<float2*>(y1) = make_float2(dh[2] + dl[2], dh[3] + dl[3]);
    }
  }
}

constexpr size_t kApSmem = (sizeof(NlShared) + 15) / 16 * 16 + 2 * kApG * kNlRows * 16 * sizeof(float);

__global__ void __launch_bounds__(kNlThreads, 2)
k_nl_apply(Geo g, Wave w, NlGrid grid, int max_nch, const float* __restrict__ P, size_t lo_plane,
           const int4* __restrict__ head, const int* __restrict__ img, const float2* __restrict__ X,
           const int4* __restrict__ brec, float* __restrict__ Y) {
  extern __shared__ __align__(16) unsigned char nl_smem[];
  NlShared& sh = *reinterpret_cast<NlShared*>(nl_smem);
  float* Bs = reinterpret_cast<float*>(nl_smem + (sizeof(NlShared) + 15) / 16 * 16);
  NlBrick b;
  if (!nl_brick(g, grid, b)) return;
  const int4* hd = head + b.index;
  const int total = b.cnt[0] * b.cnt[1] * b.cnt[2];
  for (int i0 = 0; i0 < total; i0 += kNlList) {
    nl_begin(g, w, 0, w.ntiles, b, i0, NlPart{nullptr, 0}, hd, img, sh);
    if (sh.n == 0) continue;
    int k0 = 0;
    for (;;) {
      const float2* Xp = X + (size_t)(sh.x0 + sh.row0) * 64;
      switch ((sh.nrows + 7) / 8) {
        case 0: nl_apply_pass<0>(g, sh, Bs, k0, max_nch, Xp, P, lo_plane, brec, Y); break;
        case 1: nl_apply_pass<1>(g, sh, Bs, k0, max_nch, Xp, P, lo_plane, brec, Y); break;
        case 2: nl_apply_pass<2>(g, sh, Bs, k0, max_nch, Xp, P, lo_plane, brec, Y); break;
        case 3: nl_apply_pass<3>(g, sh, Bs, k0, max_nch, Xp, P, lo_plane, brec, Y); break;
        case 4: nl_apply_pass<4>(g, sh, Bs, k0, max_nch, Xp, P, lo_plane, brec, Y); break;
        case 5: nl_apply_pass<5>(g, sh, Bs, k0, max_nch, Xp, P, lo_plane, brec, Y); break;
        case 6: nl_apply_pass<6>(g, sh, Bs, k0, max_nch, Xp, P, lo_plane, brec, Y); break;
        case 7: nl_apply_pass<7>(g, sh, Bs, k0, max_nch, Xp, P, lo_plane, brec, Y); break;
        default: nl_apply_pass<8>(g, sh, Bs, k0, max_nch, Xp, P, lo_plane, brec, Y); break;
      }
      k0 += sh.nimg;
      if (k0 >= sh.nb) break;
      nl_next(hd, img, k0, sh);
    }
  }
}

// Part[tile][off[tile][brick] + row][8 nodes] = X^T[rows][64 points] t[64 points][8] of every tile that holds the
// brick (rows of the brick in record order). Per group of kPrG tiles t is read once (16 bytes a load, one
// group ahead), split to TF32 (hi, lo) and staged in shared memory for the brick's row tiles: a warp owns
// 16 rows (A fragments of the 64 points in registers), 16 shared loads and 24 MMAs per tile. Loading and
// splitting t in every warp took 300 instructions per row tile and tile.
constexpr int kPrTile = 2 * 64 * 8;   // floats of one staged tile: hi and lo planes [64 points][8 nodes]
constexpr size_t kPrSmem = (sizeof(NlShared) + 15) / 16 * 16 + 2 * kPrG * kPrTile * sizeof(float);

__global__ void __launch_bounds__(kPrThreads, 2)
k_nl_project(Geo g, Wave w, NlGrid grid, int c0, int cn, const float* __restrict__ T, const int4* __restrict__ head,
             const int* __restrict__ img, const float2* __restrict__ X, NlPart part, float* __restrict__ Part) {
  extern __shared__ __align__(16) unsigned char nl_smem[];   // tiles c0 .. c0 + cn - 1 of the wave
  NlShared& sh = *reinterpret_cast<NlShared*>(nl_smem);
  float* Bs = reinterpret_cast<float*>(nl_smem + (sizeof(NlShared) + 15) / 16 * 16);
  NlBrick b;
  if (!nl_brick(g, grid, b)) return;
  const int4* hd = head + b.index;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g8 = lane >> 2, t4 = lane & 3;
  const int total = b.cnt[0] * b.cnt[1] * b.cnt[2];
  const float* Tw = T + (size_t)c0 * g.Upts * 8;
  // staging: the thread takes half (four nodes) h4 of point pt of tiles tile0, tile0 + 2, ...
  constexpr int kIt = kPrG * 128 / kPrThreads, kTs = kPrThreads / 128;
  const int pt = (threadIdx.x & 127) >> 1, h4 = threadIdx.x & 1, tile0 = threadIdx.x >> 7;
  const int py = (pt >> 2) & 3, pz = pt >> 4;
  const int toff = ((pz * g.U[1] + py) * g.U[0] + (pt & 3)) * 8 + 4 * h4;
  for (int i0 = 0; i0 < total; i0 += kNlList) {
    nl_begin(g, w, c0, cn, b, i0, part, hd, img, sh);
    const int n = sh.n;
    if (n == 0 || sh.nb == 0) continue;
    for (int k0 = 0;;) {
      const int nrows = sh.nrows, nmt = (nrows + 15) / 16, rbase = sh.row0;
      // 1 .. 4 row tiles (three: the third on two of the eight warps), every str-th tile of a group
      const int mt = warp % nmt, str = kPrThreads / 32 / nmt + (mt < (kPrThreads / 32) % nmt), r = 16 * mt + g8;
      uint32_t ah[8][4], al[8][4];
      {
        const float2 *x0p = X + (size_t)(sh.x0 + rbase + r) * 64 + t4, *x1p = x0p + 8 * 64;
        const bool in0 = r < nrows, in1 = r + 8 < nrows;   // (another pass's or brick's rows follow)
        const float2 zero = make_float2(0.f, 0.f);
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
          const float2 x0 = in0 ? __ldg(x0p + 8 * ks) : zero, x1 = in1 ? __ldg(x1p + 8 * ks) : zero;
          const float2 x2 = in0 ? __ldg(x0p + 8 * ks + 4) : zero, x3 = in1 ? __ldg(x1p + 8 * ks + 4) : zero;
          ah[ks][0] = __float_as_uint(x0.x); al[ks][0] = __float_as_uint(x0.y);
          ah[ks][1] = __float_as_uint(x1.x); al[ks][1] = __float_as_uint(x1.y);
          ah[ks][2] = __float_as_uint(x2.x); al[ks][2] = __float_as_uint(x2.y);
          ah[ks][3] = __float_as_uint(x3.x); al[ks][3] = __float_as_uint(x3.y);
        }
      }
      float4 tv[kIt];
      auto load = [&](int j0) {
#pragma unroll
        for (int i = 0; i < kIt; ++i) {
          const int j = j0 + tile0 + kTs * i;
          tv[i] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (j < n) {
            const int4 tb = sh.list[j];
            if (py < (tb.w & 15) && pz < (tb.w >> 4))
              tv[i] = *reinterpret_cast<const float4*>(Tw + (unsigned long long)(unsigned)tb.x * (unsigned)(g.Upts * 8) + (tb.z * 8 + toff));
          }
        }
      };
      auto stage = [&](int buf) {
#pragma unroll
        for (int i = 0; i < kIt; ++i) {
          uint32_t hi[4], lo[4];
          split_tf32(tv[i].x, hi[0], lo[0]);
          split_tf32(tv[i].y, hi[1], lo[1]);
          split_tf32(tv[i].z, hi[2], lo[2]);
          split_tf32(tv[i].w, hi[3], lo[3]);
          float* d = Bs + (buf * kPrG + tile0 + kTs * i) * kPrTile + pt * 8 + 4 * h4;
          *reinterpret_cast<uint4*>(d) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          *reinterpret_cast<uint4*>(d + 512) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
      };
      float* po = Part + (size_t)(rbase + r) * 8 + 2 * t4;
      load(0);
      stage(0);
      int buf = 0;
      for (int j0 = 0; j0 < n; j0 += kPrG, buf ^= 1) {
        __syncthreads();   // the group is staged; the other buffer is free
        const bool more = j0 + kPrG < n;
        if (more) load(j0 + kPrG);
        for (int tt = warp / nmt; tt < kPrG && j0 + tt < n; tt += str) {
          const int4 cur = sh.list[j0 + tt];
          const float* bt = Bs + (buf * kPrG + tt) * kPrTile + t4 * 8 + g8;
          float dh[4] = {0.f, 0.f, 0.f, 0.f}, dl[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int ks = 0; ks < 8; ++ks) {
            const uint32_t bh[2] = {__float_as_uint(bt[64 * ks]), __float_as_uint(bt[64 * ks + 32])};
            const uint32_t bl[2] = {__float_as_uint(bt[512 + 64 * ks]), __float_as_uint(bt[512 + 64 * ks + 32])};
            mma_tf32(dl, al[ks], bh);
            mma_tf32(dl, ah[ks], bl);
            float d[4];
            mma_tf32_set(d, ah[ks], bh);
#pragma unroll
            for (int i = 0; i < 4; ++i) dh[i] += d[i];
          }
          float* o = po + (size_t)cur.y * 8;
          if (r < nrows) *reinterpret_cast<float2*>(o) = make_float2(dh[0] + dl[0], dh[1] + dl[1]);
          if (r + 8 < nrows) *reinterpret_cast<float2*>(o + 64) = make_float2(dh[2] + dl[2], dh[3] + dl[3]);
        }
        if (more) stage(buf ^ 1);
      }
      k0 += sh.nimg;
      if (k0 >= sh.nb) break;
      nl_next(hd, img, k0, sh);
    }
  }
}

// Per tile: its bricks' first rows in Part (off, brick order), and per image the rows of its first channel, of the
// bricks it meets in brick order. One thread per image searches the record lists (ascending image order) of the
// bricks its box overlaps. A tile with more rows or images than the launch was sized for (a stale graph) is refused:
// off = -1 and no entries, so nothing reaches past Part or idx.
__global__ void __launch_bounds__(256)
k_nl_index(Geo g, Wave w, NlGrid grid, const AtomTab* __restrict__ atoms, const TileEntry* __restrict__ entries,
           const int* __restrict__ n_entries, const int* __restrict__ blist, const int* __restrict__ bn,
           const int4* __restrict__ head, const int* __restrict__ img, int rows_cap, int idx_cap, int* off_, int* start,
           int* __restrict__ idx, int* __restrict__ status) {
  const int tl = blockIdx.x, t = wave_tile(w, tl);
  int o[3];
  tile_origin(g, t, o);
  const int ne = n_entries[tl];
  const TileEntry* ent = entries + (size_t)tl * g.e_cap;
  int* st = start + (size_t)tl * (g.e_cap + 1);
  int* ix = idx + (size_t)tl * idx_cap;
  int* off = off_ + (size_t)tl * g.nbricks;
  int rows = 0;
  for (int b0 = 0; b0 < g.nbricks; b0 += blockDim.x) {
    const int br = b0 + threadIdx.x;
    int tot;
    const int first = block_exclusive_scan(br < g.nbricks ? head[nl_index(g, grid, t, br)].y : 0, &tot);
    if (br < g.nbricks) off[br] = rows + first;
    rows += tot;
  }
  __syncthreads();
  int base = 0;
  for (int e0 = 0; e0 < ne; e0 += blockDim.x) {
    const int e = e0 + threadIdx.x;
    int lo[3] = {0, 0, 0}, hi[3] = {-1, -1, -1};
    if (e < ne) {
      const TileEntry te = ent[e];
      const AtomTab& at = atoms[te.atom];
      for (int a = 0; a < 3; ++a) {
        const int bl = at.lo[a] + te.s[a] * g.n[a] - (o[a] - g.m[a]);   // box corner in U-local coords
        lo[a] = max(0, bl) / kBrick;
        hi[a] = min(g.nbr[a] - 1, floor_div_d(bl + at.dim[a] - 1, kBrick));
      }
    }
    auto walk = [&](bool fill, int at0) {
      int cnt = 0;
      for (int bz = lo[2]; bz <= hi[2]; ++bz)
        for (int by = lo[1]; by <= hi[1]; ++by)
          for (int bx = lo[0]; bx <= hi[0]; ++bx) {
            const int br = (bz * g.nbr[1] + by) * g.nbr[0] + bx;
            const size_t tb = (size_t)tl * g.nbricks + br;
            const int* l = blist + tb * g.br_cap;
            const int nb = bn[tb];
            int a = 0, c = nb;
            while (a < c) {
              const int mid = (a + c) >> 1;
              if (l[mid] < e) a = mid + 1;
              else c = mid;
            }
            if (a < nb && l[a] == e) {
              const int4 hd = head[nl_index(g, grid, t, br)];
              if (hd.x == 0) continue;   // a brick without a table (refused): nothing of it is in Part
              if (fill && at0 + cnt < idx_cap) ix[at0 + cnt] = off[br] + (hd.w >= 0 ? a * hd.w : img[-1 - hd.w + a] >> 4);
              ++cnt;
            }
          }
      return cnt;
    };
    int tot;
    const int first = block_exclusive_scan(e < ne ? walk(false, 0) : 0, &tot);
    if (e < ne) {
      st[e] = base + first;
      walk(true, base + first);
    }
    base += tot;
  }
  if (threadIdx.x == 0) st[ne] = base;
  if (rows <= rows_cap && base <= idx_cap) return;
  __syncthreads();
  for (int e = threadIdx.x; e <= ne; e += blockDim.x) st[e] = 0;
  for (int br = threadIdx.x; br < g.nbricks; br += blockDim.x) off[br] = -1;
  if (threadIdx.x == 0) atomicOr(status + kStOverflow, 16);
}

// P[row][q] = gamma |dOmega| times the sum of the row's partial projections over its bricks, as pairs of floats
// (two-sum; FP64 adds issue at 1.7 lanes per clock), in a fixed order: rounded once and split to TF32 planes
// (hi, lo) for the apply in P, the pair in Pp. One warp per image: its 8 nch values are 2 nch groups of four, so 16 / nch bricks are read at once
// (one brick at a time left too few loads in flight), then added over the lanes that share a group.
__device__ __forceinline__ void pair_add(float& h, float& l, float vh, float vl) {
  const float s = __fadd_rn(h, vh), z = __fsub_rn(s, h);
  l = __fadd_rn(l, __fadd_rn(__fadd_rn(__fsub_rn(h, __fsub_rn(s, z)), __fsub_rn(vh, z)), vl));
  h = s;
}

__global__ void __launch_bounds__(128)
k_nl_reduce(Geo g, int tl0, const TileEntry* __restrict__ entries, const int* __restrict__ n_entries,
            const AtomTab* __restrict__ atoms, const float2* __restrict__ gdvp, const int* __restrict__ start,
            const int* __restrict__ idx, int idx_cap, int rows_cap, const float* __restrict__ Part, float* __restrict__ P,
            size_t lo_plane, float2* __restrict__ Pp) {
  const int tc = blockIdx.x, tl = tl0 + tc, lane = threadIdx.x & 31;
  const int* st = start + (size_t)tl * (g.e_cap + 1);
  const int* ix = idx + (size_t)tl * idx_cap;
  const float4* pt = reinterpret_cast<const float4*>(Part + (size_t)tc * rows_cap * 8);
  const int ne = n_entries[tl];
  for (int e = blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5); e < ne; e += gridDim.y * (blockDim.x >> 5)) {
    const TileEntry te = entries[(size_t)tl * g.e_cap + e];
    const int nch = atoms[te.atom].nch, ch0 = atoms[te.atom].ch0;
    const int grp = nch == 3 ? 8 : 2 * nch, nsub = 32 / grp;   // lanes per brick (two idle with 3 channels)
    const int sub = lane / grp, v4 = lane % grp;
    const int i0 = st[e], i1 = st[e + 1];
    float h[4] = {0.f, 0.f, 0.f, 0.f}, l[4] = {0.f, 0.f, 0.f, 0.f};
    if (v4 < 2 * nch) {
#pragma unroll 4
      for (int i = i0 + sub; i < i1; i += nsub) {
        const float4 v = pt[ix[i] * 2 + v4];
        pair_add(h[0], l[0], v.x, 0.f);
        pair_add(h[1], l[1], v.y, 0.f);
        pair_add(h[2], l[2], v.z, 0.f);
        pair_add(h[3], l[3], v.w, 0.f);
      }
    }
    for (int d = grp; d < 32; d <<= 1)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        pair_add(h[q], l[q], __shfl_xor_sync(0xffffffffu, h[q], d), __shfl_xor_sync(0xffffffffu, l[q], d));
    if (lane < 2 * nch) {
      const float2 gd = gdvp[ch0 + (lane >> 1)];
      const size_t k = ((size_t)tl * g.r_cap + te.row0) * 8 + 4 * lane;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float p = h[q] * gd.x, t = fmaf(h[q], gd.x, -p) + (h[q] * gd.y + l[q] * gd.x);
        const float r = p + t;
        uint32_t hi, lo;
        split_tf32(r, hi, lo);
        P[k + q] = __uint_as_float(hi);
        P[lo_plane + k + q] = __uint_as_float(lo);
        Pp[k + q] = make_float2(r, t - (r - p));
      }
    }
  }
}

// ------------------------------------------------------------------------------ stencil
// t^{j+1} on ty rows (all x) of a tile, marching in z. A thread owns one (x, y) and a node pair: the z
// neighbours are a sliding window of registers, the x and y neighbours come from the plane in shared
// memory (with its halo rows, zeros past the window's edge, so no tap is checked), and W, Y, t^{j-1} of the next
// planes are copied ahead into shared memory (cp.async), which keeps tens of kilobytes per SM in
// flight without registers. 28 bytes per point and node pass (t^j, t^{j-1}, Y and W read, t^{j+1}
// written). 512 tiles of 28^3 windows: 0.71 ms, 2.15 GB of DRAM traffic, 45 % of a plain copy's rate; the block's 14
// warps (127 registers each: two planes' z windows, taps and S sums) issue in 58 % of the cycles, and that,
// not the traffic or the instruction count, bounds it (packed differences: 4 % fewer instructions, 0.73 ms; a
// second block per SM at 72 registers spills).
__device__ __forceinline__ void cp8(unsigned dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src));
}

__host__ __device__ inline int st_plane_floats(int Ux, int ty, int no) { return ((ty + 2 * no) * (Ux + no) + no) * 8; }

template <int NO, int MAXT, int MINB, int NST>
__global__ void __launch_bounds__(MAXT, MINB)
k_stencil(Geo g, Wave w, const float* __restrict__ Tc, const float* __restrict__ Tp, float* Tn, int has_y,
          const float* __restrict__ Wt, const float* __restrict__ v, const double* __restrict__ scal, int mode,
          const double* __restrict__ ncoef, int ty, double* __restrict__ Spart) {
  extern __shared__ __align__(16) float st_smem[];
  const int chunk = blockIdx.x, tl = blockIdx.y, t = wave_tile(w, tl);
  const int Ux = g.U[0], Uy = g.U[1], Uz = g.U[2];
  const int y0 = chunk * ty, tyn = min(ty, Uy - y0);
  const int pitch = (Ux + NO) * 8, plane = st_plane_floats(Ux, ty, NO), nthr = blockDim.x;
  float* planes = st_smem;                                   // [NST][2][plane]
  constexpr int kOwn = 5 * 2 * MAXT;
  float* own = planes + 2 * NST * plane;                     // [NST][2][5][MAXT * 2]: t^{j-1}, Y, W x 3
  const int nact = Ux * tyn * 4;                             // threads that own a column
  const int pair = threadIdx.x & 3, xi = (threadIdx.x >> 2) % Ux, yi = (threadIdx.x >> 2) / Ux;
  const bool act = threadIdx.x < nact;
  int o[3];
  tile_origin(g, t, o);
  const size_t tbase = (size_t)tl * g.Upts * 8;
  const float* T = Tc + tbase;
  const int zstr = Ux * Uy * 8;
  for (int i = threadIdx.x; i < 2 * NST * plane; i += nthr) planes[i] = 0.f;
  const double f = (mode == 0) ? 0.5 : 1.0;
  float caA = float(f * scal[4]), cdA = float(f * scal[6]), caB = caA, cdB = cdA;
  const int qy = pair & 1, qz = pair >> 1;
  const int qa[3] = {0, qy, qz}, qb[3] = {1, qy, qz};
  const bool va = node_valid(g, o, qa), vb = node_valid(g, o, qb);
  if (ncoef) {
    const int na = o[0] + g.n[0] * ((o[1] + qy) + g.n[1] * (o[2] + qz));
    if (va) { caA = float(f * ncoef[2 * na]); cdA = float(f * ncoef[2 * na + 1]); }
    if (vb) { caB = float(f * ncoef[2 * na + 2]); cdB = float(f * ncoef[2 * na + 3]); }
  }
  const int uy = y0 + yi;
  const bool iny = act && (unsigned)(uy - qy) <= (unsigned)(2 * g.m[1]);
  const bool inA = iny && va && (unsigned)xi <= (unsigned)(2 * g.m[0]);
  const bool inB = iny && vb && (unsigned)(xi - 1) <= (unsigned)(2 * g.m[0]);
  const float cc = mode == 0 ? 0.f : 1.f;
  // wrapped V_eff position of the column
  int wx = (o[0] - g.m[0] + xi) % g.n[0], wy = (o[1] - g.m[1] + uy) % g.n[1], wz = (o[2] - g.m[2]) % g.n[2];
  if (wx < 0) wx += g.n[0];
  if (wy < 0) wy += g.n[1];
  if (wz < 0) wz += g.n[2];
  const float* vcol = v + (act ? wx + g.n[0] * wy : 0);
  const int vz = g.n[0] * g.n[1];
  // copies of two planes: the halo rows of t^j (16 bytes, a thread keeps its column and moves 2 ty rows at a
  // time), and the thread's own t^{j-1}, Y and W (8 bytes each, one offset from five block-uniform bases).
  // Bulk copies of whole rows need a tenth of the instructions and measured 0.96 against 0.74 ms per step of
  // 512 tiles (28^3 windows, 896-byte rows).
  const int ylo = max(0, y0 - NO), nrow = min(Uy, y0 + ty + NO) - ylo;
  const bool rd_p = mode == 1, rd_y = has_y && mode != 2;
  const int cr0 = threadIdx.x < Ux * ty * 4 ? threadIdx.x / (2 * Ux) : nrow;
  const unsigned planes_s = (unsigned)__cvta_generic_to_shared(planes), own_s = (unsigned)__cvta_generic_to_shared(own);
  const unsigned cdst = planes_s + 4 * ((ylo - (y0 - NO) + cr0) * pitch + NO * 8 + 4 * (threadIdx.x - 2 * Ux * cr0));
  const unsigned odst = own_s + 8 * threadIdx.x;
  const int cstep = 2 * ty * Ux * 8, dstep = 4 * 2 * ty * pitch;
  const bool c0 = cr0 < nrow, c1 = cr0 + 2 * ty < nrow;
  const float* csrc = T + ylo * Ux * 8 + 4 * threadIdx.x;   // the thread's first halo piece of the next plane
  const unsigned oo = act ? (uy * Ux + xi) * 8 + 2 * pair : 0;
  const float *Tpt = Tp + tbase + oo, *Yt = Tn + tbase + oo, *W0 = Wt + 3 * tbase + oo;
  const size_t wfld = (size_t)g.Upts * 8;
  int zi = 0;
  auto issue = [&](int stage) {   // the next two planes into a stage
#pragma unroll
    for (int s = 0; s < 2; ++s, ++zi) {
      if (zi < Uz) {
        const unsigned d = cdst + (2 * stage + s) * (4 * plane);
        if (c0) cp16(d, csrc);
        if (c1) cp16(d + dstep, csrc + cstep);
        for (int r = cr0 + 4 * ty, k = 2; r < nrow; r += 2 * ty, ++k) cp16(d + k * dstep, csrc + k * cstep);
        if (act) {
          const unsigned ow = odst + (2 * stage + s) * (kOwn * 4);
          if (rd_p) cp8(ow, Tpt);
          if (rd_y) cp8(ow + 8 * MAXT, Yt);
          cp8(ow + 16 * MAXT, W0);
          cp8(ow + 24 * MAXT, W0 + wfld);
          cp8(ow + 32 * MAXT, W0 + 2 * wfld);
        }
      }
      csrc += zstr;
      Tpt += zstr;
      Yt += zstr;
      W0 += zstr;
    }
    asm volatile("cp.async.commit_group;");
  };
  __syncthreads();   // the planes are cleared
#pragma unroll
  for (int i = 0; i < NST - 1; ++i) issue(i);
  // z window of the column for planes z and z + 1: t(z - NO + k) in r[k]
  constexpr int kW = 2 * NO + 2;
  unsigned zofs = act ? (uy * Ux + xi) * 8 + 2 * pair : 0, nofs = zofs;   // column in the plane to load; to write
  float* Tnt = Tn + tbase;
  float2 r[kW], nx[2];
#pragma unroll
  for (int k = 0; k < kW; ++k) {
    r[k] = make_float2(0.f, 0.f);
    if (k >= NO && k < 2 * NO && k - NO < Uz) r[k] = ld2g(T + zofs + (k - NO) * zstr);
  }
  zofs += NO * zstr;
  int zl = NO;   // plane of the next window load
  auto next = [&]() {
#pragma unroll
    for (int s = 0; s < 2; ++s, ++zl, zofs += zstr) {
      nx[s] = make_float2(0.f, 0.f);
      if (zl < Uz) nx[s] = ld2g(T + zofs);
    }
  };
  next();
  float sb[18];
#pragma unroll
  for (int k = 0; k < 18; ++k) sb[k] = 0.f;
  float vloc[2];
  auto potential = [&]() {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      vloc[s] = vcol[wz * vz];
      if (++wz == g.n[2]) wz = 0;
    }
  };
  potential();
  int scur = 0, snew = NST - 1;
  const int pofs = (yi + NO) * pitch + (xi + NO) * 8 + 2 * pair;
#pragma unroll 1
  for (int z = 0; z < Uz; z += 2) {
    if constexpr (NST == 1) {   // wide windows: no room to copy ahead
      __syncthreads();
      issue(0);
      asm volatile("cp.async.wait_group 0;");
      __syncthreads();
    } else {
      asm volatile("cp.async.wait_group %0;" ::"n"(NST - 2));
      __syncthreads();
      issue(snew);
      snew = snew + 1 == NST ? 0 : snew + 1;
    }
    r[2 * NO] = nx[0];
    r[2 * NO + 1] = nx[1];
    next();
    const float vl[2] = {vloc[0], vloc[1]};
    potential();
    const float* pc = planes + 2 * scur * plane + pofs;
    const float* ow = own + 2 * scur * kOwn + 2 * threadIdx.x;
    scur = scur + 1 == NST ? 0 : scur + 1;
    if (act) {
      float2 y[2], gr[2][3];   // off-diagonal part of H t^j and the gradient, planes z and z + 1
#pragma unroll
      for (int s = 0; s < 2; ++s) y[s] = gr[s][0] = gr[s][1] = gr[s][2] = make_float2(0.f, 0.f);
      auto tap = [&](int s, int a, float wl, float wg, float2 fp, float2 fm) {
        const float2 sum = __fadd2_rn(fp, fm);   // packed: half the issue slots
        y[s].x += wl * sum.x;
        y[s].y += wl * sum.y;
        gr[s][a].x += wg * (fp.x - fm.x);
        gr[s][a].y += wg * (fp.y - fm.y);
      };
#pragma unroll
      for (int pp = 1; pp <= NO; ++pp) {
        const float wl = g.lapf[0][pp], wg = g.grdf[0][pp];
        tap(0, 0, wl, wg, ld2g(pc + pp * 8), ld2g(pc - pp * 8));
        tap(1, 0, wl, wg, ld2g(pc + plane + pp * 8), ld2g(pc + plane - pp * 8));
      }
      const float *yp = pc, *ym = pc;
#pragma unroll
      for (int pp = 1; pp <= NO; ++pp) {
        yp += pitch;
        ym -= pitch;
        const float wl = g.lapf[1][pp], wg = g.grdf[1][pp];
        tap(0, 1, wl, wg, ld2g(yp), ld2g(ym));
        tap(1, 1, wl, wg, ld2g(yp + plane), ld2g(ym + plane));
      }
#pragma unroll
      for (int pp = 1; pp <= NO; ++pp) {
        const float wl = g.lapf[2][pp], wg = g.grdf[2][pp];
        tap(0, 2, wl, wg, r[NO + pp], r[NO - pp]);
        tap(1, 2, wl, wg, r[NO + 1 + pp], r[NO + 1 - pp]);
      }
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        if (z + s >= Uz) break;   // an odd number of planes
#pragma unroll
        for (int b = 0; b < 3; ++b) {   // W is zero outside each node's window
          const float2 wb = ld2g(ow + s * kOwn + (4 + 2 * b) * MAXT);
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            sb[3 * a + b] += gr[s][a].x * wb.x;
            sb[9 + 3 * a + b] += gr[s][a].y * wb.y;
          }
        }
        if (mode != 2) {
          if (rd_y) {
            const float2 yn = ld2g(ow + s * kOwn + 2 * MAXT);
            y[s].x += yn.x;
            y[s].y += yn.y;
          }
          const float2 tp = rd_p ? ld2g(ow + s * kOwn) : make_float2(0.f, 0.f), tc = r[NO + s];
          const bool inz = (unsigned)(z + s - qz) <= (unsigned)(2 * g.m[2]);
          float2 tn = make_float2(0.f, 0.f);
          if (inA && inz) tn.x = caA * y[s].x + (cdA + caA * vl[s]) * tc.x - cc * tp.x;
          if (inB && inz) tn.y = caB * y[s].y + (cdB + caB * vl[s]) * tc.y - cc * tp.y;
          *reinterpret_cast<float2*>(Tnt + nofs + s * zstr) = tn;
        }
      }
    }
    nofs += 2 * zstr;
#pragma unroll
    for (int k = 0; k < 2 * NO; ++k) r[k] = r[k + 2];
  }
  // S sums: over the warp's eight points per node pair, then over warps in FP64, fixed order
  __syncthreads();
  float* red = st_smem;   // [warps][8 nodes][9]
#pragma unroll
  for (int k = 0; k < 18; ++k) {
    float sv = sb[k];
    sv += __shfl_xor_sync(0xffffffffu, sv, 4);
    sv += __shfl_xor_sync(0xffffffffu, sv, 8);
    sv += __shfl_xor_sync(0xffffffffu, sv, 16);
    if ((threadIdx.x & 31) < 4) red[((threadIdx.x >> 5) * 8 + 2 * pair + k / 9) * 9 + k % 9] = sv;
  }
  __syncthreads();
  for (int k2 = threadIdx.x; k2 < 72; k2 += nthr) {
    double sv = 0.0;
    for (int wv = 0; wv < (nthr >> 5); ++wv) sv += double(red[wv * 72 + k2]);
    Spart[((size_t)tl * gridDim.x + chunk) * 72 + k2] = sv;
  }
}

// ------------------------------------------------------------------------------ host
// Rows per stencil block: at most 448 threads (the rows evenly spread over the blocks; 127 registers and 142 KB at
// 28 points, one block per SM); windows wider than 112 points take one row and up to 544 threads.
int stencil_rows(const Geo& g) {
  const int most = std::max(1, 448 / (4 * g.U[0]));
  const int chunks = (g.U[1] + most - 1) / most;
  return (g.U[1] + chunks - 1) / chunks;
}
int stencil_chunks(const Geo& g) {
  const int ty = stencil_rows(g);
  return (g.U[1] + ty - 1) / ty;
}

template <int NO, int MAXT, int MINB, int NST>
static int stencil_launch(sq_handle* h, const Wave& w, const float* Tc, const float* Tp, float* Tn, int has_y, int mode) {
  const Geo& g = h->geo;
  const int ty = stencil_rows(g), nthr = (4 * g.U[0] * ty + 31) / 32 * 32;
  const size_t smem = sizeof(float) * 2 * NST * (size_t(st_plane_floats(g.U[0], ty, NO)) + 5 * 2 * size_t(MAXT));
  const double* ncoef = (h->bounds_mode == SQ_BOUNDS_PER_NODE) ? h->d.ncoef : nullptr;
  // the attribute belongs to the function: every caller sets the same value
  SQ_CUDA_TRY(h, cudaFuncSetAttribute(k_stencil<NO, MAXT, MINB, NST>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  k_stencil<NO, MAXT, MINB, NST><<<dim3(stencil_chunks(g), w.ntiles), nthr, smem, h->stream>>>(
      g, w, Tc, Tp, Tn, has_y, (const float*)h->wb.W, h->d.v32, h->d.scal, mode, ncoef, ty, h->wb.Spart);
  SQ_LAUNCH_CHECK(h);
  return SQ_OK;
}

template <int NO>
static int stencil_no(sq_handle* h, const Wave& w, const float* Tc, const float* Tp, float* Tn, int has_y, int mode) {
  if (h->geo.U[0] <= 84) return stencil_launch<NO, 448, 1, 2>(h, w, Tc, Tp, Tn, has_y, mode);
  return stencil_launch<NO, 544, 1, 1>(h, w, Tc, Tp, Tn, has_y, mode);
}

static bool nl_any(const sq_handle* h) { return h->geo.n_atoms > 0 && h->table_len > 0; }
static dim3 nl_dim(const NlGrid& n) { return dim3(n.nb[0], n.nb[1], 8 * n.nz); }

// Do the wave's tables fit their buffers (ensure_nl_buffers) and its bricks a grid?
bool nl_fits(const sq_handle* h, size_t wi) {
  if (!nl_any(h)) return true;
  if (wi >= h->wave_nl.size()) return false;
  const NlNeed& need = h->wave_nl[wi];
  const NlGrid n = nl_grid(h->geo, h->waves[wi]);
  return size_t(need.x_rows) <= h->x_rows_cap && size_t(need.imgs) <= h->img_cap && size_t(need.tile_imgs) <= h->idx_cap &&
         size_t(need.tile_rows) * 8 <= h->part_floats && n.nb[1] < 65536 && 8 * n.nb[2] < 65536;
}

// rows and images the tables of wave wi need, added to cnt[0], cnt[1] (after its lists)
int count_nl_tables(sq_handle* h, size_t wi, int* cnt) {
  if (!nl_any(h)) return SQ_OK;
  const Wave& w = h->waves[wi];
  const NlGrid n = nl_grid(h->geo, w);
  if (n.nb[1] >= 65536 || 8 * n.nb[2] >= 65536) return SQ_OK;   // nl_fits is false
  k_nl_table<<<nl_dim(n), 128, 0, h->stream>>>(h->geo, w, n, h->d.chi32s, h->wb.brick_rec, h->wb.brick_n, 0, 0, cnt,
                                               nullptr, nullptr, nullptr, nullptr);
  SQ_LAUNCH_CHECK(h);
  return SQ_OK;
}

// Buffers for the largest needs of the layout, a sixteenth larger than needed so that moving atoms seldom outgrow
// them; they never shrink. Part holds the partial projections of the largest wave, at most kNlPartFloats (the sweep
// then takes the tiles in chunks). What cannot be allocated is left out: nl_fits sends those waves to k_step.
int ensure_nl_buffers(sq_handle* h) {
  if (!nl_any(h)) return SQ_OK;
  NlNeed top;
  size_t part = 0;
  for (size_t wi = 0; wi < h->wave_nl.size(); ++wi) {
    const NlNeed& n = h->wave_nl[wi];
    top.x_rows = std::max(top.x_rows, n.x_rows);
    top.imgs = std::max(top.imgs, n.imgs);
    top.tile_imgs = std::max(top.tile_imgs, n.tile_imgs);
    const size_t tile = size_t(n.tile_rows) * 8;
    part = std::max(part, std::max(tile, std::min(kNlPartFloats, tile * h->waves[wi].ntiles)));
  }
  auto grow = [&](void** p, size_t* cap, size_t need, size_t unit, size_t most) -> int {
    if (need <= *cap && *p) return SQ_OK;
    const size_t want = std::max(need, std::min(most, need + need / 16 + 64));
    h->nl_epoch++;   // captured graphs hold the old pointer
    SQ_CUDA_TRY(h, cudaStreamSynchronize(h->stream));
    dev_free(h, *p, *cap * unit);
    *p = nullptr;
    *cap = 0;
    if (dev_alloc(h, p, want * unit) != SQ_OK) {   // no error: the other step runs
      h->err.clear();
      return SQ_OK;
    }
    *cap = want;
    return SQ_OK;
  };
  const size_t any = SIZE_MAX / 2;
  int rc = grow((void**)&h->wb.nl_X, &h->x_rows_cap, top.x_rows, 64 * sizeof(float2), any);
  if (rc == SQ_OK) rc = grow((void**)&h->wb.nl_img, &h->img_cap, top.imgs, sizeof(int), any);
  if (rc == SQ_OK) rc = grow((void**)&h->wb.proj_idx, &h->idx_cap, top.tile_imgs, sizeof(int) * size_t(h->wave_cap), any);
  if (rc == SQ_OK) rc = grow((void**)&h->wb.Part, &h->part_floats, part, sizeof(float), std::max(part, kNlPartFloats));
  return rc;
}

// the wave's brick tables and the image -> brick index, after its lists
int build_nl_tables(sq_handle* h, size_t wi) {
  if (!nl_any(h)) return SQ_OK;
  const Wave& w = h->waves[wi];
  const NlGrid n = nl_grid(h->geo, w);
  SQ_CUDA_TRY(h, cudaMemsetAsync(h->wb.nl_cnt, 0, 2 * sizeof(int), h->stream));
  k_nl_table<<<nl_dim(n), 128, 0, h->stream>>>(h->geo, w, n, h->d.chi32s, h->wb.brick_rec, h->wb.brick_n,
                                               (long long)h->x_rows_cap, (long long)h->img_cap, h->wb.nl_cnt, h->wb.nl_head,
                                               h->wb.nl_img, h->wb.nl_X, h->d.status);
  SQ_LAUNCH_CHECK(h);
  k_nl_index<<<w.ntiles, 256, 0, h->stream>>>(h->geo, w, n, h->d.atoms, h->wb.entries, h->wb.n_entries, h->wb.brick_list,
                                              h->wb.brick_n, h->wb.nl_head, h->wb.nl_img, h->wave_nl[wi].tile_rows,
                                              int(h->idx_cap), h->wb.proj_off, h->wb.proj_start, h->wb.proj_idx, h->d.status);
  SQ_LAUNCH_CHECK(h);
  return SQ_OK;
}

// Projections of t^{j+1} in chunks of tiles whose partial sums fit the Part buffer
int launch_project_mixed(sq_handle* h, size_t wi, const float* T) {
  if (!nl_any(h)) return SQ_OK;
  const Geo& g = h->geo;
  const Wave& w = h->waves[wi];
  const int rows = h->wave_nl[wi].tile_rows;
  const size_t per_tile = size_t(std::max(1, rows)) * 8;
  SQ_CUDA_TRY(h, cudaFuncSetAttribute(k_nl_project, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kPrSmem)));
  const int most = int(std::max<size_t>(1, std::min<size_t>(size_t(w.ntiles), h->part_floats / per_tile)));
  const int nchunk = (w.ntiles + most - 1) / most, ct = (w.ntiles + nchunk - 1) / nchunk;   // equal chunks
  for (int c0 = 0; c0 < w.ntiles; c0 += ct) {
    const int cn = std::min(ct, w.ntiles - c0);
    const NlGrid n = nl_grid(g, w, c0, cn);
    k_nl_project<<<nl_dim(n), kPrThreads, kPrSmem, h->stream>>>(g, w, n, c0, cn, T, h->wb.nl_head, h->wb.nl_img, h->wb.nl_X,
                                                                NlPart{h->wb.proj_off, rows}, h->wb.Part);
    SQ_LAUNCH_CHECK(h);
    k_nl_reduce<<<dim3(cn, 8), 128, 0, h->stream>>>(g, c0, h->wb.entries, h->wb.n_entries, h->d.atoms, h->d.gdvp,
                                           h->wb.proj_start, h->wb.proj_idx, int(h->idx_cap), rows, h->wb.Part,
                                           (float*)h->wb.Pg[1], nl_plane(h), (float2*)h->wb.Pg[0]);
    SQ_LAUNCH_CHECK(h);
  }
  return SQ_OK;
}

int launch_step_mixed(sq_handle* h, size_t wi, const float* Tc, const float* Tp, float* Tn, int mode) {
  const Geo& g = h->geo;
  const Wave& w = h->waves[wi];
  const bool nl = nl_any(h);
  if (nl && mode != 2) {
    const NlGrid n = nl_grid(g, w);
    SQ_CUDA_TRY(h, cudaFuncSetAttribute(k_nl_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kApSmem)));
    k_nl_apply<<<nl_dim(n), kNlThreads, kApSmem, h->stream>>>(g, w, n, h->max_nch, (const float*)h->wb.Pg[1],
                                                              nl_plane(h), h->wb.nl_head, h->wb.nl_img, h->wb.nl_X,
                                                              h->wb.brick_rec, Tn);
    SQ_LAUNCH_CHECK(h);
  }
  h->step_variant[0]++;
  switch (g.n_o) {
    case 1: return stencil_no<1>(h, w, Tc, Tp, Tn, nl, mode);
    case 2: return stencil_no<2>(h, w, Tc, Tp, Tn, nl, mode);
    case 3: return stencil_no<3>(h, w, Tc, Tp, Tn, nl, mode);
    case 4: return stencil_no<4>(h, w, Tc, Tp, Tn, nl, mode);
    case 5: return stencil_no<5>(h, w, Tc, Tp, Tn, nl, mode);
    default: return stencil_no<6>(h, w, Tc, Tp, Tn, nl, mode);
  }
}

}  // namespace sq
