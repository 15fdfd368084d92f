// mhd_gran.cu -- the granulation driver (Sect. 2.3, Eqs. 1-4) on the GPU.
//
// State: one slot per pixel (occupancy, t0, T, v_max, t_max), so granules
// need no list, compaction or host bookkeeping.
//
// Update (the population at time t):
//   1. seed:    a pixel within r_inner of a live centre is out, the rest
//               undecided; a granule with t - t0 - t_max > t_max (Eq. 2 is
//               back at v_min) no longer counts as live
//   2. rounds:  join: an undecided pixel with no undecided pixel of smaller
//               (key, index) within r_inner, and no member there, becomes a
//               member; exclude: an undecided pixel with a member within
//               r_inner is out.  Repeated until nothing is undecided, this
//               gives exactly the set the sequential visit in (key, index)
//               order accepts (the first undecided pixel in that order joins
//               every round, so the rounds end).
//   3. birth:   expired granules are cleared, members become granules with
//               the draws at their pixel.
// Velocity at time t:
//   4. amp:     per pixel, Eq. 2 of its granule (0 where none)
//   5. render:  v_gran(p) = sum over lane offsets o of amp(p - o) w(o), with
//               w(o) = profile(|o|) o / |o| tabulated on the host
//   6. FFT:     the filtered rotational part (Eq. 3), packed plane v_x + i v_y;
//               its last kernel adds it to v_gran (v_vor = v_gran + f_rot
//               v_rot') and sums |v_vor|^2 per block
//   7. total, scale: block sums of |v|^2 of both fields totalled in a fixed
//               order; v_vor scaled to the rms of v_gran (Eq. 4) into the
//               caller's array.
//
// What bounds the pixel kernels.  One pixel in ten carries a granule, but a
// warp that tests pixel by pixel does FP64 work (2 operations per clock and SM)
// for every offset at which any of its 32 lanes has one, which is nearly all
// of them.  So the neighbourhood kernels work on tiles of 32 x 8 pixels whose
// occupancy, halo included, is a 64-bit mask per row (one ballot or two per
// row): a disk test is an AND per row, and the render walks each lane's own
// hits, so a warp takes as many steps as its busiest lane has granules in
// reach (about 9) instead of one per offset (68 at 0.23 Mm pixels); amplitudes
// and births are computed on lists of the occupied pixels of a block.  Disks
// wider than 16 pixels, or planes narrower than a tile, take the plain kernels.
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <vector>

#include "mhd.h"
#include "mhd_internal.h"

namespace mhd {
namespace {

constexpr int GT = 256;             // threads per block of the pixel kernels
constexpr int GMAX_PX = 64;         // largest disk radius in pixels
constexpr int UNDECIDED = 0, MEMBER = 1, OUT = 2;

struct GranDev {
  int nx, ny;
  int* occ;
  double *t0, *life, *vmax, *tmax;  // [ny][nx] each
  int* mis;
  double* amp;
  double* vg;  // [2][ny][nx]
  double* vr;  // [2][ny][nx]: the rotational part, then v_vor
  const int2* off_in;
  int n_in;
  const int2* off_l;
  const double2* w_l;
  int n_l;
  double* part;  // [2][nblk] block sums
  double* tot;   // [2]: scale, spare
  int* cnt;      // [BATCH] undecided pixels left after each round of a batch
};

// rounds launched between two reads of the undecided counts (the rounds after
// the last needed one return at once)
constexpr int BATCH = 4;

// disk row by row: offsets (o_x, o_y) of the disk are |o_x| <= lim[|o_y|]
constexpr int MAXR = 16;
struct Disk {
  int rx, ry;                 // largest |o_x|, |o_y|
  signed char lim[MAXR + 1];  // -1: no offset in that row
};

__device__ __forceinline__ int wrap(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// a granule whose amplitude has fallen below v_min after its peak
__device__ __forceinline__ bool expired(const GranDev& g, int p, double t) {
  const double tm = g.tmax[p];
  return t - g.t0[p] - tm > tm;
}

__global__ void __launch_bounds__(GT) seed_kernel(GranDev g, double t) {
  const int p = blockIdx.x * GT + threadIdx.x;
  if (p >= g.nx * g.ny) return;
  const int y = p / g.nx, x = p - y * g.nx;
  bool blocked = g.occ[p] != 0 && !expired(g, p, t);
  for (int n = 0; n < g.n_in && !blocked; ++n) {
    const int2 o = __ldg(g.off_in + n);
    const int q = wrap(y + o.y, g.ny) * g.nx + wrap(x + o.x, g.nx);
    blocked = g.occ[q] != 0 && !expired(g, q, t);
  }
  g.mis[p] = blocked ? OUT : UNDECIDED;
}

// ---- tiles of 32 x 8 pixels with row masks (nx, ny powers of two) ----------
constexpr int TW = 32, TH = 8;
constexpr int TROWS = TH + 2 * MAXR;

// masks[r]: bit c set where flag(pixel) holds at halo column x0 - rx + c of
// halo row y0 - ry + r (periodic)
template <typename F>
__device__ __forceinline__ void row_masks(const GranDev& g, int x0, int y0, int rx, int ry,
                                          unsigned long long* masks, F flag) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int r = w; r < TH + 2 * ry; r += GT / 32) {
    const int row = ((y0 - ry + r) & (g.ny - 1)) * g.nx;
    const bool f0 = flag(row + ((x0 - rx + lane) & (g.nx - 1)));
    const bool f1 = lane < 2 * rx && flag(row + ((x0 - rx + 32 + lane) & (g.nx - 1)));
    const unsigned lo = __ballot_sync(0xffffffffu, f0), hi = __ballot_sync(0xffffffffu, f1);
    if (lane == 0) masks[r] = (unsigned long long)hi << 32 | lo;
  }
}
// the bits of a row mask within the disk's row o_y of the pixel at tile column
// tx: bit lim + o_x of the result
__device__ __forceinline__ unsigned long long disk_bits(unsigned long long m, int tx, int rx, int lim) {
  return lim < 0 ? 0ull : (m >> (tx + rx - lim)) & ((1ull << (2 * lim + 1)) - 1ull);
}
__device__ __forceinline__ bool disk_any(const unsigned long long* masks, const Disk& d, int tx, int ty) {
  unsigned long long any = 0;
  for (int oy = -d.ry; oy <= d.ry; ++oy)
    any |= disk_bits(masks[ty + d.ry + oy], tx, d.rx, d.lim[oy < 0 ? -oy : oy]);
  return any != 0;
}

__global__ void __launch_bounds__(GT) seed_tile_kernel(GranDev g, Disk d, double t) {
  __shared__ unsigned long long live[TROWS];
  const int x0 = blockIdx.x * TW, y0 = blockIdx.y * TH, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  row_masks(g, x0, y0, d.rx, d.ry, live, [&](int p) { return g.occ[p] != 0 && !expired(g, p, t); });
  __syncthreads();
  g.mis[(y0 + ty) * g.nx + x0 + tx] = disk_any(live, d, tx, ty) ? OUT : UNDECIDED;
}

// As join_kernel below: a snapshot of the neighbours' states, taken while
// other tiles may be joining, gives the same decision either way.
__global__ void __launch_bounds__(GT) join_tile_kernel(GranDev g, Disk d, const unsigned* __restrict__ keys,
                                                       int round) {
  if (round > 0 && g.cnt[round - 1] == 0) return;
  const int x0 = blockIdx.x * TW, y0 = blockIdx.y * TH, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int p = (y0 + ty) * g.nx + x0 + tx;
  const bool open = g.mis[p] == UNDECIDED;
  if (!__syncthreads_or(open)) return;
  __shared__ unsigned long long mem[TROWS], und[TROWS];
  const volatile int* mis = g.mis;
  row_masks(g, x0, y0, d.rx, d.ry, mem, [&](int q) { return mis[q] == MEMBER; });
  // every neighbour that is not out: one that joins while this tile reads is
  // still compared by its key, which precedes p's
  row_masks(g, x0, y0, d.rx, d.ry, und, [&](int q) { return mis[q] != OUT; });
  __syncthreads();
  if (!open || disk_any(mem, d, tx, ty)) return;
  const unsigned kp = keys[p];
  for (int oy = -d.ry; oy <= d.ry; ++oy) {
    const int lim = d.lim[oy < 0 ? -oy : oy];
    unsigned long long b = disk_bits(und[ty + d.ry + oy], tx, d.rx, lim);
    if (oy == 0) b &= ~(1ull << lim);  // the pixel itself
    const int row = ((y0 + ty + oy) & (g.ny - 1)) * g.nx;
    while (b) {
      const int c = __ffsll((long long)b) - 1;
      b &= b - 1;
      const int q = row + ((x0 + tx + c - lim) & (g.nx - 1));
      const unsigned kq = keys[q];
      if (kq < kp || (kq == kp && q < p)) return;
    }
  }
  g.mis[p] = MEMBER;
}

__global__ void __launch_bounds__(GT) exclude_tile_kernel(GranDev g, Disk d, int round) {
  if (round > 0 && g.cnt[round - 1] == 0) return;
  const int x0 = blockIdx.x * TW, y0 = blockIdx.y * TH, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int p = (y0 + ty) * g.nx + x0 + tx;
  const bool open = g.mis[p] == UNDECIDED;
  if (!__syncthreads_or(open)) return;
  __shared__ unsigned long long mem[TROWS];
  row_masks(g, x0, y0, d.rx, d.ry, mem, [&](int q) { return g.mis[q] == MEMBER; });
  __syncthreads();
  const bool hit = open && disk_any(mem, d, tx, ty);
  if (hit) g.mis[p] = OUT;
  const int c = __syncthreads_count(open && !hit);
  if (threadIdx.x == 0 && c) atomicAdd(g.cnt + round, c);
}

// Reads of neighbours race with their writes in the same launch; either
// value gives the same decision (a neighbour that joins now precedes p, so
// p does not join whether it reads UNDECIDED or MEMBER).
__global__ void __launch_bounds__(GT) join_kernel(GranDev g, const unsigned* __restrict__ keys, int round) {
  if (round > 0 && g.cnt[round - 1] == 0) return;
  const int p = blockIdx.x * GT + threadIdx.x;
  if (p >= g.nx * g.ny) return;
  if (g.mis[p] != UNDECIDED) return;
  const int y = p / g.nx, x = p - y * g.nx;
  const unsigned kp = keys[p];
  for (int n = 0; n < g.n_in; ++n) {
    const int2 o = __ldg(g.off_in + n);
    const int q = wrap(y + o.y, g.ny) * g.nx + wrap(x + o.x, g.nx);
    const int s = ((volatile int*)g.mis)[q];
    if (s == MEMBER) return;
    if (s == UNDECIDED) {
      const unsigned kq = keys[q];
      if (kq < kp || (kq == kp && q < p)) return;
    }
  }
  g.mis[p] = MEMBER;
}

__global__ void __launch_bounds__(GT) exclude_kernel(GranDev g, int round) {
  if (round > 0 && g.cnt[round - 1] == 0) return;
  const int p = blockIdx.x * GT + threadIdx.x;
  int undecided = 0;
  if (p < g.nx * g.ny && g.mis[p] == UNDECIDED) {
    const int y = p / g.nx, x = p - y * g.nx;
    bool hit = false;
    for (int n = 0; n < g.n_in && !hit; ++n) {
      const int2 o = __ldg(g.off_in + n);
      hit = g.mis[wrap(y + o.y, g.ny) * g.nx + wrap(x + o.x, g.nx)] == MEMBER;
    }
    if (hit) g.mis[p] = OUT;
    else undecided = 1;
  }
  const int c = __syncthreads_count(undecided);
  if (threadIdx.x == 0 && c) atomicAdd(g.cnt + round, c);
}

// The occupied (or chosen) pixels of a block's LP * GT pixels as a list in
// shared memory, so that the FP64 work on them runs in full warps; returns
// their number.  The order within the list does not matter.
constexpr int LP = 8;
template <typename F>
__device__ __forceinline__ int block_list(int N, int* list, int* count, F take) {
  if (threadIdx.x == 0) *count = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int u = 0; u < LP; ++u) {
    const int p = (blockIdx.x * LP + u) * GT + threadIdx.x;
    const bool in = p < N && take(p);
    const unsigned m = __ballot_sync(0xffffffffu, in);
    int base = 0;
    if (lane == 0 && m) base = atomicAdd(count, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (in) list[base + __popc(m & ((1u << lane) - 1))] = p;
  }
  __syncthreads();
  return *count;
}

__global__ void __launch_bounds__(GT) birth_kernel(GranDev g, mhd_gran_params gp, double t,
                                                   const double* __restrict__ c_life,
                                                   const double* __restrict__ c_amp) {
  __shared__ int list[LP * GT], count;
  const int n = block_list(g.nx * g.ny, list, &count, [&](int p) {
    if (g.occ[p] && expired(g, p, t)) {
      g.occ[p] = 0;
      g.t0[p] = g.life[p] = g.vmax[p] = g.tmax[p] = 0.0;
    }
    return g.mis[p] == MEMBER;
  });
  for (int i = threadIdx.x; i < n; i += GT) {
    const int p = list[i];
    const double cl = fmin(1.0, fmax(-1.0, c_life[p]));
    const double ca = fmin(1.0, fmax(-1.0, c_amp[p]));
    const double T = gp.lifetime * (1.0 + gp.lifetime_spread * cl);
    const double vm = gp.v0 * (1.0 + gp.amp_spread * ca);
    g.occ[p] = 1;
    g.t0[p] = t;
    g.life[p] = T;
    g.vmax[p] = vm;
    g.tmax[p] = T * sqrt(fabs(log(gp.vmin_frac * gp.v0 / vm)));  // Eq. 1
  }
}

__global__ void __launch_bounds__(GT) amp_kernel(GranDev g, double t) {
  __shared__ int list[LP * GT], count;
  const int n = block_list(g.nx * g.ny, list, &count, [&](int p) {
    const bool in = g.occ[p] != 0;
    if (!in) g.amp[p] = 0.0;
    return in;
  });
  for (int i = threadIdx.x; i < n; i += GT) {
    const int p = list[i];
    const double s = (t - g.t0[p] - g.tmax[p]) / g.life[p];
    g.amp[p] = g.vmax[p] * exp(-s * s);  // Eq. 2
  }
}

__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < GT / 32; ++i) s += sh[i];
  return s;
}

// v_gran at pixel p: the granule centred at p - o contributes amp w(o).
// Block sums of |v_gran|^2 into part[0][block].
__global__ void __launch_bounds__(GT) render_kernel(GranDev g) {
  __shared__ double sh[GT / 32];
  const int N = g.nx * g.ny;
  const int p = blockIdx.x * GT + threadIdx.x;
  double e = 0.0;
  if (p < N) {
    const int y = p / g.nx, x = p - y * g.nx;
    double vx = 0.0, vy = 0.0;
    for (int n = 0; n < g.n_l; ++n) {
      const int2 o = __ldg(g.off_l + n);
      const double a = __ldg(g.amp + wrap(y - o.y, g.ny) * g.nx + wrap(x - o.x, g.nx));
      if (a != 0.0) {
        const double2 w = __ldg(g.w_l + n);
        vx = fma(a, w.x, vx);
        vy = fma(a, w.y, vy);
      }
    }
    g.vg[p] = vx;
    g.vg[N + p] = vy;
    e = vx * vx + vy * vy;
  }
  const double s = block_sum(e, sh);
  if (threadIdx.x == 0) g.part[blockIdx.x] = s;
}

// The same sum over a tile: each lane walks the granules within its own disk,
// in the order of the offset list, so the result equals render_kernel's.
__global__ void __launch_bounds__(GT) render_tile_kernel(GranDev g, Disk d) {
  extern __shared__ double2 dyn[];
  __shared__ unsigned long long occ[TROWS];
  __shared__ double sh[GT / 32];
  const int wr = 2 * d.rx + 1, ww = TW + 2 * d.rx, hh = TH + 2 * d.ry;
  double2* wt = dyn;                                      // [2 ry + 1][2 rx + 1] weights
  double* am = reinterpret_cast<double*>(dyn + wr * (2 * d.ry + 1));  // [hh][ww] amplitudes
  const int x0 = blockIdx.x * TW, y0 = blockIdx.y * TH, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int n = threadIdx.x; n < g.n_l; n += GT) {
    const int2 o = __ldg(g.off_l + n);
    wt[(o.y + d.ry) * wr + o.x + d.rx] = __ldg(g.w_l + n);
  }
  for (int r = ty; r < hh; r += GT / 32) {
    const int row = ((y0 - d.ry + r) & (g.ny - 1)) * g.nx;
    const double a0 = __ldg(g.amp + row + ((x0 - d.rx + tx) & (g.nx - 1)));
    const double a1 = tx < 2 * d.rx ? __ldg(g.amp + row + ((x0 - d.rx + 32 + tx) & (g.nx - 1))) : 0.0;
    am[r * ww + tx] = a0;
    if (tx < 2 * d.rx) am[r * ww + 32 + tx] = a1;
    const unsigned lo = __ballot_sync(0xffffffffu, a0 != 0.0), hi = __ballot_sync(0xffffffffu, a1 != 0.0);
    if (tx == 0) occ[r] = (unsigned long long)hi << 32 | lo;
  }
  __syncthreads();
  double vx = 0.0, vy = 0.0;
  int oy = -d.ry - 1, lim = 0;
  unsigned long long bits = 0;
  for (;;) {
    // next granule of this lane: rows by ascending o_y, and within a row the
    // columns by descending x (ascending o_x; the centre sits at p - o)
    while (!bits && oy < d.ry) {
      ++oy;
      lim = d.lim[oy < 0 ? -oy : oy];
      bits = disk_bits(occ[ty + d.ry - oy], tx, d.rx, lim);
      if (oy == 0) bits &= ~(1ull << lim);
    }
    if (!__any_sync(0xffffffffu, bits != 0)) break;
    if (bits) {
      const int c = 63 - __clzll((long long)bits);
      bits &= ~(1ull << c);
      const double a = am[(ty + d.ry - oy) * ww + tx + d.rx - lim + c];
      const double2 w = wt[(oy + d.ry) * wr + d.rx + lim - c];
      vx = fma(a, w.x, vx);
      vy = fma(a, w.y, vy);
    }
  }
  const int N = g.nx * g.ny, p = (y0 + ty) * g.nx + x0 + tx;
  g.vg[p] = vx;
  g.vg[N + p] = vy;
  const double s = block_sum(vx * vx + vy * vy, sh);
  if (threadIdx.x == 0) g.part[blockIdx.y * gridDim.x + blockIdx.x] = s;
}

// the filter of Eq. 3 on a quarter of the spectrum (it is even in k_x and k_y
// but for the sign of sin 2 theta): w = exp(-(2 |k| / k_N)^4) / 2 and w cos, w
// sin of twice the angle of k; zero on the mean and the Nyquist modes
__global__ void __launch_bounds__(GT) filter_kernel(FFTPlan fp, double* __restrict__ tab) {
  const int hx = fp.nx / 2 + 1, hy = fp.ny / 2 + 1;
  const int q = blockIdx.x * GT + threadIdx.x;
  if (q >= hx * hy) return;
  const int a = q / hy, b = q - a * hy;
  const double kx = fabs(fp.ktx[a]), ky = fabs(fp.kty[b]);
  const double k2 = kx * kx + ky * ky;
  double w = 0.0, wc = 0.0, ws = 0.0;
  if (k2 > 0.0 && 2 * a != fp.nx && 2 * b != fp.ny) {
    const double ax = kx / fp.knx, ay = ky / fp.kny;
    const double q4 = 4.0 * (ax * ax + ay * ay);
    w = 0.5 * exp(-q4 * q4);
    wc = w * ((kx * kx - ky * ky) / k2);
    ws = w * (2.0 * kx * ky / k2);
  }
  tab[3 * (size_t)q] = w;
  tab[3 * (size_t)q + 1] = wc;
  tab[3 * (size_t)q + 2] = ws;
}

// one block: totals of both block-sum rows in a fixed order, the Eq. 4 scale
__global__ void __launch_bounds__(GT) total_kernel(GranDev g, int nblk, int nvor) {
  __shared__ double sh[GT / 32];
  double sv = 0.0, sw = 0.0;
  for (int i = threadIdx.x; i < nblk; i += GT) sv += g.part[i];
  for (int i = threadIdx.x; i < nvor; i += GT) sw += g.part[nblk + i];
  const double tv = block_sum(sv, sh);
  __syncthreads();
  const double tw = block_sum(sw, sh);
  if (threadIdx.x == 0) g.tot[0] = tw > 0.0 ? sqrt(tv / tw) : 0.0;
}

template <typename R>
__global__ void __launch_bounds__(GT) scale_kernel(GranDev g, R* __restrict__ v) {
  const int N = g.nx * g.ny;
  const int p = blockIdx.x * GT + threadIdx.x;
  if (p >= N) return;
  const double s = g.tot[0];
  v[p] = (R)(g.vr[p] * s);
  v[N + p] = (R)(g.vr[N + p] * s);
}

// ---- host side ---------------------------------------------------------------

bool pow2(int n) { return n > 0 && (n & (n - 1)) == 0; }
int lg2(int n) {
  int l = 0;
  while ((1 << l) < n) ++l;
  return l;
}

// the same disk by rows (lim is symmetric and falls with |o_y|); false if it is
// wider than the tile kernels take
bool disk_rows(double r, double dx, double dy, Disk* d) {
  d->rx = d->ry = 0;
  for (int q = 0; q <= MAXR; ++q) d->lim[q] = -1;
  const int mx = (int)std::ceil(r / dx), my = (int)std::ceil(r / dy);
  for (int oy = 0; oy <= my; ++oy)
    for (int ox = 0; ox <= mx; ++ox) {
      const double ex = ox * dx, ey = oy * dy;
      if (!(ex * ex + ey * ey < r * r)) continue;
      if (ox > MAXR || oy > MAXR) return false;
      d->lim[oy] = (signed char)ox;
      if (ox > d->rx) d->rx = ox;
      if (oy > d->ry) d->ry = oy;
    }
  return true;
}

// disk offsets (o != 0) with |o| < r, |o| = sqrt((o_x dx)^2 + (o_y dy)^2)
std::vector<int2> disk(double r, double dx, double dy) {
  std::vector<int2> out;
  const int mx = (int)std::ceil(r / dx), my = (int)std::ceil(r / dy);
  for (int oy = -my; oy <= my; ++oy)
    for (int ox = -mx; ox <= mx; ++ox) {
      if (ox == 0 && oy == 0) continue;
      const double ex = ox * dx, ey = oy * dy;
      if (ex * ex + ey * ey < r * r) out.push_back(make_int2(ox, oy));
    }
  return out;
}

const char* check(int nx, int ny, double dx, double dy, const mhd_gran_params* gp) {
  if (!gp) return "gran params are NULL";
  if (!pow2(nx) || !pow2(ny) || nx < 8 || ny < 8 || nx > 1024 || ny > 1024)
    return "nx, ny must be powers of two in [8, 1024]";
  if (!(dx > 0.0) || !(dy > 0.0)) return "dx, dy must be positive";
  if (!(gp->r_inner > 0.0) || !(gp->r_granule > 0.0) || !(gp->r_lane > gp->r_granule))
    return "need 0 < r_inner and 0 < r_granule < r_lane";
  const double rmax = gp->r_inner > gp->r_lane ? gp->r_inner : gp->r_lane;
  if (!(rmax < 0.5 * nx * dx) || !(rmax < 0.5 * ny * dy)) return "r_inner and r_lane must be below half the plane";
  if (rmax / dx > GMAX_PX || rmax / dy > GMAX_PX) return "r_inner and r_lane must span at most 64 pixels";
  if (!(gp->v0 > 0.0) || !(gp->lifetime > 0.0)) return "v0 and lifetime must be positive";
  if (!(gp->lifetime_spread >= 0.0 && gp->lifetime_spread < 1.0) ||
      !(gp->amp_spread >= 0.0 && gp->amp_spread < 1.0))
    return "spreads must lie in [0, 1)";
  if (!(gp->vmin_frac > 0.0 && gp->vmin_frac < 1.0 - gp->amp_spread))
    return "vmin_frac must lie in (0, 1 - amp_spread)";
  if (!std::isfinite(gp->f_rot)) return "f_rot must be finite";
  return nullptr;
}

struct Carve {
  size_t off = 0;
  size_t take(size_t bytes) {
    const size_t o = off;
    off += (bytes + 255) / 256 * 256;
    return o;
  }
};

struct Layout2 {
  size_t occ, par, mis, amp, vg, vr, keys, cl, ca, twx, twy, ktx, kty, P, Q, off_in, off_l, w_l, part, tot, cnt, filt;
  size_t total;
  int n_in, n_l, nblk;
};

Layout2 carve(int nx, int ny, double dx, double dy, const mhd_gran_params* gp) {
  Layout2 o;
  const size_t N = (size_t)nx * ny;
  o.n_in = (int)disk(gp->r_inner, dx, dy).size();
  o.n_l = (int)disk(gp->r_lane, dx, dy).size();
  o.nblk = (int)((N + GT - 1) / GT);
  Carve c;
  o.occ = c.take(N * 4);
  o.par = c.take(4 * N * 8);
  o.mis = c.take(N * 4);
  o.amp = c.take(N * 8);
  o.vg = c.take(2 * N * 8);
  o.vr = c.take(2 * N * 8);
  o.keys = c.take(N * 4);
  o.cl = c.take(N * 8);
  o.ca = c.take(N * 8);
  o.twx = c.take((size_t)nx * 16);
  o.twy = c.take((size_t)ny * 16);
  o.ktx = c.take((size_t)nx * 8);
  o.kty = c.take((size_t)ny * 8);
  // one complex plane: the column kernel reads and writes the columns its block
  // owns, so it works in place; the place of a second plane holds the filter
  // table, 24 (nx / 2 + 1) (ny / 2 + 1) <= 16 N bytes for nx, ny >= 8
  o.P = o.Q = c.take(N * 16);
  o.filt = c.take(N * 16);
  o.off_in = c.take((size_t)(o.n_in > 0 ? o.n_in : 1) * 8);
  o.off_l = c.take((size_t)o.n_l * 8);
  o.w_l = c.take((size_t)o.n_l * 16);
  // block sums of the render, then of the last FFT kernel (at most one per row)
  o.part = c.take((size_t)(o.nblk + (o.nblk > ny ? o.nblk : ny)) * 8);
  o.tot = c.take(2 * 8);
  o.cnt = c.take(BATCH * 4);
  o.total = c.off;
  return o;
}

}  // namespace
}  // namespace mhd

using namespace mhd;

struct mhd_gran_ctx {
  int nx, ny;
  double dx, dy;
  mhd_gran_params gp;
  char* ws;
  Layout2 o;
  GranDev g;
  FFTPlan fp;
  cudaStream_t st;
  bool tiles;       // the tile kernels serve this plane and these radii
  Disk din, dl;     // r_inner, r_lane
  size_t smem_l;    // dynamic shared memory of the tiled render
  long long launches = 0;
  char err[512] = "no error";
};

static int gfail(mhd_gran_ctx* g, int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  if (g) snprintf(g->err, sizeof g->err, "%s", buf);
  else set_global_error("%s", buf);
  return code;
}

static int gcheck(mhd_gran_ctx* g, cudaError_t e, const char* what) {
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) return gfail(g, MHD_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
  return MHD_OK;
}

// A host table to the device, ordered on the generator's stream: cudaMemcpy may
// return once the table is staged, with its transfer still under way on the
// legacy stream, which a non-blocking stream does not wait for.  (Pageable
// memory is staged before the call returns, so the table may go.)
static int upload(mhd_gran_ctx* g, const void* dst, const void* src, size_t bytes, const char* what) {
  return gcheck(g, cudaMemcpyAsync((void*)dst, src, bytes, cudaMemcpyHostToDevice, g->st), what);
}

extern "C" size_t mhd_gran_workspace_bytes(int nx, int ny, double dx, double dy, const mhd_gran_params* gp) {
  if (check(nx, ny, dx, dy, gp)) return 0;
  return carve(nx, ny, dx, dy, gp).total;
}

extern "C" int mhd_gran_create(int nx, int ny, double dx, double dy, const mhd_gran_params* gp, void* workspace,
                               size_t ws_bytes, void* stream, mhd_gran_handle* out) {
  if (!out) return gfail(nullptr, MHD_ERR_ARG, "out is NULL");
  *out = nullptr;
  const char* bad = check(nx, ny, dx, dy, gp);
  if (bad) return gfail(nullptr, MHD_ERR_ARG, "%s", bad);
  const Layout2 o = carve(nx, ny, dx, dy, gp);
  if (!workspace || ((uintptr_t)workspace & 255) || ws_bytes < o.total)
    return gfail(nullptr, MHD_ERR_WORKSPACE, "workspace must be 256-byte aligned with at least %zu bytes", o.total);
  mhd_gran_ctx* g = new mhd_gran_ctx;
  g->nx = nx;
  g->ny = ny;
  g->dx = dx;
  g->dy = dy;
  g->gp = *gp;
  g->ws = (char*)workspace;
  g->o = o;
  g->st = (cudaStream_t)stream;
  const size_t N = (size_t)nx * ny;
  GranDev& d = g->g;
  d.nx = nx;
  d.ny = ny;
  d.occ = (int*)(g->ws + o.occ);
  d.t0 = (double*)(g->ws + o.par);
  d.life = d.t0 + N;
  d.vmax = d.t0 + 2 * N;
  d.tmax = d.t0 + 3 * N;
  d.mis = (int*)(g->ws + o.mis);
  d.amp = (double*)(g->ws + o.amp);
  d.vg = (double*)(g->ws + o.vg);
  d.vr = (double*)(g->ws + o.vr);
  d.off_in = (const int2*)(g->ws + o.off_in);
  d.n_in = o.n_in;
  d.off_l = (const int2*)(g->ws + o.off_l);
  d.w_l = (const double2*)(g->ws + o.w_l);
  d.n_l = o.n_l;
  d.part = (double*)(g->ws + o.part);
  d.tot = (double*)(g->ws + o.tot);
  d.cnt = (int*)(g->ws + o.cnt);
  FFTPlan& fp = g->fp;
  memset(&fp, 0, sizeof fp);
  fp.nx = nx;
  fp.ny = ny;
  fp.lognx = lg2(nx);
  fp.logny = lg2(ny);
  fp.twx = (const double2*)(g->ws + o.twx);
  fp.twy = (const double2*)(g->ws + o.twy);
  fp.ktx = (const double*)(g->ws + o.ktx);
  fp.kty = (const double*)(g->ws + o.kty);
  fp.P = (double2*)(g->ws + o.P);
  fp.Q = (double2*)(g->ws + o.Q);
  fp.filt = (const double*)(g->ws + o.filt);
  fp.p0 = 0;
  fp.knx = M_PI / dx;
  fp.kny = M_PI / dy;
  // host tables: twiddles, signed wavenumbers 2 pi m / L, disk offsets and
  // the lane weights profile(|o|) o / |o| (linear rise to r_granule, cos^2
  // fall to r_lane)
  int rc = MHD_OK;
  for (int axis = 0; axis < 2 && rc == MHD_OK; ++axis) {
    const int n = axis == 0 ? nx : ny;
    const double L = n * (axis == 0 ? dx : dy);
    std::vector<double> tw((size_t)2 * n), k((size_t)n);
    for (int r = 0; r < n; ++r) {
      const double2 w = twiddle_pair(cos(2.0 * M_PI * r / n), -sin(2.0 * M_PI * r / n), r,
                                     axis == 0 ? fp.lognx : fp.logny);
      tw[2 * r] = w.x;
      tw[2 * r + 1] = w.y;
      k[r] = 2.0 * M_PI * (2 * r > n ? r - n : r) / L;
    }
    rc = upload(g, axis == 0 ? fp.twx : fp.twy, tw.data(), (size_t)n * 16, "upload twiddles");
    if (rc == MHD_OK) rc = upload(g, axis == 0 ? fp.ktx : fp.kty, k.data(), (size_t)n * 8, "upload wavenumbers");
  }
  const std::vector<int2> din = disk(gp->r_inner, dx, dy), dl = disk(gp->r_lane, dx, dy);
  std::vector<double2> wl(dl.size());
  for (size_t n = 0; n < dl.size(); ++n) {
    const double ex = dl[n].x * dx, ey = dl[n].y * dy;
    const double r = sqrt(ex * ex + ey * ey);
    double f;
    if (r <= gp->r_granule) {
      f = r / gp->r_granule;
    } else {
      const double c = cos(0.5 * M_PI * (r - gp->r_granule) / (gp->r_lane - gp->r_granule));
      f = c * c;
    }
    wl[n] = make_double2(f * ex / r, f * ey / r);
  }
  if (rc == MHD_OK && !din.empty()) rc = upload(g, d.off_in, din.data(), din.size() * 8, "upload disk");
  if (rc == MHD_OK) rc = upload(g, d.off_l, dl.data(), dl.size() * 8, "upload lane");
  if (rc == MHD_OK) rc = upload(g, d.w_l, wl.data(), wl.size() * 16, "upload weights");
  if (rc == MHD_OK)
    rc = gcheck(g, cudaMemsetAsync(g->ws + o.occ, 0, N * 4, g->st), "clear granules");
  if (rc == MHD_OK)
    rc = gcheck(g, cudaMemsetAsync(g->ws + o.par, 0, 4 * N * 8, g->st), "clear granules");
  if (rc == MHD_OK)
    rc = gcheck(g, cudaMemsetAsync(g->ws + o.vg, 0, 4 * N * 8, g->st), "clear fields");
  if (rc == MHD_OK) {
    const bool in = disk_rows(gp->r_inner, dx, dy, &g->din), lane = disk_rows(gp->r_lane, dx, dy, &g->dl);
    g->tiles = in && lane && nx >= TW;
    g->smem_l = sizeof(double2) * (2 * g->dl.rx + 1) * (2 * g->dl.ry + 1) +
                sizeof(double) * (TW + 2 * g->dl.rx) * (TH + 2 * g->dl.ry);
    const int nq = (nx / 2 + 1) * (ny / 2 + 1);
    filter_kernel<<<(nq + GT - 1) / GT, GT, 0, g->st>>>(fp, (double*)(g->ws + o.filt));
    rc = gcheck(g, cudaGetLastError(), "filter table");
  }
  if (rc == MHD_OK) rc = gcheck(g, cudaStreamSynchronize(g->st), "create");
  if (rc != MHD_OK) {
    set_global_error("%s", g->err);
    delete g;
    return rc;
  }
  *out = g;
  return MHD_OK;
}

static const void* stage(mhd_gran_ctx* g, const void* src, size_t off, size_t bytes, int mem, int* rc) {
  if (mem == MHD_MEM_DEVICE) return src;
  *rc = gcheck(g, cudaMemcpyAsync(g->ws + off, src, bytes, cudaMemcpyHostToDevice, g->st), "stage input");
  return g->ws + off;
}

extern "C" int mhd_gran_update(mhd_gran_handle g, double t, const unsigned int* keys, const double* c_life,
                               const double* c_amp, int mem, int* rounds) {
  if (!g) return gfail(nullptr, MHD_ERR_ARG, "generator is NULL");
  if (!keys || !c_life || !c_amp) return gfail(g, MHD_ERR_ARG, "keys, c_life and c_amp are required");
  if (mem != MHD_MEM_DEVICE && mem != MHD_MEM_HOST) return gfail(g, MHD_ERR_ARG, "bad mem flag");
  if (!std::isfinite(t)) return gfail(g, MHD_ERR_ARG, "t must be finite");
  const size_t N = (size_t)g->nx * g->ny;
  int rc = MHD_OK;
  const unsigned* k = (const unsigned*)stage(g, keys, g->o.keys, N * 4, mem, &rc);
  const double* cl = rc ? nullptr : (const double*)stage(g, c_life, g->o.cl, N * 8, mem, &rc);
  const double* ca = rc ? nullptr : (const double*)stage(g, c_amp, g->o.ca, N * 8, mem, &rc);
  if (rc) return rc;
  const int nb = g->o.nblk, nl = (int)((N + (size_t)LP * GT - 1) / ((size_t)LP * GT));
  const dim3 tiles(g->nx / TW, g->ny / TH);
  if (g->tiles) seed_tile_kernel<<<tiles, GT, 0, g->st>>>(g->g, g->din, t);
  else seed_kernel<<<nb, GT, 0, g->st>>>(g->g, t);
  g->launches += 1;
  // each round the first undecided pixel in (key, index) order joins, so
  // N + 1 rounds always suffice.  The host reads the undecided counts once per
  // batch of rounds (a steady update takes about three rounds).
  int r = 0, left = 1;
  while (left > 0) {
    if (r > (int)N) return gfail(g, MHD_ERR_TIMEOUT, "placement did not settle in %d rounds", r);
    rc = gcheck(g, cudaMemsetAsync(g->g.cnt, 0, BATCH * 4, g->st), "clear count");
    if (rc) return rc;
    for (int b = 0; b < BATCH; ++b) {
      if (g->tiles) {
        join_tile_kernel<<<tiles, GT, 0, g->st>>>(g->g, g->din, k, b);
        exclude_tile_kernel<<<tiles, GT, 0, g->st>>>(g->g, g->din, b);
      } else {
        join_kernel<<<nb, GT, 0, g->st>>>(g->g, k, b);
        exclude_kernel<<<nb, GT, 0, g->st>>>(g->g, b);
      }
    }
    g->launches += 2 * BATCH;
    int cnt[BATCH];
    rc = gcheck(g, cudaMemcpyAsync(cnt, g->g.cnt, sizeof cnt, cudaMemcpyDeviceToHost, g->st), "read count");
    if (rc == MHD_OK) rc = gcheck(g, cudaStreamSynchronize(g->st), "placement round");
    if (rc) return rc;
    for (int b = 0; b < BATCH && left > 0; ++b) {
      left = cnt[b];
      ++r;
    }
  }
  birth_kernel<<<nl, GT, 0, g->st>>>(g->g, g->gp, t, cl, ca);
  g->launches += 1;
  if (rounds) *rounds = r;
  rc = gcheck(g, cudaGetLastError(), "update");
  if (rc == MHD_OK && mem == MHD_MEM_HOST) rc = gcheck(g, cudaStreamSynchronize(g->st), "update");
  return rc;
}

extern "C" int mhd_gran_velocity(mhd_gran_handle g, double t, int precision, void* v, int mem) {
  if (!g) return gfail(nullptr, MHD_ERR_ARG, "generator is NULL");
  if (!v) return gfail(g, MHD_ERR_ARG, "v is NULL");
  if (precision != 32 && precision != 64) return gfail(g, MHD_ERR_ARG, "precision must be 32 or 64");
  if (mem != MHD_MEM_DEVICE && mem != MHD_MEM_HOST) return gfail(g, MHD_ERR_ARG, "bad mem flag");
  if (!std::isfinite(t)) return gfail(g, MHD_ERR_ARG, "t must be finite");
  const size_t N = (size_t)g->nx * g->ny;
  const int nb = g->o.nblk;
  const GranDev& d = g->g;
  amp_kernel<<<(int)((N + (size_t)LP * GT - 1) / ((size_t)LP * GT)), GT, 0, g->st>>>(d, t);
  if (g->tiles) render_tile_kernel<<<dim3(g->nx / TW, g->ny / TH), GT, g->smem_l, g->st>>>(d, g->dl);
  else render_kernel<<<nb, GT, 0, g->st>>>(d);
  const int nvor = launch_rotational(g->fp, d.vg, d.vg + N, d.vr, d.vr + N, true, g->gp.f_rot, d.part + nb, g->st);
  total_kernel<<<1, GT, 0, g->st>>>(d, nb, nvor);
  g->launches += 6;
  // device output straight into v; host output through the FFT's plane (2N
  // doubles), free once the inverse rows have read it
  void* dst = mem == MHD_MEM_DEVICE ? v : (void*)(g->ws + g->o.P);
  if (precision == 64) scale_kernel<double><<<nb, GT, 0, g->st>>>(d, (double*)dst);
  else scale_kernel<float><<<nb, GT, 0, g->st>>>(d, (float*)dst);
  g->launches += 1;
  int rc = gcheck(g, cudaGetLastError(), "velocity");
  if (rc == MHD_OK && mem == MHD_MEM_HOST) {
    rc = gcheck(g, cudaMemcpyAsync(v, dst, 2 * N * (precision == 64 ? 8 : 4), cudaMemcpyDeviceToHost, g->st),
                "read velocity");
    if (rc == MHD_OK) rc = gcheck(g, cudaStreamSynchronize(g->st), "read velocity");
  }
  return rc;
}

static int copy_out(mhd_gran_ctx* g, void* dst, const void* src, size_t bytes, int mem) {
  const cudaMemcpyKind kind = mem == MHD_MEM_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  int rc = gcheck(g, cudaMemcpyAsync(dst, src, bytes, kind, g->st), "read");
  if (rc == MHD_OK && mem == MHD_MEM_HOST) rc = gcheck(g, cudaStreamSynchronize(g->st), "read");
  return rc;
}

extern "C" int mhd_gran_read_granules(mhd_gran_handle g, int* occ, double* par, int mem) {
  if (!g) return gfail(nullptr, MHD_ERR_ARG, "generator is NULL");
  if (!occ) return gfail(g, MHD_ERR_ARG, "occ is NULL");
  if (mem != MHD_MEM_DEVICE && mem != MHD_MEM_HOST) return gfail(g, MHD_ERR_ARG, "bad mem flag");
  const size_t N = (size_t)g->nx * g->ny;
  int rc = copy_out(g, occ, g->g.occ, N * 4, mem);
  if (rc == MHD_OK && par) rc = copy_out(g, par, g->g.t0, 4 * N * 8, mem);
  return rc;
}

extern "C" int mhd_gran_read_field(mhd_gran_handle g, int which, double* dst, int mem) {
  if (!g) return gfail(nullptr, MHD_ERR_ARG, "generator is NULL");
  if (!dst) return gfail(g, MHD_ERR_ARG, "dst is NULL");
  if (which != 0 && which != 1) return gfail(g, MHD_ERR_ARG, "which must be 0 or 1");
  if (mem != MHD_MEM_DEVICE && mem != MHD_MEM_HOST) return gfail(g, MHD_ERR_ARG, "bad mem flag");
  const size_t N = (size_t)g->nx * g->ny;
  if (which == 0) return copy_out(g, dst, g->g.vg, 2 * N * 8, mem);
  // v_rot' is not kept (the FFT's last kernel adds it to v_gran): recompute it
  // from v_gran in the place of v_vor, which the next velocity forms anew
  launch_rotational(g->fp, g->g.vg, g->g.vg + N, g->g.vr, g->g.vr + N, false, 0.0, nullptr, g->st);
  g->launches += 3;
  int rc = gcheck(g, cudaGetLastError(), "rotational part");
  if (rc) return rc;
  return copy_out(g, dst, g->g.vr, 2 * N * 8, mem);
}

extern "C" long long mhd_gran_launch_count(mhd_gran_handle g) { return g ? g->launches : 0; }

extern "C" const char* mhd_gran_last_error(mhd_gran_handle g) { return g ? g->err : mhd_last_error(nullptr); }

extern "C" void mhd_gran_destroy(mhd_gran_handle g) { delete g; }
