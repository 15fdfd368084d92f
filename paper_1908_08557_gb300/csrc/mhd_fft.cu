// mhd_fft.cu -- FP64 horizontal FFT of the potential-field boundary
// (Sect. 4.2, Eqs. 16-17; Sect. 2.4 inverted extrapolation) and of the
// magnetogram inversion (Sect. 2.4, Eq. 7).
//
// The six real boundary planes (A_x, A_y, A_z at the top layer and at the
// photosphere) travel as three complex planes:
//   P0 = A_x(top) + i A_y(top),  P1 = A_x(bot) + i A_y(bot),
//   P2 = A_z(top) + i A_z(bot).
// The extrapolation multiplier M(k) is real and even in k, so applying it to
// a packed plane extrapolates both real parts at once.  P2 carries two planes
// with different multipliers M_t, M_b; with F = FFT(P2) the spectrum to invert
// is a F(k) + b conj(F(-k)), a = (M_t + M_b)/2, b = (M_t - M_b)/2, whose inverse
// has real part = top ghost and imaginary part = bottom ghost.
//
// Kernels (radix-4 Stockham autosort in shared memory, FP64):
//   1. rows_fwd: pack rows from the state, FFT along x, store transposed
//   2. cols:     FFT along y, for each ghost layer j = 1..3 form the
//                extrapolated spectrum (M_t = exp(-|k| j dz),
//                M_b = exp(+f_b |k| j dz)), inverse FFT along y
//   3. rows_inv: inverse FFT along x, write real/imaginary parts into the
//                ghost layers (with their periodic x,y images)
#include "mhd_bc.cuh"
#include "mhd_internal.h"

namespace mhd {

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// One radix-2 butterfly with its twiddle, (b0 + w b1, b0 - w b1), in six FP64
// multiply-adds (four for the product and four for the sums otherwise; the
// transforms are bound by the FP64 pipe): with w = m (1 + i t) the product is
// m (u, v), u = x - t y, v = y + t x, and the factor m rides on the sums.
// Where |Im w| > |Re w| the same with w = i m (1 + i t), i.e. for (-y, x), so
// that |t| <= 1 and nothing is lost (twiddle_pair, mhd_internal.h); the tangent
// form of a twiddle for fused multiply-adds is that of Linzer and Feig (1993).
// inv: conjugate twiddle.
// Signs and swaps go by integer operations (a negated copy can cost an FP64
// one).
__device__ __forceinline__ double flip(double x, int sign) {
  return __hiloint2double(__double2hiint(x) ^ sign, __double2loint(x));
}
__device__ __forceinline__ void bfly(double2 b0, double2 b1, double2 w, bool swap, bool inv, double2& s, double2& d) {
  constexpr int S = (int)0x80000000;
  const double ny = flip(b1.y, S);
  const double p = __hiloint2double(swap ? __double2hiint(ny) : __double2hiint(b1.x),
                                    swap ? __double2loint(ny) : __double2loint(b1.x));
  const double q = __hiloint2double(swap ? __double2hiint(b1.x) : __double2hiint(b1.y),
                                    swap ? __double2loint(b1.x) : __double2loint(b1.y));
  const double t = flip(w.y, inv ? S : 0), m = flip(w.x, inv && swap ? S : 0);
  const double u = fma(-t, q, p), v = fma(t, p, q);
  s = make_double2(fma(m, u, b0.x), fma(m, v, b0.y));
  d = make_double2(fma(-m, u, b0.x), fma(-m, v, b0.y));
}

// nb lines of n = 2^logn complex points in a (b is scratch of equal size).
// Stockham autosort, radix 4, with one radix-2 stage first when logn is odd.
// With p the length of the sub-transforms done so far, radix-4 butterfly
// i in [0, n/4) has k = i mod p, j = i div p; it takes x[i + m n/4]
// (m = 0..3) times w^(m k), w = exp(-+2 pi i / (4p)), and writes their
// 4-point DFT c_q to y[4 j p + k + q p] = y[4i - 3k + q p]; the twiddles
// enter as two levels of radix-2 butterflies, w^(2k) then w^k.  At p = 1
// every k is 0 and the twiddles drop out; the radix-2 stage (p = 1) writes
// x[i] +- x[i + n/2] to y[2i], y[2i + 1].  Returns the buffer holding the
// (unnormalised) transform.
__device__ double2* fft_lines(double2* a, double2* b, int n, int logn, int nb, const double2* __restrict__ tw,
                              bool inverse) {
  int p = 1, lp = 0;
  if (2 * (int)blockDim.x >= nb * n) {
    // a thread per radix-2 butterfly: where threads are plenty the transform is
    // a chain of FP64 instructions of 64 clocks each, 34 here against 64 in the
    // radix-4 form below for 64 points (64 x 64 planes, three fills of a step:
    // 148 -> 143 us a step at 64^3)
    const int half = n >> 1;
    const int q = threadIdx.x, line = q >> (logn - 1), i = q & (half - 1);
    const bool on = q < nb * half;
    for (; p < n; p <<= 1, ++lp) {
      if (on) {
        const int k = i & (p - 1);
        const double2 u0 = a[line * n + i], u1 = a[line * n + i + half];
        double2* y = b + line * n + 2 * i - k;
        double2 s, d;
        if (p > 1) {
          const int r = k << (logn - 1 - lp);
          bfly(u0, u1, __ldg(tw + r), twiddle_swap(r, logn), inverse, s, d);
        } else {
          s = cadd(u0, u1);
          d = csub(u0, u1);
        }
        y[0] = s;
        y[p] = d;
      }
      __syncthreads();
      double2* t = a;
      a = b;
      b = t;
    }
    return a;
  }
  if (logn & 1) {
    const int half = n >> 1;
    const int total = nb * half;
    for (int q = threadIdx.x; q < total; q += blockDim.x) {
      const int line = q >> (logn - 1);
      const int i = q & (half - 1);
      const double2 u0 = a[line * n + i], u1 = a[line * n + i + half];
      b[line * n + 2 * i] = cadd(u0, u1);
      b[line * n + 2 * i + 1] = csub(u0, u1);
    }
    __syncthreads();
    double2* t = a;
    a = b;
    b = t;
    p = 2;
    lp = 1;
  }
  const int quarter = n >> 2;
  const int total = nb * quarter;
  const int rs = inverse ? (int)0x80000000 : 0;
  for (; p < n; p <<= 2, lp += 2) {
    const int tws = logn - 2 - lp;  // twiddle index m k n / (4p) = (m k) << tws
    for (int q = threadIdx.x; q < total; q += blockDim.x) {
      const int line = q >> (logn - 2);
      const int i = q & (quarter - 1);
      const int k = i & (p - 1);
      const double2* x = a + line * n + i;
      const double2 b0 = x[0], b1 = x[quarter], b2 = x[2 * quarter], b3 = x[3 * quarter];
      double2* y = b + line * n + 4 * i - 3 * k;
      if (p > 1) {
        const int r1 = k << tws, r2 = (2 * k) << tws;
        const double2 w1 = __ldg(tw + r1), w2 = __ldg(tw + r2);
        const bool s1 = twiddle_swap(r1, logn), s2 = twiddle_swap(r2, logn);
        double2 t0, t1, t2, t3, y0, y1, y2, y3;
        bfly(b0, b2, w2, s2, inverse, t0, t1);
        bfly(b1, b3, w2, s2, inverse, t2, t3);
        bfly(t0, t2, w1, s1, inverse, y0, y2);
        // -i t3 for the forward transform, +i t3 for the inverse
        bfly(t1, make_double2(flip(t3.y, rs), flip(t3.x, ~rs & (int)0x80000000)), w1, s1, inverse, y1, y3);
        y[0] = y0;
        y[p] = y1;
        y[2 * p] = y2;
        y[3 * p] = y3;
      } else {
        const double2 t0 = cadd(b0, b2), t1 = csub(b0, b2), t2 = cadd(b1, b3), t3 = csub(b1, b3);
        const double2 r3 = inverse ? make_double2(-t3.y, t3.x) : make_double2(t3.y, -t3.x);
        y[0] = cadd(t0, t2);
        y[p] = cadd(t1, r3);
        y[2 * p] = csub(t0, t2);
        y[3 * p] = csub(t1, r3);
      }
    }
    __syncthreads();
    double2* t = a;
    a = b;
    b = t;
  }
  return a;
}

// ---------------------------------------------------------------------------
// 1. forward rows.  mode 0: three boundary planes of the state; mode 1: one
// real plane `src2d` ([ny][nx], the magnetogram).
// mode 2 (adjoint of the potential-field ghosts): plane p = 3c + m - 1 packs
// the ghost adjoints of A_c at the top layer nz-1+m (real) and at -m
// (imaginary); mode 3: the complex plane dre + i dim (FP64 inputs).
template <typename R>
__global__ void __launch_bounds__(256) rows_fwd_kernel(FFTPlan fp, Layout L, const R* f, const R* src2d, int mode,
                                                       const StepState* ss, int nb, const double* dre,
                                                       const double* dim) {
  extern __shared__ double2 sm[];
  chain_enter();
  if (ss && halted(ss)) return;
  const int nx = fp.nx, ny = fp.ny;
  const int y0 = blockIdx.x * nb;
  const int p = fp.p0 + blockIdx.y;
  double2* a = sm;
  double2* b = sm + nb * nx;
  const int kt = L.nz - 1;
  for (int q = threadIdx.x; q < nb * nx; q += blockDim.x) {
    const int line = q / nx, x = q - line * nx, y = y0 + line;
    double re, im;
    if (mode == 1) {
      re = (double)src2d[(long long)y * nx + x];
      im = 0.0;
    } else if (mode == 2) {
      const int cc = p / 3, m = p - 3 * cc + 1;
      re = (double)f[L.at(AX + cc, kt + m, y, x)];
      im = (double)f[L.at(AX + cc, -m, y, x)];
    } else if (mode == 3) {
      re = dre[(long long)y * nx + x];
      im = dim[(long long)y * nx + x];
    } else if (p == 0) {
      re = (double)f[L.at(AX, kt, y, x)];
      im = (double)f[L.at(AY, kt, y, x)];
    } else if (p == 1) {
      re = (double)f[L.at(AX, 0, y, x)];
      im = (double)f[L.at(AY, 0, y, x)];
    } else {
      re = (double)f[L.at(AZ, kt, y, x)];
      im = (double)f[L.at(AZ, 0, y, x)];
    }
    a[line * nx + x] = make_double2(re, im);
  }
  __syncthreads();
  double2* r = fft_lines(a, b, nx, fp.lognx, nb, fp.twx, false);
  // transposed store: P[p][x][y], consecutive threads walk y
  for (int q = threadIdx.x; q < nb * nx; q += blockDim.x) {
    const int x = q / nb, line = q - x * nb;
    fp.P[((long long)p * nx + x) * ny + y0 + line] = r[line * nx + x];
  }
}

// ---------------------------------------------------------------------------
// 2. columns.  A block owns column pairs (kx, nx - kx); both columns of a pair
// are needed to split the packed plane P2 (F(-k) lives in the mirror column).
// mode 0: potential-field extrapolation, 3 layers; mode 1: magnetogram
// inversion (Eq. 7): A^_x + i A^_y = (kt_x + i kt_y) B^_z / kt^2; mode 2: its
// transpose; mode 4: the filtered rotational part of the granulation field
// (Sect. 2.3, Eq. 3).  The spectra of lg output layers at a time are formed and
// inverted as one batch of lines, so each stage of the inverse transform has
// lg times the butterflies between two barriers; with all of the layers o_first
// .. o_end - 1 in one batch two buffers of lg layers do (the forward spectrum's
// buffer becomes the scratch), otherwise three (the spectrum is kept).  A block
// reads and writes its own columns only, so with one output plane P and Q may be
// the same.
__device__ __forceinline__ void cols_block(const FFTPlan& fp, int mode, int ppb, int lg, int o_first, int o_end) {
  extern __shared__ double2 sm[];
  const int nx = fp.nx, ny = fp.ny;
  const int npairs = nx / 2 + 1;
  const int pair0 = blockIdx.x * ppb;  // ppb column pairs per block
  const int np = min(ppb, npairs - pair0);
  const int nl = 2 * np;
  const int p = fp.p0 + blockIdx.y;
  const int npts = nl * ny;            // points of one layer
  const int bsz = lg * 2 * ppb * ny;   // points of one buffer
  double2* A = sm;
  double2* B = sm + bsz;
  double2* Z = sm + 2 * bsz;           // more than one batch
  // columns of line l: pair (l >> 1), mirror if odd
  for (int q = threadIdx.x; q < npts; q += blockDim.x) {
    const int line = q / ny, y = q - line * ny;
    const int kx = pair0 + (line >> 1);
    const int col = (line & 1) ? ((nx - kx) & (nx - 1)) : kx;
    A[line * ny + y] = fp.P[((long long)p * nx + col) * ny + y];
  }
  __syncthreads();
  double2* spec = fft_lines(A, B, ny, fp.logny, nl, fp.twy, false);
  double2* G = (spec == A) ? B : A;  // layer o0 + o's lines at G + o npts
  double2* T = lg == o_end - o_first ? spec : Z;
  const int nplanes = mode == 0 ? 3 : 1;
  for (int o0 = o_first; o0 < o_end; o0 += lg) {
  for (int q = threadIdx.x; q < lg * npts; q += blockDim.x) {
    const int o = o0 + q / npts, qq = q - (o - o0) * npts;
    const int line = qq / ny, ky = qq - line * ny;
    const int kx = pair0 + (line >> 1);
    const int col = (line & 1) ? ((nx - kx) & (nx - 1)) : kx;
    const double2 F = spec[qq];
    double2 g;
    if (mode == 1) {
      const double kxm = fp.ktx[col], kym = fp.kty[ky];
      const double k2 = kxm * kxm + kym * kym;
      if (k2 > 0.0) {
        const double2 m = make_double2(kxm / k2, kym / k2);
        g = cmul(m, F);
      } else {
        g = make_double2(0.0, 0.0);
      }
    } else if (mode == 4) {
      // F = FFT(v_x + i v_y).  With V_x = (F + conj F(-k)) / 2 and
      // V_y = (F - conj F(-k)) / 2i, the divergence-free part
      // V - k (k . V) / |k|^2 packs as (F - e^(2 i theta) conj F(-k)) / 2,
      // e^(i theta) = (k_x + i k_y) / |k|; times the filter
      // exp(-(2 |k| / k_N)^4).  The mean and the Nyquist modes (whose signed
      // wavenumber has no partner) carry none.
      // (w, w cos 2 theta, w sin 2 theta) from the quarter table: formed
      // here, the exponential and the divisions took half of the launch
      const int ka = col <= nx / 2 ? col : nx - col, kb = ky <= ny / 2 ? ky : ny - ky;
      const double* t = fp.filt + 3 * ((long long)ka * (ny / 2 + 1) + kb);
      const double w = __ldg(t), wc = __ldg(t + 1), ws0 = __ldg(t + 2);
      const double ws = (col > nx / 2) != (ky > ny / 2) ? -ws0 : ws0;
      const double2 Fm = spec[(line ^ 1) * ny + ((ny - ky) & (ny - 1))];
      g = make_double2(w * F.x - (wc * Fm.x + ws * Fm.y), w * F.y - (ws * Fm.x - wc * Fm.y));
    } else if (mode == 2) {
      // transpose of Eq. 7's inversion: with F = FFT(X + i Y) for real X,
      // Y (the adjoints of A_x, A_y), the spectrum of the B_z adjoint is
      // conj(m_x) X + conj(m_y) Y = [(kt_x - i kt_y) F - (kt_x + i kt_y) conj F(-k)] / (2 kt^2)
      const double kxm = fp.ktx[col], kym = fp.kty[ky];
      const double k2 = kxm * kxm + kym * kym;
      if (k2 > 0.0) {
        const double2 Fm = spec[(line ^ 1) * ny + ((ny - ky) & (ny - 1))];
        const double2 Fc = make_double2(Fm.x, -Fm.y);
        const double2 t1 = cmul(make_double2(kxm, -kym), F);
        const double2 t2 = cmul(make_double2(kxm, kym), Fc);
        g = make_double2((t1.x - t2.x) / (2.0 * k2), (t1.y - t2.y) / (2.0 * k2));
      } else {
        g = make_double2(0.0, 0.0);
      }
    } else {
      // ghost layer o + 1: the multipliers of its distance from the top
      // layer (M_t) and, below the photosphere, from the bottom one (M_b)
      const long long e = (long long)o * nx * ny + (long long)col * ny + ky;
      const double mt = fp.et[e], mb = fp.eb[e];
      if (p == 0) {
        g = make_double2(mt * F.x, mt * F.y);
      } else if (p == 1) {
        g = make_double2(mb * F.x, mb * F.y);
      } else {
        const double2 Fm = spec[(line ^ 1) * ny + ((ny - ky) & (ny - 1))];
        const double ca = 0.5 * (mt + mb), cb = 0.5 * (mt - mb);
        g = make_double2(ca * F.x + cb * Fm.x, ca * F.y - cb * Fm.y);
      }
    }
    G[q] = g;
  }
  __syncthreads();
  const double2* r = fft_lines(G, T, ny, fp.logny, lg * nl, fp.twy, true);
  for (int q = threadIdx.x; q < lg * npts; q += blockDim.x) {
    const int o = o0 + q / npts, qq = q - (o - o0) * npts;
    const int line = qq / ny, y = qq - line * ny;
    const int kx = pair0 + (line >> 1);
    const bool self = (kx == 0 || 2 * kx == nx);
    if ((line & 1) && self) continue;  // the mirror of a self-paired column
    const int col = (line & 1) ? ((nx - kx) & (nx - 1)) : kx;
    fp.Q[(((long long)o * nplanes + p) * nx + col) * ny + y] = r[q];
  }
  __syncthreads();
  }
}

// gridDim.z = 3: one ghost layer per block, the forward transform repeated in
// each.  While that leaves at most two blocks per SM the repetition costs no
// time and the inverse has a third of the serial FP64 instructions.
__global__ void __launch_bounds__(256) cols_kernel(FFTPlan fp, int mode, const StepState* ss, int ppb, int lg) {
  chain_enter();
  if (ss && halted(ss)) return;
  const int o = gridDim.z > 1 ? (int)blockIdx.z : 0, n = mode == 0 && gridDim.z == 1 ? 3 : 1;
  cols_block(fp, mode, ppb, lg, o, o + n);
}

// The columns of the potential-field ghosts with the pointwise ghost rules in
// the same launch, on planes whose boundary chain is a row of short kernels:
// the rules touch no plane of the transforms, and the blocks from x = ncol on
// take them, both ends of all columns, beside the transforms (ghost
// fill 64 x 64 31 -> 23 us, 32 x 32 21 -> 17: the rules' launch is gone from the
// chain, and their time is hidden).
template <typename R>
__global__ void __launch_bounds__(256) cols_rules_kernel(FFTPlan fp, const StepState* ss, int ppb, int lg, int ncol,
                                                         Layout L, Phys<R> ph, Background<R> bg, R* f) {
  chain_enter();
  if (halted(ss)) return;
  if ((int)blockIdx.x < ncol) {
    const int o = gridDim.z > 1 ? (int)blockIdx.z : 0;
    cols_block(fp, 0, ppb, lg, o, gridDim.z > 1 ? o + 1 : 3);
    return;
  }
  const int pw = L.nx + 2 * NG, n = pw * (L.ny + 2 * NG);
  const int blk = ((int)(blockIdx.x - ncol) * gridDim.y + blockIdx.y) * gridDim.z + blockIdx.z;
  const int q = blk * blockDim.x + threadIdx.x;
  if (q >= 2 * n) return;
  const int c = q < n ? q : q - n;
  ghost_rules<R>(L, ph, bg, f, c % pw - NG, c / pw - NG, q >= n);
}

// ---------------------------------------------------------------------------
// 3. inverse rows, normalised by 1/(nx ny) (modes 0 and 2: through the
// multipliers); mode 0 writes ghost layers of the state, mode 1 the compact planes out_re, out_im ([ny][nx]).
// mode 2 (adjoint): plane c adds its real part into A_c at the top layer and
// its imaginary part into A_c at the photosphere (interior x, y only);
// mode 3: real part into out_re.
struct RowsAdd {  // mode 5
  const double* vx;
  const double* vy;
  double f_rot;
  double* part;
};

template <typename R>
__global__ void __launch_bounds__(256) rows_inv_kernel(FFTPlan fp, Layout L, R* f, R* out_re,
                                                       R* out_im, int mode, const StepState* ss, int nb, RowsAdd add) {
  extern __shared__ double2 sm[];
  chain_enter();
  double energy = 0.0;
  if (ss && halted(ss)) return;
  const int nx = fp.nx, ny = fp.ny;
  const int y0 = blockIdx.x * nb;
  const int p = fp.p0 + blockIdx.y, o = blockIdx.z;
  const int nplanes = mode == 0 ? 3 : (mode == 2 ? 3 : 1);
  double2* a = sm;
  double2* b = sm + nb * nx;
  for (int q = threadIdx.x; q < nb * nx; q += blockDim.x) {
    const int x = q / nb, line = q - x * nb;
    a[line * nx + x] = fp.Q[(((long long)o * nplanes + p) * nx + x) * ny + y0 + line];
  }
  __syncthreads();
  double2* r = fft_lines(a, b, nx, fp.lognx, nb, fp.twx, true);
  const double sc = 1.0 / ((double)nx * (double)ny), frs = add.f_rot * sc;
  const int m = o + 1;
  const int ktop = L.nz - 1 + m, kbot = -m;
  for (int q = threadIdx.x; q < nb * nx; q += blockDim.x) {
    const int line = q / nx, x = q - line * nx, y = y0 + line;
    const double2 v = r[line * nx + x];
    if (mode == 5) {
      const long long o = (long long)y * nx + x;
      const double wx = fma(frs, v.x, add.vx[o]), wy = fma(frs, v.y, add.vy[o]);
      out_re[o] = (R)wx;
      out_im[o] = (R)wy;
      energy = fma(wx, wx, fma(wy, wy, energy));
      continue;
    }
    // (modes 0 and 2: the multipliers carry the normalisation)
    const bool scaled = mode == 0 || mode == 2;
    const R re = (R)(scaled ? v.x : v.x * sc), im = (R)(scaled ? v.y : v.y * sc);
    if (mode == 1) {
      out_re[(long long)y * nx + x] = re;
      out_im[(long long)y * nx + x] = im;
      continue;
    }
    if (mode == 3) {
      out_re[(long long)y * nx + x] = re;
      continue;
    }
    if (mode == 2) {
      f[L.at(AX + p, L.nz - 1, y, x)] += re;
      f[L.at(AX + p, 0, y, x)] += im;
      continue;
    }
    int f1, k1, f2, k2;
    if (p == 0) { f1 = AX; k1 = ktop; f2 = AY; k2 = ktop; }
    else if (p == 1) { f1 = AX; k1 = kbot; f2 = AY; k2 = kbot; }
    else { f1 = AZ; k1 = ktop; f2 = AZ; k2 = kbot; }
    // the cell and its periodic images (nx, ny >= 8: at most one per direction)
    const int ox = x < NG ? nx : (x >= nx - NG ? -nx : 0);
    const long long oy = y < NG ? (long long)ny * L.mx : (y >= ny - NG ? -(long long)ny * L.mx : 0);
    R* q1 = f + L.at(f1, k1, y, x);
    R* q2 = f + L.at(f2, k2, y, x);
    q1[0] = re;
    q2[0] = im;
    if (ox) {
      q1[ox] = re;
      q2[ox] = im;
    }
    if (oy) {
      q1[oy] = re;
      q2[oy] = im;
    }
    if (ox && oy) {
      q1[ox + oy] = re;
      q2[ox + oy] = im;
    }
  }
  if (mode == 5) {
    // fixed order: warp tree, then the warps in turn
    __shared__ double sh[8];
    for (int o2 = 16; o2 > 0; o2 >>= 1) energy += __shfl_down_sync(0xffffffffu, energy, o2);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = energy;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int q = 0; q < (int)(blockDim.x >> 5); ++q) s += sh[q];
      add.part[blockIdx.x] = s;
    }
  }
}

// Adjoint columns: for component c, sum over the three ghost layers m of the
// extrapolated spectra of the packed ghost adjoints (top real, bottom
// imaginary), then one inverse FFT along y.  Input planes 3c + m - 1 in
// fp.P, output plane c in fp.Q.  lg = 3: the layers' forward transforms as one
// batch of lines (two buffers of three layers); lg = 1: one after the other
// (two buffers of a layer and the sum).
// Blocks ncol .. of x take the transpose of the pointwise ghost rules, which
// touches no plane of the transforms (as in cols_rules_kernel; a taped adjoint
// step at 64 x 32 x 45 in FP64 767 -> 754 us against a launch of its own).
template <typename R>
__global__ void __launch_bounds__(256) cols_adj_kernel(FFTPlan fp, const StepState* ss, int ppb, int lg, int ncol,
                                                       Layout L, Phys<R> ph, Background<R> bg, const R* g, R* gbar,
                                                       R dz) {
  extern __shared__ double2 sm[];
  chain_enter();
  if (ss && halted(ss)) return;
  if ((int)blockIdx.x >= ncol) {
    const int n = fp.nx * fp.ny, q = (((int)blockIdx.x - ncol) * 3 + (int)blockIdx.y) * (int)blockDim.x + (int)threadIdx.x;
    const bool both = L.nz == 2 * NG + 1;
    if (q >= (both ? n : 2 * n)) return;
    const int c = q < n ? q : q - n;
    adj_ghost_rules<R>(L, ph, bg, g, gbar, dz, c % fp.nx, c / fp.nx, q < n, both || q >= n);
    return;
  }
  const int nx = fp.nx, ny = fp.ny;
  const int npairs = nx / 2 + 1;
  const int pair0 = blockIdx.x * ppb;
  const int np = min(ppb, npairs - pair0);
  const int nl = 2 * np, npts = nl * ny;
  const int c = blockIdx.y;
  const int buf = lg * 2 * ppb * ny;
  double2* X = sm;
  double2* Y = sm + buf;
  double2* acc = sm + 2 * buf;  // lg = 1
  double2* T = X;
  for (int m0 = 0; m0 < 3; m0 += lg) {
    __syncthreads();
    for (int q = threadIdx.x; q < lg * npts; q += blockDim.x) {
      const int m = q / npts, qq = q - m * npts;
      const int line = qq / ny, y = qq - line * ny;
      const int kx = pair0 + (line >> 1);
      const int col = (line & 1) ? ((nx - kx) & (nx - 1)) : kx;
      X[q] = fp.P[((long long)(3 * c + m0 + m) * nx + col) * ny + y];
    }
    __syncthreads();
    double2* spec = fft_lines(X, Y, ny, fp.logny, lg * nl, fp.twy, false);
    if (lg == 3) {
      acc = spec == X ? Y : X;  // free once transformed
      T = spec;
    }
    for (int q = threadIdx.x; q < npts; q += blockDim.x) {
      const int line = q / ny, ky = q - line * ny;
      const int kx = pair0 + (line >> 1);
      const int col = (line & 1) ? ((nx - kx) & (nx - 1)) : kx;
      const int mir = (line ^ 1) * ny + ((ny - ky) & (ny - 1));
      double2 s = lg == 3 || m0 == 0 ? make_double2(0.0, 0.0) : acc[q];
      for (int m = 0; m < lg; ++m) {
        const long long e = (long long)(m0 + m) * nx * ny + (long long)col * ny + ky;
        const double mt = fp.et[e], mb = fp.eb[e];
        const double2 F = spec[m * npts + q], Fm = spec[m * npts + mir];
        const double ca = 0.5 * (mt + mb), cb = 0.5 * (mt - mb);
        s.x += ca * F.x + cb * Fm.x;
        s.y += ca * F.y - cb * Fm.y;
      }
      acc[q] = s;
    }
  }
  __syncthreads();
  double2* r = fft_lines(acc, T, ny, fp.logny, nl, fp.twy, true);
  for (int q = threadIdx.x; q < npts; q += blockDim.x) {
    const int line = q / ny, y = q - line * ny;
    const int kx = pair0 + (line >> 1);
    const bool self = (kx == 0 || 2 * kx == nx);
    if ((line & 1) && self) continue;
    const int col = (line & 1) ? ((nx - kx) & (nx - 1)) : kx;
    fp.Q[((long long)c * nx + col) * ny + y] = r[q];
  }
}

// Dynamic shared-memory limits of the FFT kernels, set once per device (the
// attribute belongs to the device's context).
static void set_smem_once() {
  static PerDevice<bool> done;
  done.get([] {
    cudaFuncSetAttribute(rows_fwd_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * FFT_PTS * 16);
    cudaFuncSetAttribute(rows_fwd_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * FFT_PTS * 16);
    cudaFuncSetAttribute(rows_inv_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * FFT_PTS * 16);
    cudaFuncSetAttribute(rows_inv_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * FFT_PTS * 16);
    cudaFuncSetAttribute(cols_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 6 * FFT_PTS * 16);
    cudaFuncSetAttribute(cols_rules_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 6 * FFT_PTS * 16);
    cudaFuncSetAttribute(cols_rules_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 6 * FFT_PTS * 16);
    cudaFuncSetAttribute(cols_adj_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 6 * FFT_PTS * 16);
    cudaFuncSetAttribute(cols_adj_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 6 * FFT_PTS * 16);
    return true;
  });
}

// batch sizes: rows per block (nb) so a block holds ~1024 points, column
// pairs per block (ppb) so there are enough blocks for every SM; shared
// memory sized to the batch
struct FFTLaunch {
  int ppb, lg;                   // lg: ghost layers per inverse batch in cols
  int threads, threads3;         // cols: one output layer, three
  size_t smem_cols, smem_cols3;
  int layers;                    // cols of all planes in one launch: blocks per column batch (gridDim.z) ...
  int lgz, threadsz;             // ... and theirs
  size_t smemz;
};

// Threads of a block with `lines` lines of n points: one per radix-4 butterfly
// of a stage, so that every warp has FP64 work; where the launch's blocks leave
// SMs with one or two of them, one per point, so that loading, the multipliers
// and storing are one pass each instead of four serial ones.
static int line_threads(long long blocks, int lines, int n) {
  const int per = blocks <= 2LL * sm_count() ? 1 : 4;
  const int t = (lines * n / per + 31) / 32 * 32;
  return t < 32 ? 32 : (t > 256 ? 256 : t);
}

static FFTLaunch fft_launch(const FFTPlan& fp, int planes) {
  FFTLaunch l;
  // column pairs per block: up to 256 points, but no more than leaves two
  // blocks for every SM (the FP64 pipes of idle SMs are lost: 64 x 64 planes
  // with four pairs a block ran on 9 SMs, 22 us a launch)
  const int npairs = fp.nx / 2 + 1;
  l.ppb = 256 / fp.ny;
  const int spread = npairs * planes / (2 * sm_count());
  if (l.ppb > spread) l.ppb = spread;
  if (l.ppb < 1) l.ppb = 1;
  l.smem_cols = (size_t)2 * 2 * l.ppb * fp.ny * sizeof(double2);
  // the three ghost layers in one batch while that keeps two column blocks
  // per SM (at most 96 KB), one at a time otherwise (at 1024^2 the batched
  // form, 192 KB and one block per SM, measured 8 % slower)
  l.lg = (size_t)6 * 2 * l.ppb * fp.ny * sizeof(double2) <= (size_t)96 * 1024 ? 3 : 1;
  l.smem_cols3 = (size_t)(l.lg == 3 ? 6 : 3) * 2 * l.ppb * fp.ny * sizeof(double2);
  const long long blocks = (long long)planes * ((npairs + l.ppb - 1) / l.ppb);
  l.threads = line_threads(blocks, 2 * l.ppb, fp.ny);
  l.threads3 = line_threads(blocks, 2 * l.ppb * l.lg, fp.ny);
  // one ghost layer per block while that leaves at most two blocks per SM
  // (FP32 step at 32^3
  // 98.3 -> 97.6 us, FP64 at 64 x 32 x 45 477.8 -> 475.3)
  l.layers = 3 * blocks <= 2LL * sm_count() ? 3 : 1;
  l.lgz = l.layers == 3 ? 1 : l.lg;
  l.threadsz = l.layers == 3 ? line_threads(3 * blocks, 2 * l.ppb, fp.ny) : l.threads3;
  l.smemz = l.layers == 3 ? (size_t)2 * 2 * l.ppb * fp.ny * sizeof(double2) : l.smem_cols3;
  return l;
}

// Row transforms of `planes` planes: lines per block chosen so that the
// blocks spread evenly over the SMs (all blocks of these kernels are resident
// at once and share each SM's FP64 pipe, so the busiest SM sets the time).
struct RowsCfg {
  int nb, threads;
  size_t smem;
};

static RowsCfg rows_cfg(const FFTPlan& fp, int planes) {
  const int nsm = sm_count();
  int nbmax = 1024 / fp.nx;
  if (nbmax < 1) nbmax = 1;
  if (nbmax > fp.ny) nbmax = fp.ny;
  RowsCfg c{nbmax, 0, 0};
  double best = -1.0;
  for (int nb = nbmax; nb >= 1; nb >>= 1) {
    const long long blocks = (long long)planes * (fp.ny / nb);
    const long long per_sm = (blocks + nsm - 1) / nsm;
    const double eff = (double)blocks / (double)(per_sm * nsm);
    if (eff > best + 1e-9) {
      best = eff;
      c.nb = nb;
    }
  }
  c.threads = line_threads((long long)planes * (fp.ny / c.nb), c.nb, fp.nx);
  c.smem = (size_t)2 * c.nb * fp.nx * sizeof(double2);
  return c;
}

bool pfe_one_chain(int nx, int ny) { return nx * ny <= 8192; }

template <typename R>
void launch_pfe(const FFTPlan& fp, const Layout& L, R* f, const StepState* ss, cudaStream_t st,
                const PlaneStreams* ps, bool chained, const GhostRules<R>* rules) {
  set_smem_once();
  const int npairs = fp.nx / 2 + 1;
  const FFTLaunch l = fft_launch(fp, 3);
  // small planes are bound by launches and latency, not by the FP64 pipe: the
  // three planes go as one chain (64 x 64, ten steps: 2.06 -> 1.95 ms; at
  // 128 x 128 three chains are 2 % faster, at 256 x 256 5 %)
  if (!ps || pfe_one_chain(fp.nx, fp.ny)) {
    const RowsCfg rf = rows_cfg(fp, 3), ri = rows_cfg(fp, 9);
    const double* none = nullptr;
    R* nout = nullptr;
    launch_chained(chained, rows_fwd_kernel<R>, dim3(fp.ny / rf.nb, 3), rf.threads, rf.smem, st, fp, L, f, nout, 0, ss,
                   rf.nb, none, none);
    // (at 128 x 128 and above the waiting blocks of the successors cost more
    // than the launches they hide: 17 -> 23 us a kernel)
    const bool small = pfe_one_chain(fp.nx, fp.ny);
    const int ncol = (npairs + l.ppb - 1) / l.ppb;
    if (rules) {
      const int n2 = 2 * (L.nx + 2 * NG) * (L.ny + 2 * NG), per = 3 * l.layers * l.threadsz;
      launch_chained(small, cols_rules_kernel<R>, dim3(ncol + (n2 + per - 1) / per, 3, l.layers), l.threadsz, l.smemz, st,
                     fp, ss, l.ppb, l.lgz, ncol, L, rules->ph, rules->bg, f);
    } else {
      launch_chained(small, cols_kernel, dim3(ncol, 3, l.layers), l.threadsz, l.smemz, st, fp, 0, ss, l.ppb, l.lgz);
    }
    launch_chained(small, rows_inv_kernel<R>, dim3(fp.ny / ri.nb, 3, 3), ri.threads, ri.smem, st, fp, L, f, nout, nout,
                   0, ss, ri.nb, RowsAdd{});
    return;
  }
  // one chain (rows, columns, inverse rows) per packed plane, on its own
  // stream: the chains share no data, and running them side by side fills
  // the SMs' FP64 pipes where one launch's tail would leave them idle
  const RowsCfg rf = rows_cfg(fp, 1), ri = rows_cfg(fp, 3);
  cudaEventRecord(ps->fork, st);
  for (int i = 0; i < 2; ++i) cudaStreamWaitEvent(ps->s[i], ps->fork, 0);
  for (int p = 0; p < 3; ++p) {
    cudaStream_t sp = p == 0 ? st : ps->s[p - 1];
    FFTPlan fq = fp;
    fq.p0 = p;
    rows_fwd_kernel<R><<<dim3(fp.ny / rf.nb, 1), rf.threads, rf.smem, sp>>>(fq, L, f, nullptr, 0, ss, rf.nb,
                                                                            nullptr, nullptr);
    cols_kernel<<<dim3((npairs + l.ppb - 1) / l.ppb, 1), l.threads3, l.smem_cols3, sp>>>(fq, 0, ss, l.ppb, l.lg);
    rows_inv_kernel<R><<<dim3(fp.ny / ri.nb, 1, 3), ri.threads, ri.smem, sp>>>(fq, L, f, nullptr, nullptr, 0, ss,
                                                                              ri.nb, RowsAdd{});
  }
  for (int i = 0; i < 2; ++i) cudaEventRecord(ps->join[i], ps->s[i]);
}

void pfe_join(const PlaneStreams& ps, cudaStream_t st) {
  for (int i = 0; i < 2; ++i) cudaStreamWaitEvent(st, ps.join[i], 0);
}

template <typename R>
void launch_atarget(const FFTPlan& fp, const R* bz, R* axt, R* ayt, cudaStream_t st) {
  set_smem_once();
  Layout L{};
  const FFTLaunch l = fft_launch(fp, 1);
  const int npairs = fp.nx / 2 + 1;
  const RowsCfg r1 = rows_cfg(fp, 1);
  rows_fwd_kernel<R><<<dim3(fp.ny / r1.nb, 1), r1.threads, r1.smem, st>>>(fp, L, nullptr, bz, 1, nullptr, r1.nb,
                                                                          nullptr, nullptr);
  cols_kernel<<<dim3((npairs + l.ppb - 1) / l.ppb, 1), l.threads, l.smem_cols, st>>>(fp, 1, nullptr, l.ppb, 1);
  rows_inv_kernel<R><<<dim3(fp.ny / r1.nb, 1, 1), r1.threads, r1.smem, st>>>(fp, L, nullptr, axt, ayt, 1, nullptr,
                                                                             r1.nb, RowsAdd{});
}

int launch_rotational(const FFTPlan& fp, const double* vx, const double* vy, double* rx, double* ry, bool add,
                      double f_rot, double* part, cudaStream_t st) {
  set_smem_once();
  Layout L{};
  const FFTLaunch l = fft_launch(fp, 1);
  const int npairs = fp.nx / 2 + 1;
  const RowsCfg r1 = rows_cfg(fp, 1);
  rows_fwd_kernel<double><<<dim3(fp.ny / r1.nb, 1), r1.threads, r1.smem, st>>>(fp, L, nullptr, nullptr, 3, nullptr,
                                                                               r1.nb, vx, vy);
  cols_kernel<<<dim3((npairs + l.ppb - 1) / l.ppb, 1), l.threads, l.smem_cols, st>>>(fp, 4, nullptr, l.ppb, 1);
  rows_inv_kernel<double><<<dim3(fp.ny / r1.nb, 1, 1), r1.threads, r1.smem, st>>>(
      fp, L, nullptr, rx, ry, add ? 5 : 1, nullptr, r1.nb, RowsAdd{vx, vy, f_rot, part});
  return fp.ny / r1.nb;
}

// Adjoint of the potential-field ghosts: gbar (adjoint of the ghost-filled
// state) has its A ghost-layer entries mapped back onto the top layer and
// the photosphere; with them the transpose of the pointwise rules (g: the
// ghost-filled forward state).  `fp_adj` is the plan with the 9-plane buffer as P and the
// 3-plane buffer as Q.
template <typename R>
void launch_pfe_adjoint(const FFTPlan& fp_adj, const Layout& L, const GhostRules<R>& rules, const R* g, R* gbar, R dz,
                        const StepState* ss, cudaStream_t st, bool chained) {
  set_smem_once();
  const FFTLaunch l = fft_launch(fp_adj, 3);
  const int npairs = fp_adj.nx / 2 + 1;
  const RowsCfg r9 = rows_cfg(fp_adj, 9), r3 = rows_cfg(fp_adj, 3);
  const double* none = nullptr;
  R* nout = nullptr;
  launch_chained(chained, rows_fwd_kernel<R>, dim3(fp_adj.ny / r9.nb, 9), r9.threads, r9.smem, st, fp_adj, L, gbar, nout,
                 2, ss, r9.nb, none, none);
  // both ends of a column, or one thread for both (nz = 7)
  const int ncol = (npairs + l.ppb - 1) / l.ppb, per = 3 * l.threads3;
  const int ends = (L.nz == 2 * NG + 1 ? 1 : 2) * fp_adj.nx * fp_adj.ny;
  launch_chained(chained, cols_adj_kernel<R>, dim3(ncol + (ends + per - 1) / per, 3), l.threads3, l.smem_cols3, st,
                 fp_adj, ss, l.ppb, l.lg, ncol, L, rules.ph, rules.bg, g, gbar, dz);
  launch_chained(chained, rows_inv_kernel<R>, dim3(fp_adj.ny / r3.nb, 3, 1), r3.threads, r3.smem, st, fp_adj, L, gbar,
                 nout, nout, 2, ss, r3.nb, RowsAdd{});
}

// Transpose of the magnetogram inversion: B_z adjoint (out, [ny][nx]) from
// the FP64 adjoints of A_x, A_y (abx, aby).
template <typename R>
void launch_atarget_adjoint(const FFTPlan& fp, const double* abx, const double* aby, R* out, cudaStream_t st) {
  set_smem_once();
  Layout L{};
  const FFTLaunch l = fft_launch(fp, 1);
  const int npairs = fp.nx / 2 + 1;
  const RowsCfg r1 = rows_cfg(fp, 1);
  rows_fwd_kernel<R><<<dim3(fp.ny / r1.nb, 1), r1.threads, r1.smem, st>>>(fp, L, nullptr, nullptr, 3, nullptr, r1.nb,
                                                                          abx, aby);
  cols_kernel<<<dim3((npairs + l.ppb - 1) / l.ppb, 1), l.threads, l.smem_cols, st>>>(fp, 2, nullptr, l.ppb, 1);
  rows_inv_kernel<R><<<dim3(fp.ny / r1.nb, 1, 1), r1.threads, r1.smem, st>>>(fp, L, nullptr, out, nullptr, 3, nullptr,
                                                                             r1.nb, RowsAdd{});
}

template void launch_pfe_adjoint<float>(const FFTPlan&, const Layout&, const GhostRules<float>&, const float*, float*,
                                        float, const StepState*, cudaStream_t, bool);
template void launch_pfe_adjoint<double>(const FFTPlan&, const Layout&, const GhostRules<double>&, const double*,
                                         double*, double, const StepState*, cudaStream_t, bool);
template void launch_atarget_adjoint<float>(const FFTPlan&, const double*, const double*, float*, cudaStream_t);
template void launch_atarget_adjoint<double>(const FFTPlan&, const double*, const double*, double*, cudaStream_t);
template void launch_pfe<float>(const FFTPlan&, const Layout&, float*, const StepState*, cudaStream_t,
                                const PlaneStreams*, bool, const GhostRules<float>*);
template void launch_pfe<double>(const FFTPlan&, const Layout&, double*, const StepState*, cudaStream_t,
                                 const PlaneStreams*, bool, const GhostRules<double>*);
template void launch_atarget<float>(const FFTPlan&, const float*, float*, float*, cudaStream_t);
template void launch_atarget<double>(const FFTPlan&, const double*, double*, double*, cudaStream_t);

}  // namespace mhd
