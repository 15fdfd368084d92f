// mhd_adj_gather64.cu -- the transposed-stencil gather of the adjoint
// right-hand side in FP64 (see mhd_adj_gather_zm.cu for the sums it forms from
// the coefficient fields).
//
// What bounds it: the FP64 pipe (two operations per clock and SM), so the
// count of operations and their spread over the SMs matter, and the loads, all
// straight from the coefficient fields through L1, do not.  A block is one row
// of 32 cells over KZ = 8 output layers of one output group, a warp per layer.
// Each warp forms, for its own plane, the three inputs of D1z^T that mix
// in-plane differences (of bJ or of the Laplacian coefficients) and hands them
// along z through shared memory; six of the warps also do one of the planes
// beyond the block's layers.  Differences are taken in units of their smallest
// weight (60 h D1, 90 h^2 D2), the scales enter the multiply-adds that consume
// them.  About 400 operations per cell for both groups (the z-march before it
// scattered 600 in FP64 and put a 64 x 32 x 45 box on 48 SMs: 527 us a launch).
#include "mhd_adjoint_point.cuh"
#include "mhd_internal.h"

namespace mhd {
namespace g64 {

constexpr int TX = 32, KZ = 8, NT = TX * KZ;
constexpr int SW = TX + 8;  // scratch row: columns -3 .. TX + 2, padded

struct Args {
  Layout L;
  const double* coef;
  double* dbar;
  double* gbar;
  double* fbar;
  double alpha, beta;
  int klo, khi, ksw, bcz;
  double tau_A, tau_u;
  // D1 scales 1 / 60 h and their products, D2 scales 1 / 90 h^2 (host-formed)
  double cx, cy, cz, cxy, ex, ey, ez;
  const StepState* ss;
};

__device__ __forceinline__ double comb1(double a1, double b1, double a2, double b2, double a3, double b3) {
  return fma(45.0, a1 - b1, fma(-9.0, a2 - b2, a3 - b3));
}
__device__ __forceinline__ double comb2(double c, double a1, double b1, double a2, double b2, double a3, double b3) {
  return fma(-245.0, c, fma(135.0, a1 + b1, fma(-13.5, a2 + b2, a3 + b3)));
}

// group 0: A_x, A_y, A_z, ln rho; group 1: u_x, u_y, u_z, ln T (blockIdx.z odd)
template <int GRP>
__device__ __forceinline__ void gather(const Args& a, double (*tz)[3][TX], double (*scr)[SW], int k0) {
  const Layout& L = a.L;
  const int tx = threadIdx.x, w = threadIdx.y;
  const int nx = L.nx, ny = L.ny, nz = L.nz, n2 = nx * ny;
  const long long n3 = (long long)n2 * nz;
  const int x0 = blockIdx.x * TX, i = x0 + tx, j = blockIdx.y;
  const int k = k0 + w;                       // output plane, -3 .. nz + 2
  const bool in = k >= 0 && k < nz;           // a coefficient plane too
  const bool col = i < nx;
  // periodic neighbours (nx, ny powers of two) as offsets from the cell
  int xo[7], yo[7];
  const int ic = i & (nx - 1);
#pragma unroll
  for (int m = -3; m <= 3; ++m) {
    xo[m + 3] = ((i + m) & (nx - 1)) - ic;
    yo[m + 3] = (((j + m) & (ny - 1)) - j) * nx;
  }
  auto P = [&](int q, int p) { return a.coef + q * n3 + (long long)p * n2 + (long long)j * nx + ic; };
  auto d1 = [&](const double* p, const int (&o)[7]) {
    return comb1(p[o[4]], p[o[2]], p[o[5]], p[o[1]], p[o[6]], p[o[0]]);
  };
  auto d2 = [&](const double* p, const int (&o)[7]) {
    return comb2(p[0], p[o[4]], p[o[2]], p[o[5]], p[o[1]], p[o[6]],
                 p[o[0]]);
  };
  constexpr int QX = GRP == 0 ? CGA : CLU, QY = QX + 1, QZ = QX + 2;  // bJ, or the Laplacian coefficients of u
  constexpr double g = GRP == 0 ? 1.0 : 1.0 / 3.0;
  // inputs of D1z^T (times 60 dz) at plane p; yQ: d_y of QY there
  auto tin = [&](int p, double& yQ, double (&t)[3]) {
    yQ = d1(P(QY, p), yo);
    const double xq = d1(P(QZ, p), xo), yq = d1(P(QZ, p), yo), dv = fma(a.cx, d1(P(QX, p), xo), a.cy * yQ);
    if (GRP == 0) {
      t[0] = fma(-a.cx, xq, *P(CDA + 2, p));
      t[1] = -fma(a.cy, yq, *P(CDA + 7, p));
      t[2] = p >= a.ksw ? *P(CDA, p) - dv : -dv;
    } else {
      t[0] = fma(-g * a.cx, xq, *P(CDU + 2, p));
      t[1] = fma(-g * a.cy, yq, *P(CDU + 5, p));
      t[2] = fma(-g, dv, *P(CDU + 8, p));
    }
  };
  double yQ = 0.0;
  if (col) {
    double t[3] = {0.0, 0.0, 0.0};
    if (in) tin(k, yQ, t);
#pragma unroll
    for (int c = 0; c < 3; ++c) tz[w + NG][c][tx] = t[c];
    if (w < 2 * NG) {
      const int s = w < NG ? w : KZ + w, p = k0 - NG + s;
      double e[3] = {0.0, 0.0, 0.0}, y;
      if (p >= 0 && p < nz) tin(p, y, e);
#pragma unroll
      for (int c = 0; c < 3; ++c) tz[s][c][tx] = e[c];
    }
  }
  // d_y of QX and QY along the row, with an x halo
  if (in) {
    if (i < nx + NG) {
      scr[0][tx + NG] = d1(P(QX, k), yo);
      scr[1][tx + NG] = col ? yQ : d1(P(QY, k), yo);
    }
    if (tx < 4 * NG) {
      const int f = tx / (2 * NG), h = tx - f * 2 * NG, hc = h < NG ? h - NG : TX + h - NG;
      const double* p = a.coef + (f == 0 ? QX : QY) * n3 + (long long)k * n2 + (long long)j * nx +
                        ((x0 + hc) & (nx - 1));
      scr[f][hc + NG] = d1(p, yo);
    }
  }
  __syncthreads();
  if (!col || k >= nz + NG) return;
  double v[4];
  // z parts: D1z^T of the shared inputs, D2z of fields read along the column
#pragma unroll
  for (int c = 0; c < 3; ++c)
    v[c] = -a.cz * comb1(tz[w + 4][c][tx], tz[w + 2][c][tx], tz[w + 5][c][tx], tz[w + 1][c][tx], tz[w + 6][c][tx],
                         tz[w][c][tx]);
  auto zcol = [&](int q, int m) {  // coefficient q at plane k + m, zero outside
    const int p = k + m;
    return p >= 0 && p < nz ? *P(q, p) : 0.0;
  };
  auto zz = [&](int q) {
    return comb2(zcol(q, 0), zcol(q, 1), zcol(q, -1), zcol(q, 2), zcol(q, -2), zcol(q, 3), zcol(q, -3));
  };
  constexpr int QG = GRP == 0 ? CGL : CGT, QL = GRP == 0 ? CLL : CLT, QV = CV + (GRP == 0 ? LR : LT);
  v[3] = fma(-a.cz, comb1(zcol(QG + 2, 1), zcol(QG + 2, -1), zcol(QG + 2, 2), zcol(QG + 2, -2), zcol(QG + 2, 3),
                          zcol(QG + 2, -3)), a.ez * zz(QL));
  if (GRP == 0) {
    v[0] = fma(-a.ez, zz(QX), v[0]);
    v[1] = fma(-a.ez, zz(QY), v[1]);
    if (k + NG >= a.ksw) {
      // the swamp's own Laplacian coefficients live on layers k >= ksw only
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        auto sc = [&](int m) {
          const int p = k + m;
          return p >= a.ksw && p < nz ? *P(CLA + c, p) : 0.0;
        };
        v[c] = fma(a.ez, comb2(sc(0), sc(1), sc(-1), sc(2), sc(-2), sc(3), sc(-3)), v[c]);
      }
    }
  } else {
    v[0] = fma(a.ez, zz(QX), v[0]);
    v[1] = fma(a.ez, zz(QY), v[1]);
    v[2] = fma(a.ez * (4.0 / 3.0), zz(QZ), v[2]);
  }
  if (in) {
    const double* s = &scr[0][tx + NG];
    const double xyX = comb1(s[1], s[-1], s[2], s[-2], s[3], s[-3]);
    s = &scr[1][tx + NG];
    const double xyY = comb1(s[1], s[-1], s[2], s[-2], s[3], s[-3]);
    if (GRP == 0) {
      const double *b0 = P(CDA + 7, k), *b1 = P(CDA + 2, k), *b2 = P(CDA + 3, k);
      v[0] += fma(a.cxy, xyY, fma(a.cy, d1(b2, yo), -a.ey * d2(P(QX, k), yo)));
      v[1] += fma(a.cxy, xyX, fma(-a.cx, d1(b2, xo), -a.ex * d2(P(QY, k), xo)));
      v[2] += fma(a.cx, d1(b1, xo), fma(-a.cy, d1(b0, yo), fma(-a.ex, d2(P(QZ, k), xo), -a.ey * d2(P(QZ, k), yo))));
      if (k >= a.ksw) {
        v[0] = fma(-a.cx, d1(P(CDA, k), xo), v[0]);
        v[1] = fma(-a.cy, d1(P(CDA, k), yo), v[1]);
#pragma unroll
        for (int c = 0; c < 3; ++c) v[c] = fma(a.ex, d2(P(CLA + c, k), xo), fma(a.ey, d2(P(CLA + c, k), yo), v[c]));
      }
    } else {
      const double f43 = 4.0 / 3.0;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double wx = c == 0 ? f43 * a.ex : a.ex, wy = c == 1 ? f43 * a.ey : a.ey;
        v[c] += fma(wx, d2(P(QX + c, k), xo), fma(wy, d2(P(QX + c, k), yo),
                fma(-a.cx, d1(P(CDU + 3 * c, k), xo), fma(-a.cy, d1(P(CDU + 3 * c + 1, k), yo),
                                                          *P(CV + UX + c, k)))));
      }
      v[0] = fma(g * a.cxy, xyY, v[0]);
      v[1] = fma(g * a.cxy, xyX, v[1]);
    }
    v[3] += fma(a.ex, d2(P(QL, k), xo), fma(a.ey, d2(P(QL, k), yo),
            fma(-a.cx, d1(P(QG, k), xo), fma(-a.cy, d1(P(QG + 1, k), yo), *P(QV, k)))));
  }
  // the substep's update, or G with the nudging's value adjoints
  const bool fz = k >= a.klo && k < a.khi;
  const double dt = a.ss->dt;
  const long long q0 = L.at(0, k, j, i);
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int f = GRP == 0 ? (t < 3 ? AX + t : LR) : (t < 3 ? UX + t : LT);
    const long long q = q0 + (long long)f * L.fs;
    if (fz) {
      const double fv = a.fbar[q] + v[t];
      a.fbar[q] = fv;
      a.dbar[q] = fma(a.alpha, a.dbar[q], a.beta * fv);
    } else {
      double gv = v[t];
      if (a.bcz == 0 && ((k == 0 && (f == AX || f == AY)) || (k < 0 && (f == UX || f == UY))))
        gv = fma(-(f == AX || f == AY ? a.tau_A : a.tau_u) * dt, a.dbar[q], gv);
      a.gbar[q] = gv;
    }
  }
}

__global__ void __launch_bounds__(NT, 2) gather64_kernel(const __grid_constant__ Args a) {
  __shared__ double tz[KZ + 2 * NG][3][TX];
  __shared__ double scr[KZ][2][SW];
  chain_enter();
  if (halted(a.ss)) return;
  const int k0 = (int)(blockIdx.z >> 1) * KZ - NG;
  if (blockIdx.z & 1) gather<1>(a, tz, scr[threadIdx.y], k0);
  else gather<0>(a, tz, scr[threadIdx.y], k0);
}

}  // namespace g64

void launch_adj_gather64(const Layout& L, const Phys<double>& ph, const double* coef, double* dbar, double* gbar,
                         double* fbar, double alpha, double beta, int klo, int khi, int ksw, const StepState* ss,
                         cudaStream_t st, bool chained) {
  g64::Args a;
  a.L = L;
  a.coef = coef;
  a.dbar = dbar;
  a.gbar = gbar;
  a.fbar = fbar;
  a.alpha = alpha;
  a.beta = beta;
  a.klo = klo;
  a.khi = khi;
  a.ksw = ksw;
  a.bcz = ph.bcz;
  a.tau_A = ph.tau_A;
  a.tau_u = ph.tau_u;
  a.cx = ph.idx / 60.0;
  a.cy = ph.idy / 60.0;
  a.cz = ph.idz / 60.0;
  a.cxy = a.cx * a.cy;
  a.ex = ph.idx2 / 90.0;
  a.ey = ph.idy2 / 90.0;
  a.ez = ph.idz2 / 90.0;
  a.ss = ss;
  const dim3 grid((L.nx + g64::TX - 1) / g64::TX, L.ny, 2 * ((L.nz + 2 * NG + g64::KZ - 1) / g64::KZ));
  launch_chained(chained, g64::gather64_kernel, grid, dim3(g64::TX, g64::KZ), 0, st, a);
}

}  // namespace mhd
