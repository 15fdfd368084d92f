// mhd_rk64.cu -- FP64 right-hand side + RK3 update, and the FP64 pointwise
// adjoint, forming every first derivative once.
//
// What bounds it: the FP64 pipe.  An SM retires two FP64 operations per clock
// (a warp instruction holds its scheduler's share of the pipe for 64 clocks),
// so loads, index arithmetic and shared memory are nearly free and only the
// count of FP64 operations matters, and how evenly they lie on the SMs.  The
// mixed derivatives D1_a D1_b dominate a cell-by-cell evaluation: as product
// stencils they cost 36 operations each, twelve of them 432 of 1022 per cell.
// Here a mixed derivative is one more first difference (5 operations) of a
// first difference that some cell has already taken:
//  - z mixed: the x and y differences that the grad-div terms need (six sources
//    of A and u) are formed by each cell for its own plane and handed along z
//    through shared memory; the three planes at each end of the block's layers
//    are formed once per block;
//  - xy mixed: the y differences of A_x, A_y, u_x, u_y of the row with an x halo
//    pass through a scratch of the warp.
// Weights: the differences are taken in units of their smallest weight,
//   d f  = (f_3 - f_-3) - 9 (f_2 - f_-2) + 45 (f_1 - f_-1)       (D1 = d / 60 h)
//   dd f = (f_3 + f_-3) - 13.5 (f_2 + f_-2) + 135 (f_1 + f_-1) - 245 f
//                                                                (D2 = dd / 90 h^2)
// which saves a multiplication per difference; the scales enter the
// multiply-adds that consume them.  545 FP64 instructions per cell in all (1022 cell by
// cell).
//
// A block is one row of 32 cells over KZ = 8 layers, a warp per layer: a single
// barrier, and work in pieces small enough to spread over the SMs (a z-march
// of the same arithmetic, a ring of sources per column, leaves one warp per
// scheduler in small boxes, where dependent FP64 operations take 114 clocks
// each instead of 64).  Neighbours come through L1 from the padded state.
//
// Measured (GB300, a launch): 256 x 256 x 128 16.5 -> 8.9 ms against the
// cell-by-cell kernel (mhd_rk.cu), 32^3 93 -> 55 us; the FP64 pipe is active
// 85 % of the time at 128^3.
#include "mhd_adjoint_point.cuh"
#include "mhd_internal.h"

namespace mhd {
namespace r64 {

constexpr int TX = 32, KZ = 8, NT = TX * KZ;
constexpr int NSRC = 6;          // z-mixed sources: dxAz, dyAz, div_h A, dxUz, dyUz, div_h u
constexpr int NAUX = 3;          // kept by the cell itself: dyAy, D1x u_x, D1y u_y
constexpr int SW = TX + 8;       // scratch row: x0 - 3 .. x0 + TX + 2, padded
constexpr int NSC = 4;           // scratch fields: dy of A_y, A_x, u_y, u_x

// Products of the scheme constants, formed on the host: a uniform product
// costs every thread an FP64 operation as any other does.  c*: D1 scales
// 1 / 60 h and their products, e*: D2 scales 1 / 90 h^2, v*: times nu (1, 1/3
// or 4/3 of it); the z entries are replaced per layer on a non-uniform grid.
struct Coef64 {
  double cx, cy, cz, cxy, cxz, cyz, ex, ey, ez;
  double v1ex, v1ey, v1ez, v4ex, v4ey, v4ez, v3cx, v3cxy, v3cxz, v3cyz, v3cz;
  double heat, visc, cond;  // (gamma - 1) eta, (gamma - 1) nu, (gamma - 1) kappa0
};

struct Args {
  Layout L;
  Coef64 c;
  Phys<double> ph;
  Background<double> bg;
  const double* fin;
  double* fout;
  double* df;
  const double* wtab;
  const double* wptab;
  const double* axt;
  const double* ayt;
  const double* v0;
  const double* v1;
  const StepState* ss;
  int sub;
  // adjoint mode
  const double* dbar;
  double* coef;
  double* thbar;
};

__device__ __forceinline__ double comb1(double a1, double b1, double a2, double b2, double a3, double b3) {
  return fma(45.0, a1 - b1, fma(-9.0, a2 - b2, a3 - b3));
}
__device__ __forceinline__ double comb2(double c, double a1, double b1, double a2, double b2, double a3, double b3) {
  return fma(-245.0, c, fma(135.0, a1 + b1, fma(-13.5, a2 + b2, a3 + b3)));
}
// first difference along stride s; first and second
template <typename I>
__device__ __forceinline__ double dd1(const double* p, I s) {
  return comb1(p[s], p[-s], p[2 * s], p[-2 * s], p[3 * s], p[-3 * s]);
}
template <typename I>
__device__ __forceinline__ double dd12(const double* p, I s, double c, double& d2) {
  const double a1 = p[s], b1 = p[-s], a2 = p[2 * s], b2 = p[-2 * s],
               a3 = p[3 * s], b3 = p[-3 * s];
  d2 = comb2(c, a1, b1, a2, b2, a3, b3);
  return comb1(a1, b1, a2, b2, a3, b3);
}
template <typename I>
__device__ __forceinline__ double dd2(const double* p, I s, double c) {
  return comb2(c, p[s], p[-s], p[2 * s], p[-2 * s], p[3 * s],
               p[-3 * s]);
}
__device__ __forceinline__ double ds1(const double* p) {
  return comb1(p[1], p[-1], p[2], p[-2], p[3], p[-3]);
}

__device__ __forceinline__ void put_images(const Layout& L, double* f, int fl, int k, int j, int i,
                                           double v) {
  int xs[3], ys[3], nxs = 1, nys = 1;
  xs[0] = i;
  ys[0] = j;
  if (i < NG) xs[nxs++] = i + L.nx;
  if (i >= L.nx - NG) xs[nxs++] = i - L.nx;
  if (j < NG) ys[nys++] = j + L.ny;
  if (j >= L.ny - NG) ys[nys++] = j - L.ny;
  for (int b = 0; b < nys; ++b)
    for (int a = 0; a < nxs; ++a) f[L.at(fl, k, ys[b], xs[a])] = v;
}

// ADJ = false: right-hand side + RK update of substep `sub` (sub < 0: the
// right-hand side alone into df); ADJ = true: the pointwise adjoint.  ZG: a
// non-uniform vertical grid, D_z f = m1 D_xi f, D_z^2 f = m1^2 D_xi^2 f + r21 D_z f.
template <bool ADJ, bool ZG>
__global__ void __launch_bounds__(NT, 2) rk64_kernel(const __grid_constant__ Args a) {
  __shared__ double src[KZ + 2 * NG][NSRC][TX];
  __shared__ double scr_all[KZ][NSC][SW];
  chain_enter();
  if (halted(a.ss)) return;
  const Layout& L = a.L;
  const Phys<double>& ph = a.ph;
  const int tx = threadIdx.x, w_ = threadIdx.y;
  const int x0 = blockIdx.x * TX;
  const int i = x0 + tx, j = blockIdx.y, k0 = blockIdx.z * KZ, k = k0 + w_;
  const bool live = i < L.nx && k < L.nz;
  const bool near = i < L.nx + NG && k < L.nz;  // its y differences are read by live threads
  const int sy = L.mx, sz = L.mx * L.my;
  const long long fs = L.fs;
  const Coef64& C = a.c;

  const int sub = a.sub;
  const bool eval = sub < 0;
  const double dt = eval ? 1.0 : a.ss->dt;
  const double alpha = eval ? 0.0 : rk_alpha(sub);
  const double beta = eval ? 0.0 : rk_beta(sub);

  // sources of plane p at this column, into n (z-mixed) and e (kept for the centre)
  auto front = [&](int p, double (&n)[NSRC], double (&e)[NAUX]) {
    const double* q = a.fin + L.at(0, p, j, i);
    n[0] = dd1(q + AZ * fs, 1);
    n[1] = dd1(q + AZ * fs, sy);
    e[0] = dd1(q + AY * fs, sy);
    n[2] = fma(C.cx, dd1(q + AX * fs, 1), C.cy * e[0]);
    n[3] = dd1(q + UZ * fs, 1);
    n[4] = dd1(q + UZ * fs, sy);
    e[1] = C.cx * dd1(q + UX * fs, 1);
    e[2] = C.cy * dd1(q + UY * fs, sy);
    n[5] = e[1] + e[2];
  };
  const long long n2 = (long long)L.nx * L.ny, n3 = n2 * L.nz;
  double cur[NSRC], ax_[NAUX];
  if (i < L.nx) {
    // this layer's sources (a layer above the top is a neighbour's source
    // only), and one of the six planes beyond the block's layers per warp
    if (k < L.nz + NG) {
      front(k, cur, ax_);
#pragma unroll
      for (int q = 0; q < NSRC; ++q) src[w_ + NG][q][tx] = cur[q];
    }
    const int ps = w_ < NG ? w_ : KZ + w_;  // slot of the extra plane (w_ < 2 NG)
    if (w_ < 2 * NG && k0 - NG + ps < L.nz + NG) {
      double n[NSRC], e[NAUX];
      front(k0 - NG + ps, n, e);
#pragma unroll
      for (int q = 0; q < NSRC; ++q) src[ps][q][tx] = n[q];
    }
  }
  {
    const double* f = a.fin + L.at(0, k, j, i);
    double* scr = &scr_all[w_][0][0];
    // y differences of A_y, A_x, u_y, u_x of the row, with the x halo
    double dyAx = 0.0, yyAx = 0.0, dyUx = 0.0, yyUx = 0.0;
    if (near) {
      const double ca = f[AX * fs], cu = f[UX * fs];
      dyAx = dd12(f + AX * fs, sy, ca, yyAx);
      dyUx = dd12(f + UX * fs, sy, cu, yyUx);
      double* sc = scr + tx + NG;
      sc[1 * SW] = dyAx;
      sc[3 * SW] = dyUx;
      sc[0] = live ? ax_[0] : dd1(f + AY * fs, sy);
      sc[2 * SW] = live ? ax_[2] : C.cy * dd1(f + UY * fs, sy);
    }
    if (tx < NSC * 2 * NG && k < L.nz) {
      const int hf = tx / (2 * NG), hq = tx - hf * 2 * NG, hc = hq < NG ? hq - NG : TX + hq - NG;
      if (x0 + hc < L.nx + NG) {
        const int fld = hf == 0 ? AY : (hf == 1 ? AX : (hf == 2 ? UY : UX));
        const double v = dd1(a.fin + L.at(fld, k, j, x0 + hc), sy);
        scr[hf * SW + hc + NG] = hf == 2 ? C.cy * v : v;
      }
    }
    __syncthreads();
    if (live) {
      double mz[NSRC];
#pragma unroll
      for (int q = 0; q < NSRC; ++q)
        mz[q] = comb1(src[w_ + 4][q][tx], src[w_ + 2][q][tx], src[w_ + 5][q][tx], src[w_ + 1][q][tx],
                      src[w_ + 6][q][tx], src[w_][q][tx]);
      const double* sc = scr + tx + NG;
      double cz = C.cz, ez = C.ez, cxz = C.cxz, cyz = C.cyz, v1ez = C.v1ez, v4ez = C.v4ez, v3cxz = C.v3cxz,
             v3cyz = C.v3cyz, v3cz = C.v3cz, r21 = 0.0;
      if constexpr (ZG) {
        const double m1 = a.bg.zm1[k], m2 = m1 * m1;  // the host's entries are those of unit spacing
        r21 = a.bg.zr21[k];
        cz *= m1; cxz *= m1; cyz *= m1; v3cxz *= m1; v3cyz *= m1; v3cz *= m1;
        ez *= m2; v1ez *= m2; v4ez *= m2;
      }
      const double w = a.wtab[k], wp = a.wptab[k];
      const bool swamp = !ADJ && (w != 0.0 || wp != 0.0);
      // ---- A: B = curl A + B_ext, J = grad div A - lap A (the own-axis
      // second derivatives cancel), swamp terms
      double A0, A1, B[3], J[3], sw[3] = {0.0, 0.0, 0.0};
      {
        const double *pa = f + AX * fs, *pb = f + AY * fs, *pc = f + AZ * fs;
        A0 = *pa;
        A1 = *pb;
        const double A2 = *pc;
        double zz;
        double dzA = dd12(pa, sz, A0, zz);
        B[1] = fma(cz, dzA, fma(-C.cx, cur[0], ph.bext[1]));
        J[0] = fma(C.cxy, ds1(sc), fma(cxz, mz[0], fma(-C.ey, yyAx, -ez * zz)));
        if constexpr (ZG) J[0] = fma(-r21 * cz, dzA, J[0]);
        double l0 = 0.0, l1 = 0.0, l2 = 0.0, dv = 0.0;
        if (swamp) {
          l0 = fma(C.ex, dd2(pa, 1, A0), fma(C.ey, yyAx, ez * zz));
          if constexpr (ZG) l0 = fma(r21 * cz, dzA, l0);
        }
        double xx;
        const double dxA = dd12(pb, 1, A1, xx);
        dzA = dd12(pb, sz, A1, zz);
        B[0] = fma(-cz, dzA, fma(C.cy, cur[1], ph.bext[0]));
        B[2] = fma(C.cx, dxA, fma(-C.cy, dyAx, ph.bext[2]));
        J[1] = fma(C.cxy, ds1(sc + 1 * SW), fma(cyz, mz[1], fma(-C.ex, xx, -ez * zz)));
        if constexpr (ZG) J[1] = fma(-r21 * cz, dzA, J[1]);
        if (swamp) {
          l1 = fma(C.ex, xx, fma(C.ey, dd2(pb, sy, A1), ez * zz));
          if constexpr (ZG) l1 = fma(r21 * cz, dzA, l1);
        }
        xx = dd2(pc, 1, A2);
        const double yy = dd2(pc, sy, A2);
        J[2] = fma(cz, mz[2], fma(-C.ex, xx, -C.ey * yy));
        if (swamp) {
          dzA = dd12(pc, sz, A2, zz);
          l2 = fma(C.ex, xx, fma(C.ey, yy, ez * zz));
          if constexpr (ZG) l2 = fma(r21 * cz, dzA, l2);
          dv = fma(cz, dzA, cur[2]);
          const double ews = ph.eta_s * w;
          if (a.bg.bB && k >= a.bg.ksw) {
            const long long ns = n2 * (L.nz - a.bg.ksw), qs = (long long)(k - a.bg.ksw) * n2 + (long long)j * L.nx + i;
            l0 += a.bg.bL[qs];
            l1 += a.bg.bL[ns + qs];
            l2 += a.bg.bL[2 * ns + qs];
            dv += a.bg.bL[3 * ns + qs];
          }
          sw[0] = ews * l0;
          sw[1] = ews * l1;
          sw[2] = fma(ews, l2, ph.eta_s * wp * dv);
        }
        if (a.bg.bB) {
          // A stored about a background: its B and J
          const long long q3 = (long long)k * n2 + (long long)j * L.nx + i;
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            B[c] += a.bg.bB[c * n3 + q3];
            J[c] += a.bg.bJ[c * n3 + q3];
          }
        }
      }
      // ---- u: dU[c][a] = d_a u_c, and nu (lap u + grad div u / 3)
      double u[3], dU[3][3], vis[3] = {0.0, 0.0, 0.0};
      {
        const double *pa = f + UX * fs, *pb = f + UY * fs, *pc = f + UZ * fs;
        u[0] = *pa;
        u[1] = *pb;
        u[2] = *pc;
        dU[0][0] = ax_[1];
        dU[0][1] = C.cy * dyUx;
        dU[1][1] = ax_[2];
        dU[2][0] = C.cx * cur[3];
        dU[2][1] = C.cy * cur[4];
        if constexpr (ADJ) {
          dU[0][2] = cz * dd1(pa, sz);
          dU[1][0] = C.cx * dd1(pb, 1);
          dU[1][2] = cz * dd1(pb, sz);
          dU[2][2] = cz * dd1(pc, sz);
        } else {
          double xx, zz;
          dU[0][2] = cz * dd12(pa, sz, u[0], zz);
          // the scratch holds D1y u_y already scaled (field 2), d_y u_x not (field 3)
          vis[0] = fma(C.v4ex, dd2(pa, 1, u[0]),
                       fma(C.v1ey, yyUx, fma(v1ez, zz, fma(C.v3cx, ds1(sc + 2 * SW), v3cxz * mz[3]))));
          dU[1][0] = C.cx * dd12(pb, 1, u[1], xx);
          dU[1][2] = cz * dd12(pb, sz, u[1], zz);
          vis[1] = fma(C.v1ex, xx,
                       fma(C.v4ey, dd2(pb, sy, u[1]), fma(v1ez, zz, fma(C.v3cxy, ds1(sc + 3 * SW), v3cyz * mz[4]))));
          dU[2][2] = cz * dd12(pc, sz, u[2], zz);
          vis[2] = fma(C.v1ex, dd2(pc, 1, u[2]), fma(C.v1ey, dd2(pc, sy, u[2]), fma(v4ez, zz, v3cz * mz[5])));
          if constexpr (ZG) {
            vis[0] = fma(ph.nu * r21, dU[0][2], vis[0]);
            vis[1] = fma(ph.nu * r21, dU[1][2], vis[1]);
            vis[2] = fma((4.0 / 3.0) * ph.nu * r21, dU[2][2], vis[2]);
          }
        }
      }
      // ---- ln rho, ln T: stored perturbation + background
      double lr, th, gL[3], gT[3], lapL = 0.0, lapT;
      {
        const double* p = f + LR * fs;
        const double c = *p;
        lr = a.bg.lbar[k + NG] + c;
        if constexpr (ADJ) {
          gL[0] = C.cx * dd1(p, 1);
          gL[1] = C.cy * dd1(p, sy);
          gL[2] = fma(cz, dd1(p, sz), a.bg.dl[k]);
        } else {
          double xx, yy, zz;
          gL[0] = C.cx * dd12(p, 1, c, xx);
          gL[1] = C.cy * dd12(p, sy, c, yy);
          const double dz = dd12(p, sz, c, zz);
          gL[2] = fma(cz, dz, a.bg.dl[k]);
          lapL = fma(C.ex, xx, fma(C.ey, yy, fma(ez, zz, a.bg.d2l[k])));
          if constexpr (ZG) lapL = fma(r21 * cz, dz, lapL);
        }
      }
      {
        const double* p = f + LT * fs;
        const double c = *p;
        th = a.bg.tbar[k + NG] + c;
        double xx, yy, zz;
        gT[0] = C.cx * dd12(p, 1, c, xx);
        gT[1] = C.cy * dd12(p, sy, c, yy);
        const double dz = dd12(p, sz, c, zz);
        gT[2] = fma(cz, dz, a.bg.dt[k]);
        lapT = fma(C.ex, xx, fma(C.ey, yy, fma(ez, zz, a.bg.d2t[k])));
        if constexpr (ZG) lapT = fma(r21 * cz, dz, lapT);
      }

      if constexpr (ADJ) {
        // the cell record the pointwise transpose reads: J as grad div A with
        // lap A = 0 (only their difference enters), no second derivative of u
        Cell<double> c;
        c.A[0] = A0; c.A[1] = A1; c.A[2] = 0.0;
        c.L = lr;
        c.Th = th;
        c.dA[0][0] = c.dA[1][1] = c.dA[2][2] = 0.0;
        c.dA[2][1] = B[0] - ph.bext[0]; c.dA[1][2] = 0.0;
        c.dA[0][2] = B[1] - ph.bext[1]; c.dA[2][0] = 0.0;
        c.dA[1][0] = B[2] - ph.bext[2]; c.dA[0][1] = 0.0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          c.U[q] = u[q];
          c.gdA[q] = J[q];
          c.lapA[q] = c.lapU[q] = c.gdU[q] = 0.0;
          c.gL[q] = gL[q];
          c.gT[q] = gT[q];
#pragma unroll
          for (int b = 0; b < 3; ++b) c.dU[q][b] = dU[q][b];
        }
        c.lapL = 0.0;
        c.lapT = lapT;
        double wo[NF];
#pragma unroll
        for (int fl = 0; fl < NF; ++fl) wo[fl] = dt * a.dbar[L.at(fl, k, j, i)];
        const long long q2 = (long long)j * L.nx + i;
        double cf[NCOEF];
        adjoint_cell<double>(c, ph, w, wp, wo, dt, k, L.nz, a.dbar + L.at(UX, 0, j, i), a.dbar + L.at(UY, 0, j, i),
                             L.sz(), a.thbar, q2, n2, a.ss, sub, cf);
        if (k < ph.nc_k1) nc_adjoint<double>(ph, a.bg, L.nz, k, lr, th, wo[LT], cf);
        coef_swamp_part<double>(ph, w, wo, cf);
        double* co = a.coef + (long long)k * n2 + q2;
#pragma unroll
        for (int q = 0; q < NCOEF; ++q)
          if (coef_always(q) || (coef_swamp(q) && k >= a.bg.ksw)) co[q * n3] = cf[q];
      } else {
        const double T = exp(th), rho1 = exp(-lr);
        double out[NF];
        out[0] = fma(u[1], B[2], fma(-u[2], B[1], fma(-ph.eta, J[0], sw[0])));
        out[1] = fma(u[2], B[0], fma(-u[0], B[2], fma(-ph.eta, J[1], sw[1])));
        out[2] = fma(u[0], B[1], fma(-u[1], B[0], fma(-ph.eta, J[2], sw[2])));
        // traceless rate of strain, off-diagonal entries doubled (t_ab = 2 S_ab)
        const double div = ax_[1] + ax_[2] + dU[2][2], d3 = -(1.0 / 3.0) * div;
        const double s00 = dU[0][0] + d3, s11 = dU[1][1] + d3, s22 = dU[2][2] + d3;
        const double t01 = dU[0][1] + dU[1][0], t02 = dU[0][2] + dU[2][0], t12 = dU[1][2] + dU[2][1];
        // 2 S:S and 2 S . grad ln rho
        const double S2 = fma(t01, t01, fma(t02, t02, fma(t12, t12, 2.0 * fma(s00, s00, fma(s11, s11, s22 * s22)))));
        const double h0 = 2.0 * gL[0], h1 = 2.0 * gL[1], h2 = 2.0 * gL[2];
        const double g0 = fma(s00, h0, fma(t01, gL[1], t02 * gL[2]));
        const double g1 = fma(s11, h1, fma(t01, gL[0], t12 * gL[2]));
        const double g2 = fma(s22, h2, fma(t02, gL[0], t12 * gL[1]));
        const double F0 = fma(J[1], B[2], -(J[2] * B[1])), F1 = fma(J[2], B[0], -(J[0] * B[2])),
                     F2 = fma(J[0], B[1], -(J[1] * B[0]));
        out[3] = fma(F0, rho1, fma(ph.nu, g0, vis[0]));
        out[4] = fma(F1, rho1, fma(ph.nu, g1, vis[1]));
        out[5] = fma(F2, rho1, fma(ph.nu, g2, vis[2]));
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const double adv = fma(u[0], dU[c][0], fma(u[1], dU[c][1], u[2] * dU[c][2]));
          // pressure and gravity cancel in hydrostatic balance: their
          // difference is formed before the smaller terms join it
          const double hyd = fma(-T, gL[c] + gT[c], c == 2 ? ph.gz : 0.0);
          out[3 + c] += hyd - adv;
        }
        const double ugL = fma(u[0], gL[0], fma(u[1], gL[1], u[2] * gL[2]));
        const double gLs = fma(gL[0], gL[0], fma(gL[1], gL[1], gL[2] * gL[2]));
        out[6] = fma(ph.drho, gLs + lapL, -(ugL + div));
        if (swamp) out[6] = fma(ph.drho_s * w, lapL, out[6]);
        const double ugT = fma(u[0], gT[0], fma(u[1], gT[1], u[2] * gT[2]));
        const double gTs = fma(gT[0], gT[0], fma(gT[1], gT[1], gT[2] * gT[2]));
        const double JJ = fma(J[0], J[0], fma(J[1], J[1], J[2] * J[2]));
        // 1 / T and kappa0 T^{5/2} / rho from one reciprocal square root
        const double rs = rsqrt(T);
        const double heat = fma(C.heat * JJ, rho1, C.visc * S2) * (rs * rs);
        const double kt = C.cond * rho1 * (T * T * T * rs);
        double diff = lapT * kt;
        if (swamp) diff = fma(ph.chi_s * w, lapT, diff);
        out[7] = fma(3.5 * kt, gTs, diff) + (heat - fma(ph.gm1, div, ugT));
        if (k < ph.nc_k1) out[LT] += nc_term<double>(ph, a.bg, L.nz, k, lr, th, nullptr, nullptr);

        double tgx = 0.0, tgy = 0.0;
        if (ph.bcz == 0 && k == 0) {
          const double r = eval ? a.ss->eval_r : a.ss->r[sub], s = eval ? a.ss->eval_s : a.ss->s[sub];
          const long long q2 = (long long)j * L.nx + i;
          tgx = r * fma(s, a.v1[q2] - a.v0[q2], a.v0[q2]);
          tgy = r * fma(s, a.v1[n2 + q2] - a.v0[n2 + q2], a.v0[n2 + q2]);
          // photospheric rows: nudging of A_hor (Sect. 2.1) and u_hor (Eq. 5);
          // ln rho held at its initial profile and u_z = 0 (Sect. 2.5)
          out[AX] -= ph.tau_A * (A0 - a.axt[q2]);
          out[AY] -= ph.tau_A * (A1 - a.ayt[q2]);
          out[UX] -= ph.tau_u * (u[0] - tgx);
          out[UY] -= ph.tau_u * (u[1] - tgy);
          out[UZ] = 0.0;
          out[LR] = 0.0;
        }
        if (ph.bcz == 0 && k == L.nz - 1) out[UZ] = 0.0;  // closed top (Sect. 4)

        const bool edge = i < NG || i >= L.nx - NG || j < NG || j >= L.ny - NG;
        const long long q0 = L.at(0, k, j, i);
#pragma unroll
        for (int fl = 0; fl < NF; ++fl) {
          const long long q = q0 + fl * fs;
          const double dfn = sub > 0 ? fma(alpha, a.df[q], dt * out[fl]) : dt * out[fl];
          if (sub < 2) a.df[q] = dfn;
          if (!eval) {
            const double v = fma(beta, dfn, f[fl * fs]);
            if (edge) put_images(L, a.fout, fl, k, j, i, v);
            else a.fout[q] = v;
          }
        }
        if (ph.bcz == 0 && k == 0) {
          // stateful u_x, u_y ghost rows below the photosphere: nudging only
          for (int m = 1; m <= NG; ++m) {
#pragma unroll
            for (int cc = 0; cc < 2; ++cc) {
              const long long q = L.at(UX + cc, -m, j, i);
              const double ug = a.fin[q];
              const double rh = -ph.tau_u * (ug - (cc == 0 ? tgx : tgy));
              const double dfn = sub > 0 ? fma(alpha, a.df[q], dt * rh) : dt * rh;
              if (sub < 2) a.df[q] = dfn;
              if (!eval) put_images(L, a.fout, UX + cc, -m, j, i, fma(beta, dfn, ug));
            }
          }
        }
      }
    }
  }
}

static dim3 grid64(const Layout& L) { return dim3((L.nx + TX - 1) / TX, L.ny, (L.nz + KZ - 1) / KZ); }

// (the kernels' shared-memory limit is raised once per device)
static size_t spread64(bool chained, dim3 g) {
  static PerDevice<bool> done;
  done.get([] {
    cudaFuncSetAttribute(rk64_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ONE_PER_SM_BYTES);
    cudaFuncSetAttribute(rk64_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ONE_PER_SM_BYTES);
    cudaFuncSetAttribute(rk64_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ONE_PER_SM_BYTES);
    return true;
  });
  return one_per_sm(chained, g);
}

static Coef64 coef64(const Phys<double>& ph, bool zg) {
  Coef64 c;
  c.cx = ph.idx / 60.0;
  c.cy = ph.idy / 60.0;
  c.cz = (zg ? 1.0 : ph.idz) / 60.0;
  c.cxy = c.cx * c.cy;
  c.cxz = c.cx * c.cz;
  c.cyz = c.cy * c.cz;
  c.ex = ph.idx2 / 90.0;
  c.ey = ph.idy2 / 90.0;
  c.ez = (zg ? 1.0 : ph.idz2) / 90.0;
  c.v1ex = ph.nu * c.ex;
  c.v1ey = ph.nu * c.ey;
  c.v1ez = ph.nu * c.ez;
  c.v4ex = c.v1ex * 4.0 / 3.0;
  c.v4ey = c.v1ey * 4.0 / 3.0;
  c.v4ez = c.v1ez * 4.0 / 3.0;
  c.v3cx = ph.nu * c.cx / 3.0;
  c.v3cxy = ph.nu * c.cxy / 3.0;
  c.v3cxz = ph.nu * c.cxz / 3.0;
  c.v3cyz = ph.nu * c.cyz / 3.0;
  c.v3cz = ph.nu * c.cz / 3.0;
  c.heat = ph.gm1 * ph.eta;
  c.visc = ph.gm1 * ph.nu;
  c.cond = ph.gm1 * ph.kappa0;
  return c;
}

}  // namespace r64

void launch_rk64(const Layout& L, const Phys<double>& ph, const Background<double>& bg, const double* fin,
                 double* fout, double* df, const double* wtab, const double* wptab, const Driver& drv,
                 const StepState* ss, int sub, cudaStream_t st, bool chained) {
  r64::Args a{};
  a.L = L;
  a.ph = ph;
  a.bg = bg;
  a.fin = fin;
  a.fout = fout;
  a.df = df;
  a.wtab = wtab;
  a.wptab = wptab;
  a.axt = (const double*)drv.axt;
  a.ayt = (const double*)drv.ayt;
  a.v0 = (const double*)drv.v0;
  a.v1 = (const double*)drv.v1;
  a.ss = ss;
  a.sub = sub;
  const bool zg = bg.zm1 != nullptr;
  a.c = r64::coef64(ph, zg);
  const dim3 g = r64::grid64(L), b(r64::TX, r64::KZ);
  const size_t smem = r64::spread64(chained, g);
  if (zg) launch_chained(chained, r64::rk64_kernel<false, true>, g, b, smem, st, a);
  else launch_chained(chained, r64::rk64_kernel<false, false>, g, b, smem, st, a);
}

void launch_adj_point64(const Layout& L, const Phys<double>& ph, const Background<double>& bg, const double* gst,
                        const double* dbar, double* coef, double* thbar, const double* wtab, const double* wptab,
                        const StepState* ss, int sub, cudaStream_t st, bool chained) {
  r64::Args a{};
  a.L = L;
  a.ph = ph;
  a.bg = bg;
  a.fin = gst;
  a.wtab = wtab;
  a.wptab = wptab;
  a.ss = ss;
  a.sub = sub;
  a.dbar = dbar;
  a.coef = coef;
  a.thbar = thbar;
  a.c = r64::coef64(ph, false);
  const dim3 g = r64::grid64(L);
  launch_chained(chained, r64::rk64_kernel<true, false>, g, dim3(r64::TX, r64::KZ), r64::spread64(chained, g), st, a);
}

}  // namespace mhd
