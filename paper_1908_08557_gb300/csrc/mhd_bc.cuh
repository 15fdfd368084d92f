// mhd_bc.cuh -- the pointwise ghost rules of one column, for the kernels that
// apply them (mhd_ghost.cu, mhd_fft.cu).
#pragma once
#include "mhd_internal.h"

namespace mhd {

constexpr int BC_TH = 64;  // threads of a block of columns

// Pointwise ghost rules over whole padded planes (rims included, so no rim
// pass is needed afterwards).  In full variables:
//  bottom: ln rho fixed to the initial profile ('fg', Sect. 2.5);
//          ln T from hydrostatic equilibrium downward (Eq. 8 with p = rho T):
//          lnT_j = lnT_{j+1} + lnrho_{j+1} - lnrho_j - dz g_z / T_{j+1};
//          u_z antisymmetric (closed, u_z = 0 at z = 0).
//  top:    ln T symmetric (Eq. 11); ln rho hydrostatic with the boundary
//          temperature (Eq. 13, signed g_z): lnrho_{nz-1+m} = lnrho_{nz-1-m}
//          + 2 m dz g_z / T_{nz-1}; u_z antisymmetric, u_x, u_y symmetric.
// ln rho and ln T are stored as perturbations about the background; the
// background differences enter through the constants cb, ctT, ctL (FP64 on
// the host), and the background ghost values of ln rho equal the fixed
// profile, so their perturbation is zero.
//
// The lower or upper end of column (i, j) on closed boundaries (bc_z = 0).
template <typename R>
__device__ __forceinline__ void ghost_rules(const Layout& L, const Phys<R>& ph, const Background<R>& bg, R* f, int i,
                                            int j, bool top) {
  const int kt = L.nz - 1;
  // (layer distances from the vertical grid: bg.dzb[m] = z_{1-m} - z_{-m},
  // bg.dzt[m] = z_{nz-1+m} - z_{nz-1-m}; dz and 2 m dz on the uniform grid)
  if (!top) {
    R th1 = f[L.at(LT, 0, j, i)];
    R l1 = f[L.at(LR, 0, j, i)];
    R uz[NG];
#pragma unroll
    for (int m = 1; m <= NG; ++m) uz[m - 1] = f[L.at(UZ, m, j, i)];
#pragma unroll
    for (int m = 1; m <= NG; ++m) {
      const R T1 = rexp<R>(bg.tbar[NG - m + 1] + th1);
      const R l0 = R(0);
      const R th0 = th1 + l1 - l0 + bg.cb[m] - bg.dzb[m] * ph.gz / T1;
      f[L.at(LR, -m, j, i)] = l0;
      f[L.at(LT, -m, j, i)] = th0;
      f[L.at(UZ, -m, j, i)] = -uz[m - 1];
      th1 = th0;
      l1 = l0;
    }
    return;
  }
  R v[NG][5];
#pragma unroll
  for (int m = 1; m <= NG; ++m)
#pragma unroll
    for (int c = 0; c < 5; ++c) v[m - 1][c] = f[L.at(UX + c, kt - m, j, i)];
  const R Ttop = rexp<R>(bg.tbar[NG + kt] + f[L.at(LT, kt, j, i)]);
#pragma unroll
  for (int m = 1; m <= NG; ++m) {
    f[L.at(LT, kt + m, j, i)] = v[m - 1][LT - UX] + bg.ctT[m];
    f[L.at(LR, kt + m, j, i)] = v[m - 1][LR - UX] + bg.ctL[m] + bg.dzt[m] * ph.gz / Ttop;
    f[L.at(UZ, kt + m, j, i)] = -v[m - 1][UZ - UX];
    f[L.at(UX, kt + m, j, i)] = v[m - 1][0];
    f[L.at(UY, kt + m, j, i)] = v[m - 1][1];
  }
}

// Transpose of the rules (one column, interior x, y): ghost adjoints are routed
// into the layers they were computed from.  Bound by latency, as the rules
// themselves: the two ends of a column are separate threads, and each loads all
// it needs before it computes.  nz >= 7, so the layers the two ends write
// (k <= 3 and k >= nz - 4) are disjoint but for the middle one of seven, whose
// u_z both touch: that box takes one thread for both ends.
template <typename R>
__device__ __forceinline__ void adj_ghost_rules(const Layout& L, const Phys<R>& ph, const Background<R>& bg, const R* g,
                                                R* gbar, R dz, int i, int j, bool bottom, bool top) {
  const int kt = L.nz - 1;
  const R dzg = dz * ph.gz;
  // bottom: ln T recursion (ln rho ghosts are constants)
  if (bottom) {
    R th[NG], at[NG + 1], uz[NG], gz[NG];
#pragma unroll
    for (int m = 0; m < NG; ++m) {
      th[m] = bg.tbar[NG - m] + g[L.at(LT, -m, j, i)];
      uz[m] = gbar[L.at(UZ, m + 1, j, i)];
      gz[m] = gbar[L.at(UZ, -m - 1, j, i)];
    }
#pragma unroll
    for (int m = 0; m <= NG; ++m) at[m] = gbar[L.at(LT, -m, j, i)];
    const R al = gbar[L.at(LR, 0, j, i)];
    const R a2 = at[2] + at[3] * (R(1) + dzg * rexp<R>(-th[2]));
    const R a1 = at[1] + a2 * (R(1) + dzg * rexp<R>(-th[1]));
    gbar[L.at(LT, 0, j, i)] = at[0] + a1 * (R(1) + dzg * rexp<R>(-th[0]));
    gbar[L.at(LR, 0, j, i)] = al + a1;
#pragma unroll
    for (int m = 0; m < NG; ++m) gbar[L.at(UZ, m + 1, j, i)] = uz[m] - gz[m];
  }
  // top
  if (top) {
    R in[NG][5], gh[NG][5];
#pragma unroll
    for (int m = 1; m <= NG; ++m)
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        in[m - 1][c] = gbar[L.at(UX + c, kt - m, j, i)];
        gh[m - 1][c] = gbar[L.at(UX + c, kt + m, j, i)];
      }
    const R at = gbar[L.at(LT, kt, j, i)];
    const R Ttop = rexp<R>(bg.tbar[NG + kt] + g[L.at(LT, kt, j, i)]);
    R bth = R(0);
#pragma unroll
    for (int m = 1; m <= NG; ++m) {
      const R bl = gh[m - 1][LR - UX];
      gbar[L.at(LT, kt - m, j, i)] = in[m - 1][LT - UX] + gh[m - 1][LT - UX];
      gbar[L.at(LR, kt - m, j, i)] = in[m - 1][LR - UX] + bl;
      bth -= bl * (R(2 * m) * dz) * ph.gz / Ttop;
      gbar[L.at(UZ, kt - m, j, i)] = in[m - 1][UZ - UX] - gh[m - 1][UZ - UX];
      gbar[L.at(UX, kt - m, j, i)] = in[m - 1][0] + gh[m - 1][0];
      gbar[L.at(UY, kt - m, j, i)] = in[m - 1][1] + gh[m - 1][1];
    }
    gbar[L.at(LT, kt, j, i)] = at + bth;
  }
}

}  // namespace mhd
