// mhd_adj_gather_zm.cu -- the transposed-stencil gather of the adjoint right-
// hand side as a z-march.
//
// Given the coefficient fields h of a substep (the adjoints of the cell values
// and of every derivative the right-hand side read, [q][nz][ny][nx], in the
// reduced set of coef_always), the adjoint of the ghost-filled input is, per
// output field,
//   sum over first-derivative coefficients   D1_a^T h = -D1_a h,
//   + Laplacian coefficients                  (D2x + D2y + D2z) h,
//   + gradient-of-divergence coefficients     D2_a h (own axis) and
//                                             D1_a D1_c h (c != a, symmetric),
//   + value coefficients (u, ln rho, ln T),
// periodic in x and y, zero outside the interior layers, evaluated on the
// interior and the three z ghost layers on each side.  For A the first
// derivatives add up to -curl bB and the second ones to (grad div - lap) bJ, in
// which the own-axis second derivatives cancel; the swamp layers add
// lap (eta_s w dt D_A) and -grad bdivA.
//
// A CTA (128 threads, two x-adjacent cells each in packed f32x2) owns a 32 x 8
// tile and one output group -- {A_x, A_y, A_z, ln rho} or {u_x, u_y, u_z, ln T}
// -- and marches over the coefficient planes p of a z chunk.  The fields of
// plane p whose in-plane stencils the group takes (9 and 12 of them, with a
// 3-cell x, y halo, wrapped periodically) are staged in shared memory by
// cp.async in 16-byte chunks, one plane ahead; of the ones read at the cell
// alone (2 and 8) each thread copies its own pair along.  In-plane terms go
// to the output at plane p; the z terms are first combined into one input of
// D1z^T and one of D2z per output and scattered from the cell's column:
// h(p) contributes to outputs p - 3 .. p + 3, held in a 7-plane accumulator
// ring per output field in registers.  When plane p is done, output plane
// p - 3 is complete and is written.  The in-plane mixed terms D1x D1y use the
// commuted form D1x(D1y h) through a scratch row with an x halo.
//
// Measured: a taped adjoint step at 256^3 (three of these launches and the point
// kernel's) 6.52 ms with all 40 coefficients and the centre-only ones loaded
// into registers as they were needed, 5.41 ms as it stands.
//
// Output: on layers klo <= k < khi the substep's update F += G,
// D = alpha D + beta F; elsewhere G into gbar, with the value adjoints of the
// photospheric nudging (A_x, A_y at k = 0, Eq. 4) and of the stateful u_x, u_y
// ghost rows (Eq. 5).
#include "mhd_adjoint_point.cuh"
#include "mhd_internal.h"
#include "mhd_pair.cuh"
#include "mhd_zmarch.cuh"

namespace mhd {
namespace gzm {

using namespace pk;

constexpr int TX = 32, TY = 8;
constexpr int XO = 4;                 // staged rows start 4 columns left of the tile
constexpr int SX = TX + 8, SY = TY + 6;
constexpr int SP = SX * SY;           // elements of one staged field plane
constexpr int NO = 4;                 // output fields of a group
constexpr int NT = TX / 2 * TY;       // 128 threads
constexpr int CP = SX / 4 * SY;       // 16-byte chunks of a staged field plane (140)
constexpr int NH = 12;                // staged fields, at most (group 1; group 0 stages 9)
constexpr int NC = 8;                 // centre-only fields, at most (group 1; group 0 reads 2)
constexpr int NB = 2;                 // plane buffers: one in flight while one is used (three, with two in
                                      // flight and less L1 beside them, take 7 % longer at 256^3)
constexpr int PL = NH * SP + NC * 2 * NT;  // floats per plane buffer: staged planes, then the threads' own pairs
constexpr size_t SMEM = (size_t)NB * PL * 4 + (size_t)4 * TY * SX * 4;

// staged slots
enum { B0 = 0, B1, B2, J0, J1, J2, G0, G1, LL };                             // group 0
enum { UX0 = 0, UY0, UX1, UY1, UX2, UY2, L0, L1, L2, T0, T1, TT };           // group 1: d_x, d_y of u_c; nu D; ...
// centre-only slots
enum { VL = 0, GL2 };                                                        // group 0
enum { UZ0 = 0, UZ1, UZ2, V0, V1, V2, VT, GT2 };                             // group 1
__host__ __device__ constexpr int nstage(int grp) { return grp == 0 ? 9 : 12; }
__host__ __device__ constexpr int ncentre(int grp) { return grp == 0 ? 2 : 8; }
__host__ __device__ constexpr int qstage(int grp, int s) {
  constexpr int a[9] = {CDA + 7, CDA + 2, CDA + 3, CGA, CGA + 1, CGA + 2, CGL, CGL + 1, CLL};
  constexpr int u[12] = {CDU, CDU + 1, CDU + 3, CDU + 4, CDU + 6, CDU + 7, CLU, CLU + 1, CLU + 2, CGT, CGT + 1, CLT};
  return grp == 0 ? a[s] : u[s];
}
__host__ __device__ constexpr int qcentre(int grp, int s) {
  constexpr int a[2] = {CV + LR, CGL + 2};
  constexpr int u[8] = {CDU + 2, CDU + 5, CDU + 8, CV + UX, CV + UY, CV + UZ, CV + LT, CGT + 2};
  return grp == 0 ? a[s] : u[s];
}

struct Args {
  Layout L;
  Phys<float> ph;
  const float* coef;
  float* dbar;
  float* gbar;
  float* fbar;
  float alpha, beta;
  int klo, khi, ksw;
  StepState* ss;
  int ntx, nty, nch, kchunk;
  Coef cx, cy;  // D1, D2 weights over dx, dy
  int dyn;      // items claimed from the step state's counter (else grid stride)
};

// z scatters into a 7-plane ring (index 3 = the current plane)
__device__ __forceinline__ void zs_d1t(f2 (&a)[7], f2 v) {  // D1z^T: +c_m h into p + m, -c_m h into p - m
  a[4] = fma2(F2(W<float>::c1), v, a[4]); a[2] = fma2(F2(-W<float>::c1), v, a[2]);
  a[5] = fma2(F2(W<float>::c2), v, a[5]); a[1] = fma2(F2(-W<float>::c2), v, a[1]);
  a[6] = fma2(F2(W<float>::c3), v, a[6]); a[0] = fma2(F2(-W<float>::c3), v, a[0]);
}
__device__ __forceinline__ void zs_d2(f2 (&a)[7], f2 v) {  // D2z (symmetric)
  a[3] = fma2(F2(W<float>::e0), v, a[3]);
  a[4] = fma2(F2(W<float>::e1), v, a[4]); a[2] = fma2(F2(W<float>::e1), v, a[2]);
  a[5] = fma2(F2(W<float>::e2), v, a[5]); a[1] = fma2(F2(W<float>::e2), v, a[1]);
  a[6] = fma2(F2(W<float>::e3), v, a[6]); a[0] = fma2(F2(W<float>::e3), v, a[0]);
}
__device__ __forceinline__ f2 dxx(const float* p, const Coef& c) {
  f2 d1, d2;
  dx_pair(p, c, d1, &d2);
  return d2;
}
__device__ __forceinline__ f2 dyy(const float* p, const Coef& c) {
  f2 d1, d2;
  ds_pair(p, SX, c, d1, &d2);
  return d2;
}
__device__ __forceinline__ f2 dx1(const float* p, const Coef& c) {
  f2 d1;
  dx_pair(p, c, d1, nullptr);
  return d1;
}
__device__ __forceinline__ f2 dy1(const float* p, const Coef& c) {
  f2 d1;
  ds_pair(p, SX, c, d1, nullptr);
  return d1;
}

// The swamp layers' own terms at the pair (i, j) of plane p: per component the
// in-plane Laplacian of s_c = eta_s w dt D_c and its value for D2z, and the
// divergence term's -D1x, -D1y and value.  A few layers of a box, so the
// neighbours are read straight from memory, one cell after the other (nx, ny
// powers of two).
__device__ __noinline__ void swamp_pair(const Args& a, int p, int j, int i, f2 (&in)[3], f2 (&s)[3], f2& dv) {
  const int nx = a.L.nx, ny = a.L.ny;
  const long long n2 = (long long)nx * ny, n3 = n2 * a.L.nz;
  const float* base = a.coef + (long long)p * n2;
  auto at = [&](int q, int jj, int ii) { return base[q * n3 + (long long)(jj & (ny - 1)) * nx + (ii & (nx - 1))]; };
  const float c1[4] = {0.f, W<float>::c1, W<float>::c2, W<float>::c3};
  const float e[4] = {W<float>::e0, W<float>::e1, W<float>::e2, W<float>::e3};
  float r[3][2], v[3][2], d[2];
  for (int t = 0; t < 2; ++t) {
    const int x = i + t;
    float gx = 0.f, gy = 0.f;
    for (int c = 0; c < 3; ++c) {
      v[c][t] = at(CLA + c, j, x);
      float lx = e[0] * v[c][t], ly = lx;
      for (int m = 1; m <= 3; ++m) {
        lx += e[m] * (at(CLA + c, j, x + m) + at(CLA + c, j, x - m));
        ly += e[m] * (at(CLA + c, j + m, x) + at(CLA + c, j - m, x));
      }
      r[c][t] = a.ph.idx2 * lx + a.ph.idy2 * ly;
    }
    for (int m = 1; m <= 3; ++m) {
      gx += c1[m] * (at(CDA, j, x + m) - at(CDA, j, x - m));
      gy += c1[m] * (at(CDA, j + m, x) - at(CDA, j - m, x));
    }
    r[0][t] -= a.ph.idx * gx;
    r[1][t] -= a.ph.idy * gy;
    d[t] = at(CDA, j, x);
  }
  for (int c = 0; c < 3; ++c) {
    in[c] = make_float2(r[c][0], r[c][1]);
    s[c] = make_float2(v[c][0], v[c][1]);
  }
  dv = make_float2(d[0], d[1]);
}

// One item: output group GRP of a tile over output planes [n0, n1).
template <int GRP>
__device__ __forceinline__ void item_pair(const Args& a, float* buf, float* scrb, int x0, int y0, int n0, int n1) {
  const Layout& L = a.L;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int nx = L.nx, ny = L.ny, nz = L.nz;
  const long long n2 = (long long)nx * ny, n3 = n2 * nz;
  const Phys<float>& ph = a.ph;
  const f2 idz = F2(ph.idz), idz2 = F2(ph.idz2);
  const float dt = (float)a.ss->dt;
  const int e = 2 * tx + XO;
  const int cen = (ty + 3) * SX + e;
  const int pa = max(0, n0 - NG), pb = min(nz - 1, n1 + NG - 1);  // valid input planes
  auto chunk_off = [&](int c) -> long long {
    if (c >= CP) return 0;
    const int r = c / (SX / 4), cc = c - r * (SX / 4);
    const int yy = ((y0 - 3 + r) % ny + ny) % ny, xx = ((x0 - XO + cc * 4) % nx + nx) % nx;
    return (long long)yy * nx + xx;
  };
  const long long off0 = chunk_off(tid), off1 = chunk_off(tid + NT);
  auto cp16 = [](float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(zm::sa(dst)), "l"(src) : "memory");
  };
  auto cp8 = [](float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(zm::sa(dst)), "l"(src) : "memory");
  };
  const int i = x0 + 2 * tx, j = y0 + ty;
  const bool live = i < nx && j < ny;
  const long long qc = (long long)j * nx + i;  // the pair's offset within a plane
  // planes past pb commit an empty group, so that the wait below is the same
  // for every plane
  auto stage = [&](int p, int bb) {
    if (p <= pb) {
      float* dst = buf + bb * PL;
      const float* src = a.coef + (long long)p * n2;
      // the field stride is hidden from the compiler, which would otherwise
      // keep the addresses of all fields in registers across the planes
      long long fs = n3;
      asm volatile("" : "+l"(fs));
#pragma unroll
      for (int s = 0; s < nstage(GRP); ++s) {
        const float* f = src + qstage(GRP, s) * fs;
        cp16(dst + s * SP + tid * 4, f + off0);
        if (tid + NT < CP) cp16(dst + s * SP + (tid + NT) * 4, f + off1);
      }
      if (live) {
#pragma unroll
        for (int s = 0; s < ncentre(GRP); ++s)
          cp8(dst + NH * SP + (s * NT + tid) * 2, src + qcentre(GRP, s) * fs + qc);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int q = 0; q < NB - 1; ++q) stage(pa + q, q);
  int b = 0;
  f2 acc[NO][7];
#pragma unroll
  for (int t = 0; t < NO; ++t)
#pragma unroll
    for (int d = 0; d < 7; ++d) acc[t][d] = F2(0.f);
  // x-halo pairs of the in-plane mixed scratch: 2 fields x 8 rows x 4 pairs
  const int hf = tid >> 5, hr = (tid & 31) >> 2, hx = (tid & 3) < 2 ? 2 * (tid & 3) : 32 + 2 * (tid & 3);
  const Coef& cx = a.cx;
  const Coef& cy = a.cy;

  for (int p = n0 - NG; p <= n1 + NG - 1; ++p) {
    // output plane p - 3 is written at the end of this plane: its accumulator
    // and D values are fetched now, ahead of the compute
    const int n = p - NG;
    const bool emit = n >= n0 && live;
    const bool fz = n >= a.klo && n < a.khi;
    f2 fo[NO], dd[NO];
    long long qo = 0;
    if (emit) qo = L.at(0, n, j, i);
#pragma unroll
    for (int t = 0; t < NO; ++t) {
      const int f = GRP == 0 ? (t < 3 ? AX + t : LR) : (t < 3 ? UX + t : LT);
      const long long q = qo + (long long)f * L.fs;
      fo[t] = (emit && fz) ? ld2(a.fbar + q) : F2(0.f);
      dd[t] = (emit && (fz || (ph.bcz == 0 && n <= 0))) ? ld2(a.dbar + q) : F2(0.f);
    }
    if (p >= pa && p <= pb) {
      stage(p + NB - 1, b == 0 ? NB - 1 : b - 1);
      asm volatile("cp.async.wait_group %0;" ::"n"(NB - 1) : "memory");
      __syncthreads();
      const float* s = buf + b * PL;
      auto S = [&](int q) { return s + q * SP + cen; };
      auto C = [&](int q) { return ld2(s + NH * SP + (q * NT + tid) * 2); };
      float* scr = scrb + ((p - pa) & 1) * 2 * TY * SX;
      auto scratch = [&](f2 v0, f2 v1, int s0, int s1) {
        // D1y of two fields on the tile's rows, with the x halo
        *reinterpret_cast<f2*>(scr + ty * SX + e) = v0;
        *reinterpret_cast<f2*>(scr + TY * SX + ty * SX + e) = v1;
        if (tid < 64)
          *reinterpret_cast<f2*>(scr + hf * TY * SX + hr * SX + hx) =
              dy1(s + (hf == 0 ? s0 : s1) * SP + (hr + 3) * SX + hx, cy);
      };
      if constexpr (GRP == 0) {
        const f2 yJ0 = dy1(S(J0), cy), yJ1 = dy1(S(J1), cy);
        scratch(yJ0, yJ1, J0, J1);
        // -curl bB, and (grad div - lap) bJ without its cancelling parts
        f2 d1, d2;
        acc[0][3] = add(acc[0][3], dif(dy1(S(B2), cy), dyy(S(J0), cy)));
        acc[1][3] = dif(acc[1][3], add(dx1(S(B2), cx), dxx(S(J1), cx)));
        acc[2][3] = add(acc[2][3], dif(dx1(S(B1), cx), dy1(S(B0), cy)));
        dx_pair(S(J2), cx, d1, &d2);
        zs_d1t(acc[0], mul(idz, dif(ld2(S(B1)), d1)));
        f2 e1, e2;
        ds_pair(S(J2), SX, cy, e1, &e2);
        acc[2][3] = dif(acc[2][3], add(d2, e2));
        zs_d1t(acc[1], mul(mul(idz, F2(-1.f)), add(ld2(S(B0)), e1)));
        f2 t2 = mul(F2(-1.f), add(dx1(S(J0), cx), yJ1));
        f2 s0 = mul(F2(-1.f), ld2(S(J0))), s1 = mul(F2(-1.f), ld2(S(J1)));
        if (p >= a.ksw && live) {
          f2 in[3], sv[3], dv;
          swamp_pair(a, p, j, i, in, sv, dv);
#pragma unroll
          for (int c = 0; c < 3; ++c) acc[c][3] = add(acc[c][3], in[c]);
          s0 = add(s0, sv[0]);
          s1 = add(s1, sv[1]);
          zs_d2(acc[2], mul(idz2, sv[2]));
          t2 = add(t2, dv);
        }
        zs_d1t(acc[2], mul(idz, t2));
        zs_d2(acc[0], mul(idz2, s0));
        zs_d2(acc[1], mul(idz2, s1));
        // ln rho: value, -D1x, -D1y, D1z^T, Laplacian
        dx_pair(S(LL), cx, d1, &d2);
        acc[3][3] = add(acc[3][3], dif(add(C(VL), add(d2, dyy(S(LL), cy))), add(dx1(S(G0), cx), dy1(S(G1), cy))));
        zs_d1t(acc[3], mul(idz, C(GL2)));
        zs_d2(acc[3], mul(idz2, ld2(S(LL))));
      } else {
        // grad div u enters as a third of the Laplacian's coefficients: own-axis
        // second derivatives get 4/3, the mixed ones 1/3
        const f2 third = F2(1.f / 3.f), f43 = F2(4.f / 3.f);
        const f2 yL0 = dy1(S(L0), cy);
        f2 yL1, yyL1;
        ds_pair(S(L1), SX, cy, yL1, &yyL1);
        scratch(yL0, yL1, L0, L1);
        f2 d1, d2, e1, e2;
        dx_pair(S(L0), cx, d1, &d2);
        acc[0][3] = add(acc[0][3], fma2(f43, d2, add(dyy(S(L0), cy), dif(C(V0), add(dx1(S(UX0), cx), dy1(S(UY0), cy))))));
        zs_d1t(acc[2], mul(idz, dif(C(UZ2), mul(third, add(d1, yL1)))));
        zs_d2(acc[0], mul(idz2, ld2(S(L0))));
        acc[1][3] = add(acc[1][3], fma2(f43, yyL1, add(dxx(S(L1), cx), dif(C(V1), add(dx1(S(UX1), cx), dy1(S(UY1), cy))))));
        zs_d2(acc[1], mul(idz2, ld2(S(L1))));
        dx_pair(S(L2), cx, d1, &d2);
        ds_pair(S(L2), SX, cy, e1, &e2);
        acc[2][3] = add(acc[2][3], add(add(d2, e2), dif(C(V2), add(dx1(S(UX2), cx), dy1(S(UY2), cy)))));
        zs_d1t(acc[0], mul(idz, dif(C(UZ0), mul(third, d1))));
        zs_d1t(acc[1], mul(idz, dif(C(UZ1), mul(third, e1))));
        zs_d2(acc[2], mul(mul(idz2, f43), ld2(S(L2))));
        // ln T: value, -D1x, -D1y, D1z^T, Laplacian
        dx_pair(S(TT), cx, d1, &d2);
        acc[3][3] = add(acc[3][3], dif(add(C(VT), add(d2, dyy(S(TT), cy))), add(dx1(S(T0), cx), dy1(S(T1), cy))));
        zs_d1t(acc[3], mul(idz, C(GT2)));
        zs_d2(acc[3], mul(idz2, ld2(S(TT))));
      }
      __syncthreads();
      // xy mixed: D1x(D1y h_x) -> y, D1x(D1y h_y) -> x
      const f2 g = F2(GRP == 0 ? 1.f : 1.f / 3.f);
      acc[1][3] = fma2(g, dx1(scr + ty * SX + e, cx), acc[1][3]);
      acc[0][3] = fma2(g, dx1(scr + TY * SX + ty * SX + e, cx), acc[0][3]);
      b = b == NB - 1 ? 0 : b + 1;
    }
    if (emit) {
#pragma unroll
      for (int t = 0; t < NO; ++t) {
        const int f = GRP == 0 ? (t < 3 ? AX + t : LR) : (t < 3 ? UX + t : LT);
        const long long q = qo + (long long)f * L.fs;
        const f2 v = acc[t][0];
        if (fz) {
          const f2 fv = add(fo[t], v);
          *reinterpret_cast<f2*>(a.fbar + q) = fv;
          *reinterpret_cast<f2*>(a.dbar + q) = fma2(F2(a.alpha), dd[t], mul(F2(a.beta), fv));
        } else {
          f2 gv = v;
          if (ph.bcz == 0 && ((n == 0 && (f == AX || f == AY)) || (n < 0 && (f == UX || f == UY))))
            gv = dif(gv, mul(F2((f == AX || f == AY ? ph.tau_A : ph.tau_u) * dt), dd[t]));
          *reinterpret_cast<f2*>(a.gbar + q) = gv;
        }
      }
    }
#pragma unroll
    for (int t = 0; t < NO; ++t) {
#pragma unroll
      for (int d = 0; d < 6; ++d) acc[t][d] = acc[t][d + 1];
      acc[t][6] = F2(0.f);
    }
  }
}

__global__ void __launch_bounds__(NT, 2) gather_pair_kernel(const __grid_constant__ Args a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* buf = reinterpret_cast<float*>(smem_raw);
  float* scr = buf + NB * PL;
  chain_enter();
  if (halted(a.ss)) return;
  const int nzo = a.L.nz + 2 * NG;
  const int tiles = a.ntx * a.nty;
  const int nitems = tiles * a.nch * 2;
  // items group-major within a z chunk: the CTAs running together hold all
  // tiles of one output group, whose halo planes they share in L2.  With
  // several items per CTA (dyn) each CTA claims its next item from the step
  // state's counter as it starts one (the claim is handed to the CTA at the
  // end-of-item barrier), so that CTAs meeting dearer items (the x, y edges'
  // wrapped halos, the update layers) do not hold up the launch.
  __shared__ int s_next;
  if (a.dyn) {
    if (threadIdx.x == 0) s_next = atomicAdd(&a.ss->items, 1);
    __syncthreads();
  }
  for (int item = a.dyn ? s_next : (int)blockIdx.x; item < nitems;) {
    int next = 0;
    if (a.dyn && threadIdx.x == 0) next = atomicAdd(&a.ss->items, 1);
    const int ch = item / (2 * tiles), r = item - ch * 2 * tiles;
    const int grp = r >= tiles ? 1 : 0;
    const int tile = r - grp * tiles;
    const int x0 = (tile % a.ntx) * TX, y0 = (tile / a.ntx) * TY;
    const int n0 = ch * a.kchunk - NG, n1 = min(nzo, (ch + 1) * a.kchunk) - NG;
    __syncthreads();
    if (grp == 0)
      item_pair<0>(a, buf, scr, x0, y0, n0, n1);
    else
      item_pair<1>(a, buf, scr, x0, y0, n0, n1);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (a.dyn) {
      __syncthreads();
      if (threadIdx.x == 0) s_next = next;
      __syncthreads();
      item = s_next;
    } else {
      item += gridDim.x;
    }
  }
}

}  // namespace gzm

void launch_adj_gather_zm(const Layout& L, const Phys<float>& ph, const float* coef, float* dbar, float* gbar,
                          float* fbar, double alpha, double beta, int klo, int khi, int ksw, StepState* ss,
                          cudaStream_t st, bool chained) {
  // persistent CTAs on the current device (shared-memory limit set there)
  static PerDevice<int> per_dev;
  const int ctas = per_dev.get([] {
    cudaFuncSetAttribute(gzm::gather_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gzm::SMEM);
    int per = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, gzm::gather_pair_kernel, gzm::NT, gzm::SMEM);
    return sm_count() * (per > 0 ? per : 1);
  });
  gzm::Args a;
  a.L = L;
  a.ph = ph;
  a.coef = coef;
  a.dbar = dbar;
  a.gbar = gbar;
  a.fbar = fbar;
  a.alpha = (float)alpha;
  a.beta = (float)beta;
  a.klo = klo;
  a.khi = khi;
  a.ksw = ksw;
  a.ss = ss;
  a.ntx = (L.nx + gzm::TX - 1) / gzm::TX;
  a.nty = (L.ny + gzm::TY - 1) / gzm::TY;
  const int tiles = a.ntx * a.nty;
  a.kchunk = zm::zchunk(L.nz + 2 * NG, 2 * tiles, ctas);
  a.nch = (L.nz + 2 * NG + a.kchunk - 1) / a.kchunk;
  const double W1[4] = {0.0, 45.0 / 60.0, -9.0 / 60.0, 1.0 / 60.0};
  const double W2[4] = {-490.0 / 180.0, 270.0 / 180.0, -27.0 / 180.0, 2.0 / 180.0};
  auto weights = [&](double h) {
    pk::Coef c;
    c.c1 = pk::F2((float)(W1[1] / h)); c.c2 = pk::F2((float)(W1[2] / h)); c.c3 = pk::F2((float)(W1[3] / h));
    c.e0 = pk::F2((float)(W2[0] / (h * h))); c.e1 = pk::F2((float)(W2[1] / (h * h)));
    c.e2 = pk::F2((float)(W2[2] / (h * h))); c.e3 = pk::F2((float)(W2[3] / (h * h)));
    return c;
  };
  a.cx = weights(1.0 / (double)ph.idx);
  a.cy = weights(1.0 / (double)ph.idy);
  const int nitems = 2 * tiles * a.nch;
  const int grid = nitems < ctas ? nitems : ctas;
  a.dyn = nitems >= 4 * grid;
  if (a.dyn) cudaMemsetAsync(&ss->items, 0, sizeof(int), st);
  launch_chained(chained && !a.dyn, gzm::gather_pair_kernel, grid, gzm::NT, gzm::SMEM, st, a);
}

}  // namespace mhd
