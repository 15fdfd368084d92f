// mhd_ghost.cu -- ghost-zone kernels: the pointwise bottom/top atmospheric
// rules and periodic-z copies; and the copies between interior and padded
// arrays (which fill the periodic x,y rims).
#include "mhd_bc.cuh"
#include "mhd_internal.h"

namespace mhd {

// The ghost rules (mhd_bc.cuh) of both ends; bc_z = 1: periodic copies in z of
// all fields (test geometry; the background is zero there).
//
// Bound by latency: each column is a chain of exponentials and divisions (in
// FP64 some hundred dependent operations), and there are few columns.  The
// two ends are separate threads and blocks hold 64 of them, so that the
// chains run side by side over all SMs (32^2 columns in FP64: blocks of 256
// threads with both ends in a thread took 19 us on 6 SMs).
template <typename R>
__global__ void __launch_bounds__(BC_TH) bc_kernel(Layout L, Phys<R> ph, Background<R> bg, R* f, const StepState* ss) {
  chain_enter();
  const int pw = L.nx + 2 * NG, phh = L.ny + 2 * NG;
  const int q = blockIdx.x * BC_TH + threadIdx.x;
  if (q >= pw * phh) return;
  if (halted(ss)) return;
  const int i = q % pw - NG, j = q / pw - NG;
  const int nz = L.nz, kt = nz - 1;
  const bool top = blockIdx.y != 0;
  if (ph.bcz == 1) {
    for (int fl = 0; fl < NF; ++fl)
      for (int m = 1; m <= NG; ++m) {
        if (!top) f[L.at(fl, -m, j, i)] = f[L.at(fl, nz - m, j, i)];
        else f[L.at(fl, kt + m, j, i)] = f[L.at(fl, m - 1, j, i)];
      }
    return;
  }
  ghost_rules<R>(L, ph, bg, f, i, j, top);
}

template <typename R>
void launch_bc(const Layout& L, const Phys<R>& ph, const Background<R>& bg, R* f, const StepState* ss,
               cudaStream_t st, bool chained) {
  int n = (L.nx + 2 * NG) * (L.ny + 2 * NG);
  launch_chained(chained, bc_kernel<R>, dim3((n + BC_TH - 1) / BC_TH, 2), BC_TH, 0, st, L, ph, bg, f, ss);
}

// interior [field][nz][ny][nx] <-> padded; the background is added on the
// way out and removed on the way in (ln rho, ln T: the profiles; A: the
// background field when A is stored about one)
template <typename R>
__device__ __forceinline__ R bg_at(const Layout& L, const Background<R>& bg, int fl, int k, int j, int i) {
  if (fl == LR) return bg.lbar[k + NG];
  if (fl == LT) return bg.tbar[k + NG];
  if (fl <= AZ && bg.abg) return bg.abg[L.at(fl, k, j, i)];
  return R(0);
}

// Interior <-> padded copies.  Bound by memory: a plane is walked as a flat
// run of 16-byte vectors (four per thread, all loads issued before the
// stores), with the field and layer in the grid, so the only index division
// is one 32-bit one per vector; the element-by-element form with its 64-bit
// divisions took 0.68 ms for the 256^3 FP32 state against a floor of 0.16.
// Rows that are no multiple of a vector (odd nx), or a caller's array that is
// not 16-byte aligned, take the same kernel one element at a time (E = 1).
template <typename R, int E>
struct Vec {
  R v[E];
  __device__ __forceinline__ static Vec ld(const R* p) {
    Vec r;
    if constexpr (E * sizeof(R) == 16) {
      *reinterpret_cast<float4*>(r.v) = *reinterpret_cast<const float4*>(p);
    } else {
#pragma unroll
      for (int e = 0; e < E; ++e) r.v[e] = p[e];
    }
    return r;
  }
  __device__ __forceinline__ void st(R* p) const {
    if constexpr (E * sizeof(R) == 16) {
      *reinterpret_cast<float4*>(p) = *reinterpret_cast<const float4*>(v);
    } else {
#pragma unroll
      for (int e = 0; e < E; ++e) p[e] = v[e];
    }
  }
};
constexpr int CPT = 4;  // vectors per thread
constexpr int CTH = 256;

// FOLD: the adjoint's copy: no background, and the adjoints of the stateful
// u_x, u_y ghost rows are added to the photospheric layer they start from
template <typename R, int E, bool FOLD>
__global__ void __launch_bounds__(CTH) pack_kernel(Layout L, Background<R> bg, const R* __restrict__ f,
                                                   R* __restrict__ out, int f0, bool fold) {
  const int fl = f0 + (int)blockIdx.z;
  const int nv = L.nx / E, total = nv * L.ny;
  const long long n2 = (long long)L.nx * L.ny;
  for (int k = blockIdx.y; k < L.nz; k += gridDim.y) {
    R* o = out + ((long long)blockIdx.z * L.nz + k) * n2;
    const R add = FOLD ? R(0) : (fl == LR ? bg.lbar[k + NG] : (fl == LT ? bg.tbar[k + NG] : R(0)));
    const bool ab = !FOLD && fl <= AZ && bg.abg;
    const bool fd = FOLD && fold && k == 0 && (fl == UX || fl == UY);
    Vec<R, E> v[CPT];
    long long q[CPT];
#pragma unroll
    for (int u = 0; u < CPT; ++u) {
      const int x = blockIdx.x * (CTH * CPT) + u * CTH + threadIdx.x;
      if (x >= total) continue;
      const int j = x / nv;
      q[u] = L.at(fl, k, j, (x - j * nv) * E);
      v[u] = Vec<R, E>::ld(f + q[u]);
    }
#pragma unroll
    for (int u = 0; u < CPT; ++u) {
      const int x = blockIdx.x * (CTH * CPT) + u * CTH + threadIdx.x;
      if (x >= total) continue;
      if (ab) {
        const Vec<R, E> b = Vec<R, E>::ld(bg.abg + q[u]);
#pragma unroll
        for (int e = 0; e < E; ++e) v[u].v[e] += b.v[e];
      } else if (fd) {
        for (int m = 1; m <= NG; ++m) {
          const Vec<R, E> b = Vec<R, E>::ld(f + q[u] - m * L.sz());
#pragma unroll
          for (int e = 0; e < E; ++e) v[u].v[e] += b.v[e];
        }
      } else if (!FOLD) {
#pragma unroll
        for (int e = 0; e < E; ++e) v[u].v[e] += add;
      }
      v[u].st(o + (long long)x * E);
    }
  }
}

// A whole padded set from the interior array in one pass: interior cells and
// their periodic x, y images on the interior layers, u_x, u_y below the
// photosphere equal to the photospheric layer (the stateful ghosts' start;
// only when `ughost`), zero elsewhere.  ADJ: no background, no images, and a
// second array gets beta times the same (the adjoint of the RK accumulator).
template <typename R, int E, bool ADJ>
__global__ void __launch_bounds__(CTH) unpack_kernel(Layout L, Background<R> bg, const R* __restrict__ in,
                                                     R* __restrict__ f, R* __restrict__ f2, R beta, bool ughost) {
  constexpr int P = 16 / sizeof(R);  // the padded rows are always whole vectors
  const int fl = blockIdx.z;
  const int nv = L.mx / P, total = nv * L.my;
  const long long n2 = (long long)L.nx * L.ny;
  for (int kp = blockIdx.y; kp < L.mz; kp += gridDim.y) {
    const int kg = kp - NG;
    const bool ug = ughost && kg < 0 && (fl == UX || fl == UY);
    const int k = ug ? 0 : kg;
    const bool layer = k >= 0 && k < L.nz;
    const R sub = ADJ || !layer ? R(0) : (fl == LR ? bg.lbar[k + NG] : (fl == LT ? bg.tbar[k + NG] : R(0)));
    const bool ab = !ADJ && layer && fl <= AZ && bg.abg;
    const R* src = in + ((long long)fl * L.nz + (layer ? k : 0)) * n2;
    const long long base = L.at(fl, kg, -NG, -XOFF);
    Vec<R, P> v[CPT];
    if constexpr (E == P) {
      // whole vectors throughout, the periodic images too (a vector that holds
      // one may carry a further cell into the row padding), so that no warp
      // splits at the row ends; all loads go out before the first is used
      int off[CPT];
      bool take[CPT];
#pragma unroll
      for (int u = 0; u < CPT; ++u) {
        const int x = min((int)blockIdx.x * (CTH * CPT) + u * CTH + (int)threadIdx.x, total - 1);
        const int r = x / nv, i0 = (x - r * nv) * P - XOFF;
        int j = r - NG;
        const bool rim = j < 0 || j >= L.ny;
        j = j < 0 ? j + L.ny : (j >= L.ny ? j - L.ny : j);
        take[u] = layer && (ADJ ? !rim && i0 >= 0 && i0 < L.nx : i0 + P > -NG && i0 < L.nx + NG);
        off[u] = take[u] ? j * L.nx + (i0 < 0 ? i0 + L.nx : (i0 >= L.nx ? i0 - L.nx : i0)) : 0;
      }
#pragma unroll
      for (int u = 0; u < CPT; ++u) v[u] = Vec<R, P>::ld(src + off[u]);
      if (ab) {
#pragma unroll
        for (int u = 0; u < CPT; ++u) {
          const int j = off[u] / L.nx;
          const Vec<R, P> b = Vec<R, P>::ld(bg.abg + L.at(fl, k, j, off[u] - j * L.nx));
#pragma unroll
          for (int e = 0; e < P; ++e) v[u].v[e] -= b.v[e];
        }
      }
#pragma unroll
      for (int u = 0; u < CPT; ++u)
#pragma unroll
        for (int e = 0; e < P; ++e) v[u].v[e] = take[u] ? (ADJ || ab ? v[u].v[e] : v[u].v[e] - sub) : R(0);
    } else {
      for (int u = 0; u < CPT; ++u) {
        const int x = min((int)blockIdx.x * (CTH * CPT) + u * CTH + (int)threadIdx.x, total - 1);
        const int r = x / nv, i0 = (x - r * nv) * P - XOFF;
        int j = r - NG;
        const bool rim = j < 0 || j >= L.ny;
        j = j < 0 ? j + L.ny : (j >= L.ny ? j - L.ny : j);
        for (int e = 0; e < P; ++e) {
          int i = i0 + e;
          const bool cell = layer && (ADJ ? !rim && i >= 0 && i < L.nx : i >= -NG && i < L.nx + NG);
          if (i < 0) i += L.nx;
          else if (i >= L.nx) i -= L.nx;
          R t = R(0);
          if (cell) t = src[(long long)j * L.nx + i] - (ab ? bg.abg[L.at(fl, k, j, i)] : sub);
          v[u].v[e] = t;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < CPT; ++u) {
      const int x = blockIdx.x * (CTH * CPT) + u * CTH + threadIdx.x;
      if (x >= total) continue;
      v[u].st(f + base + (long long)x * P);
      if (ADJ) {
#pragma unroll
        for (int e = 0; e < P; ++e) v[u].v[e] *= beta;
        v[u].st(f2 + base + (long long)x * P);
      }
    }
  }
}

// whole vectors per row and a 16-byte aligned caller array
template <typename R>
static bool vec_ok(const Layout& L, const void* p) {
  return L.nx % (16 / (int)sizeof(R)) == 0 && ((uintptr_t)p & 15u) == 0;
}
static dim3 copy_grid(int vecs, int layers, int fields) {
  return dim3((vecs + CTH * CPT - 1) / (CTH * CPT), layers < 65535 ? layers : 65535, fields);
}

// padded [field][nz+6][ny+6][nx+6] copy, background added
template <typename R>
__global__ void pack_padded_kernel(Layout L, Background<R> bg, const R* __restrict__ f, R* __restrict__ out) {
  const int pw = L.nx + 2 * NG, ph = L.ny + 2 * NG;
  const long long n = (long long)pw * ph * L.mz * NF;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n;
       q += (long long)gridDim.x * blockDim.x) {
    int i = (int)(q % pw) - NG;
    long long r = q / pw;
    int j = (int)(r % ph) - NG;
    r /= ph;
    int k = (int)(r % L.mz) - NG;
    int fl = (int)(r / L.mz);
    out[q] = f[L.at(fl, k, j, i)] + bg_at(L, bg, fl, k, j, i);
  }
}

// one z layer k of one field, interior [ny][nx], background added
template <typename R>
__global__ void pack_plane_kernel(Layout L, Background<R> bg, const R* __restrict__ f, R* __restrict__ out, int field,
                                  int k) {
  const long long n2 = (long long)L.nx * L.ny;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n2; q += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(q % L.nx), j = (int)(q / L.nx);
    out[q] = f[L.at(field, k, j, i)] + bg_at(L, bg, field, k, j, i);
  }
}

// per-layer mean of one field of an interior-packed state, FP64, fixed order
template <typename R>
__global__ void layer_mean_kernel(Layout L, const R* __restrict__ in, int field, double* out) {
  __shared__ double sm[256];
  const int k = blockIdx.x;
  const long long n2 = (long long)L.nx * L.ny;
  const R* p = in + ((long long)field * L.nz + k) * n2;
  double s = 0.0;
  for (long long q = threadIdx.x; q < n2; q += blockDim.x) s += (double)p[q];
  sm[threadIdx.x] = s;
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) sm[threadIdx.x] += sm[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[k] = sm[0] / (double)n2;
}

template <typename R>
void launch_pack(const Layout& L, const Background<R>& bg, const R* f, R* out, int field, cudaStream_t st) {
  constexpr int E = 16 / sizeof(R);
  const int f0 = field < 0 ? 0 : field, nf = field < 0 ? NF : 1;
  if (vec_ok<R>(L, out))
    pack_kernel<R, E, false><<<copy_grid(L.nx / E * L.ny, L.nz, nf), CTH, 0, st>>>(L, bg, f, out, f0, false);
  else
    pack_kernel<R, 1, false><<<copy_grid(L.nx * L.ny, L.nz, nf), CTH, 0, st>>>(L, bg, f, out, f0, false);
}
template <typename R>
void launch_adj_pack(const Layout& L, int bcz, const R* fbar, R* out, cudaStream_t st) {
  constexpr int E = 16 / sizeof(R);
  const Background<R> none{};
  if (vec_ok<R>(L, out))
    pack_kernel<R, E, true><<<copy_grid(L.nx / E * L.ny, L.nz, NF), CTH, 0, st>>>(L, none, fbar, out, 0, bcz == 0);
  else
    pack_kernel<R, 1, true><<<copy_grid(L.nx * L.ny, L.nz, NF), CTH, 0, st>>>(L, none, fbar, out, 0, bcz == 0);
}
template <typename R>
void launch_unpack(const Layout& L, const Background<R>& bg, const R* in, R* f, bool ughost, cudaStream_t st) {
  constexpr int E = 16 / sizeof(R);
  const dim3 g = copy_grid(L.mx / E * L.my, L.mz, NF);
  if (vec_ok<R>(L, in)) unpack_kernel<R, E, false><<<g, CTH, 0, st>>>(L, bg, in, f, nullptr, R(0), ughost);
  else unpack_kernel<R, 1, false><<<g, CTH, 0, st>>>(L, bg, in, f, nullptr, R(0), ughost);
}
template <typename R>
void launch_adj_unpack(const Layout& L, const R* in, R* fbar, R* dbar, double beta, cudaStream_t st) {
  constexpr int E = 16 / sizeof(R);
  const Background<R> none{};
  const dim3 g = copy_grid(L.mx / E * L.my, L.mz, NF);
  if (vec_ok<R>(L, in)) unpack_kernel<R, E, true><<<g, CTH, 0, st>>>(L, none, in, fbar, dbar, (R)beta, false);
  else unpack_kernel<R, 1, true><<<g, CTH, 0, st>>>(L, none, in, fbar, dbar, (R)beta, false);
}
template <typename R>
void launch_pack_padded(const Layout& L, const Background<R>& bg, const R* f, R* out, cudaStream_t st) {
  pack_padded_kernel<R><<<1216, 256, 0, st>>>(L, bg, f, out);
}
template <typename R>
void launch_pack_plane(const Layout& L, const Background<R>& bg, const R* f, R* out, int field, int k, cudaStream_t st) {
  const long long n2 = (long long)L.nx * L.ny;
  pack_plane_kernel<R><<<(int)((n2 + 255) / 256 < 1216 ? (n2 + 255) / 256 : 1216), 256, 0, st>>>(L, bg, f, out, field, k);
}
template <typename R>
void launch_layer_mean(const Layout& L, const R* in, int field, double* out, cudaStream_t st) {
  layer_mean_kernel<R><<<L.nz, 256, 0, st>>>(L, in, field, out);
}

#define INST(R)                                                                               \
  template void launch_bc<R>(const Layout&, const Phys<R>&, const Background<R>&, R*,          \
                             const StepState*, cudaStream_t, bool);                            \
  template void launch_pack<R>(const Layout&, const Background<R>&, const R*, R*, int, cudaStream_t); \
  template void launch_adj_pack<R>(const Layout&, int, const R*, R*, cudaStream_t);           \
  template void launch_adj_unpack<R>(const Layout&, const R*, R*, R*, double, cudaStream_t);  \
  template void launch_unpack<R>(const Layout&, const Background<R>&, const R*, R*, bool, cudaStream_t); \
  template void launch_pack_padded<R>(const Layout&, const Background<R>&, const R*, R*, cudaStream_t); \
  template void launch_layer_mean<R>(const Layout&, const R*, int, double*, cudaStream_t);                 \
  template void launch_pack_plane<R>(const Layout&, const Background<R>&, const R*, R*, int, int, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace mhd
