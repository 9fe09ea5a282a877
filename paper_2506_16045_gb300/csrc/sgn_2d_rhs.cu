// Gradient (a2) and right-hand side (a7) on 2d power-of-two grids by one-dimensional derivative
// passes: f_x needs transforms along the rows only and f_y along the columns only, so a
// derivative costs two 1d transforms of a packed pair of real fields instead of four (and no
// pass over a half spectrum).  The right-hand side is four kernels:
//   x1  rows:    x derivatives of u, eta u, zeta, s, eta u u, eta u v
//   y1  columns: y derivatives of v, eta v, zeta, s, eta u v, eta v v; d = div u, m = div(eta u),
//                p = -g eta grad zeta - div(eta u (x) u); d_y
//   x2  rows:    d_x, then Phi and Psi, Phi_x; f_eta = -m, f_U's x component
//   y2  columns: Phi_y, f_U's y component
// with s = grad h . u, Q = u . grad d - d^2, S = u . grad s,
//   Phi = eta^3 Q / 3 + eta^2 m d + eta^2 S / 2 + eta m s,  Psi = eta^2 Q / 2 + eta m d + eta S + m s
// (Def:bigF; the four pieces of f_U share these two).  The transforms run in T (float64, or
// double-float for the mixed path) and the planes between them hold T; the products at a point
// are float64 (in double-float they made f_eta's error 1.2 to 1.5 times as large, since a
// derivative follows).
//
// What bounds it: the issue of the double-float stages (or the float64 pipe), and latency where
// a grid has few rows.  Against 26 two-dimensional half-spectrum transforms in 23 launches (one
// GB300): 512 x 512 mixed, 4 RK4 steps 15.5 -> 13.0 ms (about 160 us less per evaluation), the
// 256 x 256 float64 run 1.09 times as fast.
#include "sgn_2d_fft.cuh"

namespace sgn {

using namespace d2;

namespace {

constexpr int kRhsColNT = 512;

template <typename T>
struct RhsArgs2d {
  int nx, ny, lx, ly;
  long long P;
  double kxn, kyn;           // 2 pi / (Lx nx), 2 pi / (Ly ny)
  double g;
  const double *eta, *u, *h, *gh;
  T* w;                      // planes, see W_* (W_PX, W_PY and W_R hold float64)
  double *f_eta, *f_U;
  const void *t64, *t32;
};
// planes: x derivatives of x1 (W_UX .. W_TXY), then what y1 leaves, then x2
enum { W_UX = 0, W_MX, W_ZX, W_SX, W_TXX, W_TXY, W_D, W_M, W_PX, W_PY, W_SY, W_DY, W_PHI, W_R };

// Columns per CTA: four float64 fill a 32-byte sector; fewer on narrow grids, where tiles of
// four would leave SMs idle (nx = 256: 64 tiles; the 256 x 256 float64 run is 1.02 times as fast
// with two as with four).
int rhs_tw(int nx) { return nx >= 512 ? 4 : (nx >= 256 ? 2 : 1); }

template <typename T>
__global__ void __launch_bounds__(kMatvecNT, 2) k2_rhs_x1(const __grid_constant__ RhsArgs2d<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int nx = a.nx;
  const long long P = a.P, row = (long long)blockIdx.x * nx;
  cplx<T>* z = reinterpret_cast<cplx<T>*>(smem);
  cplx<T>* tab = z + 3 * nx;
  fill_tw2(tab, a.lx, Tw<T>::get(a.t64, a.t32));
  for (int x = threadIdx.x; x < nx; x += blockDim.x) {
    const long long j = row + x;
    const double e = a.eta[j], u = a.u[j], v = a.u[P + j], eu = e * u;
    const double s = a.gh[j] * u + a.gh[P + j] * v;
    cplx<T>* q = z + sw2(x);
    q[0] = mk(num<T>(u), num<T>(eu));
    q[nx] = mk(num<T>(e - a.h[j]), num<T>(s));
    q[2 * nx] = mk(num<T>(eu * u), num<T>(eu * v));
  }
  __syncthreads();
  deriv2d<T>(z, a.lx, 3, nx, tab, num<T>(a.kxn));
  for (int x = threadIdx.x; x < nx; x += blockDim.x) {
    T* w = a.w + row + x;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const cplx<T> v = z[q * nx + sw2(x)];
      w[(2 * q) * P] = v.x;
      w[(2 * q + 1) * P] = v.y;
    }
  }
}

template <typename T, int TW>
__global__ void __launch_bounds__(kRhsColNT, 1) k2_rhs_y1(const __grid_constant__ RhsArgs2d<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int nx = a.nx, ny = a.ny, st = col_stride<TW>(ny);
  const long long P = a.P;
  cplx<T>* z = reinterpret_cast<cplx<T>*>(smem);             // pair q of column c at (q TW + c) st
  cplx<T>* tab = z + 3 * TW * st;
  fill_tw2(tab, a.ly, Tw<T>::get(a.t64, a.t32));
  const int c0 = blockIdx.x * TW;
  for (int i = threadIdx.x; i < TW * ny; i += kRhsColNT) {
    const int y = i / TW, c = i % TW;
    const long long j = (long long)y * nx + c0 + c;
    const double e = a.eta[j], u = a.u[j], v = a.u[P + j], ev = e * v;
    const double s = a.gh[j] * u + a.gh[P + j] * v;
    cplx<T>* q = z + c * st + sw2(y);
    q[0] = mk(num<T>(v), num<T>(ev));
    q[TW * st] = mk(num<T>(e - a.h[j]), num<T>(s));
    q[2 * TW * st] = mk(num<T>(ev * u), num<T>(ev * v));
  }
  __syncthreads();
  const T kn = num<T>(a.kyn);
  deriv2d<T>(z, a.ly, 3 * TW, st, tab, kn);
  for (int i = threadIdx.x; i < TW * ny; i += kRhsColNT) {
    const int y = i / TW, c = i % TW;
    const long long j = (long long)y * nx + c0 + c;
    cplx<T>* q = z + c * st + sw2(y);
    const cplx<T> vm = q[0], zs = q[TW * st], t = q[2 * TW * st];
    T* w = a.w + j;
    const T d = w[W_UX * P] + vm.x;
    const double ge = a.g * a.eta[j];
    double* wd = reinterpret_cast<double*>(a.w) + j;
    w[W_D * P] = d;
    w[W_M * P] = w[W_MX * P] + vm.y;
    wd[W_PX * P] = -ge * to_f64(w[W_ZX * P]) - to_f64(w[W_TXX * P] + t.x);
    wd[W_PY * P] = -ge * to_f64(zs.x) - to_f64(w[W_TXY * P] + t.y);
    w[W_SY * P] = zs.y;
    q[0] = mk(d, from_int<T>(0));
  }
  __syncthreads();
  // d_y, two columns to a sequence
  constexpr int NB = TW > 1 ? TW / 2 : 1, ST = TW > 1 ? 2 : 1;
  if constexpr (TW > 1) {
    for (int i = threadIdx.x; i < NB * ny; i += kRhsColNT) {
      cplx<T>* q = z + 2 * (i / ny) * st + sw2(i % ny);
      q[0].y = q[st].x;
    }
    __syncthreads();
  }
  deriv2d<T>(z, a.ly, NB, ST * st, tab, kn);
  for (int i = threadIdx.x; i < TW * ny; i += kRhsColNT) {
    const int y = i / TW, c = i % TW;
    const cplx<T> v = z[(c / ST) * ST * st + sw2(y)];
    a.w[W_DY * P + (long long)y * nx + c0 + c] = (c % ST) ? v.y : v.x;
  }
}

template <typename T>
__global__ void __launch_bounds__(kRowNT, 3) k2_rhs_x2(const __grid_constant__ RhsArgs2d<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int nx = a.nx;
  const long long P = a.P, row = 2ll * blockIdx.x * nx;      // two rows to a sequence
  cplx<T>* z = reinterpret_cast<cplx<T>*>(smem);
  cplx<T>* tab = z + nx;
  fill_tw2(tab, a.lx, Tw<T>::get(a.t64, a.t32));
  for (int x = threadIdx.x; x < nx; x += blockDim.x)
    z[sw2(x)] = mk(a.w[W_D * P + row + x], a.w[W_D * P + row + nx + x]);
  __syncthreads();
  const T kn = num<T>(a.kxn);
  deriv2d<T>(z, a.lx, 1, nx, tab, kn);
  for (int x = threadIdx.x; x < nx; x += blockDim.x) {
    const cplx<T> dx = z[sw2(x)];
    T phi0, phi1;
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {
      const long long j = row + r * nx + x;
      T* w = a.w + j;
      double* wd = reinterpret_cast<double*>(a.w) + j;
      const double e = a.eta[j], u = a.u[j], v = a.u[P + j], hx = a.gh[j], hy = a.gh[P + j];
      const double d = to_f64(w[W_D * P]), m = to_f64(w[W_M * P]), s = hx * u + hy * v;
      const double Sv = u * to_f64(w[W_SX * P]) + v * to_f64(w[W_SY * P]);
      const double Q = u * to_f64(r ? dx.y : dx.x) + v * to_f64(w[W_DY * P]) - d * d;
      const double e2 = e * e, md = m * d, ms = m * s;
      const T Phi = num<T>(e2 * e * Q * (1.0 / 3.0) + e2 * md + 0.5 * (e2 * Sv) + e * ms);
      const double Psi = 0.5 * (e2 * Q) + e * md + e * Sv + ms;
      w[W_PHI * P] = Phi;
      wd[W_PX * P] -= hx * Psi;
      wd[W_R * P] = wd[W_PY * P] - hy * Psi;
      a.f_eta[j] = -m;
      if (r) phi1 = Phi; else phi0 = Phi;
    }
    z[sw2(x)] = mk(phi0, phi1);
  }
  __syncthreads();
  deriv2d<T>(z, a.lx, 1, nx, tab, kn);
  for (int x = threadIdx.x; x < nx; x += blockDim.x) {
    const cplx<T> v = z[sw2(x)];
    const long long j = row + x;
    const double* px = reinterpret_cast<const double*>(a.w) + W_PX * P + j;
    a.f_U[j] = to_f64(v.x) + px[0];
    a.f_U[j + nx] = to_f64(v.y) + px[nx];
  }
}

// out = (y derivative of the plane `in`) + add (nullable), TW columns per CTA.
template <typename T, int TW>
__device__ __forceinline__ void y_pass(int nx, int ny, int ly, const T* in, const double* add,
                                       double* out,
                                       double kyn, const cplx<T>* tw) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int NB = TW > 1 ? TW / 2 : 1, ST = TW > 1 ? 2 : 1;
  const int st = col_stride<NB>(ny), c0 = blockIdx.x * TW;
  cplx<T>* z = reinterpret_cast<cplx<T>*>(smem);
  cplx<T>* tab = z + NB * st;
  fill_tw2(tab, ly, tw);
  for (int i = threadIdx.x; i < NB * ny; i += blockDim.x) {
    const int y = i / NB, k = i % NB;
    const T* p = in + (long long)y * nx + c0 + ST * k;
    z[k * st + sw2(y)] = mk(p[0], TW > 1 ? p[ST - 1] : from_int<T>(0));
  }
  __syncthreads();
  deriv2d<T>(z, ly, NB, st, tab, num<T>(kyn));
  for (int i = threadIdx.x; i < NB * ny; i += blockDim.x) {
    const int y = i / NB, k = i % NB;
    const long long j = (long long)y * nx + c0 + ST * k;
    const cplx<T> v = z[k * st + sw2(y)];
    if (add) {
      out[j] = to_f64(v.x) + add[j];
      if (TW > 1) out[j + 1] = to_f64(v.y) + add[j + 1];
    } else {
      out[j] = to_f64(v.x);
      if (TW > 1) out[j + 1] = to_f64(v.y);
    }
  }
}

template <typename T, int TW>
__global__ void __launch_bounds__(kRowNT, 3) k2_rhs_y2(const __grid_constant__ RhsArgs2d<T> a) {
  y_pass<T, TW>(a.nx, a.ny, a.ly, a.w + W_PHI * a.P,
                reinterpret_cast<const double*>(a.w) + W_R * a.P, a.f_U + a.P, a.kyn,
                Tw<T>::get(a.t64, a.t32));
}

// Gradient: f_y into `fy` (scratch), then f_x with f_y copied along, so that f may be one of
// the two output planes.
template <int TW>
__global__ void __launch_bounds__(kRowNT, 3) k2_grad_y(int nx, int ny, int ly, const double* f,
                                                       double* fy, double kyn, const void* t64) {
  y_pass<double, TW>(nx, ny, ly, f, nullptr, fy, kyn, Tw<double>::get(t64, nullptr));
}

__global__ void __launch_bounds__(kRowNT, 3) k2_grad_x(int nx, int lx, long long P,
                                                       const double* f, const double* fy,
                                                       double* out, double kxn, const void* t64) {
  extern __shared__ __align__(16) unsigned char smem[];
  const long long row = 2ll * blockIdx.x * nx;
  cplx<double>* z = reinterpret_cast<cplx<double>*>(smem);
  cplx<double>* tab = z + nx;
  fill_tw2(tab, lx, Tw<double>::get(t64, nullptr));
  for (int x = threadIdx.x; x < nx; x += blockDim.x)
    z[sw2(x)] = mk(f[row + x], f[row + nx + x]);
  __syncthreads();
  deriv2d<double>(z, lx, 1, nx, tab, kxn);
  for (int x = threadIdx.x; x < nx; x += blockDim.x) {
    const cplx<double> v = z[sw2(x)];
    out[row + x] = v.x;
    out[row + nx + x] = v.y;
    out[P + row + x] = fy[row + x];
    out[P + row + nx + x] = fy[row + nx + x];
  }
}

// Threads of a CTA: one per butterfly of a stage, within [64, most].
int rhs_threads(int butterflies, int most) {
  const int t = (butterflies + 31) / 32 * 32;
  return t < 64 ? 64 : (t > most ? most : t);
}

template <typename K, typename... A>
cudaError_t go(K k, int grid, int nt, size_t sm, cudaStream_t s, A... args) {
  cudaError_t e = raise_smem(k, sm);
  if (e) return e;
  k<<<grid, nt, sm, s>>>(args...);
  return cudaGetLastError();
}

template <int TW>
size_t y_smem(int ny) {
  constexpr int NB = TW > 1 ? TW / 2 : 1;
  return ((size_t)NB * col_stride<NB>(ny) + ny) * 16;
}

template <typename T, int TW>
cudaError_t rhs_cols1(const RhsArgs2d<T>& a, cudaStream_t s) {
  const size_t sm = ((size_t)3 * TW * col_stride<TW>(a.ny) + a.ny) * sizeof(cplx<T>);
  return go(k2_rhs_y1<T, TW>, a.nx / TW, kRhsColNT, sm, s, a);
}
template <typename T, int TW>
cudaError_t rhs_cols2(const RhsArgs2d<T>& a, cudaStream_t s) {
  return go(k2_rhs_y2<T, TW>, a.nx / TW, rhs_threads(TW * a.ny / 4, kRowNT), y_smem<TW>(a.ny), s,
            a);
}

template <typename T>
cudaError_t rhs2d(const Layout2d& L, const void* tw64, const void* tw32, double g,
                  const double* eta, const double* u, const double* h, const double* gradh,
                  double* f_eta, double* f_U, cudaStream_t s) {
  const Modes2d M = modes_of(L);
  const RhsArgs2d<T> a{L.nx, L.ny, L.lx, L.ly, L.P, M.kxu / L.nx, M.kyu / L.ny, g, eta, u, h,
                       gradh, reinterpret_cast<T*>(L.rhs_w), f_eta, f_U, tw64, tw32};
  static_assert(sizeof(T) == sizeof(double), "planes of L.P doubles");
  cudaError_t e;
  const size_t row = sizeof(cplx<T>) * L.nx;
  const int tw = rhs_tw(L.nx);
  if ((e = go(k2_rhs_x1<T>, L.ny, rhs_threads(3 * L.nx / 4, kMatvecNT), 4 * row, s, a))) return e;
  if ((e = tw == 4 ? rhs_cols1<T, 4>(a, s) : tw == 2 ? rhs_cols1<T, 2>(a, s) : rhs_cols1<T, 1>(a, s)))
    return e;
  if ((e = go(k2_rhs_x2<T>, L.ny / 2, rhs_threads(L.nx / 2, kRowNT), 2 * row, s, a))) return e;
  return tw == 4 ? rhs_cols2<T, 4>(a, s) : tw == 2 ? rhs_cols2<T, 2>(a, s) : rhs_cols2<T, 1>(a, s);
}

template <int TW>
cudaError_t grad_cols(const Layout2d& L, const void* tw64, const double* f, double* fy,
                      cudaStream_t s) {
  return go(k2_grad_y<TW>, L.nx / TW, rhs_threads(TW * L.ny / 4, kRowNT), y_smem<TW>(L.ny), s,
            L.nx, L.ny, L.ly, f, fy, modes_of(L).kyu / L.ny, tw64);
}

}  // namespace

cudaError_t launch_grad2d(const Layout2d& L, const void* tw64, const double* f, double* gradf,
                          cudaStream_t s) {
  if (L.mr) return mr2d_grad(L, f, gradf, s);
  double* fy = static_cast<double*>(L.tp);
  const int tw = rhs_tw(L.nx);
  cudaError_t e = tw == 4   ? grad_cols<4>(L, tw64, f, fy, s)
                  : tw == 2 ? grad_cols<2>(L, tw64, f, fy, s)
                            : grad_cols<1>(L, tw64, f, fy, s);
  if (e) return e;
  return go(k2_grad_x, L.ny / 2, rhs_threads(L.nx / 4, kRowNT), 2 * sizeof(cplx<double>) * L.nx, s,
            L.nx, L.lx, L.P, f, static_cast<const double*>(fy), gradf, modes_of(L).kxu / L.nx,
            tw64);
}

cudaError_t launch_rhs2d(const Layout2d& L, const void* tw64, const void* tw32, int precision,
                         double g, const double* eta, const double* u, const double* h,
                         const double* gradh, double* f_eta, double* f_U, cudaStream_t s) {
  if (L.mr) return mr2d_rhs(L, g, eta, u, h, gradh, f_eta, f_U, s);
  return precision == SGN_PREC_MIXED
             ? rhs2d<df>(L, tw64, tw32, g, eta, u, h, gradh, f_eta, f_U, s)
             : rhs2d<double>(L, tw64, tw32, g, eta, u, h, gradh, f_eta, f_U, s);
}

}  // namespace sgn
