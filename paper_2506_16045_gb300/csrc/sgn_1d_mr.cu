// 1d instances whose n is not a power of two: n = 2^a 3^b 5^c (a >= 1, 6 <= n <= 16384), the
// grids of §6.1 at sizes the register-blocked power-of-two kernels do not take.  One CTA per
// instance (kMrNT threads, 256 for float64 solves up to kMrSmall64), with a mixed-radix Stockham
// FFT (radices 8, 4, 2 for the power of two, then 5 and 3) in shared memory up to kMrSmemN and in
// global memory above, two buffers used in turn, and per-size twiddle tables built when the
// layout is created.  Every spectral operation follows the same
// formulas as the power-of-two kernels (D = F^{-1}(iK)F with the n/2 wavenumber set to 0,
// Def:G in its weak form, A^{-1} per mode, PCG with the stopping rule R7, the right-hand
// side of Eq:DAE_DSWE with Def:bigF):
//   k_mr_deriv   f -> D f                                   (float64)
//   k_mr_apply_G u -> G u                                   (float64)
//   k_mr_precond r -> A^{-1} r                              (float64)
//   k_mr_pcg     G x = b: float64 PCG, or float32 inner PCG inside double-float refinement
//   k_mr_rhs     (f_eta, f_U)                               (float64 or double-float)
#include <vector>

#include "sgn_1d_dev.cuh"
#include "sgn_mr_fft.cuh"

namespace sgn {
namespace {

using d1::kPi;
using mr::MrPlan;
using mr::mr_plan;
using mr::k_mr_twiddles;
constexpr int kMrNT = 512;
// Largest n whose float64 solve takes 256 threads: the float64 pipe is the bound
// either way, and the barriers of 16 warps cost more than they hide while a thread has one or
// two modes.  512 against 256 threads, one float64 solve (one call): n = 240 532 and 475 us, 768
// 579 and 543, 960 700 and 679, 1500 1126 and 1153 us.  The mixed solve has 512 at every size
// (n = 240 210 us, 192 with 256; 768 213 and 206; 960 238 and 238; 1500 300 and 305), and so has
// the right-hand side, where the two are equal up to 768 (n = 1500: 209 and 234 us).
constexpr int kMrSmall64 = 768;
constexpr int kMrMaxN = 16384;       // largest generic n
constexpr int kMrSmemN = 6144;       // largest n whose two transform buffers (192 KB) are in
                                     // shared memory; above it they are in global memory

// wavenumber of mode m (Nyquist 0), in T: ku = 2 pi / L in T.  No float64 in the float32 and
// double-float forms (a float64 operation costs 62 float32 ones here, and a wavenumber is
// formed for every mode of every transform).
template <typename T>
__device__ __forceinline__ T mr_k(int m, int n, T ku) {
  return ku * from_int<T>(wave_index(m, n));
}
// the mirror n - m of mode m
__device__ __forceinline__ int mr_mirror(int m, int n) { return m == 0 ? 0 : n - m; }

struct MrTw {            // the instance's twiddle tables (n - 1 entries each)
  const cplx<double>* d;
  const cplx<float>* f;
  const cplx<df>* h;
};
template <typename T>
__device__ __forceinline__ const cplx<T>* tw_of(const MrTw& t);
template <>
__device__ __forceinline__ const cplx<double>* tw_of<double>(const MrTw& t) { return t.d; }
template <>
__device__ __forceinline__ const cplx<float>* tw_of<float>(const MrTw& t) { return t.f; }
template <>
__device__ __forceinline__ const cplx<df>* tw_of<df>(const MrTw& t) { return t.h; }

struct MrArgs {
  const Inst1d* insts;
  const int* ids;          // the generic instances' ids
  cplx<double>* big;       // global transform buffers of the instances above kMrSmemN
  const cplx<double>* tw64;
  const cplx<float>* tw32;
  const cplx<df>* twdf;
};

__device__ __forceinline__ MrTw mr_tw(const MrArgs& A, const Inst1d& I) {
  return MrTw{A.tw64 + I.tw, A.tw32 + I.tw, A.twdf + I.tw};
}

// The instance's two transform buffers (n entries of 16 bytes each): shared memory, or its
// slot of the layout's global buffer (I.gbuf >= 0, n > kMrSmemN; the CTA's own L2-resident
// copy, written and read by this CTA only, ordered by the same barriers).
template <typename T>
__device__ __forceinline__ cplx<T>* tbuf(const MrArgs& A, const Inst1d& I, int which) {
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned char* base = I.gbuf >= 0 ? reinterpret_cast<unsigned char*>(A.big + I.gbuf) : smem;
  return reinterpret_cast<cplx<T>*>(base + (size_t)which * 16 * I.n);
}

// f_x of the real fields a + i b packed in buf (transform, i k / n, inverse): re / im
template <int NT, typename T>
__device__ __forceinline__ cplx<T>* mr_deriv_pair(cplx<T>* A, cplx<T>* B, const MrPlan& P,
                                                  double kunit, const cplx<T>* tw) {
  const int n = P.n;
  cplx<T>* F = mr::mr_fft<T, NT>(A, B, P, false, tw);
  const T kn = num<T>(kunit / n);
  for (int m = threadIdx.x; m < n; m += NT) F[m] = mul_pi(F[m]) * mr_k<T>(m, n, kn);
  __syncthreads();
  return mr::mr_fft<T, NT>(F, F == A ? B : A, P, true, tw);
}

// ---- operators (float64) ----------------------------------------------------------------
__global__ void __launch_bounds__(kMrNT) k_mr_deriv(const MrArgs A, const double* __restrict__ f,
                                                   double* __restrict__ fx) {
  const Inst1d I = A.insts[A.ids[blockIdx.x]];
  MrPlan P;
  mr_plan(I.n, P);
  cplx<double>* a = tbuf<double>(A, I, 0);
  cplx<double>* b = tbuf<double>(A, I, 1);
  for (int j = threadIdx.x; j < I.n; j += kMrNT) a[j] = mk(f[I.off + j], 0.0);
  __syncthreads();
  const cplx<double>* o = mr_deriv_pair<kMrNT, double>(a, b, P, 2.0 * kPi / I.L, mr_tw(A, I).d);
  for (int j = threadIdx.x; j < I.n; j += kMrNT) fx[I.off + j] = o[j].x;
}

// The transform of v + i v_x from the half spectrum of the real field v: a_m = (1 - k) v_m and
// a_{n-m} = (1 + k) conj v_m, the DC and Nyquist coefficients taken real (their imaginary
// parts are rounding residue).  get(m): v_m, m = 0..n/2.  Ends with a barrier.
template <int NT, typename T, typename Get>
__device__ __forceinline__ void mr_fill(cplx<T>* a, int n, T ku, Get get) {
  const int h = n / 2;
  const T one = from_int<T>(1);
  for (int m = threadIdx.x; m <= h; m += NT) {
    const cplx<T> v = get(m);
    if (m == 0 || m == h) {
      a[m] = mk(v.x, from_int<T>(0));
    } else {
      const T k = mr_k<T>(m, n, ku);
      a[m] = v * (one - k);
      a[n - m] = conj(v) * (one + k);
    }
  }
  __syncthreads();
}

// With Z = F(v + i v_x) in a (mr_fill): back to real space, pointwise w = c1 v + c2 v_x,
// q = c2 v + c3 v_x, and the transform Y of w + i q, from which mr_gv takes (G v)^ (Def:G as
// w - q_x).  point(j, v, v_x) may keep the field.  Returns Y, after a barrier.
template <int NT, typename T, typename Coef, typename Point>
__device__ __forceinline__ cplx<T>* mr_wq(cplx<T>* a, cplx<T>* b, const MrPlan& P, T inv_n,
                                          const cplx<T>* tw, const Coef& coef, Point point) {
  const int n = P.n;
  cplx<T>* z = mr::mr_fft<T, NT>(a, b, P, true, tw);
  for (int j = threadIdx.x; j < n; j += NT) {
    const T v = z[j].x * inv_n, vx = z[j].y * inv_n;
    T c1, c2, c3;
    coef(j, c1, c2, c3);
    point(j, v, vx);
    z[j] = mk(c1 * v + c2 * vx, c2 * v + c3 * vx);
  }
  __syncthreads();
  return mr::mr_fft<T, NT>(z, z == a ? b : a, P, false, tw);
}
struct NoPoint {
  template <typename T>
  __device__ __forceinline__ void operator()(int, T, T) const {}
};

// (G v)^_m = ((1 - k_m) Y_m + (1 + k_m) conj Y_{n-m}) / 2, m = 0..n/2
template <typename T>
__device__ __forceinline__ cplx<T> mr_gv(const cplx<T>* Y, int m, int n, T ku) {
  const T one = from_int<T>(1), k = mr_k<T>(m, n, ku);
  const cplx<T> y = Y[m], ym = conj(Y[mr_mirror(m, n)]);
  const cplx<T> s = y * (one - k) + ym * (one + k);
  return mk(half(s.x), half(s.y));
}

struct Coef64 {
  const double* eta;
  const double* hx;
  __device__ void operator()(int j, double& c1, double& c2, double& c3) const {
    const double e = eta[j], g = hx[j];
    c1 = e * (1.0 + g * g);
    c2 = 0.5 * e * e * g;
    c3 = e * e * e / 3.0;
  }
};

__global__ void __launch_bounds__(kMrNT) k_mr_apply_G(const MrArgs A, const double* __restrict__ eta,
                                                     const double* __restrict__ hx,
                                                     const double* __restrict__ u,
                                                     double* __restrict__ Gu) {
  const Inst1d I = A.insts[A.ids[blockIdx.x]];
  MrPlan P;
  mr_plan(I.n, P);
  const int n = I.n, h = n / 2;
  cplx<double>* a = tbuf<double>(A, I, 0);
  cplx<double>* b = tbuf<double>(A, I, 1);
  const cplx<double>* tw = mr_tw(A, I).d;
  const double kunit = 2.0 * kPi / I.L;
  for (int j = threadIdx.x; j < n; j += kMrNT) a[j] = mk(u[I.off + j], 0.0);
  __syncthreads();
  // (1 - k) times the spectrum of a real field is that of v + i v_x
  cplx<double>* V = mr::mr_fft<double, kMrNT>(a, b, P, false, tw);
  cplx<double>* o = V == a ? b : a;
  for (int m = threadIdx.x; m < n; m += kMrNT) V[m] = V[m] * (1.0 - mr_k<double>(m, n, kunit));
  __syncthreads();
  cplx<double>* Y = mr_wq<kMrNT, double>(V, o, P, 1.0 / n, tw, Coef64{eta + I.off, hx + I.off}, NoPoint());
  o = Y == a ? b : a;
  // the Hermitian full spectrum of G u into the other buffer, and back
  for (int m = threadIdx.x; m <= h; m += kMrNT) {
    const cplx<double> g = mr_gv<double>(Y, m, n, kunit);
    o[m] = g;
    if (m > 0 && m < h) o[n - m] = conj(g);
  }
  __syncthreads();
  const cplx<double>* x = mr::mr_fft<double, kMrNT>(o, Y, P, true, tw);
  for (int j = threadIdx.x; j < n; j += kMrNT) Gu[I.off + j] = x[j].x / n;
}

__global__ void __launch_bounds__(kMrNT) k_mr_precond(const MrArgs A, const SolveRec* __restrict__ rec,
                                                     const double* __restrict__ r,
                                                     double* __restrict__ z) {
  const int id = A.ids[blockIdx.x];
  const Inst1d I = A.insts[id];
  MrPlan P;
  mr_plan(I.n, P);
  const int n = I.n;
  cplx<double>* a = tbuf<double>(A, I, 0);
  cplx<double>* b = tbuf<double>(A, I, 1);
  const cplx<double>* tw = mr_tw(A, I).d;
  const double kunit = 2.0 * kPi / I.L, sigma = rec[id].sigma, alpha = rec[id].alpha;
  for (int j = threadIdx.x; j < n; j += kMrNT) a[j] = mk(r[I.off + j], 0.0);
  __syncthreads();
  cplx<double>* F = mr::mr_fft<double, kMrNT>(a, b, P, false, tw);
  for (int m = threadIdx.x; m < n; m += kMrNT) {
    const double k = kunit * wave_index(m, n);
    F[m] = F[m] * (1.0 / ((sigma + alpha * k * k) * (double)n));
  }
  __syncthreads();
  const cplx<double>* x = mr::mr_fft<double, kMrNT>(F, F == a ? b : a, P, true, tw);
  for (int j = threadIdx.x; j < n; j += kMrNT) z[I.off + j] = x[j].x;
}

// ---- PCG -------------------------------------------------------------------------------
struct MrPcgArgs {
  const double* eta;
  const double* hx;
  const double* b;
  double* x;
  const SolveRec* given;
  int kind;
  double rtol, rtol_inner;
  int maxit, max_refine;
  SolveRec* rec;
  cplx<double>* ws;
  void* ux;              // nullable: also store x_x here (double-float or float64)
};

// coefficients of Def:MatrixM in double-float and float32
struct CoefDf {
  const double* eta;
  const double* hx;
  __device__ void operator()(int j, df& c1, df& c2, df& c3) const {
    const df e(eta[j]), g(hx[j]);
    const df e2 = e * e;
    c1 = e + e * g * g;
    c2 = half(e2 * g);
    c3 = e2 * e * df(0.3333333432674408f, -9.934107758624577e-09f);   // 1/3
  }
};
struct Coef32 {            // from float32 copies of eta and h_x
  const float2* eh;
  __device__ void operator()(int j, float& c1, float& c2, float& c3) const {
    const float2 v = eh[j];
    const float e = v.x, g = v.y;
    c1 = e * (1.0f + g * g);
    c2 = 0.5f * e * e * g;
    c3 = e * e * e * (1.0f / 3.0f);
  }
};

// The mixed path's sums over the CTA in double-float (48 bits; no float64 in its loops), by a
// fixed tree; slot[2][warps] and out[2] are used in turn, so a half is written
// again only after the barriers of the sum between
template <int NT>
__device__ __forceinline__ df mr_sum(df v, df* slots, df* outs, int& turn) {
  df* slot = slots + turn * (NT / 32);
  df* out = outs + turn;
  turn ^= 1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = v + df(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) slot[w] = v;
  __syncthreads();
  if (w == 0) {
    df r = l < NT / 32 ? slot[l] : df(0.0f, 0.0f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      r = r + df(__shfl_xor_sync(0xffffffffu, r.hi, o), __shfl_xor_sync(0xffffffffu, r.lo, o));
    if (l == 0) *out = r;
  }
  __syncthreads();
  return *out;
}
// The float64 sum over the CTA of values of the modes m <= h (thread t holds m = t + k kMrNT):
// block_sum's tree over the warps that hold any, with the same bits (the others add zeros).  A
// float64 add costs a warp 64 clocks of its sub-partition, idle lanes or not: n = 240 in
// float64, 6 RK4 steps, took 6.47 ms with all 16 warps in every sum.
template <int NT>
__device__ __forceinline__ double mr_sum64(double v, double* scratch, int h) {
  const int nw = min(NT / 32, (h >> 5) + 1), w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();                       // scratch may still be read by a previous call
  if (w < nw) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (l == 0) scratch[w] = v;
  }
  __syncthreads();
  if (w == 0) {
    double r = l < nw ? scratch[l] : 0.0;
    for (int o = nw > 8 ? 8 : nw > 4 ? 4 : nw > 2 ? 2 : nw - 1; o > 0; o >>= 1)
      r += __shfl_xor_sync(0xffffffffu, r, o);
    if (l == 0) scratch[NT / 32] = r;
  }
  __syncthreads();
  return scratch[NT / 32];
}

// One CTA per instance.  Bound by its SM: transforms through shared memory (n = 6144: 192 KB,
// one CTA per SM) with a barrier per stage.  The mixed form had wavenumbers, 1/(sigma + alpha
// k^2), Parseval weights, dot products and the float32 coefficients in float64 inside the
// float32 loop; they are float32 and double-float now (the two norms of a refinement pass stay
// float64).
template <bool MIXED, int NT>
__device__ __forceinline__ void mr_pcg(const MrArgs& A, const MrPcgArgs& a) {
  __shared__ double red[NT / 32 + 1];
  __shared__ df slot[2 * (NT / 32)];
  __shared__ df sums[2];
  int turn = 0;
  const int id = A.ids[blockIdx.x];
  const Inst1d I = A.insts[id];
  MrPlan P;
  mr_plan(I.n, P);
  const int n = I.n, h = n / 2;
  const long long S = h + 1;
  const double kunit = 2.0 * kPi / I.L;
  const MrTw tws = mr_tw(A, I);
  const double* eta = a.eta + I.off;
  const double* hx = a.hx + I.off;
  // ---- a1: coefficients (or the caller's)
  SolveRec R = {};
  if (a.given) {
    R = a.given[id];
    R.status = SGN_OK;
  } else {
    d1::coeffs_block<NT>(eta, hx, n, a.kind, red, R);
  }
  R.iters = 0;
  R.refinements = 0;
  R.ratio = 0.0;
  if (R.status != SGN_OK) {
    if (threadIdx.x == 0) a.rec[id] = R;
    return;
  }
  const double sigma = R.sigma, alpha = R.alpha;
  using TH = typename std::conditional<MIXED, df, double>::type;
  const TH kuh = num<TH>(kunit);
  cplx<double>* ws = a.ws + I.ws;
  // ---- b^ and x0^ (slots 0 and 1) from one transform of b + i x0, and b.A^{-1}b
  cplx<TH>* d0 = tbuf<TH>(A, I, 0);
  cplx<TH>* d1 = tbuf<TH>(A, I, 1);
  for (int j = threadIdx.x; j < n; j += NT)
    d0[j] = mk(num<TH>(a.b[I.off + j]), num<TH>(a.x[I.off + j]));
  __syncthreads();
  cplx<TH>* Y = mr::mr_fft<TH, NT>(d0, d1, P, false, tw_of<TH>(tws));
  cplx<TH>* Bh = reinterpret_cast<cplx<TH>*>(ws);
  cplx<TH>* Xh = reinterpret_cast<cplx<TH>*>(ws + S);
  auto half_of = [&](int m, cplx<TH>& bh, cplx<TH>& xh) {
    const cplx<TH> y = Y[m], ym = conj(Y[mr_mirror(m, n)]);
    const cplx<TH> sb = y + ym, sx = mul_mi(y - ym);
    bh = mk(half(sb.x), half(sb.y));
    xh = mk(half(sx.x), half(sx.y));
  };
  int iters = 0, status = SGN_OK;
  // b = 0 solves exactly, else a breakdown; x_x goes to the right-hand side with x
  auto no_rhs = [&](double bb) {
    for (int j = threadIdx.x; j < n; j += NT) {
      a.x[I.off + j] = 0.0;
      if (a.ux) static_cast<TH*>(a.ux)[I.off + j] = from_int<TH>(0);
    }
    R.status = (bb == 0.0) ? SGN_OK : SGN_ERR_BREAKDOWN;
    if (threadIdx.x == 0) a.rec[id] = R;
  };
  if constexpr (!MIXED) {
    // float64: b^, x^, r^, p^, (G p)^ in slots 0..4, 1/(sigma + alpha k^2) in slot 5
    cplx<double>* Rh = ws + 2 * S;
    cplx<double>* Ph = ws + 3 * S;
    cplx<double>* Gh = ws + 4 * S;
    double* Dv = reinterpret_cast<double*>(ws + 5 * S);
    auto wgt = [&](int m) { return (m == 0 || m == h) ? 1.0 : 2.0; };
    double bb = 0.0;
    for (int m = threadIdx.x; m <= h; m += NT) {
      const double k = kunit * wave_index(m, n), di = 1.0 / (sigma + alpha * k * k);
      Dv[m] = di;
      cplx<double> bh, xh;
      half_of(m, bh, xh);
      Bh[m] = bh;
      Xh[m] = xh;
      bb += wgt(m) * (bh.x * bh.x + bh.y * bh.y) * di;
    }
    bb = mr_sum64<NT>(bb, red, h);
    const double bnorm = sqrt(bb);
    if (!(bnorm > 0.0)) {
      no_rhs(bb);
      return;
    }
    const Coef64 coef{eta, hx};
    const double inv_n = 1.0 / n;
    auto matvec = [&](const cplx<double>* Vh) {     // Gh = (G v)^
      mr_fill<NT, double>(d0, n, kunit, [&](int m) { return Vh[m]; });
      const cplx<double>* W = mr_wq<NT, double>(d0, d1, P, inv_n, tws.d, coef, NoPoint());
      for (int m = threadIdx.x; m <= h; m += NT) Gh[m] = mr_gv<double>(W, m, n, kunit);
      __syncthreads();
    };
    matvec(Xh);
    double rz = 0.0;
    for (int m = threadIdx.x; m <= h; m += NT) {
      const cplx<double> r = Bh[m] - Gh[m];
      const double di = Dv[m];
      Rh[m] = r;
      Ph[m] = r * di;
      rz += wgt(m) * (r.x * r.x + r.y * r.y) * di;
    }
    rz = mr_sum64<NT>(rz, red, h);
    const double tol = a.rtol * bnorm;
    while (sqrt(rz) > tol) {
      if (iters >= a.maxit) {
        status = SGN_ERR_NOT_CONVERGED;
        break;
      }
      __syncthreads();
      matvec(Ph);
      double pq = 0.0;
      for (int m = threadIdx.x; m <= h; m += NT)
        pq += wgt(m) * (Ph[m].x * Gh[m].x + Ph[m].y * Gh[m].y);
      pq = mr_sum64<NT>(pq, red, h);
      if (!(pq > 0.0) || !isfinite(pq)) {
        status = SGN_ERR_BREAKDOWN;
        break;
      }
      const double al = rz / pq;
      double rzn = 0.0;
      for (int m = threadIdx.x; m <= h; m += NT) {
        Xh[m] = Xh[m] + Ph[m] * al;
        const cplx<double> r = Rh[m] - Gh[m] * al;
        Rh[m] = r;
        rzn += wgt(m) * (r.x * r.x + r.y * r.y) * Dv[m];
      }
      rzn = mr_sum64<NT>(rzn, red, h);
      ++iters;
      if (!isfinite(rzn)) {
        status = SGN_ERR_BREAKDOWN;
        break;
      }
      const double be = rzn / rz;
      rz = rzn;
      for (int m = threadIdx.x; m <= h; m += NT) Ph[m] = Rh[m] * Dv[m] + Ph[m] * be;
    }
    R.ratio = sqrt(rz) / bnorm;
    __syncthreads();
    // x + i x_x from one transform
    mr_fill<NT, double>(d0, n, kunit, [&](int m) { return Xh[m]; });
    const cplx<double>* x = mr::mr_fft<double, NT>(d0, d1, P, true, tws.d);
    double* ux = a.ux ? static_cast<double*>(a.ux) + I.off : nullptr;
    for (int j = threadIdx.x; j < n; j += NT) {
      a.x[I.off + j] = x[j].x * inv_n;
      if (ux) ux[j] = x[j].y * inv_n;
    }
  } else {
    // double-float refinement: b^ and x^ (slots 0, 1) and the residual (slot 4) in
    // double-float, float32 eta, h_x in slot 5.  The float32 inner solve lives in the two
    // transform buffers' 32 n bytes: its two transform buffers (16 n), then p, r and the
    // correction d (half spectra, 12 n + 24).  x and x_x come from the residual's own
    // transform; until the solve ends x holds double-float bits.
    cplx<df>* Gd = reinterpret_cast<cplx<df>*>(ws + 4 * S);
    float2* eh = reinterpret_cast<float2*>(ws + 5 * S);
    cplx<float>* f0 = tbuf<float>(A, I, 0);
    cplx<float>* f1 = f0 + n;
    cplx<float>* Pf = f1 + n;
    cplx<float>* Rf = Pf + S;
    cplx<float>* Df = Rf + S;
    double* xo = a.x + I.off;
    df* ux = a.ux ? static_cast<df*>(a.ux) + I.off : nullptr;
    const float sigf = (float)sigma, alf = (float)alpha, kf = (float)kunit;
    const float inv_nf = recip((float)n);
    const df sigh(sigma), alh(alpha), inv_n = recip(df(n));
    auto dinvf = [&](int m) {
      const float k = kf * (float)wave_index(m, n);
      return recip(fmaf(alf * k, k, sigf));
    };
    auto wf = [&](int m) { return (m == 0 || m == h) ? 1.0f : 2.0f; };
    // w_m |v|^2 / (sigma + alpha k^2) in float64 (|v|^2 may leave the float32 range), the
    // symbol's reciprocal by double-float
    auto term = [&](int m, cplx<df> v) {
      const df k = mr_k<df>(m, n, kuh);
      const double x = to_f64(v.x), y = to_f64(v.y);
      const double q = (x * x + y * y) * to_f64(recip(sigh + alh * (k * k)));
      return (m == 0 || m == h) ? q : q + q;
    };
    double bb = 0.0;
    for (int m = threadIdx.x; m <= h; m += NT) {
      cplx<df> bh, xh;
      half_of(m, bh, xh);
      Bh[m] = bh;
      Xh[m] = xh;
      bb += term(m, bh);
    }
    for (int j = threadIdx.x; j < n; j += NT)
      eh[j] = make_float2(df(eta[j]).hi, df(hx[j]).hi);
    bb = mr_sum64<NT>(bb, red, h);
    const double bnorm = sqrt(bb);
    if (!(bnorm > 0.0)) {
      no_rhs(bb);
      return;
    }
    const CoefDf cdf{eta, hx};
    const Coef32 c32{eh};
    int refinements = 0;
    double ratio = 0.0;
    for (;;) {
      // r^ = b^ - (G x)^ in double-float, and r.A^{-1}r; the real-space x on the way
      mr_fill<NT, df>(d0, n, kuh, [&](int m) { return Xh[m]; });
      const cplx<df>* W = mr_wq<NT, df>(d0, d1, P, inv_n, tws.h, cdf, [&](int j, df v, df vx) {
        xo[j] = __hiloint2double(__float_as_int(v.lo), __float_as_int(v.hi));
        if (ux) ux[j] = vx;
      });
      double rs = 0.0;
      for (int m = threadIdx.x; m <= h; m += NT) {
        const cplx<df> r = Bh[m] - mr_gv<df>(W, m, n, kuh);
        Gd[m] = r;
        rs += term(m, r);
      }
      const double nr = sqrt(mr_sum64<NT>(rs, red, h));
      ratio = nr / bnorm;
      if (ratio <= a.rtol) {
        status = SGN_OK;
        break;
      }
      if (status != SGN_OK) break;
      if (refinements >= a.max_refine || iters >= a.maxit) {
        status = SGN_ERR_NOT_CONVERGED;
        break;
      }
      const double tin = a.rtol_inner > 0.0 ? a.rtol_inner
                                            : fmin(0.1, fmax(1e-6, 0.3 * a.rtol / ratio));
      const float sc = (float)(1.0 / nr);
      const df tin2(tin * tin);
      // float32 PCG for G d = r / ||r||; p = A^{-1} r + beta p is formed with its transform's
      // input (beta = 0 first), and (G p)^ is taken from Y twice instead of being kept
      DfSum z0;
      for (int m = threadIdx.x; m <= h; m += NT) {
        const cplx<df> g = Gd[m];
        const cplx<float> r = mk((g.x.hi + g.x.lo) * sc, (g.y.hi + g.y.lo) * sc);
        Rf[m] = r;
        Df[m] = Pf[m] = mk(0.0f, 0.0f);
        z0.add(wf(m) * ((r.x * r.x + r.y * r.y) * dinvf(m)));
      }
      df rz = mr_sum<NT>(z0.s, slot, sums, turn);
      float beta = 0.0f;
      const int it0 = iters;
      int st_in = SGN_OK;
      while ((rz - tin2).hi > 0.0f) {
        if (iters >= a.maxit) {
          st_in = SGN_ERR_NOT_CONVERGED;
          break;
        }
        mr_fill<NT, float>(f0, n, kf, [&](int m) {
          const cplx<float> p = Rf[m] * dinvf(m) + Pf[m] * beta;
          Pf[m] = p;
          return p;
        });
        const cplx<float>* Yf = mr_wq<NT, float>(f0, f1, P, inv_nf, tws.f, c32, NoPoint());
        DfSum ps;
        for (int m = threadIdx.x; m <= h; m += NT) {
          const cplx<float> p = Pf[m], g = mr_gv<float>(Yf, m, n, kf);
          ps.add(wf(m) * (p.x * g.x + p.y * g.y));
        }
        const df pq = mr_sum<NT>(ps.s, slot, sums, turn);
        if (!(pq.hi > 0.0f) || !isfinite(pq.hi)) {
          st_in = SGN_ERR_BREAKDOWN;
          break;
        }
        const float al = quot(rz, pq);
        DfSum zs;
        for (int m = threadIdx.x; m <= h; m += NT) {
          Df[m] = Df[m] + Pf[m] * al;
          const cplx<float> r = Rf[m] - mr_gv<float>(Yf, m, n, kf) * al;
          Rf[m] = r;
          zs.add(wf(m) * ((r.x * r.x + r.y * r.y) * dinvf(m)));
        }
        const df rzn = mr_sum<NT>(zs.s, slot, sums, turn);
        ++iters;
        if (!isfinite(rzn.hi)) {
          st_in = SGN_ERR_BREAKDOWN;
          break;
        }
        beta = quot(rzn, rz);
        rz = rzn;
      }
      // a float32 breakdown after some progress keeps the correction (the next residual
      // decides); the iteration cap is reported by the refinement loop
      if (st_in == SGN_ERR_BREAKDOWN && iters == it0) status = SGN_ERR_BREAKDOWN;
      const df un(nr);
      for (int m = threadIdx.x; m <= h; m += NT)
        Xh[m] = mk(Xh[m].x + df(Df[m].x, 0.0f) * un, Xh[m].y + df(Df[m].y, 0.0f) * un);
      ++refinements;
      __syncthreads();                             // d has been read; d0 is filled next
    }
    R.refinements = refinements;
    R.ratio = ratio;
    for (int j = threadIdx.x; j < n; j += NT) {
      const double v = xo[j];
      xo[j] = to_f64(df(__int_as_float(__double2loint(v)), __int_as_float(__double2hiint(v))));
    }
  }
  R.iters = iters;
  R.status = status;
  if (threadIdx.x == 0) a.rec[id] = R;
}

// The threads follow the instance, so that its result does not depend on the ones beside it.
template <bool MIXED>
__global__ void __launch_bounds__(kMrNT) k_mr_pcg(const MrArgs A, const MrPcgArgs a) {
  if (!MIXED && A.insts[A.ids[blockIdx.x]].n <= kMrSmall64) {
    if (threadIdx.x >= 256) return;      // the barriers wait for the threads that are left
    mr_pcg<MIXED, 256>(A, a);
    return;
  }
  mr_pcg<MIXED, kMrNT>(A, a);
}

// ---- right-hand side (Eq:DAE_DSWE with Def:bigF, reading R6) ----------------------------
// Derivative pairs (u, eta u) -> (d, m); (zeta, s) -> (zeta_x, s_x); d -> d_x; Phi' -> Phi'_x
// with Phi' = eta^3 Q/3 + eta^2 m d + eta^2 S/2 + eta m s - eta u^2 (the flux folded in),
// Q = u d_x - d^2, S = u s_x; f_eta = -m, f_U = -g eta zeta_x + Phi'_x - h_x Psi,
// Psi = eta^2 Q/2 + eta m d + eta S + m s.  Intermediates in scratch planes (T per point).
// UXG: d = u_x is already in the first scratch plane (from the solve that produced u), so the
// pairs are (eta u, zeta) -> (m, zeta_x), (s, d) -> (s_x, d_x) and Phi': six transforms
// instead of eight.
template <typename T, bool UXG>
__global__ void __launch_bounds__(kMrNT) k_mr_rhs(const MrArgs A, double g, const double* __restrict__ eta,
                                                 const double* __restrict__ u,
                                                 const double* __restrict__ hgt,
                                                 const double* __restrict__ hx,
                                                 double* __restrict__ f_eta, double* __restrict__ f_U,
                                                 double* __restrict__ scr, long long Ptot) {
  const Inst1d I = A.insts[A.ids[blockIdx.x]];
  MrPlan P;
  mr_plan(I.n, P);
  const int n = I.n;
  const long long o = I.off;
  const double kunit = 2.0 * kPi / I.L;
  const cplx<T>* tw = tw_of<T>(mr_tw(A, I));
  cplx<T>* b0 = tbuf<T>(A, I, 0);
  cplx<T>* b1 = tbuf<T>(A, I, 1);
  // planes of Ptot 8-byte values (float64 or double-float), indexed by point
  T* D = reinterpret_cast<T*>(scr) + o;                 // d, then Psi
  T* M = reinterpret_cast<T*>(scr + Ptot) + o;          // m
  T* ZX = reinterpret_cast<T*>(scr + 2 * Ptot) + o;     // zeta_x
  T* SX = reinterpret_cast<T*>(scr + 3 * Ptot) + o;     // s_x
  static_assert(sizeof(T) == sizeof(double), "8-byte plane elements");
  const T third = num<T>(1.0 / 3.0), gT = num<T>(g);
  constexpr int passes = UXG ? 3 : 4;
#pragma unroll 1
  for (int pass = 0; pass < passes; ++pass) {
    // 0: (eta u, zeta), 1: (s, d); or 2: (u, eta u), 3: (zeta, s), 4: d; then 5: Phi'
    const int what = UXG ? (pass == 0 ? 0 : pass == 1 ? 1 : 5) : (pass < 3 ? 2 + pass : 5);
    if (what != 5) {
      for (int j = threadIdx.x; j < n; j += kMrNT) {
        if (what == 4) {
          b0[j] = mk(D[j], from_int<T>(0));
          continue;
        }
        const T uu = num<T>(u[o + j]), e = num<T>(eta[o + j]);
        if (what == 0) b0[j] = mk(e * uu, e - num<T>(hgt[o + j]));
        else if (what == 1) b0[j] = mk(num<T>(hx[o + j]) * uu, D[j]);
        else if (what == 2) b0[j] = mk(uu, e * uu);
        else b0[j] = mk(e - num<T>(hgt[o + j]), num<T>(hx[o + j]) * uu);
      }
      __syncthreads();
    }
    const cplx<T>* r = mr_deriv_pair<kMrNT, T>(b0, b1, P, kunit, tw);
    if (what == 5) {
      for (int j = threadIdx.x; j < n; j += kMrNT) {
        const T e = num<T>(eta[o + j]), g1 = num<T>(hx[o + j]);
        f_U[o + j] = to_f64(r[j].x - gT * e * ZX[j] - g1 * D[j]);
      }
    } else if (pass == passes - 2) {
      // all derivatives are there: Phi' (the next input), Psi (kept for f_U) and f_eta; the
      // result r may be b0 itself, each point read before it is written
      for (int j = threadIdx.x; j < n; j += kMrNT) {
        const T uu = num<T>(u[o + j]), e = num<T>(eta[o + j]), g1 = num<T>(hx[o + j]);
        const T d = D[j], m = M[j], s = g1 * uu;
        const T dx = UXG ? r[j].y : r[j].x, sx = UXG ? r[j].x : SX[j];
        const T Q = uu * dx - d * d, Sv = uu * sx;
        const T e2 = e * e;
        const T phi = e2 * e * Q * third + e2 * m * d + half(e2 * Sv) + e * m * s - e * uu * uu;
        D[j] = half(e2 * Q) + e * m * d + e * Sv + m * s;     // d is no longer needed
        b0[j] = mk(phi, from_int<T>(0));
        f_eta[o + j] = -to_f64(m);
      }
      __syncthreads();
    } else {
      for (int j = threadIdx.x; j < n; j += kMrNT) {
        if (what == 0) {
          M[j] = r[j].x;
          ZX[j] = r[j].y;
        } else if (what == 2) {
          D[j] = r[j].x;
          M[j] = r[j].y;
        } else {
          ZX[j] = r[j].x;
          SX[j] = r[j].y;
        }
      }
      __syncthreads();
    }
  }
}

// ---- launchers (one launch over the generic instances ids[first, first + num)) ---------
MrArgs mr_args(const Layout1d& lay, int first) {
  MrArgs A;
  A.insts = lay.d_inst;
  A.ids = lay.d_ids + first;
  A.big = static_cast<cplx<double>*>(lay.mr_big);
  const long long len = lay.mr_tw_len;
  const char* base = static_cast<const char*>(lay.mr_tw);
  A.tw64 = reinterpret_cast<const cplx<double>*>(base);
  A.tw32 = reinterpret_cast<const cplx<float>*>(base + sizeof(cplx<double>) * len);
  A.twdf = reinterpret_cast<const cplx<df>*>(base + (sizeof(cplx<double>) + sizeof(cplx<float>)) * len);
  return A;
}

// Two transform buffers of the layout's largest generic n up to kMrSmemN, 16 bytes per
// entry.  The twiddle tables lie back to back (float64, float32, double-float; mr_tw_len
// entries each, an even count so that the double-float table starts on a 16-byte boundary).
size_t mr_smem(const Layout1d& lay) { return (size_t)2 * 16 * lay.mr_smem_n; }

template <typename K>
cudaError_t mr_attr(K k, size_t sm) {
  return raise_smem(k, sm);
}

}  // namespace

bool mr_in_smem(int n) { return n <= kMrSmemN; }

bool mr_size_ok(int n) {
  MrPlan P;
  return n >= 6 && n <= kMrMaxN && (n & (n - 1)) != 0 && mr_plan(n, P);
}

long long mr_twiddle_len(int n) { return n - 1; }

cudaError_t mr_twiddles_init(int n, long long off, const Layout1d& lay, cudaStream_t s) {
  const MrArgs A = mr_args(lay, 0);
  k_mr_twiddles<<<(n + 255) / 256, 256, 0, s>>>(
      n, const_cast<cplx<double>*>(A.tw64) + off, const_cast<cplx<float>*>(A.tw32) + off,
      const_cast<cplx<df>*>(A.twdf) + off);
  return cudaGetLastError();
}

cudaError_t mr_launch_deriv(const Layout1d& lay, int first, int num, const double* f,
                            double* fx, cudaStream_t s) {
  const size_t sm = mr_smem(lay);
  cudaError_t e = mr_attr(k_mr_deriv, sm);
  if (e) return e;
  k_mr_deriv<<<num, kMrNT, sm, s>>>(mr_args(lay, first), f, fx);
  return cudaGetLastError();
}

cudaError_t mr_launch_apply_G(const Layout1d& lay, int first, int num, const double* eta,
                              const double* hx, const double* u, double* Gu, cudaStream_t s) {
  const size_t sm = mr_smem(lay);
  cudaError_t e = mr_attr(k_mr_apply_G, sm);
  if (e) return e;
  k_mr_apply_G<<<num, kMrNT, sm, s>>>(mr_args(lay, first), eta, hx, u, Gu);
  return cudaGetLastError();
}

cudaError_t mr_launch_precond(const Layout1d& lay, int first, int num, const SolveRec* rec,
                              const double* r, double* z, cudaStream_t s) {
  const size_t sm = mr_smem(lay);
  cudaError_t e = mr_attr(k_mr_precond, sm);
  if (e) return e;
  k_mr_precond<<<num, kMrNT, sm, s>>>(mr_args(lay, first), rec, r, z);
  return cudaGetLastError();
}

cudaError_t mr_launch_pcg(const Layout1d& lay, int first, int num, int precision,
                          const double* eta, const double* hx, const double* b, double* x,
                          const SolveRec* given, int kind, double rtol, double rtol_inner,
                          int maxit, int max_refine, SolveRec* rec, void* ws, void* ux,
                          cudaStream_t s) {
  MrPcgArgs a;
  a.ux = ux;
  a.eta = eta;
  a.hx = hx;
  a.b = b;
  a.x = x;
  a.given = given;
  a.kind = kind;
  a.rtol = rtol;
  a.rtol_inner = rtol_inner;
  a.maxit = maxit;
  a.max_refine = max_refine;
  a.rec = rec;
  a.ws = static_cast<cplx<double>*>(ws);
  const size_t sm = mr_smem(lay);
  cudaError_t e;
  if (precision == SGN_PREC_MIXED) {
    if ((e = mr_attr(k_mr_pcg<true>, sm))) return e;
    k_mr_pcg<true><<<num, kMrNT, sm, s>>>(mr_args(lay, first), a);
  } else {
    if ((e = mr_attr(k_mr_pcg<false>, sm))) return e;
    k_mr_pcg<false><<<num, kMrNT, sm, s>>>(mr_args(lay, first), a);
  }
  return cudaGetLastError();
}

cudaError_t mr_launch_rhs(const Layout1d& lay, int first, int num, int precision, double g,
                          const double* eta, const double* u, const double* h,
                          const double* hx, double* f_eta, double* f_U, double* scratch,
                          bool ux_given, cudaStream_t s) {
  const size_t sm = mr_smem(lay);
  auto go = [&](auto k) -> cudaError_t {
    const cudaError_t e = mr_attr(k, sm);
    if (e) return e;
    k<<<num, kMrNT, sm, s>>>(mr_args(lay, first), g, eta, u, h, hx, f_eta, f_U, scratch,
                             lay.points);
    return cudaGetLastError();
  };
  if (precision == SGN_PREC_MIXED) return ux_given ? go(k_mr_rhs<df, true>) : go(k_mr_rhs<df, false>);
  return ux_given ? go(k_mr_rhs<double, true>) : go(k_mr_rhs<double, false>);
}

}  // namespace sgn
