// 1d kernels for n = 2^8 .. 2^14 on the split transforms of sgn_split_fft.cuh: the constraint
// solve (a5/a6, float64 and mixed), the right-hand side (a7) and the SBDF2 velocity update
// (a10).  One instance is held by 1, 2, 4 or 8 CTAs of a thread-block cluster; the launchers
// choose the number by the load (split_lcl), and every choice gives bitwise the same result.
//
// What bounds them: an instance's data is on chip, so time is the issue of its SMs plus one
// barrier per transform stage and the cluster barriers (n = 8192 in a batch that fills the GPU:
// the mixed solve issues in 39 % of cycles and waits at those barriers first, the right-hand
// side in 53 %).  The float64 kernels are bound by the float64 pipe (0.5 lanes
// per clock for a warp's own sub-partition, 1.7 per SM): a thread holds 2 or 4 elements, so
// that even n = 256 spreads over all four sub-partitions, the coefficients, symbols and
// wavenumber factors are formed once per solve, and no division is left in the iteration
// (14.5 float64 instructions per point and iteration beside the transforms).
//
// Against one CTA per instance of sgn_1d_pcg.cuh's kind (one GB300): a float64 solve at n = 256
// 1164 -> 426 us, a batch of 64 float64 instances (512 .. 8192, 2 RK4 steps) 40.2 -> 9.9 ms,
// 24 mixed AB4 steps at n = 4096 11.8 -> 5.7 ms, 32 SBDF2 steps 10.0 -> 4.3 ms, the mixed
// ensemble of 256 (4 RK4 steps) 12.2 -> 10.0 ms.
#pragma once
#include "sgn_1d_pcg.cuh"
#include "sgn_1d_rhs.cuh"
#include "sgn_split_fft.cuh"

namespace sgn {
namespace sp {

using d1::kPi;

template <int L>
using Plan64 = Plan<L, 1 << split_log_e(L, false)>;
template <int L>
using PlanMx = Plan<L, 1 << split_log_e(L, true)>;
// CTAs of 256 threads per SM that the registers leave room for.  3 (80 registers) for the mixed
// solve and the double-float right-hand side: a batch that fills the GPU hides more latency
// (ensemble of 256, 4 RK4 steps: 11.15 ms with 2, 10.25 with 3, 10.50 with 4, which spills),
// a single instance loses a few per cent.  2 (128 registers) for the others.
#define SGN_SPLIT_BOUNDS(PL, CTAS) \
  __launch_bounds__(PL::kMaxNT, PL::kMaxNT > 256 ? 1 : CTAS)

// ---- sums over the instance ---------------------------------------------------------------
__device__ __forceinline__ df shfl_x(df v, int o) {
  return df(__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o));
}
__device__ __forceinline__ double shfl_x(double v, int o) {
  return __shfl_xor_sync(0xffffffffu, v, o);
}

// Lane 0's sum.  A double-float sum is symmetric in its operands only for finite values; were
// the lanes' sums taken, inputs that overflow could send the CTAs of a cluster different
// ways, past each other's barriers.
__device__ __forceinline__ df lane0(df v) {
  return df(__shfl_sync(0xffffffffu, v.hi, 0), __shfl_sync(0xffffffffu, v.lo, 0));
}
template <typename V>
__device__ __forceinline__ V lane0(V v) {
  return v;                              // commutative
}

// Sum over all threads of the instance: per warp by a shuffle tree, then over its W warps (of
// all CTAs, in the order of T) by warp 0 of every CTA, whose lane 0 runs fin(total).  slots:
// [2][W], the two halves used in turn (a half is written again only after a barrier that
// follows its last reading).  sum_put before a cluster-wide barrier, sum_take after it, and a
// CTA barrier before the others read what fin left.
template <typename PL, typename V>
__device__ __forceinline__ void sum_put(V a, V* s, const Geo<PL>& g) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a = a + shfl_x(a, o);
  a = lane0(a);                          // every CTA gets the same bits
  const int lane = threadIdx.x & 31;
  if (lane < (1 << g.lcl))
    at_rank(s, lane, g.lcl)[((g.rank << g.lNT) + (int)threadIdx.x) >> 5] = a;
  __syncwarp();
}
template <typename PL, typename V, typename Fin>
__device__ __forceinline__ void sum_take(const V* s, Fin fin) {
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    V r = s[lane & (PL::W - 1)];
#pragma unroll
    for (int i = 32; i < PL::W; i += 32) r = r + s[i + lane];
#pragma unroll
    for (int o = (PL::W < 32 ? PL::W : 32) / 2; o > 0; o >>= 1) r = r + shfl_x(r, o);
    if (lane == 0) fin(r);
    __syncwarp();
  }
}
template <typename PL, typename V, typename Fin>
__device__ __forceinline__ void reduce(V a, V* slots, int& half_, const Geo<PL>& g, Fin fin) {
  V* s = slots + half_ * PL::W;
  sum_put<PL>(a, s, g);
  cta_or_cluster_sync(g.lcl);
  sum_take<PL>(s, fin);
  __syncthreads();
  half_ ^= 1;
}
// ---- a1: coefficients -----------------------------------------------------------------------
// Maxima of non-negative doubles by their bits (integer compares; a float64 compare costs 64
// clocks per warp here).
struct Extrema {
  unsigned long long nmin, emax, gmax, sopt;   // ~bits of eta_min, bits of the maxima
};
__device__ __forceinline__ unsigned long long umax(unsigned long long a, unsigned long long b) {
  return a > b ? a : b;
}
__device__ __forceinline__ Extrema operator+(Extrema a, Extrema b) {
  return Extrema{umax(a.nmin, b.nmin), umax(a.emax, b.emax), umax(a.gmax, b.gmax),
                 umax(a.sopt, b.sopt)};
}
__device__ __forceinline__ Extrema shfl_x(Extrema v, int o) {
  return Extrema{__shfl_xor_sync(0xffffffffu, v.nmin, o), __shfl_xor_sync(0xffffffffu, v.emax, o),
                 __shfl_xor_sync(0xffffffffu, v.gmax, o), __shfl_xor_sync(0xffffffffu, v.sopt, o)};
}
constexpr unsigned long long kBad = ~0ull;     // gmax of an instance with a bad point

__device__ __forceinline__ Extrema extrema_of(double e, double gx) {
  const unsigned long long eb = (unsigned long long)__double_as_longlong(e);
  const unsigned long long gb =
      (unsigned long long)__double_as_longlong(gx) & 0x7fffffffffffffffull;
  // eta <= 0, NaN (sign set, zero or above infinity), or |h_x| not below 1e150
  const bool bad = eb - 1ull >= 0x7ff0000000000000ull || gb >= 0x5f138d352e5096afull;
  const double s = fma(d1::kLambdaPlus * e, gx * gx, e);
  return Extrema{~eb, eb, bad ? kBad : gb, (unsigned long long)__double_as_longlong(s)};
}

struct Setup {           // per instance, formed by one thread
  SolveRec R;
  double kunit;
  df kh;
  float kf, sigf, alf;
};

__device__ inline void make_setup(const Extrema& x, const SolveRec* given, int kind, double L,
                                  Setup& S) {
  SolveRec R = {};
  if (given) {
    R = *given;
    R.status = SGN_OK;
  } else {
    const double emax = __longlong_as_double((long long)x.emax);
    const double gmax = __longlong_as_double((long long)x.gmax);
    R.eta_min = __longlong_as_double((long long)~x.nmin);
    R.eta_max = emax;
    if (x.gmax == kBad) {
      R.status = SGN_ERR_NONPOSITIVE_DEPTH;
    } else {
      const double e3 = emax * emax * emax;
      R.flat = gmax <= d1::kFlatSlope;
      R.status = SGN_OK;
      if (R.flat) {
        R.sigma = emax;
        R.alpha = e3 / 3.0;
      } else {
        R.sigma = kind == SGN_COEF_OPT ? __longlong_as_double((long long)x.sopt)
                                       : emax * (1.0 + d1::kLambdaPlus * gmax * gmax);
        R.alpha = d1::kLambdaPlus * e3;
      }
    }
  }
  R.iters = 0;
  R.refinements = 0;
  R.ratio = 0.0;
  S.R = R;
  S.kunit = 2.0 * kPi / L;
  S.kh = df(S.kunit);
  S.kf = (float)S.kunit;
  S.sigf = (float)R.sigma;
  S.alf = (float)R.alpha;
}

// Stage twiddles w_N^m from the table of e^{-2 pi i j / 2^kTwiddleLog2}
template <int LN, typename T>
__device__ __forceinline__ void fill_tw(cplx<T>* w, const cplx<T>* __restrict__ tw, int nt) {
  for (int m = threadIdx.x; m < (1 << LN); m += nt) w[m] = tw[m << (kTwiddleLog2 - LN)];
}

// a double-float kept as the bits of a double (the solve's x before it is final)
__device__ __forceinline__ double pack_df(df v) {
  return __hiloint2double(__float_as_int(v.lo), __float_as_int(v.hi));
}
__device__ __forceinline__ df unpack_df(double d) {
  return df(__int_as_float(__double2loint(d)), __int_as_float(__double2hiint(d)));
}

// exact, subnormal parts included
__device__ __forceinline__ double f64(df v) { return (double)v.hi + (double)v.lo; }
// the root of a >= 0, and a / b rounded twice (48 bits)
__device__ __forceinline__ df root(df a) {
  const float r = sqrtf(a.hi);
  return df(r, r > 0.0f ? 0.5f * (fmaf(-r, r, a.hi) + a.lo) / r : 0.0f);
}
__device__ __forceinline__ df quot_df(df a, df b) {
  const float q = a.hi / b.hi;
  return df(q, (a - b * df(q, 0.0f)).hi / b.hi);
}

// ---- solve, mixed precision ---------------------------------------------------------------
struct MixedScalars {
  df bb, rz2, unscale;      // b.A^{-1}b; r.A^{-1}r and its root
  float tol;                // rtol ||b||_{A^{-1}}
  float scale, tin2;        // 1 / ||r||_{A^{-1}}; (inner tolerance)^2
  int go, status;
  float rz, alpha, beta;    // inner solve
  int state;                // 0 iterate, 1 converged, 2 breakdown, 3 iteration cap
};

template <typename PL>
struct SmemMixed {
  static constexpr size_t tabs = (size_t)(PL::N1 + PL::N2) * 24 + (size_t)2 * PL::W * 8;
  static size_t bytes(int lcl) { return tabs + ((size_t)40 << (PL::L - lcl)); }
};

// Iterative refinement as in sgn_1d_pcg.cuh (k_pcg1d): double-float residual, float32 PCG.  r,
// p and the correction d stay in registers; x^ and b^ in the workspace (slots 1 and 0).
template <typename PL>
__global__ void SGN_SPLIT_BOUNDS(PL, 3)
    k_solve_mixed(const __grid_constant__ PcgArgs A, int first, int lcl) {
  using SL = Slot<PL>;
  constexpr int n = PL::n, E = PL::E, RP = PL::RP, h = n / 2, PS = n / E, NYQ = PL::NYQ;
  // 128: the partners' stores travel by 128-byte lines (n = 4096, 24 AB4 steps: 5.65 ms, 5.71
  // with the buffers 32 bytes off)
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ Setup st;
  __shared__ MixedScalars sc;
  __shared__ Extrema exs[PL::W];
  const int NT = 1 << (PL::LNTA - lcl), NL = n >> lcl;
  unsigned char* q0 = smem;
  auto take = [&](size_t b) {
    unsigned char* p = q0;
    q0 += b;
    return p;
  };
  unsigned char* bA = take((size_t)16 * NL);
  unsigned char* bB = take((size_t)16 * NL);
  float2* eh = reinterpret_cast<float2*>(take((size_t)8 * NL));     // eta, h_x of the points
  cplx<df>* wAh = reinterpret_cast<cplx<df>*>(take(16 * PL::N1));
  cplx<df>* wBh = reinterpret_cast<cplx<df>*>(take(16 * PL::N2));
  cplx<float>* wAf = reinterpret_cast<cplx<float>*>(take(8 * PL::N1));
  cplx<float>* wBf = reinterpret_cast<cplx<float>*>(take(8 * PL::N2));
  df* slots = reinterpret_cast<df*>(take((size_t)2 * PL::W * 8));
  const Bufs<df> MH{reinterpret_cast<cplx<df>*>(bA), reinterpret_cast<cplx<df>*>(bB), wAh, wBh};
  const Bufs<float> MF{reinterpret_cast<cplx<float>*>(bA), reinterpret_cast<cplx<float>*>(bB), wAf,
                       wBf};
  const int t = threadIdx.x;
  const Geo<PL> g(t, lcl ? (int)cluster_rank() : 0, lcl);
  const bool ts = g.t0;
  int hb = 0;
  const int id = A.ids[first + (blockIdx.x >> lcl)];
  const long long off = A.insts[id].off, wso = A.insts[id].ws;
  const double* eta = A.eta + off;
  const double* hx = A.hx + off;
  const double* b = A.b + off;
  double* x = A.x + off;
  df* ux = A.ux ? static_cast<df*>(A.ux) + off : nullptr;
  float* cdf = A.coef_df + 6 * off;
  cplx<df>* Bh = reinterpret_cast<cplx<df>*>(A.ws + wso);
  cplx<df>* Xh = reinterpret_cast<cplx<df>*>(A.ws + wso + (h + 1));

  // ---- tables, coefficients (a1), double-float and float32 forms of eta, h_x
  fill_tw<PL::L1>(wAh, A.twdf, NT);
  fill_tw<PL::L2>(wBh, A.twdf, NT);
  for (int m = t; m < PL::N1; m += NT) {
    const cplx<df> w = A.twdf[m << (kTwiddleLog2 - PL::L1)];
    wAf[m] = mk(w.x.hi, w.y.hi);
  }
  for (int m = t; m < PL::N2; m += NT) {
    const cplx<df> w = A.twdf[m << (kTwiddleLog2 - PL::L2)];
    wBf[m] = mk(w.x.hi, w.y.hi);
  }
  cplx<df> v[E];
  {
    Extrema ex{0, 0, 0, 0};
    const df third(0.3333333432674408f, -9.934107758624577e-09f);   // 1/3
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int j = g.pt + e * PS;
      const double ed = eta[j], gd = hx[j];
      ex = ex + extrema_of(ed, gd);
      const df ef(ed), gf(gd), e2 = ef * ef;
      const df c[3] = {ef + ef * gf * gf, half(e2 * gf), e2 * ef * third};
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        cdf[q * n + j] = c[q].hi;
        cdf[(3 + q) * n + j] = c[q].lo;
      }
      eh[e * NT + t] = make_float2(ef.hi, gf.hi);
      v[e] = mk(df(b[j]), df(x[j]));
    }
    if (lcl) cluster_sync();             // the partners have started: their memory may be written
    int h0 = 0;
    reduce<PL>(ex, exs, h0, g, [&](const Extrema& m) {
      make_setup(m, A.given ? A.given + id : nullptr, A.kind, A.insts[id].L, st);
    });
  }
  if (st.R.status != SGN_OK) {
    if (ts) A.rec[id] = st.R;
    if (lcl) cluster_sync();
    return;
  }
  const float kf = st.kf, sigf = st.sigf, alf = st.alf, dN = recip(sigf);
  const df kh = st.kh;
  auto dinv = [&](int m) {
    const float k = kf * (float)m;
    return recip(sigf + alf * k * k);
  };
  auto xth = [&](int e) { return A.twdf[cross_index(g, e) << (kTwiddleLog2 - PL::L)]; };
  cplx<float> xf[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const cplx<df> w = xth(e);
    xf[e] = mk(w.x.hi, w.y.hi);
  }
  auto xtf = [&](int e) { return xf[e]; };

  // ---- b^ and x0^ from one transform of b + i x0
  fft_fwd<PL>(MH, g, v, xth);
  {
    float bb = 0.0f;
#pragma unroll
    for (int q = 0; q < RP; ++q) {
      const int m = g.mode(SL::b(q), SL::s(q));
      const cplx<df> y = v[SL::reg(q)], ym = conj(mirror_get<PL>(v, ts, SL::b(q), SL::s(q)));
      const cplx<df> s = y + ym, d = mul_mi(y - ym);
      const cplx<df> bh = mk(half(s.x), half(s.y));
      Bh[m] = bh;
      Xh[m] = mk(half(d.x), half(d.y));
      bb += ((ts && q == 0) ? 1.0f : 2.0f) * (bh.x.hi * bh.x.hi + bh.y.hi * bh.y.hi) * dinv(m);
    }
    if (ts) {
      const cplx<df> y = v[NYQ];
      Bh[h] = mk(y.x, df(0.0f, 0.0f));
      Xh[h] = mk(y.y, df(0.0f, 0.0f));
      bb += y.x.hi * y.x.hi * dN;
    }
    reduce<PL>(df(bb, 0.0f), slots, hb, g, [&](df s) {
      sc.bb = s;
      sc.tol = (float)A.rtol * sqrtf(s.hi);
    });
  }
  const float bb = sc.bb.hi;
  const df zero(0.0f, 0.0f);
  if (!(bb > 0.0f)) {                    // x = 0, and its derivative for the right-hand side
#pragma unroll
    for (int e = 0; e < E; ++e) {
      x[g.pt + e * PS] = 0.0;
      if (ux) ux[g.pt + e * PS] = zero;
    }
    if (ts) {
      st.R.status = bb == 0.0f ? SGN_OK : SGN_ERR_BREAKDOWN;
      A.rec[id] = st.R;
    }
    if (lcl) cluster_sync();
    return;
  }

  const df inv_n(1.0f / (float)n, 0.0f);                              // exact
  const float inv_nf = 1.0f / (float)n;
  const df one(1.0f, 0.0f);
  int iters = 0, status = SGN_OK, refinements = 0;
  for (;;) {
    // ---- double-float residual r^ = b^ - (G x)^, keeping the real-space x on the way
    cplx<float> r[RP], rN = mk(0.0f, 0.0f);
    {
#pragma unroll
      for (int q = 0; q < RP; ++q) {
        const int m = g.mode(SL::b(q), SL::s(q));
        const df k = kh * df((float)m, 0.0f);
        const cplx<df> xv = Xh[m];
        if (ts && q == 0) {
          v[0] = mk(xv.x, zero);
        } else {
          v[SL::reg(q)] = xv * (one - k);
          mirror_set<PL>(v, ts, SL::b(q), SL::s(q), conj(xv) * (one + k));
        }
      }
      if (ts) v[NYQ] = mk(Xh[h].x, zero);
      fft_inv<PL>(MH, g, v, xth);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int j = g.pt + e * PS;
        const df pv = v[e].x * inv_n, px = v[e].y * inv_n;
        x[j] = pack_df(pv);
        if (ux) ux[j] = px;
        const df c1(cdf[j], cdf[3 * n + j]), c2(cdf[n + j], cdf[4 * n + j]),
            c3(cdf[2 * n + j], cdf[5 * n + j]);
        v[e] = mk(dot2(c1, pv, c2, px), dot2(c2, pv, c3, px));
      }
      fft_fwd<PL>(MH, g, v, xth);
      float rz = 0.0f;
#pragma unroll
      for (int q = 0; q < RP; ++q) {
        const int m = g.mode(SL::b(q), SL::s(q));
        const df k = kh * df((float)m, 0.0f), k0 = one - k, k1 = one + k;
        const cplx<df> y = v[SL::reg(q)], ym = conj(mirror_get<PL>(v, ts, SL::b(q), SL::s(q)));
        const df sx = dot2(y.x, k0, ym.x, k1), sy = dot2(y.y, k0, ym.y, k1);
        const cplx<df> rr = Bh[m] - mk(half(sx), half(sy));
        r[q] = mk(rr.x.hi + rr.x.lo, rr.y.hi + rr.y.lo);
        rz += ((ts && q == 0) ? 1.0f : 2.0f) * (r[q].x * r[q].x + r[q].y * r[q].y) * dinv(m);
      }
      if (ts) {
        const df rr = Bh[h].x - v[NYQ].x;
        rN = mk(rr.hi + rr.lo, 0.0f);
        rz += rN.x * rN.x * dN;
      }
      // one thread decides the pass: converged (r.A^{-1}r against rtol^2 b.A^{-1}b, which may
      // leave the float32 range: in float64 unless the first is clearly above), out of budget,
      // or the next inner solve
      reduce<PL>(df(rz, 0.0f), slots, hb, g, [&](df s) {
        sc.rz2 = s;
        sc.go = 0;
        sc.status = status;
        if ((!(s.hi > 2.0f * (sc.tol * sc.tol)) && f64(s) <= A.rtol * A.rtol * f64(sc.bb)) ||
            status != SGN_OK)
          return;
        if (refinements >= A.max_refine || iters >= A.maxit) {
          sc.status = SGN_ERR_NOT_CONVERGED;
          return;
        }
        const df nr = root(s);
        const float in = recip(nr.hi), tin = fminf(0.1f, fmaxf(1e-6f, 0.3f * (in * sc.tol)));
        sc.tin2 = A.rtol_inner > 0.0 ? (float)(A.rtol_inner * A.rtol_inner) : tin * tin;
        sc.unscale = nr;
        sc.scale = in;
        sc.go = 1;
      });
    }
    status = sc.status;
    if (!sc.go) break;
    const float scale = sc.scale, tin2 = sc.tin2;

    // ---- float32 PCG for G d = r / ||r||
    const int it_before = iters;
    int st_in = SGN_OK;
    cplx<float> p[RP], d[RP];
    float pN = 0.0f, dNy = 0.0f;
    float dv[RP];                        // 1 / (sigma + alpha k^2) of the slots
    {
      float loc = 0.0f;
#pragma unroll
      for (int q = 0; q < RP; ++q) {
        dv[q] = dinv(g.mode(SL::b(q), SL::s(q)));
        r[q] = r[q] * scale;
        p[q] = r[q] * dv[q];
        d[q] = mk(0.0f, 0.0f);
        loc += ((ts && q == 0) ? 1.0f : 2.0f) * (r[q].x * p[q].x + r[q].y * p[q].y);
      }
      if (ts) {
        rN = rN * scale;
        pN = rN.x * dN;
        loc += rN.x * pN;
      }
      reduce<PL>(df(loc, 0.0f), slots, hb, g, [&](df s) {
        const float rz = s.hi + s.lo;
        sc.rz = rz;
        sc.state = (rz <= tin2) ? 1 : (iters >= A.maxit ? 3 : 0);
      });
    }
    for (;;) {
      const int state = sc.state;
      if (state != 0) {
        if (state == 3) st_in = SGN_ERR_NOT_CONVERGED;
        if (state == 2) st_in = SGN_ERR_BREAKDOWN;
        break;
      }
      Geo<PL> gi = g;
      // addresses are formed anew in each iteration: kept across it, they spill
      asm volatile("" : "+r"(gi.t), "+r"(gi.ap0), "+r"(gi.ap1));
      cplx<float> w[E];
#pragma unroll
      for (int q = 0; q < RP; ++q) {
        const float k = kf * (float)g.mode(SL::b(q), SL::s(q));
        if (ts && q == 0) {
          w[0] = mk(p[0].x, 0.0f);
        } else {
          w[SL::reg(q)] = p[q] * (1.0f - k);
          mirror_set<PL>(w, ts, SL::b(q), SL::s(q), conj(p[q]) * (1.0f + k));
        }
      }
      if (ts) w[NYQ] = mk(pN, 0.0f);
      fft_inv<PL>(MF, gi, w, xtf);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const float pv = w[e].x * inv_nf, px = w[e].y * inv_nf;
        const float2 eg = eh[e * NT + t];
        const float et = eg.x, gx = eg.y, e2 = et * et;
        const float c1 = fmaf(et * gx, gx, et), c2 = 0.5f * e2 * gx, c3 = e2 * et * (1.0f / 3.0f);
        w[e] = mk(c1 * pv + c2 * px, c2 * pv + c3 * px);
      }
      fft_fwd<PL>(MF, gi, w, xtf);
      cplx<float> gq[RP];
      float gN = 0.0f, pq_loc = 0.0f;
#pragma unroll
      for (int q = 0; q < RP; ++q) {
        const float k = kf * (float)g.mode(SL::b(q), SL::s(q));
        const cplx<float> y = w[SL::reg(q)], ym = conj(mirror_get<PL>(w, ts, SL::b(q), SL::s(q)));
        const cplx<float> s = y * (1.0f - k) + ym * (1.0f + k);
        gq[q] = mk(0.5f * s.x, 0.5f * s.y);
        pq_loc += ((ts && q == 0) ? 1.0f : 2.0f) * (p[q].x * gq[q].x + p[q].y * gq[q].y);
      }
      if (ts) {
        gN = w[NYQ].x;
        pq_loc += pN * gN;
      }
      reduce<PL>(df(pq_loc, 0.0f), slots, hb, g, [&](df s) {
        const float pq = s.hi + s.lo;
        if (!(pq > 0.0f) || !isfinite(pq)) sc.state = 2;
        else sc.alpha = sc.rz / pq;
      });
      if (sc.state == 2) {
        st_in = SGN_ERR_BREAKDOWN;
        break;
      }
      const float at = sc.alpha;
      float rz_loc = 0.0f;
#pragma unroll
      for (int q = 0; q < RP; ++q) {
        d[q] = d[q] + p[q] * at;
        r[q] = r[q] - gq[q] * at;
        rz_loc += ((ts && q == 0) ? 1.0f : 2.0f) * (r[q].x * r[q].x + r[q].y * r[q].y) * dv[q];
      }
      if (ts) {
        dNy += pN * at;
        rN.x -= gN * at;
        rz_loc += rN.x * rN.x * dN;
      }
      ++iters;
      reduce<PL>(df(rz_loc, 0.0f), slots, hb, g, [&](df s) {
        const float rz = s.hi + s.lo;
        if (!isfinite(rz)) {
          sc.state = 2;
        } else {
          sc.beta = rz / sc.rz;
          sc.rz = rz;
          sc.state = (rz <= tin2) ? 1 : (iters >= A.maxit ? 3 : 0);
        }
      });
      if (sc.state == 2) {
        st_in = SGN_ERR_BREAKDOWN;
        break;
      }
      const float beta = sc.beta;
#pragma unroll
      for (int q = 0; q < RP; ++q) p[q] = r[q] * dv[q] + p[q] * beta;
      if (ts) pN = rN.x * dN + pN * beta;
    }
    // A float32 breakdown after some progress only means float32 has resolved what it can:
    // keep the correction and let the next refinement pass decide.
    if (st_in == SGN_ERR_BREAKDOWN && iters == it_before) status = SGN_ERR_BREAKDOWN;
    ++refinements;
    const df unscale = sc.unscale;
#pragma unroll
    for (int q = 0; q < RP; ++q) {
      const int m = g.mode(SL::b(q), SL::s(q));
      const cplx<df> xv = Xh[m];
      Xh[m] = mk(xv.x + df(d[q].x, 0.0f) * unscale, xv.y + df(d[q].y, 0.0f) * unscale);
    }
    if (ts) Xh[h] = mk(Xh[h].x + df(dNy, 0.0f) * unscale, zero);
  }
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int j = g.pt + e * PS;
    x[j] = to_f64(unpack_df(x[j]));
  }
  if (ts) {
    SolveRec R = st.R;
    R.ratio = f64(quot_df(root(sc.rz2), root(sc.bb)));
    R.refinements = refinements;
    R.iters = iters;
    R.status = status;
    A.rec[id] = R;
  }
  if (lcl) cluster_sync();               // shared memory outlives the partners' last use of it
}

// ---- solve, float64 -----------------------------------------------------------------------
struct Scalars64 {
  double bb, rz, at, beta, tol, tol2;
  int state;                // 0 iterate, 2 breakdown
};
template <typename PL>
struct Smem64 {
  static constexpr size_t tabs = (size_t)(PL::N1 + PL::N2) * 16 + (size_t)2 * PL::W * 8;
  static size_t bytes(int lcl) { return tabs + ((size_t)64 << (PL::L - lcl)); }
};

template <typename PL>
__global__ void SGN_SPLIT_BOUNDS(PL, 2)
    k_solve64(const __grid_constant__ PcgArgs A, int first, int lcl) {
  using SL = Slot<PL>;
  constexpr int n = PL::n, E = PL::E, RP = PL::RP, h = n / 2, PS = n / E, NYQ = PL::NYQ;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Setup st;
  __shared__ Scalars64 sc;
  __shared__ Extrema exs[PL::W];
  const int NT = 1 << (PL::LNTA - lcl), NL = n >> lcl;
  unsigned char* q0 = smem;
  auto take = [&](size_t b) {
    unsigned char* p = q0;
    q0 += b;
    return p;
  };
  cplx<double>* bA = reinterpret_cast<cplx<double>*>(take((size_t)16 * NL));
  cplx<double>* bB = reinterpret_cast<cplx<double>*>(take((size_t)16 * NL));
  cplx<double>* xs = reinterpret_cast<cplx<double>*>(take((size_t)8 * NL));   // x^ [RP][NT]
  double* cs = reinterpret_cast<double*>(take((size_t)24 * NL));              // c1, c2, c3 / 2n
  cplx<double>* wA = reinterpret_cast<cplx<double>*>(take(16 * PL::N1));
  cplx<double>* wB = reinterpret_cast<cplx<double>*>(take(16 * PL::N2));
  double* slots = reinterpret_cast<double*>(take((size_t)2 * PL::W * 8));
  const Bufs<double> M{bA, bB, wA, wB};
  const int t = threadIdx.x;
  const Geo<PL> g(t, lcl ? (int)cluster_rank() : 0, lcl);
  const bool ts = g.t0;
  int hb = 0;
  const int id = A.ids[first + (blockIdx.x >> lcl)];
  const long long off = A.insts[id].off;
  const double* eta = A.eta + off;
  const double* hx = A.hx + off;
  const double* b = A.b + off;
  double* x = A.x + off;
  double* ux = A.ux ? static_cast<double*>(A.ux) + off : nullptr;

  fill_tw<PL::L1>(wA, A.tw64, NT);
  fill_tw<PL::L2>(wB, A.tw64, NT);
  cplx<double> v[E];
  {
    Extrema ex{0, 0, 0, 0};
    constexpr double sc2n = 0.5 / (double)n;                          // exact
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int j = g.pt + e * PS;
      const double ed = eta[j], gd = hx[j], e2 = ed * ed;
      ex = ex + extrema_of(ed, gd);
      cs[e * NT + t] = ed * (1.0 + gd * gd) * sc2n;
      cs[(E + e) * NT + t] = 0.5 * e2 * gd * sc2n;
      cs[(2 * E + e) * NT + t] = e2 * ed * (1.0 / 3.0) * sc2n;
      v[e] = mk(b[j], x[j]);
    }
    if (lcl) cluster_sync();             // the partners have started: their memory may be written
    int h0 = 0;
    reduce<PL>(ex, exs, h0, g, [&](const Extrema& m) {
      make_setup(m, A.given ? A.given + id : nullptr, A.kind, A.insts[id].L, st);
    });
  }
  if (st.R.status != SGN_OK) {
    if (ts) A.rec[id] = st.R;
    if (lcl) cluster_sync();
    return;
  }
  auto xt = [&](int e) { return A.tw64[cross_index(g, e) << (kTwiddleLog2 - PL::L)]; };
  // per slot: 1 - k and 1 + k, and the weighted and plain symbol of A^{-1}
  double km[RP], kp[RP], dv[RP];
#pragma unroll
  for (int q = 0; q < RP; ++q) {
    const double k = st.kunit * (double)g.mode(SL::b(q), SL::s(q));
    km[q] = 1.0 - k;
    kp[q] = 1.0 + k;
    dv[q] = 1.0 / fma(st.R.alpha * k, k, st.R.sigma);
  }
  const double dN = 1.0 / st.R.sigma;
  const double wt0 = ts ? 1.0 : 2.0;     // Parseval weight of slot 0 (mode 0 counts once)
  // real space from the half spectrum f(q), fN: v = n (f + i f_x) (with_k) or n f
  auto to_real = [&](auto f, double fN, bool with_k) {
#pragma unroll
    for (int q = 0; q < RP; ++q) {
      const cplx<double> p = f(q);
      if (ts && q == 0) {
        v[0] = mk(p.x, 0.0);
      } else {
        v[SL::reg(q)] = with_k ? p * km[q] : p;
        mirror_set<PL>(v, ts, SL::b(q), SL::s(q), conj(with_k ? p * kp[q] : p));
      }
    }
    if (ts) v[NYQ] = mk(fN, 0.0);
    fft_inv<PL>(M, g, v, xt);
  };
  // (G f)^ of the slots into gq, gN
  auto matvec = [&](auto f, double fN, cplx<double>* gq, double& gN) {
    to_real(f, fN, true);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const double c1 = cs[e * NT + t], c2 = cs[(E + e) * NT + t], c3 = cs[(2 * E + e) * NT + t];
      const double pv = v[e].x, px = v[e].y;
      v[e] = mk(c1 * pv + c2 * px, c2 * pv + c3 * px);
    }
    fft_fwd<PL>(M, g, v, xt);
#pragma unroll
    for (int q = 0; q < RP; ++q) {
      const cplx<double> y = v[SL::reg(q)], ym = conj(mirror_get<PL>(v, ts, SL::b(q), SL::s(q)));
      gq[q] = mk(y.x * km[q] + ym.x * kp[q], y.y * km[q] + ym.y * kp[q]);
    }
    gN = 2.0 * v[NYQ].x;
  };

  // ---- b^ and x0^ from one transform of b + i x0
  cplx<double> r[RP], p[RP];
  double rN = 0.0, pN = 0.0, xN = 0.0;
  fft_fwd<PL>(M, g, v, xt);
  {
    double bb = 0.0;
#pragma unroll
    for (int q = 0; q < RP; ++q) {
      const cplx<double> y = v[SL::reg(q)], ym = conj(mirror_get<PL>(v, ts, SL::b(q), SL::s(q)));
      const cplx<double> s = y + ym, d = mul_mi(y - ym);
      r[q] = mk(half(s.x), half(s.y));
      xs[q * NT + t] = mk(half(d.x), half(d.y));
      bb += (q == 0 ? wt0 : 2.0) * (r[q].x * r[q].x + r[q].y * r[q].y) * dv[q];
    }
    if (ts) {
      rN = v[NYQ].x;
      xN = v[NYQ].y;
      bb += rN * rN * dN;
    }
    reduce<PL>(bb, slots, hb, g, [&](double s) {
      sc.bb = s;
      sc.tol = A.rtol * sqrt(s);
      sc.tol2 = sc.tol * sc.tol;
    });
  }
  if (!(sc.bb > 0.0)) {                  // x = 0, and its derivative for the right-hand side
#pragma unroll
    for (int e = 0; e < E; ++e) {
      x[g.pt + e * PS] = 0.0;
      if (ux) ux[g.pt + e * PS] = 0.0;
    }
    if (ts) {
      st.R.status = sc.bb == 0.0 ? SGN_OK : SGN_ERR_BREAKDOWN;
      A.rec[id] = st.R;
    }
    if (lcl) cluster_sync();
    return;
  }
  int iters = 0, status = SGN_OK;
  // r = b - G x0, p = A^{-1} r
  {
    cplx<double> gq[RP];
    double gN, loc = 0.0;
    matvec([&](int q) { return xs[q * NT + t]; }, xN, gq, gN);
#pragma unroll
    for (int q = 0; q < RP; ++q) {
      r[q] = r[q] - gq[q];
      p[q] = r[q] * dv[q];
      loc += (q == 0 ? wt0 : 2.0) * (r[q].x * p[q].x + r[q].y * p[q].y);
    }
    if (ts) {
      rN -= gN;
      pN = rN * dN;
      loc += rN * pN;
    }
    reduce<PL>(loc, slots, hb, g, [&](double s) {
      sc.rz = s;
      sc.state = 0;
    });
  }
  // sqrt(rz) > rtol sqrt(bb), without the square root where the squares are in range
  auto above = [&]() {
    return sc.tol2 > 1e-290 ? sc.rz > sc.tol2 : sqrt(sc.rz) > sc.tol;
  };
  while (above()) {
    if (iters >= A.maxit) {
      status = SGN_ERR_NOT_CONVERGED;
      break;
    }
    cplx<double> gq[RP];
    double gN, pq = 0.0;
    matvec([&](int q) { return p[q]; }, pN, gq, gN);
#pragma unroll
    for (int q = 0; q < RP; ++q)
      pq += (q == 0 ? wt0 : 2.0) * (p[q].x * gq[q].x + p[q].y * gq[q].y);
    if (ts) pq += pN * gN;
    reduce<PL>(pq, slots, hb, g, [&](double s) {
      if (!(s > 0.0) || !isfinite(s)) sc.state = 2;
      else sc.at = sc.rz / s;
    });
    if (sc.state == 2) {
      status = SGN_ERR_BREAKDOWN;
      break;
    }
    const double at = sc.at;
    double rz = 0.0;
#pragma unroll
    for (int q = 0; q < RP; ++q) {
      xs[q * NT + t] = xs[q * NT + t] + p[q] * at;
      r[q] = r[q] - gq[q] * at;
      rz += (q == 0 ? wt0 : 2.0) * (r[q].x * r[q].x + r[q].y * r[q].y) * dv[q];
    }
    if (ts) {
      xN += pN * at;
      rN -= gN * at;
      rz += rN * rN * dN;
    }
    ++iters;
    reduce<PL>(rz, slots, hb, g, [&](double s) {
      if (!isfinite(s)) {
        sc.state = 2;
      } else {
        sc.beta = s / sc.rz;
        sc.rz = s;
      }
    });
    if (sc.state == 2) {
      status = SGN_ERR_BREAKDOWN;
      break;
    }
    const double beta = sc.beta;
#pragma unroll
    for (int q = 0; q < RP; ++q) p[q] = r[q] * dv[q] + p[q] * beta;
    if (ts) pN = rN * dN + pN * beta;
  }
  // x = F^{-1} x^; with ux, the transform of (1 - k) x^ (mirror (1 + k) conj x^), x + i x_x
  __syncthreads();
  to_real([&](int q) { return xs[q * NT + t]; }, xN, ux != nullptr);
  constexpr double inv_n = 1.0 / (double)n;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int j = g.pt + e * PS;
    x[j] = v[e].x * inv_n;
    if (ux) ux[j] = v[e].y * inv_n;
  }
  if (ts) {
    SolveRec R = st.R;
    R.ratio = sqrt(sc.rz / sc.bb);
    R.iters = iters;
    R.status = status;
    A.rec[id] = R;
  }
  if (lcl) cluster_sync();               // shared memory outlives the partners' last use of it
}

// ---- right-hand side ----------------------------------------------------------------------
// As rhs1d::rhs_body (sgn_1d_rhs.cuh): derivative pairs in T, each one forward and one inverse
// transform whose spectra never leave the registers.  m and zeta_x stay in shared memory, and
// with u_x not given d and s_x in the scratch planes 0 and 3.
template <typename PL>
struct SmemRhs {
  static constexpr size_t tabs = (size_t)(PL::N1 + PL::N2) * 16;
  static size_t bytes(int lcl) { return tabs + ((size_t)48 << (PL::L - lcl)); }
};

template <typename T>
__device__ __forceinline__ const cplx<T>* table_of(const cplx<double>* t64, const cplx<df>* tdf) {
  if constexpr (std::is_same<T, df>::value) return tdf;
  else return t64;
}

template <typename PL, typename T, bool UXG>
__global__ void SGN_SPLIT_BOUNDS(PL, (std::is_same<T, df>::value ? 3 : 2))
    k_rhs(const __grid_constant__ RhsArgs A, int first, int lcl) {
  constexpr int n = PL::n, E = PL::E, RP = PL::RP, PS = n / E;
  extern __shared__ __align__(16) unsigned char smem[];
  const int NT = 1 << (PL::LNTA - lcl), NL = n >> lcl, t = threadIdx.x;
  cplx<T>* bA = reinterpret_cast<cplx<T>*>(smem);
  cplx<T>* bB = bA + NL;
  T* sm = reinterpret_cast<T*>(bB + NL);                     // m, then the local part of f_U
  T* sz = sm + NL;                                           // zeta_x
  cplx<T>* wA = reinterpret_cast<cplx<T>*>(sz + NL);
  cplx<T>* wB = wA + PL::N1;
  const cplx<T>* tw = table_of<T>(A.tw64, A.twdf);
  const Bufs<T> M{bA, bB, wA, wB};
  const Geo<PL> g(t, lcl ? (int)cluster_rank() : 0, lcl);
  const Inst1d I = A.insts[A.ids[first + (blockIdx.x >> lcl)]];
  const double* eta = A.eta + I.off;
  const double* u = A.u + I.off;
  const double* hh = A.h + I.off;
  const double* hx = A.hx + I.off;
  T* sd = reinterpret_cast<T*>(A.scratch + I.off);                    // d = u_x
  T* ssx = reinterpret_cast<T*>(A.scratch + 3 * A.P + I.off);         // s_x
  fill_tw<PL::L1>(wA, tw, NT);
  fill_tw<PL::L2>(wB, tw, NT);
  __shared__ double kn_s;                // by one thread: a float64 division takes 640 clocks
  if (t == 0) kn_s = 2.0 * kPi / I.L * (1.0 / (double)n);
  const T third = num<T>(1.0 / 3.0), gT = num<T>(A.g);
  auto xt = [&](int e) { return tw[cross_index(g, e) << (kTwiddleLog2 - PL::L)]; };
  if (lcl) cluster_sync();               // the partners have started
  else __syncthreads();                  // the tables are filled
  const T kn = num<T>(kn_s);
  constexpr int passes = UXG ? 3 : 4;
  cplx<T> v[E];
#pragma unroll 1
  for (int pass = 0; pass < passes; ++pass) {
    const int what = UXG ? (pass == 0 ? 0 : pass == 1 ? 1 : 5) : (pass < 3 ? 2 + pass : 5);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int j = g.pt + e * PS;
      if (what == 0) {                   // (eta u, zeta)
        const T ej = num<T>(eta[j]);
        v[e] = mk(ej * num<T>(u[j]), ej - num<T>(hh[j]));
      } else if (what == 1) {            // (s, d)
        v[e] = mk(num<T>(hx[j]) * num<T>(u[j]), sd[j]);
      } else if (what == 2) {            // (u, eta u)
        const T uj = num<T>(u[j]);
        v[e] = mk(uj, num<T>(eta[j]) * uj);
      } else if (what == 3) {            // (zeta, s)
        v[e] = mk(num<T>(eta[j]) - num<T>(hh[j]), num<T>(hx[j]) * num<T>(u[j]));
      } else if (what == 4) {            // d
        v[e] = mk(sd[j], from_int<T>(0));
      } else {                           // Phi' (and the local part of f_U)
        const T ej = num<T>(eta[j]), uj = num<T>(u[j]), hj = num<T>(hx[j]);
        const T d = sd[j], m = sm[e * NT + t];
        const T dx = UXG ? v[e].y : v[e].x, sx = UXG ? v[e].x : ssx[j];
        const T s = hj * uj, Q = uj * dx - d * d, Sv = uj * sx, e2 = ej * ej, md = m * d;
        const T Phi = e2 * ej * Q * third + e2 * md + half(e2 * Sv) + ej * m * s - ej * uj * uj;
        const T Psi = half(e2 * Q) + ej * md + ej * Sv + m * s;
        A.f_eta[I.off + j] = -to_f64(m);
        sm[e * NT + t] = -(gT * ej * sz[e * NT + t]) - hj * Psi;
        v[e] = mk(Phi, from_int<T>(0));
      }
    }
    fft_fwd<PL>(M, g, v, xt);
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int s = 0; s < RP; ++s) {
        const T k = kn * from_int<T>(wave_index(g.mode(b, s), n));
        v[b * RP + s] = mul_pi(v[b * RP + s]) * k;
      }
    fft_inv<PL>(M, g, v, xt);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int j = g.pt + e * PS;
      if (what == 0) {
        sm[e * NT + t] = v[e].x;
        sz[e * NT + t] = v[e].y;
      } else if (what == 2) {
        sd[j] = v[e].x;
        sm[e * NT + t] = v[e].y;
      } else if (what == 3) {
        sz[e * NT + t] = v[e].x;
        ssx[j] = v[e].y;
      } else if (what == 5) {
        A.f_U[I.off + j] = to_f64(v[e].x + sm[e * NT + t]);
      }
    }
  }
  if (lcl) cluster_sync();               // shared memory outlives the partners' last use of it
}

// ---- SBDF2 velocity update ----------------------------------------------------------------
// As k_linimp_step1d (sgn_1d.cu): res1^ = (sigma + alpha k^2) u^ - (G u - U)^, and with SOLVE
// u_out = F^{-1}[(c1 res1^ + c0 res0^) / (sigma + alpha k^2)].  u^ stays in registers.
struct LinArgs {
  const Inst1d* insts;
  const int* ids;
  const cplx<double>* tw64;
  const cplx<df>* twdf;
  const SolveRec* A;
  const double* eta;
  const double* hx;
  const double* u;
  const double* U;
  const cplx<double>* res0;
  cplx<double>* res1;
  double c1, c0;
  double* u_out;
  void* ux;
  int precision;
  int solve;
};
template <typename PL>
struct SmemLin {
  static constexpr size_t tabs = (size_t)(PL::N1 + PL::N2) * 16;
  static size_t bytes(int lcl) { return tabs + ((size_t)32 << (PL::L - lcl)); }
};

__device__ __forceinline__ void coef_of(double e, double gx, double& c1, double& c2, double& c3) {
  c1 = e * (1.0 + gx * gx);
  c2 = 0.5 * e * e * gx;
  c3 = e * e * e * (1.0 / 3.0);
}
__device__ __forceinline__ void coef_of(double ed, double gd, df& c1, df& c2, df& c3) {
  const df e(ed), gx(gd), e2 = e * e;
  c1 = e + e * (gx * gx);
  c2 = half(e2 * gx);
  c3 = e2 * e * df(0.3333333432674408f, -9.934107758624577e-09f);   // 1/3, double-float
}

template <typename PL, typename T>
__global__ void SGN_SPLIT_BOUNDS(PL, 2)
    k_linimp(const __grid_constant__ LinArgs A, int first, int lcl) {
  using SL = Slot<PL>;
  constexpr int n = PL::n, E = PL::E, RP = PL::RP, h = n / 2, PS = n / E, NYQ = PL::NYQ;
  extern __shared__ __align__(16) unsigned char smem[];
  const int NT = 1 << (PL::LNTA - lcl), NL = n >> lcl, t = threadIdx.x;
  cplx<T>* bA = reinterpret_cast<cplx<T>*>(smem);
  cplx<T>* bB = bA + NL;
  cplx<T>* wA = bB + NL;
  cplx<T>* wB = wA + PL::N1;
  const cplx<T>* tw = table_of<T>(A.tw64, A.twdf);
  const Bufs<T> M{bA, bB, wA, wB};
  const Geo<PL> g(t, lcl ? (int)cluster_rank() : 0, lcl);
  const bool ts = g.t0;
  const int id = A.ids[first + (blockIdx.x >> lcl)];
  const Inst1d I = A.insts[id];
  const long long hs = I.ws / kWsVectors;
  const double* eta = A.eta + I.off;
  const double* hx = A.hx + I.off;
  const double* u = A.u + I.off;
  const double* U = A.U + I.off;
  T* ux = A.ux ? static_cast<T*>(A.ux) + I.off : nullptr;
  fill_tw<PL::L1>(wA, tw, NT);
  fill_tw<PL::L2>(wB, tw, NT);
  auto xt = [&](int e) { return tw[cross_index(g, e) << (kTwiddleLog2 - PL::L)]; };
  __shared__ double ku_s;                // by one thread: a float64 division takes 640 clocks
  if (t == 0) ku_s = 2.0 * kPi / I.L;
  const T sigma = num<T>(A.A[id].sigma), alpha = num<T>(A.A[id].alpha);
  const T one = from_int<T>(1), zero = from_int<T>(0), inv_n = num<T>(1.0 / (double)n);
  if (lcl) cluster_sync();               // the partners have started
  else __syncthreads();                  // the tables are filled
  const T ku = num<T>(ku_s);
  cplx<T> v[E], uh[RP];
  T uN = zero;
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = mk(num<T>(u[g.pt + e * PS]), zero);
  fft_fwd<PL>(M, g, v, xt);
#pragma unroll
  for (int q = 0; q < RP; ++q) uh[q] = v[SL::reg(q)];
  if (ts) {                              // real DC and Nyquist
    uh[0].y = zero;
    uN = v[NYQ].x;
  }
#pragma unroll
  for (int q = 0; q < RP; ++q) {
    const T k = ku * from_int<T>(g.mode(SL::b(q), SL::s(q)));
    if (ts && q == 0) {
      v[0] = uh[0];
    } else {
      v[SL::reg(q)] = uh[q] * (one - k);
      mirror_set<PL>(v, ts, SL::b(q), SL::s(q), conj(uh[q]) * (one + k));
    }
  }
  if (ts) v[NYQ] = mk(uN, zero);
  fft_inv<PL>(M, g, v, xt);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int j = g.pt + e * PS;
    const T pv = v[e].x * inv_n, px = v[e].y * inv_n;
    if (ux) ux[j] = px;
    T c1, c2, c3;
    coef_of(eta[j], hx[j], c1, c2, c3);
    v[e] = mk(c1 * pv + c2 * px - num<T>(U[j]), c2 * pv + c3 * px);
  }
  fft_fwd<PL>(M, g, v, xt);
  cplx<T> z[RP];
  T zN = zero;
  const T c1 = num<T>(A.c1), c0 = num<T>(A.c0);
#pragma unroll
  for (int q = 0; q < RP; ++q) {
    const int m = g.mode(SL::b(q), SL::s(q));
    const T k = ku * from_int<T>(m);
    const cplx<T> y = v[SL::reg(q)], ym = conj(mirror_get<PL>(v, ts, SL::b(q), SL::s(q)));
    const cplx<T> s = y * (one - k) + ym * (one + k);
    const T sym = sigma + alpha * (k * k);
    cplx<T> r = mk(uh[q].x * sym - half(s.x), uh[q].y * sym - half(s.y));
    if (ts && q == 0) r.y = zero;
    A.res1[hs + m] = mk(to_f64(r.x), to_f64(r.y));
    if (A.solve) {
      const cplx<double> p = A.res0[hs + m];
      const T is = recip(sym);
      z[q] = mk((c1 * r.x + c0 * num<T>(p.x)) * is, (c1 * r.y + c0 * num<T>(p.y)) * is);
      if (ts && q == 0) z[q].y = zero;
    }
  }
  if (ts) {
    const T r = uN * sigma - v[NYQ].x;
    A.res1[hs + h] = mk(to_f64(r), 0.0);
    if (A.solve) zN = (c1 * r + c0 * num<T>(A.res0[hs + h].x)) * recip(sigma);
  }
  if (A.solve) {                         // uniform over the grid
#pragma unroll
    for (int q = 0; q < RP; ++q) {
      v[SL::reg(q)] = z[q];
      if (!(ts && q == 0)) mirror_set<PL>(v, ts, SL::b(q), SL::s(q), conj(z[q]));
    }
    if (ts) v[NYQ] = mk(zN, zero);
    fft_inv<PL>(M, g, v, xt);
#pragma unroll
    for (int e = 0; e < E; ++e) A.u_out[I.off + g.pt + e * PS] = to_f64(v[e].x * inv_n);
  }
  if (lcl) cluster_sync();               // shared memory outlives the partners' last use of it
}

// ---- derivative and operator (float64) ------------------------------------------------------
// out = f_x, or out = G f = (c1 f + c2 f_x) - (c2 f + c3 f_x)_x with eta given (Def:G).  Bound by
// the float64 pipe and latency; as one CTA with gathered twiddles n = 4096 took 119 and 248 us.
struct FieldArgs {
  const Inst1d* insts;
  const int* ids;
  const cplx<double>* tw64;
  const double* f;
  const double* eta;       // null: the derivative
  const double* hx;
  double* out;
};

template <typename PL>
__global__ void SGN_SPLIT_BOUNDS(PL, 2)
    k_field(const __grid_constant__ FieldArgs A, int first, int lcl) {
  constexpr int n = PL::n, E = PL::E, RP = PL::RP, PS = n / E;
  extern __shared__ __align__(16) unsigned char smem[];
  const int NT = 1 << (PL::LNTA - lcl), NL = n >> lcl, t = threadIdx.x;
  cplx<double>* bA = reinterpret_cast<cplx<double>*>(smem);
  cplx<double>* bB = bA + NL;
  cplx<double>* wA = bB + NL;
  cplx<double>* wB = wA + PL::N1;
  const Bufs<double> M{bA, bB, wA, wB};
  const Geo<PL> g(t, lcl ? (int)cluster_rank() : 0, lcl);
  const Inst1d I = A.insts[A.ids[first + (blockIdx.x >> lcl)]];
  const double* f = A.f + I.off;
  fill_tw<PL::L1>(wA, A.tw64, NT);
  fill_tw<PL::L2>(wB, A.tw64, NT);
  auto xt = [&](int e) { return A.tw64[cross_index(g, e) << (kTwiddleLog2 - PL::L)]; };
  __shared__ double kn_s;                // by one thread: a float64 division takes 640 clocks
  if (t == 0) kn_s = 2.0 * kPi / I.L * (1.0 / (double)n);
  cplx<double> v[E];
  double w[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    w[e] = f[g.pt + e * PS];
    v[e] = mk(w[e], 0.0);
  }
  if (lcl) cluster_sync();               // the partners have started
  else __syncthreads();                  // the tables are filled
  const double kn = kn_s;
#pragma unroll 1
  for (int pass = 0; pass < (A.eta ? 2 : 1); ++pass) {
    fft_fwd<PL>(M, g, v, xt);
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int s = 0; s < RP; ++s)
        v[b * RP + s] = mul_pi(v[b * RP + s]) * (kn * (double)wave_index(g.mode(b, s), n));
    fft_inv<PL>(M, g, v, xt);
    if (A.eta && pass == 0) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const long long j = I.off + g.pt + e * PS;
        double c1, c2, c3;
        coef_of(A.eta[j], A.hx[j], c1, c2, c3);
        v[e] = mk(c2 * w[e] + c3 * v[e].x, c1 * w[e] + c2 * v[e].x);
        w[e] = v[e].y;
        v[e].y = 0.0;
      }
    }
  }
#pragma unroll
  for (int e = 0; e < E; ++e)
    A.out[I.off + g.pt + e * PS] = A.eta ? w[e] - v[e].x : v[e].x;
  if (lcl) cluster_sync();               // shared memory outlives the partners' last use of it
}

// ---- launches -----------------------------------------------------------------------------
template <typename PL, typename K, typename Args>
cudaError_t launch_split(K kernel, int num, int lcl, size_t smem, cudaStream_t s, const Args& a,
                         int first) {
  if (lcl < PL::kMinLcl || lcl > PL::kMaxLcl) return cudaErrorInvalidConfiguration;
  const int threads = 1 << (PL::LNTA - lcl);
  cudaError_t e = raise_smem(kernel, smem);
  if (e) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(num << lcl), 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1u << lcl;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = lcl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, a, first, lcl);
}

}  // namespace sp

// lcl: log2 of the CTAs per instance (split_lcl)
template <int L>
cudaError_t split_pcg_launch(const PcgArgs& a, int first, int num, int lcl, cudaStream_t s) {
  if (a.precision == SGN_PREC_MIXED) {
    using PL = sp::PlanMx<L>;
    return sp::launch_split<PL>(sp::k_solve_mixed<PL>, num, lcl, sp::SmemMixed<PL>::bytes(lcl), s,
                                a, first);
  }
  using PL = sp::Plan64<L>;
  return sp::launch_split<PL>(sp::k_solve64<PL>, num, lcl, sp::Smem64<PL>::bytes(lcl), s, a, first);
}

template <int L>
cudaError_t split_rhs_launch(const RhsArgs& a, int first, int num, int lcl, cudaStream_t s) {
  auto go = [&](auto k, auto pl) {
    using PL = decltype(pl);
    return sp::launch_split<PL>(k, num, lcl, sp::SmemRhs<PL>::bytes(lcl), s, a, first);
  };
  using PM = sp::PlanMx<L>;
  using PD = sp::Plan64<L>;
  if (a.precision == SGN_PREC_MIXED)
    return a.ux_given ? go(sp::k_rhs<PM, df, true>, PM{}) : go(sp::k_rhs<PM, df, false>, PM{});
  return a.ux_given ? go(sp::k_rhs<PD, double, true>, PD{}) : go(sp::k_rhs<PD, double, false>, PD{});
}

template <int L>
cudaError_t split_linimp_launch(const sp::LinArgs& a, int first, int num, int lcl, cudaStream_t s) {
  auto go = [&](auto k, auto pl) {
    using PL = decltype(pl);
    return sp::launch_split<PL>(k, num, lcl, sp::SmemLin<PL>::bytes(lcl), s, a, first);
  };
  if (a.precision == SGN_PREC_MIXED) return go(sp::k_linimp<sp::PlanMx<L>, df>, sp::PlanMx<L>{});
  return go(sp::k_linimp<sp::Plan64<L>, double>, sp::Plan64<L>{});
}

template <int L>
cudaError_t split_field_launch(const sp::FieldArgs& a, int first, int num, int lcl,
                               cudaStream_t s) {
  using PL = sp::Plan64<L>;
  return sp::launch_split<PL>(sp::k_field<PL>, num, lcl, sp::SmemLin<PL>::bytes(lcl), s, a, first);
}

}  // namespace sgn
