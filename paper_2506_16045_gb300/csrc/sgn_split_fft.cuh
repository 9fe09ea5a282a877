// Transforms of one 1d instance split over the CTAs of a thread-block cluster (1, 2, 4 or 8
// CTAs), or held by one CTA, with the same arithmetic for every split.
//
// n = 2^L points are read as an N1 x N2 matrix, j = j1 N2 + j2, and modes as k = k1 + N1 k2:
//   X[k1 + N1 k2] = sum_j2 w_N2^{j2 k2} w_n^{j2 k1} sum_j1 w_N1^{j1 k1} x[j1 N2 + j2].
// Phase A transforms the columns (length N1, fixed j2), phase B the rows (length N2, fixed
// k1).  CTA r of CL holds C = N2/CL columns of the real-space points, and in spectral space
// the rows k1 = +-v for VR = N1/(2 CL) consecutive v (v = 0 stands for the rows 0 and N1/2),
// so a mode and its mirror n - m always lie in one CTA.  A transform therefore needs one
// exchange between CTAs, the transposition between the phases (through distributed shared
// memory, one cluster barrier).  A transform of 2^13 points on one SM is bound by that SM's
// issue rate (double-float: 40 us; float64: 1.7 lanes per clock); the split divides it by
// the CTAs for the price of that barrier (370 clocks) and of the remote stores.
//
// Within a phase the stages are in place: a stage of radix R loads R elements at distance
// sigma, transforms them in registers and stores them where they were (decimation in
// frequency forward, the same stages backwards for the inverse), so a stage costs one
// barrier, results come out in digit-reversed positions, and nothing is permuted: positions
// are only translated to indices once per thread.
//
// Each of the n/E threads of an instance (T = rank NT + t) holds E elements: on the real side
// the points pt + e n/E, on the spectral side the outputs of two radix-E/2 butterflies, the
// modes i0 + s n/RP and i1 + s n/RP (RP = E/2) with i1 = n/RP - i0 (thread 0: 0 and
// n/(2 RP)), so the mirror of each of its modes is in the same thread.  T's modes do not
// depend on CL: sums over modes are taken per thread, per warp of 32 consecutive T and then
// over the warps in order, and come out bitwise the same for every CL.
//
// Shared memory: buffer A [N1][C] (column fastest) and buffer B [2 VR][N2], the latter
// through a GF(2)-linear XOR swizzle of the element index that spreads every stage's accesses
// over the banks.  Both are written remotely only between the barriers that end their
// owner's use.
#pragma once
#include "sgn_fft1d.cuh"
#include "sgn_split_plan.h"

namespace sgn {
namespace sp {

using f1::IC;
using f1::static_for;

template <int L_, int E_>
struct Plan {
  static constexpr int L = L_, n = 1 << L, E = E_;
  static constexpr int LE = E == 8 ? 3 : (E == 4 ? 2 : 1);
  static constexpr int LP = LE - 1, RP = 1 << LP;
  static constexpr int HS = RP > 1 ? RP / 2 : 1;             // half-spectrum slots per butterfly
  static constexpr int NYQ = RP > 1 ? HS : 1;                // thread 0's register of mode n/2
  static constexpr int L1 = split_log_n1(L), L2 = L - L1;
  static constexpr int N1 = 1 << L1, N2 = 1 << L2;
  // phase A: a stage of radix E, then the rest as evenly as possible; phase B: plain stages
  // as evenly as possible, then the paired one of radix RP
  static constexpr int nA = 1 + (L1 - LE + LE - 1) / LE;
  static constexpr int restB = L2 - LP;
  static constexpr int nB = (restB + LE - 1) / LE;
  static constexpr int bitsA(int q) {
    return q == 0 ? LE : (L1 - LE) / (nA - 1) + (q - 1 < (L1 - LE) % (nA - 1) ? 1 : 0);
  }
  static constexpr int bitsB(int q) { return restB / nB + (q < restB % nB ? 1 : 0); }
  // bits before stage q, and log2 of its element distance sigma
  static constexpr int cumA(int q) {
    int s = 0;
    for (int i = 0; i < q; ++i) s += bitsA(i);
    return s;
  }
  static constexpr int cumB(int q) {
    int s = 0;
    for (int i = 0; i < q; ++i) s += bitsB(i);
    return s;
  }
  static constexpr int sA(int q) { return L1 - cumA(q) - bitsA(q); }
  static constexpr int sB(int q) { return L2 - cumB(q) - bitsB(q); }
  static constexpr int LNTA = L - LE;                        // log2 threads of an instance
  static constexpr int W = LNTA > 5 ? 1 << (LNTA - 5) : 1;   // their warps
  static constexpr int kMinLcl = split_min_lcl(L, LE), kMaxLcl = split_max_lcl(L, LE);
  static constexpr int kMaxNT = LNTA - kMinLcl > 8 ? 1 << (LNTA - kMinLcl) : 256;
};

__host__ __device__ constexpr int swz(int a) {
  return a ^ ((a >> 2) & 3) ^ ((((a >> 4) ^ (a >> 5) ^ (a >> 6)) & 1) << 2) ^
         (((a >> 5) & 1) << 3);
}

// Digit reversals between positions and indices (phase A: position p1 -> k1 and back; phase
// B's plain stages: group g = position / RP -> kappa, and kappa -> position).
template <typename PL>
__host__ __device__ inline int revA(int p) {
  int k = 0;
#pragma unroll
  for (int q = 0; q < PL::nA; ++q)
    k |= ((p >> PL::sA(q)) & ((1 << PL::bitsA(q)) - 1)) << PL::cumA(q);
  return k;
}
template <typename PL>
__host__ __device__ inline int posA(int k1) {
  int p = 0;
#pragma unroll
  for (int q = 0; q < PL::nA; ++q)
    p |= ((k1 >> PL::cumA(q)) & ((1 << PL::bitsA(q)) - 1)) << PL::sA(q);
  return p;
}
template <typename PL>
__host__ __device__ inline int revB(int g) {
  int k = 0;
#pragma unroll
  for (int q = 0; q < PL::nB; ++q)
    k |= (((g << PL::LP) >> PL::sB(q)) & ((1 << PL::bitsB(q)) - 1)) << PL::cumB(q);
  return k;
}
template <typename PL>
__host__ __device__ inline int posB(int kappa) {             // position of group kappa
  int p = 0;
#pragma unroll
  for (int q = 0; q < PL::nB; ++q)
    p |= ((kappa >> PL::cumB(q)) & ((1 << PL::bitsB(q)) - 1)) << PL::sB(q);
  return p;
}

// A thread's place: its CTA's share and the points and modes it holds.
template <typename PL>
struct Geo {
  int t, rank, lcl;          // thread of the CTA, CTA of the cluster, log2 CTAs
  int lC, lNT, lVR;
  int pt;                    // first real point (of the instance)
  int i0, i1;                // paired butterflies
  int ap0, ap1;              // their swizzled addresses in buffer B
  bool t0;                   // owner of the modes 0 and n/2
  __host__ __device__ Geo(int t_, int rank_, int lcl_) : t(t_), rank(rank_), lcl(lcl_) {
    lC = PL::L2 - lcl;
    lNT = PL::LNTA - lcl;
    lVR = PL::L1 - 1 - lcl;
    pt = ((t >> lC) << PL::L2) + (rank << lC) + (t & ((1 << lC) - 1));
    const int T = (rank << lNT) + t;
    constexpr int G = PL::N2 / PL::RP;
    const int v = T / G, g = T & (G - 1), kap = revB<PL>(g);
    const int vloc = v & ((1 << lVR) - 1), VR = 1 << lVR;
    int r0, r1, k0, k1;      // rows of buffer B and kappas
    if (v != 0) {
      r0 = vloc;
      r1 = VR + vloc;
      k0 = kap;
      k1 = G - 1 - kap;
      i0 = v + (k0 << PL::L1);
      i1 = PL::N1 - v + (k1 << PL::L1);
    } else if (kap < G / 2) {                    // row 0
      r0 = r1 = 0;
      k0 = kap;
      k1 = kap ? G - kap : G / 2;
      i0 = k0 << PL::L1;
      i1 = k1 << PL::L1;
    } else {                                     // row N1 / 2
      r0 = r1 = VR;
      k0 = kap - G / 2;
      k1 = G - 1 - k0;
      i0 = PL::N1 / 2 + (k0 << PL::L1);
      i1 = PL::N1 / 2 + (k1 << PL::L1);
    }
    if (PL::RP == 1 && i0 > i1) {                // the slot's mode is the one below n/2
      const int i = i0, r = r0, k = k0;
      i0 = i1;
      r0 = r1;
      k0 = k1;
      i1 = i;
      r1 = r;
      k1 = k;
    }
    ap0 = swz((r0 << PL::L2) | posB<PL>(k0));
    ap1 = swz((r1 << PL::L2) | posB<PL>(k1));
    t0 = T == 0;
  }
  __host__ __device__ int mode(int b, int s) const { return (b ? i1 : i0) + s * (PL::n / PL::RP); }
};

// Half-spectrum slot q < RP of a thread: register, and mode below n/2.
template <typename PL>
struct Slot {
  static constexpr int b(int q) { return q / PL::HS; }
  static constexpr int s(int q) { return q % PL::HS; }
  static constexpr int reg(int q) { return b(q) * PL::RP + s(q); }
};

template <typename PL, typename V>
__host__ __device__ __forceinline__ V mirror_get(const V (&v)[PL::E], bool t0, int b, int s) {
  if (b == 0) {
    const V x = v[(PL::RP - s) & (PL::RP - 1)], y = v[2 * PL::RP - 1 - s];
    return t0 ? x : y;
  }
  const V x = v[2 * PL::RP - 1 - s], y = v[PL::RP - 1 - s];
  return t0 ? x : y;
}
template <typename PL, typename V>
__host__ __device__ __forceinline__ void mirror_set(V (&v)[PL::E], bool t0, int b, int s, V val) {
  if (b == 0) {
    if (t0) v[(PL::RP - s) & (PL::RP - 1)] = val;
    else v[2 * PL::RP - 1 - s] = val;
  } else {
    if (t0) v[2 * PL::RP - 1 - s] = val;
    else v[PL::RP - 1 - s] = val;
  }
}

// Address of element r = 0 of butterfly jj of a stage (element r lies r sigma further: in A
// r << (sA + lC), in B an XOR with swz(r << sB)), and the butterfly's index i mod sigma.
template <typename PL, int Q>
__host__ __device__ __forceinline__ int addrA(const Geo<PL>& g, int jj, int& i) {
  constexpr int S = PL::sA(Q), R = PL::bitsA(Q);
  const int bi = g.t + (jj << g.lNT), c = bi & ((1 << g.lC) - 1), y = bi >> g.lC;
  i = y & ((1 << S) - 1);
  return (((((y >> S) << (S + R)) | i)) << g.lC) + c;
}
template <typename PL, int Q>
__host__ __device__ __forceinline__ int addrB(const Geo<PL>& g, int jj, int& rho, int& i) {
  constexpr int S = PL::sB(Q), R = PL::bitsB(Q);
  const int bi = g.t + (jj << g.lNT), y = bi & ((1 << (PL::L2 - R)) - 1);
  rho = bi >> (PL::L2 - R);
  i = y & ((1 << S) - 1);
  return swz((rho << PL::L2) | ((y >> S) << (S + R)) | i);
}

// The row k1 of buffer B: its owner and its place there.
template <typename PL>
__host__ __device__ __forceinline__ void row_of(const Geo<PL>& g, int k1, int& rank, int& rho) {
  const int hi = k1 >= PL::N1 / 2;
  const int v = (hi ? PL::N1 - k1 : k1) & (PL::N1 / 2 - 1);     // N1/2 -> 0
  rank = v >> g.lVR;
  rho = (v & ((1 << g.lVR) - 1)) | (hi << g.lVR);
}
// and the other way: k1 of row rho of CTA `rank`
template <typename PL>
__host__ __device__ __forceinline__ int k1_of(const Geo<PL>& g, int rho) {
  const int hi = rho >> g.lVR, v = (g.rank << g.lVR) | (rho & ((1 << g.lVR) - 1));
  return hi ? (v ? PL::N1 - v : PL::N1 / 2) : v;
}

#ifdef __CUDACC__

__device__ __forceinline__ void cta_or_cluster_sync(int lcl) {
  if (lcl) cluster_sync();
  else __syncthreads();
}
template <typename P>
__device__ __forceinline__ P* at_rank(P* p, int rank, int lcl) {
  if (lcl == 0) return p;
  return static_cast<P*>(__cluster_map_shared_rank(static_cast<void*>(p), (unsigned)rank));
}

template <typename T, int R, bool INV>
__device__ __forceinline__ void dft_r(cplx<T> (&a)[R]) {
  if constexpr (R > 1) f1::dft<T, R, INV>(a);
}

// Buffers and tables of a transform in T: buffers A and B (this CTA's), the stage twiddles
// w_N1^m and w_N2^m in shared memory, and xt(e) = w_n^{j2 k1} of element e of the thread's
// last phase-A stage (cross_index).
template <typename T>
struct Bufs {
  cplx<T>* A;
  cplx<T>* B;
  const cplx<T>* wA;
  const cplx<T>* wB;
};

// Index m of the cross twiddle e^{-2 pi i m / n} of element e = jj R + s of the last A stage.
template <typename PL>
__device__ __forceinline__ int cross_index(const Geo<PL>& g, int e) {
  constexpr int Q = PL::nA - 1, R = 1 << PL::bitsA(Q);
  int i;
  const int a = addrA<PL, Q>(g, e / R, i);
  const int k1 = revA<PL>((a >> g.lC) + e % R);
  const int j2 = (g.rank << g.lC) + (a & ((1 << g.lC) - 1));
  return (k1 * j2) & (PL::n - 1);
}

// Forward transform, stages unrolled (float32 and float64).
template <typename PL, typename T, typename XT>
__device__ __forceinline__ void fwd_unrolled(const Bufs<T>& M, const Geo<PL>& g,
                                             cplx<T> (&v)[PL::E], XT xt) {
  constexpr int E = PL::E;
  static_for<0, PL::nA>([&](auto Qc) {
    constexpr int Q = decltype(Qc)::value, S = PL::sA(Q), LR = PL::bitsA(Q), R = 1 << LR;
#pragma unroll
    for (int jj = 0; jj < E / R; ++jj) {
      int i;
      const int a0 = addrA<PL, Q>(g, jj, i);
      cplx<T> a[R];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = Q == 0 ? v[jj * R + r] : M.A[a0 + (r << (S + g.lC))];
      dft_r<T, R, false>(a);
      if constexpr (Q + 1 < PL::nA) {
#pragma unroll
        for (int s = 1; s < R; ++s) a[s] = cmul(a[s], M.wA[(i * s) << PL::cumA(Q)]);
#pragma unroll
        for (int s = 0; s < R; ++s) M.A[a0 + (s << (S + g.lC))] = a[s];
      } else {
        const int j2 = (g.rank << g.lC) + (a0 & ((1 << g.lC) - 1));
        const int kap = revA<PL>(a0 >> g.lC);
#pragma unroll
        for (int s = 0; s < R; ++s) {
          int rk, rho;
          row_of<PL>(g, kap + (s << PL::cumA(Q)), rk, rho);
          at_rank(M.B, rk, g.lcl)[swz((rho << PL::L2) | j2)] = cmul(a[s], xt(jj * R + s));
        }
      }
    }
    if constexpr (Q + 1 < PL::nA) {
      __syncthreads();
    } else {
      cta_or_cluster_sync(g.lcl);
    }
  });
  static_for<0, PL::nB>([&](auto Qc) {
    constexpr int Q = decltype(Qc)::value, S = PL::sB(Q), LR = PL::bitsB(Q), R = 1 << LR;
#pragma unroll
    for (int jj = 0; jj < E / R; ++jj) {
      int i, rho;
      const int a0 = addrB<PL, Q>(g, jj, rho, i);
      cplx<T> a[R];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = M.B[a0 ^ swz(r << S)];
      dft_r<T, R, false>(a);
      if constexpr (S > 0) {
#pragma unroll
        for (int s = 1; s < R; ++s) a[s] = cmul(a[s], M.wB[(i * s) << PL::cumB(Q)]);
      }
#pragma unroll
      for (int s = 0; s < R; ++s) M.B[a0 ^ swz(s << S)] = a[s];
    }
    __syncthreads();
  });
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    cplx<T> a[PL::RP];
#pragma unroll
    for (int r = 0; r < PL::RP; ++r) a[r] = M.B[(b ? g.ap1 : g.ap0) ^ r];
    dft_r<T, PL::RP, false>(a);
#pragma unroll
    for (int s = 0; s < PL::RP; ++s) v[b * PL::RP + s] = a[s];
  }
}

// Inverse transform, stages unrolled.
template <typename PL, typename T, typename XT>
__device__ __forceinline__ void inv_unrolled(const Bufs<T>& M, const Geo<PL>& g,
                                             cplx<T> (&v)[PL::E], XT xt) {
  constexpr int E = PL::E;
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    cplx<T> a[PL::RP];
#pragma unroll
    for (int s = 0; s < PL::RP; ++s) a[s] = v[b * PL::RP + s];
    dft_r<T, PL::RP, true>(a);
#pragma unroll
    for (int r = 0; r < PL::RP; ++r) M.B[(b ? g.ap1 : g.ap0) ^ r] = a[r];
  }
  __syncthreads();
  static_for<0, PL::nB>([&](auto Qc) {
    constexpr int Q = PL::nB - 1 - decltype(Qc)::value;
    constexpr int S = PL::sB(Q), LR = PL::bitsB(Q), R = 1 << LR;
#pragma unroll
    for (int jj = 0; jj < E / R; ++jj) {
      int i, rho;
      const int a0 = addrB<PL, Q>(g, jj, rho, i);
      cplx<T> a[R];
#pragma unroll
      for (int s = 0; s < R; ++s) a[s] = M.B[a0 ^ swz(s << S)];
      if constexpr (S > 0) {
#pragma unroll
        for (int s = 1; s < R; ++s) a[s] = cmul(a[s], conj(M.wB[(i * s) << PL::cumB(Q)]));
      }
      dft_r<T, R, true>(a);
      if constexpr (Q > 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) M.B[a0 ^ swz(r << S)] = a[r];
      } else {
        // column j2 = i + r sigma of row k1: to its owner's buffer A
        const int k1 = k1_of<PL>(g, rho), p1 = posA<PL>(k1);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int j2 = i + (r << S);
          at_rank(M.A, j2 >> g.lC, g.lcl)[(p1 << g.lC) + (j2 & ((1 << g.lC) - 1))] = a[r];
        }
      }
    }
    if constexpr (Q > 0) {
      __syncthreads();
    } else {
      cta_or_cluster_sync(g.lcl);
    }
  });
  static_for<0, PL::nA>([&](auto Qc) {
    constexpr int Q = PL::nA - 1 - decltype(Qc)::value;
    constexpr int S = PL::sA(Q), LR = PL::bitsA(Q), R = 1 << LR;
#pragma unroll
    for (int jj = 0; jj < E / R; ++jj) {
      int i;
      const int a0 = addrA<PL, Q>(g, jj, i);
      cplx<T> a[R];
#pragma unroll
      for (int s = 0; s < R; ++s) a[s] = M.A[a0 + (s << (S + g.lC))];
      if constexpr (Q + 1 == PL::nA) {
#pragma unroll
        for (int s = 0; s < R; ++s) a[s] = cmul(a[s], conj(xt(jj * R + s)));
      } else {
#pragma unroll
        for (int s = 1; s < R; ++s) a[s] = cmul(a[s], conj(M.wA[(i * s) << PL::cumA(Q)]));
      }
      dft_r<T, R, true>(a);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if constexpr (Q > 0) M.A[a0 + (r << (S + g.lC))] = a[r];
        else v[jj * R + r] = a[r];
      }
    }
    if constexpr (Q > 0) __syncthreads();
  });
}

// ---- double-float: stages in a loop ---------------------------------------------------------
// A double-float butterfly is hundreds of instructions, and a transform with every stage
// unrolled runs its code once per transform from the instruction caches' outer levels: at 64
// threads per CTA it measured 25 us at n = 4096, about ten times its issue time.  Here the
// stages of one radix share a body in a runtime loop (both phases: the position arithmetic
// differs only in the digit's place and in the swizzle).
// One stage of radix R on the thread's E/R butterflies: buf's digit at bits [S, S + log2 R)
// of the position, lb of the S lower bits being the batch (phase A's columns), twiddles
// w^{(i s) << cum}.
template <typename PL, typename T, bool INV, int LR>
__device__ __forceinline__ void stage_loop(cplx<T>* buf, const cplx<T>* w, int t, int lNT, int S,
                                           int lb, int cum, bool sw) {
  constexpr int R = 1 << LR, J = PL::E / R;
  const int m = (1 << S) - 1;
#pragma unroll 1
  for (int jj = 0; jj < J; ++jj) {
    const int bi = t + (jj << lNT), x0 = ((bi & ~m) << LR) | (bi & m), i = (bi & m) >> lb;
    const int a0 = sw ? swz(x0) : x0;
    int ad[R];
#pragma unroll
    for (int r = 0; r < R; ++r) ad[r] = a0 ^ (sw ? swz(r << S) : r << S);
    cplx<T> a[R];
#pragma unroll
    for (int r = 0; r < R; ++r) a[r] = buf[ad[r]];
    if (INV && S > lb) {
#pragma unroll
      for (int s = 1; s < R; ++s) a[s] = cmul(a[s], conj(w[(i * s) << cum]));
    }
    dft_r<T, R, INV>(a);
    if (!INV && S > lb) {
#pragma unroll
      for (int s = 1; s < R; ++s) a[s] = cmul(a[s], w[(i * s) << cum]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) buf[ad[r]] = a[r];
  }
}
template <typename PL, typename T, bool INV>
__device__ __forceinline__ void stage_any(int LR, cplx<T>* buf, const cplx<T>* w, int t, int lNT,
                                          int S, int lb, int cum, bool sw) {
  if (PL::LE >= 3 && LR == 3) stage_loop<PL, T, INV, (PL::LE >= 3 ? 3 : 1)>(buf, w, t, lNT, S, lb, cum, sw);
  if (PL::LE >= 2 && LR == 2) stage_loop<PL, T, INV, (PL::LE >= 2 ? 2 : 1)>(buf, w, t, lNT, S, lb, cum, sw);
  if (LR == 1) stage_loop<PL, T, INV, 1>(buf, w, t, lNT, S, lb, cum, sw);
}

template <typename PL, typename T, typename XT>
__device__ __forceinline__ void fwd_looped(const Bufs<T>& M, const Geo<PL>& g,
                                           cplx<T> (&v)[PL::E], XT xt) {
  constexpr int E = PL::E, QA = PL::nA - 1, RA = 1 << PL::bitsA(QA);
  cplx<T> xw[E];                       // the exchange's twiddles, loaded ahead
#pragma unroll
  for (int e = 0; e < E; ++e) xw[e] = xt(e);
  {
    int i;
    const int a0 = addrA<PL, 0>(g, 0, i);
#pragma unroll
    for (int e = 0; e < E; ++e) M.A[a0 + (e << (PL::sA(0) + g.lC))] = v[e];
  }
  int S = PL::L1, cum = 0;
#pragma unroll 1
  for (int q = 0; q < PL::nA; ++q) {
    const int LR = PL::bitsA(q);
    if (q) __syncthreads();
    S -= LR;
    stage_any<PL, T, false>(LR, M.A, M.wA, g.t, g.lNT, S + g.lC, g.lC, cum, false);
    cum += LR;
  }
#pragma unroll
  for (int e = 0; e < E; ++e) {        // the thread's own elements of the last stage
    int i, rk, rho;
    const int a0 = addrA<PL, QA>(g, e / RA, i) + ((e % RA) << g.lC);
    row_of<PL>(g, revA<PL>(a0 >> g.lC), rk, rho);
    at_rank(M.B, rk, g.lcl)[swz((rho << PL::L2) | ((g.rank << g.lC) + (a0 & ((1 << g.lC) - 1))))] =
        cmul(M.A[a0], xw[e]);
  }
  cta_or_cluster_sync(g.lcl);
  S = PL::L2;
  cum = 0;
#pragma unroll 1
  for (int q = 0; q < PL::nB; ++q) {
    const int LR = PL::bitsB(q);
    S -= LR;
    stage_any<PL, T, false>(LR, M.B, M.wB, g.t, g.lNT, S, 0, cum, true);
    cum += LR;
    __syncthreads();
  }
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    cplx<T> a[PL::RP];
#pragma unroll
    for (int r = 0; r < PL::RP; ++r) a[r] = M.B[(b ? g.ap1 : g.ap0) ^ r];
    dft_r<T, PL::RP, false>(a);
#pragma unroll
    for (int s = 0; s < PL::RP; ++s) v[b * PL::RP + s] = a[s];
  }
}

template <typename PL, typename T, typename XT>
__device__ __forceinline__ void inv_looped(const Bufs<T>& M, const Geo<PL>& g,
                                           cplx<T> (&v)[PL::E], XT xt) {
  constexpr int E = PL::E, QA = PL::nA - 1, RA = 1 << PL::bitsA(QA), RB = 1 << PL::bitsB(0);
  cplx<T> xw[E];
#pragma unroll
  for (int e = 0; e < E; ++e) xw[e] = xt(e);
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    cplx<T> a[PL::RP];
#pragma unroll
    for (int s = 0; s < PL::RP; ++s) a[s] = v[b * PL::RP + s];
    dft_r<T, PL::RP, true>(a);
#pragma unroll
    for (int r = 0; r < PL::RP; ++r) M.B[(b ? g.ap1 : g.ap0) ^ r] = a[r];
  }
  int S = PL::LP, cum = PL::restB;
#pragma unroll 1
  for (int q = PL::nB - 1; q >= 0; --q) {
    const int LR = PL::bitsB(q);
    __syncthreads();
    cum -= LR;
    stage_any<PL, T, true>(LR, M.B, M.wB, g.t, g.lNT, S, 0, cum, true);
    S += LR;
  }
#pragma unroll
  for (int e = 0; e < E; ++e) {        // the thread's own elements: to their columns' owners
    int i, rho;
    const int r = e % RB, a0 = addrB<PL, 0>(g, e / RB, rho, i), j2 = i + (r << PL::sB(0));
    at_rank(M.A, j2 >> g.lC, g.lcl)[(posA<PL>(k1_of<PL>(g, rho)) << g.lC) +
                                    (j2 & ((1 << g.lC) - 1))] = M.B[a0 ^ swz(r << PL::sB(0))];
  }
  cta_or_cluster_sync(g.lcl);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    int i;
    const int a0 = addrA<PL, QA>(g, e / RA, i) + ((e % RA) << g.lC);
    M.A[a0] = cmul(M.A[a0], conj(xw[e]));
  }
  S = 0;
  cum = PL::L1;
#pragma unroll 1
  for (int q = PL::nA - 1; q >= 0; --q) {
    const int LR = PL::bitsA(q);
    if (q < PL::nA - 1) __syncthreads();
    cum -= LR;
    stage_any<PL, T, true>(LR, M.A, M.wA, g.t, g.lNT, S + g.lC, g.lC, cum, false);
    S += LR;
  }
  {
    int i;
    const int a0 = addrA<PL, 0>(g, 0, i);
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = M.A[a0 + (e << (PL::sA(0) + g.lC))];
  }
}

// Forward transform: v[e] = x[pt + e n/E] in; v[b RP + s] = X[mode(b, s)] out.
template <typename PL, typename T, typename XT>
__device__ __forceinline__ void fft_fwd(const Bufs<T>& M, const Geo<PL>& g, cplx<T> (&v)[PL::E],
                                        XT xt) {
  if constexpr (std::is_same<T, df>::value) fwd_looped<PL>(M, g, v, xt);
  else fwd_unrolled<PL>(M, g, v, xt);
}
// Inverse transform (unnormalised): the same layouts the other way round.
template <typename PL, typename T, typename XT>
__device__ __forceinline__ void fft_inv(const Bufs<T>& M, const Geo<PL>& g, cplx<T> (&v)[PL::E],
                                        XT xt) {
  if constexpr (std::is_same<T, df>::value) inv_looped<PL>(M, g, v, xt);
  else inv_unrolled<PL>(M, g, v, xt);
}

#endif  // __CUDACC__

}  // namespace sp
}  // namespace sgn
