// Launchers of the register-FFT 1d kernels: one launch per size class.  The kernels
// (sgn_1d_pcg.cuh: a5/a6 solve, sgn_1d_rhs.cuh: a7 right-hand side; sgn_split_1d.cuh from
// n = 256) are instantiated per size in the sgn_1d_*.cu and sgn_split_*.cu translation units, which compile in parallel.
#include "sgn_1d_pcg.cuh"
#include "sgn_1d_rhs.cuh"
#include "sgn_split_1d.cuh"

namespace sgn {

extern template cudaError_t pcg1d_launch<3, 1>(const PcgArgs&, int, int, cudaStream_t);
extern template cudaError_t pcg1d_launch<4, 1>(const PcgArgs&, int, int, cudaStream_t);
extern template cudaError_t pcg1d_launch<5, 1>(const PcgArgs&, int, int, cudaStream_t);
extern template cudaError_t pcg1d_launch<6, 1>(const PcgArgs&, int, int, cudaStream_t);
extern template cudaError_t pcg1d_launch<7, 1>(const PcgArgs&, int, int, cudaStream_t);
extern template cudaError_t pcg1d_launch<12, 2>(const PcgArgs&, int, int, cudaStream_t);
extern template cudaError_t pcg1d_launch<13, 2>(const PcgArgs&, int, int, cudaStream_t);
extern template cudaError_t rhs1d_launch<3, 1>(const RhsArgs&, int, int, cudaStream_t);
extern template cudaError_t rhs1d_launch<4, 1>(const RhsArgs&, int, int, cudaStream_t);
extern template cudaError_t rhs1d_launch<5, 1>(const RhsArgs&, int, int, cudaStream_t);
extern template cudaError_t rhs1d_launch<6, 1>(const RhsArgs&, int, int, cudaStream_t);
extern template cudaError_t rhs1d_launch<7, 1>(const RhsArgs&, int, int, cudaStream_t);
extern template cudaError_t rhs1d_launch<12, 2>(const RhsArgs&, int, int, cudaStream_t);
extern template cudaError_t rhs1d_launch<13, 2>(const RhsArgs&, int, int, cudaStream_t);
extern template cudaError_t split_pcg_launch<8>(const PcgArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_rhs_launch<8>(const RhsArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_linimp_launch<8>(const sp::LinArgs&, int, int, int,
                                                     cudaStream_t);
extern template cudaError_t split_field_launch<8>(const sp::FieldArgs&, int, int, int,
                                                   cudaStream_t);
extern template cudaError_t split_pcg_launch<9>(const PcgArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_rhs_launch<9>(const RhsArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_linimp_launch<9>(const sp::LinArgs&, int, int, int,
                                                     cudaStream_t);
extern template cudaError_t split_field_launch<9>(const sp::FieldArgs&, int, int, int,
                                                   cudaStream_t);
extern template cudaError_t split_pcg_launch<10>(const PcgArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_rhs_launch<10>(const RhsArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_linimp_launch<10>(const sp::LinArgs&, int, int, int,
                                                     cudaStream_t);
extern template cudaError_t split_field_launch<10>(const sp::FieldArgs&, int, int, int,
                                                   cudaStream_t);
extern template cudaError_t split_pcg_launch<11>(const PcgArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_rhs_launch<11>(const RhsArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_linimp_launch<11>(const sp::LinArgs&, int, int, int,
                                                     cudaStream_t);
extern template cudaError_t split_field_launch<11>(const sp::FieldArgs&, int, int, int,
                                                   cudaStream_t);
extern template cudaError_t split_pcg_launch<12>(const PcgArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_rhs_launch<12>(const RhsArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_linimp_launch<12>(const sp::LinArgs&, int, int, int,
                                                     cudaStream_t);
extern template cudaError_t split_field_launch<12>(const sp::FieldArgs&, int, int, int,
                                                   cudaStream_t);
extern template cudaError_t split_pcg_launch<13>(const PcgArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_rhs_launch<13>(const RhsArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_linimp_launch<13>(const sp::LinArgs&, int, int, int,
                                                     cudaStream_t);
extern template cudaError_t split_field_launch<13>(const sp::FieldArgs&, int, int, int,
                                                   cudaStream_t);
extern template cudaError_t split_pcg_launch<14>(const PcgArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_rhs_launch<14>(const RhsArgs&, int, int, int, cudaStream_t);
extern template cudaError_t split_linimp_launch<14>(const sp::LinArgs&, int, int, int,
                                                     cudaStream_t);
extern template cudaError_t split_field_launch<14>(const sp::FieldArgs&, int, int, int,
                                                   cudaStream_t);

// log2 of the CTAs per instance that class l's split kernel takes beside the layout's other
// classes; ctas(c) is 2 where class c runs on the two-CTA kernels.
static_assert(kSplitMinLog == kSplitLog1d && kSplitMaxLog == kMaxLog1d, "the split classes");
template <typename Ctas>
static int split_lcl(const Layout1d& lay, int l, bool mixed, Ctas ctas) {
  int num[kSplitClasses], two[kSplitClasses], lcl[kSplitClasses];
  for (int c = 0; c < kSplitClasses; ++c) {
    num[c] = lay.class_end[c] - lay.class_begin[c];
    two[c] = c >= kClusterLog1d && c <= kSmemLog1d && ctas(c) == 2 ? 2 : 1;
  }
  split_plan(num, two, mixed, kSMs, lcl);
  return lcl[l];
}

namespace {

// The form of size class LG in this layout: up to n = 128 one CTA per instance; above, the
// split kernels with the CTAs per instance that split_lcl chooses, or, where set_form(s) asked
// for two CTAs (n = 4096 and 8192, solve and right-hand side separately), the two-CTA
// clusters of sgn_1d_pcg.cuh and sgn_1d_rhs.cuh.  The solve's u_x hand-off is stored in natural
// point order by every form, so the two kernels may take different forms.
struct PcgKernels {
  template <int LG, int CL>
  static cudaError_t go(const PcgArgs& a, int first, int num, cudaStream_t s) {
    return pcg1d_launch<LG, CL>(a, first, num, s);
  }
  template <int LG>
  static cudaError_t split(const PcgArgs& a, int first, int num, int lcl, cudaStream_t s) {
    return split_pcg_launch<LG>(a, first, num, lcl, s);
  }
  static int ctas(const Layout1d& lay, int l) { return lay.ctas(l); }
};
struct RhsKernels {
  template <int LG, int CL>
  static cudaError_t go(const RhsArgs& a, int first, int num, cudaStream_t s) {
    return rhs1d_launch<LG, CL>(a, first, num, s);
  }
  template <int LG>
  static cudaError_t split(const RhsArgs& a, int first, int num, int lcl, cudaStream_t s) {
    return split_rhs_launch<LG>(a, first, num, lcl, s);
  }
  static int ctas(const Layout1d& lay, int l) { return lay.rhs_ctas(l); }
};

template <int LG, typename K, typename Args>
cudaError_t launch_form(const Layout1d& lay, const Args& a, int first, int num, cudaStream_t s,
                        K) {
  if constexpr (LG >= kSplitLog1d) {
    if constexpr (LG >= kClusterLog1d && LG <= kSmemLog1d)
      if (K::ctas(lay, LG) == 2) return K::template go<LG, 2>(a, first, num, s);
    return K::template split<LG>(a, first, num,
                                 split_lcl(lay, LG, a.precision == SGN_PREC_MIXED,
                                           [&](int c) { return K::ctas(lay, c); }),
                                 s);
  } else {
    return K::template go<LG, 1>(a, first, num, s);
  }
}

PcgArgs pcg_args(const Layout1d& lay, const void* tw64, const void* tw32, int precision,
                 const double* eta, const double* hx, const double* b, double* x,
                 const SolveRec* given, int kind, double rtol, double rtol_inner, int maxit,
                 int max_refine, SolveRec* rec, void* ws, float* coef_df) {
  PcgArgs a;
  a.insts = lay.d_inst;
  a.ids = lay.d_ids;
  a.tw64 = static_cast<const cplx<double>*>(tw64);
  a.twdf = reinterpret_cast<const cplx<df>*>(static_cast<const char*>(tw32) + kTw32Bytes);
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
  a.coef_df = precision == SGN_PREC_MIXED ? coef_df : nullptr;
  a.precision = precision;
  a.ux = nullptr;
  return a;
}

RhsArgs rhs_args(const Layout1d& lay, const void* tw64, const void* tw32, int precision,
                 double g, const double* eta, const double* u, const double* h,
                 const double* hx, double* f_eta, double* f_U, double* scratch) {
  RhsArgs a;
  a.insts = lay.d_inst;
  a.ids = lay.d_ids;
  a.tw64 = static_cast<const cplx<double>*>(tw64);
  a.twdf = reinterpret_cast<const cplx<df>*>(static_cast<const char*>(tw32) + kTw32Bytes);
  a.g = g;
  a.eta = eta;
  a.u = u;
  a.h = h;
  a.hx = hx;
  a.f_eta = f_eta;
  a.f_U = f_U;
  a.scratch = scratch;
  a.P = lay.points;
  a.precision = precision;
  a.ux_given = 0;
  return a;
}

}  // namespace

cudaError_t launch_pcg1d(const Layout1d& lay, const void* tw64, const void* tw32, int precision,
                         const double* eta, const double* hx, const double* b, double* x,
                         const SolveRec* given, int kind, double rtol, double rtol_inner,
                         int maxit, int max_refine, SolveRec* rec, void* ws, float* coef_df,
                         cudaStream_t s) {
  const PcgArgs a = pcg_args(lay, tw64, tw32, precision, eta, hx, b, x, given, kind, rtol,
                             rtol_inner, maxit, max_refine, rec, ws, coef_df);
  return d1::for_each_size(lay, s, [&](auto Lc, int first, int num, cudaStream_t cs) {
    return launch_form<decltype(Lc)::value>(lay, a, first, num, cs, PcgKernels{});
  }, [&](int first, int num, cudaStream_t cs) {
    return mr_launch_pcg(lay, first, num, precision, eta, hx, b, x, given, kind, rtol,
                         rtol_inner, maxit, max_refine, rec, ws, nullptr, cs);
  });
}

cudaError_t launch_pcg1d_ux(const Layout1d& lay, const void* tw64, const void* tw32,
                            int precision, const double* eta, const double* hx, const double* b,
                            double* x, int kind, double rtol, double rtol_inner, int maxit,
                            int max_refine, SolveRec* rec, void* ws, float* coef_df,
                            double* scratch, cudaStream_t s) {
  PcgArgs a = pcg_args(lay, tw64, tw32, precision, eta, hx, b, x, nullptr, kind, rtol,
                       rtol_inner, maxit, max_refine, rec, ws, coef_df);
  a.ux = scratch;
  return d1::for_each_size(lay, s, [&](auto Lc, int first, int num, cudaStream_t cs) {
    return launch_form<decltype(Lc)::value>(lay, a, first, num, cs, PcgKernels{});
  }, [&](int first, int num, cudaStream_t cs) {
    return mr_launch_pcg(lay, first, num, precision, eta, hx, b, x, nullptr, kind, rtol,
                         rtol_inner, maxit, max_refine, rec, ws, scratch, cs);
  });
}

cudaError_t launch_rhs1d(const Layout1d& lay, const void* tw64, const void* tw32, int precision,
                         double g, const double* eta, const double* u, const double* h,
                         const double* hx, double* f_eta, double* f_U, double* scratch,
                         cudaStream_t s) {
  const RhsArgs a = rhs_args(lay, tw64, tw32, precision, g, eta, u, h, hx, f_eta, f_U, scratch);
  return d1::for_each_size(lay, s, [&](auto Lc, int first, int num, cudaStream_t cs) {
    return launch_form<decltype(Lc)::value>(lay, a, first, num, cs, RhsKernels{});
  }, [&](int first, int num, cudaStream_t cs) {
    return mr_launch_rhs(lay, first, num, precision, g, eta, u, h, hx, f_eta, f_U, scratch, false, cs);
  });
}

cudaError_t launch_rhs1d_ux(const Layout1d& lay, const void* tw64, const void* tw32,
                            int precision, double g, const double* eta, const double* u,
                            const double* h, const double* hx, double* f_eta, double* f_U,
                            double* scratch, cudaStream_t s) {
  RhsArgs a = rhs_args(lay, tw64, tw32, precision, g, eta, u, h, hx, f_eta, f_U, scratch);
  a.ux_given = 1;
  return d1::for_each_size(lay, s, [&](auto Lc, int first, int num, cudaStream_t cs) {
    return launch_form<decltype(Lc)::value>(lay, a, first, num, cs, RhsKernels{});
  }, [&](int first, int num, cudaStream_t cs) {
    return mr_launch_rhs(lay, first, num, precision, g, eta, u, h, hx, f_eta, f_U, scratch, true, cs);
  });
}

cudaError_t launch_linimp_split(const Layout1d& lay, int l, int first, int num, const void* tw64,
                                const void* tw32, int precision, const SolveRec* A,
                                const double* eta, const double* hx, const double* u,
                                const double* U, const void* res0_hat, void* res1_hat, double c1,
                                double c0, bool solve, double* u_out, void* ux_out,
                                cudaStream_t s) {
  sp::LinArgs a;
  a.insts = lay.d_inst;
  a.ids = lay.d_ids;
  a.tw64 = static_cast<const cplx<double>*>(tw64);
  a.twdf = reinterpret_cast<const cplx<df>*>(static_cast<const char*>(tw32) + kTw32Bytes);
  a.A = A;
  a.eta = eta;
  a.hx = hx;
  a.u = u;
  a.U = U;
  a.res0 = static_cast<const cplx<double>*>(res0_hat);
  a.res1 = static_cast<cplx<double>*>(res1_hat);
  a.c1 = c1;
  a.c0 = c0;
  a.u_out = u_out;
  a.ux = ux_out;
  a.precision = precision;
  a.solve = solve;
  const int lcl = split_lcl(lay, l, precision == SGN_PREC_MIXED, [](int) { return 1; });
  switch (l) {
    case 8: return split_linimp_launch<8>(a, first, num, lcl, s);
    case 9: return split_linimp_launch<9>(a, first, num, lcl, s);
    case 10: return split_linimp_launch<10>(a, first, num, lcl, s);
    case 11: return split_linimp_launch<11>(a, first, num, lcl, s);
    case 12: return split_linimp_launch<12>(a, first, num, lcl, s);
    case 13: return split_linimp_launch<13>(a, first, num, lcl, s);
    case 14: return split_linimp_launch<14>(a, first, num, lcl, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_field_split(const Layout1d& lay, int l, int first, int num, const void* tw64,
                               const double* f, const double* eta, const double* hx, double* out,
                               cudaStream_t s) {
  const sp::FieldArgs a{lay.d_inst, lay.d_ids, static_cast<const cplx<double>*>(tw64), f, eta, hx,
                        out};
  const int lcl = split_lcl(lay, l, false, [](int) { return 1; });
  switch (l) {
    case 8: return split_field_launch<8>(a, first, num, lcl, s);
    case 9: return split_field_launch<9>(a, first, num, lcl, s);
    case 10: return split_field_launch<10>(a, first, num, lcl, s);
    case 11: return split_field_launch<11>(a, first, num, lcl, s);
    case 12: return split_field_launch<12>(a, first, num, lcl, s);
    case 13: return split_field_launch<13>(a, first, num, lcl, s);
    case 14: return split_field_launch<14>(a, first, num, lcl, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sgn
