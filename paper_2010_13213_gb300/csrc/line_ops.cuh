// line_ops.cuh -- host side of the line transforms (lines.cuh): the launch of one pass for a line shape.
#pragma once
#include "internal.h"
#include "lines.cuh"

namespace lgf {

enum LineKind { LINE_FWD_X, LINE_FWD_Y, LINE_MID, LINE_INV_Y, LINE_INV_X };

template <class R>
struct LinePass {
  const typename Ar<R>::M *in = nullptr;
  typename Ar<R>::M *out = nullptr;
  LineGeom g;
  const LineTw<R> *tw = nullptr;          // of the pass's axis
  const typename Ar<R>::T *twl = nullptr;
  const FwdSpecs *sp = nullptr;
  const InvOuts<R> *outs = nullptr;
  const R *Gf = nullptr;
  double scale = 1.0;
  int nfields = 0, wmax = 0;              // fields of the launch, their widest frequency row
  bool fine = false;                      // renormalised sums where the shape has them (LineFine)
  cudaStream_t st = nullptr;
};

template <class R, int M, int NB, bool FINE>
void line_launch_as(LineKind kind, const LinePass<R> &p) {
  constexpr int TL = LineTile<M, NB>::TL, NT = LineTile<M, NB>::NT;
  constexpr size_t smx = line_smem<R, M, NB, true>(), smy = line_smem<R, M, NB, false>(),
                   smm = line_smem_mid<R, M, NB>();
  static PerDevice done[5];
  const unsigned tiles_yz = (unsigned)((p.g.n[1] * p.g.n[2] + TL - 1) / TL), tiles_w = (unsigned)((p.wmax + TL - 1) / TL);
  const unsigned nz = (unsigned)p.g.n[2], nf = (unsigned)p.nfields;
  switch (kind) {
    case LINE_FWD_X:
      smem_limit(done[kind], k_line_fwd<R, M, NB, true>, smx);
      k_line_fwd<R, M, NB, true><<<dim3(tiles_yz, 1, nf), NT, smx, p.st>>>(p.in, p.out, p.g, *p.tw, p.twl, *p.sp);
      break;
    case LINE_FWD_Y:
      smem_limit(done[kind], k_line_fwd<R, M, NB, false>, smy);
      k_line_fwd<R, M, NB, false><<<dim3(tiles_w, nz, nf), NT, smy, p.st>>>(p.in, p.out, p.g, *p.tw, p.twl, *p.sp);
      break;
    case LINE_MID: {
      const unsigned tiles = (unsigned)(((int64_t)p.g.P[1] * p.g.M[1] * p.wmax + TL - 1) / TL);
      smem_limit(done[kind], k_line_mid<R, M, NB, FINE>, smm);
      k_line_mid<R, M, NB, FINE><<<dim3(tiles, 1, nf), NT, smm, p.st>>>(p.out, p.Gf, p.g, *p.tw, p.twl);
      break;
    }
    case LINE_INV_Y:
      smem_limit(done[kind], k_line_inv<R, M, NB, false, FINE>, smy);
      k_line_inv<R, M, NB, false, FINE><<<dim3(tiles_w, nz, nf), NT, smy, p.st>>>(p.in, p.out, p.g, *p.tw, p.twl, *p.outs,
                                                                                 1.0);
      break;
    case LINE_INV_X:
      smem_limit(done[kind], k_line_inv<R, M, NB, true, FINE>, smx);
      k_line_inv<R, M, NB, true, FINE><<<dim3(tiles_yz, 1, nf), NT, smx, p.st>>>(p.in, p.out, p.g, *p.tw, p.twl, *p.outs,
                                                                                p.scale);
      break;
  }
}
template <class R, int M, int NB>
void line_launch(LineKind kind, const LinePass<R> &p) {
  if constexpr (LineFine<R, M>::value) {
    if (p.fine) return line_launch_as<R, M, NB, true>(kind, p);
  }
  line_launch_as<R, M, NB, false>(kind, p);
}

// The pass for NB in [LO, HI] (steps of ST); one translation unit per range and arithmetic.
template <class R, int M, int LO, int HI, int ST>
bool line_range(int nb, LineKind kind, const LinePass<R> &p);

#define LINE_RANGE_DEFINE(R, M, LO, HI, ST)                                                   \
  template <int NB>                                                                           \
  static bool line_step_##M(int nb, LineKind kind, const LinePass<R> &p) {                    \
    if (nb == NB) {                                                                           \
      line_launch<R, M, NB>(kind, p);                                                         \
      return true;                                                                            \
    }                                                                                         \
    if constexpr (NB + ST <= HI) return line_step_##M<NB + ST>(nb, kind, p);                  \
    return false;                                                                             \
  }                                                                                           \
  template <>                                                                                 \
  bool line_range<R, M, LO, HI, ST>(int nb, LineKind kind, const LinePass<R> &p) {            \
    return line_step_##M<LO>(nb, kind, p);                                                    \
  }

// The instantiated ranges (line_{f64,f32,df}_{a,b,c,d}.cu).
#define LINE_RANGE_DECLARE(R)                                                       \
  template <>                                                                       \
  bool line_range<R, 16, 1, 6, 1>(int, LineKind, const LinePass<R> &);              \
  template <>                                                                       \
  bool line_range<R, 16, 7, 11, 1>(int, LineKind, const LinePass<R> &);             \
  template <>                                                                       \
  bool line_range<R, 16, 12, 16, 1>(int, LineKind, const LinePass<R> &);            \
  template <>                                                                       \
  bool line_range<R, 8, 1, 15, 2>(int, LineKind, const LinePass<R> &);              \
  template <>                                                                       \
  bool line_range<R, 8, 2, 4, 2>(int, LineKind, const LinePass<R> &);
LINE_RANGE_DECLARE(double)
LINE_RANGE_DECLARE(float)
LINE_RANGE_DECLARE(df)

template <class R>
inline bool line_pass(int B, int nb, LineKind kind, const LinePass<R> &p) {
  const int NB = line_NB(B, nb);
  if (line_M(B, nb) == 8 && NB % 2 == 0) return line_range<R, 8, 2, 4, 2>(NB, kind, p);
  if (line_M(B, nb) == 8) return line_range<R, 8, 1, 15, 2>(NB, kind, p);
  if (NB <= 6) return line_range<R, 16, 1, 6, 1>(NB, kind, p);
  if (NB <= 11) return line_range<R, 16, 7, 11, 1>(NB, kind, p);
  return line_range<R, 16, 12, 16, 1>(NB, kind, p);
}

}  // namespace lgf
