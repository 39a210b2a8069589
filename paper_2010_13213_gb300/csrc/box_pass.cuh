// box_pass.cuh -- block-index DFT passes of the seven-launch box convolution (direct conjugate-pair form; box_fft.cuh
// has the in-register FFT form for 4..16 blocks), around k_box_mid.
//
// They serve FP32 arithmetic on FP64 fields, whose results the callers read in double: the order of the FP32 operations,
// and with it every digit beyond the sixth, is as it was before the line passes (lines.cuh), which everything else runs.
// The interface promises about 1e-6 and no order of operations, so this is a choice, not an accuracy requirement; it costs
// seven launches instead of five (96 x 96 x 48 ring: 108 us; FP32 fields take the line passes).
#pragma once
#include "box.cuh"

template <class R>
struct BoxTw {  // W_P^n = e^{-2 pi i n / P}, n < P = 2 nb of the pass's axis
  cx<R> w[2 * BOX_NB_MAX];
};

// The same with the block indices resolved by the caller: ob = scatter[bidx] (-1: skip), ab = the
// addend / mask block (aux[bidx], or ob without aux).
template <class R>
LGF_D void box_store_at(const OutSpec<R> &o, int ob, int ab, int m, int B3, R v) {
  if (ob < 0) return;
  const int64_t a = (int64_t)ab * B3 + m;
  if (o.add) v = v + o.add[a];
  if (o.mask && !(o.mask[a] & o.bits)) return;
  store_field<R>(o.dst, o.off + (int64_t)ob * B3 + m, o.dtype, v);
}

// ------------------------------------------------------------------ block-index DFTs
// Pass along axis `ax` for every line (the two other block coordinates within `ext`) and local cell m:
//   forward  X[.. k ..][m] = sum_{j < nb} W_P^{ j k} x[.. j ..][m],   k < P = 2 nb
//   inverse  y[.. j ..][m] = sum_{k < P}  W_P^{-j k} X[.. k ..][m],   j < nb (unnormalised)
// Both use the conjugate symmetry W_P^{j(P-k)} = conj(W_P^{jk}) (c = cos(2 pi jk/P), s = sin(2 pi jk/P)):
//   forward  A_k = sum_j c x_j, B_k = sum_j s x_j, X_k = A_k - i B_k, X_{P-k} = A_k + i B_k (1 <= k < P/2),
//   inverse  y_j += c (X_k + X_{P-k}) + i s (X_k - X_{P-k}) per input pair,
// so every multiply has a real coefficient: half the work of the complex products.  k = 0 and k = P/2
// (coefficients 1 and (-1)^j) are sums.  A real field keeps K1x in [0, P/2] (Hermitian half): its
// forward x pass stores X_k only and its inverse x pass takes X_{P-k} = conj(X_k) (real output).
// A CTA of NT threads owns REP groups of NT consecutive cells (taken one after the other) and a chunk of
// CH pair slots (forward) or outputs (inverse); grid = (B^3 / (NT REP), lines, field * nchunk + chunk).  The chunk's (c, s) sit in a shared table;
// the next input is fetched while the current one multiplies.  The first forward pass (gather) reads
// through the field's input specs, the last inverse pass (final) writes through its output specs.
// Field f's arrays start at in + f * fstride, out + f * fstride.
// NBT > 0 fixes nb = NBT at compile time for one-chunk passes (NBT - 1 <= CH forward, NBT <= CH inverse):
// the loops unroll, every coefficient index j q mod P is a constant, and the coefficients are read
// from the parameter table itself (no shared table, no barrier unless the gather/scatter tables need one).
template <class R>
LGF_D cx<R> box_coef(const BoxTw<R> &tw, int n) {  // (cos, sin)(2 pi n / P) from W_P^n
  return cx<R>{tw.w[n].re, -tw.w[n].im};
}

template <class R, int B, int CH, int NT, int REP, int NBT = 0>
__global__ void __launch_bounds__(NT) k_bdft_fwd(const cx<R> *__restrict__ in, cx<R> *__restrict__ out,
                                                 int64_t fstride, BoxGeom g, int ax, int3 ext, BoxTw<R> tw,
                                                 int gather, int nchunk, FwdSpecs sp) {
  constexpr int B3 = B * B * B;
  constexpr bool FIX = NBT > 0;
  __shared__ cx<R> TW[FIX ? 1 : BOX_NB_MAX][CH];  // (cos, sin)(2 pi j q / P) of the chunk's general slots
  const int nb = FIX ? NBT : geo_nb(g, ax), P = 2 * nb, half = nb;
  const int a1 = ax == 0 ? 1 : 0, a2 = ax == 2 ? 1 : 2;
  const int e1 = ax == 0 ? ext.y : ext.x;
  const int l1 = (int)blockIdx.y % e1, l2 = (int)blockIdx.y / e1;
  const int field = FIX ? (int)blockIdx.z : (int)blockIdx.z / nchunk, chunk = FIX ? 0 : (int)blockIdx.z % nchunk;
  const int pxf = box_pxu(g, field);
  if (ax != 0 && l1 >= pxf) return;  // a line beyond this field's K1x range (l1 is K1x for y and z)
  const bool realx = ax == 0 && pxf < P;
  // general slots q = 1 .. half - 1 in chunks of CH; chunk 0 also sums the slots q = 0 and q = half
  const int q0 = 1 + chunk * CH;
  const int nq = FIX ? NBT - 1 : max(0, min(CH, half - q0));
  const bool ends = chunk == 0;
  if (!FIX)
    for (int i = threadIdx.x; i < nb * CH; i += NT) {
      const int j = i / CH, c = i % CH;
      const int n = (j * (q0 + c)) % P;  // < 32 * 32: 32-bit
      TW[j][c] = box_coef(tw, n);
    }
  const int64_t bsa = geo_bs(g, ax) * (int64_t)B3;
  const int64_t lbase = ((int64_t)l1 * geo_bs(g, a1) + (int64_t)l2 * geo_bs(g, a2)) * B3;
  const int gsa = ax == 0 ? 1 : (ax == 1 ? g.nb[0] : g.nb[0] * g.nb[1]);
  const int gbase = l1 * (a1 == 0 ? 1 : g.nb[0]) + l2 * (a2 == 1 ? g.nb[0] : g.nb[0] * g.nb[1]);
  InSpec s0{}, s1{}, s2{};
  int ns = 0;
  if (gather) {
#pragma unroll
    for (int f = 0; f < BOX_MAXF; ++f)
      if (f == field) {
        s0 = sp.s[f][0];
        s1 = sp.s[f][1];
        s2 = sp.s[f][2];
        ns = sp.n[f];
      }
  }
  // the line's source block of every input j and spec (the same for all cells of the CTA)
  __shared__ int GI[3][BOX_NB_MAX];
  if (gather)
    for (int j = threadIdx.x; j < nb; j += NT) {
      const int bidx = gbase + j * gsa;
      GI[0][j] = ns > 0 ? s0.gather[bidx] : -1;
      GI[1][j] = ns > 1 ? s1.gather[bidx] : -1;
      GI[2][j] = ns > 2 ? s2.gather[bidx] : -1;
    }
  const cx<R> *src = in + field * fstride + lbase;
  cx<R> *dst = out + field * fstride + lbase;
  if (!FIX || gather) __syncthreads();
  // REP groups of NT consecutive cells per CTA, one after the other (the table serves them all)
#pragma unroll 1
  for (int rep = 0; rep < REP; ++rep) {
  const int m = (blockIdx.x * REP + rep) * NT + threadIdx.x;
  auto fetch = [&](int j) -> cx<R> {
    if (!gather) return ld_stream(src + j * bsa + m);  // dead after this pass: keep L2 for its output
    R re = RT<R>::zero(), im = RT<R>::zero();
    auto add = [&](const InSpec &q, int si) {
      const int idx = GI[si][j];
      if (idx < 0) return;
      const int64_t e = (int64_t)idx * B3 + m;
      if (q.mask && !(q.mask[e] & q.bits)) return;
      const R v = load_field<R>(q.src, e, q.dtype);
      if (q.part != 0) im = im + v;
      if (q.part != 1) re = re + v;
    };
    if (ns > 0) add(s0, 0);
    if (ns > 1) add(s1, 1);
    if (ns > 2) add(s2, 2);
    return cx<R>{re, im};
  };
  // j = 0: every coefficient is 1
  cx<R> x = fetch(0);
  cx<R> A[CH], Bv[CH];
#pragma unroll
  for (int k = 0; k < CH; ++k) {
    A[k] = x;
    Bv[k] = cx_zero<R>();
  }
  // slots 0 and half (coefficients 1 and (-1)^j) from the sums over even and odd j
  cx<R> Se = x, So = cx_zero<R>();
  auto accumulate = [&](int j, const cx<R> &xj) {
    if (ends) {
      if (j & 1) So = cadd(So, xj);
      else Se = cadd(Se, xj);
    }
#pragma unroll
    for (int k = 0; k < CH; ++k) {
      if (k < nq) {
        const cx<R> w = FIX ? box_coef(tw, (j * (q0 + k)) % P) : TW[FIX ? 0 : j][k];
        A[k] = cx<R>{rfma(A[k].re, w.re, xj.re), rfma(A[k].im, w.re, xj.im)};
        Bv[k] = cx<R>{rfma(Bv[k].re, w.im, xj.re), rfma(Bv[k].im, w.im, xj.im)};
      }
    }
  };
  if constexpr (FIX) {
    cx<R> xs[NBT];
#pragma unroll
    for (int j = 1; j < NBT; ++j) xs[j] = fetch(j);
#pragma unroll
    for (int j = 1; j < NBT; ++j) accumulate(j, xs[j]);
  } else {
    cx<R> xn = nb > 1 ? fetch(1) : cx_zero<R>();
    for (int j = 1; j < nb; ++j) {
      x = xn;
      if (j + 1 < nb) xn = fetch(j + 1);
      accumulate(j, x);
    }
  }
  if (ends) {
    dst[m] = cnorm(cadd(Se, So));
    dst[half * bsa + m] = cnorm(csub(Se, So));
  }
#pragma unroll
  for (int k = 0; k < CH; ++k) {
    if (k < nq) {
      const int q = q0 + k;
      const cx<R> a = A[k], b = Bv[k];
      dst[q * bsa + m] = cx<R>{rnorm(a.re + b.im), rnorm(a.im - b.re)};
      if (!realx) dst[(P - q) * bsa + m] = cx<R>{rnorm(a.re - b.im), rnorm(a.im + b.re)};
    }
  }
  }
}

template <class R, int B, int CH, int NT, int REP, int NBT = 0>
__global__ void __launch_bounds__(NT) k_bdft_inv(const cx<R> *__restrict__ in, cx<R> *__restrict__ out,
                                                 int64_t fstride, BoxGeom g, int ax, int3 ext, BoxTw<R> tw,
                                                 int final, int nchunk, InvOuts<R> outs, double scale) {
  constexpr int B3 = B * B * B;
  constexpr bool FIX = NBT > 0;
  __shared__ cx<R> TW[FIX ? 1 : BOX_NB_MAX][CH];  // (cos, sin)(2 pi q o / P) for the general input slots
  const int nb = FIX ? NBT : geo_nb(g, ax), P = 2 * nb, half = nb;
  const int a1 = ax == 0 ? 1 : 0, a2 = ax == 2 ? 1 : 2;
  const int e1 = ax == 0 ? ext.y : ext.x;
  const int l1 = (int)blockIdx.y % e1, l2 = (int)blockIdx.y / e1;
  const int field = FIX ? (int)blockIdx.z : (int)blockIdx.z / nchunk, chunk = FIX ? 0 : (int)blockIdx.z % nchunk;
  const int pxf = box_pxu(g, field);
  if (ax != 0 && l1 >= pxf) return;  // a line beyond this field's K1x range (l1 is K1x for y and z)
  const bool realx = ax == 0 && pxf < P;
  const int o0 = chunk * CH;
  const int no = FIX ? NBT : min(CH, nb - o0);
  if (!FIX)
    for (int i = threadIdx.x; i < half * CH; i += NT) {
      const int q = i / CH, c = i % CH;
      const int n = (q * (o0 + c)) % P;  // < 32 * 32: 32-bit
      TW[q][c] = box_coef(tw, n);
    }
  const int64_t bsa = geo_bs(g, ax) * (int64_t)B3;
  const int64_t lbase = ((int64_t)l1 * geo_bs(g, a1) + (int64_t)l2 * geo_bs(g, a2)) * B3;
  const int gsa = ax == 0 ? 1 : (ax == 1 ? g.nb[0] : g.nb[0] * g.nb[1]);
  const int gbase = l1 * (a1 == 0 ? 1 : g.nb[0]) + l2 * (a2 == 1 ? g.nb[0] : g.nb[0] * g.nb[1]);
  OutSpec<R> ore{}, oim{};
  if (final) {
#pragma unroll
    for (int f = 0; f < BOX_MAXF; ++f)
      if (f == field) {
        ore = outs.re[f];
        oim = outs.im[f];
      }
  }
  const R sc = RT<R>::from(scale);
  // output blocks of the chunk's outputs (the same for all cells of the CTA): scatter and addend / mask
  __shared__ int SO[2][CH], SX[2][CH];
  if (final && threadIdx.x < CH) {
    const int k = threadIdx.x, bidx = gbase + (o0 + k) * gsa;
    int ob = -1, ab = -1;
    if (k < no && ore.scatter) {
      ob = ore.scatter[bidx];
      ab = ob >= 0 ? (ore.aux ? ore.aux[bidx] : ob) : -1;
    }
    SO[0][k] = ob;
    SX[0][k] = ab;
    ob = ab = -1;
    if (k < no && oim.scatter) {
      ob = oim.scatter[bidx];
      ab = ob >= 0 ? (oim.aux ? oim.aux[bidx] : ob) : -1;
    }
    SO[1][k] = ob;
    SX[1][k] = ab;
  }
  if (!FIX || final) __syncthreads();
  // REP groups of NT consecutive cells per CTA, one after the other (the table serves them all)
#pragma unroll 1
  for (int rep = 0; rep < REP; ++rep) {
  const int m = (blockIdx.x * REP + rep) * NT + threadIdx.x;
  const cx<R> *src = in + field * fstride + lbase + m;
  // general input slot q (1 <= q < half): X_q and X_{P-q}, the latter conj(X_q) for a real field
  // the input is dead after this pass: streaming loads keep L2 for its output
  auto fetch = [&](int q, cx<R> &xa, cx<R> &xb) {
    xa = ld_stream(src + q * bsa);
    xb = realx ? conj(xa) : ld_stream(src + (P - q) * bsa);
  };
  // slots 0 and half: coefficients 1 and (-1)^o
  const cx<R> X0 = ld_stream(src), Xh = ld_stream(src + half * bsa);
  cx<R> y[CH];
#pragma unroll
  for (int k = 0; k < CH; ++k) y[k] = ((o0 + k) & 1) ? csub(X0, Xh) : cadd(X0, Xh);
  auto accumulate = [&](int q, const cx<R> &xa, const cx<R> &xb) {
    const cx<R> U = cadd(xa, xb), V = csub(xa, xb);
#pragma unroll
    for (int k = 0; k < CH; ++k) {
      if (k < no) {
        if (o0 + k == 0) {
          y[k] = cadd(y[k], U);
        } else {
          const cx<R> w = FIX ? box_coef(tw, (q * (o0 + k)) % P) : TW[FIX ? 0 : q][k];
          y[k].re = rdot2(y[k].re, w.re, U.re, w.im, V.im, -1.0f);
          if (!realx) y[k].im = rdot2(y[k].im, w.re, U.im, w.im, V.re, 1.0f);
        }
      }
    }
  };
  if constexpr (FIX) {
    cx<R> xa[NBT], xb[NBT];
#pragma unroll
    for (int q = 1; q < NBT; ++q) fetch(q, xa[q], xb[q]);
#pragma unroll
    for (int q = 1; q < NBT; ++q) accumulate(q, xa[q], xb[q]);
  } else {
    cx<R> na = cx_zero<R>(), nbv = cx_zero<R>();
    if (half > 1) fetch(1, na, nbv);
    for (int q = 1; q < half; ++q) {
      const cx<R> xa = na, xb = nbv;
      if (q + 1 < half) fetch(q + 1, na, nbv);
      accumulate(q, xa, xb);
    }
  }
  if (!final) {
    cx<R> *dst = out + field * fstride + lbase + m;
#pragma unroll
    for (int k = 0; k < CH; ++k)
      if (k < no) dst[(o0 + k) * bsa] = cnorm(y[k]);
    continue;
  }
#pragma unroll
  for (int k = 0; k < CH; ++k) {
    if (k >= no) continue;
    const cx<R> v = cnorm(y[k]);
    box_store_at<R>(ore, SO[0][k], SX[0][k], m, B3, v.re * sc);
    if (!realx) box_store_at<R>(oim, SO[1][k], SX[1][k], m, B3, v.im * sc);
  }
  }
}

