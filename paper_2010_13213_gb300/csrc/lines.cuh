// lines.cuh -- block-index FFT mode: the lattice convolution of a level box (Sec. 2.2, Eq. (eq:lgf_convolution)) as
// five passes of whole-line transforms.
//
// The box of n_a cells per axis is embedded in a periodic lattice of L_a = 2 n_a, large enough that the circular
// convolution with the circularly laid out LGF equals the linear one on the box.  The passes take one axis each:
//     x forward  caller's blocks (gathered) -> A[z][y][fx]
//     y forward  A -> C[z][fy][fx]
//     z          C -> C: forward, times Ghat(fz, fy, fx), inverse, in shared memory
//     y inverse  C -> A[z][y][fx]
//     x inverse  A -> caller's blocks (scattered)
// The zero padding is never stored: a line holds n_a values between passes of its own axis, so the arrays are two
// and four times the box instead of eight, and an axis is transformed only on the lines that the passes before it
// have made (2, 4 and 8 n^3 points instead of 8 on every axis).
//
// A line has n = M NB cells (M = 16, or 8 for 8^3 blocks of an odd count, of two and of four), L = 2 n = P M frequencies.
// Its even and odd frequencies K = 2 K' + h (h = 0, 1) are the n-point DFTs of x_i and of x_i W_L^i, each in two steps:
// one thread per (line, m) runs NB-point DFTs over the inputs of its m, one per (line, K1) M-point DFTs over m, with
// one exchange through shared memory.
//   NB = NO N2 with NO odd, N2 a power of two; the NO-point DFT is coprime to the rest and takes no twiddles (Good's
//   mapping): i = (NO (M j2 + m) + M N2 j3) mod n,  K' = k3 mod NO = k2 + N2 K2 mod M N2,  slot K1 = 2 (k3 N2 + k2) + h,
//     t[K1][m] = W_{M N2}^{m k2} sum_{j2, j3} x_i W_NO^{j3 k3} W_N2^{j2 k2},    X[K] = sum_m t[K1][m] W_M^{m K2}.
//   For NB = 3 that is 3 complex products per m of both halves (the turns by W_L^i) where the form i = M J + m,
//   t[K1][m] = W_L^{m K1} sum_J x_i W_P^{J K1} has 7; NB = 7: 7 for 19; NB = 6: 12 for 16.
// The inverse is the conjugate of the forward transform of the conjugate, so every pass runs forward code: the z pass
// conjugates when it multiplies by Ghat (real, G is even), and the last pass negates the imaginary part.  The inverse
// needs the first n outputs only: the sum of the even K's n-point DFT and of the odd K's turned by W_L^i.
// Double-float values are renormalised (norm) around every product and when they leave a step: sums and products round
// in proportion to the low part.  With one renormalisation per product alone the error of the two rings was 7.1e-15;
// with these it is 4.9e-15, for 3 % of the time; the block-index passes had 5.7e-15.  Where a result is differenced the
// inverse passes also renormalise after every sum (LineFine).
//
// Two real fields ride as real and imaginary part of one complex field.  A field with a zero imaginary part keeps one
// of every pair of x slots K1 that the frequencies K and -K share: NB + 1 of them.
// A frequency row is [K2][kept K1]; LineGeom::fx gives the frequency K of a row's element.
//
// What bounds them: the FP32 pipe in double-float, the FP64 pipe in double (2 lanes a clock and SM), traffic and latency
// in FP32.  One double-float solve of the 96 x 96 x 48 ring (three components) takes 154 us, 62 us of it in the z pass
// (its FP32 pipe busy 72 % of the time); as block-index passes around k_box_mid it took 236 us.  Two rings on
// 96 x 96 x 112: 374 us (546), FP64 ring 753 us (1,141), FP32 two rings 113 us (204).
#pragma once
#include <type_traits>

#include "arith.cuh"
#include "box.cuh"

namespace lgf {

// Lines per CTA: enough (line, K1) tasks for the 128 threads with small NB, shared memory for three or four CTAs per SM
// with large NB.  Measured on the rings: CTAs of 64 and 96 threads 2 to 6 % slower, of 256 threads 3 % (NB = 6) to 20 %
// (NB = 10, 14), half as many lines 23 % slower for NB = 3.  Lines of one or two M-point steps come from boxes of a few
// thousand lines: small CTAs spread their arithmetic over the chip (32^3 cells in FP64, 32 lines and 128 threads per CTA:
// 92 us, these: 72 us; in double-float, one component, 53 and 42 us).
template <int M, int NB>
struct LineTile {
  static constexpr int NT = NB <= 2 ? 64 : 128;
  static constexpr int TL = NB == 2 ? 8 : (NB <= 5 ? 16 : 8);
  // CTAs per SM that the registers are limited for: 80 registers up to NB = 6 (the M-point step alone holds 64),
  // more for the NB-point step of wide boxes, where spills cost more than the occupancy gains
  static constexpr int MB = NB <= 2 ? 12 : NB <= 6 ? 6 : (NB == 7 ? 5 : (NB <= 10 ? 4 : (NB < 16 ? 3 : 2)));
};

// 4- or 8-byte asynchronous copies to shared memory, and the wait for the thread's own.
template <class R>
LGF_D void line_copy_async(R *dst, const R *src) {
  static_assert(sizeof(R) == 4 || sizeof(R) == 8, "cp.async size");
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "n"(sizeof(R)));
}
LGF_D void line_copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

struct LineGeom {
  int n[3], P[3], M[3];   // per axis: cells, block frequencies, points of the second step
  int nb[3];              // caller's blocks per axis
  int shift;              // log2 of the caller's block edge
  int nc;                 // fields [0, nc) are complex, the others real
  int wc, wr;             // frequency row length of a complex and of a real field
  const int32_t *fxc, *fxr;  // x frequency of a row's element, complex and real fields
  int64_t astride, cstride;  // field strides of A and C
};
// Line shapes whose inverse and z kernels have a form with renormalised sums (FINE, ArFine): double-float in 16-point
// steps.  It serves composite solves and the velocity refresh, which difference the result (corrections, the curl).  With
// lazy sums composite solves on 16^3 blocks had 1.15 times the error of the block-index passes (mean of 24 meshes, up to
// 1.5 times) and have 0.99 times now, refreshes of a few blocks 1.28 and 1.15; plain solves have 0.81 times with lazy sums
// and keep them.  Three-level ring 4.45 -> 4.68 ms, refresh of 6 x 6 x 3 blocks 311 -> 324 us.  Lines in 8-point steps come
// from 8^3 blocks, where lazy sums have 0.48 to 0.86 times that error in composite solves too (5 x 7 x 3 blocks with
// renormalised sums: 36.9 -> 40.5 us).
template <class R, int M>
struct LineFine {
  static constexpr bool value = std::is_same<R, df>::value && M == 16;
};
LGF_HD int line_width(const LineGeom &g, int field) { return field < g.nc ? g.wc : g.wr; }

// Shared memory element of (K1, m, line).  x passes run m (first step) and K1 (second step) over the lanes, y and z
// passes the line: the strides keep eight neighbouring lanes of either on different banks.
template <int M, int TL, bool X>
struct LineSmem {
  static constexpr int SM = X ? TL + 1 : TL, SK = X ? M * (TL + 1) + 1 : M * TL + (TL < 8 ? TL : (TL % 8 ? TL % 8 : 8));
  static LGF_D int at(int k1, int m, int line) { return k1 * SK + m * SM + line; }
};
template <class R, int M, int NB, bool X>
constexpr size_t line_smem() {
  return sizeof(typename Ar<R>::M) * (size_t)(2 * NB) * LineSmem<M, LineTile<M, NB>::TL, X>::SK;
}
template <class R, int M, int NB>
constexpr size_t line_smem_mid() {
  return line_smem<R, M, NB, false>() + sizeof(R) * (size_t)(M * NB + 1) * LineTile<M, NB>::TL;
}

// The factors of a line (see above) and its index maps.
template <int M, int NB>
struct LineMap {
  static constexpr int N2 = NB & -NB, NO = NB / N2, Q2 = M * N2, n = M * NB;
  static constexpr int CO = Q2 * inverse_mod(Q2, NO) % n, C2 = NO * inverse_mod(NO, Q2) % n;  // CRT weights of k3, k'
  // cell of input j = j3 N2 + j2 of thread m
  static LGF_D int cell(int j, int m) {
    const int c = NO * M * (j % N2) + Q2 * (j / N2);
    const int i = (c >= n ? c - n : c) + NO * m;
    return i >= n ? i - n : i;
  }
  // K' of slot q = k3 N2 + k2 at K2 = 0, and its step from K2 to K2 + 1 (mod n)
  static LGF_D int freq(int q) { return ((q / N2) * CO + (q % N2) * C2) % n; }
  static constexpr int STEP = (int)((int64_t)N2 * C2 % n);
  // the slot of the frequencies -K: -K = 2 (-K' - h) + h
  static LGF_HD constexpr int mirror(int q, int h) {
    const int k3 = q / N2, k2 = q % N2;
    return h ? (NO - 1 - k3) * N2 + N2 - 1 - k2 : (NO - k3) % NO * N2 + (N2 - k2) % N2;
  }
  // slot K1 that holds frequency K at K2 = 0
  static LGF_D int slot(int K) { return 2 * (((K >> 1) % NO) * N2 + (K >> 1) % N2) + (K & 1); }
};
template <class A, int M, int NB>
LGF_D void line_dft(typename A::V (&v)[NB], const LineTw<typename A::Real> &tw) {  // over (j3, j2)
  typedef LineMap<M, NB> Mp;
  constexpr int NO = Mp::NO, N2 = Mp::N2;
  if constexpr (NO == 1) {
    Dft<A, NB, 2 * NB>::run(v, tw);
  } else {
    if constexpr (N2 > 1) {
#pragma unroll
      for (int j3 = 0; j3 < NO; ++j3) {
        typename A::V z[N2];
#pragma unroll
        for (int j = 0; j < N2; ++j) z[j] = v[j3 * N2 + j];
        Dft<A, N2, 2 * NB>::run(z, tw);
#pragma unroll
        for (int j = 0; j < N2; ++j) v[j3 * N2 + j] = z[j];
      }
    }
#pragma unroll
    for (int k2 = 0; k2 < N2; ++k2) {
      typename A::V z[NO];
#pragma unroll
      for (int j = 0; j < NO; ++j) z[j] = v[j * N2 + k2];
      Dft<A, NO, 2 * NB>::run(z, tw);
#pragma unroll
      for (int j = 0; j < NO; ++j) v[j * N2 + k2] = z[j];
    }
  }
}

// First step of a (line, m): the NB inputs from load(v) (kept in the odd slots for the odd half), t[2 q + h][m] to S.
// `twl` is W_L^n, n < L.  One copy of the DFT serves both halves (the loop stays rolled: instruction cache).
// x lines load their cells in memory order (v[j] = cell M j + m, coalesced) and pick the inputs of m out of shared
// memory: the M threads of a line are in one warp.
template <class R, int M, int NB, int TL, bool X, class Load>
LGF_D void line_split(typename Ar<R>::M *S, int m, int line, const LineTw<R> &tw,
                      const typename Ar<R>::T *__restrict__ twl, Load load) {
  typedef Ar<R> A;
  typedef LineSmem<M, TL, X> Sm;
  typedef LineMap<M, NB> Mp;
  constexpr bool PERM = X && Mp::NO > 1;  // otherwise cell(j, m) = M j + m, or load gives that order
  auto kept = [&](int j) {
    if (!PERM) return A::ld(S + Sm::at(2 * j + 1, m, line));
    const int i = Mp::cell(j, m);
    return A::ld(S + Sm::at(2 * (i / M) + 1, i % M, line));
  };
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    typename A::V v[NB];
    if (h == 0) {
      load(v);
#pragma unroll
      for (int j = 0; j < NB; ++j) A::st(S + Sm::at(2 * j + 1, m, line), v[j]);
      if (PERM) {
        __syncwarp();
#pragma unroll
        for (int j = 0; j < NB; ++j) v[j] = kept(j);
      }
    } else {
#pragma unroll
      for (int j = 0; j < NB; ++j) v[j] = kept(j);
      if (PERM) __syncwarp();
#pragma unroll
      for (int j = 0; j < NB; ++j) v[j] = A::mul(v[j], twl[Mp::cell(j, m)]);
    }
    line_dft<A, M, NB>(v, tw);
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      v[q] = A::norm(v[q]);
      if (q % Mp::N2) v[q] = A::mul(v[q], twl[m * (q % Mp::N2) * 2 * Mp::NO]);
      A::st(S + Sm::at(2 * q + h, m, line), v[q]);
    }
  }
}

// Last step of an inverse (line, m): the M-point sums of slot K1 from S (twiddled here), the NB outputs to put(y), cells
// as load gives them; pre() before the odd half, for loads that put needs.  `half` (x axis): of a slot and its mirror
// only the lower is held; with u the twiddled sum of the held one, the other's is conj(u), times W_{M N2}^{-m} for h = 1.
template <class A, int M, int NB, int TL, bool X, class Pre, class Put>
LGF_D void line_merge(typename A::M *S, int m, int line, bool half, const LineTw<typename A::Real> &tw,
                      const typename A::T *__restrict__ twl, Pre pre, Put put) {
  typedef LineSmem<M, TL, X> Sm;
  typedef LineMap<M, NB> Mp;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    typename A::V v[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int mq = h ? Mp::mirror(q, 1) : Mp::mirror(q, 0);
      if (X && half && mq < q) {  // uniform over the CTA
        const int ex = mq % Mp::N2 + h;
        v[q] = A::ld(S + Sm::at(2 * mq + h, m, line));
        if (ex) v[q] = A::mul(v[q], twl[m * ex * 2 * Mp::NO]);
        v[q] = A::conj(v[q]);
      } else {
        v[q] = A::ld(S + Sm::at(2 * q + h, m, line));
        if (q % Mp::N2) v[q] = A::mul(v[q], twl[m * (q % Mp::N2) * 2 * Mp::NO]);
      }
    }
    if (h) pre();
    line_dft<A, M, NB>(v, tw);
    if (h == 0) {
#pragma unroll
      for (int j = 0; j < NB; ++j) A::st(S + Sm::at(2 * j, m, line), v[j]);
    } else {
#pragma unroll
      for (int j = 0; j < NB; ++j)
        v[j] = A::add(A::ld(S + Sm::at(2 * j, m, line)), A::mul(A::norm(v[j]), twl[Mp::cell(j, m)]));
      if constexpr (X && Mp::NO > 1) {  // to memory order
        __syncwarp();
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          const int i = Mp::cell(j, m);
          A::st(S + Sm::at(i / M, i % M, line), v[j]);
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < NB; ++j) v[j] = A::ld(S + Sm::at(j, m, line));
      }
      put(v);
    }
  }
}

// x forward (X): grid (n_y n_z / TL, 1, fields), lines (y, z) with y fastest (n_y n_z is a multiple of 64, so that
// every x tile is full); y forward: grid (ceil(width / TL), n_z,
// fields), lines the frequency slots of a row.
template <class R, int M, int NB, bool X>
__global__ void __launch_bounds__(LineTile<M, NB>::NT, LineTile<M, NB>::MB)
    k_line_fwd(const typename Ar<R>::M *__restrict__ in, typename Ar<R>::M *__restrict__ out,
               const __grid_constant__ LineGeom g, const __grid_constant__ LineTw<R> tw,
               const typename Ar<R>::T *__restrict__ twl, const __grid_constant__ FwdSpecs sp) {
  typedef Ar<R> A;
  constexpr int NT = LineTile<M, NB>::NT, TL = LineTile<M, NB>::TL, P = 2 * NB;
  typedef LineSmem<M, TL, X> Sm;
  extern __shared__ __align__(16) unsigned char line_smem_raw[];
  typename A::M *S = reinterpret_cast<typename A::M *>(line_smem_raw);
  const int field = blockIdx.z, W = line_width(g, field);
  const int line0 = blockIdx.x * TL;
  const int nlines = X ? g.n[1] * g.n[2] : W;
  if (line0 >= nlines) return;
  const bool half = X && field >= g.nc;
  bool any = !X;
  for (int t = threadIdx.x; t < TL * M; t += NT) {
    const int m = X ? t % M : t / TL, l = X ? t / M : t % TL, line = line0 + l;
    if (line >= nlines) continue;
    if constexpr (X) {
      const int sh = g.shift, msk = (1 << sh) - 1, ns = sp.n[field];
      const int y = line % g.n[1], z = line / g.n[1];
      const int64_t brow = ((int64_t)(z >> sh) * g.nb[1] + (y >> sh)) * g.nb[0];
      const int crow = (((z & msk) << sh) + (y & msk)) << sh;
      line_split<R, M, NB, TL, X>(S, m, l, tw, twl, [&](typename A::V (&v)[NB]) {
        R re[NB], im[NB];
#pragma unroll
        for (int j = 0; j < NB; ++j) re[j] = im[j] = RT<R>::zero();
#pragma unroll 1
        for (int s = 0; s < ns; ++s) {  // all block indices, then all masks, then all values
          const int32_t *gather = sp.s[field][s].gather + brow;
          const void *src = sp.s[field][s].src;
          const uint8_t *mask = sp.s[field][s].mask;
          const int dtype = sp.s[field][s].dtype, bits = sp.s[field][s].bits, part = sp.s[field][s].part;
          int64_t e[NB];
#pragma unroll
          for (int j = 0; j < NB; ++j) {
            const int x = M * j + m, idx = __ldg(gather + (x >> sh));
            any |= idx >= 0;
            e[j] = idx < 0 ? -1 : ((int64_t)idx << (3 * sh)) + crow + (x & msk);
          }
          if (mask) {
            int mk[NB];
#pragma unroll
            for (int j = 0; j < NB; ++j) mk[j] = e[j] < 0 ? 0 : __ldg(mask + e[j]) & bits;
#pragma unroll
            for (int j = 0; j < NB; ++j)
              if (!mk[j]) e[j] = -1;
          }
          R val[NB];
          if (dtype == 2) {
#pragma unroll
            for (int j = 0; j < NB; ++j) val[j] = e[j] < 0 ? RT<R>::zero() : ((const R *)src)[e[j]];
          } else if (dtype == 0) {
            double w[NB];
#pragma unroll
            for (int j = 0; j < NB; ++j) w[j] = e[j] < 0 ? 0.0 : ((const double *)src)[e[j]];
#pragma unroll
            for (int j = 0; j < NB; ++j) val[j] = RT<R>::from(w[j]);
          } else {
            float w[NB];
#pragma unroll
            for (int j = 0; j < NB; ++j) w[j] = e[j] < 0 ? 0.0f : ((const float *)src)[e[j]];
#pragma unroll
            for (int j = 0; j < NB; ++j) val[j] = RT<R>::from(w[j]);
          }
          if (part != 1) {
#pragma unroll
            for (int j = 0; j < NB; ++j) re[j] = re[j] + val[j];
          }
          if (part != 0) {
#pragma unroll
            for (int j = 0; j < NB; ++j) im[j] = im[j] + val[j];
          }
        }
#pragma unroll
        for (int j = 0; j < NB; ++j) v[j] = A::make(re[j], im[j]);
      });
    } else {
      const typename A::M *src = in + field * g.astride + (int64_t)blockIdx.y * g.n[1] * W + line;
      line_split<R, M, NB, TL, X>(S, m, l, tw, twl, [&](typename A::V (&v)[NB]) {
#pragma unroll
        for (int j = 0; j < NB; ++j) v[j] = A::ld(src + (int64_t)LineMap<M, NB>::cell(j, m) * W);
      });
    }
  }
  any = __syncthreads_or(any);
  const int nk = half ? NB + 1 : P;
  for (int t = threadIdx.x; t < TL * nk; t += NT) {
    const int c = X ? t % nk : t / TL, l = X ? t / nk : t % TL, line = line0 + l;
    if (line >= nlines) continue;
    const int k1 = half ? LineMap<M, NB>::slot(__ldg(g.fxr + c)) : c;
    typename A::V v[M];
    if (any) {
#pragma unroll
      for (int m = 0; m < M; ++m) v[m] = A::ld(S + Sm::at(k1, m, l));
      Dft<A, M, M>::run(v, tw);
    } else {  // no source on these lines
#pragma unroll
      for (int m = 0; m < M; ++m) v[m] = A::zero();
    }
    if constexpr (X) {  // row of the line, element K2 nk + c
      typename A::M *dst = out + field * g.astride + (int64_t)line * W + c;
#pragma unroll
      for (int k2 = 0; k2 < M; ++k2) A::st(dst + k2 * nk, A::norm(v[k2]));
    } else {  // row fy of the plane
      typename A::M *dst = out + field * g.cstride + (int64_t)blockIdx.y * (P * M) * W + line;
      int kp = LineMap<M, NB>::freq(k1 >> 1);
#pragma unroll
      for (int k2 = 0; k2 < M; ++k2) {
        A::st(dst + (int64_t)(2 * kp + (k1 & 1)) * W, A::norm(v[k2]));
        kp += LineMap<M, NB>::STEP;
        if (kp >= M * NB) kp -= M * NB;
      }
    }
  }
}

// The NB outputs of an (x line, m) through an output spec, ob[J] the output block of cell M J + m (-1: none): all
// addend and mask loads before the stores.
template <class R, int M, int NB>
LGF_D void line_store(const OutSpec<R> &o, const int (&ob)[NB], int brow, int crow, int m, int sh, R (&w)[NB]) {
  const int msk = (1 << sh) - 1;
  const int32_t *aux = o.aux;
  const R *add = o.add;
  const uint8_t *mask = o.mask;
  bool on[NB];
#pragma unroll
  for (int j = 0; j < NB; ++j) on[j] = ob[j] >= 0;
  if (add || mask) {
    int64_t a[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j)
      a[j] = on[j] ? ((int64_t)(aux ? __ldg(aux + brow + ((M * j + m) >> sh)) : ob[j]) << (3 * sh)) + crow + ((M * j + m) & msk) : 0;
    if (mask) {
      int mk[NB];
#pragma unroll
      for (int j = 0; j < NB; ++j) mk[j] = on[j] ? __ldg(mask + a[j]) & o.bits : 0;
#pragma unroll
      for (int j = 0; j < NB; ++j) on[j] = mk[j] != 0;
    }
    if (add) {
      R t[NB];
#pragma unroll
      for (int j = 0; j < NB; ++j) t[j] = on[j] ? add[a[j]] : RT<R>::zero();
#pragma unroll
      for (int j = 0; j < NB; ++j) w[j] = w[j] + t[j];
    }
  }
  const int64_t base = o.off + crow;
#pragma unroll
  for (int j = 0; j < NB; ++j)
    if (on[j]) store_field<R>(o.dst, base + ((int64_t)ob[j] << (3 * sh)) + ((M * j + m) & msk), o.dtype, w[j]);
}

// y inverse and x inverse (X, writing through the output specs); grids as k_line_fwd.  Fine: all sums renormalised, as what
// these two passes round is not smoothed by anything after them (two-level rings of 48 to 160 cells: error 4.9e-15 ->
// 4.3e-15 for 4 % of the time).
template <class R, int M, int NB, bool X, bool FINE>
__global__ void __launch_bounds__(LineTile<M, NB>::NT, LineTile<M, NB>::MB)
    k_line_inv(const typename Ar<R>::M *__restrict__ in, typename Ar<R>::M *__restrict__ out,
               const __grid_constant__ LineGeom g, const __grid_constant__ LineTw<R> tw,
               const typename Ar<R>::T *__restrict__ twl, const __grid_constant__ InvOuts<R> outs, double scale) {
  typedef Ar<R> A;
  typedef std::conditional_t<FINE, ArFine<R>, Ar<R>> I;
  constexpr int NT = LineTile<M, NB>::NT, TL = LineTile<M, NB>::TL, P = 2 * NB;
  typedef LineSmem<M, TL, X> Sm;
  extern __shared__ __align__(16) unsigned char line_smem_raw[];
  typename A::M *S = reinterpret_cast<typename A::M *>(line_smem_raw);
  const int field = blockIdx.z, W = line_width(g, field);
  const int line0 = blockIdx.x * TL;
  const int nlines = X ? g.n[1] * g.n[2] : W;
  if (line0 >= nlines) return;
  const bool half = X && field >= g.nc;
  const int nk = half ? NB + 1 : P;
  for (int t = threadIdx.x; t < TL * nk; t += NT) {
    const int c = X ? t % nk : t / TL, l = X ? t / nk : t % TL, line = line0 + l;
    if (line >= nlines) continue;
    const int k1 = half ? LineMap<M, NB>::slot(__ldg(g.fxr + c)) : c;
    typename A::V v[M];
    if constexpr (X) {
      const typename A::M *src = in + field * g.astride + (int64_t)line * W + c;
#pragma unroll
      for (int k2 = 0; k2 < M; ++k2) v[k2] = A::ld(src + k2 * nk);
    } else {
      const typename A::M *src = in + field * g.cstride + (int64_t)blockIdx.y * (P * M) * W + line;
      int kp = LineMap<M, NB>::freq(k1 >> 1);
#pragma unroll
      for (int k2 = 0; k2 < M; ++k2) {
        v[k2] = A::ld(src + (int64_t)(2 * kp + (k1 & 1)) * W);
        kp += LineMap<M, NB>::STEP;
        if (kp >= M * NB) kp -= M * NB;
      }
    }
    Dft<I, M, M>::run(v, tw);
#pragma unroll
    for (int m = 0; m < M; ++m) A::st(S + Sm::at(k1, m, l), A::norm(v[m]));
  }
  __syncthreads();
  const R sc = RT<R>::from(scale);
  for (int t = threadIdx.x; t < TL * M; t += NT) {
    const int m = X ? t % M : t / TL, l = X ? t / M : t % TL, line = line0 + l;
    if (line >= nlines) continue;
    if constexpr (X) {
      const int sh = g.shift, msk = (1 << sh) - 1;
      const int y = line % g.n[1], z = line / g.n[1];
      const int brow = ((z >> sh) * g.nb[1] + (y >> sh)) * g.nb[0];
      const int crow = (((z & msk) << sh) + (y & msk)) << sh;
      int ore[NB], oim[NB];  // the scatter indices of the line's blocks, loaded while the odd half runs
      line_merge<I, M, NB, TL, X>(
          S, m, l, half, tw, twl,
          [&]() {
            const int32_t *sr = outs.re[field].scatter, *si = half ? nullptr : outs.im[field].scatter;
#pragma unroll
            for (int j = 0; j < NB; ++j) ore[j] = sr ? __ldg(sr + brow + ((M * j + m) >> sh)) : -1;
#pragma unroll
            for (int j = 0; j < NB; ++j) oim[j] = si ? __ldg(si + brow + ((M * j + m) >> sh)) : -1;
          },
          [&](typename A::V (&v)[NB]) {
            R w[NB];
#pragma unroll
            for (int j = 0; j < NB; ++j) w[j] = A::re(v[j]) * sc;
            line_store<R, M, NB>(outs.re[field], ore, brow, crow, m, sh, w);
            if (!half) {
#pragma unroll
              for (int j = 0; j < NB; ++j) w[j] = -(A::im(v[j]) * sc);
              line_store<R, M, NB>(outs.im[field], oim, brow, crow, m, sh, w);
            }
          });
    } else {
      typename A::M *dst = out + field * g.astride + (int64_t)blockIdx.y * g.n[1] * W + line;
      line_merge<I, M, NB, TL, X>(S, m, l, false, tw, twl, []() {}, [&](typename A::V (&v)[NB]) {
#pragma unroll
        for (int j = 0; j < NB; ++j) A::st(dst + (int64_t)LineMap<M, NB>::cell(j, m) * W, A::norm(v[j]));
      });
    }
  }
}

// z: forward, kernel product, inverse; grid (ceil(L_y width / TL), 1, fields), lines the slots (fy, fx) of a plane.
// Gf is Ghat on 0 <= f_a <= L_a / 2 (it is even in every axis), x fastest.
// Ghat grows as 1 / f^2 towards f = 0: the few lines of low f_y and f_x carry most of a smooth result, and what they round
// in the inverse is seen as one smooth error all over the box.  Fine: a tile that holds a line with both frequencies within
// L / 32 renormalises its sums (three-level ring over 16 seeds, beside fine y and x passes: 6.5e-15, up to 10.9e-15 ->
// 5.4e-15, up to 7.4e-15, for 1.5 % of the time; in all tiles 5.2e-15 and 6.4e-15 for another 4 %).
template <class R, int M, int NB, bool FINE>
__global__ void __launch_bounds__(LineTile<M, NB>::NT, LineTile<M, NB>::MB)
    k_line_mid(typename Ar<R>::M *__restrict__ C, const R *__restrict__ Gf, const __grid_constant__ LineGeom g,
               const __grid_constant__ LineTw<R> tw, const typename Ar<R>::T *__restrict__ twl) {
  typedef Ar<R> A;
  constexpr int NT = LineTile<M, NB>::NT, TL = LineTile<M, NB>::TL, P = 2 * NB, L = P * M;
  typedef LineSmem<M, TL, false> Sm;
  extern __shared__ __align__(16) unsigned char line_smem_raw[];
  typename A::M *S = reinterpret_cast<typename A::M *>(line_smem_raw);
  const int field = blockIdx.z, W = line_width(g, field);
  const int Lx = g.P[0] * g.M[0], Ly = g.P[1] * g.M[1];
  const int nlines = Ly * W, line0 = blockIdx.x * TL;
  if (line0 >= nlines) return;
  typename A::M *Cf = C + field * g.cstride;
  // Ghat of the tile's lines, [fz <= L / 2][line], on its way to shared memory under the first step
  R *G = reinterpret_cast<R *>(S + P * Sm::SK);
  bool low = false;
  {
    const int l = threadIdx.x % TL, line = min(line0 + l, nlines - 1), fy = line / W, s = line - fy * W;
    const int fx = __ldg((field < g.nc ? g.fxc : g.fxr) + s);
    const R *src = Gf + (int64_t)min(fy, Ly - fy) * (Lx / 2 + 1) + min(fx, Lx - fx);
    const int64_t gz = (int64_t)(Ly / 2 + 1) * (Lx / 2 + 1);
    for (int fz = threadIdx.x / TL; fz <= L / 2; fz += NT / TL) line_copy_async(G + fz * TL + l, src + fz * gz);
    if constexpr (FINE) low = 32 * min(fy, Ly - fy) <= Ly && 32 * min(fx, Lx - fx) <= Lx;
  }
  for (int t = threadIdx.x; t < TL * M; t += NT) {
    const int m = t / TL, l = t % TL, line = line0 + l;
    if (line >= nlines) continue;
    const typename A::M *src = Cf + line;
    line_split<R, M, NB, TL, false>(S, m, l, tw, twl, [&](typename A::V (&v)[NB]) {
#pragma unroll
      for (int j = 0; j < NB; ++j) v[j] = A::ld(src + (int64_t)LineMap<M, NB>::cell(j, m) * nlines);
    });
  }
  line_copy_wait();
  if constexpr (FINE) low = __syncthreads_or(low);
  else __syncthreads();
  auto rest = [&](auto inverse) {
    typedef decltype(inverse) I;
    for (int t = threadIdx.x; t < TL * P; t += NT) {
      const int k1 = t / TL, l = t % TL;
      if (line0 + l >= nlines) continue;
      typename A::V v[M];
#pragma unroll
      for (int m = 0; m < M; ++m) v[m] = A::ld(S + Sm::at(k1, m, l));
      Dft<A, M, M>::run(v, tw);
      int kp = LineMap<M, NB>::freq(k1 >> 1);
#pragma unroll
      for (int k2 = 0; k2 < M; ++k2) {
        const int fz = 2 * kp + (k1 & 1);
        v[k2] = A::norm(A::scale_conj(A::norm(v[k2]), G[min(fz, L - fz) * TL + l]));
        kp += LineMap<M, NB>::STEP;
        if (kp >= M * NB) kp -= M * NB;
      }
      Dft<I, M, M>::run(v, tw);
#pragma unroll
      for (int m = 0; m < M; ++m) A::st(S + Sm::at(k1, m, l), A::norm(v[m]));
    }
    __syncthreads();
    for (int t = threadIdx.x; t < TL * M; t += NT) {
      const int m = t / TL, l = t % TL, line = line0 + l;
      if (line >= nlines) continue;
      typename A::M *dst = Cf + line;
      line_merge<I, M, NB, TL, false>(S, m, l, false, tw, twl, []() {}, [&](typename A::V (&v)[NB]) {
#pragma unroll
        for (int j = 0; j < NB; ++j) A::st(dst + (int64_t)LineMap<M, NB>::cell(j, m) * nlines, A::norm(v[j]));
      });
    }
  };
  if constexpr (FINE) {
    if (low) {
      rest(ArFine<R>());
      return;
    }
  }
  rest(Ar<R>());
}

}  // namespace lgf
