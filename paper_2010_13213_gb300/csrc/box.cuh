// box.cuh -- level boxes: input and output specs of a box convolution, the generator of its kernel spectrum, and the
// local transforms of the tensor-core path.
//
// A level box of nb = (nbx, nby, nbz) blocks of B^3 cells is embedded in a periodic lattice of
// P = 2 nb blocks per axis (Pc = P B cells), large enough that the circular convolution with the
// circularly laid out LGF equals the linear one on the box (Sec. 2.2 Eq. (eq:lgf_convolution)).  The CUDA-core
// evaluation transforms whole lines (lines.cuh).  The tensor-core path and the kernel spectrum work on blocks:
// writing a cell index n = B J + m (block J, local cell m) and a frequency K = K1 + P K2 (K1 in [0, P), K2 in
// [0, B)) per axis, the Pc-point DFT factors as ("four-step"):
//     Y[K1][m]  = sum_J x[J][m] W_P^{J.K1}                  block-index DFT   (k_bdft_tc / k_bdft_dense, per axis)
//     Y'        = Y W_Pc^{m.K1}                              twiddle          (k_box_mid)
//     X[K1][K2] = sum_m Y'[K1][m] W_B^{m.K2}                 local B^3 FFT     (k_box_mid)
// The convolution multiplies X by the (real, since G is even) spectrum Ghat[K1][K2] and runs the three
// steps backwards; the inverse block-index DFT is evaluated only on the box's blocks.  Inputs are
// complex: two real fields ride as real and imaginary part (G is real).
#pragma once
#include "common.cuh"

#define BOX_NB_MAX 16

// Layout of a box array: [bz][by][bx][B^3] with full extents (Px, Py, Pz) blocks.
struct BoxGeom {
  int nb[3];    // box blocks per axis
  int P[3];     // 2 nb
  int64_t bs[3];  // block strides (in blocks) of the full P-array: 1, Px, Px*Py
  int nc;       // fields [0, nc) of a launch are complex (K1x < Px); the others are real fields kept on
                // the Hermitian half K1x <= Px/2
};
// Per-axis members picked by selects: indexing a kernel parameter's array with a runtime axis would copy
// the whole struct to local memory.
LGF_HD int geo_nb(const BoxGeom &g, int a) { return a == 0 ? g.nb[0] : (a == 1 ? g.nb[1] : g.nb[2]); }
LGF_HD int geo_P(const BoxGeom &g, int a) { return a == 0 ? g.P[0] : (a == 1 ? g.P[1] : g.P[2]); }
LGF_HD int64_t geo_bs(const BoxGeom &g, int a) { return a == 0 ? g.bs[0] : (a == 1 ? g.bs[1] : g.bs[2]); }
// Block frequencies K1x a field keeps, and the most any field of the launch keeps.
LGF_HD int box_pxu(const BoxGeom &g, int field) { return field < g.nc ? g.P[0] : g.P[0] / 2 + 1; }
LGF_HD int box_pxmax(const BoxGeom &g) { return g.nc > 0 ? g.P[0] : g.P[0] / 2 + 1; }

// Source of the first forward pass: box block -> buffer block (gather, -1 = absent), a field
// (dtype per load_field, the component already applied to the pointer) and an optional cell mask.
// Each spec adds into the real (part 0), the imaginary (part 1) or both parts (part 2) of the complex input.
struct InSpec {
  const int32_t *gather;
  const void *src;
  const uint8_t *mask;
  int dtype, bits, part;
};
// Destination of the last inverse pass for the real (re) or imaginary (im) part: box block ->
// output block (scatter, -1 = skip), output field (component applied) with element offset, the
// internal-R addend and mask indexed by aux (or by the output block when aux is null).
template <class R>
struct OutSpec {
  const int32_t *scatter;
  const int32_t *aux;
  void *dst;
  const R *add;
  const uint8_t *mask;
  int64_t off;
  int dtype, bits;
};

#define BOX_MAXF 4  // complex fields per launch

struct InSpec3 {  // the input specs of one complex field
  InSpec s[3];
};

struct FwdSpecs {   // per field: up to three input specs (first forward pass only)
  InSpec s[BOX_MAXF][3];
  int n[BOX_MAXF];
};

template <class R>
struct InvOuts {  // per field: destinations of the real and imaginary parts (last inverse pass)
  OutSpec<R> re[BOX_MAXF], im[BOX_MAXF];
};

template <class R>
LGF_D void box_store(const OutSpec<R> &o, int bidx, int m, int B3, R v) {
  if (!o.scatter) return;
  const int ob = o.scatter[bidx];
  if (ob < 0) return;
  const int64_t a = (int64_t)(o.aux ? o.aux[bidx] : ob) * B3 + m;
  if (o.add) v = v + o.add[a];
  if (o.mask && !(o.mask[a] & o.bits)) return;
  store_field<R>(o.dst, o.off + (int64_t)ob * B3 + m, o.dtype, v);
}

// ------------------------------------------------------------------ dense block-index DFT (kernel spectra, FP64)
// out[.. k ..][m] = sum_{j < P} W_P^{j k} in[.. j ..][m] over all P blocks; the first pass reads the
// circularly laid out unit-lattice LGF: cell n (per axis, 0 <= n < Pc) holds G(d), d = n for
// n <= Pc/2 and n - Pc above.
template <int B>
__global__ void __launch_bounds__(256) k_bdft_dense(const cx<double> *__restrict__ in, cx<double> *__restrict__ out,
                                                    BoxGeom g, int ax, const cx<double> *__restrict__ wP,
                                                    const double *__restrict__ Gd, int K) {
  constexpr int B3 = B * B * B;
  const int P = geo_P(g, ax);
  const int a1 = ax == 0 ? 1 : 0, a2 = ax == 2 ? 1 : 2;
  const int e1 = geo_P(g, a1);
  const int64_t line = blockIdx.y;
  const int l1 = (int)(line % e1), l2 = (int)(line / e1);
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= B3) return;
  int coord[3];
  coord[a1] = l1;
  coord[a2] = l2;
  const int mloc[3] = {m % B, (m / B) % B, m / (B * B)};
  auto value = [&](int j) -> cx<double> {
    coord[ax] = j;
    if (Gd) {
      int d[3];
      for (int a = 0; a < 3; ++a) {
        const int Pc = geo_P(g, a) * B, n = coord[a] * B + mloc[a];
        d[a] = n <= Pc / 2 ? n : Pc - n;
      }
      return cx<double>{Gd[((int64_t)d[2] * K + d[1]) * K + d[0]], 0.0};
    }
    return in[((int64_t)coord[0] * g.bs[0] + coord[1] * g.bs[1] + coord[2] * g.bs[2]) * B3 + m];
  };
  for (int k = 0; k < P; ++k) {
    cx<double> acc{0.0, 0.0};
    for (int j = 0; j < P; ++j) acc = acc + value(j) * wP[(j * k) % P];
    coord[ax] = k;
    out[((int64_t)coord[0] * g.bs[0] + coord[1] * g.bs[1] + coord[2] * g.bs[2]) * B3 + m] = acc;
  }
}

// ------------------------------------------------------------------ fused twiddle + local FFT + kernel
// One CTA per (K1 block, field): Y'[m] = Y[m] W_Pc^{m.K1}; X = FFT_B^3(Y'); X *= Ghat; back.  Six
// line-FFT steps over the B^2 lines (l0, l1) of each axis, one thread per line (two for FP32, see
// MidSplit):
//   0  z lines (x, y): global Y, twiddle, FFT_z              -> shared
//   1  y lines (x, z): FFT_y                                 -> shared
//   2  x lines (y, z): FFT_x, X Ghat, conjugate              (registers)
//   3  x lines      : FFT_x                                  -> shared
//   4  y lines      : FFT_y                                  -> shared
//   5  z lines      : FFT_z, conjugate, conjugate twiddle    -> global Y
// (the inverse is conj(FFT(conj(.))), so one FFT body serves every step: small code, no
// instruction-cache stalls).  Four barriers, one shared store and load per cell and step.  Ghat is stored
// per block as [x][z][y] so the x lines of step 2 read it coalesced.  Shared memory: B^3 complex with
// rows padded to B + 1 (every line direction conflict-free).  Without MULTIPLY (kernel-spectrum
// generation) the real part of step 2 goes to `kout` in the same [x][z][y] order.  The per-cell twiddle
// is one load from a table of W_L^n, L = lcm of the three lattice periods, at an integer exponent.
template <int B>
struct MidGeom {
  static constexpr int RS = B + 1;          // padded row
  static constexpr int N = B * B * RS;      // padded elements
};

// Exchange with the lane 16 apart in the warp (the other half of the same line).
LGF_D double shfl16(double v) { return __shfl_xor_sync(0xffffffffu, v, 16); }
LGF_D float shfl16(float v) { return __shfl_xor_sync(0xffffffffu, v, 16); }
LGF_D df shfl16(df v) { return df{__shfl_xor_sync(0xffffffffu, v.hi, 16), __shfl_xor_sync(0xffffffffu, v.lo, 16)}; }
template <class R>
LGF_D cx<R> shfl16(cx<R> v) { return cx<R>{shfl16(v.re), shfl16(v.im)}; }

// Line FFT split over two threads: half h holds the points 2r + h (r < H = B/2) and runs the H-point
// FFT of its half (E: even points, O: odd points); the last radix-2 stage X_k = E_k + W_B^k O_k,
// X_{k+H} = E_k - W_B^k O_k is shared out by k, half h taking k in [hQ, hQ + Q), Q = B/4, after one
// exchange of Q values.  Output slot j of half h then holds X at mid_out_index(B, h, j).
LGF_HD constexpr int mid_out_index(int B, int h, int j) { return h * (B / 4) + j % (B / 4) + (B / 2) * (j / (B / 4)); }

template <class R, int B>
LGF_D void fft_split(cx<R> (&u)[B / 2], int h, const Tw64<R> &tw) {
  constexpr int Q = B / 4;
  fft_reg<R, B / 2, false, false>(u, tw);
#pragma unroll
  for (int r = 0; r < Q; ++r) {
    const cx<R> recv = shfl16(h ? u[r] : u[Q + r]);  // half 0 sends E_{Q+r}, half 1 sends O_r
    const cx<R> E = h ? recv : u[r], O = h ? u[Q + r] : recv;
    cx<R> t;
    if (r == 0) {  // k = 0 (W = 1) or k = B/4 (W = -i, an exact swap)
      t = h ? cx<R>{O.im, -O.re} : O;
    } else {
      const cx<R> w0 = twiddle<R, 64, false>(tw, r * (64 / B)), w1 = twiddle<R, 64, false>(tw, (Q + r) * (64 / B));
      t = cmul(O, h ? w1 : w0);
    }
    u[r] = cadd(E, t);
    u[Q + r] = csub(E, t);
  }
}

// Source of slot r (point 2r + h) of half h when the output of fft_split feeds another split FFT of the
// same line: >= 0, the half's own slot; < 0, -(s + 1) for the s-th value received from the other half,
// which sends its slots 2s + h.
LGF_HD constexpr int mid_regroup_src(int B, int h, int r) {
  const int m = 2 * r + h, H = B / 2, Q = B / 4;
  if ((m % H) / Q == h) return (m % H) % Q + Q * (m / H);
  int src = 0;
  for (int s = 0; s < H / 2; ++s)
    if (mid_out_index(B, 1 - h, 2 * s + h) == m) src = -(s + 1);
  return src;
}

template <class R, int B>
LGF_D void mid_regroup(cx<R> (&u)[B / 2], int h) {
  constexpr int H = B / 2;
  cx<R> recv[H / 2], nu[H];
#pragma unroll
  for (int s = 0; s < H / 2; ++s) recv[s] = shfl16(h ? u[2 * s] : u[2 * s + 1]);
#pragma unroll
  for (int r = 0; r < H; ++r) {
    const int c0 = mid_regroup_src(B, 0, r), c1 = mid_regroup_src(B, 1, r);
    const cx<R> v0 = c0 >= 0 ? u[c0 >= 0 ? c0 : 0] : recv[c0 < 0 ? -c0 - 1 : 0];
    const cx<R> v1 = c1 >= 0 ? u[c1 >= 0 ? c1 : 0] : recv[c1 < 0 ? -c1 - 1 : 0];
    nu[r] = h ? v1 : v0;
  }
#pragma unroll
  for (int r = 0; r < H; ++r) u[r] = nu[r];
}

// Lines per thread of k_box_mid: FP32 splits each line over two threads (half the registers per thread,
// twice the resident warps, one exchange per FFT); double-float and FP64 keep a whole line per thread,
// where the exchanges (two or four words per complex value) and the register limit of the doubled block
// cost more than the occupancy gains.
template <class R>
struct MidSplit {
  static constexpr bool value = false;
};
template <>
struct MidSplit<float> {
  static constexpr bool value = true;
};
template <class R, int B>
constexpr int mid_threads() { return (MidSplit<R>::value ? 2 : 1) * B * B; }

template <class R, int B, bool MULTIPLY>
__global__ void __launch_bounds__(mid_threads<R, B>(), 512 / (B * B)) k_box_mid(
    cx<R> *__restrict__ Y, int64_t fstride, const R *__restrict__ Gh, BoxGeom g, const cx<R> *__restrict__ twl,
    int L, int3 twf, Tw64<R> tw, R *__restrict__ kout) {
  constexpr bool SPLIT = MidSplit<R>::value;
  constexpr int B2 = B * B, B3 = B * B * B, RS = B + 1, NV = SPLIT ? B / 2 : B, Q = B / 4;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<R> *S = reinterpret_cast<cx<R> *>(smem_raw);
  // K1 block: blockIdx.x runs over K1x < the launch's widest range; a real field stops at Px/2
  const int pxm = box_pxmax(g);
  const int k1x = (int)(blockIdx.x % pxm), k1y = (int)((blockIdx.x / pxm) % g.P[1]);
  const int k1z = (int)(blockIdx.x / ((unsigned)pxm * g.P[1]));
  if (k1x >= box_pxu(g, blockIdx.y)) return;
  const int64_t kb = k1x + (int64_t)g.P[0] * (k1y + (int64_t)g.P[1] * k1z);  // linear in the full P array
  cx<R> *Yb = Y + blockIdx.y * fstride + kb * B3;  // field blockIdx.y
  // line t = (l0, l1).  SPLIT: lanes 0-15 of warp w hold the even points of the lines 16w .. 16w + 15,
  // lanes 16-31 the odd points of the same lines (each quarter-warp keeps the one-line-per-lane pattern)
  const int h = SPLIT ? (threadIdx.x >> 4) & 1 : 0;
  const int t = SPLIT ? (threadIdx.x >> 5) * 16 + (threadIdx.x & 15) : threadIdx.x, l0 = t % B, l1 = t / B;
  // point of the line in input slot r / output slot j of this thread
  auto in_idx = [h](int r) { return SPLIT ? 2 * r + h : r; };
  auto out_idx = [h](int j) { return SPLIT ? mid_out_index(B, h, j) : j; };
  // twiddle W_Pc^{m.K1} of the cell (x, y, z) = (l0, l1, i) of this z line: W_L^{e0 + i ez mod L} with
  // L = lcm(Pcx, Pcy, Pcz) (m_a K1_a < Pc_a, so each term below is below L: 32-bit)
  // (kept in shared memory between the first and the last step: no registers held across the FFTs)
  __shared__ int s_e0[B2];
  __shared__ int s_ez;
  if (h == 0) s_e0[t] = (l0 * k1x * twf.x + l1 * k1y * twf.y) % L;
  if (threadIdx.x == 0) s_ez = (k1z * twf.z) % L;
  __syncthreads();
  cx<R> v[NV];
  const int nstep = MULTIPLY ? 6 : 3;
  for (int step = 0; step < nstep; ++step) {
    const int ax = step < 3 ? 2 - step : step - 3;
    int base, stride;
    if (ax == 0) base = (l1 * B + l0) * RS, stride = 1;             // x lines: (y, z) = (l0, l1)
    else if (ax == 1) base = l1 * B * RS + l0, stride = RS;         // y lines: (x, z) = (l0, l1)
    else base = l1 * RS + l0, stride = B * RS;                      // z lines: (x, y) = (l0, l1)
    if (step == 0) {
      const int ez = s_ez, dez = SPLIT ? (2 * ez) % L : ez;
      int e = (s_e0[t] + h * ez) % L;
#pragma unroll
      for (int r = 0; r < NV; ++r) {
        const int i = in_idx(r);
        v[r] = cmul(ld_stream(Yb + (i * B + l1) * B + l0), twl[e]);
        e += dez;
        if (e >= L) e -= L;
      }
    } else if (step == 3) {
      if constexpr (SPLIT) mid_regroup<R, B>(v, h);  // the same x lines, in registers
    } else {
#pragma unroll
      for (int r = 0; r < NV; ++r) v[r] = S[base + in_idx(r) * stride];
    }
    // no renormalisation between the line FFTs: the next step's butterflies add lazily, and the kernel
    // product and the final twiddle product renormalise
    if constexpr (SPLIT) fft_split<R, B>(v, h, tw);
    else fft_reg<R, B, false, false>(v, tw);
    if (step == 2) {
      if (!MULTIPLY) {
#pragma unroll
        for (int j = 0; j < NV; ++j) kout[kb * B3 + out_idx(j) * B2 + t] = v[j].re;
      } else {
#pragma unroll
        for (int j = 0; j < NV; ++j) {
          const R gk = ld_stream(Gh + kb * B3 + out_idx(j) * B2 + t);  // read once per solve
          v[j] = cx<R>{v[j].re * gk, -(v[j].im * gk)};
        }
      }
      continue;
    }
    if (step == 5) {
      const int ez = s_ez, e0 = s_e0[t];
      int e = 0;
#pragma unroll
      for (int j = 0; j < NV; ++j) {
        const int i = out_idx(j);
        if (j == 0 || (SPLIT && j == Q)) {
          e = (e0 + i * ez) % L;
        } else {
          e += ez;
          if (e >= L) e -= L;
        }
        Yb[(i * B + l1) * B + l0] = conj(cmul(v[j], twl[e]));
      }
    } else {
#pragma unroll
      for (int j = 0; j < NV; ++j) S[base + out_idx(j) * stride] = v[j];
      __syncthreads();
    }
  }
}
