// box_spec.cu -- kernel spectra and transform tables of the block-index FFT mode, one set per level-box shape, cached
// in the table.
//
// For a box of nb blocks per axis (periodic lattice Pc = 2 nb B), Ghat is the Pc^3 DFT of the circularly laid out
// unit-lattice LGF (cell n holds G(d), d = n for n <= Pc/2, n - Pc above).  G is real and even in every axis, and so
// is Ghat: it is kept on 0 <= f_a <= Pc_a / 2, an eighth of the padded lattice.  Computed once in FP64 in block order
// (dense block-index DFTs + the local FFT of k_box_mid), then folded, rounded to FP32 and split into double-float.
#include <math.h>
#include <string.h>

#include <numeric>
#include <vector>

#include "box.cuh"
#include "internal.h"

namespace lgf {

// Ghat on the folded lattice [f_z][f_y][f_x], 0 <= f_a <= Pc_a / 2, from block order (k_box_mid: [K1 block][x][z][y],
// f = K1 + P K2 per axis); n = values.
__global__ void k_spec_fold(const double *__restrict__ g, int B, BoxGeom geo, int64_t n, double mant8, double *__restrict__ g64,
                            float *__restrict__ g32, df *__restrict__ gdf) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int nx = geo.P[0] * B / 2 + 1, ny = geo.P[1] * B / 2 + 1;
  const int fx = (int)(i % nx), fy = (int)((i / nx) % ny), fz = (int)(i / ((int64_t)nx * ny));
  const int64_t kb = fx % geo.P[0] + (int64_t)geo.P[0] * (fy % geo.P[1] + (int64_t)geo.P[1] * (fz % geo.P[2]));
  const double v = g[((kb * B + fx / geo.P[0]) * B + fz / geo.P[2]) * B + fy / geo.P[1]];
  g64[i] = v;
  g32[i] = (float)v;
  // with the 1 / (8 cells) of the inverse transform up to a power of two: the last pass then scales by h^2 and that
  // power, which rounds nothing for an h that is one (error of the two rings 5.8e-15 -> 5.0e-15).  The power stays out, as
  // it would take low parts of small fields below the floats' range.
  gdf[i] = df_make(v * mant8);
}

// Block order from the folded spectrum (k_box_mid of the block-index paths); n = P^3 B^3 values.
__global__ void k_spec_unfold(const double *__restrict__ g, int B, BoxGeom geo, int64_t n, float *__restrict__ g32,
                              df *__restrict__ gdf) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int y = (int)(i % B), z = (int)((i / B) % B), x = (int)((i / (B * B)) % B);
  const int64_t kb = i / ((int64_t)B * B * B);
  int f[3] = {(int)(kb % geo.P[0]) + geo.P[0] * x, (int)((kb / geo.P[0]) % geo.P[1]) + geo.P[1] * y,
              (int)(kb / ((int64_t)geo.P[0] * geo.P[1])) + geo.P[2] * z};
  for (int a = 0; a < 3; ++a) f[a] = min(f[a], geo.P[a] * B - f[a]);
  const int64_t nx = geo.P[0] * B / 2 + 1, ny = geo.P[1] * B / 2 + 1;
  const double v = g[((int64_t)f[2] * ny + f[1]) * nx + f[0]];
  g32[i] = (float)v;
  gdf[i] = df_make(v);
}

__global__ void k_tw_convert(const double *__restrict__ c, const double *__restrict__ s, int n,
                             cx<double> *__restrict__ t64, cx<float> *__restrict__ t32, cx<df> *__restrict__ tdf) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  t64[i] = cx<double>{c[i], -s[i]};
  t32[i] = cx<float>{(float)c[i], -(float)s[i]};
  tdf[i] = cx<df>{df_make(c[i]), df_make(-s[i])};
}

// e^{-2 pi i n / N}, n < N, from long-double cos/sin folded into the first octant.
void twiddles_host(int N, std::vector<double> &c, std::vector<double> &s) {
  const long double pi = 3.141592653589793238462643383279502884L;
  c.resize(N);
  s.resize(N);
  for (int n = 0; n < N; ++n) {
    // reduce 2 pi n / N to [0, pi/4] with exact symmetries (N multiple of 4 here)
    long double a = 2.0L * pi * (long double)n / (long double)N;
    c[n] = (double)cosl(a);
    s[n] = (double)sinl(a);
    if (4 * n == N) c[n] = 0.0, s[n] = 1.0;
    if (2 * n == N) c[n] = -1.0, s[n] = 0.0;
    if (4 * n == 3 * N) c[n] = 0.0, s[n] = -1.0;
    if (n == 0) c[n] = 1.0, s[n] = 0.0;
  }
}

// Coefficient digits of one block-index DFT pass (box_tc.cuh): C_jo = W_P^{-+jo} (dir -1 forward, +1
// inverse); `realw`: the Hermitian-folded real inverse, weights 1 (j = 0, 2j = P) or 2 and real output
// only.  M^T[n = 2o + p][k = 2j + q] / sigma = 2^{-7} sum_t c_t 2^{-8t} with integer digits |c_t| <= 128.
static void tc_matrix(int P, int nin, int nout, int dir, bool realw, const std::vector<double> &c,
                      const std::vector<double> &s, std::vector<uint16_t> &buf, TcMat &M) {
  const int K = 2 * nin, N = 2 * nout;
  M.nin = nin;
  M.nout = nout;
  M.Kp = (K + 15) / 16 * 16;
  M.Np = (N + 15) / 16 * 16;
  M.sigma = realw ? 2.0f : 1.0f;
  M.plane16 = M.Np * M.Kp * 2 / 16;
  const size_t off = buf.size(), plane = (size_t)M.Np * M.Kp;
  buf.resize(off + TC_SMAX * plane, 0);
  for (int n = 0; n < N; ++n)
    for (int k = 0; k < K; ++k) {
      const int j = k / 2, q = k % 2, o = n / 2, p = n % 2;
      const int idx = (int)(((int64_t)j * o) % P);
      const double w = realw ? ((j == 0 || 2 * j == P) ? 1.0 : 2.0) : 1.0;
      const double cr = w * c[idx], ci = w * (dir < 0 ? -s[idx] : s[idx]);
      double v;
      if (p == 0) v = q == 0 ? cr : -ci;
      else v = realw ? 0.0 : (q == 0 ? ci : cr);
      double r = v / (double)M.sigma * 128.0;
      const size_t pos = ((size_t)(n / 8) * (M.Kp / 8) + k / 8) * 64 + (n % 8) * 8 + (k % 8);
      for (int t = 0; t < TC_SMAX; ++t) {
        const double d = nearbyint(r);
        r = (r - d) * 256.0;
        const float fd = (float)d;  // |d| <= 128: exact in bf16 (the top half of the float)
        uint32_t bits;
        memcpy(&bits, &fd, 4);
        buf[off + t * plane + pos] = (uint16_t)(bits >> 16);
      }
    }
  M.d = reinterpret_cast<const uint16_t *>(off);  // offset for now; rebased after the upload
}

static int tc_matrices(BoxSpec *S, const BoxGeom &g, cudaStream_t st) {
  std::vector<uint16_t> buf;
  for (int a = 0; a < 3; ++a) {
    std::vector<double> c, s;
    twiddles_host(g.P[a], c, s);
    tc_matrix(g.P[a], g.nb[a], g.P[a], -1, false, c, s, buf, S->tcm[a][0]);
    tc_matrix(g.P[a], g.P[a], g.nb[a], +1, false, c, s, buf, S->tcm[a][1]);
    if (a == 0) tc_matrix(g.P[a], g.P[a] / 2 + 1, g.nb[a], +1, true, c, s, buf, S->tcm[a][2]);
  }
  if (cudaMalloc(&S->tcw, buf.size() * 2) != cudaSuccess) return set_error(LGF_E_OOM, "tensor-core coefficients");
  cudaMemcpyAsync(S->tcw, buf.data(), buf.size() * 2, cudaMemcpyHostToDevice, st);
  for (int a = 0; a < 3; ++a)
    for (int v = 0; v < 3; ++v)
      if (S->tcm[a][v].Np) S->tcm[a][v].d = S->tcw + reinterpret_cast<size_t>(S->tcm[a][v].d);
  S->bytes += buf.size() * 2;
  cudaError_t e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? LGF_OK : set_error(LGF_E_CUDA, "coefficient upload: %s", cudaGetErrorString(e));
}

BoxSpec::~BoxSpec() {
  cudaFree(tcw);
  cudaFree(gf64);
  cudaFree(gf32);
  cudaFree(gfdf);
  cudaFree(ltl64);
  cudaFree(ltl32);
  cudaFree(ltldf);
  cudaFree(fx);
  cudaFree(g32);
  cudaFree(gdf);
  cudaFree(twl64);
  cudaFree(twl32);
  cudaFree(twldf);
}

static BoxGeom spec_geom(const BoxSpec *S) {
  BoxGeom g;
  for (int a = 0; a < 3; ++a) {
    g.nb[a] = S->nb[a];
    g.P[a] = 2 * S->nb[a];
  }
  g.bs[0] = 1;
  g.bs[1] = g.P[0];
  g.bs[2] = (int64_t)g.P[0] * g.P[1];
  g.nc = 1;
  return g;
}

// The parameter tables of one axis's line transforms, P = 2 NB.
template <class R>
static void line_tables(int P, LineTw<R> &t) {
  memset(&t, 0, sizeof t);
  std::vector<double> c, s;
  twiddles_host(P, c, s);
  for (int i = 0; i < P && i < LINE_P_MAX; ++i) make_T(c[i], -s[i], t.p[i]);
  twiddles_host(16, c, s);
  const int at[4] = {1, 2, 3, 9};
  for (int i = 0; i < 4; ++i) make_T(c[at[i]], -s[at[i]], t.w16[i]);
  twiddles_host(3, c, s);
  make_T(c[1], -s[1], t.c3);
}

// W_{L_a}^n of the three axes, one array per arithmetic.
template <class R>
static int line_rows(const BoxSpec *S, int B, typename Ar<R>::T **dst, cudaStream_t st) {
  std::vector<typename Ar<R>::T> all;
  for (int a = 0; a < 3; ++a) {
    const int L = 2 * S->nb[a] * B;
    std::vector<double> c, s;
    twiddles_host(L, c, s);
    for (int i = 0; i < L; ++i) {
      typename Ar<R>::T t;
      make_T(c[i], -s[i], t);
      all.push_back(t);
    }
  }
  if (cudaMalloc(dst, all.size() * sizeof(all[0])) != cudaSuccess) {
    cudaGetLastError();
    return set_error(LGF_E_OOM, "line twiddles");
  }
  cudaMemcpyAsync(*dst, all.data(), all.size() * sizeof(all[0]), cudaMemcpyHostToDevice, st);
  return cudaStreamSynchronize(st) == cudaSuccess ? LGF_OK : set_error(LGF_E_CUDA, "line twiddle upload");
}

// x frequency K of every row element [K2][kept K1] of the line transforms (lines.cuh), complex then real fields: slot
// K1 = 2 (k3 N2 + k2) + h holds K = 2 K' + h with K' = k3 mod NO, K' = k2 + N2 K2 mod M N2; a real field keeps the
// slots that are not above their mirror, in order.
static int line_freqs(BoxSpec *S, int B, cudaStream_t st) {
  const int nb = S->nb[0], M = line_M(B, nb), NB = line_NB(B, nb);
  const int N2 = NB & -NB, NO = NB / N2, Q2 = M * N2, n = M * NB;
  auto freq = [&](int k1, int k2big) {  // by search: tables of at most 512 entries
    const int q = k1 / 2, k3 = q / N2, kk = q % N2 + N2 * k2big;
    for (int k = 0; k < n; ++k)
      if (k % NO == k3 % NO && k % Q2 == kk % Q2) return 2 * k + k1 % 2;
    return 0;
  };
  std::vector<int32_t> all;
  for (int real = 0; real < 2; ++real) {
    std::vector<int> keep;
    for (int k1 = 0; k1 < 2 * NB; ++k1) {
      const int q = k1 / 2, h = k1 % 2, k3 = q / N2, k2 = q % N2;
      const int mir = h ? (NO - 1 - k3) * N2 + N2 - 1 - k2 : (NO - k3) % NO * N2 + (N2 - k2) % N2;
      if (!real || q <= mir) keep.push_back(k1);
    }
    for (int k2 = 0; k2 < M; ++k2)
      for (int k1 : keep) all.push_back(freq(k1, k2));
  }
  if (cudaMalloc(&S->fx, all.size() * sizeof(int32_t)) != cudaSuccess) {
    cudaGetLastError();
    return set_error(LGF_E_OOM, "line frequencies");
  }
  cudaMemcpyAsync(S->fx, all.data(), all.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st);
  return cudaStreamSynchronize(st) == cudaSuccess ? LGF_OK : set_error(LGF_E_CUDA, "line frequency upload");
}

// Four-step twiddles W_L^n, L = lcm of the three lattice periods Pc = P B (k_box_mid).
static int block_twiddles(BoxSpec *S, const BoxGeom &g, int B, cudaStream_t st) {
  const int Pc[3] = {g.P[0] * B, g.P[1] * B, g.P[2] * B};
  const int L = std::lcm(std::lcm(Pc[0], Pc[1]), Pc[2]);
  S->twL = L;
  for (int a = 0; a < 3; ++a) S->twf[a] = L / Pc[a];
  std::vector<double> c, s;
  twiddles_host(L, c, s);
  double *dc = nullptr, *ds = nullptr;
  const bool ok = cudaMalloc(&dc, sizeof(double) * L) == cudaSuccess && cudaMalloc(&ds, sizeof(double) * L) == cudaSuccess &&
                  cudaMalloc(&S->twl64, sizeof(cx<double>) * L) == cudaSuccess &&
                  cudaMalloc(&S->twl32, sizeof(cx<float>) * L) == cudaSuccess &&
                  cudaMalloc(&S->twldf, sizeof(cx<df>) * L) == cudaSuccess;
  if (ok) {
    cudaMemcpyAsync(dc, c.data(), sizeof(double) * L, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(ds, s.data(), sizeof(double) * L, cudaMemcpyHostToDevice, st);
    k_tw_convert<<<(L + 127) / 128, 128, 0, st>>>(dc, ds, L, S->twl64, S->twl32, S->twldf);
    cudaStreamSynchronize(st);
  }
  cudaFree(dc);
  cudaFree(ds);
  S->bytes += (size_t)L * (16 + 8 + 16);
  if (ok) return LGF_OK;
  cudaGetLastError();
  return set_error(LGF_E_OOM, "box spectrum: twiddles");
}

// The block-index paths' tables, from the folded spectrum.
static int gen_blocks(BoxSpec *S, int B, cudaStream_t st) {
  const BoxGeom g = spec_geom(S);
  const int64_t n = (int64_t)g.P[0] * g.P[1] * g.P[2] * B * B * B;
  if (cudaMalloc(&S->g32, sizeof(float) * n) != cudaSuccess || cudaMalloc(&S->gdf, sizeof(df) * n) != cudaSuccess) {
    cudaGetLastError();
    return set_error(LGF_E_OOM, "block-order spectrum");
  }
  S->bytes += (size_t)n * 12;
  k_spec_unfold<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(S->gf64, B, g, n, S->g32, S->gdf);
  return tc_matrices(S, g, st);  // synchronises
}

template <int B>
static int gen_spectrum(lgf_table *t, BoxSpec *S, cudaStream_t st) {
  constexpr int B3 = B * B * B;
  const BoxGeom g = spec_geom(S);
  const int64_t nblk = (int64_t)g.P[0] * g.P[1] * g.P[2];
  const int64_t n = nblk * B3;
  int64_t nf = 1;
  for (int a = 0; a < 3; ++a) nf *= g.P[a] * B / 2 + 1;
  cx<double> *Y0 = nullptr, *Y1 = nullptr, *wP[3] = {nullptr, nullptr, nullptr};
  auto release = [&]() {
    cudaFree(Y0);
    cudaFree(Y1);
    for (int a = 0; a < 3; ++a) cudaFree(wP[a]);
  };
  auto fail = [&](int code, const char *what) {
    release();
    cudaGetLastError();
    return set_error(code, "box spectrum: %s", what);
  };
  if (cudaMalloc(&Y0, sizeof(cx<double>) * n) || cudaMalloc(&Y1, sizeof(cx<double>) * n)) return fail(LGF_E_OOM, "scratch");
  if (cudaMalloc(&S->gf64, sizeof(double) * nf) || cudaMalloc(&S->gf32, sizeof(float) * nf) ||
      cudaMalloc(&S->gfdf, sizeof(df) * nf))
    return fail(LGF_E_OOM, "spectrum");
  S->bytes = nf * (8 + 4 + 8);
  for (int a = 0; a < 3; ++a) {  // W_P of the dense block DFTs
    std::vector<double> c, s;
    twiddles_host(g.P[a], c, s);
    std::vector<cx<double>> w(g.P[a]);
    for (int i = 0; i < g.P[a]; ++i) w[i] = cx<double>{c[i], -s[i]};
    if (cudaMalloc(&wP[a], sizeof(cx<double>) * g.P[a])) return fail(LGF_E_OOM, "tables");
    cudaMemcpyAsync(wP[a], w.data(), sizeof(cx<double>) * g.P[a], cudaMemcpyHostToDevice, st);
    for (int i = 0; i < g.P[a] && i < 32; ++i) S->bw32[a][i] = cx<float>{(float)c[i], -(float)s[i]};
    const int P = 2 * line_NB(B, g.nb[a]);  // 2 NB of the line transforms
    line_tables<double>(P, S->lt64[a]);
    line_tables<float>(P, S->lt32[a]);
    line_tables<df>(P, S->ltdf[a]);
    S->ltl_off[a] = a == 0 ? 0 : S->ltl_off[a - 1] + g.P[a - 1] * B;
  }
  int rc;
  if ((rc = line_rows<double>(S, B, &S->ltl64, st)) || (rc = line_rows<float>(S, B, &S->ltl32, st)) ||
      (rc = line_rows<df>(S, B, &S->ltldf, st)) || (rc = line_freqs(S, B, st)) ||
      (rc = block_twiddles(S, g, B, st))) {
    release();
    return rc;
  }
  // dense block-index DFTs of the embedded LGF: x (from G), y, z
  const dim3 blk(256);
  const unsigned gx = (B3 + 255) / 256;
  k_bdft_dense<B><<<dim3(gx, g.P[1] * g.P[2]), blk, 0, st>>>(nullptr, Y0, g, 0, wP[0], t->Gd, t->N + 1);
  k_bdft_dense<B><<<dim3(gx, g.P[0] * g.P[2]), blk, 0, st>>>(Y0, Y1, g, 1, wP[1], nullptr, 0);
  k_bdft_dense<B><<<dim3(gx, g.P[0] * g.P[1]), blk, 0, st>>>(Y1, Y0, g, 2, wP[2], nullptr, 0);
  const size_t sm = sizeof(cx<double>) * (size_t)B * B * (B + 1);
  double *block_order = reinterpret_cast<double *>(Y1);  // n values; Y1 is dead after the z pass
  cudaFuncSetAttribute(k_box_mid<double, B, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_box_mid<double, B, false><<<dim3((unsigned)nblk, 1), mid_threads<double, B>(), sm, st>>>(
      Y0, 0, nullptr, g, S->twl64, S->twL, make_int3(S->twf[0], S->twf[1], S->twf[2]), make_tw64<double>(), block_order);
  k_spec_fold<<<(unsigned)((nf + 255) / 256), 256, 0, st>>>(block_order, B, g, nf, box_pow2(n) / (double)n, S->gf64, S->gf32,
                                                          S->gfdf);
  const cudaError_t e = cudaStreamSynchronize(st);
  release();
  if (e != cudaSuccess || cudaGetLastError() != cudaSuccess)
    return set_error(LGF_E_CUDA, "box spectrum kernels failed: %s", cudaGetErrorString(e));
  return gen_blocks(S, B, st);
}

int box_spectrum(lgf_table *t, const int nb[3], BoxSpec **out, cudaStream_t st) {
  for (int a = 0; a < 3; ++a) {
    if (nb[a] < 1 || nb[a] > BOX_NB_MAX)
      return set_error(LGF_E_UNSUPPORTED, "box mode supports 1..%d blocks per axis (got %d)", BOX_NB_MAX, nb[a]);
    if (nb[a] * t->B > t->N)
      return set_error(LGF_E_TABLE_RANGE, "box of %d blocks along axis %d exceeds the table's LGF extent", nb[a], a);
  }
  std::lock_guard<std::mutex> g(t->mu);
  const auto key = std::make_tuple(nb[0], nb[1], nb[2]);
  auto it = t->box.find(key);
  BoxSpec *S = it != t->box.end() ? it->second : nullptr;
  if (!S) {
    S = new BoxSpec();
    for (int a = 0; a < 3; ++a) S->nb[a] = nb[a];
    const int rc = t->B == 8 ? gen_spectrum<8>(t, S, st) : gen_spectrum<16>(t, S, st);
    if (rc) {
      delete S;
      return rc;
    }
    t->box[key] = S;
  }
  *out = S;
  return LGF_OK;
}

}  // namespace lgf
