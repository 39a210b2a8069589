// refresh.cu -- velocity refresh u = -C^T L_E^{-1} omega on one level (Sec. 4.1, Eq. (eq:vel_update)).
//
// Staggered lattice (Sec. 2.1): the velocity lives on the positive faces of a cell, the vorticity and the
// streamfunction on its positive edges; component a of cell n is stored at index n (face centre
// n + (1,1,1)/2 + e_a/2, edge centre n + (1,1,1) - e_a/2, in cells).  The LGF of the edge Laplacian is
// the cell one (the lattice is shift-invariant), so L_E^{-1} is the library's three-component Poisson
// solve; C^T, the curl from edges to faces (the transpose of the face-to-edge curl C, Eq. (eq:mimetic)),
// is a backward difference:
//   (C^T psi)_x[n] = (psi_z[n] - psi_z[n - e_y] - psi_y[n] + psi_y[n - e_z]) / h   (and cyclically).
// The backward differences reach one cell below a block toward -x, -y, -z, so the streamfunction is
// solved on the caller's blocks (sources and targets) and on their -x, -y, -z neighbour blocks (targets).
#include <cuda_runtime.h>
#include <string.h>

#include <list>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "internal.h"
#include "solver.h"

namespace lgf {

template <class T>
__device__ __forceinline__ double ld(const T *p, int64_t i) {
  return (double)p[i];
}

// u = -C^T psi on the caller's blocks; grid (nblocks, 3 components), 256 threads.
// psi: [3][next][B^3] over the extended block set whose first n blocks are the caller's; nbr[b][a] is the
// extended index of block b's neighbour toward -e_a.
template <class T>
__global__ void __launch_bounds__(256) k_curl_t(const T *__restrict__ psi, int64_t pcs, const int32_t *__restrict__ nbr,
                                                int shift, double inv_h, T *__restrict__ u, int64_t ucs) {
  const int b = blockIdx.x, comp = blockIdx.y, B = 1 << shift, B3 = 1 << (3 * shift);
  const int a1 = (comp + 1) % 3, a2 = (comp + 2) % 3;  // (C^T psi)_c = d_{a1} psi_{a2} - d_{a2} psi_{a1}
  const int nb1 = nbr[3 * b + a1], nb2 = nbr[3 * b + a2];
  for (int off = threadIdx.x; off < B3; off += blockDim.x) {
    const int c[3] = {off & (B - 1), (off >> shift) & (B - 1), off >> (2 * shift)};
    const int st1 = 1 << (a1 * shift), st2 = 1 << (a2 * shift);  // element strides along a1, a2
    // index of the cell one step toward -e_a1 (-e_a2): this block, or the neighbour's last layer
    const int64_t own = (int64_t)b * B3 + off;
    const int64_t m1 = c[a1] > 0 ? own - st1 : (int64_t)nb1 * B3 + off + (int64_t)(B - 1) * st1;
    const int64_t m2 = c[a2] > 0 ? own - st2 : (int64_t)nb2 * B3 + off + (int64_t)(B - 1) * st2;
    const double d1 = ld(psi, a2 * pcs + own) - ld(psi, a2 * pcs + m1);  // backward difference along a1 of psi_a2
    const double d2 = ld(psi, a1 * pcs + own) - ld(psi, a1 * pcs + m2);  // along a2 of psi_a1
    u[comp * ucs + own] = (T)(-(d1 - d2) * inv_h);
  }
}

// Extended block set of a mesh (the caller's blocks first, then their missing -x, -y, -z neighbours as targets only)
// and the neighbour table on the device, cached by geometry as the solver's plans are.
struct RefreshPlan {
  std::vector<int32_t> ijk;
  std::vector<uint8_t> roles;
  int32_t *d_nbr = nullptr;
  int next = 0;
  ~RefreshPlan() { cudaFree(d_nbr); }
};
static std::mutex g_rp_mu;
static std::list<std::pair<std::string, std::shared_ptr<RefreshPlan>>> g_rp;  // most recent first

static int refresh_plan(const lgf_mesh *m, std::shared_ptr<RefreshPlan> &out, cudaStream_t st) {
  const int n = m->nblocks[0];
  int dev = 0;
  cudaGetDevice(&dev);
  std::string key((const char *)&dev, sizeof dev);
  key.append((const char *)&m->block, 4);
  key.append((const char *)m->block_ijk, 12 * (size_t)n);
  std::lock_guard<std::mutex> g(g_rp_mu);
  for (auto it = g_rp.begin(); it != g_rp.end(); ++it)
    if (it->first == key) {
      g_rp.splice(g_rp.begin(), g_rp, it);
      out = it->second;
      return LGF_OK;
    }
  auto P = std::make_shared<RefreshPlan>();
  std::map<std::tuple<int, int, int>, int> index;
  P->ijk.assign(m->block_ijk, m->block_ijk + 3 * (size_t)n);
  for (int i = 0; i < n; ++i) index[std::make_tuple(P->ijk[3 * i], P->ijk[3 * i + 1], P->ijk[3 * i + 2])] = i;
  std::vector<int32_t> nbr(3 * (size_t)n);
  for (int i = 0; i < n; ++i)
    for (int a = 0; a < 3; ++a) {
      int c[3] = {m->block_ijk[3 * i], m->block_ijk[3 * i + 1], m->block_ijk[3 * i + 2]};
      --c[a];
      const auto at = std::make_tuple(c[0], c[1], c[2]);
      auto it = index.find(at);
      if (it == index.end()) {
        it = index.emplace(at, (int)(P->ijk.size() / 3)).first;
        P->ijk.insert(P->ijk.end(), c, c + 3);
      }
      nbr[3 * i + a] = it->second;
    }
  P->next = (int)(P->ijk.size() / 3);
  P->roles.assign(P->next, 2);
  for (int i = 0; i < n; ++i) P->roles[i] = 3;
  if (cudaMalloc(&P->d_nbr, sizeof(int32_t) * nbr.size()) != cudaSuccess) {
    cudaGetLastError();
    return set_error(LGF_E_OOM, "velocity refresh neighbour table");
  }
  // on the device before any stream can find the plan: a copy from pageable memory on the legacy stream may return before
  // the transfer has ended, and the caller's streams do not wait for that stream
  if (cudaMemcpyAsync(P->d_nbr, nbr.data(), sizeof(int32_t) * nbr.size(), cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess) {
    cudaGetLastError();
    return set_error(LGF_E_CUDA, "velocity refresh neighbour table upload");
  }
  g_rp.emplace_front(key, P);
  while (g_rp.size() > 1024) g_rp.pop_back();  // cudaFree inside orders against in-flight work
  out = P;
  return LGF_OK;
}

}  // namespace lgf

using namespace lgf;

extern "C" int lgf_velocity_refresh(lgf_table *t, const lgf_mesh *m, const void *omega_dev, void *u_dev,
                                    int32_t dtype, const lgf_solve_opts *opts, lgf_report *rep, void *cuda_stream) {
  if (!t) return set_error(LGF_E_INVALID_ARG, "table is NULL");
  int rc = check_mesh(m, t->B);
  if (rc) return rc;
  if (m->nlevels != 1) return set_error(LGF_E_MESH, "the velocity refresh takes one level (got %d)", m->nlevels);
  if (!omega_dev || !u_dev) return set_error(LGF_E_INVALID_ARG, "field pointer NULL");
  if (omega_dev == u_dev) return set_error(LGF_E_INVALID_ARG, "omega and u alias");
  if (dtype != LGF_F64 && dtype != LGF_F32) return set_error(LGF_E_INVALID_ARG, "dtype %d", dtype);
  lgf_solve_opts o{LGF_PREC_FP64, LGF_MAC_AUTO, 0, 0, 0.0, 0, 0};
  if (opts) o = *opts;
  if (o.precision < 0 || o.precision > 2) return set_error(LGF_E_INVALID_ARG, "precision %d", o.precision);
  if (o.mac_mode < 0 || o.mac_mode > 2) return set_error(LGF_E_INVALID_ARG, "mac_mode %d", o.mac_mode);
  if ((rc = check_slices(o))) return rc;
  if (rep) memset(rep, 0, sizeof(*rep));
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const int B = m->block, n = m->nblocks[0];
  const int shift = B == 8 ? 3 : 4;
  const int64_t B3 = (int64_t)B * B * B;
  std::shared_ptr<RefreshPlan> P;
  if ((rc = refresh_plan(m, P, st))) return rc;
  const int next = P->next;
  lgf_mesh me = *m;
  const int32_t nb_ext[1] = {next};
  me.nblocks = nb_ext;
  me.block_ijk = P->ijk.data();
  me.block_role = P->roles.data();
  // scratch of the table's workspace for this stream: omega on the extended set (the added blocks are not sources,
  // never read) and psi on the extended set
  const size_t es = dtype == LGF_F64 ? 8 : 4;
  const int64_t ext_cs = (int64_t)next * B3, ucs = (int64_t)n * B3;
  Workspace *ws = workspace_for(t, st);
  if ((rc = ws->buf[21].reserve(es * 3 * (size_t)ext_cs)) || (rc = ws->buf[22].reserve(es * 3 * (size_t)ext_cs))) return rc;
  void *om = ws->buf[21].p, *psi = ws->buf[22].p;
  for (int c = 0; c < 3; ++c)
    cudaMemcpyAsync((char *)om + es * c * ext_cs, (const char *)omega_dev + es * c * ucs, es * ucs,
                    cudaMemcpyDeviceToDevice, st);
  rc = solve_poisson(t, &me, 3, om, psi, dtype, o, rep, st, true);
  if (rc == LGF_OK) {
    const double inv_h = 1.0 / m->h0;
    if (dtype == LGF_F64)
      k_curl_t<double><<<dim3(n, 3), 256, 0, st>>>((const double *)psi, ext_cs, P->d_nbr, shift, inv_h,
                                                  (double *)u_dev, ucs);
    else
      k_curl_t<float><<<dim3(n, 3), 256, 0, st>>>((const float *)psi, ext_cs, P->d_nbr, shift, inv_h,
                                                 (float *)u_dev, ucs);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) rc = set_error(LGF_E_CUDA, "curl launch: %s", cudaGetErrorString(e));
    else if (rep) rep->kernel_launches += 1;
  }
  return rc;
}
