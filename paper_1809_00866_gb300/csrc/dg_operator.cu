// Matrix-free DG operator on sm_103a: residual f_h (Eq. (NSdiscrRes)), its exact linearisation
// (Eqs. (jacTrilFnotNU), (jacTrilnu)) and the finite-difference action (Eqs. (matrix-free), (epsdef)),
// as a face pass (dg_face.cu) and a volume pass (dg_volume.cu); projections onto the modal basis.
#include <algorithm>
#include <mutex>
#include <vector>

#include "dg_opargs.h"

namespace dg {

template <int K>
struct Sz {
  static constexpr int NB = nb_of(K), N1 = K + 1, NQ = N1 * N1 * N1, NQF = N1 * N1;
};

// ------------------------------------------------------- Taylor-Green vortex
template <int K>
__global__ void __launch_bounds__(128) tgv_kernel(MeshDev M, const double* Bvol, const double* wvol,
                                                  const double* xg, double* w) {
  using S = Sz<K>;
  constexpr int NB = S::NB, NQ = S::NQ, N1 = S::N1;
  __shared__ double sF[4 * NQ];
  for (int e = blockIdx.x; e < M.ne; e += gridDim.x) {
    const ElemGeom g = elem_geom(M, e);
    for (int q = threadIdx.x; q < NQ; q += blockDim.x) {
      const int q0 = q / (N1 * N1), q1 = (q / N1) % N1, q2 = q % N1;
      const double x = g.lo[0] + 0.5 * g.h[0] * (xg[q0] + 1.0);
      const double y = g.lo[1] + 0.5 * g.h[1] * (xg[q1] + 1.0);
      const double z = g.lo[2] + 0.5 * g.h[2] * (xg[q2] + 1.0);
      const double wq = wvol[q];
      sF[0 * NQ + q] = sin(x) * cos(y) * cos(z) * wq;
      sF[1 * NQ + q] = -cos(x) * sin(y) * cos(z) * wq;
      sF[2 * NQ + q] = 0.0;
      sF[3 * NQ + q] = (cos(2.0 * x) + cos(2.0 * y)) * (cos(2.0 * z) + 2.0) * (1.0 / 16.0) * wq;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 4 * NB; t += blockDim.x) {
      const int v = t / NB, m = t - v * NB;
      double acc = 0.0;
      for (int q = 0; q < NQ; ++q) acc += Bvol[q * NB + m] * sF[v * NQ + q];
      w[(size_t)e * 4 * NB + t] = acc * g.s;
    }
    __syncthreads();
  }
}

// ------------------------------------------------ points and projections of given fields
template <int K>
__global__ void __launch_bounds__(128) quad_points_kernel(MeshDev M, const double* xg, double* xyz) {
  constexpr int N1 = K + 1, NQ = N1 * N1 * N1;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)M.ne * NQ;
       i += (long long)gridDim.x * blockDim.x) {
    const int e = (int)(i / NQ), q = (int)(i - (long long)e * NQ);
    const int q0 = q / (N1 * N1), q1 = (q / N1) % N1, q2 = q % N1;
    const ElemGeom g = elem_geom(M, e);
    double* o = xyz + i * 3;
    o[0] = g.lo[0] + 0.5 * g.h[0] * (xg[q0] + 1.0);
    o[1] = g.lo[1] + 0.5 * g.h[1] * (xg[q1] + 1.0);
    o[2] = g.lo[2] + 0.5 * g.h[2] * (xg[q2] + 1.0);
  }
}

// w[e][v][m] = s_e sum_q phi_hat_m(x_q) wvol_q vals[e][v][q]: the Gauss-rule L2 projection onto the
// orthonormal basis phi_m = phi_hat_m / s_e (the |K|/8 of dx and the 1/s of phi_m give s_e)
template <int K>
__global__ void __launch_bounds__(128) project_points_kernel(MeshDev M, const double* Bvol, const double* wvol,
                                                             const double* vals, double* w) {
  using S = Sz<K>;
  constexpr int NB = S::NB, NQ = S::NQ;
  for (int e = blockIdx.x; e < M.ne; e += gridDim.x) {
    const ElemGeom g = elem_geom(M, e);
    const double* ve = vals + (size_t)e * 4 * NQ;
    for (int t = threadIdx.x; t < 4 * NB; t += blockDim.x) {
      const int v = t / NB, m = t - v * NB;
      double acc = 0.0;
      for (int q = 0; q < NQ; ++q) acc += Bvol[q * NB + m] * wvol[q] * ve[v * NQ + q];
      w[(size_t)e * 4 * NB + t] = acc * g.s;
    }
  }
}

// ------------------------------------------------------------- FD helpers
__global__ void fd_perturb_kernel(long long n, const double* w, const double* v, const double* wnorm2,
                                  const double* vnorm2, double* out) {
  const double nv = sqrt(*vnorm2);
  const double delta = nv > 0.0 ? 1e-9 * sqrt(1.0 + sqrt(*wnorm2)) / nv : 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = w[i] + delta * v[i];
}
__global__ void fd_finish_kernel(long long n, int nb, const double* f1, const double* f0, const double* v,
                                 const double* wnorm2, const double* vnorm2, double inv_gdt, const double* geo,
                                 double* out) {
  const double nv = sqrt(*vnorm2);
  const double delta = nv > 0.0 ? 1e-9 * sqrt(1.0 + sqrt(*wnorm2)) / nv : 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int var = (int)((i / nb) & 3);
    const long long e = i / (4 * nb);
    const double mass = var < 3 ? inv_gdt * geo[e * kGeo + 11] * v[i] : 0.0;
    out[i] = (delta > 0.0 ? (f1[i] - f0[i]) / delta : 0.0) + mass;
  }
}

// ------------------------------------------------------------- launchers
template <class R>
static OpArgsT<R> make_args(Handle* h, const R* in, R* out) {
  OpArgsT<R> a;
  a.M = mesh_dev(h);
  a.in = in;
  a.out = out;
  if constexpr (sizeof(R) == 8) {
    a.face_buf = h->face_buf;
    a.ubar = h->ubar;
    a.dFlux = h->dFlux;
  } else {
    a.face_buf = h->face_buf_f;
    a.ubar = h->ubar_f;
    a.dFlux = h->dFlux_f;
  }
  a.nu = R(h->p.nu);
  a.eta8 = R(0.125 * h->p.eta);
  a.c = h->p.ac_c;
  a.inv_gdt = h->inv_gdt;
  a.status = h->status;
  a.riemann_its = h->dbg.riemann_its;
  return a;
}

// The grids of the passes are one wave of the GPU, so that no SM runs a second, thinner wave of a
// grid-stride loop.
int resident_ctas(const void* fn, int threads, size_t smem) {
  struct Entry {
    const void* fn;
    int threads;
    size_t smem;
    int n;
  };
  static std::mutex mu;
  static std::vector<Entry> cache;
  std::lock_guard<std::mutex> lk(mu);
  for (const Entry& c : cache)
    if (c.fn == fn && c.threads == threads && c.smem == smem) return c.n;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, smem) != cudaSuccess || n < 1) {
    cudaGetLastError();
    return 0;  // unknown: the caller keeps its own bound
  }
  cache.push_back(Entry{fn, threads, smem, n});
  return n;
}

// The tangent passes (the hot products of the solver) take the handle's launch shapes. Every output
// entry is computed by the same arithmetic in the same order whatever the shape, so the results do
// not depend on it.
template <class R>
static int run_operator(Handle* h, const OpArgsT<R>& a, int mode, cudaStream_t st, bool face_only = false) {
  const bool tan = mode == MODE_TAN || mode == MODE_LINPART;
  const OpTune tu = mode == MODE_TAN ? h->tune[sizeof(R) == 4 ? 1 : 0] : OpTune{};
  const int cf = tan ? (sizeof(R) == 4 ? DG_PROF_FACE_TAN32 : DG_PROF_FACE_TAN) : DG_PROF_FACE_RES;
  const int cv = tan ? (sizeof(R) == 4 ? DG_PROF_VOL_TAN32 : DG_PROF_VOL_TAN) : DG_PROF_VOL_RES;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  int rc;
  if ((rc = prof_begin(h, st, &e0))) return rc;
  if ((rc = face_pass<R>(h, a, mode, tu, st))) return rc;
  if ((rc = prof_end(h, cf, st, e0))) return rc;
  if (face_only) return DG_OK;
  if ((rc = prof_begin(h, st, &e1))) return rc;
  if ((rc = volume_pass<R>(h, a, mode, tu, st))) return rc;
  if ((rc = prof_end(h, cv, st, e1))) return rc;
  ++h->op_apps;
  return DG_OK;
}

int op_residual(Handle* h, const double* w, double* f, bool store_lin, cudaStream_t st) {
  OpArgs a = make_args(h, w, f);
  if (store_lin) a.status = h->status + 1;  // the linearisation's own word, read by dg_set_linearization
  return run_operator(h, a, store_lin ? MODE_RES_LIN : MODE_RES, st);
}

int op_tangent(Handle* h, const double* v, double* out, cudaStream_t st) {
  return run_operator(h, make_args(h, v, out), MODE_TAN, st);
}

int op_tangent_f32(Handle* h, const float* v, float* out, int tc, cudaStream_t st) {
  const OpArgsT<float> a = make_args(h, v, out);
  if (!tc) return run_operator(h, a, MODE_TAN, st);
  // the face pass as usual, then the volume pass with its contractions on the tensor cores
  int rc = run_operator(h, a, MODE_TAN, st, true);
  if (rc) return rc;
  cudaEvent_t e1 = nullptr;
  if ((rc = prof_begin(h, st, &e1))) return rc;
  if ((rc = tc_volume_tangent(h, v, out, tc, st))) return rc;
  if ((rc = prof_end(h, DG_PROF_VOL_TC32, st, e1))) return rc;
  ++h->op_apps;
  return DG_OK;
}

int op_linear_part(Handle* h, const double* v, double* out, cudaStream_t st) {
  return run_operator(h, make_args(h, v, out), MODE_LINPART, st);
}

int op_fd(Handle* h, const double* v, double* out, cudaStream_t st) {
  const long long n = h->lev[0].n;
  int rc = vec_norm2(h, v, n, h->red_out, st);
  if (rc) return rc;
  const int blocks = h->nsm * 8;
  fd_perturb_kernel<<<blocks, 256, 0, st>>>(n, h->wlin, v, h->wnorm2, h->red_out, h->fd_w);
  DG_LAUNCH_CHECK(h);
  rc = op_residual(h, h->fd_w, h->fd_f, false, st);
  if (rc) return rc;
  fd_finish_kernel<<<blocks, 256, 0, st>>>(n, h->lev[0].nb, h->fd_f, h->flin, v, h->wnorm2, h->red_out,
                                           h->inv_gdt, h->geo, out);
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

int op_quad_points(Handle* h, double* xyz, cudaStream_t st) {
  const MeshDev M = mesh_dev(h);
  const int grid = h->nsm * 8;
  switch (h->tab.k) {
    case 1: quad_points_kernel<1><<<grid, 128, 0, st>>>(M, h->tab.xg, xyz); break;
    case 2: quad_points_kernel<2><<<grid, 128, 0, st>>>(M, h->tab.xg, xyz); break;
    case 3: quad_points_kernel<3><<<grid, 128, 0, st>>>(M, h->tab.xg, xyz); break;
    case 4: quad_points_kernel<4><<<grid, 128, 0, st>>>(M, h->tab.xg, xyz); break;
  }
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

int op_project_points(Handle* h, const double* vals, double* w, cudaStream_t st) {
  const MeshDev M = mesh_dev(h);
  const int grid = std::min(h->ne, h->nsm * 8);
  switch (h->tab.k) {
    case 1: project_points_kernel<1><<<grid, 128, 0, st>>>(M, h->tab.Bvol, h->tab.wvol, vals, w); break;
    case 2: project_points_kernel<2><<<grid, 128, 0, st>>>(M, h->tab.Bvol, h->tab.wvol, vals, w); break;
    case 3: project_points_kernel<3><<<grid, 128, 0, st>>>(M, h->tab.Bvol, h->tab.wvol, vals, w); break;
    case 4: project_points_kernel<4><<<grid, 128, 0, st>>>(M, h->tab.Bvol, h->tab.wvol, vals, w); break;
  }
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

int op_project_tgv(Handle* h, double* w, cudaStream_t st) {
  const MeshDev M = mesh_dev(h);
  const int grid = h->ne < h->nsm * 8 ? h->ne : h->nsm * 8;
  switch (h->tab.k) {
    case 1: tgv_kernel<1><<<grid, 128, 0, st>>>(M, h->tab.Bvol, h->tab.wvol, h->tab.xg, w); break;
    case 2: tgv_kernel<2><<<grid, 128, 0, st>>>(M, h->tab.Bvol, h->tab.wvol, h->tab.xg, w); break;
    case 3: tgv_kernel<3><<<grid, 128, 0, st>>>(M, h->tab.Bvol, h->tab.wvol, h->tab.xg, w); break;
    case 4: tgv_kernel<4><<<grid, 128, 0, st>>>(M, h->tab.Bvol, h->tab.wvol, h->tab.xg, w); break;
    default: return fail(h, DG_ERR_ARG, "unsupported degree");
  }
  DG_LAUNCH_CHECK(h);
  return DG_OK;
}

// ------------------------------------------------- residual without allocation
// Scratch of dg_residual_noalloc: the face pass's output (the documented limit of N_e * 6 * 7 * N_2
// doubles, N_2 = (k+1)(k+2)/2, holds it twice over), in a file-scope device array instead of the handle's own buffers. Every GPU that
// loads the library holds it until the process exits.
static __device__ __align__(256) double g_noalloc_scratch[DG_NOALLOC_SCRATCH_DOUBLES];

// Device address of g_noalloc_scratch on the handle's device, looked up once per device with
// that device current (the caller's device must be the handle's). In host code the array's name
// is only a host-side stand-in, never a device address, so it must not be passed to a kernel.
static int noalloc_scratch(Handle* h, double** out) {
  static std::mutex mu;
  static double* addr[64] = {};
  const int dev = h->device;
  int cur = -1;
  DG_CUDA(h, cudaGetDevice(&cur));
  if (cur != dev)
    return fail(h, DG_ERR_ARG, "dg_residual_noalloc: make the handle's device (" + std::to_string(dev) +
                                   ") current; device " + std::to_string(cur) + " is");
  if (dev < 0 || dev >= 64) return fail(h, DG_ERR_ARG, "device index out of range for the static scratch");
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[dev]) {
    double* p = nullptr;
    DG_CUDA(h, cudaGetSymbolAddress((void**)&p, g_noalloc_scratch));
    if (!p) return fail(h, DG_ERR_CUDA, "cudaGetSymbolAddress returned a null address");
    addr[dev] = p;
  }
  *out = addr[dev];
  return DG_OK;
}

}  // namespace dg

extern "C" int dg_residual_noalloc(dg_handle* hh, const double* w, double* f, void* stream) {
  using namespace dg;
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h) return DG_ERR_ARG;
  if (!w || !f || w == f) return fail(h, DG_ERR_ARG, "w and f must be distinct non-null device pointers");
  const int n2 = h->tab.n2;
  const long long need = (long long)h->ne * 6 * 7 * n2;
  if (need > (long long)DG_NOALLOC_SCRATCH_DOUBLES)
    return fail(h, DG_ERR_ARG,
                "mesh too large for the static scratch of dg_residual_noalloc: it needs N_e*42*N_2 = " +
                    std::to_string(need) + " doubles, the limit is " + std::to_string(DG_NOALLOC_SCRATCH_DOUBLES));
  double* scratch = nullptr;
  int rc = noalloc_scratch(h, &scratch);
  if (rc) return rc;
  OpArgs a = make_args(h, w, f);
  a.face_buf = scratch;  // face_buf_size: about half of N_e * 42 * N_2
  return run_operator(h, a, MODE_RES, as_stream(stream));
}
