// Pseudo-spectral incompressible Navier-Stokes (paper Sec. 2.2, Eqs. (7)-(8))
// in rotational form, fused into the FFT passes of Sec. 3.
//
// One evaluation of the nonlinear term is five kernels:
//   1. ns_invx_curl : uhat (3) -> inverse x pass of u and omega = i k x u (6)
//   2. ns_invy      : inverse y pass of the 6 fields
//   3. ns_z_product : per z line: c2r of the 6 fields, n = u x omega in
//                     registers, r2c of the 3 products (real fields never
//                     touch global memory)
//   4. ns_fwdy      : forward y pass of the 3 fields
//   5. ns_fwdx      : forward x pass + 1/N^3 + 2/3 dealias + projection
//                     + forcing + the RK2 integrating-factor update
//
// The 2/3 rule is used throughout, not only to zero the products: modes
// with 3|k| >= n on any axis are zero in the state, so every pass reads only
// the rows and columns that can be nonzero and writes only those a later
// pass reads.  The arrays keep the full [n][n][n/2+1] layout; the untouched
// parts are never read.
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#define FFTK_PAIRED_FP32 2  // see fft_engine.cuh
#include "ns_passes.cuh"

namespace fftk {
// ------------------------------------------------------------ reductions ---
// Energy of the forced modes, 1/2 sum w |u|^2 over k2min <= |k|^2 <= k2max,
// in FP64; one block, fixed order.
__global__ void k_forced_energy(const float2* __restrict__ u, NSGeom g, int kr, int k2min,
                                int k2max, double* ef) {
  pdl_wait();
  __shared__ double red[256];
  const int side = 2 * kr + 1;
  const int count = side * side * (kr + 1);
  double acc = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) {
    const int kz = i % (kr + 1);
    const int t = i / (kr + 1);
    const int ky = t % side - kr, kx = t / side - kr;
    const int k2 = kx * kx + ky * ky + kz * kz;
    if (k2 < k2min || k2 > k2max) continue;
    const int ax = kx < 0 ? kx + g.n : kx, ay = ky < 0 ? ky + g.n : ky;
    const long long idx = ((long long)ax * g.n + ay) * g.h1 + kz;
    const double w = kz == 0 ? 1.0 : 2.0;
    double s = 0.0;
    for (int f = 0; f < 3; ++f) {
      const float2 v = u[idx + f * g.M];
      s += (double)v.x * v.x + (double)v.y * v.y;
    }
    acc += 0.5 * w * s;
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *ef = red[0];
}


int ns_kmax(int n) { return (int)std::floor(std::sqrt(3.0) * (n / 2) + 0.5) + 1; }

NSGeom make_geom(int n) {
  NSGeom g;
  g.n = n;
  g.h1 = n / 2 + 1;
  g.kd = (n - 1) / 3;
  g.kc = g.kd + 1;
  g.nk = 2 * g.kd + 1;
  g.M = (long long)n * n * g.h1;
  return g;
}

fftk_status ns_ensure(fftk_plan p) {
  std::lock_guard<std::mutex> lk(p->mu);
  if (p->ns) return FFTK_OK;
  NSWork* s = new (std::nothrow) NSWork;
  if (!s) return FFTK_ERR_OOM;
  s->g = make_geom(p->nx);
  s->kmax = ns_kmax(p->nx);
  s->etab_len = 3 * s->g.kd * s->g.kd + 1;
  const size_t fb = sizeof(float2) * (size_t)s->g.M;
  const size_t fw = sizeof(float2) * (size_t)p->nx * p->nx * (size_t)ns_row(p->nx);  // padded rows (fused path)
  const int width = 2 + s->kmax + 1;
  cudaError_t e = cudaMalloc(&s->w, 6 * (fw > fb ? fw : fb));
  if (e == cudaSuccess) e = cudaMalloc(&s->u1, 3 * fb);
  if (e == cudaSuccess) e = cudaMemset(s->u1, 0, 3 * fb);
  if (e == cudaSuccess) e = cudaMalloc(&s->etab, sizeof(float2) * 2 * (size_t)s->etab_len);
  if (e == cudaSuccess) e = cudaMalloc(&s->ef, sizeof(double));
  if (e == cudaSuccess) e = cudaMemset(s->ef, 0, sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&s->part, sizeof(double) * (size_t)diag_blocks(width) * width);
  if (e == cudaSuccess) e = cudaMalloc(&s->dout, sizeof(double) * (size_t)width);
  if (e == cudaSuccess) e = cudaMallocHost(&s->hout, sizeof(double) * (size_t)width);
  s->diag_smem = (int)(sizeof(double) * DIAG_WARPS * (s->kmax + 1));
  if (e == cudaSuccess) e = diag_attr();
  if (e != cudaSuccess) {
    cudaGetLastError();
    cudaFree(s->w);
    cudaFree(s->u1);
    cudaFree(s->etab);
    cudaFree(s->ef);
    cudaFree(s->part);
    cudaFree(s->dout);
    if (s->hout) cudaFreeHost(s->hout);
    delete s;
    return e == cudaErrorMemoryAllocation ? FFTK_ERR_OOM : FFTK_ERR_CUDA;
  }
  p->ns = s;
  return FFTK_OK;
}

// exp(-nu k^2 dt) for integer k^2, FP64 on the host, split into an FP32 pair
// hi = fl(E), lo = fl(E - hi).
static fftk_status ns_etab(fftk_plan p, double nu, double dt) {
  NSWork* s = p->ns;
  if (s->etab_nu == nu && s->etab_dt == dt) return FFTK_OK;
  std::vector<float2> h(2 * (size_t)s->etab_len);
  for (int half = 0; half < 2; ++half)
    for (int k2 = 0; k2 < s->etab_len; ++k2) {
      const double E = std::exp(-nu * (double)k2 * (half ? 0.5 * dt : dt));
      const float hi = (float)E;
      h[(size_t)half * s->etab_len + k2] = make_float2(hi, (float)(E - (double)hi));
    }
  cudaError_t e = cudaMemcpy(s->etab, h.data(), sizeof(float2) * h.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return from_cuda(e);
  s->etab_nu = nu;
  s->etab_dt = dt;
  return FFTK_OK;
}

// The fused passes' second six-field workspace (padded rows), on first use.
cudaError_t ns_second_workspace(fftk_plan p) {
  NSWork* s = p->ns;
  std::lock_guard<std::mutex> lk(p->mu);
  if (s->w2) return cudaSuccess;
  const size_t fw = sizeof(float2) * (size_t)p->nx * p->nx * (size_t)ns_row(p->nx);
  cudaError_t e = cudaMalloc(&s->w2, 6 * fw);
  if (e != cudaSuccess) {
    cudaGetLastError();
    s->w2 = nullptr;
  }
  return e;
}

// ---------------------------------------------- split-precision NS step ----
// Plans of dtype FFTK_R32_SPLIT16 evaluate the right-hand side with the x and
// y passes on the tensor cores (split FP16 radix-16 stages, restricted to the
// 2/3-rule set): u and omega = i k x u on the kept modes, inverse x and y
// passes of the six fields, the fused FP32 z pass (u x omega in registers),
// forward y and x passes of n, and the per-mode update of the fused path.

// w6 = (u, i k x u) on the kept modes; the derivative of the Nyquist wavenumber is 0
__global__ void k_curl_full(const float2* __restrict__ u, float2* __restrict__ w6, NSGeom g) {
  const long long items = (long long)g.nk * g.nk * g.kc;  // k_z fastest
  for (long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x; it < items;
       it += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(it % g.kc);
    const long long ab = it / g.kc;
    const int a = dense_to_a((int)(ab / g.nk), g.n, g.kd), b = dense_to_a((int)(ab % g.nk), g.n, g.kd);
    const long long idx = ((long long)a * g.n + b) * g.h1 + c;
    const int ka = kwav(a, g.n), kb = kwav(b, g.n);
    const float kx = (2 * abs(ka) == g.n) ? 0.f : (float)ka, ky = (2 * abs(kb) == g.n) ? 0.f : (float)kb;
    const float kz = (2 * c == g.n) ? 0.f : (float)c;
    const float2 ux = u[idx], uy = u[idx + g.M], uz = u[idx + 2 * g.M];
    w6[idx] = ux;
    w6[idx + g.M] = uy;
    w6[idx + 2 * g.M] = uz;
    w6[idx + 3 * g.M] = csub(mul_i(uz, ky), mul_i(uy, kz));
    w6[idx + 4 * g.M] = csub(mul_i(ux, kz), mul_i(uz, kx));
    w6[idx + 5 * g.M] = csub(mul_i(uy, kx), mul_i(ux, ky));
  }
}

// the update of every kept mode from n_hat (already scaled by the transform)
__global__ void k_update_full(const float2* __restrict__ nh, const float2* u0, const float2* u1, float2* out,
                              NSGeom g, NSUpdate upd, int mode, const float2* __restrict__ extra) {
  float gforce = 0.f;
  if (upd.feps > 0.0) {
    const double ef = *upd.ef;
    gforce = ef > 0.0 ? (float)(upd.feps / (2.0 * ef)) : 0.f;
  }
  const long long items = (long long)g.nk * g.nk * g.kc;  // the kept modes, k_z fastest
  for (long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x; it < items;
       it += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(it % g.kc);
    const long long ab = it / g.kc;
    const int a = dense_to_a((int)(ab / g.nk), g.n, g.kd), b = dense_to_a((int)(ab % g.nk), g.n, g.kd);
    const long long idx = ((long long)a * g.n + b) * g.h1 + c;
    const int kx = kwav(a, g.n), ky = kwav(b, g.n);
    NSModeIn in;
    ns_mode_load(in, kx * kx + ky * ky + c * c, idx, g.M, upd, mode, u0, u1);
    ns_mode_update(in, nh[idx], nh[idx + g.M], nh[idx + 2 * g.M], kwav(a, g.n), kwav(b, g.n), c, idx, g.M, upd, mode,
                   gforce, u0, u1, extra, out);
  }
}

static cudaError_t ns_z_dispatch(fftk_plan p, cudaStream_t st);

static cudaError_t ns_rhs_split(fftk_plan p, const float2* u, const float2* u0, const float2* u1, float2* out,
                                const NSUpdate& upd, int mode, const float2* extra, cudaStream_t st) {
  NSWork* s = p->ns;
  const NSGeom g = s->g;
  const unsigned grid = 152 * 8;
  const bool tc = cpass_tc_supported(g.n) && g.n <= 1024;
  const float scale = (float)(1.0 / ((double)g.n * g.n * g.n));
  {
    LaunchScope ls(p, KK_AUX, st);
    k_curl_full<<<grid, 256, 0, st>>>(u, s->w, g);
  }
  cudaError_t e = tc ? launch_cpass_tc_pruned(p, 0, +1, s->w, s->w, 6, 1.f, KK_X_INV, st)
                     : launch_pruned_x(p, +1, s->w, s->w, 6, 1.f, st);
  if (e == cudaSuccess)
    e = tc ? launch_cpass_tc_pruned(p, 1, +1, s->w, s->w, 6, 1.f, KK_Y_INV, st)
           : launch_pruned_y(p, +1, s->w, s->w, 6, 1.f, st);
  if (e == cudaSuccess) e = ns_z_dispatch(p, st);
  if (e == cudaSuccess)
    e = tc ? launch_cpass_tc_pruned(p, 1, -1, s->w, s->w, 3, 1.f, KK_Y_FWD, st)
           : launch_pruned_y(p, -1, s->w, s->w, 3, 1.f, st);
  if (e == cudaSuccess)
    e = tc ? launch_cpass_tc_pruned(p, 0, -1, s->w, s->w, 3, scale, KK_X_FWD, st)
           : launch_pruned_x(p, -1, s->w, s->w, 3, scale, st);
  if (e != cudaSuccess) return e;
  {
    LaunchScope ls(p, KK_AUX, st);
    k_update_full<<<grid, 256, 0, st>>>(s->w, u0, u1, out, g, upd, mode, extra);
  }
  return cudaGetLastError();
}

#define NS_SIZES(X) X(8) X(16) X(32) X(64) X(128) X(256) X(512) X(1024)

static cudaError_t ns_z_dispatch(fftk_plan p, cudaStream_t st) {
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return NSLaunch<n>::z(p, st);
    NS_SIZES(CASE)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

static cudaError_t ns_rhs_dispatch(fftk_plan p, const float2* u, const float2* u0, const float2* u1,
                                   float2* out, const NSUpdate& upd, int mode, const float2* extra,
                                   cudaStream_t st) {
  if (!is_pow2(p->nx)) return ns_rhs_radix3(p, u, u0, u1, out, upd, mode, extra, st);
  if (p->dtype == FFTK_R32_SPLIT16) return ns_rhs_split(p, u, u0, u1, out, upd, mode, extra, st);
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return NSLaunch<n>::rhs(p, u, u0, u1, out, upd, mode, extra, st);
    NS_SIZES(CASE)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

static cudaError_t forced_energy(fftk_plan p, const float2* u, const tarang_params* prm,
                                 cudaStream_t st) {
  int kr = 0;
  while ((kr + 1) * (kr + 1) <= prm->force_k2max) ++kr;
  LaunchScope ls(p, KK_NS_REDUCE, st);
  launch_pdl(k_forced_energy, 1, 256, 0, st, u, p->ns->g, kr, prm->force_k2min, prm->force_k2max,
                                     p->ns->ef);
  return cudaGetLastError();
}

fftk_status ns_check(fftk_plan p, const tarang_params* prm, bool need_dt) {
  if (!p || !prm) return FFTK_ERR_INVALID_ARG;
  if (p->nx != p->ny || p->nx != p->nz) return FFTK_ERR_UNSUPPORTED_SIZE;
  if (!ns_size_ok(p->nx)) return FFTK_ERR_UNSUPPORTED_SIZE;
  if (!(prm->nu >= 0.0) || !std::isfinite(prm->nu)) return FFTK_ERR_INVALID_ARG;
  if (need_dt && (!(prm->dt > 0.0) || !std::isfinite(prm->dt))) return FFTK_ERR_INVALID_ARG;
  if (prm->sgs_model && !prm->sgs_model->params) return FFTK_ERR_INVALID_ARG;
  if (prm->sgs_model && !is_pow2(p->nx)) return FFTK_ERR_UNSUPPORTED_SIZE;  // the learned closure: 2^m grids
  if (prm->scheme != TARANG_RK2 && prm->scheme != TARANG_RK4) return FFTK_ERR_INVALID_ARG;
  if (prm->force_eps != 0.0) {
    const int kd = (p->nx - 1) / 3;
    if (!(prm->force_eps > 0.0) || prm->force_k2min < 1 || prm->force_k2max < prm->force_k2min ||
        prm->force_k2max > kd * kd)
      return FFTK_ERR_INVALID_ARG;
  }
  return FFTK_OK;
}

}  // namespace fftk

using namespace fftk;

void ns_free(fftk_plan p) {
  NSWork* s = p->ns;
  if (!s) return;
  cudaFree(s->w);
  cudaFree(s->w2);
  cudaFree(s->u1);
  cudaFree(s->etab);
  cudaFree(s->ef);
  cudaFree(s->part);
  cudaFree(s->dout);
  if (s->hout) cudaFreeHost(s->hout);
  cudaFree(s->r3);
  cudaFree(s->acc);
  rbc_free(s->rbc);
  cudaFree(s->sout);
  sgs_free(s->sgs);
  delete s;
  p->ns = nullptr;
}


// The right-hand side of a checked state into the kept modes of `out`.
cudaError_t fftk::ns_rhs_kept(fftk_plan p, const float2* u, float2* out, const tarang_params* prm, cudaStream_t st) {
  const NSGeom g = p->ns->g;
  NSUpdate upd{p->ns->etab, p->ns->etab_len, nullptr, p->ns->ef, prm->force_eps, prm->force_k2min,
               prm->force_k2max, 0.f,
               (float)(1.0 / ((double)g.n * g.n * g.n))};
  cudaError_t e = cudaSuccess;
  if (prm->force_eps > 0.0) e = forced_energy(p, u, prm, st);
  const float2* extra = nullptr;
  if (e == cudaSuccess && prm->sgs_model) e = sgs_term(p, &p->ns->sgs, u, prm->sgs_model, st, &extra);
  if (e == cudaSuccess) e = ns_rhs_dispatch(p, u, u, nullptr, out, upd, NS_RHS, extra, st);
  return e;
}

extern "C" fftk_status tarang_ns_rhs(fftk_plan p, const void* uhat, void* nhat,
                                     const tarang_params* prm, void* cuda_stream) {
  fftk_status s = ns_check(p, prm, false);
  if (s != FFTK_OK) return s;
  if (!uhat || !nhat || uhat == nhat || misaligned16(uhat) || misaligned16(nhat))
    return FFTK_ERR_INVALID_ARG;
  s = ns_ensure(p);
  if (s != FFTK_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t e = cudaMemsetAsync(nhat, 0, sizeof(float2) * 3 * (size_t)p->ns->g.M, st);
  if (e == cudaSuccess)
    e = ns_rhs_kept(p, static_cast<const float2*>(uhat), static_cast<float2*>(nhat), prm, st);
  return from_cuda(e);
}

extern "C" fftk_status tarang_ns_step(fftk_plan p, void* uhat, const tarang_params* prm, int nsteps,
                                      double* diag_host, void* cuda_stream) {
  fftk_status s = ns_check(p, prm, true);
  if (s != FFTK_OK) return s;
  if (!uhat || nsteps < 0 || misaligned16(uhat)) return FFTK_ERR_INVALID_ARG;
  s = ns_ensure(p);
  if (s != FFTK_OK) return s;
  s = ns_etab(p, prm->nu, prm->dt);
  if (s != FFTK_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  NSWork* w = p->ns;
  const NSGeom g = w->g;
  float2* u = static_cast<float2*>(uhat);
  if (prm->scheme == TARANG_RK4 && !w->acc) {
    cudaError_t ea = cudaMalloc(&w->acc, sizeof(float2) * 3 * (size_t)g.M);
    if (ea != cudaSuccess) {
      cudaGetLastError();
      return from_cuda(ea);
    }
  }
  NSUpdate upd{w->etab, w->etab_len, w->acc, w->ef, prm->force_eps, prm->force_k2min, prm->force_k2max,
               (float)prm->dt, (float)(1.0 / ((double)g.n * g.n * g.n))};
  cudaError_t e = cudaSuccess;
  if (prm->scheme == TARANG_RK4) {
    // four evaluations of N: from u, then from the stage state u1
    for (int it = 0; it < nsteps && e == cudaSuccess; ++it)
      for (int stage = 0; stage < 4 && e == cudaSuccess; ++stage) {
        const float2* in = stage == 0 ? u : w->u1;
        const float2* extra = nullptr;
        if (prm->force_eps > 0.0) e = forced_energy(p, in, prm, st);
        if (e == cudaSuccess && prm->sgs_model) e = sgs_term(p, &w->sgs, in, prm->sgs_model, st, &extra);
        if (e == cudaSuccess)
          e = ns_rhs_dispatch(p, in, u, w->u1, stage == 3 ? u : w->u1, upd, NS_RK4_1 + stage, extra, st);
      }
    if (e != cudaSuccess) return from_cuda(e);
    if (diag_host) return tarang_diag(p, u, prm->nu, diag_host, cuda_stream);
    return FFTK_OK;
  }
  for (int it = 0; it < nsteps && e == cudaSuccess; ++it) {
    const float2* extra = nullptr;
    if (prm->force_eps > 0.0) e = forced_energy(p, u, prm, st);
    if (e == cudaSuccess && prm->sgs_model) e = sgs_term(p, &w->sgs, u, prm->sgs_model, st, &extra);
    if (e == cudaSuccess) e = ns_rhs_dispatch(p, u, u, nullptr, w->u1, upd, NS_STAGE1, extra, st);
    if (e == cudaSuccess && prm->force_eps > 0.0) e = forced_energy(p, w->u1, prm, st);
    if (e == cudaSuccess && prm->sgs_model) e = sgs_term(p, &w->sgs, w->u1, prm->sgs_model, st, &extra);
    if (e == cudaSuccess) e = ns_rhs_dispatch(p, w->u1, u, w->u1, u, upd, NS_STAGE2, extra, st);
  }
  if (e != cudaSuccess) return from_cuda(e);
  if (diag_host) return tarang_diag(p, u, prm->nu, diag_host, cuda_stream);
  return FFTK_OK;
}

// --------------------------------------------------------- initial field ---
namespace fftk {

// Zero every mode outside the 2/3 set and project the kept ones (Eq. (8)).
__global__ void k_ic_shape(float2* u, NSGeom g) {
  const long long total = g.M;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % g.h1);
    const long long ab = i / g.h1;
    const int b = (int)(ab % g.n), a = (int)(ab / g.n);
    if (!(kept_xy(a, g.n, g.kd) && kept_xy(b, g.n, g.kd) && c < g.kc)) {
      u[i] = u[i + g.M] = u[i + 2 * g.M] = make_float2(0.f, 0.f);
      continue;
    }
    const float kx = (float)kwav(a, g.n), ky = (float)kwav(b, g.n), kz = (float)c;
    const float k2 = kx * kx + ky * ky + kz * kz;
    if (k2 == 0.f) {
      u[i] = u[i + g.M] = u[i + 2 * g.M] = make_float2(0.f, 0.f);
      continue;
    }
    const float2 ux = u[i], uy = u[i + g.M], uz = u[i + 2 * g.M];
    const float2 kd = make_float2((kx * ux.x + ky * uy.x + kz * uz.x) / k2,
                                  (kx * ux.y + ky * uy.y + kz * uz.y) / k2);
    u[i] = csub(ux, cscale(kd, kx));
    u[i + g.M] = csub(uy, cscale(kd, ky));
    u[i + 2 * g.M] = csub(uz, cscale(kd, kz));
  }
}

// Make the k_z = 0 plane exactly Hermitian: f(-kx,-ky) = conj f(kx,ky).
__global__ void k_ic_herm(float2* u, NSGeom g) {
  const long long total = 3LL * g.n * g.n;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int f = (int)(i / ((long long)g.n * g.n));
    const int ab = (int)(i % ((long long)g.n * g.n));
    const int a = ab / g.n, b = ab % g.n;
    const int a2 = (g.n - a) % g.n, b2 = (g.n - b) % g.n;
    const long long i1 = ((long long)a * g.n + b) * g.h1, i2 = ((long long)a2 * g.n + b2) * g.h1;
    if (i2 < i1) continue;
    float2* base = u + f * g.M;
    if (i1 == i2) {
      base[i1].y = 0.f;
    } else {
      const float2 p = base[i1], q = base[i2];
      const float2 avg = make_float2(0.5f * (p.x + q.x), 0.5f * (p.y - q.y));
      base[i1] = avg;
      base[i2] = cconj(avg);
    }
  }
}

// u *= s[nint|k|] on the kept modes.
__global__ void k_ic_rescale(float2* u, NSGeom g, const double* __restrict__ s, int kmax) {
  const long long total = (long long)g.nk * g.nk * g.kc;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int kz = (int)(i % g.kc);
    const long long t = i / g.kc;
    const int a = dense_to_a((int)(t / g.nk), g.n, g.kd), b = dense_to_a((int)(t % g.nk), g.n, g.kd);
    const long long kx = kwav(a, g.n), ky = kwav(b, g.n);
    const long long k2 = kx * kx + ky * ky + (long long)kz * kz;
    long long K = (long long)floor(sqrt((double)k2));
    while (K * K > k2) --K;
    while ((K + 1) * (K + 1) <= k2) ++K;
    if (k2 >= K * K + K + 1) ++K;
    const float sc = K <= kmax ? (float)s[K] : 0.f;
    const long long idx = ((long long)a * g.n + b) * g.h1 + kz;
    for (int f = 0; f < 3; ++f) u[idx + f * g.M] = cscale(u[idx + f * g.M], sc);
  }
}

}  // namespace fftk

extern "C" fftk_status tarang_ic_random(fftk_plan p, const float* normals, void* uhat, double k0,
                                        double E0, void* cuda_stream) {
  if (!p || !normals || !uhat || !(k0 > 0.0) || !(E0 > 0.0) || !std::isfinite(k0) ||
      !std::isfinite(E0))
    return FFTK_ERR_INVALID_ARG;
  if (p->nx != p->ny || p->nx != p->nz || !ns_size_ok(p->nx)) return FFTK_ERR_UNSUPPORTED_SIZE;
  fftk_status s = ns_ensure(p);
  if (s != FFTK_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  NSWork* w = p->ns;
  const NSGeom g = w->g;
  float2* u = static_cast<float2*>(uhat);
  s = fftk_r2c(p, normals, uhat, 3, cuda_stream);
  if (s != FFTK_OK) return s;
  {
    LaunchScope ls(p, KK_AUX, st);
    k_ic_shape<<<152 * 8, 256, 0, st>>>(u, g);
  }
  {
    LaunchScope ls(p, KK_AUX, st);
    k_ic_herm<<<152 * 4, 256, 0, st>>>(u, g);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return from_cuda(e);
  const int kmax = w->kmax;
  std::vector<double> d((size_t)(2 + kmax + 1));
  s = tarang_diag(p, uhat, 0.0, d.data(), cuda_stream);
  if (s != FFTK_OK) return s;
  // per-shell factors so that E(K) ~ K^4 exp(-2 (K/k0)^2), then total E0
  std::vector<double> sc((size_t)kmax + 1, 0.0);
  double tsum = 0.0;
  for (int K = 1; K <= kmax; ++K) {
    const double eK = d[(size_t)(2 + K)];
    if (eK > 0.0) {
      const double t = std::pow((double)K, 4.0) * std::exp(-2.0 * ((double)K / k0) * ((double)K / k0));
      sc[(size_t)K] = std::sqrt(t / eK);
      tsum += t;
    }
  }
  if (!(tsum > 0.0)) return FFTK_ERR_NONFINITE;
  const double gscale = std::sqrt(E0 / tsum);
  for (auto& v : sc) v *= gscale;
  double* dsc = nullptr;
  e = cudaMalloc(&dsc, sizeof(double) * sc.size());
  if (e == cudaSuccess) e = cudaMemcpy(dsc, sc.data(), sizeof(double) * sc.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    LaunchScope ls(p, KK_AUX, st);
    k_ic_rescale<<<152 * 8, 256, 0, st>>>(u, g, dsc, kmax);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (dsc) cudaFree(dsc);
  return from_cuda(e);
}

// Dealias and project a caller's state (Eq. (8) and the 2/3 rule): the entry
// point that turns any transformed velocity, e.g. a filtered resolved field on
// a coarse grid, into a valid solver state.
extern "C" fftk_status tarang_dealias_project(fftk_plan p, void* uhat, void* cuda_stream) {
  if (!p || !uhat || misaligned16(uhat)) return FFTK_ERR_INVALID_ARG;
  if (p->nx != p->ny || p->nx != p->nz || !ns_size_ok(p->nx)) return FFTK_ERR_UNSUPPORTED_SIZE;
  fftk_status s = ns_ensure(p);
  if (s != FFTK_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  {
    LaunchScope ls(p, KK_AUX, st);
    k_ic_shape<<<152 * 8, 256, 0, st>>>(static_cast<float2*>(uhat), p->ns->g);
  }
  return from_cuda(cudaGetLastError());
}
