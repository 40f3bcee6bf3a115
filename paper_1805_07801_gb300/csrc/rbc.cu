// Rayleigh-Benard convection through the plan's transforms: the periodic
// cube (FFF basis) and free-slip, isothermal plates (SFF basis).
#include <cmath>
#include <mutex>
#include <new>
#include <vector>

#include "rbc_passes.cuh"

// ------------------------------------------------ Rayleigh-Benard (FFF) ---
// Sec. 2.2, Eqs. (12)-(13), non-dimensional, on the 2 pi-periodic cube with
// gravity along z; state float2 [4][n][n][n/2+1] = (u_x, u_y, u_z, theta).
//   N_u = P[F(u x omega) + theta z],   N_theta = -i k . F(u theta) + u_z,
// evaluated with seven inverse transforms (u, omega, theta) and six forward
// ones (u x omega, u theta) per right-hand side, 13 per stage and 52 per RK4
// step as counted in the paper's Sec. 7: x and y passes restricted to the
// 2/3 set (fft_pruned.cu, fft_sc.cu) and one fused z pass per stage that
// forms the products in registers.
namespace fftk {

struct RBCWork {
  float2* w7 = nullptr;   // 7 spectra (rows of ns_row): u, omega, theta; then n (u x omega), u theta, in place
  float2* s1 = nullptr;   // stage state (4 fields)
  float2* acc = nullptr;  // RK4 accumulator (4 fields)
  float2* tab = nullptr;  // integrating factors, hi + lo by integer k^2: E_nu, E_kappa, H_nu, H_kappa
  int tab_len = 0;
  double Ra = -1.0, Pr = -1.0, dt = -1.0;
};

void rbc_free(RBCWork* r) {
  if (!r) return;
  cudaFree(r->w7);
  cudaFree(r->s1);
  cudaFree(r->acc);
  cudaFree(r->tab);
  delete r;
}

static fftk_status rbc_ensure(fftk_plan p) {
  fftk_status st = ns_ensure(p);
  if (st != FFTK_OK) return st;
  NSWork* s = p->ns;
  std::lock_guard<std::mutex> lk(p->mu);
  if (s->rbc) return FFTK_OK;
  RBCWork* r = new (std::nothrow) RBCWork;
  if (!r) return FFTK_ERR_OOM;
  const NSGeom g = s->g;
  const size_t fb = sizeof(float2) * (size_t)g.M;
  // |k|^2 up to 3 kd^2 on the cube, (2n-1)/3 squared + 2 kd^2 between plates
  const int kxs = (2 * g.n - 1) / 3;
  r->tab_len = kxs * kxs + 2 * g.kd * g.kd + 1;
  const size_t fw = sizeof(float2) * (size_t)g.n * g.n * (size_t)ns_row(g.n);  // padded rows
  // the periodic cube pads the rows of the stage state and of the accumulator too;
  // plates leave them at n/2 + 1 in the same arrays (a plan serves both bases, and
  // the second one may come up under stream capture, where nothing is allocated)
  const size_t fs = fw > fb ? fw : fb;
  cudaError_t e = cudaMalloc(&r->w7, 7 * fw);
  if (e == cudaSuccess) e = cudaMalloc(&r->s1, 4 * fs);
  if (e == cudaSuccess) e = cudaMemset(r->s1, 0, 4 * fs);
  if (e == cudaSuccess) e = cudaMalloc(&r->acc, 4 * fs);
  if (e == cudaSuccess) e = cudaMemset(r->acc, 0, 4 * fs);
  if (e == cudaSuccess) e = cudaMalloc(&r->tab, sizeof(float2) * 4 * (size_t)r->tab_len);
  if (e != cudaSuccess) {
    cudaGetLastError();
    rbc_free(r);
    return e == cudaErrorMemoryAllocation ? FFTK_ERR_OOM : FFTK_ERR_CUDA;
  }
  s->rbc = r;
  return FFTK_OK;
}

static fftk_status rbc_tables(fftk_plan p, double Ra, double Pr, double dt) {
  RBCWork* r = p->ns->rbc;
  if (r->Ra == Ra && r->Pr == Pr && r->dt == dt) return FFTK_OK;
  const double nu = std::sqrt(Pr / Ra), kappa = 1.0 / std::sqrt(Ra * Pr);
  const double coef[4] = {nu * dt, kappa * dt, 0.5 * nu * dt, 0.5 * kappa * dt};
  std::vector<float2> h(4 * (size_t)r->tab_len);
  for (int t = 0; t < 4; ++t)
    for (int k2 = 0; k2 < r->tab_len; ++k2) {
      const double E = std::exp(-coef[t] * (double)k2);
      const float hi = (float)E;
      h[(size_t)t * r->tab_len + k2] = make_float2(hi, (float)(E - (double)hi));
    }
  cudaError_t e = cudaMemcpy(r->tab, h.data(), sizeof(float2) * h.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return from_cuda(e);
  r->Ra = Ra;
  r->Pr = Pr;
  r->dt = dt;
  return FFTK_OK;
}

// ---- free-slip plates (SFF): wall-normal axis x on [0, pi], gravity along x.
// u_x and theta are sine series along x (storage index a is k_x = a + 1),
// u_y and u_z cosine series (index a is k_x = a); y and z Fourier.  d_x of a
// sine coefficient s_k is the cosine coefficient k s_k, d_x of a cosine
// coefficient c_k the sine coefficient -k c_k.  Kept: 3 k_x < 2n, 3|k_y| < n,
// 3 k_z < n.  A thread owns the wavenumber triple (k_x = a, k_y, k_z): the
// cosine entry at index a and the sine entry at index a - 1.

// w7 = [u_x, omega_y, omega_z, theta | u_y, u_z, omega_x]: sine group, then
// cosine group (each contiguous, for one batched transform per group)
__global__ void k_rbc_sff_prep(const float2* __restrict__ x, float2* __restrict__ w7, NSGeom g) {
  pdl_wait();
  const long long M = g.M, rowa = (long long)g.n * g.h1;  // one step of the x index
  const long long HW = ns_row(g.n), MW = (long long)g.n * g.n * HW, roww = (long long)g.n * HW;  // of w7
  // the kept modes only (the pruned inverse passes read nothing else; the
  // sine entry of k_x = a is kept with the cosine one, k_x = n never is)
  const int nx = (2 * g.n - 1) / 3 + 1;  // k_x = 0 .. nx - 1 (3 k_x < 2n)
  const long long items = (long long)nx * g.nk * g.kc;
  for (long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x; it < items;
       it += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(it % g.kc);
    const long long ab = it / g.kc;
    const int a = (int)(ab / g.nk), b = dense_to_a((int)(ab % g.nk), g.n, g.kd);
    const long long idx = ((long long)a * g.n + b) * g.h1 + c;
    const long long iw = ((long long)a * g.n + b) * HW + c;
    const int kb = kwav(b, g.n);
    const float ky = (2 * abs(kb) == g.n) ? 0.f : (float)kb, kz = (2 * c == g.n) ? 0.f : (float)c;
    const float2 uy = x[idx + M], uz = x[idx + 2 * M];
    // cosine entries at index a
    w7[iw + 4 * MW] = uy;
    w7[iw + 5 * MW] = uz;
    w7[iw + 6 * MW] = csub(mul_i(uz, ky), mul_i(uy, kz));  // omega_x = d_y u_z - d_z u_y
    // sine entries of k_x = a at index a - 1
    if (a == 0) continue;
    const long long sidx = idx - rowa;
    const float kx = (float)a;
    const float2 ux = x[sidx], th = x[sidx + 3 * M];
    const float2 uyc = uy, uzc = uz;
    w7[iw - roww] = ux;
    w7[iw - roww + MW] = cadd(mul_i(ux, kz), cscale(uzc, kx));      // omega_y = d_z u_x - d_x u_z
    w7[iw - roww + 2 * MW] = csub(cscale(uyc, -kx), mul_i(ux, ky));  // omega_z = d_x u_y - d_y u_x
    w7[iw - roww + 3 * MW] = th;
  }
}

// w7 (spectra): [(u x omega)_x, (u_y theta), (u_z theta) in sine | (u x omega)_y,
// (u x omega)_z, (u_x theta) in cosine].  v = u x omega + theta x, minus the
// gradient of the cosine pressure p = -div v / k^2; N_theta = -div(u theta) + u_x.
template <int MODE>
__global__ void k_rbc_sff_update(const float2* __restrict__ w7, const float2* x, const float2* u0, const float2* s1,
                                 float2* acc, float2* out, NSGeom g, RBCUpdate upd) {
  pdl_wait();
  const long long M = g.M, rowa = (long long)g.n * g.h1;
  const long long HW = ns_row(g.n), MW = (long long)g.n * g.n * HW, roww = (long long)g.n * HW;  // of w7
  const int nx = (2 * g.n - 1) / 3 + 1;  // the kept modes, k_z fastest
  const long long items = (long long)nx * g.nk * g.kc;
  for (long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x; it < items;
       it += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(it % g.kc);
    const long long ab = it / g.kc;
    const int a = (int)(ab / g.nk), b = dense_to_a((int)(ab % g.nk), g.n, g.kd);
    const long long idx = ((long long)a * g.n + b) * g.h1 + c;
    const long long iw = ((long long)a * g.n + b) * HW + c, sw = iw - roww;
    const int ky = kwav(b, g.n), kz = c, kx = a;
    const int k2 = kx * kx + ky * ky + kz * kz;
    const float fkx = (float)kx, fky = (float)ky, fkz = (float)kz;
    const bool has_s = a >= 1;  // the sine entry of k_x = a (index a - 1)
    const long long sidx = idx - rowa;
    // velocity
    float2 vx = make_float2(0.f, 0.f);
    if (has_s) vx = cadd(w7[sw], x[sidx + 3 * M]);  // (u x omega)_x + theta
    float2 vy = w7[iw + 3 * MW], vz = w7[iw + 4 * MW];
    // k = 0 (cosine k_x = 0, k_y = k_z = 0): a uniform flow along the plates,
    // with no pressure gradient to remove
    if (k2 != 0) {
      const float inv = 1.f / (float)k2;
      // div v = k_x v_x + i k_y v_y + i k_z v_z (cosine); p = -div / k^2
      const float2 dv = make_float2(fkx * vx.x - fky * vy.y - fkz * vz.y, fkx * vx.y + fky * vy.x + fkz * vz.x);
      const float2 pc = make_float2(-dv.x * inv, -dv.y * inv);
      vy = csub(vy, mul_i(pc, fky));
      vz = csub(vz, mul_i(pc, fkz));
      vx = cadd(vx, cscale(pc, fkx));
    }
    float2 nt = make_float2(0.f, 0.f);
    if (has_s) {
      // -(d_x (u_x theta) + d_y (u_y theta) + d_z (u_z theta)) + u_x
      const float2 cx = w7[iw + 5 * MW], sy = w7[sw + MW], sz = w7[sw + 2 * MW];
      const float2 ux = x[sidx];
      const float2 d = csub(cadd(mul_i(sy, fky), mul_i(sz, fkz)), cscale(cx, fkx));
      nt = cadd(make_float2(-d.x, -d.y), ux);
    }
    // entry e of one field, its factors at offset t of each pair
    auto update = [&](long long e, float2 n, int t) {
      const float2 z = make_float2(0.f, 0.f);
      const float2 a = MODE != NS_RHS && MODE != NS_RK4_4 ? u0[e] : z;
      const float2 b = MODE == NS_STAGE2 ? s1[e] : (MODE >= NS_RK4_2 ? acc[e] : z);
      const float2 E = MODE != NS_RHS && MODE != NS_RK4_4 ? __ldg(&upd.tab[t * upd.tab_len + k2]) : z;
      const float2 H = MODE >= NS_RK4_1 && MODE != NS_RK4_4 ? __ldg(&upd.tab[(2 + t) * upd.tab_len + k2]) : z;
      rbc_entry_store<MODE>(e, e, n, a, b, E, H, upd.dt, acc, out);
    };
    update(idx + M, vy, 0);
    update(idx + 2 * M, vz, 0);
    if (has_s) {
      update(sidx, vx, 0);
      update(sidx + 3 * M, nt, 1);
    }
  }
}

// One right-hand side of the stage input x and the update of `mode`.
// Periodic cube: four fused kernels and two y passes as in the Navier-Stokes
// solver (inverse x with the curl, y, z with the products, y, forward x with
// projection and update).  Plates: the sine and cosine series couple k_x = a
// and a - 1 between fields, so the spectral preparation and the update are
// kernels of their own around the sine/cosine x passes.
static cudaError_t rbc_stage(fftk_plan p, const float2* x, const float2* u0, float2* out, const RBCUpdate& upd,
                             int mode, int basis, cudaStream_t st) {
  NSWork* s = p->ns;
  RBCWork* r = s->rbc;
  const NSGeom g = s->g;
  const float scale = (float)(1.0 / ((double)g.n * g.n * g.n));
  float2* w = r->w7;
  cudaError_t e = cudaSuccess;
  if (basis == TARANG_RBC_SFF) {
    const unsigned grid = 152 * 8;
    const long long mw = (long long)g.n * g.n * ns_row(g.n);
    // w7 = [u_x, omega_y, omega_z, theta | u_y, u_z, omega_x]: sine group, cosine group
    {
      LaunchScope ls(p, KK_RBC_PREP, st);
      launch_pdl(k_rbc_sff_prep, grid, 256, 0, st, x, w, g);
    }
    e = launch_scpass_pruned(p, true, +1, w, w, 4, 1.f, st);
    if (e == cudaSuccess) e = launch_scpass_pruned(p, false, +1, w + 4 * mw, w + 4 * mw, 3, 1.f, st);
    if (e == cudaSuccess) e = ns_ypass(p, w, w, 7, +1, KK_Y_INV, st);
    // products: [(u x omega)_x, u_y theta, u_z theta | (u x omega)_y, (u x omega)_z, u_x theta]
    const RBCSlots sl{{0, 4, 5, 6, 1, 2, 3}, {0, 3, 4, 5, 1, 2}};
    if (e == cudaSuccess) e = rbc_z(p, w, sl, st);
    if (e == cudaSuccess) e = ns_ypass(p, w, w, 6, -1, KK_Y_FWD, st);
    if (e == cudaSuccess) e = launch_scpass_pruned(p, true, -1, w, w, 3, scale, st);
    if (e == cudaSuccess) e = launch_scpass_pruned(p, false, -1, w + 3 * mw, w + 3 * mw, 3, scale, st);
    if (e != cudaSuccess) return e;
    {
      LaunchScope ls(p, KK_RBC_UPDATE, st);
      switch (mode) {
#define MODE(m)                                                                                            \
  case m:                                                                                                  \
    launch_pdl(k_rbc_sff_update<m>, grid, 256, 0, st, w, x, u0, r->s1, r->acc, out, g, upd);               \
    break;
        MODE(NS_RHS) MODE(NS_STAGE1) MODE(NS_STAGE2) MODE(NS_RK4_1) MODE(NS_RK4_2) MODE(NS_RK4_3) MODE(NS_RK4_4)
#undef MODE
        default:
          return cudaErrorInvalidValue;
      }
    }
    return cudaGetLastError();
  }
  // w7 = [u_x, u_y, u_z, omega_x, omega_y, omega_z, theta] -> [n_x, n_y, n_z, u_x theta, ...]
  e = rbc_invx(p, x, x == r->s1, w, st);
  if (e == cudaSuccess) e = ns_ypass(p, w, w, 7, +1, KK_Y_INV, st);
  const RBCSlots sl{{0, 1, 2, 3, 4, 5, 6}, {0, 1, 2, 3, 4, 5}};
  if (e == cudaSuccess) e = rbc_z(p, w, sl, st);
  if (e == cudaSuccess) e = ns_ypass(p, w, w, 6, -1, KK_Y_FWD, st);
  if (e != cudaSuccess) return e;
  return rbc_fwdx(p, RBCStage{w, x, u0, r->s1, r->acc, out, upd, mode, scale}, st);
}

// Cubes as for the Navier-Stokes solver (powers of two in [8, 1024], 3 * 2^m
// in [12, 768]); the plates (SFF) need power-of-two axes for their sine and
// cosine transforms.
static fftk_status rbc_check(fftk_plan p, const void* state, int basis = TARANG_RBC_FFF) {
  if (!p || !state || misaligned16(state)) return FFTK_ERR_INVALID_ARG;
  if (p->nx != p->ny || p->nx != p->nz) return FFTK_ERR_UNSUPPORTED_SIZE;
  if (!ns_size_ok(p->nx)) return FFTK_ERR_UNSUPPORTED_SIZE;
  if (basis == TARANG_RBC_SFF && !is_pow2(p->nx)) return FFTK_ERR_UNSUPPORTED_SIZE;
  return FFTK_OK;
}

}  // namespace fftk

using namespace fftk;

extern "C" fftk_status tarang_rbc_rhs(fftk_plan p, int basis, const void* state, void* out, void* cuda_stream) {
  if (basis != TARANG_RBC_FFF && basis != TARANG_RBC_SFF) return FFTK_ERR_INVALID_ARG;
  fftk_status s = rbc_check(p, state, basis);
  if (s != FFTK_OK) return s;
  if (!out || out == state || misaligned16(out)) return FFTK_ERR_INVALID_ARG;
  s = rbc_ensure(p);
  if (s != FFTK_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const NSGeom g = p->ns->g;
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(float2) * 4 * (size_t)g.M, st);
  RBCUpdate upd{p->ns->rbc->tab, p->ns->rbc->tab_len, 0.f};
  if (e == cudaSuccess)
    e = rbc_stage(p, static_cast<const float2*>(state), static_cast<const float2*>(state),
                  static_cast<float2*>(out), upd, NS_RHS, basis, st);
  return from_cuda(e);
}

extern "C" fftk_status tarang_rbc_step(fftk_plan p, void* state, const tarang_rbc_params* prm, int nsteps,
                                       void* cuda_stream) {
  fftk_status s = rbc_check(p, state, prm ? prm->basis : TARANG_RBC_FFF);
  if (s != FFTK_OK) return s;
  if (!prm || nsteps < 0 || !(prm->Ra > 0.0) || !(prm->Pr > 0.0) || !(prm->dt > 0.0) || !std::isfinite(prm->Ra) ||
      !std::isfinite(prm->Pr) || !std::isfinite(prm->dt) || (prm->scheme != TARANG_RK2 && prm->scheme != TARANG_RK4) ||
      (prm->basis != TARANG_RBC_FFF && prm->basis != TARANG_RBC_SFF))
    return FFTK_ERR_INVALID_ARG;
  s = rbc_ensure(p);
  if (s != FFTK_OK) return s;
  s = rbc_tables(p, prm->Ra, prm->Pr, prm->dt);
  if (s != FFTK_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  RBCWork* r = p->ns->rbc;
  float2* u = static_cast<float2*>(state);
  const RBCUpdate upd{r->tab, r->tab_len, (float)prm->dt};
  cudaError_t e = cudaSuccess;
  for (int it = 0; it < nsteps && e == cudaSuccess; ++it) {
    if (prm->scheme == TARANG_RK2) {
      e = rbc_stage(p, u, u, r->s1, upd, NS_STAGE1, prm->basis, st);
      if (e == cudaSuccess) e = rbc_stage(p, r->s1, u, u, upd, NS_STAGE2, prm->basis, st);
    } else {
      for (int stage = 0; stage < 4 && e == cudaSuccess; ++stage)
        e = rbc_stage(p, stage == 0 ? u : r->s1, u, stage == 3 ? u : r->s1, upd, NS_RK4_1 + stage, prm->basis,
                      st);
    }
  }
  return from_cuda(e);
}

// Kinetic and thermal energy transfer of the periodic convection (the flux
// computation of the paper's Sec. 7, Pi_u(k) and Pi_theta(k)): with N the
// right-hand side of tarang_rbc_rhs,
//   T_u(K) = sum_shell w Re(conj(u) . N_u) - sum_shell w Re(conj(u_z) theta),
//   T_theta(K) = sum_shell w Re(conj(theta) N_theta) - sum_shell w Re(conj(theta) u_z)
// (the buoyancy and conduction-source exchanges removed, advection left),
// Pi(K) = -sum_{K' <= K} T(K').
extern "C" fftk_status tarang_rbc_transfer(fftk_plan p, const void* state, double* out_host, void* cuda_stream) {
  fftk_status s = rbc_check(p, state);
  if (s != FFTK_OK) return s;
  if (!out_host) return FFTK_ERR_INVALID_ARG;
  s = rbc_ensure(p);
  if (s != FFTK_OK) return s;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  NSWork* w = p->ns;
  RBCWork* r = w->rbc;
  const NSGeom g = w->g;
  const float2* x = static_cast<const float2*>(state);
  float2* nh = r->acc;  // free between steps
  const RBCUpdate upd{r->tab, r->tab_len, 0.f};
  cudaError_t e = rbc_stage(p, x, x, nh, upd, NS_RHS, TARANG_RBC_FFF, st);
  const int nb = w->kmax + 1, width = 2 + nb;
  // three reductions: u . N_u (3 components), u_z theta, theta N_theta
  const float2* ua[3] = {x, x + 2 * g.M, x + 3 * g.M};
  const float2* na[3] = {nh, x + 3 * g.M, nh + 3 * g.M};
  const int nfs[3] = {3, 1, 1};
  std::vector<double> h(3 * (size_t)width);
  for (int q = 0; q < 3 && e == cudaSuccess; ++q) {
    e = diag_launch(p, ua[q], na[q], 0.0, st, nfs[q]);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(h.data() + (size_t)q * width, w->dout, sizeof(double) * width, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  if (e != cudaSuccess) return from_cuda(e);
  // out: sum T_u, T_u(0..kmax), Pi_u(0..kmax), sum T_theta, T_theta(...), Pi_theta(...)
  bool finite = true;
  for (int fld = 0; fld < 2; ++fld) {
    double* o = out_host + (size_t)fld * (1 + 2 * nb);
    const double* adv = h.data() + (size_t)(fld == 0 ? 0 : 2) * width;
    const double* buoy = h.data() + (size_t)width;
    double pi = 0.0, tot = 0.0;
    for (int K = 0; K < nb; ++K) {
      const double t = adv[2 + K] - buoy[2 + K];
      o[1 + K] = t;
      pi -= t;
      o[1 + nb + K] = pi;
      tot += t;
    }
    o[0] = tot;
    finite = finite && std::isfinite(tot);
  }
  return finite ? FFTK_OK : FFTK_ERR_NONFINITE;
}
