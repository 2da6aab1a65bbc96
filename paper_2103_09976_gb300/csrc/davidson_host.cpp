// Host control of the device Davidson solver (FP64 vectors on the device).
//
// Appendix A names the Davidson method for the solving step (Eq. eff-eigsh);
// the steps follow E. R. Davidson (J. Comput. Phys. 17, 87 (1975)) with the
// choices stated in include/dmrg.h: diagonal preconditioner clamped at 1e-8,
// classical Gram-Schmidt applied twice, thick restart from the two lowest
// Ritz vectors, convergence when the squared residual norm is below tol.
#include <cmath>
#include <cstring>

#include "context.h"

namespace dmrg {

namespace {

constexpr uint64_t KEY_GUESS = 0x4755455353505349ull;  // "GUESSPSI" stream of the seed
constexpr int LDH = 32;                                // leading dimension of the projected matrix

}  // namespace

// Davidson buffers of a problem and the diagonal of H_eff (built once).
void ensure_davidson_workspace(Context& c, Problem& p) {
  const int S = c.opts.dav_max_space;
  if (p.dav_ready && p.dav_space == S) return;
  const long long n = p.psi_size;
  cudaStream_t st = c.stream;
  p.dav_V.alloc((size_t)S * n * sizeof(double));
  p.dav_AV.alloc((size_t)S * n * sizeof(double));
  p.dav_diag.alloc(n * sizeof(double));
  p.dav_x.alloc(n * sizeof(double));
  p.dav_ax.alloc(n * sizeof(double));
  p.dav_r.alloc(n * sizeof(double));
  p.dav_t.alloc(n * sizeof(double));
  p.dav_x2.alloc(n * sizeof(double));
  p.dav_partial.alloc((size_t)DAV_MAX_BLOCKS * DAV_PSTRIDE * sizeof(double));
  p.dav_cnt.alloc(16);
  DMRG_CUDA(cudaMemsetAsync(p.dav_cnt.p, 0, 16, st));
  p.dav_H.alloc(LDH * LDH * sizeof(double));
  p.dav_w.alloc(LDH * sizeof(double));
  p.dav_Y.alloc(LDH * LDH * sizeof(double));
  p.dav_Yf.alloc(32 * 32 * sizeof(float));
  p.dav_s.alloc(128 * sizeof(double));
  // diagonal of H_eff: the tasks whose output block is their input block
  std::vector<int> dstart(p.blocks.size() + 1, 0), dtask;
  for (size_t b = 0; b < p.blocks.size(); ++b) {
    for (int t = p.wl.out_start[b]; t < p.wl.out_start[b + 1]; ++t)
      if (p.wl.tasks[t].in_blk == (int)b) dtask.push_back(t);
    dstart[b + 1] = (int)dtask.size();
  }
  if (dtask.empty()) dtask.push_back(0);
  p.d_dstart.upload(dstart, st);
  p.d_dtask.upload(dtask, st);
  {
    ProfScope ps(c.prof, 2, st);
    launch_heff_diag(p.store.as<double>(), p.d_tasks.as<Task>(), p.d_dstart.as<int>(), p.d_dtask.as<int>(),
                     p.d_blocks.as<PsiBlock>(), (int)p.blocks.size(), p.dav_diag.as<double>(), st);
  }
  DMRG_CUDA(cudaGetLastError());
  DMRG_CUDA(cudaStreamSynchronize(st));
  p.dav_space = S;
  p.dav_ready = true;
}

bool run_davidson(Context& c, Problem& p, const double* x0, double tol, double* energy, double* x_out,
                  int* iters, unsigned long long guess_counter_base) {
  ensure_davidson_workspace(c, p);
  const long long n = p.psi_size;
  const int S = c.opts.dav_max_space;
  const int max_iter = c.opts.dav_max_iter;
  cudaStream_t st = c.stream;
  double* V = p.dav_V.as<double>();
  double* AV = p.dav_AV.as<double>();
  double* H = p.dav_H.as<double>();
  double* w = p.dav_w.as<double>();
  double* Y = p.dav_Y.as<double>();
  // s[0..31], s[64..95]: Gram-Schmidt coefficients, s[40]: |r|^2, s[41]: theta, s[42]: |new direction|^2,
  // s[43], s[44]: Rayleigh quotient
  double* s = p.dav_s.as<double>();
  const DavScratch part = p.dav_scratch();
  double* xb[2] = {p.dav_x.as<double>(), p.dav_x2.as<double>()};  // this Ritz vector and the one before
  int cur = 0;
  double* x = xb[0];
  double* ax = p.dav_ax.as<double>();
  double* r = p.dav_r.as<double>();
  double* t = p.dav_t.as<double>();
  float* Yf = p.dav_Yf.as<float>();
  const double* diag = p.dav_diag.as<double>();
  auto row = [&](double* M, int i) { return M + (long long)i * n; };
  double host[4];
  struct Event {
    cudaEvent_t e = nullptr;
    Event() { DMRG_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming)); }
    ~Event() { cudaEventDestroy(e); }
  } ready;

  auto sigma = [&](const double* in, double* out) { run_sigma(c, p, in, out); };
  double* const pinned = c.h_scalars.get();
  double* const got = pinned ? pinned : host;
  // projected-matrix entries of the newest vector j: H[i][j] = V_i . AV_j, H[j][i] = V_j . AV_i
  auto update_H = [&](int k) {
    const int j = k - 1;
    dav_dots2(V, row(AV, j), H + j, LDH, AV, row(V, j), H + (long long)j * LDH, 1, n, k, n, part, st);
  };
  // row k of V <- t made orthogonal to the k vectors before it (classical Gram-Schmidt twice, the first products
  // V_i . t in s already) and normalised; zero if nothing of norm 1e-14 is left
  constexpr double VANISHED = 1e-14;
  auto extend = [&](int k) {
    double* vk = row(V, k);
    dav_project_dots(V, n, k, s, t, vk, n, part, s + 64, st);
    dav_project_norm(V, n, k, s + 64, vk, vk, n, part, s + 42, st);
    dav_scale(vk, s + 42, VANISHED, n, st);
  };

  ProfScope prof_all(c.prof, 2, st);
  // initial vector, normalised
  if (x0)
    DMRG_CUDA(cudaMemcpyAsync(row(V, 0), x0, n * sizeof(double), cudaMemcpyDeviceToDevice, st));
  else
    launch_gen_vector(row(V, 0), n, (uint64_t)(c.opts.seed ^ KEY_GUESS), guess_counter_base, st);
  dav_dots(V, n, 1, row(V, 0), n, part, s + 42, 1, st);
  dav_scale(row(V, 0), s + 42, 0.0, n, st);
  sigma(row(V, 0), row(AV, 0));
  int k = 1, nmv = 1;
  update_H(k);
  bool converged = false;
  bool extended = false;  // V's newest row comes from extend(); its norm is read with the next residual
  double theta = 0.0, theta_before = 0.0;
  int warm = 0;           // size of the projected matrix whose vectors Yf holds
  for (;;) {
    const bool full = k >= S;  // the restart needs two Ritz vectors
    if (full)
      dav_eigh(H, k, LDH, w, Y, st);
    else
      dav_eigh_lowest(H, k, LDH, w, Y, Yf, warm, st);
    warm = full ? 0 : k;
    x = xb[cur];
    dav_ritz(V, AV, n, k, Y, LDH, w, diag, x, ax, t, n, part, s, s + 40, st);
    DMRG_CUDA(cudaMemcpyAsync(got, s + 40, 3 * sizeof(double), cudaMemcpyDeviceToHost, st));
    DMRG_CUDA(cudaEventRecord(ready.e, st));
    // the next direction is prepared while the host waits for the residual
    // (unused if this was the last iteration)
    if (!full && nmv < max_iter) extend(k);
    DMRG_CUDA(cudaEventSynchronize(ready.e));
    const double rr = got[0];
    if (extended && std::sqrt(got[2]) < VANISHED) {  // the newest direction was rounding noise: the result without it
      --nmv;
      x = xb[cur ^ 1];
      theta = theta_before;
      break;
    }
    theta = got[1];
    if (!(rr == rr)) throw Error(DMRG_ECUDA, "Davidson: residual is not a number");
    if (rr < tol) {
      converged = true;
      break;
    }
    if (nmv >= max_iter) break;
    if (full) {  // thick restart from the two lowest Ritz vectors
      dav_lincomb(V, n, k, Y + 1, LDH, 1.0, r, n, false, st);   // r <- second Ritz vector
      DMRG_CUDA(cudaMemcpyAsync(row(V, 0), x, n * sizeof(double), cudaMemcpyDeviceToDevice, st));
      DMRG_CUDA(cudaMemcpyAsync(row(V, 1), r, n * sizeof(double), cudaMemcpyDeviceToDevice, st));
      dav_lincomb(AV, n, k, Y + 1, LDH, 1.0, r, n, false, st);  // r <- H times it
      DMRG_CUDA(cudaMemcpyAsync(row(AV, 0), ax, n * sizeof(double), cudaMemcpyDeviceToDevice, st));
      DMRG_CUDA(cudaMemcpyAsync(row(AV, 1), r, n * sizeof(double), cudaMemcpyDeviceToDevice, st));
      k = 2;
      update_H(1);
      update_H(2);
      dav_dots(V, n, k, t, n, part, s, 1, st);  // V changed: first Gram-Schmidt products again
      extend(k);
    }
    sigma(row(V, k), row(AV, k));
    ++nmv;
    ++k;
    update_H(k);
    extended = true;
    theta_before = theta;
    cur ^= 1;
  }
  if (c.opts.sigma_prec != DMRG_FP64) {
    // The mixed-precision operator differs from H by a relative 1e-5 or so,
    // which moves its eigenvalue at first order. The Rayleigh quotient of
    // the final vector with the FP64 sigma is off only at second order in
    // the vector's error, so it is the energy returned.
    run_sigma_f64(c, p, x, ax);
    dav_dots2(x, ax, s + 43, 1, x, x, s + 44, 1, n, 1, n, part, st);
    DMRG_CUDA(cudaMemcpyAsync(got, s + 43, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
    DMRG_CUDA(cudaStreamSynchronize(st));
    theta = got[0] / got[1];
  }
  if (x_out) DMRG_CUDA(cudaMemcpyAsync(x_out, x, n * sizeof(double), cudaMemcpyDeviceToDevice, st));
  DMRG_CUDA(cudaStreamSynchronize(st));
  check_device_error(c, p);
  *energy = theta;
  *iters = nmv;
  return converged;
}

}  // namespace dmrg
