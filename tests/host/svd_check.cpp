// Decimation SVD, direct: blocks of the given sizes through the kernels the
// size rule picks, and once more with every block on the grid-wide kernel.
//   svd_check <left 0|1> <spectrum: flat|graded|lowrank|zero> <d m>...
// Prints, per block, "d m cluster orth off sig": max |V^T V - 1|, the largest
// product of two columns of A V over |A|_F^2, and the largest difference of the
// two runs' singular values over |A|_F. Sums in long double.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "kernels.h"

using namespace dmrg;

#define CK(x) do { if ((x) != cudaSuccess) { fprintf(stderr, "cuda: %s\n", cudaGetErrorString(cudaGetLastError())); return 1; } } while (0)

int main(int argc, char** argv) {
  const bool left = atoi(argv[1]) != 0;
  const std::string spec = argv[2];
  std::vector<int> D, M;
  for (int i = 3; i + 1 < argc; i += 2) {
    D.push_back(atoi(argv[i]));
    M.push_back(atoi(argv[i + 1]));
  }
  const int nb = (int)D.size();
  std::mt19937_64 gen(7);
  std::normal_distribution<double> nd;
  std::vector<long long> off(nb), qoff(nb), woff(nb);
  long long no = 0, nq = 0, nw = 0;
  for (int b = 0; b < nb; ++b) {
    off[b] = no, qoff[b] = nq, woff[b] = nw;
    no += (long long)D[b] * M[b], nq += (long long)D[b] * D[b], nw += D[b];
  }
  std::vector<double> psi(no, 0.0);
  for (int b = 0; b < nb; ++b) {  // sum of scaled outer products: graded 10^-(k/4), lowrank a third of the rank
    const int d = D[b], m = M[b], r = std::min(d, m);
    const int terms = spec == "zero" ? 0 : spec == "lowrank" ? (r + 2) / 3 : r;
    for (int k = 0; k < terms; ++k) {
      const double sc = spec == "graded" ? std::pow(10.0, -0.25 * k) : 1.0;
      std::vector<double> u(d), v(m);
      for (double& x : u) x = nd(gen);
      for (double& x : v) x = nd(gen);
      for (int i = 0; i < d; ++i)
        for (int j = 0; j < m; ++j) psi[off[b] + (left ? (long long)i * m + j : (long long)j * d + i)] += sc * u[i] * v[j];
    }
  }
  double *dpsi, *dQ, *dw, *dwork;
  SvdBlock* dsb;
  int dev = 0, n_sm = 0;
  CK(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev));
  CK(cudaMalloc(&dpsi, no * 8));
  CK(cudaMalloc(&dQ, nq * 8));
  CK(cudaMalloc(&dw, nw * 8));
  CK(cudaMalloc(&dwork, (64 + no + nq) * 8));
  CK(cudaMalloc(&dsb, nb * sizeof(SvdBlock)));
  CK(cudaMemcpy(dpsi, psi.data(), no * 8, cudaMemcpyHostToDevice));
  if (!svd_clusters_launch()) {
    fprintf(stderr, "no cluster can be placed\n");
    return 1;
  }
  std::vector<SvdDims> dims(nb);
  for (int b = 0; b < nb; ++b) dims[b] = {off[b], D[b], M[b]};
  std::vector<double> W[2], Q(nq);
  std::vector<int> cls(nb);
  for (int run = 1; run >= 0; --run) {  // 1: all grid-wide, 0: as the rule picks
    std::vector<SvdBlock> sb;
    const SvdShape sh = plan_svd_blocks(dims, run == 0, sb);
    if (sh.q_elems != nq || sh.w_elems != nw || sh.work_elems != 64 + no + nq) {
      fprintf(stderr, "sizes of the plan\n");
      return 1;
    }
    for (int b = 0; b < nb; ++b) cls[b] = sb[b].cluster;
    CK(cudaMemcpy(dsb, sb.data(), nb * sizeof(SvdBlock), cudaMemcpyHostToDevice));
    launch_svd_blocks(dpsi, dsb, sh, dQ, dw, dwork, left, n_sm, 0);
    CK(cudaGetLastError());
    CK(cudaDeviceSynchronize());
    W[run].resize(nw);
    CK(cudaMemcpy(W[run].data(), dw, nw * 8, cudaMemcpyDeviceToHost));
    CK(cudaMemcpy(Q.data(), dQ, nq * 8, cudaMemcpyDeviceToHost));
  }
  for (int b = 0; b < nb; ++b) {
    const int d = D[b], m = M[b];
    auto a = [&](int i, int j) { return psi[off[b] + (left ? (long long)i * m + j : (long long)j * d + i)]; };
    auto q = [&](int r, int c) { return Q[qoff[b] + (long long)r * d + c]; };
    long double fro = 0, orth = 0, cosm = 0, sig = 0;
    for (int i = 0; i < d; ++i)
      for (int j = 0; j < m; ++j) fro += (long double)a(i, j) * a(i, j);
    for (int x = 0; x < d; ++x)
      for (int y = x; y < d; ++y) {
        long double v = x == y ? -1 : 0;
        for (int r = 0; r < d; ++r) v += (long double)q(r, x) * q(r, y);
        orth = std::max(orth, std::fabs(v));
      }
    std::vector<long double> av((size_t)d * m), n2(d, 0);  // columns of A V (A: d columns of m)
    for (int x = 0; x < d; ++x)
      for (int r = 0; r < d; ++r)
        for (int j = 0; j < m; ++j) av[(size_t)x * m + j] += (long double)q(r, x) * a(r, j);
    for (int x = 0; x < d; ++x)
      for (int j = 0; j < m; ++j) n2[x] += av[(size_t)x * m + j] * av[(size_t)x * m + j];
    for (int x = 0; x < d; ++x)
      for (int y = 0; y < x; ++y) {
        long double g = 0;
        for (int j = 0; j < m; ++j) g += av[(size_t)x * m + j] * av[(size_t)y * m + j];
        if (fro > 0) cosm = std::max(cosm, std::fabs(g) / fro);
      }
    for (int x = 0; x < d; ++x)  // w holds squared norms
      if (fro > 0)
        sig = std::max(sig, std::fabs(std::sqrt((long double)W[0][woff[b] + x]) - std::sqrt((long double)W[1][woff[b] + x])) /
                                std::sqrt(fro));
    printf("%d %d %d %.3Le %.3Le %.3Le\n", d, m, cls[b], orth, cosm, sig);
  }
  return 0;
}
