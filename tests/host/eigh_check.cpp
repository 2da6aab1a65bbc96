// Projected eigenproblem of the Davidson solver, direct.
//   eigh_check <constant> <gap>
// H (32 x 32) has the values 0, gap and others in [0.5, 8] plus the constant;
// its leading k x k blocks, k = 1 .. 32, go through dav_eigh_lowest, each
// started from the vectors of the one before, as the solver does. Prints per k
// "k value resid norm orth": errors of the lowest value (against Jacobi in long
// double) and of the residual over |H - constant|_F, | |y| - 1 |, and max
// |Q^T Q - 1| of the FP32 vectors kept for the next call. Then "time lowest full":
// us of a call on all of H by dav_eigh_lowest and by dav_eigh, neither warm.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "kernels.h"

using namespace dmrg;
typedef long double ld;

#define CK(x) do { if ((x) != cudaSuccess) { fprintf(stderr, "cuda: %s\n", cudaGetErrorString(cudaGetLastError())); return 1; } } while (0)

constexpr int N = 32;

// values of the symmetric k x k matrix a (destroyed), cyclic Jacobi; lowest one
static ld lowest(std::vector<ld> a, int k) {
  for (int sweep = 0; sweep < 60; ++sweep) {
    ld off = 0, tot = 0;
    for (int i = 0; i < k; ++i)
      for (int j = 0; j < k; ++j) (i == j ? tot : off) += a[i * k + j] * a[i * k + j];
    if (off <= 1e-37L * (tot + off)) break;
    for (int p = 0; p < k; ++p)
      for (int q = p + 1; q < k; ++q) {
        if (a[p * k + q] == 0) continue;
        const ld z = (a[q * k + q] - a[p * k + p]) / (2 * a[p * k + q]);
        const ld t = (z >= 0 ? 1 : -1) / (std::fabs(z) + std::sqrt(z * z + 1)), c = 1 / std::sqrt(t * t + 1), s = t * c;
        for (int r = 0; r < k; ++r) {
          const ld x = a[r * k + p], y = a[r * k + q];
          a[r * k + p] = c * x - s * y, a[r * k + q] = s * x + c * y;
        }
        for (int r = 0; r < k; ++r) {
          const ld x = a[p * k + r], y = a[q * k + r];
          a[p * k + r] = c * x - s * y, a[q * k + r] = s * x + c * y;
        }
      }
  }
  ld v = a[0];
  for (int i = 1; i < k; ++i) v = std::min(v, a[i * k + i]);
  return v;
}

int main(int, char** argv) {
  const double cst = atof(argv[1]), gap = atof(argv[2]);
  std::mt19937_64 gen(5);
  std::normal_distribution<double> nd;
  std::uniform_real_distribution<double> ud(0.5, 8.0);
  std::vector<ld> U(N * N), lam(N);
  for (int i = 0; i < N; ++i) {
    lam[i] = i == 0 ? 0.0L : i == 1 ? (ld)gap : (ld)ud(gen);
    for (int j = 0; j < N; ++j) U[i * N + j] = nd(gen);
    for (int pass = 0; pass < 2; ++pass)
      for (int q = 0; q < i; ++q) {
        ld d = 0;
        for (int j = 0; j < N; ++j) d += U[i * N + j] * U[q * N + j];
        for (int j = 0; j < N; ++j) U[i * N + j] -= d * U[q * N + j];
      }
    ld n = 0;
    for (int j = 0; j < N; ++j) n += U[i * N + j] * U[i * N + j];
    for (int j = 0; j < N; ++j) U[i * N + j] /= std::sqrt(n);
  }
  std::vector<double> H(N * N);
  for (int i = 0; i < N; ++i)
    for (int j = 0; j <= i; ++j) {
      ld s = i == j ? (ld)cst : 0.0L;
      for (int q = 0; q < N; ++q) s += lam[q] * U[q * N + i] * U[q * N + j];
      H[i * N + j] = H[j * N + i] = (double)s;
    }
  double *dH, *dw, *dY;
  float* dYf;
  CK(cudaMalloc(&dH, N * N * 8));
  CK(cudaMalloc(&dw, N * 8));
  CK(cudaMalloc(&dY, N * N * 8));
  CK(cudaMalloc(&dYf, N * N * 4));
  CK(cudaMemcpy(dH, H.data(), N * N * 8, cudaMemcpyHostToDevice));
  std::vector<double> w(N), Y(N * N);
  std::vector<float> Yf(N * N);
  for (int k = 1; k <= N; ++k) {
    dav_eigh_lowest(dH, k, N, dw, dY, dYf, k - 1, 0);
    CK(cudaGetLastError());
    CK(cudaDeviceSynchronize());
    CK(cudaMemcpy(w.data(), dw, N * 8, cudaMemcpyDeviceToHost));
    CK(cudaMemcpy(Y.data(), dY, N * N * 8, cudaMemcpyDeviceToHost));
    CK(cudaMemcpy(Yf.data(), dYf, N * N * 4, cudaMemcpyDeviceToHost));
    std::vector<ld> a(k * k);
    ld fro = 0, nn = 0, rr = 0, orth = 0;
    for (int i = 0; i < k; ++i)
      for (int j = 0; j < k; ++j) {
        a[i * k + j] = (ld)H[i * N + j] - (i == j ? (ld)cst : 0.0L);
        fro += a[i * k + j] * a[i * k + j];
      }
    fro = std::sqrt(fro);
    const ld theta = (ld)w[0] - (ld)cst;
    for (int i = 0; i < k; ++i) {
      ld r = -theta * (ld)Y[i * N];
      for (int j = 0; j < k; ++j) r += a[i * k + j] * (ld)Y[j * N];
      rr += r * r;
      nn += (ld)Y[i * N] * (ld)Y[i * N];
      for (int j = 0; j < k; ++j) {
        ld d = i == j ? -1 : 0;
        for (int q = 0; q < k; ++q) d += (ld)Yf[q * N + i] * (ld)Yf[q * N + j];
        orth = std::max(orth, std::fabs(d));
      }
    }
    printf("%d %.3Le %.3Le %.3Le %.3Le\n", k, std::fabs(theta - lowest(a, k)) / fro, std::sqrt(rr) / fro,
           std::fabs(std::sqrt(nn) - 1), orth);
  }
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  float ms[2];
  for (int full = 0; full < 2; ++full) {
    for (int rep = 0; rep < 25; ++rep) {
      if (rep == 5) CK(cudaEventRecord(e0));
      if (full) dav_eigh(dH, N, N, dw, dY, 0);
      else dav_eigh_lowest(dH, N, N, dw, dY, dYf, 0, 0);
    }
    CK(cudaEventRecord(e1));
    CK(cudaEventSynchronize(e1));
    CK(cudaEventElapsedTime(&ms[full], e0, e1));
  }
  printf("time %.2f %.2f\n", ms[0] * 50, ms[1] * 50);
  return 0;
}
