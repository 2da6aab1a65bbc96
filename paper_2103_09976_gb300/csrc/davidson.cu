// Davidson eigensolver on the device (FP64 control path).
//
// Appendix A (solving step, Eq. eff-eigsh) names the Davidson method. The
// steps here: projected matrix V^T H V, its lowest eigenpair, Ritz vector and
// residual, diagonal preconditioner clamped at 1e-8, classical Gram-Schmidt
// twice, thick restart from the two lowest Ritz vectors. Three scalars per
// iteration (Ritz value, squared residual norm, squared norm of the previous
// new direction) cross to the host. All reductions have a fixed order, so
// results are deterministic.
//
// The vectors of a solve are short (1e3 - 1e6) and the FP64 pipe takes about
// 67 cycles per warp instruction and SM sub-partition, so an iteration is
// bound by launches and by the instructions of its reductions, not by memory.
// Hence a few kernels that each do all that one pass over the subspace can
// (Ritz vector, residual, preconditioner and the first Gram-Schmidt products
// in one), sums of up to 32 products over a warp that halve the number of
// values with the number of lanes (31 additions instead of 160), and the last
// block of a grid summing the blocks' partial results instead of a second
// launch. An iteration took 28 launches and, without its sigma, 390 us at
// K=16, M=150 (224 us of them the eigenproblem, 98 us dot products); now 8
// launches and 140 us.
#include <algorithm>

#include "kernels.h"

namespace dmrg {

namespace {

constexpr int KMAX = DAV_KMAX;     // vectors per call (subspace size limit)
constexpr int DT = 128;            // threads of a vector kernel
constexpr int PSTRIDE = DAV_PSTRIDE;  // partial results per block: two sets of KMAX, or one and a scalar
static_assert(PSTRIDE >= 2 * KMAX, "two sets of partial results");

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sums of KB values per lane over the warp; returns the sum of value
// lane / (32 / KB). KB = 8, 16 or 32.
template <int KB>
__device__ __forceinline__ double warp_sums(double (&v)[KB], int lane) {
#pragma unroll
  for (int c = KB / 2, o = 16; o > 0; o >>= 1, c >>= 1) {
    if (c > 0) {  // lanes with bit o keep the upper half of the values
      const bool up = lane & o;
#pragma unroll
      for (int i = 0; i < KB / 2; ++i)
        if (i < c) {
          const double send = up ? v[i] : v[i + c], keep = up ? v[i + c] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
  return v[0];
}

// Sums over the block of v[0..KB) into row[0..KB) (global memory), and of
// `extra` into row[KMAX] when with_extra. All threads of the block call it.
template <int KB>
__device__ __forceinline__ void block_sums(double (&v)[KB], double extra, bool with_extra, double* __restrict__ row) {
  __shared__ double red[DT / 32][KB + 1];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const double s = warp_sums<KB>(v, lane);
  if (lane % (32 / KB) == 0) red[wid][lane / (32 / KB)] = s;
  if (with_extra) {
    extra = warp_sum(extra);
    if (lane == 0) red[wid][KB] = extra;
  }
  __syncthreads();
  if (threadIdx.x < KB + (with_extra ? 1 : 0)) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < DT / 32; ++w) t += red[w][threadIdx.x];
    row[threadIdx.x < KB ? threadIdx.x : KMAX] = t;
  }
}

// True in every thread of the last block of the grid (of `nblk` blocks that
// share the counter) to get here; everything the blocks wrote before is then
// visible. The counter is left at zero.
__device__ __forceinline__ bool last_block(unsigned int* counter, unsigned int nblk) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(counter, 1u) == nblk - 1;
    if (last) *counter = 0u;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// Column `lane` of the partial results, summed over the blocks in a fixed
// order (each warp every 4th block, then the warps), by all threads of the
// last block; valid in warp 0.
__device__ __forceinline__ double sum_blocks(const double* __restrict__ part, int nblk, int col) {
  __shared__ double red[DT / 32][33];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  double s = 0.0;
  __syncthreads();
#pragma unroll 4
  for (int b = wid; b < nblk; b += DT / 32) s += __ldcg(part + (long long)b * PSTRIDE + col);
  red[wid][lane] = s;
  __syncthreads();
  double t = 0.0;
  if (wid == 0)
#pragma unroll
    for (int w = 0; w < DT / 32; ++w) t += red[w][lane];
  return t;
}

// out[i * stride] = V[i] . w for i < k, one set of vectors per blockIdx.y
struct DotSet {
  const double* V;
  const double* w;
  double* out;
  int stride;
};
template <int KB>
__global__ void __launch_bounds__(DT) dots_kernel(DotSet a, DotSet b, long long ld, int k, long long n,
                                                  double* __restrict__ partial, unsigned int* __restrict__ counter) {
  const DotSet d = blockIdx.y ? b : a;
  double acc[KB];
#pragma unroll
  for (int i = 0; i < KB; ++i) acc[i] = 0.0;
  for (long long e = blockIdx.x * (long long)DT + threadIdx.x; e < n; e += (long long)gridDim.x * DT) {
    const double we = d.w[e];
#pragma unroll
    for (int i = 0; i < KB; ++i)
      if (i < k) acc[i] = fma(d.V[i * ld + e], we, acc[i]);
  }
  double* part = partial + blockIdx.y * KMAX;
  block_sums<KB>(acc, 0.0, false, part + (long long)blockIdx.x * PSTRIDE);
  if (!last_block(counter + blockIdx.y, gridDim.x)) return;
  const double s = sum_blocks(part, gridDim.x, threadIdx.x & 31);
  if (threadIdx.x < k) d.out[(long long)threadIdx.x * d.stride] = s;
}

// One pass over the subspace after the projected eigenproblem: Ritz vector
// x = sum_i y_i V_i and ax = sum_i y_i AV_i, residual r = ax - theta x,
// preconditioned direction t = r / clamp(theta - diag), r . r, and the
// products c_i = V_i . t of the first Gram-Schmidt pass. sc = {r . r, theta}.
template <int KB>
__global__ void __launch_bounds__(DT)
ritz_kernel(const double* __restrict__ V, const double* __restrict__ AV, long long ld, int k,
            const double* __restrict__ Y, int ys, const double* __restrict__ theta, const double* __restrict__ diag,
            double* __restrict__ x, double* __restrict__ ax, double* __restrict__ t, long long n,
            double* __restrict__ partial, unsigned int* __restrict__ counter, double* __restrict__ c,
            double* __restrict__ sc) {
  __shared__ double y[KMAX];
  if (threadIdx.x < KMAX) y[threadIdx.x] = threadIdx.x < k ? Y[threadIdx.x * ys] : 0.0;
  __syncthreads();
  const double th = *theta;
  double acc[KB], rr = 0.0;
#pragma unroll
  for (int i = 0; i < KB; ++i) acc[i] = 0.0;
  for (long long e = blockIdx.x * (long long)DT + threadIdx.x; e < n; e += (long long)gridDim.x * DT) {
    double v[KB], xe = 0.0, axe = 0.0;
#pragma unroll
    for (int i = 0; i < KB; ++i)
      if (i < k) {
        v[i] = V[i * ld + e];
        xe = fma(y[i], v[i], xe);
        axe = fma(y[i], AV[i * ld + e], axe);
      }
    x[e] = xe;
    ax[e] = axe;
    const double re = axe - th * xe;
    rr = fma(re, re, rr);
    double den = th - diag[e];
    if (fabs(den) < 1e-8) den = den < 0.0 ? -1e-8 : 1e-8;
    const double te = re / den;
    t[e] = te;
#pragma unroll
    for (int i = 0; i < KB; ++i)
      if (i < k) acc[i] = fma(v[i], te, acc[i]);
  }
  block_sums<KB>(acc, rr, true, partial + (long long)blockIdx.x * PSTRIDE);
  if (!last_block(counter, gridDim.x)) return;
  const int lane = threadIdx.x & 31;
  const double s = sum_blocks(partial, gridDim.x, lane);
  if (threadIdx.x < k) c[threadIdx.x] = s;
  const double q = sum_blocks(partial, gridDim.x, KMAX);
  if (threadIdx.x == 0) {
    sc[0] = q;
    sc[1] = th;
  }
}

// out = t - sum_i c_i V_i. dots: also c2_i = V_i . out (the next Gram-Schmidt
// pass); otherwise out . out into *c2.
template <int KB, bool DOTS>
__global__ void __launch_bounds__(DT)
project_kernel(const double* __restrict__ V, long long ld, int k, const double* __restrict__ c, const double* t,
               double* out, long long n, double* __restrict__ partial, unsigned int* __restrict__ counter,
               double* __restrict__ c2) {
  __shared__ double cc[KMAX];
  if (threadIdx.x < KMAX) cc[threadIdx.x] = threadIdx.x < k ? c[threadIdx.x] : 0.0;
  __syncthreads();
  double acc[KB], nn = 0.0;
#pragma unroll
  for (int i = 0; i < KB; ++i) acc[i] = 0.0;
  for (long long e = blockIdx.x * (long long)DT + threadIdx.x; e < n; e += (long long)gridDim.x * DT) {
    double v[KB], s = 0.0;
#pragma unroll
    for (int i = 0; i < KB; ++i)
      if (i < k) {
        v[i] = V[i * ld + e];
        s = fma(cc[i], v[i], s);
      }
    const double o = t[e] - s;
    out[e] = o;
    if (DOTS) {
#pragma unroll
      for (int i = 0; i < KB; ++i)
        if (i < k) acc[i] = fma(v[i], o, acc[i]);
    } else {
      nn = fma(o, o, nn);
    }
  }
  if (DOTS) {
    block_sums<KB>(acc, 0.0, false, partial + (long long)blockIdx.x * PSTRIDE);
    if (!last_block(counter, gridDim.x)) return;
    const double s = sum_blocks(partial, gridDim.x, threadIdx.x & 31);
    if (threadIdx.x < k) c2[threadIdx.x] = s;
  } else {
    double one[8] = {nn, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    block_sums<8>(one, 0.0, false, partial + (long long)blockIdx.x * PSTRIDE);
    if (!last_block(counter, gridDim.x)) return;
    const double s = sum_blocks(partial, gridDim.x, 0);
    if (threadIdx.x == 0) *c2 = s;
  }
}

// out = sum_i c[i*cs] V[i] (+ beta * out when add)
__global__ void lincomb_kernel(const double* __restrict__ V, long long ld, int k, const double* __restrict__ c,
                               int cs, double sign, double* __restrict__ out, long long n, int add) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int i = 0; i < k; ++i) s = fma(c[i * cs], V[i * ld + e], s);
    out[e] = add ? out[e] + sign * s : sign * s;
  }
}

// x <- sign(x . z) x + a z / sqrt(z . z); xz_zz = {x . z, z . z}
__global__ void axpy_unit_kernel(double* __restrict__ x, const double* __restrict__ z,
                                 const double* __restrict__ xz_zz, double a, long long n) {
  const double sg = xz_zz[0] < 0.0 ? -1.0 : 1.0;
  const double s = a / sqrt(xz_zz[1]);
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    x[e] = fma(s, z[e], sg * x[e]);
}

// x /= sqrt(*nrm2); zero when the norm is below `floor` (the host then drops it)
__global__ void scale_kernel(double* __restrict__ x, const double* __restrict__ nrm2, double floor, long long n) {
  const double nrm = sqrt(*nrm2);
  const double s = nrm < floor ? 0.0 : 1.0 / nrm;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    x[e] *= s;
}

// Eigenpairs of the symmetric k x k matrix A (shared memory; overwritten) in the
// basis Q by cyclic Jacobi in round-robin order (Brent-Luk): each
// round rotates up to 16 disjoint index pairs at once. Four warps share the
// work (the FP64 rate of one SM sub-partition would otherwise bound it):
// pair i's rotation is computed by warp i % 4, and every thread applies the
// rotations of its warp's pairs to its row (and its column). w = values + shift
// ascending, Y columns = vectors Q v (Y row-major k x ldh). k <= 32; 128 threads,
// which see A and Q (a barrier since they were written).
constexpr int EIGH_WARPS = 4;
__device__ void jacobi_eigh(double (*A)[33], double (*Q)[33], int k, int ldh, double shift, double* __restrict__ w,
                            double* __restrict__ Y) {
  __shared__ double cs[16], sn[16];
  __shared__ int pp[16], qq[16];
  __shared__ double red[2][EIGH_WARPS];
  __shared__ int stop;
  const int tid = threadIdx.x, r = tid & 31, wid = tid >> 5;
  const int kp = k + (k & 1);            // players, one dummy when k is odd
  const int npairs = kp / 2;
  for (int sweep = 0; sweep < 60 && k > 1; ++sweep) {
    double off = 0.0, tot = 0.0;
    for (int e = tid; e < k * k; e += blockDim.x) {
      const int i = e / k, c = e % k;
      const double a = A[i][c];
      tot += a * a;
      if (c != i) off += a * a;
    }
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if (r == 0) {
      red[0][wid] = off;
      red[1][wid] = tot;
    }
    __syncthreads();
    if (tid == 0) {
      double o2 = 0.0, t2 = 0.0;
      for (int j = 0; j < EIGH_WARPS; ++j) {
        o2 += red[0][j];
        t2 += red[1][j];
      }
      stop = (o2 <= 1e-30 * t2 || o2 == 0.0) ? 1 : 0;
    }
    __syncthreads();
    if (stop) break;
    for (int round = 0; round < kp - 1; ++round) {
      // pair i = r * EIGH_WARPS + wid: lane r of warp wid
      const int i = r * EIGH_WARPS + wid;
      if (r < 4 && i < npairs) {
        auto player = [&](int x) { return x == 0 ? 0 : 1 + (x - 1 + round) % (kp - 1); };
        int p = player(i), q = player(kp - 1 - i);
        if (p > q) { const int t = p; p = q; q = t; }
        double c = 1.0, sv = 0.0;
        if (q < k) {
          const double apq = A[p][q];
          if (apq != 0.0) {
            const double th = (A[q][q] - A[p][p]) / (2.0 * apq);
            const double t = (th >= 0.0 ? 1.0 : -1.0) / (fabs(th) + sqrt(th * th + 1.0));
            c = 1.0 / sqrt(t * t + 1.0);
            sv = t * c;
          }
        }
        cs[i] = c;
        sn[i] = sv;
        pp[i] = p;
        qq[i] = q < k ? q : -1;
      }
      __syncthreads();
      // columns: A <- A J, Q <- Q J (thread (r, wid): row r, pairs wid, wid + 4, ...)
      if (r < k)
        for (int j = wid; j < npairs; j += EIGH_WARPS) {
          const int q = qq[j];
          if (q < 0 || sn[j] == 0.0) continue;
          const int p = pp[j];
          const double c = cs[j], sv = sn[j];
          const double arp = A[r][p], arq = A[r][q];
          A[r][p] = c * arp - sv * arq;
          A[r][q] = sv * arp + c * arq;
          const double qp = Q[r][p], qv = Q[r][q];
          Q[r][p] = c * qp - sv * qv;
          Q[r][q] = sv * qp + c * qv;
        }
      __syncthreads();
      // rows: A <- J^T A (thread (r, wid): column r, pairs wid, wid + 4, ...)
      if (r < k)
        for (int j = wid; j < npairs; j += EIGH_WARPS) {
          const int q = qq[j];
          if (q < 0 || sn[j] == 0.0) continue;
          const int p = pp[j];
          const double c = cs[j], sv = sn[j];
          const double apc = A[p][r], aqc = A[q][r];
          A[p][r] = c * apc - sv * aqc;
          A[q][r] = sv * apc + c * aqc;
        }
      __syncthreads();
    }
  }
  // sort ascending: rank of each eigenvalue (ties by index), then scatter
  if (tid < k) {
    const double v = A[tid][tid];
    int rank = 0;
    for (int j = 0; j < k; ++j) {
      const double u = A[j][j];
      rank += (u < v) || (u == v && j < tid);
    }
    w[rank] = v + shift;
    for (int rr = 0; rr < k; ++rr) Y[rr * ldh + rank] = Q[rr][tid];
  }
}

__global__ void __launch_bounds__(32 * EIGH_WARPS)
eigh_full_kernel(const double* __restrict__ H, int k, int ldh, double* __restrict__ w, double* __restrict__ Y) {
  __shared__ double A[32][33], Q[32][33];
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) {
    const int i = e / k, c = e % k;
    A[i][c] = 0.5 * (H[i * ldh + c] + H[c * ldh + i]);
    Q[i][c] = i == c ? 1.0 : 0.0;
  }
  __syncthreads();
  jacobi_eigh(A, Q, k, ldh, 0.0, w, Y);
}

// Lowest eigenpair of the symmetric part of the k x k matrix H (k <= 32):
// w[0] and column 0 of Y. One FP64 Jacobi sweep of a 24 x 24 matrix costs 22 us
// of one SM's FP64 pipe, so the whole spectrum is found by Jacobi in FP32 (256
// times the rate; the two-sided rotation of a 2 x 2 block of pairs per thread,
// two barriers per round), warm-started from the previous call's vectors in Yf,
// and the lowest pair is then refined in FP64: with residual r = H y - theta y,
// y -= sum_i q_i (q_i . r) / (lambda_i - theta) over the other FP32
// eigenvectors, which multiplies its error by about 1e-6 per step, until |r| <=
// 1e-15 |H|_F, the bound the FP64 Jacobi stops at. Where the lowest two values are
// closer than FP32 can tell apart, or the residual does not reach it in a few
// steps, the FP64 Jacobi above decides, started from these vectors.
//
// All of it on H - H[0][0]: the scale that FP32 and the bounds see is then the
// spread of the projected spectrum, not a constant in the Hamiltonian (at -88 Ha
// any gap below 1.8 mHa used to go to the FP64 Jacobi).
// Per call at K=16, M=150: 43 us (FP64 Jacobi of the whole spectrum: 224 us).
__global__ void __launch_bounds__(32 * EIGH_WARPS)
eigh_lowest_kernel(const double* __restrict__ H, int k, int ldh, double* __restrict__ w, double* __restrict__ Y,
                   float* __restrict__ Yf, int k0) {
  __shared__ double Hs[32][33];
  __shared__ float A[32][33], Q[32][33], T[32][33];
  __shared__ float sn[16], th[16];
  __shared__ int pp[16], qq[16];
  __shared__ double part[EIGH_WARPS][32], yv[32], rv[32];
  __shared__ float coef[32], redf[2][EIGH_WARPS];
  __shared__ int state;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nt = 32 * EIGH_WARPS;
  const int kp = k + (k & 1), npairs = kp / 2;  // odd k: one empty row and column
  const double shift = H[0];
  double mx = 0.0;
  for (int e = tid; e < kp * kp; e += nt) {
    const int i = e / kp, c = e - i * kp;
    double h = 0.0;
    if (i < k && c < k) h = i == c ? H[i * (ldh + 1)] - shift : 0.5 * (H[i * ldh + c] + H[c * ldh + i]);
    Hs[i][c] = h;
    Q[i][c] = (i < k0 && c < k0) ? Yf[i * 32 + c] : (i == c ? 1.0f : 0.0f);
    mx = fmax(mx, fabs(h));
  }
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) part[wid][0] = mx;
  __syncthreads();
  mx = fmax(fmax(part[0][0], part[1][0]), fmax(part[2][0], part[3][0]));
  const int ex = mx > 0.0 ? ilogb(mx) : 0;
  const double sc = ldexp(1.0, -ex);  // FP32 works on the shifted H / 2^ex
  // Every fourth call Q <- Q (3 - Q^T Q) / 2 (2.5 us): Q is then orthonormal to 1e-6 or so
  // whatever the number of calls (8e-5 was seen after 32 calls), below the gap of 2e-5 that the selection asks for
  const bool again = k0 > 0 && k0 % 4 == 0;
  if (again) {
    for (int e = tid; e < kp * kp; e += nt) {
      const int i = e / kp, c = e - i * kp;
      float s = 0.0f;
      for (int j = 0; j < kp; ++j) s = fmaf(Q[j][i], Q[j][c], s);
      T[i][c] = s;
    }
    __syncthreads();
    for (int e = tid; e < kp * kp; e += nt) {
      const int i = e / kp, c = e - i * kp;
      float s = 0.0f;
      for (int j = 0; j < kp; ++j) s = fmaf(Q[i][j], (j == c ? 1.0f : 0.0f) - T[j][c], s);
      A[i][c] = fmaf(0.5f, s, Q[i][c]);
    }
    __syncthreads();
  }
  for (int e = tid; e < kp * kp; e += nt) {
    const int i = e / kp, c = e - i * kp;
    if (again) Q[i][c] = A[i][c];
    A[i][c] = (float)(Hs[i][c] * sc);
  }
  __syncthreads();
  if (k0 > 0) {  // A <- Q^T A Q
    for (int e = tid; e < kp * kp; e += nt) {
      const int i = e / kp, c = e - i * kp;
      float s = 0.0f;
      for (int j = 0; j < kp; ++j) s = fmaf(A[i][j], Q[j][c], s);
      T[i][c] = s;
    }
    __syncthreads();
    for (int e = tid; e < kp * kp; e += nt) {
      const int i = e / kp, c = e - i * kp;
      if (c > i) continue;
      float s = 0.0f;
      for (int j = 0; j < kp; ++j) s = fmaf(Q[j][i], T[j][c], s);
      A[i][c] = s;
      A[c][i] = s;
    }
    __syncthreads();
  }
  // the (up to two) pair blocks (bi <= bj) of this thread
  const int nblocks = npairs * (npairs + 1) / 2;
  int bi[2], bj[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    int x = tid + u * nt, i = 0;
    while (i < npairs && x >= npairs - i) x -= npairs - i++;
    bi[u] = i;
    bj[u] = i + x;
  }
  float fro2 = 0.0f;  // |shifted H|_F^2 / 2^(2 ex)
  for (int sweep = 0; sweep < 10 && k > 1; ++sweep) {
    float off = 0.0f, tot = 0.0f;
    for (int e = tid; e < kp * kp; e += nt) {
      const int i = e / kp, c = e - i * kp;
      const float a2 = A[i][c] * A[i][c];
      tot += a2;
      if (c != i) off += a2;
    }
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if (lane == 0) {
      redf[0][wid] = off;
      redf[1][wid] = tot;
    }
    __syncthreads();
    off = redf[0][0] + redf[0][1] + redf[0][2] + redf[0][3];
    tot = redf[1][0] + redf[1][1] + redf[1][2] + redf[1][3];
    fro2 = tot;
    if (!(off > 1e-11f * tot)) break;
    for (int round = 0; round < kp - 1; ++round) {
      if (tid < npairs) {
        auto player = [&](int x) { return x == 0 ? 0 : 1 + (x - 1 + round) % (kp - 1); };
        int p = player(tid), q = player(kp - 1 - tid);
        if (p > q) { const int t = p; p = q; q = t; }
        const float apq = A[p][q];
        // sine and tan(angle / 2): with them a rotation by a small angle is orthogonal to
        // rounding, where a cosine of FP32 is not
        float sv = 0.0f, tau = 0.0f;
        if (apq != 0.0f) {
          const float z = (A[q][q] - A[p][p]) / (2.0f * apq), az = fabsf(z);
          const float t = (z >= 0.0f ? 1.0f : -1.0f) * (az > 1e8f ? 0.5f / az : 1.0f / (az + sqrtf(1.0f + az * az)));
          const float c = rsqrtf(1.0f + t * t);
          sv = t * c;
          tau = __fdividef(sv, 1.0f + c);
        }
        sn[tid] = sv;
        th[tid] = tau;
        pp[tid] = p;
        qq[tid] = q;
      }
      __syncthreads();
      auto rotate = [](float s, float tau, float& x, float& y) {  // x' = c x - s y, y' = s x + c y
        const float u = fmaf(tau, x, y), v = fmaf(-tau, y, x);
        x = fmaf(-s, u, x);
        y = fmaf(s, v, y);
      };
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (tid + u * nt < nblocks) {  // A block (pairs i, j) <- J_i^T block J_j
          const int i = bi[u], j = bj[u], p = pp[i], q = qq[i], r = pp[j], s = qq[j];
          float a2 = A[p][r], b2 = A[p][s], c2 = A[q][r], d2 = A[q][s];
          rotate(sn[j], th[j], a2, b2);
          rotate(sn[j], th[j], c2, d2);
          rotate(sn[i], th[i], a2, c2);
          rotate(sn[i], th[i], b2, d2);
          if (i == j) b2 = c2 = 0.0f;
          A[p][r] = a2;
          A[r][p] = a2;
          A[p][s] = b2;
          A[s][p] = b2;
          A[q][r] = c2;
          A[r][q] = c2;
          A[q][s] = d2;
          A[s][q] = d2;
        }
      }
      for (int e = tid; e < kp * npairs; e += nt) {
        const int i = e / npairs, j = e - i * npairs, p = pp[j], q = qq[j];
        float x = Q[i][p], y = Q[i][q];
        rotate(sn[j], th[j], x, y);
        Q[i][p] = x;
        Q[i][q] = y;
      }
      __syncthreads();
    }
  }
  __syncthreads();
  // lowest and second-lowest FP32 values
  if (wid == 0) {
    float v = lane < k ? A[lane][lane] : 3e38f, best = v;
    int arg = lane;
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, arg, o);
      if (ov < best || (ov == best && oi < arg)) {
        best = ov;
        arg = oi;
      }
    }
    float second = lane == arg ? 3e38f : v, big = lane < k ? fabsf(v) : 0.0f;
    for (int o = 16; o > 0; o >>= 1) {
      second = fminf(second, __shfl_xor_sync(0xffffffffu, second, o));
      big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
    }
    if (lane == 0) state = second - best > 2e-5f * big ? arg : -1;
    yv[lane] = lane < k ? (double)Q[lane][arg] : 0.0;
  }
  __syncthreads();
  const int arg = state;
  bool ok = arg >= 0;
  double theta = 0.0;
  for (int step = 0; ok; ++step) {
    // r = H y - theta y with y normalized; row `lane`, a quarter of the columns per warp
    double s = 0.0;
    for (int j = wid; j < k; j += EIGH_WARPS) s = fma(Hs[lane][j], yv[j], s);
    part[wid][lane] = lane < k ? s : 0.0;
    __syncthreads();
    if (wid == 0) {
      const double y = yv[lane], hy = (part[0][lane] + part[1][lane]) + (part[2][lane] + part[3][lane]);
      const double yy = warp_sum(y * y), yhy = warp_sum(y * hy);
      theta = yhy / yy;
      const double r = fma(-theta, y, hy);
      const double rr = warp_sum(r * r);
      rv[lane] = r;
      if (lane == 0) {
        const double lim = 1e-15 * ((double)sqrtf(fro2) / sc);
        state = rr <= lim * lim * yy ? 2 : (step < 6 && rr == rr ? 1 : 0);
      }
      part[0][lane] = theta;
    }
    __syncthreads();
    theta = part[0][0];
    const int st = state;
    if (st == 2) break;
    if (st == 0) {
      ok = false;
      break;
    }
    if (wid == 0) {
      float g = 0.0f;
      const float rs = (float)(lane < k ? rv[lane] * sc : 0.0);
      __syncwarp();
      for (int j = 0; j < k; ++j) g = fmaf(Q[j][lane < k ? lane : 0], __shfl_sync(0xffffffffu, rs, j), g);
      const float den = (lane < k ? A[lane][lane] : 0.0f) - (float)(theta * sc);
      coef[lane] = (lane < k && lane != arg) ? g / (fabsf(den) > 1e-5f ? den : 1e-5f) : 0.0f;
      __syncwarp();
      double y = yv[lane], d = 0.0;
      if (lane < k) {
        float df = 0.0f;
        for (int i = 0; i < k; ++i) df = fmaf(Q[lane][i], coef[i], df);
        d = (double)df;
      }
      yv[lane] = y - d;
    }
    __syncthreads();
  }
  __syncthreads();
  for (int e = tid; e < k * k; e += nt) Yf[(e / k) * 32 + e % k] = Q[e / k][e % k];
  if (!ok) {
    // FP64 Jacobi from the FP32 vectors: orthonormal in FP64 after two steps Q <- Q (3 -
    // Q^T Q) / 2 (1e-6, 1e-12, 1e-24), they leave it two sweeps instead of nine (596 us at
    // 32 vectors, 1284 from the identity, 1087 by eigh_full_kernel)
    __shared__ double Ad[32][33], Qd[32][33];
    auto product = [&](double (*X)[33], bool xt, double (*Z)[33], double (*out)[33]) {  // out = X Z or X^T Z
      for (int e = tid; e < k * k; e += nt) {
        const int i = e / k, c = e - i * k;
        double s = 0.0;
        for (int j = 0; j < k; ++j) s = fma(xt ? X[j][i] : X[i][j], Z[j][c], s);
        out[i][c] = s;
      }
      __syncthreads();
    };
    for (int e = tid; e < k * k; e += nt) Qd[e / k][e % k] = (double)Q[e / k][e % k];
    __syncthreads();
    for (int step = 0; step < 2; ++step) {
      product(Qd, true, Qd, Ad);
      for (int e = tid; e < k * k; e += nt) Ad[e / k][e % k] = (e / k == e % k ? 1.5 : 0.0) - 0.5 * Ad[e / k][e % k];
      __syncthreads();
      product(Qd, false, Ad, Hs);
      for (int e = tid; e < k * k; e += nt) Qd[e / k][e % k] = Hs[e / k][e % k];
      __syncthreads();
    }
    for (int e = tid; e < k * k; e += nt) {
      const int i = e / k, c = e - i * k;
      Hs[i][c] = i == c ? H[i * (ldh + 1)] - shift : 0.5 * (H[i * ldh + c] + H[c * ldh + i]);
    }
    __syncthreads();
    product(Hs, false, Qd, Ad);
    product(Qd, true, Ad, Hs);
    for (int e = tid; e < k * k; e += nt) {
      const int i = e / k, c = e - i * k;
      if (c < i) Hs[i][c] = Hs[c][i] = 0.5 * (Hs[i][c] + Hs[c][i]);
    }
    __syncthreads();
    jacobi_eigh(Hs, Qd, k, ldh, shift, w, Y);
    return;
  }
  if (wid == 0) {
    const double y = yv[lane];
    const double yy = warp_sum(y * y);
    if (lane < k) Y[lane * ldh] = y / sqrt(yy);
    if (lane == 0) w[0] = theta + shift;
  }
}

int vec_blocks(long long n) { return (int)std::min<long long>(DAV_MAX_BLOCKS, std::max<long long>(1, (n + DT - 1) / DT)); }

}  // namespace

// k = number of vectors -> register block of the kernels
#define DAV_DISPATCH(k, CALL)  \
  do {                         \
    if ((k) <= 8) {            \
      constexpr int KB = 8;    \
      CALL;                    \
    } else if ((k) <= 16) {    \
      constexpr int KB = 16;   \
      CALL;                    \
    } else {                   \
      constexpr int KB = 32;   \
      CALL;                    \
    }                          \
  } while (0)

void dav_dots2(const double* V, const double* w, double* out, int stride, const double* V2, const double* w2,
               double* out2, int stride2, long long ld, int k, long long n, const DavScratch& sc, cudaStream_t st) {
  if (k <= 0) return;
  if (k > KMAX) k = KMAX;  // the subspace size is checked against this limit on the host
  const DotSet a{V, w, out, stride}, b{V2, w2, out2, stride2};
  const dim3 grid(vec_blocks(n), V2 ? 2 : 1);
  DAV_DISPATCH(k, (dots_kernel<KB><<<grid, DT, 0, st>>>(a, b, ld, k, n, sc.partial, sc.counters)));
}

void dav_dots(const double* V, long long ld, int k, const double* w, long long n, const DavScratch& sc, double* out,
              int out_stride, cudaStream_t st) {
  dav_dots2(V, w, out, out_stride, nullptr, nullptr, nullptr, 0, ld, k, n, sc, st);
}

void dav_ritz(const double* V, const double* AV, long long ld, int k, const double* Y, int ys, const double* theta,
              const double* diag, double* x, double* ax, double* t, long long n, const DavScratch& sc, double* c,
              double* scal, cudaStream_t st) {
  DAV_DISPATCH(k, (ritz_kernel<KB><<<vec_blocks(n), DT, 0, st>>>(V, AV, ld, k, Y, ys, theta, diag, x, ax, t, n,
                                                                 sc.partial, sc.counters, c, scal)));
}

void dav_project_dots(const double* V, long long ld, int k, const double* c, const double* t, double* out, long long n,
                      const DavScratch& sc, double* c2, cudaStream_t st) {
  DAV_DISPATCH(k, (project_kernel<KB, true><<<vec_blocks(n), DT, 0, st>>>(V, ld, k, c, t, out, n, sc.partial,
                                                                          sc.counters, c2)));
}

void dav_project_norm(const double* V, long long ld, int k, const double* c, const double* t, double* out, long long n,
                      const DavScratch& sc, double* nrm2, cudaStream_t st) {
  DAV_DISPATCH(k, (project_kernel<KB, false><<<vec_blocks(n), DT, 0, st>>>(V, ld, k, c, t, out, n, sc.partial,
                                                                           sc.counters, nrm2)));
}

void dav_lincomb(const double* V, long long ld, int k, const double* c, int cs, double sign, double* out,
                 long long n, bool add, cudaStream_t st) {
  long long grid = (n + 255) / 256;
  if (grid > 152 * 8) grid = 152 * 8;
  if (grid < 1) grid = 1;
  lincomb_kernel<<<(unsigned)grid, 256, 0, st>>>(V, ld, k, c, cs, sign, out, n, add ? 1 : 0);
}

void dav_scale(double* x, const double* nrm2, double floor, long long n, cudaStream_t st) {
  long long grid = (n + 255) / 256;
  if (grid > 152 * 8) grid = 152 * 8;
  if (grid < 1) grid = 1;
  scale_kernel<<<(unsigned)grid, 256, 0, st>>>(x, nrm2, floor, n);
}

void dav_axpy_unit(double* x, const double* z, const double* xz_zz, double a, long long n, cudaStream_t st) {
  long long grid = (n + 255) / 256;
  if (grid > 152 * 8) grid = 152 * 8;
  if (grid < 1) grid = 1;
  axpy_unit_kernel<<<(unsigned)grid, 256, 0, st>>>(x, z, xz_zz, a, n);
}

void dav_eigh(const double* H, int k, int ldh, double* w, double* Y, cudaStream_t st) {
  eigh_full_kernel<<<1, 32 * EIGH_WARPS, 0, st>>>(H, k, ldh, w, Y);
}

void dav_eigh_lowest(const double* H, int k, int ldh, double* w, double* Y, float* Yf, int k0, cudaStream_t st) {
  eigh_lowest_kernel<<<1, 32 * EIGH_WARPS, 0, st>>>(H, k, ldh, w, Y, Yf, k0 < k ? k0 : 0);
}

}  // namespace dmrg

namespace dmrg {

namespace {

// diag[b][i, j] = sum over the diagonal tasks of block b of
// scale * X_L[i, i] * X_R[j, j] (identity factors contribute 1)
__global__ void heff_diag_kernel(const double* __restrict__ store, const Task* __restrict__ tasks,
                                 const int* __restrict__ dstart, const int* __restrict__ dtask,
                                 const PsiBlock* __restrict__ blocks, int nblk, double* __restrict__ diag) {
  for (int b = blockIdx.y; b < nblk; b += gridDim.y) {
    const PsiBlock pb = blocks[b];
    const long long ne = (long long)pb.mL * pb.mR;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < ne; e += (long long)gridDim.x * blockDim.x) {
      const int i = (int)(e / pb.mR), j = (int)(e % pb.mR);
      double s = 0.0;
      for (int q = dstart[b]; q < dstart[b + 1]; ++q) {
        const Task t = tasks[dtask[q]];
        const double dl = t.aoff < 0 ? 1.0 : store[t.aoff + (long long)i * (pb.mL + 1)];
        const double dr = t.boff < 0 ? 1.0 : store[t.boff + (long long)j * (pb.mR + 1)];
        s = fma(t.scale * dl, dr, s);
      }
      diag[pb.off + e] = s;
    }
  }
}

}  // namespace

void launch_heff_diag(const double* store, const Task* tasks, const int* dstart, const int* dtask,
                      const PsiBlock* blocks, int nblk, double* diag, cudaStream_t st) {
  if (nblk <= 0) return;
  dim3 grid(64, nblk < 65535 ? nblk : 65535);
  heff_diag_kernel<<<grid, 256, 0, st>>>(store, tasks, dstart, dtask, blocks, nblk, diag);
}

}  // namespace dmrg
