// Sweep kernels: blocking (Eq. blocked-ops), the normal-to-complementary
// sums of the mixed NC/CN scheme (Sec. III.A), decimation (one-sided Jacobi
// SVD of the psi blocks), orthonormal bases for the initial MPS, and the
// small GEMMs that carry a wavefunction to the next bond. The
// transformation of Eq. op-trans runs on the FP64 sigma kernel with a
// dedicated work list (see sweep.cpp).
#include <cooperative_groups.h>

#include <algorithm>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/dmrg.h"
#include "kernels.h"

namespace dmrg {

namespace {

__constant__ int c_site_n[4] = {0, 1, 1, 2};
__constant__ int c_site_s[4] = {0, 1, -1, 0};

// index of sector (n, s) in a basis sorted by (n, s), or -1
__device__ __forceinline__ int find_sector(const int* q, int nq, int n, int s) {
  int lo = 0, hi = nq - 1;
  while (lo <= hi) {
    const int mid = (lo + hi) >> 1;
    const int mn = q[2 * mid], ms = q[2 * mid + 1];
    if (mn == n && ms == s) return mid;
    if (mn < n || (mn == n && ms < s)) lo = mid + 1;
    else hi = mid - 1;
  }
  return -1;
}

// One destination block per CTA (grid-stride): for every term of its
// operator, in order, find the block sector ib the term reads (enlarged
// input sector minus the site state's quantum numbers), the source block
// and its output sector ob, and add coef * sign * source into the chunk
// (rows of ob within Qout, columns of ib within Qin). Terms are resolved 256
// at a time, one per thread, into shared memory (the lookups are dependent
// global loads, so doing them in parallel hides their latency), then applied
// in term order. Each destination element (row R, column C) is owned by one
// thread - warp R mod 8, lane C mod 32 - for every update, so terms are
// applied in order without atomics and the sums are deterministic; a warp
// walks its rows of a chunk and its lanes read consecutive columns. Signs:
// block x site takes (-1)^{N(block in)} when the site part is odd; site x
// block takes (-1)^{N(site in)} when the block operator is odd.
struct RTerm {        // one resolved term
  long long soff;     // source block offset
  double w;           // coefficient times sign
  int r0, c0, rows, cols;
  int kind;           // 0 skip, 1 identity, 2 source, 3 source transposed
  int store2;         // source in the second store
};
constexpr int BLK_THREADS = 256;
static_assert(BLK_THREADS == 256, "the update ownership assumes 8 warps");

__global__ void __launch_bounds__(BLK_THREADS) blocking_kernel(BlockingDev d) {
  __shared__ RTerm rt[BLK_THREADS];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int warp = tid >> 5, lane = tid & 31;  // 8 warps (BLK_THREADS = 256)
  for (int bi = blockIdx.x; bi < d.ndst; bi += gridDim.x) {
    const BDst db = d.dsts[bi];
    double* dst = d.dst_store + db.off;
    const long long ne = (long long)db.rows * db.cols;
    for (long long e = tid; e < ne; e += nt) dst[e] = 0.0;
    __syncthreads();  // zeroing and the updates below own elements differently
    const int qin_n = d.eq[2 * db.Qin], qin_s = d.eq[2 * db.Qin + 1];
    const int qout_n = d.eq[2 * db.Qout], qout_s = d.eq[2 * db.Qout + 1];
    const int t_end = d.term_start[db.k + 1];
    for (int t0 = d.term_start[db.k]; t0 < t_end; t0 += nt) {
      const int nhere = min(nt, t_end - t0);
      if (tid < nhere) {
        RTerm& r = rt[tid];
        r.kind = 0;
        const BTerm tm = d.terms[t0 + tid];
        const int ib = find_sector(d.bq, d.nb, qin_n - c_site_n[tm.nin], qin_s - c_site_s[tm.nin]);
        const int c0 = ib >= 0 ? d.chunk_off[db.Qin * d.nb + ib] : -1;
        int ob = ib, par = 0;
        long long soff = -1;
        bool ok = c0 >= 0;
        if (ok && tm.src >= 0) {
          const int dn = d.src_dq[2 * tm.src], ds = d.src_dq[2 * tm.src + 1];
          par = d.src_par[tm.src];
          if (!tm.trans) {
            soff = d.srcblk[(long long)tm.src * d.nb + ib];
            ob = soff < 0 ? -1 : find_sector(d.bq, d.nb, d.bq[2 * ib] + dn, d.bq[2 * ib + 1] + ds);
          } else {
            ob = find_sector(d.bq, d.nb, d.bq[2 * ib] - dn, d.bq[2 * ib + 1] - ds);
            if (ob >= 0) soff = d.srcblk[(long long)tm.src * d.nb + ob];
          }
          ok = soff >= 0 && ob >= 0;
        }
        if (ok && (d.bq[2 * ob] + c_site_n[tm.nout] != qout_n || d.bq[2 * ob + 1] + c_site_s[tm.nout] != qout_s)) {
          atomicExch(d.err, 1);
          ok = false;
        }
        const int r0 = ok ? d.chunk_off[db.Qout * d.nb + ob] : -1;
        if (ok && r0 >= 0) {
          bool neg;
          if (d.left) neg = ((c_site_n[tm.nout] - c_site_n[tm.nin]) & 1) && (d.bq[2 * ib] & 1);
          else neg = par && (c_site_n[tm.nin] & 1);
          r.soff = soff;
          r.w = neg ? -tm.coef : tm.coef;
          r.r0 = r0;
          r.c0 = c0;
          r.rows = d.bdim[ob];
          r.cols = d.bdim[ib];
          r.kind = tm.src < 0 ? 1 : (tm.trans ? 3 : 2);
          r.store2 = tm.src >= d.nsrc1;
        }
      }
      __syncthreads();
      for (int q = 0; q < nhere; ++q) {
        const RTerm r = rt[q];
        if (r.kind == 0) continue;
        const double* __restrict__ S = r.store2 ? d.src_store2 : d.src_store;
        // rows of the destination with (row mod 8) = warp, columns with (col mod 32) = lane
        for (int i = (warp - r.r0) & 7; i < r.rows; i += 8) {
          double* drow = dst + (long long)(r.r0 + i) * db.cols + r.c0;
          for (int j = (lane - r.c0) & 31; j < r.cols; j += 32) {
            double v;
            if (r.kind == 1) v = (i == j) ? 1.0 : 0.0;
            else if (r.kind == 2) v = S[r.soff + (long long)i * r.cols + j];
            else v = S[r.soff + (long long)j * r.rows + i];
            drow[j] += r.w * v;
          }
        }
      }
      __syncthreads();
    }
  }
}

// Y_o = sum_i C[o][i] X_i for one 64 x 128 (operator, element) tile per
// iteration: the coefficient tile (64 x 16) and 16 source rows of 128
// elements are staged in shared memory, each warp owns 8 output operators x
// 128 elements (16 sub-tiles of 8 x 8) and accumulates them with the FP64
// m8n8k4 tensor instruction (lane g = lane/4, c = lane%4 holds A[g][c],
// B[c][g], D[g][2c..2c+1]). Each output element is written once.
constexpr int CB_K = 16;
struct CombSmem {
  double C[COMB_TM][CB_K + 4];
  double X[CB_K][COMB_TN + 4];
};

__device__ __forceinline__ void dmma8(double (&d)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};\n"
               : "+d"(d[0]), "+d"(d[1])
               : "d"(a), "d"(b));
}

__global__ void __launch_bounds__(256, 2)
opcomb_kernel(const double* __restrict__ src, const long long* __restrict__ xoff, const double* __restrict__ coef,
              const CombClass* __restrict__ cls, int ncls, int ntiles, double* __restrict__ dst) {
  __shared__ __align__(16) CombSmem sm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, c = lane & 3;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    int k = 0;
    while (k + 1 < ncls && cls[k + 1].tile_start <= t) ++k;
    const CombClass cc = cls[k];
    const int local = t - cc.tile_start;
    const int to = local / cc.tiles_e, te = local - to * cc.tiles_e;
    const int o0 = to * COMB_TM;
    const long long e0 = (long long)te * COMB_TN;
    double acc[COMB_TN / 8][2];
#pragma unroll
    for (int q = 0; q < COMB_TN / 8; ++q) acc[q][0] = acc[q][1] = 0.0;
    for (int i0 = 0; i0 < cc.n_in; i0 += CB_K) {
      for (int x = tid; x < COMB_TM * CB_K; x += blockDim.x) {
        const int r = x / CB_K, kk = x - r * CB_K;
        const int o = o0 + r, i = i0 + kk;
        sm.C[r][kk] = (o < cc.n_out && i < cc.n_in) ? coef[cc.c_off + (long long)o * cc.n_in + i] : 0.0;
      }
      for (int x = tid; x < CB_K * COMB_TN; x += blockDim.x) {
        const int kk = x / COMB_TN, j = x - kk * COMB_TN;
        const int i = i0 + kk;
        const long long e = e0 + j;
        sm.X[kk][j] = (i < cc.n_in && e < cc.E) ? src[xoff[cc.x_start + i] + e] : 0.0;
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < CB_K; kk += 4) {
        const double a = sm.C[warp * 8 + g][kk + c];
#pragma unroll
        for (int q = 0; q < COMB_TN / 8; ++q) dmma8(acc[q], a, sm.X[kk + c][q * 8 + g]);
      }
      __syncthreads();
    }
    const int o = o0 + warp * 8 + g;
    if (o < cc.n_out) {
      double* y = dst + cc.y_off + (long long)o * cc.E;
#pragma unroll
      for (int q = 0; q < COMB_TN / 8; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const long long e = e0 + q * 8 + 2 * c + h;
          if (e < cc.E) y[e] = acc[q][h];
        }
    }
  }
}

// One strided GEMM job per CTA (grid-stride): 16 x 16 output tiles, one
// element per thread, k staged in shared memory 16 at a time.
__global__ void bgemm_kernel(const double* __restrict__ A, const double* __restrict__ B, double* __restrict__ C,
                             const GJob* __restrict__ jobs, int njobs) {
  __shared__ double sa[16][17], sb[16][17];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  for (int jb = blockIdx.x; jb < njobs; jb += gridDim.x) {
    const GJob g = jobs[jb];
    for (int i0 = 0; i0 < g.m; i0 += 16)
      for (int j0 = 0; j0 < g.n; j0 += 16) {
        double acc = 0.0;
        for (int k0 = 0; k0 < g.kk; k0 += 16) {
          {
            const int i = i0 + ty, k = k0 + tx;
            sa[ty][tx] = (i < g.m && k < g.kk)
                             ? A[g.a + (g.ta ? (long long)k * g.lda + i : (long long)i * g.lda + k)] : 0.0;
            const int kb = k0 + ty, j = j0 + tx;
            sb[ty][tx] = (kb < g.kk && j < g.n)
                             ? B[g.b + (g.tb ? (long long)j * g.ldb + kb : (long long)kb * g.ldb + j)] : 0.0;
          }
          __syncthreads();
#pragma unroll
          for (int q = 0; q < 16; ++q) acc = fma(sa[ty][q], sb[q][tx], acc);
          __syncthreads();
        }
        const int i = i0 + ty, j = j0 + tx;
        if (i < g.m && j < g.n) C[g.c + (long long)i * g.ldc + j] = acc;
      }
  }
}

// Orthonormalise the columns of each d x m block (row-major, in place) by
// classical Gram-Schmidt applied twice per column.
__global__ void orthonormalize_kernel(double* __restrict__ store, const GramBlock* __restrict__ gb, int nb) {
  __shared__ double coef[1024];
  __shared__ double red[256];
  for (int b = blockIdx.x; b < nb; b += gridDim.x) {
    const GramBlock g = gb[b];
    double* G = store + g.g_off;
    const int d = g.d, m = g.m;
    for (int j = 0; j < m; ++j) {
      for (int pass = 0; pass < 2; ++pass) {
        for (int i = threadIdx.x; i < j; i += blockDim.x) {
          double s = 0.0;
          for (int r = 0; r < d; ++r) s = fma(G[(long long)r * m + i], G[(long long)r * m + j], s);
          coef[i] = s;
        }
        __syncthreads();
        for (int r = threadIdx.x; r < d; r += blockDim.x) {
          double s = 0.0;
          for (int i = 0; i < j; ++i) s = fma(coef[i], G[(long long)r * m + i], s);
          G[(long long)r * m + j] -= s;
        }
        __syncthreads();
      }
      double s = 0.0;
      for (int r = threadIdx.x; r < d; r += blockDim.x) s = fma(G[(long long)r * m + j], G[(long long)r * m + j], s);
      red[threadIdx.x] = s;
      __syncthreads();
      for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
      }
      const double inv = red[0] > 0.0 ? 1.0 / sqrt(red[0]) : 0.0;
      __syncthreads();
      for (int r = threadIdx.x; r < d; r += blockDim.x) G[(long long)r * m + j] *= inv;
      __syncthreads();
    }
  }
}

// dst[b] (d x k, row-major) = first k columns of Q[b] (d x d), each column
// with the sign that makes its entry of largest magnitude positive (first
// such entry on ties). Eigenvectors carry an arbitrary sign; this fixes the
// gauge of the kept states, so a basis is a function of the wavefunction
// alone. One warp per column.
__global__ void take_columns_kernel(const double* __restrict__ Qall, const TakeBlock* __restrict__ tb, int nb,
                                    double* __restrict__ dst) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int b = blockIdx.y; b < nb; b += gridDim.y) {
    const TakeBlock t = tb[b];
    for (int c = blockIdx.x * nw + wid; c < t.k; c += gridDim.x * nw) {
      double best = -1.0, val = 0.0;
      int bi = 0x7fffffff;
      for (int r = lane; r < t.d; r += 32) {
        const double v = Qall[t.q_off + (long long)r * t.d + c];
        if (fabs(v) > best) {  // r ascends per lane, so ties keep the first
          best = fabs(v);
          bi = r;
          val = v;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        const double ov = __shfl_xor_sync(0xffffffffu, val, o);
        if (ob > best || (ob == best && oi < bi)) {
          best = ob;
          bi = oi;
          val = ov;
        }
      }
      const double sg = val < 0.0 ? -1.0 : 1.0;
      for (int r = lane; r < t.d; r += 32)
        dst[t.dst_off + (long long)r * t.k + c] = sg * Qall[t.q_off + (long long)r * t.d + c];
    }
  }
}

// ---------------------------------------------------------------- SVD
// One-sided (Hestenes) Jacobi: the d columns of A (d x m data, each column a
// contiguous vector of length m) are rotated in pairs until mutually
// orthogonal; the rotations, accumulated in V (d x d), are the singular
// vectors of the psi block's d-dimensional side, and the final column norms
// are the singular values. Pairs of one round are disjoint (round-robin
// order), so every warp of the grid takes pairs of any block, and the grid
// synchronizes between rounds.
__global__ void svd_setup_kernel(const double* __restrict__ psi, const SvdBlock* __restrict__ sb, int nb,
                                 double* __restrict__ work, int left) {
  for (int b = blockIdx.y; b < nb; b += gridDim.y) {
    const SvdBlock s = sb[b];
    if (s.cluster) continue;
    const long long na = (long long)s.d * s.m;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < na; e += (long long)gridDim.x * blockDim.x) {
      const int c = (int)(e / s.m), i = (int)(e % s.m);
      // left: column c = row c of X (d = rows, m = cols); right: column c = column c of X (d = cols, m = rows)
      work[s.a_off + e] = left ? psi[s.psi_off + (long long)c * s.m + i] : psi[s.psi_off + (long long)i * s.d + c];
    }
    const long long nv = (long long)s.d * s.d;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nv; e += (long long)gridDim.x * blockDim.x)
      work[s.v_off + e] = (e / s.d == e % s.d) ? 1.0 : 0.0;
  }
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// |A|_F^2 of every block's work matrix into w[w_off] (scratch until the
// singular values are written there).
__global__ void svd_norm_kernel(const SvdBlock* __restrict__ sb, int nb, const double* __restrict__ work,
                                double* __restrict__ w) {
  __shared__ double red[32];
  for (int b = blockIdx.x; b < nb; b += gridDim.x) {
    const SvdBlock s = sb[b];
    if (s.cluster) continue;
    const long long na = (long long)s.d * s.m;
    double v = 0.0;
    for (long long e = threadIdx.x; e < na; e += blockDim.x) v = fma(work[s.a_off + e], work[s.a_off + e], v);
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
      double x = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
      x = warp_sum(x);
      if (threadIdx.x == 0) w[s.w_off] = x;
    }
    __syncthreads();
  }
}

// A pair is rotated while its cosine |a_p . a_q| / (|a_p| |a_q|) is at least
// tol = max(1e-15, eps sqrt(m)) (the rounding floor of an m-term dot
// product), and only if both vectors exceed 1e-15 |A|_F: vectors below that
// are numerical zeros (a block with more rows than columns has them), whose
// mutual cosines are rounding noise and would never settle. Sweeps stop when
// no pair of any block is above its tolerance (at most 30).
//
// On this GPU a round is bound by the FP64 pipe: a warp instruction takes about
// 67 cycles of its SM sub-partition, whatever the number of warps, so a pair
// costs what its FP64 instructions cost, one after the other. Hence:
//  - angle, scaling and the clear cases of the test in FP32, on exponent-shifted
//    bits (a conversion instruction would go through the same pipe): an angle off
//    by 1e-7 leaves 1e-7 of the product, which later sweeps remove;
//  - the rotation is fixed by tau = tan(angle / 2), any FP32 number, and its
//    sine 2 tau / (1 + tau^2), found in FP64 by Newton's step from an FP32
//    reciprocal; applied as three shears (x -= tau y, y += s x, x -= tau y), three
//    instructions per element pair where a rotation by sine and cosine takes four;
//  - the squared column norms are carried along (al - t ga, be + t ga; exact to
//    first order in the angle's error) and recomputed at the start of every sweep.
constexpr int SVD_THREADS = 256;
constexpr int SVD_REG = 8;         // vectors up to 32 * SVD_REG long stay in registers

// v * 2^-(e - 1023) in FP32 (truncated), e a biased exponent not below that
// of v by construction; 0 where that is below FP32's range
__device__ __forceinline__ float scaled_float(double v, int e) {
  const int h = __double2hiint(v), l = __double2loint(v);
  const int ef = ((h >> 20) & 0x7ff) - e + 127;
  const int bits = (h & 0x80000000) | (ef << 23) | ((h & 0xfffff) << 3) | ((unsigned)l >> 29);
  return ef <= 0 ? 0.0f : __int_as_float(bits);
}

// exact (a normal number or zero)
__device__ __forceinline__ double wide(float v) {
  const int b = __float_as_int(v), e = (b >> 23) & 0xff;
  return e == 0 ? 0.0 : __hiloint2double((b & 0x80000000) | ((e + 896) << 20) | ((b & 0x7fffff) >> 3), b << 29);
}

struct SvdRotation {
  double tau, s, t;  // tan(angle / 2), sine, tangent (FP32 accuracy, for the norms)
};

// What the angle needs of the norms alone: ready before the product is
struct SvdNorms {
  bool large;    // both squared norms above floor2 (numbers, or NaN)
  int e;         // biased exponent of the larger
  float d, lim;  // (be - al) and tol |a_p| |a_q|, over 2^(e - 1023)
};

__device__ __forceinline__ SvdNorms svd_norms(double al, double be, double floor2, double tol2) {
  const long long ia = __double_as_longlong(al), ib = __double_as_longlong(be), fl = __double_as_longlong(floor2);
  SvdNorms n;
  n.large = ia > fl && ib > fl;
  n.e = (int)((ia > ib ? ia : ib) >> 52);
  n.d = scaled_float(be - al, n.e);
  const float ab = scaled_float(al, n.e) * scaled_float(be, n.e);
  n.lim = sqrtf((float)tol2) * (ab * rsqrtf(ab));  // ab >= 1e-30 where it is used
  return n;
}

// Rotation that makes two columns of squared norms al, be and product ga
// orthogonal; false when the pair is within its tolerance. Uniform over a warp.
__device__ __forceinline__ bool svd_angle(const SvdNorms& n, double al, double be, double ga, double tol2,
                                          SvdRotation& rot) {
  if (!n.large || (__double_as_longlong(ga) << 1) == 0) return false;
  const int eg = (__double2hiint(ga) >> 20) & 0x7ff;
  float t;
  if (n.e >= 64 && n.e <= 1980 && eg <= n.e + 1) {
    const float g = scaled_float(ga, n.e), ag = fabsf(g);
    if (ag < 0.999f * n.lim) return false;
    if (!(ag > 1.001f * n.lim) && !(ga * ga >= tol2 * (al * be))) return false;
    const float z = __fdividef(n.d, 2.0f * g);
    const float az = fabsf(z), q = fmaf(z, z, 1.0f);
    t = az > 1e8f ? __fdividef(0.5f, az) : __fdividef(1.0f, fmaf(q, rsqrtf(q), az));
    t = z >= 0.0f ? t : -t;
  } else {  // outside FP32's reach, or not finite: plain FP64
    if (!(ga * ga >= tol2 * (al * be))) return false;
    const double zeta = (be - al) / (2.0 * ga);
    t = (float)((zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta)));
  }
  const float u = fmaf(t, t, 1.0f);
  const float tau = __fdividef(t, fmaf(u, rsqrtf(u), 1.0f));
  rot.t = wide(t);
  rot.tau = wide(tau);
  // s = 2 tau / w, w = 1 + tau^2: 1 / w = r (1 + e1 + e1^2 + ...), e1 ~ 1e-7
  const double r = wide(__fdividef(1.0f, fmaf(tau, tau, 1.0f)));
  const double e1 = fma(-r, fma(rot.tau, rot.tau, 1.0), 1.0), s0 = wide(2.0f * tau) * r;
  rot.s = fma(s0, fma(e1, e1, e1), s0);
  return true;
}

__device__ __forceinline__ void svd_rotate(const SvdRotation& rot, double& x, double& y) {
  x = fma(-rot.tau, y, x);
  y = fma(rot.s, x, y);
  x = fma(-rot.tau, y, x);
}

// Round `r` of block s, pair i: true when the pair was above its tolerance.
// fresh: the norms are recomputed (first round of a sweep).
__device__ bool svd_pair(const SvdBlock& s, int i, int r, bool fresh, double* __restrict__ work,
                         double* __restrict__ nrm, double floor2, int lane) {
  const int dp = s.d + (s.d & 1);
  auto player = [&](int x) { return x == 0 ? 0 : 1 + (x - 1 + r) % (dp - 1); };
  int p = player(i), q = player(dp - 1 - i);
  if (p > q) { const int t = p; p = q; q = t; }
  double* ap = work + s.a_off + (long long)p * s.m;
  if (q >= s.d) {  // p sits this round out
    if (fresh) {
      double al = 0.0;
      for (int e = lane; e < s.m; e += 32) al = fma(ap[e], ap[e], al);
      al = warp_sum(al);
      if (lane == 0) nrm[s.q_off + p] = al;
    }
    return false;
  }
  double* aq = work + s.a_off + (long long)q * s.m;
  double* vp = work + s.v_off + (long long)p * s.d;
  double* vq = work + s.v_off + (long long)q * s.d;
  const bool in_regs = s.m <= 32 * SVD_REG && s.d <= 32 * SVD_REG;
  double x[SVD_REG], y[SVD_REG], vx[SVD_REG], vy[SVD_REG];
  double al = 0.0, be = 0.0, ga = 0.0;
  if (!fresh) {
    al = nrm[s.q_off + p];
    be = nrm[s.q_off + q];
  }
  if (in_regs) {
#pragma unroll
    for (int k = 0; k < SVD_REG; ++k) {
      const int e = lane + 32 * k;
      if (32 * k < s.m) {
        x[k] = e < s.m ? ap[e] : 0.0;
        y[k] = e < s.m ? aq[e] : 0.0;
      }
      if (32 * k < s.d) {
        vx[k] = e < s.d ? vp[e] : 0.0;
        vy[k] = e < s.d ? vq[e] : 0.0;
      }
    }
#pragma unroll
    for (int k = 0; k < SVD_REG; ++k)
      if (32 * k < s.m) {
        ga = fma(x[k], y[k], ga);
        if (fresh) {
          al = fma(x[k], x[k], al);
          be = fma(y[k], y[k], be);
        }
      }
  } else {
    for (int e = lane; e < s.m; e += 32) {
      const double u = ap[e], v = aq[e];
      ga = fma(u, v, ga);
      if (fresh) {
        al = fma(u, u, al);
        be = fma(v, v, be);
      }
    }
  }
  if (fresh) {
    al = warp_sum(al);
    be = warp_sum(be);
  }
  const double tol2 = fmax(1e-30, 4.930380657631324e-32 * (double)s.m);
  const SvdNorms norms = svd_norms(al, be, floor2, tol2);
  ga = warp_sum(ga);
  SvdRotation rot;
  rot.t = 0.0;
  const bool rotate = svd_angle(norms, al, be, ga, tol2, rot);
  if (rotate) {
    if (in_regs) {
#pragma unroll
      for (int k = 0; k < SVD_REG; ++k) {
        const int e = lane + 32 * k;
        if (32 * k < s.m && e < s.m) {
          svd_rotate(rot, x[k], y[k]);
          ap[e] = x[k];
          aq[e] = y[k];
        }
        if (32 * k < s.d && e < s.d) {
          svd_rotate(rot, vx[k], vy[k]);
          vp[e] = vx[k];
          vq[e] = vy[k];
        }
      }
    } else {
      for (int e = lane; e < s.m; e += 32) {
        double u = ap[e], v = aq[e];
        svd_rotate(rot, u, v);
        ap[e] = u;
        aq[e] = v;
      }
      for (int e = lane; e < s.d; e += 32) {
        double u = vp[e], v = vq[e];
        svd_rotate(rot, u, v);
        vp[e] = u;
        vq[e] = v;
      }
    }
  }
  if (lane == 0 && (rotate || fresh)) {
    nrm[s.q_off + p] = fma(-rot.t, ga, al);
    nrm[s.q_off + q] = fma(rot.t, ga, be);
  }
  return rotate;
}

// Wait for a phase of an mbarrier, at most about a second; false: it did not come.
__device__ __forceinline__ bool svd_wait(unsigned bar, unsigned parity) {
  for (int k = 0; k < (1 << 20); ++k) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, 1000;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

__device__ __forceinline__ unsigned cluster_addr(const void* p, int rank) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}

// v to a shared-memory address of the cluster, its 8 bytes counted by the mbarrier beside it
__device__ __forceinline__ void svd_send(unsigned addr, double v, unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr),
               "l"(__double_as_longlong(v)), "r"(bar)
               : "memory");
}

// Both columns of a warp's buffer are awaited: 2 ld doubles
__device__ __forceinline__ void svd_arm(unsigned bar, int ld) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(2 * ld * 8) : "memory");
}

// Blocks that fit: one cluster each. Warp w of CTA k holds the pair
// k * ppc + w, its two columns (A, V and squared norm) in the CTA's shared
// memory, and after a round sends them where the next round's pairs want
// them, in its own CTA or a neighbour's, into the other of two buffers: a pair
// waits for its two columns and for nothing else. Clusters of 16 CTAs (the most
// there is), so that up to 64 pairs have an SM sub-partition each: 2.1 ms a
// decimation against 2.6 with 8 (K=16, M=150, an earlier form). Bound by the latency of
// a round, a chain of some 25 FP64 instructions, the FP32 angle and the way of
// the columns. C: 32-element chunks of the longer of A's and V's
// columns; what lies past the shorter's end is skipped by branches that
// the compiler is kept from turning into selects (all the instructions
// would go through the FP64 pipe: 4200 of a round's 9000 cycles).
// One 96 x 96 block takes 1.9 us a round, 4.9 on the grid-wide kernel (columns
// through L2, a grid barrier a round, every block waiting for the largest);
// 26 blocks of up to 96 2.8 ms against 6.7, up to 200 16.6 against 30.4, 80 of
// up to 250 93 against 109. Decimations of two sweeps: 113 -> 35 ms at K=16,
// M=150 (30 steps), 447 -> 222 at K=24, M=300 (46 steps).
template <int C>
__device__ __forceinline__ void svd_cluster_block(const SvdBlock& s, const double* __restrict__ psi,
                                                  double* __restrict__ work, int left, double* cols, double* part,
                                                  unsigned int* above, unsigned long long* full) {
  namespace cgp = cooperative_groups;
  cgp::cluster_group cluster = cgp::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int ppc = (s.npairs + SVD_CLUSTER - 1) / SVD_CLUSTER;
  const int pair = rank * ppc + wid;
  const bool active = wid < ppc && pair < s.npairs;
  const int m = s.m, d = s.d, dp = d + (d & 1), ld = m + d + 1;
  const int px = pair, py = dp - 1 - pair;  // positions of the pair; the next round finds position x at x - 1, 1 at dp - 1
  double *cx = cols + wid * 4 * ld, *cy = cx + ld;  // buffer 1: 2 ld doubles on
  const unsigned my_full = (unsigned)__cvta_generic_to_shared(full + 2 * wid);  // buffer 1: 8 bytes on
  unsigned tx = 0, ty = 0, tx_full = 0, ty_full = 0;  // where the columns go, and the mbarriers there (of buffer 0)
  if (active) {
    auto home = [&](int x, unsigned& col, unsigned& bar) {
      const int pr = x < s.npairs ? x : dp - 1 - x, w = pr % ppc, k = pr / ppc;
      col = cluster_addr(cols + (w * 4 + (x < s.npairs ? 0 : 1)) * ld, k);
      bar = cluster_addr(full + 2 * w, k);
    };
    home(px == 0 ? 0 : px == 1 ? dp - 1 : px - 1, tx, tx_full);
    home(py == 1 ? dp - 1 : py - 1, ty, ty_full);
    if (lane == 0)
      for (int b = 0; b < 2; ++b) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(my_full + 8 * b) : "memory");
        svd_arm(my_full + 8 * b, ld);
      }
    double nn = 0.0;
    for (int h = 0; h < 2; ++h) {
      double* c = h ? cy : cx;
      const int col = h ? py : px;  // a column past d: zero
      for (int e = lane; e < m; e += 32) {
        const double v = col >= d ? 0.0
                         : left   ? psi[s.psi_off + (long long)col * m + e]
                                  : psi[s.psi_off + (long long)e * d + col];
        c[e] = v;
        nn = fma(v, v, nn);
      }
      for (int e = lane; e < d; e += 32) c[m + e] = e == col ? 1.0 : 0.0;
    }
    nn = warp_sum(nn);
    if (lane == 0) part[wid] = nn;
  }
  if (threadIdx.x < 3) above[threadIdx.x] = 0u;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  cluster.sync();
  double floor2 = 0.0;  // 1e-30 |A|_F^2
  for (int pr = lane; pr < s.npairs; pr += 32) floor2 += *cluster.map_shared_rank(part + pr % ppc, pr / ppc);
  floor2 = 1e-30 * warp_sum(floor2);
  const double tol2 = fmax(1e-30, 4.930380657631324e-32 * (double)m);
  unsigned int* flags = cluster.map_shared_rank(above, 0);
  // Columns of round g (counted over all sweeps) lie in buffer g & 1. A neighbour
  // writes a buffer again only after it has the columns sent from it, so
  // the two buffers need no other guard.
  unsigned g = 0;
  bool lost = false;  // a wait ran out: no more waits, the caller sees an error
  auto arrived = [&]() {
    if (g == 0) return;
    const unsigned bar = my_full + 8 * (g & 1);
    if (!lost) lost = !svd_wait(bar, ((g - 1) >> 1) & 1);
    if (lane == 0) svd_arm(bar, ld);  // for round g + 2
  };
  for (int sweep = 0; sweep < 30; ++sweep) {
    bool any = false;
    for (int r = 0; r < s.rounds; ++r, ++g) {
      if (!active) continue;
      arrived();
      const int from = (g & 1) * 2 * ld, to = 2 * ld - from;
      const double *bx = cx + from, *by = cy + from;
      double x[C], y[C], vx[C], vy[C];
      double al = bx[ld - 1], be = by[ld - 1], ga = 0.0;
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const int e = lane + 32 * k;
        x[k] = y[k] = vx[k] = vy[k] = 0.0;
        if (e < m) {
          x[k] = bx[e];
          y[k] = by[e];
        }
        if (e < d) {
          vx[k] = bx[m + e];
          vy[k] = by[m + e];
        }
      }
      if (r == 0) {
        al = be = 0.0;
#pragma unroll
        for (int k = 0; k < C; ++k)
          if (32 * k < m) {
            asm volatile("" ::: "memory");
            al = fma(x[k], x[k], al);
            be = fma(y[k], y[k], be);
          }
        al = warp_sum(al);
        be = warp_sum(be);
      }
      const SvdNorms norms = svd_norms(al, be, floor2, tol2);
#pragma unroll
      for (int k = 0; k < C; ++k)
        if (32 * k < m) {
          asm volatile("" ::: "memory");
          ga = fma(x[k], y[k], ga);
        }
      ga = warp_sum(ga);
      SvdRotation rot;
      if (svd_angle(norms, al, be, ga, tol2, rot)) {  // never with a column past d: its norm is 0
        any = true;
#pragma unroll
        for (int k = 0; k < C; ++k) {
          if (32 * k < m) {
            asm volatile("" ::: "memory");
            svd_rotate(rot, x[k], y[k]);
          }
          if (32 * k < d) {
            asm volatile("" ::: "memory");
            svd_rotate(rot, vx[k], vy[k]);
          }
        }
        al = fma(-rot.t, ga, al);
        be = fma(rot.t, ga, be);
      }
      const unsigned ox = tx + 8 * to, oy = ty + 8 * to, fx = tx_full + 8 * (~g & 1), fy = ty_full + 8 * (~g & 1);
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const int e = lane + 32 * k;
        if (e < m) {
          svd_send(ox + 8 * e, x[k], fx);
          svd_send(oy + 8 * e, y[k], fy);
        }
        if (e < d) {
          svd_send(ox + 8 * (m + e), vx[k], fx);
          svd_send(oy + 8 * (m + e), vy[k], fy);
        }
      }
      if (lane == 0) {
        svd_send(ox + 8 * (ld - 1), al, fx);
        svd_send(oy + 8 * (ld - 1), be, fy);
      }
    }
    lost = __any_sync(0xffffffffu, lost);
    // above[sweep % 3] of CTA 0, as in the grid-wide kernel; bit 1: give up
    if (lane == 0 && (any || lost)) atomicOr(flags + sweep % 3, lost ? 2u : 1u);
    cluster.sync();
    const unsigned int more = *(volatile unsigned int*)(flags + sweep % 3);
    if (rank == 0 && threadIdx.x == 0) above[(sweep + 2) % 3] = 0u;
    if (more & 2u) lost = true;
    if (more != 1u) break;
  }
  if (active) arrived();
  if (lost) {
    atomicOr(reinterpret_cast<unsigned int*>(work) + SVD_LOST, 1u);
    __nanosleep(100000);  // columns that nobody awaits any more may still be on their way
  }
  cluster.sync();  // no CTA leaves while its flags or columns are in use
  if (active)      // a whole number of cycles: every column is back at its first position
    for (int h = 0; h < 2; ++h) {
      const double* c = (h ? cy : cx) + (g & 1) * 2 * ld;
      const int col = h ? py : px;
      if (col >= d) continue;
      for (int e = lane; e < m; e += 32) work[s.a_off + (long long)col * m + e] = c[e];
      for (int e = lane; e < d; e += 32) work[s.v_off + (long long)col * d + e] = c[m + e];
    }
}

__global__ void __launch_bounds__(32 * SVD_CLUSTER_WARPS, 1)
svd_cluster_kernel(const SvdBlock* __restrict__ sb, const double* __restrict__ psi, double* __restrict__ work, int left) {
  extern __shared__ double svd_cols[];
  __shared__ double part[SVD_CLUSTER_WARPS];
  __shared__ unsigned int above[3];
  __shared__ unsigned long long full[2 * SVD_CLUSTER_WARPS];  // mbarriers: the columns of a warp's buffers
  const SvdBlock s = sb[sb[blockIdx.x / SVD_CLUSTER].order];
  auto run = [&](auto c) { svd_cluster_block<decltype(c)::value>(s, psi, work, left, svd_cols, part, above, full); };
  const int chunks = ((s.m > s.d ? s.m : s.d) + 31) / 32;
  if (chunks <= 1)
    run(std::integral_constant<int, 1>());
  else if (chunks <= 2)
    run(std::integral_constant<int, 2>());
  else if (chunks <= 3)
    run(std::integral_constant<int, 3>());
  else if (chunks <= 4)
    run(std::integral_constant<int, 4>());
  else
    run(std::integral_constant<int, SVD_REG>());
}

// The other blocks: columns in global memory, one pair per warp over the whole
// grid, one CTA per SM in the barrier and consecutive pairs on different SMs.
__global__ void __launch_bounds__(SVD_THREADS, 1)
svd_jacobi_kernel(const SvdBlock* __restrict__ sb, int nb, int total_pairs, int max_rounds, double* __restrict__ work,
                  double* __restrict__ nrm, const double* __restrict__ fro, unsigned int* __restrict__ above) {
  namespace cgp = cooperative_groups;
  cgp::grid_group grid = cgp::this_grid();
  const int lane = threadIdx.x & 31;
  const int warp = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;  // consecutive pairs on different SMs
  const int nwarps = (blockDim.x >> 5) * gridDim.x;
  auto block_of = [&](int pid) {  // last b with pair0 <= pid
    int lo = 0, hi = nb - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (sb[mid].pair0 <= pid) lo = mid;
      else hi = mid - 1;
    }
    return sb[lo];
  };
  const SvdBlock first = block_of(min(warp, total_pairs - 1));
  const double floor_first = 1e-30 * fro[first.w_off];
  for (int sweep = 0; sweep < 30; ++sweep) {
    bool any = false;
    for (int round = 0; round < max_rounds; ++round) {
      for (int pid = warp; pid < total_pairs; pid += nwarps) {
        const SvdBlock s = pid == warp ? first : block_of(pid);
        const int i = pid - s.pair0;
        if (i >= s.npairs || s.rounds <= 0) continue;
        const double floor2 = pid == warp ? floor_first : 1e-30 * fro[s.w_off];
        any |= svd_pair(s, i, round % s.rounds, round == 0, work, nrm, floor2, lane);
      }
      grid.sync();
    }
    // above[sweep % 3]: raised in this sweep, read after the barrier, cleared for reuse two sweeps later
    if (lane == 0 && any) atomicOr(above + sweep % 3, 1u);
    grid.sync();
    const bool more = *(volatile unsigned int*)(above + sweep % 3) != 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) above[(sweep + 2) % 3] = 0u;
    if (!more) break;
  }
}

// singular values (column norms) sorted descending (ties by index); Q row r,
// column rank(c) = V[c][r]
__global__ void svd_finish_kernel(const SvdBlock* __restrict__ sb, int nb, const double* __restrict__ work,
                                  double* __restrict__ Q, double* __restrict__ w) {
  extern __shared__ double sig[];
  for (int b = blockIdx.x; b < nb; b += gridDim.x) {
    const SvdBlock s = sb[b];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int c = wid; c < s.d; c += nw) {
      const double* a = work + s.a_off + (long long)c * s.m;
      double v = 0.0;
      for (int e = lane; e < s.m; e += 32) v = fma(a[e], a[e], v);
      v = warp_sum(v);
      if (lane == 0) sig[c] = v;
    }
    __syncthreads();
    for (int c = threadIdx.x; c < s.d; c += blockDim.x) {
      const double v = sig[c];
      int rank = 0;
      for (int j = 0; j < s.d; ++j) rank += (sig[j] > v) || (sig[j] == v && j < c);
      w[s.w_off + rank] = v;
      for (int r = 0; r < s.d; ++r) Q[s.q_off + (long long)r * s.d + rank] = work[s.v_off + (long long)c * s.d + r];
    }
    __syncthreads();
  }
}

}  // namespace

void launch_blocking(const BlockingDev& d, cudaStream_t st) {
  if (d.ndst <= 0) return;
  const int grid = d.ndst < 152 * 64 ? d.ndst : 152 * 64;
  blocking_kernel<<<grid, BLK_THREADS, 0, st>>>(d);
}

void launch_opcomb(const double* src, const long long* xoff, const double* coef, const CombClass* cls, int ncls,
                   int ntiles, double* dst, cudaStream_t st) {
  if (ntiles <= 0) return;
  const int grid = ntiles < 152 * 2 * 8 ? ntiles : 152 * 2 * 8;
  opcomb_kernel<<<grid, 256, 0, st>>>(src, xoff, coef, cls, ncls, ntiles, dst);
}

void launch_bgemm(const double* A, const double* B, double* C, const GJob* jobs, int njobs, cudaStream_t st) {
  if (njobs <= 0) return;
  bgemm_kernel<<<njobs < 152 * 16 ? njobs : 152 * 16, 256, 0, st>>>(A, B, C, jobs, njobs);
}

void launch_orthonormalize(double* store, const GramBlock* gb, int nb, cudaStream_t st) {
  if (nb <= 0) return;
  orthonormalize_kernel<<<nb < 65535 ? nb : 65535, 256, 0, st>>>(store, gb, nb);
}

void launch_take_columns(const double* Q, const TakeBlock* tb, int nb, double* dst, cudaStream_t st) {
  if (nb <= 0) return;
  dim3 grid(8, nb < 65535 ? nb : 65535);
  take_columns_kernel<<<grid, 256, 0, st>>>(Q, tb, nb, dst);
}

}  // namespace dmrg

namespace dmrg {

bool svd_cluster_fits(int d, int m) {
  const int npairs = (d + 1) / 2, ppc = (npairs + SVD_CLUSTER - 1) / SVD_CLUSTER;
  static_assert((32 * SVD_REG / 2 + SVD_CLUSTER - 1) / SVD_CLUSTER == SVD_CLUSTER_WARPS, "a warp for every pair of a CTA");
  return d >= 1 && d <= 32 * SVD_REG && m <= 32 * SVD_REG &&
         (size_t)ppc * 4 * (m + d + 1) * sizeof(double) <= SVD_CLUSTER_SMEM;
}

// Launch of n clusters; the kernel's attributes are set on the way.
static cudaLaunchConfig_t cluster_config(int n, int warps, int smem, cudaStream_t st, cudaLaunchAttribute& at) {
  set_max_dynamic_smem((const void*)svd_cluster_kernel, (int)SVD_CLUSTER_SMEM);
  const cudaError_t e = cudaFuncSetAttribute((const void*)svd_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) throw Error(DMRG_ECUDA, std::string("cudaFuncSetAttribute(cluster size): ") + cudaGetErrorString(e));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)n * SVD_CLUSTER);
  cfg.blockDim = dim3(32u * warps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = SVD_CLUSTER;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cfg;
}

bool svd_clusters_launch() {
  int n = 0;
  try {
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = cluster_config(1, SVD_CLUSTER_WARPS, (int)SVD_CLUSTER_SMEM, nullptr, at);
    if (cudaOccupancyMaxActiveClusters(&n, svd_cluster_kernel, &cfg) != cudaSuccess) n = 0;
  } catch (const Error&) {
  }
  if (n <= 0) cudaGetLastError();  // the answer, not an error of the caller's
  return n > 0;
}

SvdShape plan_svd_blocks(const std::vector<SvdDims>& dims, bool clusters, std::vector<SvdBlock>& sb) {
  SvdShape s;
  s.nb = (int)dims.size();
  sb.resize(dims.size());
  std::vector<int> cl;  // blocks of the cluster kernel
  for (int b = 0; b < s.nb; ++b) {
    const int d = dims[b].d, m = dims[b].m, dp = d + (d & 1);
    const bool fits = clusters && svd_cluster_fits(d, m);
    sb[b] = {dims[b].psi_off, s.q_elems, s.w_elems, s.work_elems, s.work_elems + (long long)d * m, d, m,
             s.grid_pairs, dp / 2, dp - 1, fits ? 1 : 0, 0, 0};
    if (fits) {
      const int ppc = (dp / 2 + SVD_CLUSTER - 1) / SVD_CLUSTER;
      s.cluster_warps = std::max(s.cluster_warps, ppc);
      s.cluster_smem = std::max(s.cluster_smem, (int)(ppc * 4 * (m + d + 1) * sizeof(double)));
      cl.push_back(b);
    } else {
      s.grid_pairs += dp / 2;
      s.grid_rounds = std::max(s.grid_rounds, dp - 1);
    }
    s.max_d = std::max(s.max_d, d);
    s.work_elems += (long long)d * m + (long long)d * d;
    s.q_elems += (long long)d * d;
    s.w_elems += d;
  }
  std::stable_sort(cl.begin(), cl.end(), [&](int a, int b) { return sb[a].d > sb[b].d; });  // the longest first
  for (size_t i = 0; i < cl.size(); ++i) sb[i].order = cl[i];
  s.n_cluster = (int)cl.size();
  return s;
}

void launch_svd_blocks(const double* psi, const SvdBlock* sb, const SvdShape& shape, double* Q, double* w, double* work,
                       bool left, int n_sm, cudaStream_t st) {
  int nb = shape.nb, total_pairs = shape.grid_pairs, max_rounds = shape.grid_rounds;
  if (nb <= 0) return;
  const size_t sig_bytes = (size_t)shape.max_d * sizeof(double);
  if (sig_bytes > 48 * 1024) set_max_dynamic_smem((const void*)svd_finish_kernel, (int)sig_bytes);
  if (cudaMemsetAsync(work, 0, 64, st) != cudaSuccess) return;  // the flags of both kernels; the caller's cudaGetLastError reports it
  if (shape.n_cluster > 0) {
    cudaLaunchAttribute at;
    cudaLaunchConfig_t cfg = cluster_config(shape.n_cluster, shape.cluster_warps, shape.cluster_smem, st, at);
    if (cudaLaunchKernelEx(&cfg, svd_cluster_kernel, sb, psi, work, left ? 1 : 0) != cudaSuccess) return;
  }
  if (total_pairs > 0 && max_rounds > 0) {
    dim3 grid(32, nb < 65535 ? nb : 65535);
    svd_setup_kernel<<<grid, 256, 0, st>>>(psi, sb, nb, work, left ? 1 : 0);
    unsigned int* above = reinterpret_cast<unsigned int*>(work);  // first words of work
    svd_norm_kernel<<<nb < 65535 ? nb : 65535, 256, 0, st>>>(sb, nb, work, w);
    const double* fro = w;
    double* nrm = Q;  // Q is written by the finish kernel: until then the squared column norms, d per block
    void* args[] = {(void*)&sb,   (void*)&nb,  (void*)&total_pairs, (void*)&max_rounds,
                    (void*)&work, (void*)&nrm, (void*)&fro,         (void*)&above};
    const cudaError_t e = cudaLaunchCooperativeKernel((void*)svd_jacobi_kernel, dim3(n_sm), dim3(SVD_THREADS), args, 0, st);
    if (e != cudaSuccess) return;  // the caller's cudaGetLastError reports it
  }
  svd_finish_kernel<<<nb < 65535 ? nb : 65535, 256, sig_bytes, st>>>(sb, nb, work, Q, w);
}

}  // namespace dmrg
