// FP64 sigma = H_eff . psi as fused back-to-back GEMMs per (term, sector).
//
// Sec. II.D-E: sigma is a sum over NC operator pairs (Eq. hpsi-thread),
// each split into dense products over symmetry sectors, with the two
// parallel levels (terms, sectors) collapsed into one flat task list. Here a
// persistent CTA takes one work item = (output block tile, run of tasks) and
// accumulates, for every task,
//     S[r0:r0+32, c0:c0+nc] += scale * (X_L[r0:, :] psi_b) X_R[c0:, :]^T
// chunk by chunk (32 columns of the intermediate at a time, the intermediate
// never leaves a warp's registers), then writes its partial tile to a private
// scratch slot. A second kernel sums each output tile's slots in fixed order
// (Sec. II.D's final reduction), so sigma is bitwise deterministic whatever
// the schedule of the items.
//
// The FP64 path is bound by the FP64 multiply-add rate, which on this GPU
// is the same for the FP64 tensor instruction (mma.sync m8n8k4 .f64: 256
// multiply-adds per warp instruction) and for scalar FMAs: about 1.9 FMAs per
// cycle and SM, so one such instruction occupies its SM sub-partition for
// about 540 cycles. The tensor form is used because its 8x8x4 granularity keeps
// padding small: every output tile, intermediate chunk and contraction is
// padded only to multiples of 8 (rows, columns) and 4 (k). At that rate a load
// straight from global memory (L1 / L2) into a fragment is never the limit, so
// nothing is staged in shared memory and no barrier stands between the warps:
// a warp owns rows of the tile and a share of the item's tasks, computes the
// intermediate of 32 columns in registers and feeds it to the second product
// from the registers it is in (below). Per sigma, against 8 warps sharing
// operands staged in shared memory with 4 barriers per 32 k steps: 9.6 us
// (before: 74) at K=8, M=64; 1.92 ms (2.84) at K=36, M=501, with the FP64 pipe
// busy 75% of one launch (blocks of 1-30 rows, padded to twice their
// multiply-adds); 22.9 ms (26.3) at K=54, M=1000; 635 ms (658) at K=108,
// M=2000.
#include <algorithm>
#include <mutex>
#include <set>
#include <string>
#include <tuple>

#include "../../include/dmrg.h"
#include "kernels.h"

namespace dmrg {

namespace {

constexpr int NW = 4;             // warps per CTA
constexpr int NT = 32 * NW;
constexpr int CTAS_PER_SM = 2;
constexpr int NX = 4;             // 8-column groups of the intermediate per chunk
constexpr int WARP_ELEMS = 2048;  // output elements of a warp: 16 x 128 or 8 x 256
static_assert(F64_TM == 32 && F64_TN == 256, "warp layouts of a tile");

struct Smem {
  double part[NW][WARP_ELEMS];  // the warps' sums of an item
  int item;
};

// D = A(8x4) B(4x8) + D; lane (g = lane/4, c = lane%4) holds A[g][c],
// B[c][g] and D[g][2c], D[g][2c+1].
__device__ __forceinline__ void dmma(double (&d)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};\n"
               : "+d"(d[0]), "+d"(d[1])
               : "d"(a), "d"(b));
}

// s += sum of the tasks t0, t0 + step, ... < t1 on rows r0 .. r0 + 8 nrs - 1
// (nrs <= RG groups of 8) and columns c0 .. c0 + 8 ncs - 1 (ncs <= CG groups)
// of output block ob. Rows and columns past the block are computed from its
// last row or column (never stored, so only finite or not matters to
// themselves); contraction indices past the end enter as zeros on both sides.
//
// The second product contracts the columns of X. Its A fragment wants X[g][k]
// for four k in lane order c = 0..3, and the lane already holds X[g][2c] and
// X[g][2c + 1] of every 8-column group: the order of a contraction is free, so
// one instruction takes the columns 2c and the next the columns 2c + 1, with
// the right operator's columns loaded in the same order, and X never moves.
// Only a last group of 2-4 valid columns is brought into natural order by
// shuffles, where one instruction then replaces two.
template <int RG, int CG>
__device__ __forceinline__ void run_tasks(const SigmaDev& a, const PsiBlock& ob, int r0, int nrs, int c0, int ncs,
                                          int t0, int t1, int step, int lane, double (&s)[RG][CG][2]) {
  const int g = lane >> 2, c = lane & 3;
  const int mo = ob.mL, no = ob.mR;
  int row[RG];
#pragma unroll
  for (int r = 0; r < RG; ++r) row[r] = min(r0 + 8 * r + g, mo - 1);
  const int col_first = min(c0 + g, no - 1), col_last = min(c0 + 8 * (ncs - 1) + g, no - 1);
  Task nx{};
  if (t0 < t1) nx = a.tasks[t0];
  for (int t = t0; t < t1; t += step) {
    const Task tk = nx;
    if (t + step < t1) nx = a.tasks[t + step];  // in flight during this task
    const PsiBlock ib = a.blocks[tk.in_blk];
    const int m = ib.mL, n = ib.mR;
    const double* __restrict__ psib = a.psi + ib.off;
    const bool tA = tk.flags & 1, tB = tk.flags & 2;
    // element (i, k) of the left block used: la[i * ars + k * aks]; of the right one likewise
    const long long ars = tA ? 1 : m, aks = tA ? mo : 1, rrs = tB ? 1 : n, rks = tB ? no : 1;
    const double* __restrict__ la = a.store + (tk.aoff < 0 ? 0 : tk.aoff);
    const double* __restrict__ lr = a.store + (tk.boff < 0 ? 0 : tk.boff);
    for (int nc0 = 0; nc0 < n; nc0 += 8 * NX) {
      const int nleft = n - nc0, nxs = min(NX, (nleft + 7) >> 3);
      // ---- X = scale * L[rows, :] psi_b[:, nc0 .. nc0 + 8 nxs)
      double x[RG][NX][2];
      if (tk.aoff < 0) {
#pragma unroll
        for (int r = 0; r < RG; ++r)
#pragma unroll
          for (int q = 0; q < NX; ++q)
#pragma unroll
            for (int h = 0; h < 2; ++h)
              x[r][q][h] = psib[(long long)row[r] * n + min(nc0 + 8 * q + 2 * c + h, n - 1)];
      } else {
#pragma unroll
        for (int r = 0; r < RG; ++r)
#pragma unroll
          for (int q = 0; q < NX; ++q) x[r][q][0] = x[r][q][1] = 0.0;
        const double* pa[RG];
#pragma unroll
        for (int r = 0; r < RG; ++r) pa[r] = la + row[r] * ars + c * aks;
        const double* pb = psib + (long long)c * n;
        int ob_[NX];
#pragma unroll
        for (int q = 0; q < NX; ++q) ob_[q] = min(nc0 + 8 * q + g, n - 1);
        auto kstep = [&](bool valid) {
          double av[RG], bv[NX];
#pragma unroll
          for (int r = 0; r < RG; ++r) av[r] = (valid && r < nrs) ? __ldg(pa[r]) : 0.0;
#pragma unroll
          for (int q = 0; q < NX; ++q) bv[q] = (valid && q < nxs) ? __ldg(pb + ob_[q]) : 0.0;
#pragma unroll
          for (int q = 0; q < NX; ++q)
            if (q < nxs)
#pragma unroll
              for (int r = 0; r < RG; ++r)
                if (r < nrs) dmma(x[r][q], av[r], bv[q]);
        };
        for (int k = 0; k + 4 <= m; k += 4) {
          kstep(true);
#pragma unroll
          for (int r = 0; r < RG; ++r) pa[r] += 4 * aks;
          pb += 4ll * n;
        }
        if (m & 3) kstep(c < (m & 3));
      }
      if (tk.scale != 1.0) {
#pragma unroll
        for (int r = 0; r < RG; ++r)
#pragma unroll
          for (int q = 0; q < NX; ++q)
#pragma unroll
            for (int h = 0; h < 2; ++h) x[r][q][h] *= tk.scale;
      }
      if (nleft < 8 * NX) {  // columns past the block
#pragma unroll
        for (int r = 0; r < RG; ++r)
#pragma unroll
          for (int q = 0; q < NX; ++q)
#pragma unroll
            for (int h = 0; h < 2; ++h)
              if (8 * q + 2 * c + h >= nleft) x[r][q][h] = 0.0;
      }
      // ---- S += X R[columns, nc0 ..]^T
      if (tk.boff < 0) {  // identity: output column j is intermediate column j
#pragma unroll
        for (int j = 0; j < CG; ++j)
#pragma unroll
          for (int q = 0; q < NX; ++q)
            if (c0 + 8 * j == nc0 + 8 * q) {
#pragma unroll
              for (int r = 0; r < RG; ++r)
#pragma unroll
                for (int h = 0; h < 2; ++h) s[r][j][h] += x[r][q][h];
            }
        continue;
      }
#pragma unroll
      for (int q = 0; q < NX; ++q) {
        if (q >= nxs) break;
        const int left = nleft - 8 * q;        // valid columns of this group
        const bool natural = left >= 2 && left <= 4;
        double a0[RG], a1[RG];
        if (natural) {
#pragma unroll
          for (int r = 0; r < RG; ++r) {
            const int src = (lane & ~3) | (c >> 1);
            const double u = __shfl_sync(0xffffffffu, x[r][q][0], src), v = __shfl_sync(0xffffffffu, x[r][q][1], src);
            a0[r] = (c & 1) ? v : u;
            a1[r] = 0.0;
          }
        } else {
#pragma unroll
          for (int r = 0; r < RG; ++r) {
            a0[r] = x[r][q][0];
            a1[r] = x[r][q][1];
          }
        }
        const int k0 = nc0 + 8 * q + (natural ? c : 2 * c);  // this lane's first contraction column
        const bool two = !natural && left > 1;               // the columns 2c + 1 hold something
        const bool v0 = k0 < n, v1 = two && k0 + 1 < n;
        const double* p0 = lr + col_first * rrs + k0 * rks;
        const double* pl = lr + col_last * rrs + k0 * rks;
#pragma unroll
        for (int j = 0; j < CG; ++j) {
          if (j >= ncs) break;
          const double* p = j == ncs - 1 ? pl : p0 + 8ll * j * rrs;
          const double b0 = v0 ? __ldg(p) : 0.0, b1 = v1 ? __ldg(p + rks) : 0.0;
#pragma unroll
          for (int r = 0; r < RG; ++r)
            if (r < nrs) dmma(s[r][j], a0[r], b0);
          if (two) {
#pragma unroll
            for (int r = 0; r < RG; ++r)
              if (r < nrs) dmma(s[r][j], a1[r], b1);
          }
        }
      }
    }
  }
}

// One item on one CTA: RG x CG register tiles, rows [8 RG i, ..) of the tile
// on row slice i, and the item's tasks shared by NW / n_rows warps per row
// slice. `flip` swaps the row slices between the two resident CTAs, so that a
// short last slice does not leave the same SM sub-partitions idle in both.
template <int RG, int CG>
__device__ __forceinline__ void run_item(const SigmaDev& a, const Item& it, const PsiBlock& ob, bool flip, Smem& sm) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, c = lane & 3;
  int n_rows = (it.nrows + 8 * RG - 1) / (8 * RG);  // 1, 2 or 4 (3 leaves a warp idle)
  if (n_rows == 3) n_rows = 4;
  const int n_slices = NW / n_rows;
  const int w = flip ? NW - 1 - warp : warp;
  const int rs = w / n_slices, sl = w - rs * n_slices;
  const int r0 = 8 * RG * rs, nr = min(8 * RG, it.nrows - r0);
  double s[RG][CG][2];
#pragma unroll
  for (int r = 0; r < RG; ++r)
#pragma unroll
    for (int j = 0; j < CG; ++j) s[r][j][0] = s[r][j][1] = 0.0;
  if (nr > 0)
    run_tasks<RG, CG>(a, ob, it.r0 + r0, (nr + 7) >> 3, it.c0, (it.ncols + 7) >> 3, it.t_begin + sl, it.t_end,
                      n_slices, lane, s);
  double* out = a.scratch + it.slot;
  if (n_slices == 1) {  // the warp holds its rows' sums
#pragma unroll
    for (int r = 0; r < RG; ++r)
#pragma unroll
      for (int j = 0; j < CG; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int row = 8 * r + g, col = 8 * j + 2 * c + h;
          if (row < nr && col < it.ncols) out[(long long)(r0 + row) * it.ncols + col] = s[r][j][h];
        }
    return;
  }
  // add the slices of every row slice in order
  double* mine = sm.part[rs * n_slices + sl];
#pragma unroll
  for (int r = 0; r < RG; ++r)
#pragma unroll
    for (int j = 0; j < CG; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = 8 * r + g, col = 8 * j + 2 * c + h;
        if (row < nr && col < it.ncols) mine[row * it.ncols + col] = s[r][j][h];
      }
  __syncthreads();
  for (int e = threadIdx.x; e < it.nrows * it.ncols; e += NT) {
    const int i = e / (8 * RG * it.ncols), le = e - i * (8 * RG * it.ncols);
    double v = sm.part[i * n_slices][le];
    for (int k = 1; k < n_slices; ++k) v += sm.part[i * n_slices + k][le];
    out[e] = v;
  }
}

__global__ void __launch_bounds__(NT, CTAS_PER_SM)
sigma_f64_kernel(SigmaDev a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
  const bool flip = blockIdx.x >= gridDim.x / 2;
  for (;;) {
    if (threadIdx.x == 0) {
      unsigned k = atomicAdd(a.counter, 1u);
      sm.item = (k < (unsigned)a.n_items) ? a.schedule[k] : -1;
    }
    __syncthreads();
    const int it_idx = sm.item;
    __syncthreads();  // the slot and sm.part are rewritten from here on
    if (it_idx < 0) return;
    const Item it = a.items[it_idx];
    const PsiBlock ob = a.blocks[it.out];
    // tiles up to 128 columns: 16 x 128 per warp; wider: 8 x 256, so that the
    // intermediate is still computed once per row
    if (it.ncols <= 128)
      run_item<2, 16>(a, it, ob, flip, sm);
    else
      run_item<1, 32>(a, it, ob, flip, sm);
  }
}

// Work lists whose output tiles are one item of one task each (the
// transformation of Eq. op-trans: 1e3-1e6 tiles): the warps of a CTA share the
// 16 x 128 pieces of NW items at a time (each piece one warp's register tile)
// and write them straight into sigma: no partial tiles, no reduction pass, one
// counter access per NW items. (An item per warp, whatever its size, left a
// tail of single warps on the widest sectors.) The transformations of two
// sweeps at K=24, M=300 take 87 ms, mostly host lists (90 ms with partial tiles
// as large as the store written and reduced).
__global__ void __launch_bounds__(NT, CTAS_PER_SM)
sigma_f64_direct_kernel(SigmaDev a) {
  __shared__ int next;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
  for (;;) {
    if (threadIdx.x == 0) next = (int)min(atomicAdd(a.counter, (unsigned)NW), 0x7ffffff0u);
    __syncthreads();
    const int q0 = next;
    __syncthreads();
    if (q0 >= a.n_items) return;
    int p = warp;  // this warp's next piece, counted from the current item's first
    for (int q = q0; q < min(q0 + NW, a.n_items); ++q) {
      const Item it = a.items[a.schedule[q]];
      const int n_cols = (it.ncols + 127) >> 7, n_pieces = ((it.nrows + 15) >> 4) * n_cols;
      if (p < n_pieces) {
        const PsiBlock ob = a.blocks[it.out];
        double* out = a.sigma + ob.off + (long long)it.r0 * ob.mR + it.c0;
        for (; p < n_pieces; p += NW) {
          const int r0 = 16 * (p / n_cols), c0 = 128 * (p % n_cols);
          const int nr = min(16, it.nrows - r0), nc = min(128, it.ncols - c0);
          double s[2][16][2];
#pragma unroll
          for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int j = 0; j < 16; ++j) s[r][j][0] = s[r][j][1] = 0.0;
          run_tasks<2, 16>(a, ob, it.r0 + r0, (nr + 7) >> 3, it.c0 + c0, (nc + 7) >> 3, it.t_begin, it.t_end, 1, lane,
                           s);
#pragma unroll
          for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int j = 0; j < 16; ++j)
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const int row = 8 * r + g, col = 8 * j + 2 * c + h;
                if (row < nr && col < nc) out[(long long)(r0 + row) * ob.mR + c0 + col] = s[r][j][h];
              }
        }
      }
      p -= n_pieces;
    }
  }
}

// Sum of every output tile's partial tiles, in item order: blockIdx.x the
// group, blockIdx.y a run of RED_THREADS elements of its tile (the work lists
// give the items of a group consecutive slots of one tile each, so element e
// of the k-th item is at slot + k * n + e). Bound by latency: a tile has 5-30
// partials of a few thousand elements. One CTA per group walking its items
// one load at a time took 402 us at K=76, M=2000 (104 groups, BF16X3) and
// 292 us at K=16, M=150 (31 groups); spreading the elements over CTAs, with
// RED_UNROLL loads in flight per thread and the same order of additions,
// takes 21 us and 19 us.
constexpr int RED_THREADS = 128;
constexpr int RED_UNROLL = 8;
__global__ void __launch_bounds__(RED_THREADS) reduce_kernel(SigmaDev a) {
  const Group g = a.groups[blockIdx.x];
  const int n = g.nrows * g.ncols, ni = g.i_end - g.i_begin;
  const PsiBlock ob = a.blocks[g.out];
  const double* __restrict__ part = a.scratch + a.items[g.i_begin].slot;
  for (int e = blockIdx.y * RED_THREADS + threadIdx.x; e < n; e += gridDim.y * RED_THREADS) {
    const double* __restrict__ src = part + e;
    double acc = 0.0;
    int k = 0;
    for (; k + RED_UNROLL <= ni; k += RED_UNROLL) {
      double v[RED_UNROLL];
#pragma unroll
      for (int u = 0; u < RED_UNROLL; ++u) v[u] = src[(long long)(k + u) * n];
#pragma unroll
      for (int u = 0; u < RED_UNROLL; ++u) acc += v[u];
    }
    for (; k < ni; ++k) acc += src[(long long)k * n];
    const int r = e / g.ncols, c = e - r * g.ncols;
    a.sigma[ob.off + (long long)(g.r0 + r) * ob.mR + g.c0 + c] = acc;
  }
}

}  // namespace

void set_max_dynamic_smem(const void* fn, int bytes) {
  static std::mutex mu;
  static std::set<std::tuple<const void*, int, int>> done;  // (kernel, device, bytes)
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) throw Error(DMRG_ECUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
  std::lock_guard<std::mutex> lk(mu);
  if (done.count({fn, dev, bytes})) return;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess)
    throw Error(DMRG_ECUDA, std::string("cudaFuncSetAttribute(max dynamic shared memory): ") + cudaGetErrorString(e));
  done.insert({fn, dev, bytes});
}

void launch_sigma_f64_direct(const SigmaDev& a, int n_sm, cudaStream_t st) {
  if (a.n_items < 1) return;
  int grid = CTAS_PER_SM * n_sm;
  if (grid > (a.n_items + NW - 1) / NW) grid = (a.n_items + NW - 1) / NW;
  sigma_f64_direct_kernel<<<grid, NT, 0, st>>>(a);
}

void launch_sigma_f64(const SigmaDev& a, int n_sm, cudaStream_t st) {
  const int smem = (int)sizeof(Smem);
  set_max_dynamic_smem((const void*)sigma_f64_kernel, smem);
  int grid = CTAS_PER_SM * n_sm;
  if (grid > a.n_items) grid = a.n_items;
  if (grid < 1) grid = 1;
  sigma_f64_kernel<<<grid, NT, smem, st>>>(a);
}

void launch_reduce(const SigmaDev& a, cudaStream_t st) {
  if (a.n_groups < 1 || a.max_tile < 1) return;
  // a CTA per run of elements until that fills the GPU many times over (a
  // plan has one group per output tile: a few for small bonds, thousands for large ones)
  int ny = (a.max_tile + RED_THREADS - 1) / RED_THREADS;
  ny = std::min(ny, std::max(1, 152 * 64 / a.n_groups));
  const dim3 grid((unsigned)a.n_groups, (unsigned)ny);
  reduce_kernel<<<grid, RED_THREADS, 0, st>>>(a);
}

}  // namespace dmrg
