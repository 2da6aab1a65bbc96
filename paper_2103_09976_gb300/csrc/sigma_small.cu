// Products of small classes with warp-level matrix instructions (part of the
// mixed-precision sigma, Sec. II.D-E: the same (term, sector) products as the
// tensor-core kernel, for the classes whose output tile and psi block are all at
// most TC_SMALL_MAX wide).
//
// A tcgen05 instruction is at least 128 x 16 x 16, so a product of 8x8 or
// 16x16 blocks would use it by a few percent, and such products are most of
// the (term, block) pairs of a middle bond while carrying about 1% of the
// flops. Here one warp computes one term at a time,
//     sigma[tile] += c * (L psi_b) R^T,
// with mma.sync (16 x 8 x 16), whose granularity fits. The split store's 8x8
// tiles are its fragments: lane l of a warp needs bytes 4l .. 4l+3 of a tile's
// slice, so operands go from global memory to registers with 128-byte coalesced
// loads and no shared memory; a transposed use transposes the fragments
// (movmatrix). psi's fragments stay in registers while the block is the same.
// The accumulators of X = L psi have the layout of the second product's left
// fragments, so X only has to be split again.
//
// Arithmetic: FP32 accumulation of slice products, the error of FP32 multiply-adds
// on the summed slices or less (mma_step). The fp16 split (hi + lo) takes all four
// products in the first product and, with X as three fp16 slices, five in the second
// (lo x the third slice, below 2^-33, is left out); every row of X is scaled so that
// its largest element fills the range of fp16 (row_scales). The bf16 split (hi + mid +
// lo) takes the six products above 2^-24 in both, X as three bf16 slices; what is left
// out is below 2^-25. Terms of a warp are summed in FP32 over groups of 8, groups in
// float-float (48 bits), warps in FP64 in warp order, so the result does not depend on
// scheduling.
//
// Bound by instruction issue (<= 16: 65% of issue slots) and load latency (<= 32:
// 12-16 warps per SM of 128-162 registers); a term of 16 x 16 blocks reads 2-3 KB
// for 18-24 matrix instructions. So a warp takes 16 rows (a term of more rows is
// shared by two), CTAs are 4 warps, items come from a counter, the next term's
// record is loaded a term ahead and its L and R before psi and the first product.
// Both kernels per sigma, against FP32 multiply-adds from shared memory: 1.63 ->
// 0.92 ms at K=108, M=2000 (FP16X2), 0.74 -> 0.39 ms at K=54, M=1000 (BF16X2), 63
// -> 46 us at K=24, M=250.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "kernels.h"

namespace dmrg {

namespace {

// D: size class; NT 8-wide tiles per side, NW warps per CTA, MINB CTAs per SM
template <int D, bool F16>
struct SmallCfg;
template <bool F16>
struct SmallCfg<16, F16> {
  static constexpr int NT = 2, NW = 4, MINB = F16 ? 7 : 6;
};
template <bool F16>
struct SmallCfg<32, F16> {
  static constexpr int NT = 4, NW = 4, MINB = F16 ? 4 : 3;
};
static_assert(TC_SMALL_MAX == 32 && TC_SMALL_MID == 16, "size classes");

// d += a b, 16 x 8 x 16: lane (g = lane / 4, c = lane % 4) holds d[g][2c], d[g][2c+1], d[g+8][..]
template <bool F16>
__device__ __forceinline__ void mma16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  if (F16)
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
  else
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// transpose of an 8x8 fragment
__device__ __forceinline__ uint32_t trans8(uint32_t x) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(r) : "r"(x));
  return r;
}

// The NSL slices of the tile at byte offset `off` as fragments (zero when !valid).
template <int NSL>
__device__ __forceinline__ void load_tile(uint32_t (&f)[NSL], const unsigned char* __restrict__ base, int off,
                                          bool valid) {
  const uint32_t* p = reinterpret_cast<const uint32_t*>(base + off);
#pragma unroll
  for (int s = 0; s < NSL; ++s) f[s] = valid ? __ldg(p + 32 * s) : 0u;
}

// (x0, x1) as three slices, x = s[0] + s[1] + s[2]
template <bool F16>
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t (&s)[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (F16) {
      const __half2 h = __floats2half2_rn(x0, x1);
      s[k] = *reinterpret_cast<const uint32_t*>(&h);
      const float2 v = __half22float2(h);
      x0 -= v.x;
      x1 -= v.y;
    } else {
      const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
      s[k] = *reinterpret_cast<const uint32_t*>(&h);
      x0 -= __uint_as_float(s[k] << 16);
      x1 -= __uint_as_float(s[k] & 0xFFFF0000u);
    }
  }
}

// Slice pairs (A slice, B slice) of the two products, smallest first (the last pair is hi x hi).
template <bool F16>
struct Pairs;
template <>
struct Pairs<true> {  // first: 2 x 2 slices; second: X has 3
  static constexpr int N1 = 4, N2 = 5;
  __device__ static constexpr int a1(int p) { return p == 0 || p == 2 ? 1 : 0; }
  __device__ static constexpr int b1(int p) { return p <= 1 ? 1 : 0; }
  __device__ static constexpr int a2(int p) { return p == 0 ? 2 : p <= 2 ? 1 : 0; }
  __device__ static constexpr int b2(int p) { return p == 1 || p == 3 ? 1 : 0; }
};
template <>
struct Pairs<false> {  // hl, mm, lh, hm, mh, hh
  static constexpr int N1 = 6, N2 = 6;
  __device__ static constexpr int a1(int p) { return p == 1 || p == 4 ? 1 : p == 2 ? 2 : 0; }
  __device__ static constexpr int b1(int p) { return p == 0 ? 2 : p == 1 || p == 3 ? 1 : 0; }
  __device__ static constexpr int a2(int p) { return a1(p); }
  __device__ static constexpr int b2(int p) { return b1(p); }
};

// x[j] += a b[j] for the N tiles j < nj of one K step (x[j] = a b[j] when `first`);
// b(j, h, s): slice s of K tile h. The matrix instruction adds with truncation
// (measured: operands aligned to the largest exponent with two extra bits, the
// result cut to 24), so a sum left to it shrinks by up to a unit in the last place
// an instruction, always in one direction. Hence every K step has its own
// accumulator z, corrections first and hi x hi last, one cut at full size, and FP32
// additions, which round to nearest, join the steps. REST: z starts with hi x
// hi on top of its own negative, which gives what was cut off (to a quarter unit); the
// <= 16 class needs it, where FP32 multiply-adds round a few times only. Relative
// error of sigma against 64 bits (2-norm, 1e-7), one accumulator / these parts / FP32
// multiply-adds of the summed slices: bf16 slices 1.0 / 0.8 / 0.9 at K=8, M=60 (blocks up to 4
// wide), 1.0 / 0.8 / 1.0 at K=24, M=200 (10), 3.3 / 1.1 / 1.4 at K=36, M=500 (25); fp16 1.3 / 1.0 /
// 1.0, 1.2 / 0.9 / 1.2, 2.5 / 1.2 / 1.5. Time of a sigma, one accumulator and one scale for
// all X -> this: 806 -> 812 us at K=54, M=1000 (BF16X2), 7.45 -> 7.56 ms at K=108, M=2000 (FP16X2),
// launched without a graph.
template <bool F16, bool SECOND, bool REST, int NT, int NSA, class Frag>
__device__ __forceinline__ void mma_step(float (&x)[NT][4], bool first, int nj, const uint32_t (&a)[NSA][4],
                                         Frag&& b) {
  using P = Pairs<F16>;
  constexpr int NP = SECOND ? P::N2 : P::N1;
  if (!REST) {
    float z[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) z[j][e] = 0.0f;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const int as = SECOND ? P::a2(p) : P::a1(p), bs = SECOND ? P::b2(p) : P::b1(p);
#pragma unroll
      for (int j = 0; j < NT; ++j)
        if (j < nj) mma16<F16>(z[j], a[as], b(j, 0, bs), b(j, 1, bs));
    }
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) x[j][e] = first ? z[j][e] : x[j][e] + z[j][e];
    return;
  }
#pragma unroll
  for (int j = 0; j < NT; ++j)
    if (j == 0 || j < nj) {
      float z[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      mma16<F16>(z, a[0], b(j, 0, 0), b(j, 1, 0));
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        x[j][e] = first ? z[e] : x[j][e] + z[e];
        z[e] = -z[e];
      }
      mma16<F16>(z, a[0], b(j, 0, 0), b(j, 1, 0));
#pragma unroll
      for (int p = 0; p < NP - 1; ++p) {
        const int as = SECOND ? P::a2(p) : P::a1(p), bs = SECOND ? P::b2(p) : P::b1(p);
        mma16<F16>(z, a[as], b(j, 0, bs), b(j, 1, bs));
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) x[j][e] += z[e];
    }
}

// Powers of two 2^k (and 2^-k) that bring the largest |v| of each of the two rows of
// four lanes into [2^14, 2^15) (as near as FP32's exponents allow). Only the
// exponents matter, so both rows' go through the two shuffles in one word.
__device__ __forceinline__ void row_scales(float m0, float m1, float (&up)[2], float (&down)[2]) {
  unsigned m = __float_as_uint(m0) >> 23 | (__float_as_uint(m1) >> 23) << 16;
  m = __vmaxu2(m, __shfl_xor_sync(0xffffffffu, m, 1));
  m = __vmaxu2(m, __shfl_xor_sync(0xffffffffu, m, 2));
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const unsigned e = min(max((m >> (16 * h)) & 0xff, 15u), 240u) << 23;  // |v| < 2^(e - 126)
    up[h] = __uint_as_float((268u << 23) - e);
    down[h] = __uint_as_float(e - (14u << 23));
  }
}

// 8-byte slot of a running sum: a float-float pair while terms are added, an
// FP64 number when the warps' sums are added
union Slot {
  float2 ff;
  double d;
};

template <int D, bool F16>
__global__ void __launch_bounds__(32 * SmallCfg<D, F16>::NW, SmallCfg<D, F16>::MINB) sigma_small_kernel(SmallDev a) {
  constexpr int NT = SmallCfg<D, F16>::NT, NW = SmallCfg<D, F16>::NW, NSL = F16 ? 2 : 3, TILE = 128 * NSL;
  constexpr int GROUP = 8;           // terms summed in FP32 before each float-float addition
  // running sums, [warp][element of the lane][lane]
  __shared__ Slot acc[NW][NT * 4][32];
  __shared__ int next;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned char* const op = reinterpret_cast<const unsigned char*>(a.op) + 4 * lane;
  const unsigned char* const psi = reinterpret_cast<const unsigned char*>(a.psi) + 4 * lane;
  for (;;) {
    if (threadIdx.x == 0) next = (int)atomicAdd(a.counter, 1u);
    __syncthreads();
    const int qi = next;
    __syncthreads();
    if (qi >= a.n_items) return;
    const TcItem it = a.items[a.schedule[qi]];
    const int tm = it.nrows, tn = it.ncols, tm8 = (tm + 7) >> 3, tn8 = (tn + 7) >> 3;
    // a warp computes 16 rows of a term: tiles of more rows take two warps per term
    const int n_rows = tm > 16 ? 2 : 1, step = NW / n_rows, i = warp % n_rows, r8 = 2 * i;
    float grp[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        grp[j][e] = 0.0f;
        acc[warp][j * 4 + e][lane].ff = make_float2(0.0f, 0.0f);
      }
    auto flush_group = [&]() {  // acc += grp (two-sum), grp = 0
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          Slot& s = acc[warp][j * 4 + e][lane];
          const float2 v = s.ff;
          const float x = grp[j][e], sum = v.x + x, z = sum - v.x;
          const float lo = v.y + ((v.x - (sum - z)) + (x - z));
          const float hi = sum + lo;
          s.ff = make_float2(hi, lo - (hi - sum));
          grp[j][e] = 0.0f;
        }
    };
    uint32_t fp[NT][NT][NSL];  // psi^T fragments: [K tile][N tile]
    int cur = -1, ng = 0, m8 = 0, n8 = 0;
    const int t0 = it.r_begin + warp / n_rows;
    SmallTerm nx{};
    if (t0 < it.r_end) nx = a.terms[t0];
    for (int t = t0; t < it.r_end; t += step) {
      const SmallTerm tk = nx;
      if (t + step < it.r_end) nx = a.terms[t + step];  // in flight during this term
      const bool idL = tk.a_tile < 0, idR = tk.b_tile < 0, tA = tk.flags & 1, tB = tk.flags & 2;
      const unsigned char* pp = nullptr;
      int pc8 = 0;
      if (tk.in_blk != cur || idL) {
        const TcPsiBlock pb = a.pblk[tk.in_blk];
        m8 = (pb.m + 7) >> 3;
        n8 = (pb.n + 7) >> 3;
        pp = psi + pb.tile * TILE;
        pc8 = pb.C8;
      }
      // fragments of R for K step ks: [N tile][K tile of the step]
      const unsigned char* const pr = op + tk.b_tile * TILE;
      const int rj = (tB ? 1 : n8) * TILE, rk = (tB ? tn8 : 1) * TILE;
      uint32_t fr[NT][2][NSL];
      auto load_r = [&](int ks) {
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            load_tile<NSL>(fr[j][h], pr, j * rj + (2 * ks + h) * rk, !idR && j < tn8 && 2 * ks + h < n8);
      };
      const unsigned char* const pl = op + tk.a_tile * TILE;
      const int lr = (tA ? 1 : m8) * TILE, lk = (tA ? tm8 : 1) * TILE;
      uint32_t fa[NSL][4];
      auto load_l = [&](int ks) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int r = r8 + (q & 1), k = 2 * ks + (q >> 1);
          uint32_t v[NSL];
          load_tile<NSL>(v, pl, r * lr + k * lk, !idL && r < tm8 && k < m8);
#pragma unroll
          for (int s = 0; s < NSL; ++s) fa[s][q] = v[s];
        }
      };
      load_l(0);
      load_r(0);  // in flight during the first product
      if (tk.in_blk != cur) {
#pragma unroll
        for (int k = 0; k < NT; ++k)
#pragma unroll
          for (int j = 0; j < NT; ++j) load_tile<NSL>(fp[k][j], pp, (k * pc8 + j) * TILE, k < m8 && j < n8);
#pragma unroll
        for (int k = 0; k < NT; ++k)
#pragma unroll
          for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int s = 0; s < NSL; ++s) fp[k][j][s] = trans8(fp[k][j][s]);
        cur = tk.in_blk;
      }
      const float sc = (float)tk.scale;
      float x[NT][4];
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) x[j][e] = 0.0f;
      if (!idL) {  // X = L psi
#pragma unroll
        for (int ks = 0; ks < NT / 2; ++ks) {
          if (ks > 0 && 2 * ks >= m8) break;
          if (ks > 0) load_l(ks);
          if (tA) {
#pragma unroll
            for (int s = 0; s < NSL; ++s)
#pragma unroll
              for (int q = 0; q < 4; ++q) fa[s][q] = trans8(fa[s][q]);
          }
          mma_step<F16, false, D == 16 && F16>(x, ks == 0, n8, fa, [&](int j, int h, int sl) { return fp[2 * ks + h][j][sl]; });
        }
      } else {  // X = psi (the tile's rows and columns)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t v[NSL];
            load_tile<NSL>(v, pp, ((r8 + h) * pc8 + j) * TILE, r8 + h < m8 && j < n8);
#pragma unroll
            for (int s = NSL - 1; s >= 0; --s) {
              if (F16) {
                const float2 w = __half22float2(*reinterpret_cast<const __half2*>(&v[s]));
                x[j][2 * h] += w.x;
                x[j][2 * h + 1] += w.y;
              } else {
                x[j][2 * h] += __uint_as_float(v[s] << 16);
                x[j][2 * h + 1] += __uint_as_float(v[s] & 0xFFFF0000u);
              }
            }
          }
      }
      if (idR) {
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) grp[j][e] = fmaf(sc, x[j][e], grp[j][e]);
      } else {  // Y = X R^T
        // fp16: every row of X on a scale of its own, undone in Y: its elements are
        // held to 2^-39 of its largest, as the splits hold operands and psi. On one scale
        // for all (2^-20, from |X| <= 2^35) psi blocks far below max |psi| lost their bits
        float up[2], down[2] = {1.0f, 1.0f};
        if (F16) {
          float mx[2] = {0.0f, 0.0f};
#pragma unroll
          for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) mx[e >> 1] = fmaxf(mx[e >> 1], fabsf(x[j][e]));
          row_scales(mx[0], mx[1], up, down);
        }
        float y[NT][4];
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) y[j][e] = 0.0f;
#pragma unroll
        for (int ks = 0; ks < NT / 2; ++ks) {
          if (ks > 0 && 2 * ks >= n8) break;
          if (ks > 0) load_r(ks);
          if (tB) {
#pragma unroll
            for (int j = 0; j < NT; ++j)
#pragma unroll
              for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int s = 0; s < NSL; ++s) fr[j][h][s] = trans8(fr[j][h][s]);
          }
          uint32_t fx[3][4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint32_t s3[3];
            const float f = F16 ? up[q & 1] : 1.0f;
            split_pair<F16>(x[2 * ks + (q >> 1)][2 * (q & 1)] * f, x[2 * ks + (q >> 1)][2 * (q & 1) + 1] * f, s3);
#pragma unroll
            for (int s = 0; s < 3; ++s) fx[s][q] = s3[s];
          }
          mma_step<F16, true, D == 16>(y, ks == 0, tn8, fx, [&](int j, int h, int sl) { return fr[j][h][sl]; });
        }
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e)
            grp[j][e] = fmaf(sc, F16 ? y[j][e] * down[e >> 1] : y[j][e], grp[j][e]);
      }
      if (++ng == GROUP) {
        flush_group();
        ng = 0;
      }
    }
    flush_group();
#pragma unroll
    for (int e = 0; e < NT * 4; ++e) {
      Slot& s = acc[warp][e][lane];
      const float2 v = s.ff;
      s.d = (double)v.x + (double)v.y;
    }
    // add the warps' sums in warp order
    __syncthreads();
    double* out = a.scratch + it.slot;
    const double ps = F16 ? ldexp(1.0, psi_exponent(*a.psi_exp) - 14) : 1.0;  // undo psi's split scale
    for (int e = threadIdx.x; e < tm * tn; e += blockDim.x) {
      const int r = e / tn, c = e - r * tn;
      const int idx = (c >> 3) * 4 + ((r >> 3) & 1) * 2 + (c & 1), ln = (r & 7) * 4 + ((c & 7) >> 1);
      double v = acc[r >> 4][idx][ln].d;
      for (int w = (r >> 4) + n_rows; w < NW; w += n_rows) v += acc[w][idx][ln].d;
      out[e] = F16 ? v * ps : v;
    }
    // the next item's barriers come before acc is written again
  }
}

template <int D, bool F16>
void launch_class(const SmallDev& a, int n_items, const int* schedule, unsigned int* counter, int n_sm, cudaStream_t st) {
  if (n_items <= 0) return;
  SmallDev b = a;
  b.schedule = schedule;
  b.n_items = n_items;
  b.counter = counter;
  int grid = SmallCfg<D, F16>::MINB * n_sm;
  if (grid > n_items) grid = n_items;
  sigma_small_kernel<D, F16><<<grid, 32 * SmallCfg<D, F16>::NW, 0, st>>>(b);
}

// ------------------------------------------------------------ medium class
// Blocks of 33 - 64 (TC_MEDIUM_MAX): a term's tile rows are shared by up to four
// warps (16 rows each) of a CTA of 12 (a multiple of 1, 2, 3 and 4). The blocks
// of a term are contiguous tile runs, so one bulk copy each brings L and R into
// a ring slot of the group of warps that works on the term, while the group is
// busy with the term before; psi (one block per item) stays in shared memory.
// ldmatrix turns the tiles into fragments, transposing where the operator is
// used transposed. Arithmetic as the tensor-core kernel's: two slices and three
// products (fp16, or the first two bf16 slices), or three slices and six
// products, X split again into as many slices, FP32 sums over a warp's terms of
// an item, float-float over warps, FP64 over items.
//
// Bound by shared-memory reads and the matrix instructions (0.5 per cycle and SM:
// 1500 cycles for a 64 x 64 product in three products, whose fragments are 140
// KB of reads), in practice by the instruction latencies of 3 warps per scheduler:
// the matrix pipe is busy 40% of the time at K=54, M=1000 (0.40 ms per sigma).
// Fragments loaded from global memory by every warp took 0.75 ms there, a barrier
// of the group per term and FP64 sums over the warps 0.48 ms.
constexpr int MED_NT = TC_MEDIUM_MAX / 8, MED_KS = MED_NT / 2, MED_NW = 12;
constexpr int MED_DEPTH = 4;                       // most ring slots per group
constexpr uint32_t MED_WAIT = 2000000000u;         // cycles (~1 s) before a wait gives up

template <bool F16>
struct MedSmem {  // dynamic shared memory
  static constexpr int TILE = F16 ? 256 : 384;
  static constexpr int PSI = MED_NT * MED_NT * TILE;  // psi tiles
  // fragment reads past a block's last tile: at most one tile row or column (odd tile counts), 8 tiles; what they
  // read is not used or zeroed
  static constexpr int SLACK = 8 * TILE;
  static constexpr int RING = (225 * 1024 - PSI - SLACK) / 128 * 128;
  static constexpr int BYTES = PSI + RING + SLACK;
  static_assert(RING >= 4 * 2 * PSI, "two slots for two groups of the largest blocks");
  static_assert(RING >= 12 * 16 * TC_MEDIUM_MAX * 4, "the sums of 12 warps of 16 rows fit the ring");
};

// four 8x8 fragments; lane l gives the address of row l % 8 of tile l / 8
template <bool TRANS>
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  if constexpr (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

template <bool F16, int NPROD>
__global__ void __launch_bounds__(32 * MED_NW, 1) sigma_medium_kernel(SmallDev a) {
  constexpr int NT = MED_NT, KS = MED_KS, NU = NPROD == 6 ? 3 : 2, TILE = MedSmem<F16>::TILE;
  // slice pairs, smallest first
  auto pa = [](int p) constexpr { return NPROD == 6 ? Pairs<false>::a1(p) : p == 0 ? 1 : 0; };
  auto pb_ = [](int p) constexpr { return NPROD == 6 ? Pairs<false>::b1(p) : p == 1 ? 1 : 0; };
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int NB = MED_NW * MED_DEPTH;   // (group, slot) pairs
  __shared__ __align__(8) uint64_t bars[2 * NB + 1];  // slot loaded; slot read (4 arrivals); psi loaded
  __shared__ uint32_t phase[NB];           // uses of each slot so far, mod 2
  __shared__ int next;
  __shared__ volatile int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t s_psi = (uint32_t)__cvta_generic_to_shared(smem), s_ring = s_psi + MedSmem<F16>::PSI;
  const uint32_t s_bars = (uint32_t)__cvta_generic_to_shared(bars);
  float* const part = reinterpret_cast<float*>(smem + MedSmem<F16>::PSI);  // after the terms: the groups' sums
  const unsigned char* const op = reinterpret_cast<const unsigned char*>(a.op);
  auto bar = [&](int b) { return s_bars + 8u * (uint32_t)b; };
  auto expect = [&](int b, uint32_t bytes) {
    asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(bar(b)), "r"(bytes)
                 : "memory");
  };
  auto bulk = [&](uint32_t dst, const unsigned char* src, int bytes, int b) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar(b))
                 : "memory");
  };
  // bounded; a warp that gives up, or finds that another has, keeps to the barriers below but computes nothing more
  auto wait = [&](int b, uint32_t parity, bool drain = false) -> bool {
    uint32_t t0 = 0, ok = 0;
    for (int n = 0;; ++n) {
      asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                   : "=r"(ok) : "r"(bar(b)), "r"(parity) : "memory");
      if (ok) return true;
      if (abort_flag && !drain) return false;
      uint32_t t;
      asm volatile("mov.u32 %0, %%clock;\n" : "=r"(t)::"memory");
      if (n == 0) t0 = t;
      if (t - t0 > MED_WAIT) {
        abort_flag = 1;
        atomicExch(a.err, 32);
        return false;
      }
    }
  };
  if (threadIdx.x <= 2 * NB) {
    const uint32_t count = threadIdx.x >= NB && threadIdx.x < 2 * NB ? 4 : 1;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar(threadIdx.x)), "r"(count));
    if (threadIdx.x < NB) phase[threadIdx.x] = 0;
  }
  if (threadIdx.x == 0) abort_flag = 0;
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  constexpr int PSI_BAR = 2 * NB;
  uint32_t psi_phase = 0;
  for (;;) {
    if (threadIdx.x == 0) next = (int)atomicAdd(a.counter, 1u);
    __syncthreads();  // also: the previous item's tile has been read
    const int qi = next;
    if (qi >= a.n_items) return;
    const TcItem it = a.items[a.schedule[qi]];
    const int tm = it.nrows, tn = it.ncols, tm8 = (tm + 7) >> 3, tn8 = (tn + 7) >> 3;
    const TcPsiBlock pb = a.pblk[a.terms[it.r_begin].in_blk];
    const int m8 = (pb.m + 7) >> 3, n8 = (pb.n + 7) >> 3;
    // groups of n_rows warps, each with `depth` ring slots of one term
    const int n_rows = (tm + 15) >> 4;
    const int l_bytes = tm8 * m8 * TILE, r_bytes = tn8 * n8 * TILE;
    const int slots = MedSmem<F16>::RING / (l_bytes + r_bytes);
    const int groups = min(MED_NW / n_rows, slots >> 1), depth = min(MED_DEPTH, slots / groups);
    const int gi = warp / n_rows, i = warp - gi * n_rows, r8 = 2 * i;
    const bool active = gi < groups, leader = active && i == 0 && lane == 0;
    const int n_terms = active ? max(0, (it.r_end - it.r_begin - gi + groups - 1) / groups) : 0;
    if (threadIdx.x == 0) {
      expect(PSI_BAR, pb.R8 * pb.C8 * TILE);
      bulk(s_psi, reinterpret_cast<const unsigned char*>(a.psi) + pb.tile * TILE, pb.R8 * pb.C8 * TILE, PSI_BAR);
    }
    auto fetch = [&](int k) {  // the group's k-th term into slot k % depth (leader)
      const SmallTerm* t = a.terms + it.r_begin + gi + k * groups;
      const int sl = gi * depth + k % depth, b = gi * MED_DEPTH + k % depth;
      const long long at = t->a_tile, bt = t->b_tile;
      const uint32_t dst = s_ring + (uint32_t)sl * (uint32_t)(l_bytes + r_bytes);
      expect(b, (at >= 0 ? l_bytes : 0) + (bt >= 0 ? r_bytes : 0));
      if (at >= 0) bulk(dst, op + at * TILE, l_bytes, b);
      if (bt >= 0) bulk(dst + l_bytes, op + bt * TILE, r_bytes, b);
    };
    if (leader)
      for (int k = 0; k < min(depth, n_terms); ++k) fetch(k);
    bool ok = wait(PSI_BAR, psi_phase);
    psi_phase ^= 1u;
    float grp[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) grp[j][e] = 0.0f;
    // fragment addresses: lane l names row l % 8 of the tile l / 8 of four
    const int q = lane >> 3;
    const uint32_t row = (lane & 7) * 16;
    const uint32_t psi_lane = s_psi + ((q & 1) * pb.C8 + (q >> 1)) * TILE + row;  // (K tile, N tile)
    int bslot = 0, before = 0;       // barrier slot of the current term and of the one before
    uint32_t turn = 0, turn_before = 0;  // rounds of the ring completed then
    int fetched = min(depth, n_terms);
    // term k - 1 + depth into the slot of term k - 1 (barrier slot `sl`, after `rounds` rounds), once the group has read
    // it: in the middle of term k, when the group's other warps are past it
    auto refill = [&](int k, int sl, uint32_t rounds) {
      if (leader && k > 0 && k - 1 + depth < n_terms && wait(NB + gi * MED_DEPTH + sl, (phase[gi * MED_DEPTH + sl] + rounds) & 1u)) {
        fetch(k - 1 + depth);
        fetched = k + depth;
      }
      __syncwarp();
    };
    // one term from the ring slot `bslot`; the uses of its operators (transposed or not) as types: the four forms
    // are separate straight-line code, and an item's terms come in runs of one form
    auto compute = [&](const SmallTerm& tk, int k, auto TA, auto TB) {
      constexpr bool tA = decltype(TA)::value, tB = decltype(TB)::value;
      const bool idL = tk.a_tile < 0, idR = tk.b_tile < 0;
      const float sc = (float)tk.scale;
      const uint32_t sl = s_ring + (uint32_t)(gi * depth + bslot) * (uint32_t)(l_bytes + r_bytes), sr = sl + l_bytes;
      float x[NT][4];
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) x[j][e] = 0.0f;
      if (!idL) {  // X = L psi
        const int lr = (tA ? 1 : m8) * TILE, lk = (tA ? tm8 : 1) * TILE;
        uint32_t al = sl + min(r8 + (q & 1), tm8 - 1) * lr + (q >> 1) * lk + row;
        uint32_t ap = psi_lane;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          if (2 * ks >= m8) break;
          uint32_t f[NU][4];
#pragma unroll
          for (int s = 0; s < NU; ++s) {
            ldsm4<tA>(f[s], al + 128 * s);
            if (2 * ks + 1 >= m8) f[s][2] = f[s][3] = 0u;  // past the block
          }
#pragma unroll
          for (int j = 0; j < NT; j += 2) {  // pairs of N tiles; one past the block is cleared below
            if (j >= n8) break;
            uint32_t v[NU][4];
#pragma unroll
            for (int s = 0; s < NU; ++s) ldsm4<true>(v[s], ap + j * TILE + 128 * s);
#pragma unroll
            for (int p = 0; p < NPROD; ++p) {
              mma16<F16>(x[j], f[pa(p)], v[pb_(p)][0], v[pb_(p)][1]);
              mma16<F16>(x[j + 1], f[pa(p)], v[pb_(p)][2], v[pb_(p)][3]);
            }
          }
          al += 2 * lk;
          ap += 2 * pb.C8 * TILE;
        }
#pragma unroll
        for (int j = 1; j < NT; j += 2)
          if (j == n8) x[j][0] = x[j][1] = x[j][2] = x[j][3] = 0.0f;
      } else {  // X = psi (the tile's rows and columns)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (r8 + h < m8 && j < n8) {
              const unsigned char* t = smem + ((r8 + h) * pb.C8 + j) * TILE + 4 * lane;
#pragma unroll
              for (int s = TILE / 128 - 1; s >= 0; --s) {
                const uint32_t v = *reinterpret_cast<const uint32_t*>(t + 128 * s);
                if (F16) {
                  const float2 w = __half22float2(*reinterpret_cast<const __half2*>(&v));
                  x[j][2 * h] += w.x;
                  x[j][2 * h + 1] += w.y;
                } else {
                  x[j][2 * h] += __uint_as_float(v << 16);
                  x[j][2 * h + 1] += __uint_as_float(v & 0xFFFF0000u);
                }
              }
            }
      }
      refill(k, before, turn_before);
      if (idR) {
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) grp[j][e] = fmaf(sc, x[j][e], grp[j][e]);
      } else {
        // Y = X R^T; fp16: |X| <= 64 * 2^30 of the scaled operands (2^15 with an identity)
        const float f = F16 && !idL ? 0x1p-21f : 1.0f, finv = F16 && !idL ? 0x1p21f : 1.0f;
        const int rj = (tB ? 1 : n8) * TILE, rk = (tB ? tn8 : 1) * TILE;
        float y[NT][4];
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) y[j][e] = 0.0f;
        uint32_t ar = sr + (q >> 1) * rj + (q & 1) * rk + row;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          if (2 * ks >= n8) break;
          uint32_t fx[3][4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            uint32_t s3[3];
            split_pair<F16>(x[2 * ks + (u >> 1)][2 * (u & 1)] * f, x[2 * ks + (u >> 1)][2 * (u & 1) + 1] * f, s3);
#pragma unroll
            for (int s = 0; s < NU; ++s) fx[s][u] = s3[s];
          }
#pragma unroll
          for (int j = 0; j < NT; j += 2) {  // one N tile past the block is computed and never stored
            if (j >= tn8) break;
            uint32_t v[NU][4];
#pragma unroll
            for (int s = 0; s < NU; ++s) {
              ldsm4<tB>(v[s], ar + j * rj + 128 * s);
              if (2 * ks + 1 >= n8) v[s][1] = v[s][3] = 0u;  // past the block
            }
#pragma unroll
            for (int p = 0; p < NPROD; ++p) {
              mma16<F16>(y[j], fx[pa(p)], v[pb_(p)][0], v[pb_(p)][1]);
              mma16<F16>(y[j + 1], fx[pa(p)], v[pb_(p)][2], v[pb_(p)][3]);
            }
          }
          ar += 2 * rk;
        }
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) grp[j][e] = fmaf(sc, y[j][e] * finv, grp[j][e]);
      }
    };
    SmallTerm nx{};
    if (n_terms > 0) nx = a.terms[it.r_begin + gi];
    for (int k = 0; k < n_terms; ++k) {
      const SmallTerm tk = nx;
      if (k + 1 < n_terms) nx = a.terms[it.r_begin + gi + (k + 1) * groups];  // in flight during this term
      const int b = gi * MED_DEPTH + bslot;
      ok = ok && wait(b, (phase[b] + turn) & 1u);
      if (!ok) {  // the copy may still be in flight: its leader waits for it (again bounded)
        if (leader && k < fetched) wait(b, (phase[b] + turn) & 1u, true);
      } else if (tk.flags & 1) {
        if (tk.flags & 2) compute(tk, k, std::true_type{}, std::true_type{});
        else compute(tk, k, std::true_type{}, std::false_type{});
      } else {
        if (tk.flags & 2) compute(tk, k, std::false_type{}, std::true_type{});
        else compute(tk, k, std::false_type{}, std::false_type{});
      }
      __syncwarp();
      if (lane == 0)  // this warp has read the slot (4 arrivals per slot, whatever the number of warps)
        asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(bar(NB + b)),
                     "r"(i == 0 ? 5 - n_rows : 1)
                     : "memory");
      before = bslot;
      turn_before = turn;
      if (++bslot == depth) {
        bslot = 0;
        ++turn;
      }
    }
    __syncthreads();  // every slot has been read: the ring becomes the groups' sums
    if (abort_flag) return;
    if (leader)
      for (int d = 0; d < depth; ++d) phase[gi * MED_DEPTH + d] = (phase[gi * MED_DEPTH + d] + (n_terms - d + depth - 1) / depth) & 1u;
    const int g = lane >> 2, c = lane & 3, n = tm * tn;
    if (active) {
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int r = 16 * i + g + 8 * (e >> 1), col = 8 * j + 2 * c + (e & 1);
          if (r < tm && col < tn) part[gi * n + r * tn + col] = grp[j][e];
        }
    }
    __syncthreads();
    // the groups' sums in order, float-float (an FP64 addition per group would cost as much as several terms)
    double* out = a.scratch + it.slot;
    const double ps = F16 ? ldexp(1.0, psi_exponent(*a.psi_exp) - 14) : 1.0;  // undo psi's split scale
    for (int e = threadIdx.x; e < n; e += blockDim.x) {
      float hi = part[e], lo = 0.0f;
      for (int s = 1; s < groups; ++s) {
        const float v = part[s * n + e], t = hi + v, z = t - hi;
        lo += (hi - (t - z)) + (v - z);
        hi = t;
      }
      const double v = (double)hi + (double)lo;
      out[e] = F16 ? v * ps : v;
    }
    // bulk copies overwrite what was written and read here through the generic proxy
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
}

template <bool F16, int NPROD>
void launch_medium(const SmallDev& a, int n_items, const int* schedule, unsigned int* counter, int n_sm, cudaStream_t st) {
  if (n_items <= 0) return;
  set_max_dynamic_smem((const void*)sigma_medium_kernel<F16, NPROD>, MedSmem<F16>::BYTES);
  SmallDev b = a;
  b.schedule = schedule;
  b.n_items = n_items;
  b.counter = counter;
  sigma_medium_kernel<F16, NPROD>
      <<<n_sm < n_items ? n_sm : n_items, 32 * MED_NW, MedSmem<F16>::BYTES, st>>>(b);
}

template <bool F16>
void launch_classes(const SmallDev& a, int n_sm, cudaStream_t st) {
  // the schedule lists the <= 16 class, the <= 32 class, the <= 64 class
  const int n32 = a.n_items - a.n_mid - a.n_medium;
  launch_class<16, F16>(a, a.n_mid, a.schedule, a.counter, n_sm, st);
  launch_class<32, F16>(a, n32, a.schedule + a.n_mid, a.counter + 1, n_sm, st);
  const int* const med = a.schedule + a.n_mid + n32;
  if (F16 || a.nprod == 3)
    launch_medium<F16, 3>(a, a.n_medium, med, a.counter + 2, n_sm, st);
  else
    launch_medium<F16, F16 ? 3 : 6>(a, a.n_medium, med, a.counter + 2, n_sm, st);
}

}  // namespace

void launch_sigma_small(const SmallDev& a, int n_sm, cudaStream_t st) {
  if (a.f16)
    launch_classes<true>(a, n_sm, st);
  else
    launch_classes<false>(a, n_sm, st);
}

}  // namespace dmrg
