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
// Arithmetic: FP32 accumulation of slice products. The fp16 split (hi + lo)
// takes all four products in the first product, and X as three fp16 slices (at
// least 30 bits; scaled by 2^-20 so that it stays in range) in the second; the
// bf16 split (hi + mid + lo) takes the six products above 2^-24 in both, X as
// three bf16 slices. That is the accuracy of FP32 multiply-adds on the summed
// slices, which this kernel used before (measured below). Terms of a warp are
// summed in FP32 over groups of 8, groups in float-float (48 bits), warps in
// FP64 in warp order, so the result does not depend on scheduling.
//
// Bound by instruction issue (<= 16: 65% of issue slots) and load latency (<= 32:
// 12-16 warps per SM of 128-159 registers); a term of 16 x 16 blocks reads 2-3 KB
// for 18-24 matrix instructions. So a warp takes 16 rows (a term of more rows is
// shared by two), CTAs are 4 warps, items come from a counter, the next term's
// record is loaded a term ahead and its L and R before psi and the first product.
// Both kernels per sigma, against FP32 multiply-adds from shared memory: 1.63 ->
// 0.82 ms at K=108, M=2000 (FP16X2), 0.74 -> 0.38 ms at K=54, M=1000 (BF16X2), 63
// -> 41 us at K=24, M=250; error of sigma against 64 bits 1.3e-7 -> 1.2e-7 there.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

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

// Slice pairs (A slice, B slice) of the two products, smallest first.
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
  using P = Pairs<F16>;
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
      // fp16: |X| <= 32 * 2^30 of the scaled operands (2^15 with an identity)
      const float f = F16 && !idL ? 0x1p-20f : 1.0f, finv = F16 && !idL ? 0x1p20f : 1.0f;
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
#pragma unroll
          for (int p = 0; p < P::N1; ++p)
#pragma unroll
            for (int j = 0; j < NT; ++j)
              if (j < n8) mma16<F16>(x[j], fa[P::a1(p)], fp[2 * ks][j][P::b1(p)], fp[2 * ks + 1][j][P::b1(p)]);
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
            split_pair<F16>(x[2 * ks + (q >> 1)][2 * (q & 1)] * f, x[2 * ks + (q >> 1)][2 * (q & 1) + 1] * f, s3);
#pragma unroll
            for (int s = 0; s < 3; ++s) fx[s][q] = s3[s];
          }
#pragma unroll
          for (int p = 0; p < P::N2; ++p)
#pragma unroll
            for (int j = 0; j < NT; ++j)
              if (j < tn8) mma16<F16>(y[j], fx[P::a2(p)], fr[j][0][P::b2(p)], fr[j][1][P::b2(p)]);
        }
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) grp[j][e] = fmaf(sc, y[j][e] * finv, grp[j][e]);
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

template <bool F16>
void launch_both(const SmallDev& a, int n_sm, cudaStream_t st) {
  // the schedule lists the <= 16 class first
  launch_class<16, F16>(a, a.n_mid, a.schedule, a.counter, n_sm, st);
  launch_class<32, F16>(a, a.n_items - a.n_mid, a.schedule + a.n_mid, a.counter + 1, n_sm, st);
}

}  // namespace

void launch_sigma_small(const SmallDev& a, int n_sm, cudaStream_t st) {
  if (a.f16)
    launch_both<true>(a, n_sm, st);
  else
    launch_both<false>(a, n_sm, st);
}

}  // namespace dmrg
