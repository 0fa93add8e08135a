// lu_split.cu -- the FP64 LU's trailing update A22 -= L21 U12 (panels of 64 columns) on the tensor cores,
// within FP64's own error bound, by splitting the operands into 8-bit digits (the error-free splitting of
// Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication", 2012, with integer digits):
//   a row of L (a column of U) is scaled by a power of two 2^-e to below one, and x 2^(7-e) is cut into
//   SL = 9 integer digits |d| <= 128, x = 2^(e-7) sum_s d_s 2^(-8 s) up to 2^-72 of 2^e; the digits are
//   held as d_s 2^(-8 s), exact in BF16.  The products of one weight s + t, at most 2^14 each in units of
//   2^(-8 (s + t)), 128 of each of up to 8 pairs, add up to at most 2^24 units: exact in the tensor
//   cores' FP32 accumulators.  Seven accumulators hold the weights 0 .. 6, the eighth (tensor memory holds
//   no more) the weights 7 and 8, where what is below weight 7's units rounds off.
// Digit pairs with s + t < SL are kept (45 of 81).  In units of the leading digits' product, the 128 real
// products of an entry lose at most 2^-48 with the eight dropped pairs of weight 9 (the rest is smaller
// by 2^-8), 2^-50 with the operands' remainders and 2^-49 in the eighth accumulator (an ulp at each of
// its 120 instructions): below 2^-46 together.  That is a bound relative to the scales 2^er 2^ec of the
// entry's row and column; FP64 arithmetic's is 128 x 2^-53 sum |l||u|.  It is no smaller where the sum is at
// least one unit, that is, where some k has |l_ik| |u_kj| >= 2^-14 of the scales.  So a row carries for
// each of its 64 entries whether it is within 2^-3, 2^-7, 2^-11 of the scale, a column 2^-11, 2^-7, 2^-3, and an
// entry whose row and column have no bit in common (graded panels), or whose scales leave the exponents'
// range or are not finite, takes its 64 products in FP64, by the lanes of the warp together.  Share of
// such entries over spheres, two spheres and ellipsoids of 258 .. 2884 nodes: 0.03 % at the lowest
// wavenumbers, 0 .. 1e-6 above (eight digits, whose bound asks for 2^-8, with one level, 2^-4 on both
// sides: up to 3 %, and 18 ms more for the systems below).
// The accumulators of an entry are combined as 64-bit integers and enter A22 with one FP64 fused
// multiply-add.
// The complex product is a real one on the interleaved storage (as in lu_tc.cu): C (m x 2n) -= L (m x
// 128) B with B^T rows 2 c and 2 c + 1 = [ur, -ui], [ui, ur].
// Bound: the chain of a tile of 128 x 64 reals -- operands, 360 MMAs, the epilogue's FP64 instructions (four
// an entry) and rows of A22 -- of which only the next operands overlap (eight accumulators fill the tensor
// memory): FP64 pipe 30 % busy, tensor pipe 21 %.  Two systems of N = 2884: the updates 189 ms on the FP64
// pipe (0.67 of 1.1 TFLOP/s) -> 16.3 ms with the splitting (7.8 TFLOP/s of the products it replaces); error
// of the solutions against 64 bits 9.0e-15 -> 8.7e-15.  Seven digits without the bits measured 13.2 ms, but
// lost 2^g on panels graded by 2^g.
#include "tcgen05.cuh"

#include <algorithm>

namespace bie {
namespace split {

constexpr int SL = 9;              // digits
constexpr int NACC = 8;            // accumulators
constexpr int NL = 3;              // levels of the bits: 2^-(3 + 4 i) of a row's scale, 2^-(11 - 4 i) of a column's
constexpr int KR = 128;            // reals along K (64 complex)
constexpr int BM = 128, BN = 64;   // tile: rows x real columns
constexpr int KCH = 64;            // BF16 per 128-byte swizzle row
constexpr int A_SL = BM * 128, B_SL = BN * 128;  // bytes of one digit's chunk
constexpr int SMEM = SL * (A_SL + B_SL) + 1024;
constexpr int NT = 192;
constexpr int kBadExp = 5000;      // exponent of a row or column that is not finite (or above 1e308)

// Digits of t (|t| <= 128): d = rint(t), t <- 256 (t - d).
__device__ __forceinline__ int next_digit(double& t) {
  constexpr double M = 6755399441055744.0;  // 1.5 * 2^52
  const double m = t + M;
  t = (t - (m - M)) * 256.0;
  return __double2loint(m);
}
// d w in BF16: exact for |d| <= 256 and a power of two w
__device__ __forceinline__ uint32_t bf16_of(int d, float w) { return __float_as_uint((float)d * w) >> 16; }
// exponent e with |x| < 2^e for the largest magnitude x of a row
__device__ __forceinline__ int exp_of(double x) {
  if (!(x < 1e308)) return kBadExp;  // too large, infinite or NaN
  if (!(x > 0.0)) return 0;
  const int e = ((__double2hiint(x) >> 20) & 0x7ff) - 1022;
  return e > -1000 ? e : -1000;  // (2^(7 - e) stays finite)
}
// the least magnitude that counts for a row's or column's bits of one level: 2^(e - level), anything in one of
// zeros, nothing in one that is not finite
__device__ __forceinline__ double near_of(int e, double mx, int level) {
  return e == kBadExp ? INFINITY : mx > 0.0 ? __hiloint2double((1023 - level + e) << 20, 0) : 0.0;
}
__device__ __forceinline__ int row_level(int i) { return 3 + 4 * i; }
__device__ __forceinline__ int col_level(int i) { return 11 - 4 * i; }
__device__ __forceinline__ double scale_of(int e) {  // 2^(7 - e)
  return e == kBadExp ? 0.0 : __hiloint2double((1030 - e) << 20, 0);
}

// L rows r0 + r (r < m) of columns [p0, p0 + 64): digits as [z][s][m][128] BF16, exponents [z][m], bits of
// the entries near the row's scale [z][m][NL].
// One warp per row; grid (ceil(m / 8), batch), block 256.
__global__ void __launch_bounds__(256) k_split_rows(const double2* __restrict__ A, int64_t bstride, int ld, int p0, int r0,
                                                    int m, uint32_t* __restrict__ da, int32_t* __restrict__ ea,
                                                    uint64_t* __restrict__ na) {
  const int lane = threadIdx.x & 31, r = blockIdx.x * 8 + (threadIdx.x >> 5), z = blockIdx.y;
  if (r >= m) return;
  const double2* row = A + (int64_t)z * bstride + (int64_t)(r0 + r) * ld + p0;
  double2 v[2] = {row[lane], row[lane + 32]};
  double mx = fmax(fmax(fabs(v[0].x), fabs(v[0].y)), fmax(fabs(v[1].x), fabs(v[1].y)));
  if (!(v[0].x - v[0].x == 0.0 && v[0].y - v[0].y == 0.0 && v[1].x - v[1].x == 0.0 && v[1].y - v[1].y == 0.0)) mx = INFINITY;
  for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const int e = exp_of(mx);
#pragma unroll
  for (int i = 0; i < NL; ++i) {
    const double lim = near_of(e, mx, row_level(i));
    const unsigned b0 = __ballot_sync(0xffffffffu, fmax(fabs(v[0].x), fabs(v[0].y)) >= lim);
    const unsigned b1 = __ballot_sync(0xffffffffu, fmax(fabs(v[1].x), fabs(v[1].y)) >= lim);
    if (lane == 0) na[((int64_t)z * m + r) * NL + i] = e == kBadExp ? 0ull : ((uint64_t)b1 << 32) | b0;
  }
  if (lane == 0) ea[(int64_t)z * m + r] = e;
  const double sc = scale_of(e);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    double x = e == kBadExp ? 0.0 : v[h].x * sc, y = e == kBadExp ? 0.0 : v[h].y * sc;
    uint32_t* o = da + ((int64_t)z * SL * m + r) * (KR / 2) + lane + 32 * h;
#pragma unroll
    for (int s = 0; s < SL; ++s) {
      const float w = ldexpf(1.f, -8 * s);
      const uint32_t a = bf16_of(next_digit(x), w), b = bf16_of(next_digit(y), w);
      o[(int64_t)s * m * (KR / 2)] = a | (b << 16);
    }
  }
}

// U columns c0 + c (c < m) of rows [p0, p0 + 64): digits of B^T as [z][s][2 m][128] BF16, exponents [z][m]
// and bits [z][m][NL] as for the rows.
// CTA: 32 columns (lanes) x 8 warps of 8 rows; grid (ceil(m / 32), batch), block 256.
__global__ void __launch_bounds__(256) k_split_cols(const double2* __restrict__ A, int64_t bstride, int ld, int p0, int c0,
                                                    int m, uint32_t* __restrict__ db, int32_t* __restrict__ eb,
                                                    uint64_t* __restrict__ nb) {
  __shared__ uint32_t t[64][65];  // [2 c, 2 c + 1][k] pairs of one digit
  __shared__ double smx[8][32];
  __shared__ uint8_t sbit[NL][8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, z = blockIdx.y, cb = blockIdx.x * 32;
  const int c = cb + lane;
  const bool act = c < m;
  double2 v[8];
  double mx = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    v[i] = act ? A[(int64_t)z * bstride + (int64_t)(p0 + warp * 8 + i) * ld + c0 + c] : make_double2(0.0, 0.0);
    mx = fmax(mx, fmax(fabs(v[i].x), fabs(v[i].y)));
    if (!(v[i].x - v[i].x == 0.0 && v[i].y - v[i].y == 0.0)) mx = INFINITY;
  }
  smx[warp][lane] = mx;
  __syncthreads();
  for (int w = 0; w < 8; ++w) mx = fmax(mx, smx[w][lane]);
  const int e = exp_of(mx);
#pragma unroll
  for (int l = 0; l < NL; ++l) {
    const double lim = near_of(e, mx, col_level(l));
    unsigned bits = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) bits |= (unsigned)(fmax(fabs(v[i].x), fabs(v[i].y)) >= lim) << i;
    sbit[l][warp][lane] = (uint8_t)bits;
  }
  __syncthreads();
  if (warp < NL && act) {
    uint64_t all = 0;
    for (int w = 0; w < 8; ++w) all |= (uint64_t)sbit[warp][w][lane] << (8 * w);
    nb[((int64_t)z * m + c) * NL + warp] = e == kBadExp ? 0ull : all;
  }
  if (warp == 0 && act) eb[(int64_t)z * m + c] = e;
  const double sc = scale_of(e);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    v[i].x = e == kBadExp ? 0.0 : v[i].x * sc;
    v[i].y = e == kBadExp ? 0.0 : v[i].y * sc;
  }
  const int rows = min(64, 2 * (m - cb));
  float wt = 1.f;  // 2^(-8 s)
  for (int s = 0; s < SL; ++s, wt *= 0.00390625f) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t a = bf16_of(next_digit(v[i].x), wt), b = bf16_of(next_digit(v[i].y), wt);
      const uint32_t minus = b == 0u ? 0u : b ^ 0x8000u;
      t[2 * lane][warp * 8 + i] = a | (minus << 16);
      t[2 * lane + 1][warp * 8 + i] = b | (a << 16);
    }
    __syncthreads();
    uint32_t* o = db + ((int64_t)(z * SL + s) * 2 * m + 2 * cb) * (KR / 2);
    for (int e2 = threadIdx.x; e2 < rows * 64; e2 += 256) o[e2] = t[e2 >> 6][e2 & 63];
    __syncthreads();
  }
}

struct alignas(8) Bars {
  uint64_t full, empty, acc_full, acc_empty;
  uint32_t tmem_slot;
};

__device__ __forceinline__ void mbar_arrive(uint32_t a) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(a) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
// the wait names the destination registers so that no use of them is scheduled before it
__device__ __forceinline__ void tmem_wait8(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
               :
               : "memory");
}
__device__ __forceinline__ double int_to_double(int64_t v) {  // |v| < 2^51
  return __longlong_as_double(v + 0x4338000000000000ll) - 6755399441055744.0;
}

// Persistent: grid min(tiles, SMs), block NT.  Warp 0 loads the tile's digits by TMA, one K half at a time
// (216 KB), warp 1 issues the MMAs, warps 2-5 combine and subtract; the next tile's first half loads while
// the epilogue runs.  Every wait is bounded: one that gives up after `polls` polls raises *err and ends its
// role, the other roles' waits then give up too, and the copies and MMAs in flight are waited for (with
// tcx::mbar_wait's own limit) before the CTA ends.  A launch that finds *err raised does nothing.
__global__ void __launch_bounds__(NT, 1) k_update_split(const __grid_constant__ CUtensorMap ma,
                                                        const __grid_constant__ CUtensorMap mb, double* __restrict__ A,
                                                        int64_t bstride, int ld, int r0, int m, int batch,
                                                        const int32_t* __restrict__ ea, const int32_t* __restrict__ eb,
                                                        const uint64_t* __restrict__ na, const uint64_t* __restrict__ nb,
                                                        int32_t* err, uint32_t polls) {
  extern __shared__ unsigned char sm_raw[];
  __shared__ Bars bars;
  __shared__ int s_void;
  const uint32_t base = (tcx::smem_u32(sm_raw) + 1023u) & ~1023u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tm = (m + BM - 1) / BM, tn = (2 * m + BN - 1) / BN, per = tm * tn, tiles = per * batch;
  const uint32_t full = tcx::smem_u32(&bars.full), empty = tcx::smem_u32(&bars.empty);
  const uint32_t accf = tcx::smem_u32(&bars.acc_full), acce = tcx::smem_u32(&bars.acc_empty);
  if (tid == 0) s_void = *(volatile int32_t*)err;
  __syncthreads();
  if (s_void) return;  // an earlier update of this factorisation gave up
  if (warp == 0) tcx::tmem_alloc(&bars.tmem_slot, 512);
  if (tid == 0) {
    tcx::mbar_init(full, 1);
    tcx::mbar_init(empty, 1);
    tcx::mbar_init(accf, 1);
    tcx::mbar_init(acce, 4);
    asm volatile("fence.mbarrier_init.release.cluster;\n");
  }
  tcx::fence_before();
  __syncthreads();
  tcx::fence_after();
  const uint32_t tmem = bars.tmem_slot;
  if (warp == 0) {
    if (lane == 0) {
      uint32_t it = 0;
      for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int z = t / per, u = t - z * per, im = u % tm, in = u / tm;
        bool ok = true;
        for (int kc = 0; kc < 2 && ok; ++kc, ++it) {
          if (it > 0) ok = tcx::mbar_wait(empty, (it - 1) & 1, err, 1, polls);
          if (!ok) break;
          tcx::mbar_expect_tx(full, SL * (A_SL + B_SL));
          for (int s = 0; s < SL; ++s) {
            tcx::tma_load_2d(base + s * A_SL, &ma, kc * KCH, (z * SL + s) * m + im * BM, full);
            tcx::tma_load_2d(base + SL * A_SL + s * B_SL, &mb, kc * KCH, (z * SL + s) * 2 * m + in * BN, full);
          }
        }
        if (!ok) break;
      }
      if (it > 0) tcx::mbar_wait(full, (it - 1) & 1, err, 1);  // no copy is in flight when the CTA ends
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = tcx::idesc_bf16(BM, BN);
      uint32_t it = 0, n = 0;
      for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++n) {
        bool ok = true;
        if (n > 0) ok = tcx::mbar_wait(acce, (n - 1) & 1, err, 1, polls);
        if (!ok) break;
        tcx::fence_after();
        for (int kc = 0; kc < 2 && ok; ++kc, ++it) {
          ok = tcx::mbar_wait(full, it & 1, err, 1, polls);
          if (!ok) break;
          tcx::fence_after();
          for (int d = 0; d < SL; ++d)
            for (int s = 0; s <= d; ++s) {
              const uint64_t da = tcx::desc_sw128(base + s * A_SL), db = tcx::desc_sw128(base + SL * A_SL + (d - s) * B_SL);
#pragma unroll
              for (int k = 0; k < KCH / 16; ++k)  // 32 bytes along K: two descriptor units
                tcx::mma_bf16(tmem + min(d, NACC - 1) * BN, da + 2 * k, db + 2 * k, idesc,
                              (kc | s | k) || d >= NACC ? 1u : 0u);
            }
          tcx::mma_commit(empty);
        }
        if (!ok) break;
        tcx::mma_commit(accf);
      }
      if (it > 0) tcx::mbar_wait(empty, (it - 1) & 1, err, 1);  // nor an MMA
      if (n > 0) tcx::mbar_wait(accf, (n - 1) & 1, err, 1);     // nor the last tile's arrival
    }
  } else {
    const int wl = warp & 3;  // TMEM lanes 32 wl .. 32 wl + 31
    uint32_t n = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++n) {
      const int z = t / per, u = t - z * per, im = u % tm, in = u / tm;
      const bool ok = __all_sync(0xffffffffu, tcx::mbar_wait(accf, n & 1, err, 1, polls));
      if (!ok) break;
      tcx::fence_after();
      const int r = im * BM + wl * 32 + lane;
      const int er = r < m ? ea[(int64_t)z * m + r] : 0;
      uint64_t near_row[NL], near_col[NL];
      // the tile's 32 complex columns: exponent and bits, one a lane
      const int cl = in * (BN / 2) + lane;
      const int ec = cl < m ? eb[(int64_t)z * m + cl] : 0;
#pragma unroll
      for (int i = 0; i < NL; ++i) {
        near_row[i] = r < m ? na[((int64_t)z * m + r) * NL + i] : 0ull;
        near_col[i] = cl < m ? nb[((int64_t)z * m + cl) * NL + i] : 0ull;
      }
      double* row = A + 2 * ((int64_t)z * bstride + (int64_t)(r0 + (r < m ? r : 0)) * ld + r0);
      const double2* L = reinterpret_cast<const double2*>(A) + (int64_t)z * bstride + (int64_t)(r0 + im * BM + wl * 32) * ld + r0 - 64;
      const double2* U = reinterpret_cast<const double2*>(A) + (int64_t)z * bstride + (int64_t)(r0 - 64) * ld + r0;
      const uint32_t taddr = tmem + ((uint32_t)(wl * 32) << 16);
#pragma unroll 1
      for (int j0 = 0; j0 < BN; j0 += 8) {
        uint32_t a[NACC][8];
#pragma unroll
        for (int d = 0; d < NACC; ++d) tmem_ld8(taddr + d * BN + j0, a[d]);
        const int c = in * BN + j0;  // real column (even)
        double2 v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          v[q] = (r < m && c + 2 * q < 2 * m) ? *reinterpret_cast<double2*>(row + c + 2 * q) : make_double2(0.0, 0.0);
#pragma unroll
        for (int d = 0; d < NACC; ++d) tmem_wait8(a[d]);
        unsigned slow = 0;  // of the four complex columns, those where this row takes its products in FP64
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int cq = j0 / 2 + q;  // column of the tile
          // 2^(er + ec - 70): the digits' weights
          const int ex = 1023 + er + __shfl_sync(0xffffffffu, ec, cq) - 70;
          uint64_t both = 0ull;
#pragma unroll
          for (int i = 0; i < NL; ++i) both |= near_row[i] & __shfl_sync(0xffffffffu, near_col[i], cq);
          const bool digits = ex > 0 && ex < 2047 && both != 0ull;
          if (r < m && c + 2 * q < 2 * m && !digits) slow |= 1u << q;
          const double sc = digits ? __hiloint2double(ex << 20, 0) : 0.0;
          double x[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int i = 2 * q + h;
            auto iv = [&](int d) { return (int64_t)__float2int_rn(__uint_as_float(a[d][i]) * ldexpf(1.f, 8 * d)); };
            const int64_t top = (iv(0) << 24) + (iv(1) << 16) + (iv(2) << 8) + iv(3);
            const int64_t low = (iv(4) << 24) + (iv(5) << 16) + (iv(6) << 8) + iv(7);
            x[h] = fma(int_to_double(top), 4294967296.0, int_to_double(low));
          }
          v[q].x = fma(-x[0], sc, v[q].x);
          v[q].y = fma(-x[1], sc, v[q].y);
        }
        if (__any_sync(0xffffffffu, slow != 0u)) {  // each such entry by the whole warp, two of its products a lane
#pragma unroll
          for (int q = 0; q < 4; ++q)
            for (unsigned todo = __ballot_sync(0xffffffffu, (slow >> q) & 1u); todo; todo &= todo - 1u) {
              const int src = __ffs(todo) - 1;
              double2 p = make_double2(0.0, 0.0);
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const double2 l = L[(int64_t)src * ld + lane + 32 * h], w = U[(int64_t)(lane + 32 * h) * ld + (c >> 1) + q];
                p.x = fma(l.x, w.x, fma(-l.y, w.y, p.x));
                p.y = fma(l.x, w.y, fma(l.y, w.x, p.y));
              }
              for (int o = 16; o > 0; o >>= 1) {
                p.x += __shfl_xor_sync(0xffffffffu, p.x, o);
                p.y += __shfl_xor_sync(0xffffffffu, p.y, o);
              }
              if (lane == src) {
                v[q].x -= p.x;
                v[q].y -= p.y;
              }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (r < m && c + 2 * q < 2 * m) *reinterpret_cast<double2*>(row + c + 2 * q) = v[q];
      }
      tcx::fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce);
    }
  }
  tcx::fence_before();
  __syncthreads();
  tcx::fence_after();
  if (warp == 0) tcx::tmem_dealloc(tmem, 512);
}

}  // namespace split

// Scratch of lu_update_split64 for matrices of n rows.
size_t lu_split_scratch_bytes(int batch, int n) {
  const size_t m = (size_t)std::max(0, n - 64);
  return batch * (m * split::SL * split::KR * 2 * 3 + 2 * m * (sizeof(int32_t) + split::NL * sizeof(uint64_t))) + 1024;
}

// A22 -= L21 U12 for the 64-column panel at p0 (FP64, all rows and columns past it).  *err (device) is
// raised if a bounded wait gave up: the factors of the whole batch are void.
int lu_update_split64(bie_ctx* c, cd* A, int batch, int n, int ld, int64_t bstride, int p0, void* scratch, int32_t* err) {
  using namespace split;
  const int r0 = p0 + 64, m = n - r0;
  if (m <= 0) return BIE_OK;
  uint32_t* da = (uint32_t*)(((uintptr_t)scratch + 255) & ~(uintptr_t)255);
  uint32_t* db = da + (size_t)batch * SL * m * (KR / 2);
  uint64_t* na = (uint64_t*)(db + (size_t)batch * SL * 2 * m * (KR / 2));
  uint64_t* nb = na + (size_t)batch * m * NL;
  int32_t* ea = (int32_t*)(nb + (size_t)batch * m * NL);
  int32_t* eb = ea + (size_t)batch * m;
  const double2* M = reinterpret_cast<const double2*>(A);
  BIE_LAUNCH(k_split_rows<<<dim3((unsigned)((m + 7) / 8), batch), 256, 0, c->stream>>>(M, bstride, ld, p0, r0, m, da, ea, na));
  BIE_LAUNCH(k_split_cols<<<dim3((unsigned)((m + 31) / 32), batch), 256, 0, c->stream>>>(M, bstride, ld, p0, r0, m, db, eb, nb));
  CUtensorMap ma, mb;
  BIE_TRY(tcx::make_map_bf16_2d(&ma, da, KR, (uint64_t)batch * SL * m, KR, KCH, BM));
  BIE_TRY(tcx::make_map_bf16_2d(&mb, db, KR, (uint64_t)batch * SL * 2 * m, KR, KCH, BN));
  int nsm = 0;
  BIE_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device));
  const int64_t tiles = (int64_t)((m + BM - 1) / BM) * ((2 * m + BN - 1) / BN) * batch;
  BIE_TRY(set_smem_max(k_update_split));
  BIE_LAUNCH(k_update_split<<<(unsigned)std::min<int64_t>(tiles, nsm), NT, SMEM, c->stream>>>(
      ma, mb, reinterpret_cast<double*>(A), bstride, ld, r0, m, batch, ea, eb, na, nb, err, (uint32_t)c->fp64_wait_polls));
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

}  // namespace bie
