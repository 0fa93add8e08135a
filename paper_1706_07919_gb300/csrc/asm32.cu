// asm32.cu -- FP32 assembly of Eq. (BRIEF) for the mixed-precision path (same system as
// asm64.cu; see there for the row equation and the bulk/near split).
//
// Precision plan (each matrix entry to about FP32 rounding, independent of k R):
//   * positions and node normals are float-float (hi + lo), so x_q - x_i, |x_q - x_i| and
//     nu_i.(x_q - x_i) carry ~48 bits;
//   * both phases (k R for G, k nu_i.r for g and f) are formed and reduced modulo 2 pi in
//     float-float, then sincosf of the FP32 head plus a first-order correction by the tail;
//   * amplitudes (1/R, r.nu/R^3, w J N_a) are FP32;
//   * the row sums alpha_i, beta_i and b_i (over all E*Q points, with cancellation) are
//     compensated (Kahan-Babuska-Neumaier) sums.
// Output: A as interleaved complex FP32 [N][ld], b as complex FP64 [N].
#include <algorithm>

#include "bie_common.cuh"

namespace bie {

// Mixed-path point table: SoA of 13 floats per point:
//   x_hi, y_hi, z_hi, x_lo, y_lo, z_lo, nx, ny, nz, wJ, nx_lo, ny_lo, nz_lo
// (the normal's low parts let r.nu, a second-order small quantity for nearby points on one smooth
// surface, be formed in float-float).
enum { P32XH = 0, P32YH, P32ZH, P32XL, P32YL, P32ZL, P32NX, P32NY, P32NZ, P32W, P32NXL, P32NYL, P32NZL, P32COUNT };

// aos (optional): the same 13 values per point as one 64-byte record [n][16 floats].
__global__ void k_points_to32(const double* __restrict__ g, int64_t n, float* __restrict__ o,
                              float4* __restrict__ aos) {
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= n) return;
  float v[P32COUNT];
  for (int d = 0; d < 3; ++d) {
    const ff x = ff_from_double(g[(GX + d) * n + p]);
    const ff nv = ff_from_double(g[(GNX + d) * n + p]);
    v[P32XH + d] = x.hi; v[P32XL + d] = x.lo;
    v[P32NX + d] = nv.hi; v[P32NXL + d] = nv.lo;
  }
  v[P32W] = (float)g[GWJ * n + p];
  for (int f = 0; f < P32COUNT; ++f) o[f * n + p] = v[f];
  if (aos) {
    float4* a = aos + p * 4;
    a[0] = make_float4(v[0], v[1], v[2], v[3]);
    a[1] = make_float4(v[4], v[5], v[6], v[7]);
    a[2] = make_float4(v[8], v[9], v[10], v[11]);
    a[3] = make_float4(v[12], 0.f, 0.f, 0.f);
  }
}

// The bulk kernel's copy of the same table, re-ordered for coalesced loads: elements in colour
// order (position t of the colour-sorted list) and point-major, index (f * Q + q) * E + t, so
// that the lanes of a warp -- consecutive elements of one colour -- read consecutive floats.
// Element connectivity in the same order: esort[a * E + t].
__global__ void k_points_to32_sorted(const double* __restrict__ g, const int32_t* __restrict__ perm,
                                     const int32_t* __restrict__ elems, bool flip, const uint8_t* __restrict__ bc,
                                     int64_t E, int Q, float* __restrict__ o, int32_t* __restrict__ esort,
                                     float4* __restrict__ aos, uint8_t* __restrict__ esoft) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= E * Q) return;
  const int64_t t = idx % E;
  const int q = (int)(idx / E);
  const int64_t e = perm[t];
  const int64_t n = E * Q, src = e * Q + q;
  float v[P32COUNT];
  for (int d = 0; d < 3; ++d) {
    const ff x = ff_from_double(g[(GX + d) * n + src]);
    const ff nv = ff_from_double(g[(GNX + d) * n + src]);
    v[P32XH + d] = x.hi; v[P32XL + d] = x.lo;
    v[P32NX + d] = nv.hi; v[P32NXL + d] = nv.lo;
  }
  const ff w = ff_from_double(g[GWJ * n + src]);
  v[P32W] = w.hi;
  for (int f = 0; f < P32COUNT; ++f) o[((int64_t)f * Q + q) * E + t] = v[f];
  // the same 13 values as one 64-byte record, then the weight's low part (float-float kernels)
  float4* a = aos + ((int64_t)q * E + t) * 4;
  a[0] = make_float4(v[0], v[1], v[2], v[3]);
  a[1] = make_float4(v[4], v[5], v[6], v[7]);
  a[2] = make_float4(v[8], v[9], v[10], v[11]);
  a[3] = make_float4(v[12], w.lo, 0.f, 0.f);
  if (q == 0) {
    for (int a = 0; a < 6; ++a) esort[a * E + t] = elems[6 * e + a];
    esoft[t] = (uint8_t)((bc[elems[6 * e]] != 0) != flip);  // (flip: bc holds the exchanged conditions)
  }
}

// 2 pi as an unevaluated sum of three floats, and 1 / (2 pi).
struct TwoPi3 {
  float c1, c2, c3, inv;
};

struct Kern32 {
  float Gr, Gi, dGr, dGi;
  float alr, ali, ber, bei;  // g dG - dg G, f dG - df G (without w J)
};

// far_r2: beyond R^2 > far_r2 (a few element sizes) r.nu_q is formed in FP32: its absolute error
// eps R then perturbs dG by eps / R^2, the entry's own rounding.
__device__ __forceinline__ void kernel32(const ff k, const float kinv, const ff* xi, const ff* nui, const TwoPi3& tp,
                                         const float* q, Kern32& o, float far_r2 = 3.0e38f) {
  // r = x_q - x_i in float-float
  const ff rx = ff_diff_lazy(ff{q[0], q[3]}, xi[0]);
  const ff ry = ff_diff_lazy(ff{q[1], q[4]}, xi[1]);
  const ff rz = ff_diff_lazy(ff{q[2], q[5]}, xi[2]);
  const ff R2 = ff_norm2_lazy(rx, ry, rz);
  float invR;
  const ff R = ff_sqrt_lazy(R2, invR);
  const ff nr = ff_dot3_lazy(nui, rx, ry, rz);
  float c, s;
  cis_ffprod(k, R, c, s);
  const float kR = k.hi * R.hi;
  o.Gr = c * invR;
  o.Gi = s * invR;
  float rnu;
  if (R2.hi > far_r2) {
    rnu = (rx.hi + rx.lo) * q[6] + (ry.hi + ry.lo) * q[7] + (rz.hi + rz.lo) * q[8];
  } else {
    const ff nq[3] = {ff{q[6], q[10]}, ff{q[7], q[11]}, ff{q[8], q[12]}};
    const ff d = ff_dot3_lazy(nq, rx, ry, rz);
    rnu = d.hi + d.lo;
  }
  const float rn = rnu * invR * invR * invR;
  o.dGr = (-c - s * kR) * rn;
  o.dGi = (c * kR - s) * rn;
  float cg, sg;
  cis_ffprod(k, nr, cg, sg);
  const float nn = nui[0].hi * q[6] + nui[1].hi * q[7] + nui[2].hi * q[8];
  const float g = cg, f = kinv != 0.f ? sg * kinv : nr.hi, dg = -k.hi * sg * nn, df = cg * nn;
  o.alr = g * o.dGr - dg * o.Gr;
  o.ali = g * o.dGi - dg * o.Gi;
  o.ber = f * o.dGr - df * o.Gr;
  o.bei = f * o.dGi - df * o.Gi;
}

struct RowSums {
  ksum ar, ai, br, bi, sr, si;
};

__device__ __forceinline__ void load_point(const float* __restrict__ tab, int64_t n, int64_t p, float* q) {
#pragma unroll
  for (int t = 0; t < P32COUNT; ++t) q[t] = tab[t * n + p];
}

// grid: (ceil(N / rows), nk); block: 32 * rows * W (W warps share a row: the elements of one
// colour share no node, so they can scatter into the row concurrently; colours are separated by
// a barrier of the row's warps); dynamic smem: rows * N * sizeof(cf)
constexpr int ASM_W = 2;
__global__ void __launch_bounds__(512) k_asm32_bulk(
    const double* __restrict__ nodes, const double* __restrict__ normals, const uint8_t* __restrict__ bc,
    const int32_t* __restrict__ esort, int64_t N, int64_t E, int Q, const float* __restrict__ qtab,
    const float* __restrict__ qshape, const int32_t* __restrict__ color_off, int ncolors,
    const double* __restrict__ kv, const cd* __restrict__ known,
    cf* __restrict__ A, int64_t lda, double* __restrict__ rowsum /* [nk][N][6] */, int rows, TwoPi3 tp,
    float far_r2) {
  extern __shared__ cf acc32[];
  __shared__ float shp[64 * 6];
  __shared__ double part[16][ASM_W][6];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rw = warp / ASM_W, sub = warp % ASM_W;
  const int kk = blockIdx.y;
  const ff k = ff_from_double(kv[kk]);
  const float kinv = kinv32(kv[kk]);
  for (int t = threadIdx.x; t < Q * 6; t += blockDim.x) shp[t] = qshape[t];
  for (int64_t t = threadIdx.x; t < (int64_t)rows * N; t += blockDim.x) acc32[t] = {0.f, 0.f};
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * rows + rw;
  const bool valid = i < N;
  cf* row = acc32 + (int64_t)rw * N;
  const cd* kn = known + (int64_t)kk * N;
  ff xi[3], nui[3];
  for (int d = 0; d < 3; ++d) {
    xi[d] = ff_from_double(valid ? nodes[3 * i + d] : 0.0);
    nui[d] = ff_from_double(valid ? normals[3 * i + d] : 0.0);
  }
  RowSums S;
  for (int col = 0; col < ncolors; ++col) {
    for (int32_t t = color_off[col] + sub * 32 + lane; valid && t < color_off[col + 1]; t += 32 * ASM_W) {
      int32_t el[6];
      bool near = false;
#pragma unroll
      for (int a = 0; a < 6; ++a) {
        el[a] = esort[a * E + t];  // `elems` in colour order (k_points_to32_sorted)
        near |= (el[a] == i);
      }
      if (near) continue;
      float hr[6], hi[6], gr[6], gi[6];
#pragma unroll
      for (int a = 0; a < 6; ++a) { hr[a] = hi[a] = gr[a] = gi[a] = 0.f; }
      // the element's share of the row sums in FP32 (Q terms), then one compensated addition each
      float ear = 0.f, eai = 0.f, ebr = 0.f, ebi = 0.f;
      for (int qq = 0; qq < Q; ++qq) {
        float q[P32COUNT];
#pragma unroll
        for (int f = 0; f < P32COUNT; ++f) q[f] = qtab[((int64_t)f * Q + qq) * E + t];
        Kern32 K;
        kernel32(k, kinv, xi, nui, tp, q, K, far_r2);
        const float wj = q[P32W];
        ear = __fmaf_rn(wj, K.alr, ear); eai = __fmaf_rn(wj, K.ali, eai);
        ebr = __fmaf_rn(wj, K.ber, ebr); ebi = __fmaf_rn(wj, K.bei, ebi);
#pragma unroll
        for (int a = 0; a < 6; ++a) {
          const float cw = wj * shp[qq * 6 + a];
          hr[a] = __fmaf_rn(cw, K.dGr, hr[a]); hi[a] = __fmaf_rn(cw, K.dGi, hi[a]);
          gr[a] = __fmaf_rn(cw, K.Gr, gr[a]);  gi[a] = __fmaf_rn(cw, K.Gi, gi[a]);
        }
      }
      S.ar.add(ear); S.ai.add(eai);
      S.br.add(ebr); S.bi.add(ebi);
#pragma unroll
      for (int a = 0; a < 6; ++a) {
        const int32_t j = el[a];
        const float kr = (float)kn[j].re, ki = (float)kn[j].im;
        if (bc[j] == 0) {  // hard column: A += H, b += Gm P'_known
          row[j].re += hr[a]; row[j].im += hi[a];
          S.sr.add(gr[a] * kr - gi[a] * ki); S.si.add(gr[a] * ki + gi[a] * kr);
        } else {           // soft column: A -= Gm, b -= H P_known
          row[j].re -= gr[a]; row[j].im -= gi[a];
          S.sr.add(-(hr[a] * kr - hi[a] * ki)); S.si.add(-(hr[a] * ki + hi[a] * kr));
        }
      }
    }
    bar_named(1 + rw, 32 * ASM_W);  // the row's warps finish the colour (rows <= 8: ids 1..8)
  }
  // reduce the compensated sums across the warp in FP64 (12 values per row)
  double v[12] = {(double)S.ar.s, (double)S.ar.c, (double)S.ai.s, (double)S.ai.c, (double)S.br.s, (double)S.br.c,
                  (double)S.bi.s, (double)S.bi.c, (double)S.sr.s, (double)S.sr.c, (double)S.si.s, (double)S.si.c};
  double out[6];
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    double x = v[2 * t] + v[2 * t + 1];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    out[t] = x;
  }
  if (lane == 0)
    for (int t = 0; t < 6; ++t) part[rw][sub][t] = out[t];
  __syncthreads();
  if (!valid) return;
  cf* Arow = A + ((int64_t)kk * N + i) * lda;
  for (int64_t j = sub * 32 + lane; j < N; j += 32 * ASM_W) Arow[j] = row[j];
  if (sub == 0 && lane == 0) {
    double* rs = rowsum + ((int64_t)kk * N + i) * 6;
    for (int t = 0; t < 6; ++t) {
      double v = 0.0;
      for (int w = 0; w < ASM_W; ++w) v += part[rw][w][t];
      rs[t] = v;
    }
  }
}

// Known boundary values at the quadrature points of the colour-sorted elements:
//   kq[k][qq][t] = sum_a N_a(q_qq) known[k][el_t[a]]  (FP32 complex)
// so that an element whose six nodes share one boundary condition adds its right-hand-side share
// as sum_q w_q K_q kq_q (K = G on a hard element, -dG/dnu on a soft one) instead of carrying the
// six nodal sums of both kernels.  pair: wavenumbers 2 m and 2 m + 1 interleaved,
//   kq[2 m][qq][t] as float4 {re, re, im, im} (a last wavenumber alone as without pair).
// grid (ceil(E / 256), nk), block 256.
__global__ void k_known_q32(const int32_t* __restrict__ esort, int64_t E, int Q, const float* __restrict__ qshape,
                            const cd* __restrict__ known, int64_t N, cf* __restrict__ kq, int pair) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int kk = blockIdx.y;
  if (t >= E) return;
  cd kn[6];
#pragma unroll
  for (int a = 0; a < 6; ++a) kn[a] = known[(int64_t)kk * N + esort[a * E + t]];
  for (int qq = 0; qq < Q; ++qq) {
    double sr = 0.0, si = 0.0;
#pragma unroll
    for (int a = 0; a < 6; ++a) {
      const double sh = qshape[qq * 6 + a];
      sr += sh * kn[a].re;
      si += sh * kn[a].im;
    }
    if (pair && (kk | 1) < (int)gridDim.y) {
      float* o = reinterpret_cast<float*>(kq + ((int64_t)(kk & ~1) * Q + 2 * qq) * E + 2 * t) + (kk & 1);
      o[0] = (float)sr;
      o[2] = (float)si;
    } else {
      kq[((int64_t)kk * Q + qq) * E + t] = {(float)sr, (float)si};
    }
  }
}

// Bulk assembly for meshes whose elements each carry one boundary condition on all six nodes
// (every element of a sound-hard or sound-soft body), two wavenumbers per thread in the halves of
// packed FP32 registers: the geometry of a (row, quadrature point) pair -- float-float r, R, nu_i.r,
// r.nu_q -- is formed once, and each half goes through the operations of the one-wavenumber kernel
// below in its order (its own float-float phases, no recurrence: every entry keeps the accuracy of
// the one-wavenumber kernel; the same entries bit for bit).
// Per element a lane carries the six nodal sums of the one kernel that enters A (dG/dnu on a hard
// element, -G on a soft one), the right-hand-side sum against the interpolated known values kq, and
// the two regularisation sums.  A CTA is one row's 2 ASM_W warps: ASM_W warps take consecutive
// elements of a colour and a second set of ASM_W warps the other half of the same elements' quadrature
// points, so that the registers fit 16 warps per SM; the halves add into the row one after the other
// (a barrier in between: fixed order, deterministic sums).  One row per CTA: four independent CTAs
// to an SM wait for each other's barriers least.
// grid (N, ceil(nk / 2)); block 32 * 2 ASM_W.  Where a row accumulates:
//   MODE 0: shared memory, both wavenumbers' entries side by side, N float4;
//   MODE 1 (large N): A itself, each row owned by one CTA and the row's warps ordered by the same
//     barriers (scattered read-modify-writes in L2);
//   MODE 2 (large N cut into column windows, see build_colouring): shared memory, ws float4, one
//     window of columns after the other -- the window's elements of every colour, then the window
//     copied to A -- so that each entry of A is written once.
// Bound: issue slots and dependent latencies at 16 warps (FMA pipe about 60 %).  Measured, 64
// wavenumbers, the whole assembly: N = 2884 39.8 -> 31.7 ms, N = 1002 7.0 -> 5.6, two wavenumbers at
// N = 10 272 15.5 -> 12.3; of it packing gave 7 %, the first point's record, condition and nodes
// loaded together (not one after the other) 5 %, one row instead of two per CTA 10 %.  Three rows of
// 168 registers (12 warps) measured 33.4, more rows a CTA slower.
template <int MODE>
__global__ void __launch_bounds__(32 * 2 * ASM_W, 4) k_asm32_pair(
    const double* __restrict__ nodes, const double* __restrict__ normals, const uint8_t* __restrict__ esoft, bool flip,
    const int32_t* __restrict__ esort, int64_t N, int64_t E, int Q, const float4* __restrict__ qaos,
    const float* __restrict__ qshape, const int32_t* __restrict__ color_off, int ncolors,
    const double* __restrict__ kv, int nk, const cf* __restrict__ kq, cf* __restrict__ A, int64_t lda,
    double* __restrict__ rowsum /* [nk][N][6] */, float far_r2,
    const int32_t* __restrict__ win_lo, const int32_t* __restrict__ wcol_off, int nwin, int ws) {
  constexpr bool GROW = MODE == 1;
  constexpr int QS = 2, WR = ASM_W * QS;  // warps per row
  extern __shared__ float4 accp[];
  __shared__ float4 shp[64 * 3];  // shape values, each twice: {N0, N0, N1, N1}, ...
  __shared__ double part[WR][2][6];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wr = warp, sub = wr % ASM_W, h = wr / ASM_W;
  const int k0 = blockIdx.y * 2;
  const int nkb = min(2, nk - k0);  // a ragged last group repeats its wavenumber in the second half
  f2 kh, nkh, nkl, kinv;
  bool zero;
  {
    const ff a = ff_from_double(kv[k0]), b = ff_from_double(kv[k0 + nkb - 1]);
    kh = f2_make(a.hi, b.hi);
    nkh = f2_make(-a.hi, -b.hi);
    nkl = f2_make(-a.lo, -b.lo);
    const float ia = kinv32(kv[k0]), ib = kinv32(kv[k0 + nkb - 1]);
    kinv = f2_make(ia, ib);
    zero = ia == 0.f || ib == 0.f;
  }
  for (int t = threadIdx.x; t < Q * 3; t += blockDim.x) {
    const float a = qshape[2 * t], b = qshape[2 * t + 1];
    shp[t] = make_float4(a, a, b, b);
  }
  const int64_t i = blockIdx.x;
  // the row: in shared memory, or (GROW) row i of system k0 + j in A
  float4* row = accp;
  auto grow = [&](int j) -> cf* { return A + ((int64_t)(k0 + j) * N + i) * lda; };
  if constexpr (GROW) {
    for (int j = 0; j < nkb; ++j) {
      cf* r = grow(j);
      for (int64_t c2 = threadIdx.x; c2 < N; c2 += 32 * WR) r[c2] = {0.f, 0.f};
    }
  } else if constexpr (MODE == 0) {
    for (int64_t t = threadIdx.x; t < N; t += 32 * WR) row[t] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();
  const int qlo = h * Q / QS, qhi = (h + 1) * Q / QS;
  ff xi[3], nui[3];
  for (int d = 0; d < 3; ++d) {
    xi[d] = ff_from_double(nodes[3 * i + d]);
    nui[d] = ff_from_double(normals[3 * i + d]);
  }
  // compensated sums (s, c): alpha, beta and the right-hand side, re and im
  f2 ss[6], sc[6];
#pragma unroll
  for (int t = 0; t < 6; ++t) ss[t].v = sc[t].v = 0ull;
  const int nw = MODE == 2 ? nwin : 1;
  for (int w = 0; w < nw; ++w) {
  int w0 = 0;
  if constexpr (MODE == 2) {  // the row's window accumulator starts at zero
    w0 = win_lo[w];
    const int ww = win_lo[w + 1] - w0;
    for (int c2 = threadIdx.x; c2 < ww; c2 += 32 * WR) row[c2] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
  }
  for (int col = 0; col < ncolors; ++col) {
    int32_t cbeg, cend;
    if constexpr (MODE == 2) {
      cbeg = wcol_off[col * (nwin + 1) + w];
      cend = wcol_off[col * (nwin + 1) + w + 1];
    } else {
      cbeg = color_off[col];
      cend = color_off[col + 1];
    }
    const int iters = (cend - cbeg + 32 * ASM_W - 1) / (32 * ASM_W);
    for (int it = 0; it < iters; ++it) {
      const int32_t t = cbeg + it * 32 * ASM_W + sub * 32 + lane;
      bool act = t < cend;
      // the first point's 64-byte record (colour-sorted, point-major: four 16-byte loads), its known
      // values, the element's condition and nodes: independent loads, issued together
      const int32_t ts = act ? t : cbeg;
      const float4* qp = qaos + ((int64_t)qlo * E + ts) * 4;
      float4 v0 = qp[0], v1 = qp[1], v2 = qp[2], v3 = qp[3];
      const cf* kqp = kq + (int64_t)k0 * Q * E;
      auto known = [&](int qq) -> float4 {  // {re, re, im, im} of the two wavenumbers
        const int64_t at = (int64_t)qq * E + ts;
        if (nkb == 2) return reinterpret_cast<const float4*>(kqp)[at];
        const cf v = kqp[at];
        return make_float4(v.re, v.re, v.im, v.im);
      };
      float4 kqn = known(qlo);
      const bool soft = (esoft[ts] != 0) != flip;
      int32_t el[6];
#pragma unroll
      for (int a = 0; a < 6; ++a) el[a] = esort[a * E + ts];
#pragma unroll
      for (int a = 0; a < 6; ++a)
        if (el[a] == i) act = false;  // near pair: the near kernel's
      f2 ar[6], ai[6];
#pragma unroll
      for (int a = 0; a < 6; ++a) ar[a].v = ai[a].v = 0ull;
      if (act) {
        f2 es[6];  // the element's share of the six sums
#pragma unroll
        for (int u = 0; u < 6; ++u) es[u].v = 0ull;
        // (the next point's record and known values are loaded while this one's are used)
        for (int qq = qlo; qq < qhi; ++qq) {
          const float q[P32COUNT] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w, v2.x, v2.y, v2.z, v2.w, v3.x};
          const float4 kqc = kqn;
          if (qq + 1 < qhi) {
            const float4* qn = qaos + ((int64_t)(qq + 1) * E + ts) * 4;
            v0 = qn[0]; v1 = qn[1]; v2 = qn[2]; v3 = qn[3];
            kqn = known(qq + 1);
          }
          // geometry, shared by the two wavenumbers
          // float-float geometry with lazy tails (distance, 1/R, nu_i.r)
          const ff rx = ff_diff_lazy(ff{q[0], q[3]}, xi[0]);
          const ff ry = ff_diff_lazy(ff{q[1], q[4]}, xi[1]);
          const ff rz = ff_diff_lazy(ff{q[2], q[5]}, xi[2]);
          const ff R2 = ff_norm2_lazy(rx, ry, rz);
          float invR;
          const ff R = ff_sqrt_lazy(R2, invR);
          const ff nr = ff_dot3_lazy(nui, rx, ry, rz);
          float rnu;
          if (R2.hi > far_r2) {
            rnu = (rx.hi + rx.lo) * q[6] + (ry.hi + ry.lo) * q[7] + (rz.hi + rz.lo) * q[8];
          } else {
            const ff nq[3] = {ff{q[6], q[10]}, ff{q[7], q[11]}, ff{q[8], q[12]}};
            const ff d = ff_dot3_lazy(nq, rx, ry, rz);
            rnu = d.hi + d.lo;
          }
          const float nn = nui[0].hi * q[6] + nui[1].hi * q[7] + nui[2].hi * q[8];
          const float wj = q[P32W];
          // the weight rides on 1/R and on r.nu/R^3: G and dG/dnu below are w G and w dG/dnu
          const float wiR = wj * invR, wrn = wj * (rnu * invR * invR * invR);
          f2 c, s, cg, sg;
          cis_ffprod2(nkh, nkl, R, c, s);
          cis_ffprod2(nkh, nkl, nr, cg, sg);
          const f2 kR = f2_mul(kh, f2_dup(R.hi)), wiR2 = f2_dup(wiR);
          const f2 Gr = f2_mul(c, wiR2), Gi = f2_mul(s, wiR2);
          const f2 dGr = f2_mul(f2_fma(s, kR, c), f2_dup(-wrn));
          const f2 dGi = f2_mul(f2_fma(c, kR, f2_neg(s)), f2_dup(wrn));
          f2 f = f2_mul(sg, kinv);
          if (zero) {  // f's limit nu_i.r at k = 0
            float f0, f1, i0, i1;
            f2_split(f, f0, f1);
            f2_split(kinv, i0, i1);
            f = f2_make(i0 != 0.f ? f0 : nr.hi, i1 != 0.f ? f1 : nr.hi);
          }
          const f2 ndg = f2_mul(f2_mul(kh, sg), f2_dup(nn)), ndf = f2_mul(cg, f2_dup(-nn));
          es[0] = f2_fma(cg, dGr, f2_fma(ndg, Gr, es[0]));
          es[1] = f2_fma(cg, dGi, f2_fma(ndg, Gi, es[1]));
          es[2] = f2_fma(f, dGr, f2_fma(ndf, Gr, es[2]));
          es[3] = f2_fma(f, dGi, f2_fma(ndf, Gi, es[3]));
          // into A: dG (hard) or -G (soft); into b: G kq (hard) or -dG kq (soft)
          f2 war = dGr, wai = dGi, wbr = Gr, wbi = Gi;
          if (soft) {
            war = f2_neg(Gr); wai = f2_neg(Gi);
            wbr = f2_neg(dGr); wbi = f2_neg(dGi);
          }
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const float4 sh = shp[qq * 3 + a];
            const f2 s0 = f2_make(sh.x, sh.y), s1 = f2_make(sh.z, sh.w);
            ar[2 * a] = f2_fma(s0, war, ar[2 * a]);
            ai[2 * a] = f2_fma(s0, wai, ai[2 * a]);
            ar[2 * a + 1] = f2_fma(s1, war, ar[2 * a + 1]);
            ai[2 * a + 1] = f2_fma(s1, wai, ai[2 * a + 1]);
          }
          const f2 kr = f2_make(kqc.x, kqc.y), ki = f2_make(kqc.z, kqc.w);
          es[4] = f2_fma(wbr, kr, f2_fma(wbi, f2_neg(ki), es[4]));
          es[5] = f2_fma(wbr, ki, f2_fma(wbi, kr, es[5]));
        }
#pragma unroll
        for (int u = 0; u < 6; ++u) {  // ksum::add, packed
          const f2 a = ss[u], b = es[u];
          const f2 sum = f2_add(a, b), bb = f2_sub(sum, a);
          sc[u] = f2_add(sc[u], f2_add(f2_sub(a, f2_sub(sum, bb)), f2_sub(b, bb)));
          ss[u] = sum;
        }
      }
      // scatter into the row: the quadrature halves one after the other
#pragma unroll
      for (int hh = 0; hh < QS; ++hh) {
        if (act && h == hh) {
#pragma unroll
          for (int a = 0; a < 6; ++a) {
            if constexpr (GROW) {
              float r0, r1, i0, i1;
              f2_split(ar[a], r0, r1);
              f2_split(ai[a], i0, i1);
              cf* g = grow(0) + el[a];
              g->re += r0;
              g->im += i0;
              if (nkb == 2) {  // no system behind a ragged group's second half
                g = grow(1) + el[a];
                g->re += r1;
                g->im += i1;
              }
            } else {
              float4* g = row + (el[a] - w0);
              const float4 v = *g;
              const f2 r = f2_add(f2_make(v.x, v.y), ar[a]), m = f2_add(f2_make(v.z, v.w), ai[a]);
              float4 o;
              f2_split(r, o.x, o.y);
              f2_split(m, o.z, o.w);
              *g = o;
            }
          }
        }
        __syncthreads();
      }
    }
  }
  if constexpr (MODE == 2) {  // the window to A, then its accumulator is free for the next one
    __syncthreads();
    const int ww = win_lo[w + 1] - w0;
    for (int c2 = threadIdx.x; c2 < ww; c2 += 32 * WR) {
      const float4 v = row[c2];
      grow(0)[w0 + c2] = cf{v.x, v.z};
      if (nkb == 2) grow(1)[w0 + c2] = cf{v.y, v.w};
    }
    __syncthreads();
  }
  }  // windows
  // reduce the compensated sums across the warp in FP64 (6 values per row and wavenumber)
#pragma unroll
  for (int u = 0; u < 6; ++u) {
    float s2[2], c2[2];
    f2_split(ss[u], s2[0], s2[1]);
    f2_split(sc[u], c2[0], c2[1]);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      double x = (double)s2[j] + (double)c2[j];
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if (lane == 0) part[wr][j][u] = x;
    }
  }
  __syncthreads();
  if constexpr (MODE == 0)
    for (int64_t c2 = threadIdx.x; c2 < N; c2 += 32 * WR) {
      const float4 v = row[c2];
      grow(0)[c2] = cf{v.x, v.z};
      if (nkb == 2) grow(1)[c2] = cf{v.y, v.w};
    }
  for (int j = 0; j < nkb; ++j)
    if (wr == 0 && lane < 6) {
      double x = 0.0;
      for (int w = 0; w < WR; ++w) x += part[w][j][lane];
      rowsum[((int64_t)(k0 + j) * N + i) * 6 + lane] = x;
    }
}

// Bulk assembly for meshes whose elements each carry one boundary condition on all six nodes
// (every element of a sound-hard or sound-soft body), one wavenumber per thread ("mixed.asm_kb" 1).
// Per element a lane carries the six nodal sums of the one kernel that enters A (dG/dnu on a hard
// element, -G on a soft one), the right-hand-side sum against the interpolated known values kq, and
// the two regularisation sums.  A row has ASM_W warps, which take consecutive elements of a colour.
// grid (ceil(N / rows), nk); block 32 * rows * ASM_W.  Where a row accumulates:
//   MODE 0: shared memory, rows * N cf;
//   MODE 1 (large N): A itself, each row owned by one CTA and the row's warps ordered by the same
//     barriers (scattered read-modify-writes in L2).
template <int MODE>
__global__ void __launch_bounds__(256, 2) k_asm32_bulk_u(
    const double* __restrict__ nodes, const double* __restrict__ normals, const uint8_t* __restrict__ bc,
    const int32_t* __restrict__ esort, int64_t N, int64_t E, int Q, const float4* __restrict__ qaos,
    const float* __restrict__ qshape, const int32_t* __restrict__ color_off, int ncolors,
    const double* __restrict__ kv, const cf* __restrict__ kq, cf* __restrict__ A, int64_t lda,
    double* __restrict__ rowsum /* [nk][N][6] */, int rows, float far_r2) {
  constexpr bool GROW = MODE == 1;
  extern __shared__ cf acc32[];
  __shared__ float shp[64 * 6];
  __shared__ double part[8][ASM_W][6];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rw = warp / ASM_W, sub = warp % ASM_W;
  const int kk = blockIdx.y;
  const ff k = ff_from_double(kv[kk]);
  const float kinv = kinv32(kv[kk]);
  for (int t = threadIdx.x; t < Q * 6; t += blockDim.x) shp[t] = qshape[t];
  const int64_t i = (int64_t)blockIdx.x * rows + rw;
  const bool valid = i < N;
  cf* Arow = A + ((int64_t)kk * N + (valid ? i : 0)) * lda;
  cf* row = GROW ? Arow : acc32 + (int64_t)rw * N;
  if constexpr (GROW) {
    if (valid)
      for (int64_t c2 = sub * 32 + lane; c2 < N; c2 += 32 * ASM_W) row[c2] = {0.f, 0.f};
  } else {
    for (int64_t t = threadIdx.x; t < (int64_t)rows * N; t += blockDim.x) acc32[t] = {0.f, 0.f};
  }
  __syncthreads();
  ff xi[3], nui[3];
  for (int d = 0; d < 3; ++d) {
    xi[d] = ff_from_double(valid ? nodes[3 * i + d] : 0.0);
    nui[d] = ff_from_double(valid ? normals[3 * i + d] : 0.0);
  }
  RowSums S;
  for (int col = 0; col < ncolors; ++col) {
    const int32_t cbeg = color_off[col], cend = color_off[col + 1];
    for (int32_t t = cbeg + sub * 32 + lane; valid && t < cend; t += 32 * ASM_W) {
      bool act = true;
      int32_t el[6];
#pragma unroll
      for (int a = 0; a < 6; ++a) {
        el[a] = esort[a * E + t];
        if (el[a] == i) act = false;  // near pair: the near kernel's
      }
      if (!act) continue;
      float ar[6], ai[6];
#pragma unroll
      for (int a = 0; a < 6; ++a) ar[a] = ai[a] = 0.f;
      const bool soft = bc[el[0]] != 0;
      float sr = 0.f, si = 0.f, ear = 0.f, eai = 0.f, ebr = 0.f, ebi = 0.f;
      // the point's 64-byte record (colour-sorted, point-major: four 16-byte loads); the next
      // point's is loaded while this one is computed
      const float4* qp = qaos + (int64_t)t * 4;
      float4 v0 = qp[0], v1 = qp[1], v2 = qp[2], v3 = qp[3];
      const cf* kqp = kq + (int64_t)kk * Q * E + t;
      cf kqn = kqp[0];
      for (int qq = 0; qq < Q; ++qq) {
        const float q[P32COUNT] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w, v2.x, v2.y, v2.z, v2.w, v3.x};
        const cf kqv = kqn;
        if (qq + 1 < Q) {
          const float4* qn = qaos + ((int64_t)(qq + 1) * E + t) * 4;
          v0 = qn[0]; v1 = qn[1]; v2 = qn[2]; v3 = qn[3];
          kqn = kqp[(int64_t)(qq + 1) * E];
        }
        // float-float geometry with lazy tails (distance, 1/R, nu_i.r)
        const ff rx = ff_diff_lazy(ff{q[0], q[3]}, xi[0]);
        const ff ry = ff_diff_lazy(ff{q[1], q[4]}, xi[1]);
        const ff rz = ff_diff_lazy(ff{q[2], q[5]}, xi[2]);
        const ff R2 = ff_norm2_lazy(rx, ry, rz);
        float invR;
        const ff R = ff_sqrt_lazy(R2, invR);
        const ff nr = ff_dot3_lazy(nui, rx, ry, rz);
        float rnu;
        if (R2.hi > far_r2) {
          rnu = (rx.hi + rx.lo) * q[6] + (ry.hi + ry.lo) * q[7] + (rz.hi + rz.lo) * q[8];
        } else {
          const ff nq[3] = {ff{q[6], q[10]}, ff{q[7], q[11]}, ff{q[8], q[12]}};
          const ff d = ff_dot3_lazy(nq, rx, ry, rz);
          rnu = d.hi + d.lo;
        }
        const float nn = nui[0].hi * q[6] + nui[1].hi * q[7] + nui[2].hi * q[8];
        const float wj = q[P32W];
        // the weight rides on 1/R and on r.nu/R^3: G and dG/dnu below are w G and w dG/dnu
        const float wiR = wj * invR, wrn = wj * (rnu * invR * invR * invR);
        float c, s;
        cis_ffprod(k, R, c, s);
        const float kR = k.hi * R.hi;
        const float Gr = c * wiR, Gi = s * wiR;
        const float dGr = (-c - s * kR) * wrn, dGi = (c * kR - s) * wrn;
        float cg, sg;
        cis_ffprod(k, nr, cg, sg);
        const float g = cg, f = kinv != 0.f ? sg * kinv : nr.hi, dg = -k.hi * sg * nn, df = cg * nn;
        ear = __fmaf_rn(g, dGr, __fmaf_rn(-dg, Gr, ear));
        eai = __fmaf_rn(g, dGi, __fmaf_rn(-dg, Gi, eai));
        ebr = __fmaf_rn(f, dGr, __fmaf_rn(-df, Gr, ebr));
        ebi = __fmaf_rn(f, dGi, __fmaf_rn(-df, Gi, ebi));
        // into A: dG (hard) or -G (soft); into b: G kq (hard) or -dG kq (soft)
        const float war = soft ? -Gr : dGr, wai = soft ? -Gi : dGi;
        const float wbr = soft ? -dGr : Gr, wbi = soft ? -dGi : Gi;
#pragma unroll
        for (int a = 0; a < 6; ++a) {
          const float sh = shp[qq * 6 + a];
          ar[a] = __fmaf_rn(sh, war, ar[a]);
          ai[a] = __fmaf_rn(sh, wai, ai[a]);
        }
        sr = __fmaf_rn(wbr, kqv.re, __fmaf_rn(-wbi, kqv.im, sr));
        si = __fmaf_rn(wbr, kqv.im, __fmaf_rn(wbi, kqv.re, si));
      }
      S.ar.add(ear); S.ai.add(eai);
      S.br.add(ebr); S.bi.add(ebi);
      S.sr.add(sr); S.si.add(si);
#pragma unroll
      for (int a = 0; a < 6; ++a) {
        row[el[a]].re += ar[a];
        row[el[a]].im += ai[a];
      }
    }
    bar_named(1 + rw, 32 * ASM_W);  // the row's warps finish the colour (rows <= 8: ids 1..8)
  }
  // reduce the compensated sums across the warp in FP64 (6 values per row)
  const ksum* v[6] = {&S.ar, &S.ai, &S.br, &S.bi, &S.sr, &S.si};
#pragma unroll
  for (int u = 0; u < 6; ++u) {
    double x = (double)v[u]->s + (double)v[u]->c;
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) part[rw][sub][u] = x;
  }
  __syncthreads();
  if (!valid) return;
  if constexpr (!GROW)
    for (int64_t c2 = sub * 32 + lane; c2 < N; c2 += 32 * ASM_W) Arow[c2] = row[c2];
  if (sub == 0 && lane < 6) {
    double x = 0.0;
    for (int w = 0; w < ASM_W; ++w) x += part[rw][w][lane];
    rowsum[((int64_t)kk * N + i) * 6 + lane] = x;
  }
}

// One level of a warp's halving exchange: v[0 .. 2 HALF) per lane; the lane keeps the upper or
// lower half (by `upper`), adds its partner's (lane ^ o) copy of that half and stores it in
// v[0 .. HALF).
template <int HALF, class T>
__device__ __forceinline__ void halving_exchange(T* v, int o, bool upper) {
#pragma unroll
  for (int m = 0; m < HALF; ++m) {
    const T send = upper ? v[m] : v[m + HALF];
    const T keep = upper ? v[m + HALF] : v[m];
    v[m] = keep + __shfl_xor_sync(0xffffffffu, send, o);
  }
}

// Near pairs (element contains node i) and the diagonal terms; one warp per row.
__global__ void __launch_bounds__(128) k_asm32_near(
    const double* __restrict__ nodes, const double* __restrict__ normals, const uint8_t* __restrict__ bc,
    const int32_t* __restrict__ elems, int64_t N, int64_t E, int QN, const int* __restrict__ nnear_d,
    const float4* __restrict__ naos, const float* __restrict__ nshape, const int32_t* __restrict__ n2e_off,
    const int32_t* __restrict__ n2e, const double* __restrict__ kv, const cd* __restrict__ known,
    cf* __restrict__ A, int64_t lda, const double* __restrict__ rowsum, cd* __restrict__ b, TwoPi3 tp) {
  const int lane = threadIdx.x & 31;
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int kk = blockIdx.y;
  if (i >= N) return;
  const ff k = ff_from_double(kv[kk]);
  const float kinv = kinv32(kv[kk]);
  const cd* kn = known + (int64_t)kk * N;
  ff xi[3], nui[3];
  for (int d = 0; d < 3; ++d) {
    xi[d] = ff_from_double(nodes[3 * i + d]);
    nui[d] = ff_from_double(normals[3 * i + d]);
  }
  cf* Arow = A + ((int64_t)kk * N + i) * lda;
  // The regularisation sums per lane in compensated FP32 (they cancel against the bulk's) and the
  // nodal sums per lane in FP32 (a lane holds a few points of one element); across the warp the
  // nodal sums are reduced by halving exchanges, so that each of six lanes ends with one node's
  // four sums, and the right-hand side accumulates in float-float: the GB300's FP64 pipe is too
  // narrow for per-point FP64 arithmetic here (per element, six lanes split their node's known
  // value into float-float: two FP64 conversions and subtractions each).
  ksum sal_r, sal_i, sbe_r, sbe_i;
  ff bsr = {0.f, 0.f}, bsi = {0.f, 0.f};
  const int node = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
  for (int32_t t = n2e_off[i]; t < n2e_off[i + 1]; ++t) {
    const int32_t e = n2e[t] >> 3, a0 = n2e[t] & 7;
    const int np = nnear_d[a0];
    float hr[6], hi[6], gr[6], gi[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) { hr[a] = hi[a] = gr[a] = gi[a] = 0.f; }
    for (int qq = lane; qq < np; qq += 32) {
      const float4* qp = naos + (((int64_t)e * 6 + a0) * QN + qq) * 4;  // the point's 64-byte record
      const float4 v0 = qp[0], v1 = qp[1], v2 = qp[2], v3 = qp[3];
      const float q[P32COUNT] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w, v2.x, v2.y, v2.z, v2.w, v3.x};
      Kern32 K;
      kernel32(k, kinv, xi, nui, tp, q, K);
      const float wj = q[P32W];
      // w K enters exactly: the product's rounding error joins the compensation term
      auto add_exact = [&](ksum& acc, float x) {
        const float p = wj * x;
        acc.add(p);
        acc.c += __fmaf_rn(wj, x, -p);
      };
      add_exact(sal_r, K.alr); add_exact(sal_i, K.ali);
      add_exact(sbe_r, K.ber); add_exact(sbe_i, K.bei);
      const float* sh = nshape + ((int64_t)a0 * QN + qq) * 6;
#pragma unroll
      for (int a = 0; a < 6; ++a) {
        const float cw = wj * sh[a];
        hr[a] = __fmaf_rn(cw, K.dGr, hr[a]); hi[a] = __fmaf_rn(cw, K.dGi, hi[a]);
        gr[a] = __fmaf_rn(cw, K.Gr, gr[a]);  gi[a] = __fmaf_rn(cw, K.Gi, gi[a]);
      }
    }
    // node a: u[4a .. 4a+3] = h re, h im, g re, g im; nodes 6, 7 are padding.  The first two
    // levels add partial sums of 2 and 4 lanes in FP32 (small against the total), the rest in
    // float-float (FP32 pipes: the FP64 pipe of the GB300 is too narrow for this reduction).
    float u[32];
#pragma unroll
    for (int a = 0; a < 6; ++a) {
      u[4 * a] = hr[a]; u[4 * a + 1] = hi[a]; u[4 * a + 2] = gr[a]; u[4 * a + 3] = gi[a];
    }
#pragma unroll
    for (int m = 24; m < 32; ++m) u[m] = 0.f;
    halving_exchange<16>(u, 16, (lane & 16) != 0);
    halving_exchange<8>(u, 8, (lane & 8) != 0);
    ff v[4];
    {
      const bool up = (lane & 4) != 0;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float send = up ? u[m] : u[m + 4], keep = up ? u[m + 4] : u[m];
        v[m] = ff_two_sum(keep, __shfl_xor_sync(0xffffffffu, send, 4));
      }
    }
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int o = 2; o > 0; o >>= 1) {
        const ff r = {__shfl_xor_sync(0xffffffffu, v[m].hi, o), __shfl_xor_sync(0xffffffffu, v[m].lo, o)};
        v[m] = ff_add(v[m], r);
      }
    if ((lane & 3) == 0 && node < 6) {  // this lane holds node `node`'s sums
      const int32_t j = elems[6 * (int64_t)e + node];
      const ff kr = ff_from_double(kn[j].re), ki = ff_from_double(kn[j].im);
      if (bc[j] == 0) {  // hard column: A += H, b += G known
        Arow[j].re += __fadd_rn(v[0].hi, v[0].lo); Arow[j].im += __fadd_rn(v[1].hi, v[1].lo);
        bsr = ff_add(bsr, ff_sub(ff_mul(v[2], kr), ff_mul(v[3], ki)));
        bsi = ff_add(bsi, ff_add(ff_mul(v[2], ki), ff_mul(v[3], kr)));
      } else {           // soft column: A -= G, b -= H known
        Arow[j].re -= __fadd_rn(v[2].hi, v[2].lo); Arow[j].im -= __fadd_rn(v[3].hi, v[3].lo);
        bsr = ff_sub(bsr, ff_sub(ff_mul(v[0], kr), ff_mul(v[1], ki)));
        bsi = ff_sub(bsi, ff_add(ff_mul(v[0], ki), ff_mul(v[1], kr)));
      }
    }
    __syncwarp();  // the next element (sharing nodes with this one) updates after these writes
  }
  for (int o = 16; o > 0; o >>= 1) {
    bsr = ff_add(bsr, ff{__shfl_xor_sync(0xffffffffu, bsr.hi, o), __shfl_xor_sync(0xffffffffu, bsr.lo, o)});
    bsi = ff_add(bsi, ff{__shfl_xor_sync(0xffffffffu, bsi.hi, o), __shfl_xor_sync(0xffffffffu, bsi.lo, o)});
  }
  double bs_r = ff_to_double(bsr), bs_i = ff_to_double(bsi);
  double al_r = sal_r.value(), al_i = sal_i.value(), be_r = sbe_r.value(), be_i = sbe_i.value();
  for (int o = 16; o > 0; o >>= 1) {
    al_r += __shfl_xor_sync(0xffffffffu, al_r, o); al_i += __shfl_xor_sync(0xffffffffu, al_i, o);
    be_r += __shfl_xor_sync(0xffffffffu, be_r, o); be_i += __shfl_xor_sync(0xffffffffu, be_i, o);
  }
  if (lane == 0) {
    const double* rs = rowsum + ((int64_t)kk * N + i) * 6;
    al_r += rs[0]; al_i += rs[1]; be_r += rs[2]; be_i += rs[3];
    bs_r += rs[4]; bs_i += rs[5];
    const cd ki = kn[i];
    const double fr = 4.0 * kPi + al_r, fi = al_i;
    if (bc[i] == 0) {
      Arow[i].re -= (float)fr; Arow[i].im -= (float)fi;
      bs_r += be_r * ki.re - be_i * ki.im; bs_i += be_r * ki.im + be_i * ki.re;
    } else {
      Arow[i].re -= (float)be_r; Arow[i].im -= (float)be_i;
      bs_r += fr * ki.re - fi * ki.im; bs_i += fr * ki.im + fi * ki.re;
    }
    b[(int64_t)kk * N + i] = {bs_r, bs_i};
  }
}

__global__ void k_known64(const double* __restrict__ nodes, const double* __restrict__ normals,
                          const uint8_t* __restrict__ bc, int64_t N, const double* __restrict__ kv, double dx,
                          double dy, double dz, cd* __restrict__ known);

static TwoPi3 two_pi3() {
  const double tp = 2.0 * kPi;
  TwoPi3 r;
  r.c1 = (float)tp;
  r.c2 = (float)(tp - (double)r.c1);
  // third term from the FP64 remainder refined by a long-double-free split of 2 pi's digits
  const double tail = 2.4492935982947064e-16;  // 2 pi - fl64(2 pi)
  r.c3 = (float)((tp - (double)r.c1 - (double)r.c2) + tail);
  r.inv = (float)(1.0 / tp);
  return r;
}

// Layout of c->qgeo32: standard points [P32COUNT][E*Q] (element-major, used by the field kernels),
// near points [P32COUNT][E*6*QN], the colour-sorted standard points [P32COUNT][Q][E], then the
// colour-sorted connectivity as int32 [6][E].
static float* sorted_table(bie_ctx* c) {
  const int64_t nq = c->E * c->rule.Q, nn = c->E * 6 * (int64_t)c->rule.QN;
  return c->qgeo32 + P32COUNT * (nq + nn);
}
static int32_t* sorted_elems(bie_ctx* c) {
  return reinterpret_cast<int32_t*>(sorted_table(c) + P32COUNT * c->E * c->rule.Q);
}
// the colour-sorted points again as 64-byte records [Q][E][16 floats], 16-byte aligned
static size_t sorted_aos_offset(bie_ctx* c) {
  const int64_t nq = c->E * c->rule.Q, nn = c->E * 6 * (int64_t)c->rule.QN;
  return ((size_t)(P32COUNT * (2 * nq + nn) + 6 * c->E) + 63) / 64 * 64;
}
static float4* sorted_aos(bie_ctx* c) { return reinterpret_cast<float4*>(c->qgeo32 + sorted_aos_offset(c)); }
// the near points as 64-byte records [E * 6 * QN][16 floats], after the sorted records
static float4* near_aos(bie_ctx* c) {
  return reinterpret_cast<float4*>(c->qgeo32 + sorted_aos_offset(c) + 16 * (size_t)c->E * c->rule.Q);
}
// the colour-sorted elements' condition (of their first node), uint8 [E], after the near records
static size_t sorted_soft_offset(bie_ctx* c) {
  return sorted_aos_offset(c) + 16 * (size_t)(c->E * c->rule.Q + c->E * 6 * (int64_t)c->rule.QN);
}
static uint8_t* sorted_soft(bie_ctx* c) { return reinterpret_cast<uint8_t*>(c->qgeo32 + sorted_soft_offset(c)); }
const float4* sorted_aos_ptr(bie_ctx* c) { return sorted_aos(c); }

const float* sorted_table_ptr(bie_ctx* c) { return sorted_table(c); }
const int32_t* sorted_elems_ptr(bie_ctx* c) { return sorted_elems(c); }

int ensure_mixed_tables(bie_ctx* c) {
  if (c->qgeo32) return BIE_OK;
  const int64_t nq = c->E * c->rule.Q, nn = c->E * 6 * (int64_t)c->rule.QN;
  BIE_TRY(dev_alloc(c, (void**)&c->qgeo32, sorted_soft_offset(c) * sizeof(float) + (size_t)c->E));
  BIE_LAUNCH(k_points_to32<<<(unsigned)((nq + 255) / 256), 256, 0, c->stream>>>(c->qgeo, nq, c->qgeo32, nullptr));
  BIE_LAUNCH(k_points_to32<<<(unsigned)((nn + 255) / 256), 256, 0, c->stream>>>(c->ngeo, nn, c->qgeo32 + P32COUNT * nq,
                                                                                near_aos(c)));
  BIE_LAUNCH(k_points_to32_sorted<<<(unsigned)((nq + 255) / 256), 256, 0, c->stream>>>(
      c->qgeo, c->elem_perm, c->elems, c->bc == c->bc_flip, c->bc, c->E, c->rule.Q, sorted_table(c), sorted_elems(c),
      sorted_aos(c), sorted_soft(c)));
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

// Assembles nk FP32 systems: A [nk][N][lda] (cf), b [nk][N] (cd).  known [nk][N] (cd) receives the
// known boundary values; rowsum scratch: nk * N * 6 doubles; kq scratch: nk * E * Q cf (the known
// values at the quadrature points, used by the uniform-condition bulk kernel; may be NULL).
// (3 x longest element edge)^2: beyond it a pair's r.nu is formed in FP32 (once per geometry)
double far_radius2(bie_ctx* c) {
  if (!(c->far_r2 > 0.0)) {
    double h2 = 0.0;
    for (int64_t e = 0; e < c->E; ++e)
      for (int a = 0; a < 3; ++a) {
        const int32_t p = c->h_elems[6 * e + a], q = c->h_elems[6 * e + (a + 1) % 3];
        double d2 = 0.0;
        for (int x = 0; x < 3; ++x) {
          const double d = c->h_nodes[3 * p + x] - c->h_nodes[3 * q + x];
          d2 += d * d;
        }
        h2 = std::max(h2, d2);
      }
    c->far_r2 = 9.0 * h2;
  }
  return c->far_r2;
}

bool uniform_conditions(bie_ctx* c);

int assemble32(bie_ctx* c, const double* kv, int nk, cf* A, int64_t lda, cd* b, cd* known, double* rowsum, cf* kq) {
  const int64_t N = c->N;
  BIE_TRY(ensure_mixed_tables(c));
  dim3 gk((unsigned)((N + 255) / 256), nk);
  BIE_LAUNCH(k_known64<<<gk, 256, 0, c->stream>>>(c->nodes, c->normals, c->bc, N, kv, c->dir[0], c->dir[1], c->dir[2], known));
  int rows = 16 / ASM_W;
  while (rows > 1 && (size_t)rows * N * sizeof(cf) > 200 * 1024) rows /= 2;
  const size_t smem = (size_t)rows * N * sizeof(cf);
  if (smem > 200 * 1024)
    return fail(BIE_ERR_INVALID_ARG, "N = " + std::to_string(N) + " too large for the FP32 shared-memory row accumulator");
  if (c->rule.Q > 64) return fail(BIE_ERR_INVALID_ARG, "standard rule too large");
  const TwoPi3 tp = two_pi3();
  far_radius2(c);
  // the uniform-condition kernels: two wavenumbers per thread with the quadrature points of an
  // element split over two warps (one row, 128 threads), the row in shared memory while four CTAs
  // fit an SM, else (large N) window by window or in A itself; one per thread (4 rows x 2 warps) on
  // request
  int kb = (kq && uniform_conditions(c)) ? c->asm_kb : 0;
  if (kb >= 1) {
    const int64_t E = c->E;
    dim3 gq((unsigned)((E + 255) / 256), nk);
    BIE_LAUNCH(k_known_q32<<<gq, 256, 0, c->stream>>>(sorted_elems(c), E, c->rule.Q, c->qshape32, known, N, kq, kb == 2));
    if (kb == 2) {
      const size_t full = (size_t)N * sizeof(float4);
      const bool grow = full > 50 * 1024;
      // large N: window by window in shared memory where the mesh has column windows
      // ("asm.windows" 0 keeps the rows in A)
      const size_t part = (size_t)c->win_max * sizeof(float4);
      const bool win = grow && c->nwin > 1 && c->asm_windows != 0 && part <= 50 * 1024;
      dim3 gu((unsigned)N, (unsigned)((nk + 1) / 2));
      auto go = [&](auto kernel, size_t usmem) -> int {
        BIE_TRY(set_smem_max(kernel));
        BIE_LAUNCH(kernel<<<gu, 32 * 2 * ASM_W, usmem, c->stream>>>(
            c->nodes, c->normals, sorted_soft(c), c->bc == c->bc_flip, sorted_elems(c), N, E, c->rule.Q, sorted_aos(c),
            c->qshape32, c->color_off, c->ncolors, kv, nk, kq, A, lda, rowsum, (float)c->far_r2, c->win_lo, c->wcol_off, c->nwin, c->win_max));
        return BIE_OK;
      };
      if (win) BIE_TRY(go(k_asm32_pair<2>, part));
      else if (grow) BIE_TRY(go(k_asm32_pair<1>, 0));
      else BIE_TRY(go(k_asm32_pair<0>, full));
    } else {
      int urows = 4;
      while (urows > 1 && (size_t)urows * N * sizeof(cf) > 200 * 1024) urows /= 2;
      const bool grow = (size_t)urows * N * sizeof(cf) > 200 * 1024;
      if (grow) urows = 4;
      const size_t usmem = grow ? 0 : (size_t)urows * N * sizeof(cf);
      dim3 gu((unsigned)((N + urows - 1) / urows), (unsigned)nk);
      auto go = [&](auto kernel) -> int {
        BIE_TRY(set_smem_max(kernel));
        BIE_LAUNCH(kernel<<<gu, 32 * urows * ASM_W, usmem, c->stream>>>(
            c->nodes, c->normals, c->bc, sorted_elems(c), N, E, c->rule.Q, sorted_aos(c), c->qshape32, c->color_off,
            c->ncolors, kv, kq, A, lda, rowsum, urows, (float)c->far_r2));
        return BIE_OK;
      };
      if (grow) BIE_TRY(go(k_asm32_bulk_u<1>));
      else BIE_TRY(go(k_asm32_bulk_u<0>));
    }
  }
  if (kb == 0) {
    BIE_TRY((set_smem_max(k_asm32_bulk)));
    dim3 gb((unsigned)((N + rows - 1) / rows), nk);
    BIE_LAUNCH(k_asm32_bulk<<<gb, 32 * rows * ASM_W, smem, c->stream>>>(c->nodes, c->normals, c->bc, sorted_elems(c), N,
                                                                        c->E, c->rule.Q, sorted_table(c), c->qshape32,
                                                                        c->color_off, c->ncolors, kv, known, A, lda,
                                                                        rowsum, rows, tp, (float)c->far_r2));
  }
  BIE_CUDA_TRY(cudaGetLastError());
  dim3 gn((unsigned)((N * 32 + 127) / 128), nk);
  BIE_LAUNCH(k_asm32_near<<<gn, 128, 0, c->stream>>>(c->nodes, c->normals, c->bc, c->elems, N, c->E, c->rule.QN, c->d_nnear,
                                          near_aos(c), c->nshape32, c->n2e_off, c->n2e, kv, known, A, lda,
                                          rowsum, b, tp));
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

}  // namespace bie
