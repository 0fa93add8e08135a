// field.cu -- scattered field at observation points by the boundary-regularised representation
// Eq. (BRIEFdmn) (Sec. 3).  With the S_inf integrals evaluated analytically (App. B reasoning,
// applied to g and f about the foot point x0 and to the source points x_p and x0):
//   4 pi P(x_p) = 4 pi P0 + int_S { Pt [dG(x_p,x) - dG(x0,x)] - [G(x_p,x) - G(x0,x)] dPt } dS,
//   Pt = P(x) - P0 g(x) - P0' f(x),  dPt = P'(x) - P0 dg(x) - P0' df(x),
// g = cos(k nu0.(x - x0)), f = sin(k nu0.(x - x0)) / k, x0 the closest surface point of x_p,
// nu0 the surface normal there, P0 and P0' interpolated quadratically at x0.
//
// Layout: the surface values are first interpolated to every standard quadrature point
// (k_interp_q), then each CTA owns a tile of observation points for a group of wavenumbers and
// sweeps the quadrature points (an N-body style loop).
#include <algorithm>

#include "bie_common.cuh"

namespace bie {

// Pq[kk][p], Pnq[kk][p] = sum_a N_a(q) {P, P'}[node a of e], p = e*Q + q.
__global__ void k_interp_q64(const int32_t* __restrict__ elems, int64_t N, int64_t E, int Q,
                             const double* __restrict__ qshape, const cd* __restrict__ surf, cd* __restrict__ Pq,
                             cd* __restrict__ Pnq) {
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int kk = blockIdx.y;
  if (p >= E * Q) return;
  int64_t e = p / Q;
  int q = (int)(p % Q);
  const cd* P = surf + (int64_t)kk * 2 * N;
  const cd* Pn = P + N;
  cd a = {0, 0}, b = {0, 0};
  for (int t = 0; t < 6; ++t) {
    int32_t j = elems[6 * e + t];
    double s = qshape[q * 6 + t];
    a.re += s * P[j].re; a.im += s * P[j].im;
    b.re += s * Pn[j].re; b.im += s * Pn[j].im;
  }
  Pq[(int64_t)kk * E * Q + p] = a;
  Pnq[(int64_t)kk * E * Q + p] = b;
}

constexpr int FT = 128;  // points per CTA and quadrature points per shared tile (FP32 kernels)

// FP64 field.  A CTA evaluates 32 points (one per lane) for a group of F64K wavenumbers over its share z of
// `splits` of the quadrature points.  Per (point, quadrature point) pair the geometry is formed once; where
// the group's wavenumbers are equally spaced to rounding the three phases' sines and cosines are formed at
// k_0 and at the spacing and rotated to the others (at most F64K - 1 steps of one ulp each, the size of the
// rounding of k R), else per wavenumber.  The order of the sums does not depend on the points and
// wavenumbers of a call: the quadrature points are cut into `leaves` (a power of two, by the mesh alone),
// each the sum of four warps' quarters through shared memory, and the leaves are added by pairs in one
// binary tree -- the 2^b leaves of a CTA's share here (`stack`: the sums still waiting for their
// partner, one a level), the shares, a power of two of them, from `part` [splits][nk][M] by
// k_field64_sum.  With several shares the foot points' values come from k_foot_values64 (p0 [nk][M]), which
// every share's CTA would otherwise gather anew.
// Bound: the FP64 pipe.  64 wavenumbers, 1000 points, 2048 quadrature points: 51.9 -> 13.8 ms = 60 FP64
// instructions an evaluation at the pipe's measured 0.58 T/s (45 of them the rotations and the
// integrand); wavenumbers without a common spacing 23.4 ms.  Error against 64 bits unchanged.
constexpr int F64K = 16;
constexpr int kLeafLevels = 9;
__device__ __forceinline__ cd field64_value(cd p0, cd sum) {  // P0 + sum / (4 pi)
  const double inv4pi = 1.0 / (4.0 * kPi);
  return {fma(sum.re, inv4pi, p0.re), fma(sum.im, inv4pi, p0.im)};
}
// P0 re, im, P0' re, im of one wavenumber (surface values P) at point m's foot point
__device__ __forceinline__ double4 foot_value64(const int32_t* __restrict__ elems, int64_t N, const cd* __restrict__ P,
                                                const int32_t* __restrict__ foot_elem, const double* __restrict__ foot,
                                                int64_t m) {
  const double fxi = foot[8 * m + 6], feta = foot[8 * m + 7];
  const double L1 = 1.0 - fxi - feta;
  const double Nv[6] = {L1 * (2 * L1 - 1), fxi * (2 * fxi - 1), feta * (2 * feta - 1), 4 * L1 * fxi, 4 * fxi * feta,
                         4 * feta * L1};
  const int32_t* el = elems + 6 * (int64_t)foot_elem[m];
  double4 v = make_double4(0.0, 0.0, 0.0, 0.0);
  for (int a = 0; a < 6; ++a) {
    const cd x = P[el[a]], w = P[N + el[a]];
    v.x += Nv[a] * x.re; v.y += Nv[a] * x.im;
    v.z += Nv[a] * w.re; v.w += Nv[a] * w.im;
  }
  return v;
}
__global__ void k_foot_values64(const int32_t* __restrict__ elems, int64_t N, const cd* __restrict__ surf,
                                const int32_t* __restrict__ foot_elem, const double* __restrict__ foot, int64_t M,
                                double4* __restrict__ p0) {
  const int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (m < M) p0[(int64_t)blockIdx.y * M + m] = foot_value64(elems, N, surf + (int64_t)blockIdx.y * 2 * N, foot_elem, foot, m);
}

__global__ void __launch_bounds__(128, 2) k_field64(const int32_t* __restrict__ elems, int64_t N, int64_t EQ,
                                                    const double* __restrict__ qgeo, const cd* __restrict__ Pq,
                                                    const cd* __restrict__ Pnq, const cd* __restrict__ surf,
                                                    const double* __restrict__ xp, int64_t M,
                                                    const int32_t* __restrict__ foot_elem, const double* __restrict__ foot,
                                                    const double* __restrict__ kv, int nk, int splits, int leaves,
                                                    const double4* __restrict__ p0, cd* __restrict__ part,
                                                    cd* __restrict__ T) {
  __shared__ double4 s0[F64K][32];   // P0 re, im, P0' re, im at each lane's foot point
  __shared__ cd red[4][32];
  extern __shared__ double2 f64_smem[];
  cd* stack = reinterpret_cast<cd*>(f64_smem);  // [levels][F64K][32]
  __shared__ double2 sk[F64K];  // k, 1 / k (0 at k = 0)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int kbase = blockIdx.y * F64K, nkb = min(F64K, nk - kbase);
  const int64_t m0 = (int64_t)blockIdx.x * 32, m = m0 + lane < M ? m0 + lane : M - 1;
  if (threadIdx.x < nkb) {
    const double k = kv[kbase + threadIdx.x];
    sk[threadIdx.x] = make_double2(k, k > 0.0 ? 1.0 / k : 0.0);
  }
  for (int e = threadIdx.x; e < nkb * 32; e += 128) {
    const int j = e >> 5, t = e & 31;
    const int64_t mm = m0 + t < M ? m0 + t : M - 1;
    const double4 v = p0 ? p0[(int64_t)(kbase + j) * M + mm] : foot_value64(elems, N, surf + (int64_t)(kbase + j) * 2 * N, foot_elem, foot, mm);
    s0[j][t] = v;
  }
  __syncthreads();
  double p[3], x0[3], nu0[3];
  for (int d = 0; d < 3; ++d) {
    p[d] = xp[3 * m + d];
    x0[d] = foot[8 * m + d];
    nu0[d] = foot[8 * m + 3 + d];
  }
  // equally spaced: every wavenumber within an ulp of the last one of the line between the ends
  const double k0 = kv[kbase], kl = kv[kbase + nkb - 1], dk = nkb > 2 ? (kl - k0) / (nkb - 1) : 0.0;
  bool uniform = nkb > 2;
  for (int j = 1; j < nkb; ++j) uniform &= fabs(kv[kbase + j] - fma((double)j, dk, k0)) <= 2.3e-16 * fabs(kl);
  const int own = leaves / splits;
#pragma unroll 1
  for (int leaf = 0; leaf < own; ++leaf) {
  cd sum[F64K];
#pragma unroll
  for (int j = 0; j < F64K; ++j) sum[j] = cd{0, 0};
  const int64_t quarter = ((int64_t)blockIdx.z * own + leaf) * 4 + warp;
  const int64_t qlo = quarter * EQ / (4 * leaves), qhi = (quarter + 1) * EQ / (4 * leaves);
#pragma unroll 1
  for (int64_t q = qlo; q < qhi; ++q) {
    const double qx = qgeo[GX * EQ + q], qy = qgeo[GY * EQ + q], qz = qgeo[GZ * EQ + q];
    const double nx = qgeo[GNX * EQ + q], ny = qgeo[GNY * EQ + q], nz = qgeo[GNZ * EQ + q], w = qgeo[GWJ * EQ + q];
    double rx = qx - p[0], ry = qy - p[1], rz = qz - p[2];
    double Rp, iRp, R0, iR0;
    dist64(rx * rx + ry * ry + rz * rz, Rp, iRp);
    const double rnp = (rx * nx + ry * ny + rz * nz) * iRp * iRp;
    rx = qx - x0[0]; ry = qy - x0[1]; rz = qz - x0[2];
    dist64(rx * rx + ry * ry + rz * rz, R0, iR0);
    const double rn0 = (rx * nx + ry * ny + rz * nz) * iR0 * iR0;
    const double nr = nu0[0] * rx + nu0[1] * ry + nu0[2] * rz, nn = nu0[0] * nx + nu0[1] * ny + nu0[2] * nz;
    const double ap = w * iRp, a0 = w * iR0;
    double cp, sp, c0, s0v, cg, sg, dcp, dsp, dc0, ds0, dcg, dsg;
    if (uniform) {
      cis64(k0 * Rp, sp, cp);
      cis64(k0 * R0, s0v, c0);
      cis64(k0 * nr, sg, cg);
      cis64(dk * Rp, dsp, dcp);
      cis64(dk * R0, ds0, dc0);
      cis64(dk * nr, dsg, dcg);
      cp *= ap; sp *= ap;  // G = w e^{ikR} / R rides through the rotations
      c0 *= a0; s0v *= a0;
    }
#pragma unroll
    for (int j = 0; j < F64K; ++j) {
      if (j >= nkb) break;
      const double2 kj = sk[j];
      const double k = kj.x;
      if (!uniform) {
        cis64(k * Rp, sp, cp);
        cis64(k * R0, s0v, c0);
        cis64(k * nr, sg, cg);
        cp *= ap; sp *= ap;
        c0 *= a0; s0v *= a0;
      } else if (j > 0) {
        double u = cp * dcp - sp * dsp;
        sp = sp * dcp + cp * dsp;
        cp = u;
        u = c0 * dc0 - s0v * ds0;
        s0v = s0v * dc0 + c0 * ds0;
        c0 = u;
        u = cg * dcg - sg * dsg;
        sg = sg * dcg + cg * dsg;
        cg = u;
      }
      const double kRp = k * Rp, kR0 = k * R0;
      const double gdr = cp - c0, gdi = sp - s0v;  // w (Gp - G0), and w (dGp - dG0):
      const double ddr = (s0v * kR0 + c0) * rn0 - (sp * kRp + cp) * rnp;
      const double ddi = (cp * kRp - sp) * rnp - (c0 * kR0 - s0v) * rn0;
      // g, f about x0 (f -> nu0.r at k = 0) and their normal derivatives
      const double g = cg, f = k > 0.0 ? sg * kj.y : nr, dg = -k * sg * nn, df = cg * nn;
      const double4 z = s0[j][lane];
      const cd P = Pq[(int64_t)(kbase + j) * EQ + q], D = Pnq[(int64_t)(kbase + j) * EQ + q];
      const double Ptr = P.re - z.x * g - z.z * f, Pti = P.im - z.y * g - z.w * f;
      const double dPr = D.re - z.x * dg - z.z * df, dPi = D.im - z.y * dg - z.w * df;
      // sum += Pt (dGp - dG0) - (Gp - G0) dPt, product by product: a fused addition each
      sum[j].re = fma(Ptr, ddr, fma(-Pti, ddi, fma(-gdr, dPr, fma(gdi, dPi, sum[j].re))));
      sum[j].im = fma(Ptr, ddi, fma(Pti, ddr, fma(-gdr, dPi, fma(-gdi, dPr, sum[j].im))));
    }
  }
#pragma unroll
  for (int j = 0; j < F64K; ++j) {
    if (j >= nkb) break;
    __syncthreads();
    red[warp][lane] = sum[j];
    __syncthreads();
    if (warp == (j & 3)) {
      cd t = {0, 0};
      for (int w = 0; w < 4; ++w) t = cadd(t, red[w][lane]);
      int l = 0;
      for (; (leaf >> l) & 1; ++l) t = cadd(stack[(l * F64K + j) * 32 + lane], t);
      stack[(l * F64K + j) * 32 + lane] = t;  // (the last leaf's: the share's sum)
      if (leaf + 1 == own && m0 + lane < M) {
        const int64_t at = (int64_t)(kbase + j) * M + m0 + lane, n = (int64_t)nk * M;
        if (splits == 1) T[at] = field64_value(cd{s0[j][lane].x, s0[j][lane].y}, t);
        else part[blockIdx.z * n + at] = t;
      }
    }
  }
  }
}

// The shares' sums added by pairs, and the value; n = nk M
__global__ void k_field64_sum(const cd* __restrict__ part, const double4* __restrict__ p0, int splits, int64_t n,
                              cd* __restrict__ T) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  cd stack[kLeafLevels + 1];
  for (int z = 0; z < splits; ++z) {
    cd v = part[z * n + t];
    bool put = false;
#pragma unroll
    for (int l = 0; l <= kLeafLevels; ++l)  // (unrolled: the stack stays in registers)
      if (!put) {
        if ((z >> l) & 1) {
          v = cadd(stack[l], v);
        } else {
          stack[l] = v;
          put = true;
        }
      }
    if (z + 1 == splits) T[t] = field64_value(cd{p0[t].x, p0[t].y}, v);
  }
}

// Leaves of the sums: as many as leave each 32 quadrature points, 2^kLeafLevels at most.
static int field64_leaves(bie_ctx* c) {
  const int64_t EQ = c->E * c->rule.Q;
  int z = 1;
  while (z < 1 << kLeafLevels && 2 * z * 32 <= EQ) z *= 2;
  return z;
}
// Shares of the quadrature points: eight to sixty-four CTAs to an SM (two are resident), of the powers of two
// in between the one whose last, partial wave leaves the least of the SMs idle (1000 points, 64
// wavenumbers: 14 waves for 13.5 measured 15.8 ms, 27 for 26.9 15.4).
static int field64_splits(int nk, int64_t M, int nsm, int leaves) {
  const int64_t ctas = (M + 31) / 32 * ((nk + F64K - 1) / F64K), wave = 2 * nsm;
  int best = 0;
  double used = 0.0;
  for (int z = 1; z <= leaves && (best == 0 || z * ctas <= 64 * nsm); z *= 2) {
    if (z * ctas < 8 * nsm && z < leaves) continue;
    const double u = (double)(z * ctas) / (double)((z * ctas + wave - 1) / wave * wave);
    if (best == 0 || u > 1.01 * used) {
      best = z;
      used = u;
    }
  }
  return best;
}
// Scratch of field64 in bytes.
size_t field64_scratch(bie_ctx* c, int nk, int64_t M, int nsm) {
  const int z = field64_splits(nk, M, nsm, field64_leaves(c));
  return 2 * (size_t)nk * c->E * c->rule.Q * sizeof(cd) + (z > 1 ? (size_t)(z + 2) * nk * M * sizeof(cd) : 0);
}

// Evaluates nk wavenumbers: surf [nk][2][N] -> T [nk][M].  scratch: field64_scratch bytes.
int field64(bie_ctx* c, const double* kv, int nk, const cd* surf, const double* xp, int64_t M,
            const int32_t* foot_elem, const double* foot, cd* T, void* scratch, int nsm) {
  const int64_t EQ = c->E * c->rule.Q;
  cd* Pq = (cd*)scratch;
  cd* Pnq = Pq + (int64_t)nk * EQ;
  cd* part = Pnq + (int64_t)nk * EQ;
  dim3 gi((unsigned)((EQ + 255) / 256), nk);
  BIE_LAUNCH(k_interp_q64<<<gi, 256, 0, c->stream>>>(c->elems, c->N, c->E, c->rule.Q, c->qshape, surf, Pq, Pnq));
  if (M > 0) {
    const int leaves = field64_leaves(c), splits = field64_splits(nk, M, nsm, leaves);
    double4* p0 = nullptr;
    if (splits > 1) {  // (the foot points' values, then the shares' sums)
      p0 = reinterpret_cast<double4*>(part);
      part += 2 * (int64_t)nk * M;
      BIE_LAUNCH(k_foot_values64<<<dim3((unsigned)((M + 127) / 128), nk), 128, 0, c->stream>>>(c->elems, c->N, surf, foot_elem,
                                                                                              foot, M, p0));
    }
    int levels = 1;
    while ((leaves / splits) >> levels) ++levels;  // of a share's leaves
    dim3 gf((unsigned)((M + 31) / 32), (unsigned)((nk + F64K - 1) / F64K), (unsigned)splits);
    BIE_TRY(set_smem_max(k_field64));
    BIE_LAUNCH(k_field64<<<gf, 128, (size_t)levels * F64K * 32 * sizeof(cd), c->stream>>>(
        c->elems, c->N, EQ, c->qgeo, Pq, Pnq, surf, xp, M, foot_elem, foot, kv, nk, splits, leaves, p0, part, T));
    if (splits > 1)
      BIE_LAUNCH(k_field64_sum<<<(unsigned)((nk * M + 255) / 256), 256, 0, c->stream>>>(part, p0, splits, nk * M, T));
  }
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}


// ------------------------------------------------------------------------------------------
// Mixed precision: the same formula in FP32 with compensated accumulation.  ACC = true forms the
// three phases (k|x - x_p|, k|x - x0|, k nu0.(x - x0)) in float-float and reduces them modulo
// 2 pi before sincosf; ACC = false uses FP32 distances and the SFU sine/cosine after an FP32
// reduction.  Point table: asm32.cu's layout (x_hi[3], x_lo[3], nu[3], wJ).
// ------------------------------------------------------------------------------------------
struct TwoPi3f {
  float c1, c2, c3, inv;
};

__device__ __forceinline__ void cis_ff(ff a, const TwoPi3f& tp, float& c, float& s) {
  const float n = round_small(__fmul_rn(a.hi, tp.inv));
  const float h = __fmaf_rn(-n, tp.c1, a.hi);
  float t = __fmaf_rn(-n, tp.c2, a.lo);
  t = __fmaf_rn(-n, tp.c3, t);
  const ff u = ff_two_sum(h, t);
  float sh, ch;
  sincosf(u.hi, &sh, &ch);
  c = __fmaf_rn(-u.lo, sh, ch);
  s = __fmaf_rn(u.lo, ch, sh);
}

__device__ __forceinline__ void cis_fast(float t, const TwoPi3f& tp, float& c, float& s) {
  const float n = round_small(__fmul_rn(t, tp.inv));
  float u = __fmaf_rn(-n, tp.c1, t);
  u = __fmaf_rn(-n, tp.c2, u);
  __sincosf(u, &s, &c);
}

__global__ void k_interp_q32(const int32_t* __restrict__ elems, int64_t N, int64_t E, int Q,
                             const double* __restrict__ qshape, const cd* __restrict__ surf, cf* __restrict__ Pq,
                             cf* __restrict__ Pnq) {
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int kk = blockIdx.y;
  if (p >= E * Q) return;
  int64_t e = p / Q;
  int q = (int)(p % Q);
  const cd* P = surf + (int64_t)kk * 2 * N;
  const cd* Pn = P + N;
  cd a = {0, 0}, b = {0, 0};
  for (int t = 0; t < 6; ++t) {
    int32_t j = elems[6 * e + t];
    double sh = qshape[q * 6 + t];
    a.re += sh * P[j].re; a.im += sh * P[j].im;
    b.re += sh * Pn[j].re; b.im += sh * Pn[j].im;
  }
  Pq[(int64_t)kk * E * Q + p] = {(float)a.re, (float)a.im};
  Pnq[(int64_t)kk * E * Q + p] = {(float)b.re, (float)b.im};
}

template <bool ACC>
__global__ void __launch_bounds__(FT) k_field32(const int32_t* __restrict__ elems, int64_t N, int64_t EQ,
                                                const float* __restrict__ qtab, const cf* __restrict__ Pq,
                                                const cf* __restrict__ Pnq, const cd* __restrict__ surf,
                                                const double* __restrict__ xp, int64_t M,
                                                const int32_t* __restrict__ foot_elem, const double* __restrict__ foot,
                                                const double* __restrict__ kv, cd* __restrict__ T, TwoPi3f tp) {
  __shared__ float st[17][FT];
  const int kk = blockIdx.y;
  const ff k = ff_from_double(kv[kk]);
  const float kinv = kinv32(kv[kk]);
  const int64_t m = (int64_t)blockIdx.x * FT + threadIdx.x;
  const bool active = m < M;
  ff p[3] = {{0, 0}, {0, 0}, {0, 0}}, x0[3] = {{0, 0}, {0, 0}, {0, 0}}, nu0[3] = {{0, 0}, {0, 0}, {1, 0}};
  float P0r = 0, P0i = 0, Q0r = 0, Q0i = 0;
  if (active) {
    for (int d = 0; d < 3; ++d) {
      p[d] = ff_from_double(xp[3 * m + d]);
      x0[d] = ff_from_double(foot[8 * m + d]);
      nu0[d] = ff_from_double(foot[8 * m + 3 + d]);
    }
    const double fxi = foot[8 * m + 6], feta = foot[8 * m + 7];
    const double L1 = 1.0 - fxi - feta;
    const double Nv[6] = {L1 * (2 * L1 - 1), fxi * (2 * fxi - 1), feta * (2 * feta - 1), 4 * L1 * fxi, 4 * fxi * feta,
                          4 * feta * L1};
    const int32_t* el = elems + 6 * (int64_t)foot_elem[m];
    const cd* P = surf + (int64_t)kk * 2 * N;
    double a0 = 0, a1 = 0, b0 = 0, b1 = 0;
    for (int a = 0; a < 6; ++a) {
      cd v = P[el[a]], w = P[N + el[a]];
      a0 += Nv[a] * v.re; a1 += Nv[a] * v.im;
      b0 += Nv[a] * w.re; b1 += Nv[a] * w.im;
    }
    P0r = (float)a0; P0i = (float)a1; Q0r = (float)b0; Q0i = (float)b1;
  }
  const cf* Pqk = Pq + (int64_t)kk * EQ;
  const cf* Pnqk = Pnq + (int64_t)kk * EQ;
  ksum sr, si;
  for (int64_t t0 = 0; t0 < EQ; t0 += FT) {
    const int64_t t = t0 + threadIdx.x;
    if (t < EQ) {
#pragma unroll
      for (int u = 0; u < 13; ++u) st[u][threadIdx.x] = qtab[u * EQ + t];
      const cf a = Pqk[t], b = Pnqk[t];
      st[13][threadIdx.x] = a.re; st[14][threadIdx.x] = a.im;
      st[15][threadIdx.x] = b.re; st[16][threadIdx.x] = b.im;
    }
    __syncthreads();
    const int cnt = (EQ - t0) < FT ? (int)(EQ - t0) : FT;
    if (active) {
      for (int u = 0; u < cnt; ++u) {
        const ff qx = {st[0][u], st[3][u]}, qy = {st[1][u], st[4][u]}, qz = {st[2][u], st[5][u]};
        const float nx = st[6][u], ny = st[7][u], nz = st[8][u], wj = st[9][u];
        const ff rpx = ff_sub(qx, p[0]), rpy = ff_sub(qy, p[1]), rpz = ff_sub(qz, p[2]);
        const ff r0x = ff_sub(qx, x0[0]), r0y = ff_sub(qy, x0[1]), r0z = ff_sub(qz, x0[2]);
        float cp, sp, c0, s0, cg, sg, Rp, R0, rnp, rn0, nrh;
        if (ACC) {
          const ff nux = {nx, st[10][u]}, nuy = {ny, st[11][u]}, nuz = {nz, st[12][u]};
          rnp = ff_add(ff_add(ff_mul(rpx, nux), ff_mul(rpy, nuy)), ff_mul(rpz, nuz)).hi;
          rn0 = ff_add(ff_add(ff_mul(r0x, nux), ff_mul(r0y, nuy)), ff_mul(r0z, nuz)).hi;
          const ff Rpf = ff_sqrt(ff_add(ff_add(ff_sqr(rpx), ff_sqr(rpy)), ff_sqr(rpz)));
          const ff R0f = ff_sqrt(ff_add(ff_add(ff_sqr(r0x), ff_sqr(r0y)), ff_sqr(r0z)));
          const ff nr = ff_add(ff_add(ff_mul(nu0[0], r0x), ff_mul(nu0[1], r0y)), ff_mul(nu0[2], r0z));
          cis_ff(ff_mul(k, Rpf), tp, cp, sp);
          cis_ff(ff_mul(k, R0f), tp, c0, s0);
          cis_ff(ff_mul(k, nr), tp, cg, sg);
          nrh = nr.hi;
          Rp = Rpf.hi;
          R0 = R0f.hi;
        } else {
          Rp = sqrtf(rpx.hi * rpx.hi + rpy.hi * rpy.hi + rpz.hi * rpz.hi);
          R0 = sqrtf(r0x.hi * r0x.hi + r0y.hi * r0y.hi + r0z.hi * r0z.hi);
          const float nr = nu0[0].hi * r0x.hi + nu0[1].hi * r0y.hi + nu0[2].hi * r0z.hi;
          nrh = nr;
          cis_fast(k.hi * Rp, tp, cp, sp);
          cis_fast(k.hi * R0, tp, c0, s0);
          cis_fast(k.hi * nr, tp, cg, sg);
          rnp = rpx.hi * nx + rpy.hi * ny + rpz.hi * nz;
          rn0 = r0x.hi * nx + r0y.hi * ny + r0z.hi * nz;
        }
        const float iRp = 1.0f / Rp, iR0 = 1.0f / R0;
        const float kRp = k.hi * Rp, kR0 = k.hi * R0;
        rnp *= iRp * iRp * iRp;
        rn0 *= iR0 * iR0 * iR0;
        const float Gpr = cp * iRp, Gpi = sp * iRp, G0r = c0 * iR0, G0i = s0 * iR0;
        const float dGpr = (-cp - sp * kRp) * rnp, dGpi = (cp * kRp - sp) * rnp;
        const float dG0r = (-c0 - s0 * kR0) * rn0, dG0i = (c0 * kR0 - s0) * rn0;
        const float nn = nu0[0].hi * nx + nu0[1].hi * ny + nu0[2].hi * nz;
        const float g = cg, f = kinv != 0.f ? sg * kinv : nrh, dg = -k.hi * sg * nn, df = cg * nn;
        const float Ptr = st[13][u] - P0r * g - Q0r * f, Pti = st[14][u] - P0i * g - Q0i * f;
        const float dPr = st[15][u] - P0r * dg - Q0r * df, dPi = st[16][u] - P0i * dg - Q0i * df;
        const float ddr = dGpr - dG0r, ddi = dGpi - dG0i, gdr = Gpr - G0r, gdi = Gpi - G0i;
        const float tr = (Ptr * ddr - Pti * ddi) - (gdr * dPr - gdi * dPi);
        const float ti = (Ptr * ddi + Pti * ddr) - (gdr * dPi + gdi * dPr);
        sr.add(wj * tr);
        si.add(wj * ti);
      }
    }
    __syncthreads();
  }
  if (active) {
    const double inv4pi = 1.0 / (4.0 * kPi);
    T[(int64_t)kk * M + m] = {(double)P0r + sr.value() * inv4pi, (double)P0i + si.value() * inv4pi};
  }
}

// k-batched variant of the float-float kernel: each (point, quadrature point) pair's geometry --
// the float-float distances to x_p and x0, nu0.(x - x0), r.nu -- is formed once and reused for FKB
// wavenumbers; per wavenumber only the three phases (float-float product reduced by pi/2 in one
// step, cis_ffprod) and the FP32 integrand remain.
constexpr int FKB = 8;

__global__ void __launch_bounds__(FT) k_field32b(const int32_t* __restrict__ elems, int64_t N, int64_t EQ,
                                                 const float* __restrict__ qtab, const cf* __restrict__ Pq,
                                                 const cf* __restrict__ Pnq, const cd* __restrict__ surf,
                                                 const double* __restrict__ xp, int64_t M,
                                                 const int32_t* __restrict__ foot_elem,
                                                 const double* __restrict__ foot, const double* __restrict__ kv,
                                                 int nk, cd* __restrict__ T, TwoPi3f tp, int uniform,
                                                 ff dk) {
  __shared__ float sg[13][FT];        // quadrature geometry tile
  __shared__ float sq[FKB][4][FT];    // Pq, Pnq (re, im) of the tile for each wavenumber
  __shared__ float s0[FKB][4][FT];    // P0, P0' (re, im) of each thread's point for each wavenumber
  __shared__ float sk[FKB][3];        // k (hi, lo), 1/k
  const int kbase = blockIdx.y * FKB;
  const int nkb = min(FKB, nk - kbase);
  const int tid = threadIdx.x;
  const int64_t m = (int64_t)blockIdx.x * FT + tid;
  const bool active = m < M;
  if (tid < nkb) {
    const ff k = ff_from_double(kv[kbase + tid]);
    sk[tid][0] = k.hi;
    sk[tid][1] = k.lo;
    sk[tid][2] = kinv32(kv[kbase + tid]);
  }
  ff p[3] = {{0, 0}, {0, 0}, {0, 0}}, x0[3] = {{0, 0}, {0, 0}, {0, 0}}, nu0[3] = {{0, 0}, {0, 0}, {1, 0}};
  if (active) {
    for (int d = 0; d < 3; ++d) {
      p[d] = ff_from_double(xp[3 * m + d]);
      x0[d] = ff_from_double(foot[8 * m + d]);
      nu0[d] = ff_from_double(foot[8 * m + 3 + d]);
    }
    const double fxi = foot[8 * m + 6], feta = foot[8 * m + 7];
    const double L1 = 1.0 - fxi - feta;
    const double Nv[6] = {L1 * (2 * L1 - 1), fxi * (2 * fxi - 1), feta * (2 * feta - 1), 4 * L1 * fxi, 4 * fxi * feta,
                          4 * feta * L1};
    const int32_t* el = elems + 6 * (int64_t)foot_elem[m];
    for (int j = 0; j < nkb; ++j) {
      const cd* P = surf + (int64_t)(kbase + j) * 2 * N;
      double a0 = 0, a1 = 0, b0 = 0, b1 = 0;
      for (int a = 0; a < 6; ++a) {
        const cd v = P[el[a]], w = P[N + el[a]];
        a0 += Nv[a] * v.re; a1 += Nv[a] * v.im;
        b0 += Nv[a] * w.re; b1 += Nv[a] * w.im;
      }
      s0[j][0][tid] = (float)a0; s0[j][1][tid] = (float)a1;
      s0[j][2][tid] = (float)b0; s0[j][3][tid] = (float)b1;
    }
  }
  ksum accr[FKB], acci[FKB];
  for (int64_t t0 = 0; t0 < EQ; t0 += FT) {
    const int64_t t = t0 + tid;
    __syncthreads();
    if (t < EQ) {
#pragma unroll
      for (int u = 0; u < 13; ++u) sg[u][tid] = qtab[u * EQ + t];
      for (int j = 0; j < nkb; ++j) {
        const cf a = Pq[(int64_t)(kbase + j) * EQ + t], b = Pnq[(int64_t)(kbase + j) * EQ + t];
        sq[j][0][tid] = a.re; sq[j][1][tid] = a.im;
        sq[j][2][tid] = b.re; sq[j][3][tid] = b.im;
      }
    }
    __syncthreads();
    const int cnt = (EQ - t0) < FT ? (int)(EQ - t0) : FT;
    if (!active) continue;
    for (int u = 0; u < cnt; ++u) {
      const ff qx = {sg[0][u], sg[3][u]}, qy = {sg[1][u], sg[4][u]}, qz = {sg[2][u], sg[5][u]};
      const float nx = sg[6][u], ny = sg[7][u], nz = sg[8][u], wj = sg[9][u];
      const ff nux = {nx, sg[10][u]}, nuy = {ny, sg[11][u]}, nuz = {nz, sg[12][u]};
      const ff rpx = ff_sub(qx, p[0]), rpy = ff_sub(qy, p[1]), rpz = ff_sub(qz, p[2]);
      const ff r0x = ff_sub(qx, x0[0]), r0y = ff_sub(qy, x0[1]), r0z = ff_sub(qz, x0[2]);
      const ff Rp = ff_sqrt(ff_add(ff_add(ff_sqr(rpx), ff_sqr(rpy)), ff_sqr(rpz)));
      const ff R0 = ff_sqrt(ff_add(ff_add(ff_sqr(r0x), ff_sqr(r0y)), ff_sqr(r0z)));
      const ff nr = ff_add(ff_add(ff_mul(nu0[0], r0x), ff_mul(nu0[1], r0y)), ff_mul(nu0[2], r0z));
      const float iRp = 1.0f / Rp.hi, iR0 = 1.0f / R0.hi;
      // x_p is off the surface (no cancellation in r.nu); x0 is on it, so r0.nu is second-order
      // small for nearby quadrature points and is formed in float-float
      const float rnp = (rpx.hi * nx + rpy.hi * ny + rpz.hi * nz) * iRp * iRp * iRp;
      const float rn0 = ff_add(ff_add(ff_mul(r0x, nux), ff_mul(r0y, nuy)), ff_mul(r0z, nuz)).hi * iR0 * iR0 * iR0;
      const float nn = nu0[0].hi * nx + nu0[1].hi * ny + nu0[2].hi * nz;
      // phase factors: on a uniform group k_j = k_0 + j dk, e^{i k_j R} = e^{i k_0 R} (e^{i dk R})^j with
      // both factors accurate and the powers taken by FP32 rotation (drift <= nkb ulps)
      float cp = 0.f, spp = 0.f, c0 = 0.f, s0v = 0.f, cg = 0.f, sgv = 0.f;
      float dcp = 1.f, dsp = 0.f, dc0 = 1.f, ds0 = 0.f, dcg = 1.f, dsg = 0.f;
      if (uniform) {
        const ff k0 = {sk[0][0], sk[0][1]};
        cis_ffprod(k0, Rp, cp, spp);
        cis_ffprod(k0, R0, c0, s0v);
        cis_ffprod(k0, nr, cg, sgv);
        cis_ffprod(dk, Rp, dcp, dsp);
        cis_ffprod(dk, R0, dc0, ds0);
        cis_ffprod(dk, nr, dcg, dsg);
      }
#pragma unroll
      for (int j = 0; j < FKB; ++j) {
        if (j < nkb) {
          const ff k = {sk[j][0], sk[j][1]};
          const float kinv = sk[j][2];
          if (!uniform) {
            cis_ffprod(k, Rp, cp, spp);
            cis_ffprod(k, R0, c0, s0v);
            cis_ffprod(k, nr, cg, sgv);
          } else if (j > 0) {
            float t = cp * dcp - spp * dsp;
            spp = spp * dcp + cp * dsp;
            cp = t;
            t = c0 * dc0 - s0v * ds0;
            s0v = s0v * dc0 + c0 * ds0;
            c0 = t;
            t = cg * dcg - sgv * dsg;
            sgv = sgv * dcg + cg * dsg;
            cg = t;
          }
          const float kRp = k.hi * Rp.hi, kR0 = k.hi * R0.hi;
          const float Gpr = cp * iRp, Gpi = spp * iRp, G0r = c0 * iR0, G0i = s0v * iR0;
          const float dGpr = (-cp - spp * kRp) * rnp, dGpi = (cp * kRp - spp) * rnp;
          const float dG0r = (-c0 - s0v * kR0) * rn0, dG0i = (c0 * kR0 - s0v) * rn0;
          const float g = cg, f = kinv != 0.f ? sgv * kinv : nr.hi, dg = -k.hi * sgv * nn, df = cg * nn;
          const float P0r = s0[j][0][tid], P0i = s0[j][1][tid], Q0r = s0[j][2][tid], Q0i = s0[j][3][tid];
          const float Ptr = sq[j][0][u] - P0r * g - Q0r * f, Pti = sq[j][1][u] - P0i * g - Q0i * f;
          const float dPr = sq[j][2][u] - P0r * dg - Q0r * df, dPi = sq[j][3][u] - P0i * dg - Q0i * df;
          const float ddr = dGpr - dG0r, ddi = dGpi - dG0i, gdr = Gpr - G0r, gdi = Gpi - G0i;
          const float tr = (Ptr * ddr - Pti * ddi) - (gdr * dPr - gdi * dPi);
          const float ti = (Ptr * ddi + Pti * ddr) - (gdr * dPi + gdi * dPr);
          accr[j].add(wj * tr);
          acci[j].add(wj * ti);
        }
      }
    }
  }
  if (active) {
    const double inv4pi = 1.0 / (4.0 * kPi);
    for (int j = 0; j < nkb; ++j)
      T[(int64_t)(kbase + j) * M + m] = {(double)s0[j][0][tid] + accr[j].value() * inv4pi,
                                         (double)s0[j][1][tid] + acci[j].value() * inv4pi};
  }
}

// Variant of k_field32b with the wavenumber-group size KB, the points per CTA TP and the minimum
// resident CTAs MINB as template parameters: terms are summed in FP32 over runs of 32 quadrature
// points and each run is added to a compensated sum kept in shared memory, so only 2 KB partial
// sums stay in registers; every phase (group start k_0 R and step dk R) comes from the
// float-float product reduced by pi/2 in one step (cis_ffprod).  far_r2: beyond it r0.nu_q is
// formed in FP32.
// ZF: the group may hold k = 0 (f takes its limit nu0.r there); false for groups of k > 0 only,
// which keeps the zero-frequency select out of the inner loop.
template <int KB, int TP, int MINB, int UT, bool ZF>
__global__ void __launch_bounds__(TP, MINB) k_field32c(const int32_t* __restrict__ elems, int64_t N, int64_t EQ,
                                                       const float* __restrict__ qtab, const cf* __restrict__ Pq,
                                                       const cf* __restrict__ Pnq, const cd* __restrict__ surf,
                                                       const double* __restrict__ xp, int64_t M,
                                                       const int32_t* __restrict__ foot_elem,
                                                       const double* __restrict__ foot, const double* __restrict__ kv,
                                                       int nk, cd* __restrict__ T, int uniform, ff dk,
                                                       float far_r2) {
  __shared__ float4 sg[UT][4];  // a tile of UT quadrature points: 13 table values (P32 order), padded
  __shared__ float4 sq[KB][UT];  // surface values at the tile's points: P re, im, dP re, im
  __shared__ float4 s0[KB][TP];  // surface values at the foot points, same order
  __shared__ float sacc[KB][4][TP];  // compensated sums: re (s, c), im (s, c)
  __shared__ float2 sk[KB];  // k (FP32 head), 1 / k (0 at k = 0)
  __shared__ float sklo[KB];  // k - head
  const int kbase = blockIdx.y * KB;
  const int nkb = min(KB, nk - kbase);
  const int tid = threadIdx.x;
  const int64_t m = (int64_t)blockIdx.x * TP + tid;
  const bool active = m < M;
  if (tid < nkb) {
    const ff k = ff_from_double(kv[kbase + tid]);
    sk[tid] = make_float2(k.hi, kinv32(kv[kbase + tid]));
    sklo[tid] = k.lo;
  }
#pragma unroll
  for (int j = 0; j < KB; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q) sacc[j][q][tid] = 0.f;
  ff p[3] = {{0, 0}, {0, 0}, {0, 0}}, x0[3] = {{0, 0}, {0, 0}, {0, 0}}, nu0[3] = {{0, 0}, {0, 0}, {1, 0}};
  if (active) {
    for (int d = 0; d < 3; ++d) {
      p[d] = ff_from_double(xp[3 * m + d]);
      x0[d] = ff_from_double(foot[8 * m + d]);
      nu0[d] = ff_from_double(foot[8 * m + 3 + d]);
    }
    const double fxi = foot[8 * m + 6], feta = foot[8 * m + 7];
    const double L1 = 1.0 - fxi - feta;
    const double Nv[6] = {L1 * (2 * L1 - 1), fxi * (2 * fxi - 1), feta * (2 * feta - 1), 4 * L1 * fxi, 4 * fxi * feta,
                          4 * feta * L1};
    const int32_t* el = elems + 6 * (int64_t)foot_elem[m];
    for (int j = 0; j < nkb; ++j) {
      const cd* P = surf + (int64_t)(kbase + j) * 2 * N;
      double a0 = 0, a1 = 0, b0 = 0, b1 = 0;
      for (int a = 0; a < 6; ++a) {
        const cd v = P[el[a]], w = P[N + el[a]];
        a0 += Nv[a] * v.re; a1 += Nv[a] * v.im;
        b0 += Nv[a] * w.re; b1 += Nv[a] * w.im;
      }
      s0[j][tid] = make_float4((float)a0, (float)a1, (float)b0, (float)b1);
    }
  }
  float pr[KB], pim[KB];
#pragma unroll
  for (int j = 0; j < KB; ++j) pr[j] = pim[j] = 0.f;
  for (int64_t t0 = 0; t0 < EQ; t0 += UT) {
    const int cnt = (EQ - t0) < UT ? (int)(EQ - t0) : UT;
    __syncthreads();
    for (int e = tid; e < 13 * UT; e += TP) {  // consecutive threads, consecutive points
      const int f = e / UT, u = e - f * UT;
      if (u < cnt) reinterpret_cast<float*>(sg[u])[f] = qtab[f * EQ + t0 + u];
    }
    for (int e = tid; e < KB * UT; e += TP) {
      const int j = e / UT, u = e - j * UT;
      if (j < nkb && u < cnt) {
        const int64_t t = t0 + u;
        const cf a = Pq[(int64_t)(kbase + j) * EQ + t], b = Pnq[(int64_t)(kbase + j) * EQ + t];
        sq[j][u] = make_float4(a.re, a.im, b.re, b.im);
      }
    }
    __syncthreads();
    if (!active) continue;
    for (int u = 0; u < cnt; ++u) {
      const float4 g0 = sg[u][0], g1 = sg[u][1], g2 = sg[u][2], g3 = sg[u][3];
      const ff qx = {g0.x, g0.w}, qy = {g0.y, g1.x}, qz = {g0.z, g1.y};
      const float nx = g1.z, ny = g1.w, nz = g2.x, wj = g2.y;
      const ff nux = {nx, g2.z}, nuy = {ny, g2.w}, nuz = {nz, g3.x};
      // float-float geometry with lazy tails (distances, 1/R, nu0.r)
      const ff rpx = ff_diff_lazy(qx, p[0]), rpy = ff_diff_lazy(qy, p[1]), rpz = ff_diff_lazy(qz, p[2]);
      const ff r0x = ff_diff_lazy(qx, x0[0]), r0y = ff_diff_lazy(qy, x0[1]), r0z = ff_diff_lazy(qz, x0[2]);
      const ff R0sq = ff_norm2_lazy(r0x, r0y, r0z);
      float iRp, iR0;
      const ff Rp = ff_sqrt_lazy(ff_norm2_lazy(rpx, rpy, rpz), iRp);
      const ff R0 = ff_sqrt_lazy(R0sq, iR0);
      const ff nr = ff_dot3_lazy(nu0, r0x, r0y, r0z);
      // the recurrences below carry the weighted kernels Gp = w e^{ik Rp} / Rp and G0 (same for
      // the foot point); then dG/dnu = G (ik R - 1) r.nu / R^2
      const float ap = wj * iRp, a0 = wj * iR0;
      const float rnp = ((rpx.hi + rpx.lo) * nx + (rpy.hi + rpy.lo) * ny + (rpz.hi + rpz.lo) * nz) * iRp * iRp;
      // r0.nu is second-order small near the foot point (error-free products there); beyond
      // far_r2 its FP32 rounding eps R0 perturbs dG0 by eps / R0^2, the term's own rounding
      float rn0;
      if (R0sq.hi > far_r2) {
        rn0 = (r0x.hi + r0x.lo) * nx + (r0y.hi + r0y.lo) * ny + (r0z.hi + r0z.lo) * nz;
      } else {
        const ff nuq[3] = {nux, nuy, nuz};
        const ff d = ff_dot3_lazy(nuq, r0x, r0y, r0z);
        rn0 = d.hi + d.lo;
      }
      rn0 *= iR0 * iR0;
      const float nn = nu0[0].hi * nx + nu0[1].hi * ny + nu0[2].hi * nz;
      float cp = 0.f, spp = 0.f, c0 = 0.f, s0v = 0.f, cg = 0.f, sgv = 0.f;
      float dcp = 1.f, dsp = 0.f, dc0 = 1.f, ds0 = 0.f, dcg = 1.f, dsg = 0.f;
      if (uniform) {
        const ff k0 = {sk[0].x, sklo[0]};
        cis_ffprod(k0, Rp, cp, spp);
        cis_ffprod(k0, R0, c0, s0v);
        cis_ffprod(k0, nr, cg, sgv);
        // step phases dk R
        cis_ffprod(dk, Rp, dcp, dsp);
        cis_ffprod(dk, R0, dc0, ds0);
        cis_ffprod(dk, nr, dcg, dsg);
        cp *= ap; spp *= ap;
        c0 *= a0; s0v *= a0;
      }
#pragma unroll
      for (int j = 0; j < KB; ++j) {
        if (j < nkb) {
          const float2 kj = sk[j];
          const float khi = kj.x, kinv = kj.y;
          if (!uniform) {
            const ff k = {khi, sklo[j]};
            cis_ffprod(k, Rp, cp, spp);
            cis_ffprod(k, R0, c0, s0v);
            cis_ffprod(k, nr, cg, sgv);
            cp *= ap; spp *= ap;
            c0 *= a0; s0v *= a0;
          } else if (j > 0) {
            float t = cp * dcp - spp * dsp;
            spp = spp * dcp + cp * dsp;
            cp = t;
            t = c0 * dc0 - s0v * ds0;
            s0v = s0v * dc0 + c0 * ds0;
            c0 = t;
            t = cg * dcg - sgv * dsg;
            sgv = sgv * dcg + cg * dsg;
            cg = t;
          }
          const float kRp = khi * Rp.hi, kR0 = khi * R0.hi;
          // G weighted by w; dG/dnu = -(Gr + Gi kR) rn + i (Gr kR - Gi) rn, taken as the
          // difference dGp - dG0 directly
          const float gdr = cp - c0, gdi = spp - s0v;
          const float ddr = __fmaf_rn(__fmaf_rn(s0v, kR0, c0), rn0, -(__fmaf_rn(spp, kRp, cp) * rnp));
          const float ddi = __fmaf_rn(__fmaf_rn(cp, kRp, -spp), rnp, -(__fmaf_rn(c0, kR0, -s0v) * rn0));
          // f = sin(k nu0.r)/k, or its limit nu0.r at k = 0 (kinv 0)
          const float g = cg, f = (ZF && kinv == 0.f) ? nr.hi : sgv * kinv, dg = -khi * sgv * nn, df = cg * nn;
          const float4 p0 = s0[j][tid], pq = sq[j][u];
          const float P0r = p0.x, P0i = p0.y, Q0r = p0.z, Q0i = p0.w;
          const float Ptr = pq.x - P0r * g - Q0r * f, Pti = pq.y - P0i * g - Q0i * f;
          const float dPr = pq.z - P0r * dg - Q0r * df, dPi = pq.w - P0i * dg - Q0i * df;
          // run sums of w [P~ (dGp - dG0) - (Gp - G0) dP~]
          float a = __fmaf_rn(Ptr, ddr, pr[j]);
          a = __fmaf_rn(-Pti, ddi, a);
          a = __fmaf_rn(-gdr, dPr, a);
          pr[j] = __fmaf_rn(gdi, dPi, a);
          a = __fmaf_rn(Ptr, ddi, pim[j]);
          a = __fmaf_rn(Pti, ddr, a);
          a = __fmaf_rn(-gdr, dPi, a);
          pim[j] = __fmaf_rn(-gdi, dPr, a);
        }
      }
      if ((u & 31) == 31 || u == cnt - 1) {  // add the run to the compensated sums
#pragma unroll
        for (int j = 0; j < KB; ++j) {
          if (j < nkb) {
            ff a = ff_two_sum(sacc[j][0][tid], pr[j]);
            sacc[j][0][tid] = a.hi;
            sacc[j][1][tid] += a.lo;
            a = ff_two_sum(sacc[j][2][tid], pim[j]);
            sacc[j][2][tid] = a.hi;
            sacc[j][3][tid] += a.lo;
          }
          pr[j] = pim[j] = 0.f;
        }
      }
    }
  }
  if (active) {
    const double inv4pi = 1.0 / (4.0 * kPi);
    for (int j = 0; j < nkb; ++j) {
      const double sr = (double)sacc[j][0][tid] + (double)sacc[j][1][tid];
      const double si = (double)sacc[j][2][tid] + (double)sacc[j][3][tid];
      T[(int64_t)(kbase + j) * M + m] = {(double)s0[j][tid].x + sr * inv4pi, (double)s0[j][tid].y + si * inv4pi};
    }
  }
}

// ------------------------------------------------------------------------------------------
// Pairs of wavenumber groups: the evaluation of k_field32c for two consecutive groups of 16
// wavenumbers at once, wavenumber j of the first group in the low half and of the second in the
// high half of packed FP32 registers.  Both groups use one float-float geometry of the (point,
// quadrature point) pair, and every half goes through k_field32c's operations in its order (each
// group keeps its own start phase and steps by the same rotations), so that the results are the
// same bit for bit whichever kernel a group takes.
//
// Bound: the FMA pipe.  The one-group kernel issues 77.7 slots an evaluation and kept the pipe 61 %
// busy; here 43.6 slots (46 pipe cycles of packed terms and 8 of geometry an evaluation).  Measured
// on 23 040 quadrature points: 512 wavenumbers at 16 384 points 477 -> 367 ms, 64 wavenumbers 76.4
// -> 49 ms (the one-group kernel's 512 CTAs left a nearly empty second wave), 64 at 1000 points on
// 8000 quadrature points 12.7 -> 5.2 ms, two points at 20 picked wavenumbers 19.2 -> 0.43 ms.
// ------------------------------------------------------------------------------------------
constexpr int FPG = 16;      // wavenumbers per group
constexpr int FPP = 2 * FPG; // per pair

// The pairs of a call, launched from y0 on (field_pairs_max of them at a time): pair y holds wavenumbers base[y] .. base[y] + n[y] - 1 (n <= FPP) of the
// call's list, spaced by dk[y] where the launch takes the rotations.
struct PairList {
  ff dk[kMaxFieldBatch];
  int16_t base[kMaxFieldBatch];
  uint8_t n[kMaxFieldBatch];
};

// Surface values at the quadrature points in the pair kernels' layout: [pair][p][j] two float4,
// {P re (group 0), P re (group 1), P im, P im} and the same for P'; zero past the last wavenumber.
// grid (ceil(EQ / 8), pairs), block 128: 16 threads (j) per point.
__global__ void k_interp_pair(const int32_t* __restrict__ elems, int64_t N, int64_t EQ, int Q,
                              const double* __restrict__ qshape, const cd* __restrict__ surf,
                              const __grid_constant__ PairList pairs, int y0, float4* __restrict__ PQ) {
  const int j = threadIdx.x & (FPG - 1);
  const int kbase = pairs.base[y0 + blockIdx.y], nk = pairs.n[y0 + blockIdx.y];
  const int64_t p = blockIdx.x * (int64_t)(blockDim.x / FPG) + threadIdx.x / FPG;
  if (p >= EQ) return;
  const int64_t e = p / Q;
  const int q = (int)(p - e * Q);
  float v[2][4];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int kk = h * FPG + j;
    cd a = {0, 0}, b = {0, 0};
    if (kk < nk) {
      const cd* P = surf + (int64_t)(kbase + kk) * 2 * N;
      const cd* Pn = P + N;
      for (int t = 0; t < 6; ++t) {
        const int32_t i = elems[6 * e + t];
        const double sh = qshape[q * 6 + t];
        a.re += sh * P[i].re; a.im += sh * P[i].im;
        b.re += sh * Pn[i].re; b.im += sh * Pn[i].im;
      }
    }
    v[h][0] = (float)a.re; v[h][1] = (float)a.im; v[h][2] = (float)b.re; v[h][3] = (float)b.im;
  }
  float4* o = PQ + (((int64_t)blockIdx.y * EQ + p) * FPG + j) * 2;
  o[0] = make_float4(v[0][0], v[1][0], v[0][1], v[1][1]);
  o[1] = make_float4(v[0][2], v[1][2], v[0][3], v[1][3]);
}

// Negated surface values at the foot points, {-P0 re (0), -P0 re (1), -P0 im, -P0 im}, the same for P0'.
__device__ __forceinline__ void foot_values_pair(const int32_t* __restrict__ elems, int64_t N, const cd* __restrict__ surf,
                                                 const int32_t* __restrict__ foot_elem, const double* __restrict__ foot,
                                                 int64_t m, int j, int nk, float4* o) {
  const double fxi = foot[8 * m + 6], feta = foot[8 * m + 7];
  const double L1 = 1.0 - fxi - feta;
  const double Nv[6] = {L1 * (2 * L1 - 1), fxi * (2 * fxi - 1), feta * (2 * feta - 1), 4 * L1 * fxi, 4 * fxi * feta,
                        4 * feta * L1};
  const int32_t* el = elems + 6 * (int64_t)foot_elem[m];
  float v[2][4];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int kk = h * FPG + j;
    double a0 = 0, a1 = 0, b0 = 0, b1 = 0;
    if (kk < nk) {
      const cd* P = surf + (int64_t)kk * 2 * N;
      for (int a = 0; a < 6; ++a) {
        const cd v2 = P[el[a]], w = P[N + el[a]];
        a0 += Nv[a] * v2.re; a1 += Nv[a] * v2.im;
        b0 += Nv[a] * w.re; b1 += Nv[a] * w.im;
      }
    }
    v[h][0] = -(float)a0; v[h][1] = -(float)a1; v[h][2] = -(float)b0; v[h][3] = -(float)b1;
  }
  o[0] = make_float4(v[0][0], v[1][0], v[0][1], v[1][1]);
  o[1] = make_float4(v[0][2], v[1][2], v[0][3], v[1][3]);
}

struct PairPoint {  // an observation point, its foot point and the foot's normal
  ff p[3], x0[3], nu0[3];
};
__device__ __forceinline__ void load_pair_point(const double* __restrict__ xp, const double* __restrict__ foot, int64_t m,
                                                PairPoint& o) {
  for (int d = 0; d < 3; ++d) {
    o.p[d] = ff_from_double(xp[3 * m + d]);
    o.x0[d] = ff_from_double(foot[8 * m + d]);
    o.nu0[d] = ff_from_double(foot[8 * m + 3 + d]);
  }
}

// One quadrature point's terms for the pair, added to the run sums pr, pi.  g0..g3: the point's
// record (13 table values); pq: its surface values [FPG][2]; s0: the foot values, stride ss float4
// between wavenumbers; nj: wavenumbers of the longer half; sk [FPG]: {k, k, 1/k, 1/k}; skl [FPG]: the low parts of k.  UNI: uniformly
// spaced groups (phases by rotation), dk the step.
template <bool UNI, bool ZF>
__device__ __forceinline__ void pair_terms(const float4 g0, const float4 g1, const float4 g2, const float4 g3,
                                           const PairPoint& o, const float4* __restrict__ pq,
                                           const float4* __restrict__ s0, int ss, const float4* __restrict__ sk,
                                           const float2* __restrict__ skl, int nj, ff dk, float far_r2, f2* pr, f2* pi) {
  const ff qx = {g0.x, g0.w}, qy = {g0.y, g1.x}, qz = {g0.z, g1.y};
  const float nx = g1.z, ny = g1.w, nz = g2.x, wj = g2.y;
  const ff nux = {nx, g2.z}, nuy = {ny, g2.w}, nuz = {nz, g3.x};
  const ff rpx = ff_diff_lazy(qx, o.p[0]), rpy = ff_diff_lazy(qy, o.p[1]), rpz = ff_diff_lazy(qz, o.p[2]);
  const ff r0x = ff_diff_lazy(qx, o.x0[0]), r0y = ff_diff_lazy(qy, o.x0[1]), r0z = ff_diff_lazy(qz, o.x0[2]);
  const ff R0sq = ff_norm2_lazy(r0x, r0y, r0z);
  float iRp, iR0;
  const ff Rp = ff_sqrt_lazy(ff_norm2_lazy(rpx, rpy, rpz), iRp);
  const ff R0 = ff_sqrt_lazy(R0sq, iR0);
  const ff nr = ff_dot3_lazy(o.nu0, r0x, r0y, r0z);
  const float ap = wj * iRp, a0 = wj * iR0;
  const float rnp = ((rpx.hi + rpx.lo) * nx + (rpy.hi + rpy.lo) * ny + (rpz.hi + rpz.lo) * nz) * iRp * iRp;
  float rn0;
  if (R0sq.hi > far_r2) {
    rn0 = (r0x.hi + r0x.lo) * nx + (r0y.hi + r0y.lo) * ny + (r0z.hi + r0z.lo) * nz;
  } else {
    const ff nuq[3] = {nux, nuy, nuz};
    const ff d = ff_dot3_lazy(nuq, r0x, r0y, r0z);
    rn0 = d.hi + d.lo;
  }
  rn0 *= iR0 * iR0;
  const float nn = o.nu0[0].hi * nx + o.nu0[1].hi * ny + o.nu0[2].hi * nz;
  const f2 Rph = f2_dup(Rp.hi), R0h = f2_dup(R0.hi), rnp2 = f2_dup(rnp), nrnp2 = f2_dup(-rnp), rn02 = f2_dup(rn0);
  const f2 nn2 = f2_dup(nn), nnn2 = f2_dup(-nn), ap2 = f2_dup(ap), a02 = f2_dup(a0);
  f2 cp, sp, c0, s0v, cg, sg;
  f2 dcp, dsp, dc0, ds0, dcg, dsg, ndsp, nds0, ndsg;
  if (UNI) {
    const float4 k4 = sk[0];
    const float2 kl = skl[0];
    const f2 nkh = f2_make(-k4.x, -k4.y), nkl = f2_make(-kl.x, -kl.y);
    cis_ffprod2(nkh, nkl, Rp, cp, sp);
    cis_ffprod2(nkh, nkl, R0, c0, s0v);
    cis_ffprod2(nkh, nkl, nr, cg, sg);
    float a, b;
    cis_ffprod(dk, Rp, a, b);
    dcp = f2_dup(a); dsp = f2_dup(b); ndsp = f2_dup(-b);
    cis_ffprod(dk, R0, a, b);
    dc0 = f2_dup(a); ds0 = f2_dup(b); nds0 = f2_dup(-b);
    cis_ffprod(dk, nr, a, b);
    dcg = f2_dup(a); dsg = f2_dup(b); ndsg = f2_dup(-b);
    cp = f2_mul(cp, ap2); sp = f2_mul(sp, ap2);
    c0 = f2_mul(c0, a02); s0v = f2_mul(s0v, a02);
  }
#pragma unroll
  for (int j = 0; j < FPG; ++j) {
    if (j >= nj) break;  // (uniform over the CTA)
    const float4 k4 = sk[j];
    const f2 kh = f2_make(k4.x, k4.y), kinv = f2_make(k4.z, k4.w);
    if (!UNI) {
      const float2 kl = skl[j];
      const f2 nkh = f2_make(-k4.x, -k4.y), nkl = f2_make(-kl.x, -kl.y);
      cis_ffprod2(nkh, nkl, Rp, cp, sp);
      cis_ffprod2(nkh, nkl, R0, c0, s0v);
      cis_ffprod2(nkh, nkl, nr, cg, sg);
      cp = f2_mul(cp, ap2); sp = f2_mul(sp, ap2);
      c0 = f2_mul(c0, a02); s0v = f2_mul(s0v, a02);
    } else if (j > 0) {
      f2 t = f2_fma(cp, dcp, f2_mul(sp, ndsp));
      sp = f2_fma(sp, dcp, f2_mul(cp, dsp));
      cp = t;
      t = f2_fma(c0, dc0, f2_mul(s0v, nds0));
      s0v = f2_fma(s0v, dc0, f2_mul(c0, ds0));
      c0 = t;
      t = f2_fma(cg, dcg, f2_mul(sg, ndsg));
      sg = f2_fma(sg, dcg, f2_mul(cg, dsg));
      cg = t;
    }
    const f2 kRp = f2_mul(kh, Rph), kR0 = f2_mul(kh, R0h);
    const f2 ngdr = f2_sub(c0, cp), gdi = f2_sub(sp, s0v);
    const f2 ddr = f2_fma(f2_fma(s0v, kR0, c0), rn02, f2_mul(f2_fma(sp, kRp, cp), nrnp2));
    // -(dG im): kept negated, the sign returned where it enters with a plus
    const f2 nddi = f2_fma(f2_fma(cp, kRp, f2_neg(sp)), nrnp2, f2_mul(f2_fma(c0, kR0, f2_neg(s0v)), rn02));
    f2 f = f2_mul(sg, kinv);
    if (ZF) {  // f's limit nu0.r at k = 0 (kinv 0)
      float f0, f1;
      f2_split(f, f0, f1);
      f = f2_make(k4.z == 0.f ? nr.hi : f0, k4.w == 0.f ? nr.hi : f1);
    }
    const f2 dg = f2_mul(f2_mul(kh, sg), nnn2), df = f2_mul(cg, nn2);
    const float4 z0 = s0[j * ss * 2], z1 = s0[j * ss * 2 + 1], u0 = pq[2 * j], u1 = pq[2 * j + 1];
    const f2 nP0r = f2_make(z0.x, z0.y), nP0i = f2_make(z0.z, z0.w), nQ0r = f2_make(z1.x, z1.y), nQ0i = f2_make(z1.z, z1.w);
    const f2 Ptr = f2_fma(nQ0r, f, f2_fma(nP0r, cg, f2_make(u0.x, u0.y)));
    const f2 Pti = f2_fma(nQ0i, f, f2_fma(nP0i, cg, f2_make(u0.z, u0.w)));
    const f2 dPr = f2_fma(nQ0r, df, f2_fma(nP0r, dg, f2_make(u1.x, u1.y)));
    const f2 dPi = f2_fma(nQ0i, df, f2_fma(nP0i, dg, f2_make(u1.z, u1.w)));
    f2 a = f2_fma(Ptr, ddr, pr[j]);
    a = f2_fma(Pti, nddi, a);
    a = f2_fma(ngdr, dPr, a);
    pr[j] = f2_fma(gdi, dPi, a);
    a = f2_fma(Ptr, f2_neg(nddi), pi[j]);
    a = f2_fma(Pti, ddr, a);
    a = f2_fma(ngdr, dPi, a);
    pi[j] = f2_fma(f2_neg(gdi), dPr, a);
  }
}

// Adds a run sum to a compensated sum (s, c).
__device__ __forceinline__ void add_run(float run, float& s, float& c) {
  const ff a = ff_two_sum(s, run);
  s = a.hi;
  c += a.lo;
}

// A CTA of W warps evaluates P points (a power of two up to 32) for one pair.  A lane takes one
// point and one run of 32 quadrature points at a time; the W 32 / P runs in flight leave their sums
// in shared memory, and the threads of the CTA add them in the order of the runs to compensated
// sums that live in T itself between rounds (four floats in the 16 bytes of a value): the order of
// the additions, hence the result, does not depend on P or W.  DIRECT (P < 32): lanes of a warp are at
// different quadrature points, which they read from global memory; otherwise each warp stages
// tiles of 8 points.
template <bool UNI, bool ZF, bool DIRECT>
__global__ void __launch_bounds__(384, 1) k_field_pair(const int32_t* __restrict__ elems, int64_t N, int64_t EQ,
                                                       const float* __restrict__ qtab, const float4* __restrict__ PQ,
                                                       const cd* __restrict__ surf, const double* __restrict__ xp,
                                                       int64_t M, const int32_t* __restrict__ foot_elem,
                                                       const double* __restrict__ foot, const double* __restrict__ kv,
                                                       const __grid_constant__ PairList pairs, int y0, int P_, cd* __restrict__ T,
                                                       float far_r2) {
  constexpr int UT = 8;
  const int P = DIRECT ? P_ : 32;
  extern __shared__ float4 fp_smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, W = nt >> 5;
  const int G = 32 / P, pt = lane & (P - 1), rs = lane / P;
  float4* s0 = fp_smem;                                  // [FPG][2 P]: point t's values at [j][2 t], [j][2 t + 1]
  float4* sk = s0 + FPG * 2 * P;                         // [FPG]
  float2* skl = (float2*)(sk + FPG);                     // [FPG]
  float2* sr = skl + FPG;                                // [W][FPG][2][32]: the runs' sums
  float4* sg = (float4*)(sr + W * FPG * 2 * 32) + warp * UT * (4 + 2 * FPG);  // this warp's tile: [UT][4]
  float4* sq = sg + UT * 4;                              // [UT][FPG][2]
  const int kbase = pairs.base[y0 + blockIdx.y], nk = pairs.n[y0 + blockIdx.y], nj = min(nk, FPG);
  const int64_t m0 = (int64_t)blockIdx.x * P;
  ff dk = {0.f, 0.f};
  if (UNI) dk = pairs.dk[y0 + blockIdx.y];
  if (tid < FPG) {
    ff k[2] = {{0.f, 0.f}, {0.f, 0.f}};
    float ki[2] = {0.f, 0.f};
    for (int h = 0; h < 2; ++h) {
      const int kk = h * FPG + tid;
      if (kk < nk) {
        k[h] = ff_from_double(kv[kbase + kk]);
        ki[h] = kinv32(kv[kbase + kk]);
      }
    }
    sk[tid] = make_float4(k[0].hi, k[1].hi, ki[0], ki[1]);
    skl[tid] = make_float2(k[0].lo, k[1].lo);
  }
  for (int e = tid; e < P * FPG; e += nt) {
    const int t = e & (P - 1), j = e / P;
    if (m0 + t < M)
      foot_values_pair(elems, N, surf + (int64_t)kbase * 2 * N, foot_elem, foot, m0 + t, j, nk, s0 + (j * P + t) * 2);
  }
  const bool active = m0 + pt < M;
  PairPoint o;
  if (active) load_pair_point(xp, foot, m0 + pt, o);
  __syncthreads();
  const float4* pqk = PQ + (int64_t)blockIdx.y * EQ * FPG * 2;
  const int nruns = (int)((EQ + 31) / 32);
  f2 pr[FPG], pi[FPG];
  for (int r0 = 0; r0 < nruns; r0 += W * G) {
#pragma unroll
    for (int j = 0; j < FPG; ++j) pr[j].v = pi[j].v = 0ull;
    const int64_t q0 = (int64_t)(r0 + warp * G + rs) * 32;
    const int cnt = (int)(EQ - q0 < 32 ? EQ - q0 : 32);  // <= 0 past the last run
    if (DIRECT) {
      if (active)
#pragma unroll 1
        for (int u = 0; u < cnt; ++u) {
          const int64_t q = q0 + u;
          float v[13];
#pragma unroll
          for (int f = 0; f < 13; ++f) v[f] = __ldg(qtab + f * EQ + q);
          pair_terms<UNI, ZF>(make_float4(v[0], v[1], v[2], v[3]), make_float4(v[4], v[5], v[6], v[7]),
                              make_float4(v[8], v[9], v[10], v[11]), make_float4(v[12], 0.f, 0.f, 0.f), o,
                              pqk + q * FPG * 2, s0 + pt * 2, P, sk, skl, nj, dk, far_r2, pr, pi);
        }
    } else {
#pragma unroll 1
      for (int t0 = 0; t0 < cnt; t0 += UT) {
        const int tc = cnt - t0 < UT ? cnt - t0 : UT;
        __syncwarp();
        for (int e = lane; e < 13 * UT; e += 32) {
          const int f = e / UT, u = e - f * UT;
          if (u < tc) reinterpret_cast<float*>(sg + u * 4)[f] = qtab[f * EQ + q0 + t0 + u];
        }
        const float4* src = pqk + (q0 + t0) * FPG * 2;
        for (int e = lane; e < tc * FPG * 2; e += 32) sq[e] = src[e];
        __syncwarp();
        if (active)
#pragma unroll 1
          for (int u = 0; u < tc; ++u) {
            asm volatile("" ::: "memory");  // the foot values stay in shared memory (128 registers otherwise)
            pair_terms<UNI, ZF>(sg[4 * u], sg[4 * u + 1], sg[4 * u + 2], sg[4 * u + 3], o, sq + u * FPG * 2, s0 + pt * 2, P,
                                sk, skl, nj, dk, far_r2, pr, pi);
          }
      }
    }
#pragma unroll
    for (int j = 0; j < FPG; ++j) {
      float r[2], i[2];
      f2_split(pr[j], r[0], r[1]);
      f2_split(pi[j], i[0], i[1]);
      float2* d = sr + ((warp * FPG + j) * 2) * 32 + lane;
      d[0] = make_float2(r[0], i[0]);
      d[32] = make_float2(r[1], i[1]);
    }
    __syncthreads();
    const int have = min(W * G, nruns - r0);
    for (int e = tid; e < P * FPP; e += nt) {
      const int t = e & (P - 1), kk = e / P, h = kk / FPG, j = kk - h * FPG;
      if (kk >= nk || m0 + t >= M) continue;
      cd* out = T + (int64_t)(kbase + kk) * M + m0 + t;
      float2* a = reinterpret_cast<float2*>(out);
      float2 re = make_float2(0.f, 0.f), im = re;
      if (r0 > 0) { re = a[0]; im = a[1]; }
      for (int r = 0; r < have; ++r) {
        const int w = r / G, g = r - w * G;
        const float2 v = sr[((w * FPG + j) * 2 + h) * 32 + g * P + t];
        add_run(v.x, re.x, re.y);
        add_run(v.y, im.x, im.y);
      }
      if (r0 + have < nruns) {
        a[0] = re;
        a[1] = im;
      } else {
        const double inv4pi = 1.0 / (4.0 * kPi);
        const float4 z = s0[(j * P + t) * 2];
        const double P0r = -(double)(h ? z.y : z.x), P0i = -(double)(h ? z.w : z.z);
        const double vr = (double)re.x + (double)re.y, vi = (double)im.x + (double)im.y;
        *out = {P0r + vr * inv4pi, P0i + vi * inv4pi};
      }
    }
    __syncthreads();
  }
}

double far_radius2(bie_ctx* c);

template <int KB, int TP, int MINB, int UT>
static void launch_field32c(bie_ctx* c, int64_t EQ, const cf* Pq, const cf* Pnq, const cd* surf, const double* xp,
                            int64_t M, const int32_t* foot_elem, const double* foot, const double* kv, int nk, cd* T,
                            TwoPi3f tp, int uniform, ff dk, bool zero) {
  (void)tp;
  dim3 gb((unsigned)((M + TP - 1) / TP), (unsigned)((nk + KB - 1) / KB));
  const float far_r2 = (float)far_radius2(c);
  if (zero)
    BIE_LAUNCH(k_field32c<KB, TP, MINB, UT, true><<<gb, TP, 0, c->stream>>>(
        c->elems, c->N, EQ, c->qgeo32, Pq, Pnq, surf, xp, M, foot_elem, foot, kv, nk, T, uniform, dk, far_r2));
  else
    BIE_LAUNCH(k_field32c<KB, TP, MINB, UT, false><<<gb, TP, 0, c->stream>>>(
        c->elems, c->N, EQ, c->qgeo32, Pq, Pnq, surf, xp, M, foot_elem, foot, kv, nk, T, uniform, dk, far_r2));
}

int ensure_mixed_tables(bie_ctx* c);

// The pairs y0 .. y0 + np - 1 of `l` by k_field_pair.  How the points and runs are laid out: with at least
// two CTAs of 32 points and 4 warps to an SM (three are resident) that layout; fewer points leave
// SMs without work, so a CTA takes 12 warps (one CTA fills its SM's registers) and the most points
// that still give every SM one (M = 3000, 7 wavenumbers: 20 -> 4 ms; M = 1: 3.1 -> 0.1 ms).
static int launch_pairs(bie_ctx* c, const cd* surf, const double* xp, int64_t M, const int32_t* foot_elem,
                        const double* foot, const double* kv, const PairList& l, int y0, int np, bool uni, cd* T,
                        bool zero, float4* PQ, int nsm) {
  const int64_t EQ = c->E * c->rule.Q;
  const float far_r2 = (float)far_radius2(c);
  BIE_LAUNCH(k_interp_pair<<<dim3((unsigned)((EQ + 7) / 8), (unsigned)np), 128, 0, c->stream>>>(
      c->elems, c->N, EQ, c->rule.Q, c->qshape, surf, l, y0, PQ));
  int P = 32, W = 4;
  auto ctas = [&](int p) { return (M + p - 1) / p * np; };
  if (ctas(32) < 2 * nsm) {
    W = 12;
    while (P > 1 && ctas(P) < nsm) P >>= 1;
  }
  const size_t smem = (size_t)(FPG * 2 * P + FPG) * sizeof(float4) + FPG * sizeof(float2) +
                      (size_t)W * FPG * 2 * 32 * sizeof(float2) +
                      (P == 32 ? (size_t)W * 8 * (4 + 2 * FPG) * sizeof(float4) : 0);
  const dim3 g((unsigned)((M + P - 1) / P), (unsigned)np);
  auto go = [&](auto kernel) -> int {
    BIE_TRY(set_smem_max(kernel));
    BIE_LAUNCH(kernel<<<g, 32 * W, smem, c->stream>>>(c->elems, c->N, EQ, c->qgeo32, PQ, surf, xp, M, foot_elem, foot, kv, l,
                                                      y0, P, T, far_r2));
    return BIE_OK;
  };
  if (P == 32) {
    if (uni) return zero ? go(k_field_pair<true, true, false>) : go(k_field_pair<true, false, false>);
    return zero ? go(k_field_pair<false, true, false>) : go(k_field_pair<false, false, false>);
  }
  if (uni) return zero ? go(k_field_pair<true, true, true>) : go(k_field_pair<true, false, true>);
  return zero ? go(k_field_pair<false, true, true>) : go(k_field_pair<false, false, true>);
}

// Segments of a wavenumber list, (start, length): maximal runs of equally spaced wavenumbers (at
// least 4) take the phase recurrence inside their groups of 16, the rest runs without it (a
// negative length) -- so that a sweep with the zero-frequency term in front (or any uniform runs
// inside a list) keeps the recurrence where it applies.
static std::vector<std::pair<int, int>> field_segments(const double* hk, int nk) {
  std::vector<std::pair<int, int>> segs;
  int i = 0, nu_start = -1;
  while (i < nk) {
    int L = 1;
    if (i + 1 < nk) {
      const double d = hk[i + 1] - hk[i];
      L = 2;
      if (!(d > 0.0)) L = 1;
      else
        while (i + L < nk && std::fabs(hk[i + L] - (hk[i] + L * d)) <= 1e-12 * std::fabs(hk[i + L])) ++L;
    }
    if (L >= 4) {
      if (nu_start >= 0) { segs.push_back({nu_start, -(i - nu_start)}); nu_start = -1; }
      segs.push_back({i, L});
      i += L;
    } else {
      if (nu_start < 0) nu_start = i;
      ++i;
    }
  }
  if (nu_start >= 0) segs.push_back({nu_start, -(nk - nu_start)});
  return segs;
}

// Whether a segment's single last group of n <= 16 wavenumbers takes the one-group kernel (k_field32c)
// instead of a pair with an empty second half, whose packed instructions are half wasted.  The
// one-group kernel's 128-point CTAs take as long for one point as for 128 on every SM; measured on 23 040 quadrature points at M = 16 384: 26.2 ms against the pair's 28.3 for
// n = 16, 19.2 against 13.9 for n = 5 (equal near n = 13); M = 3000, n = 7: 20 against 4 ms.
static bool scalar_tail(int64_t M, int n, int nsm) { return M >= (int64_t)2 * nsm * 128 || (M >= (int64_t)100 * nsm && n > 12); }

// The pairs of wavenumber groups of a list (uniform segments' and the others'), and the scalar
// kernel's groups (start, length, segment's step or 0).
struct FieldPlan {
  PairList uni, gen;
  int nuni = 0, ngen = 0;
  bool zuni = false, zgen = false;  // k = 0 among them
  struct Tail { int start, n, uniform; double dk; };
  std::vector<Tail> tails;
};
static void field_plan(const double* hk, int nk, int64_t M, int nsm, FieldPlan& f) {
  for (const auto& sg : field_segments(hk, nk)) {
    const int r0 = sg.first, n = sg.second > 0 ? sg.second : -sg.second;
    const bool uniform = sg.second > 0;
    const double dk = uniform ? hk[r0 + 1] - hk[r0] : 0.0;
    for (int i = 0; i < n; i += FPP) {
      const int m = std::min(FPP, n - i);
      if (m <= FPG && scalar_tail(M, m, nsm)) {
        f.tails.push_back({r0 + i, m, uniform ? 1 : 0, dk});
        continue;
      }
      PairList& l = uniform ? f.uni : f.gen;
      int& np = uniform ? f.nuni : f.ngen;
      l.base[np] = (int16_t)(r0 + i);
      l.n[np] = (uint8_t)m;
      l.dk[np] = ff_from_double(dk);
      ++np;
      for (int j = 0; j < m; ++j) (uniform ? f.zuni : f.zgen) |= hk[r0 + i + j] == 0.0;
    }
  }
}

// Pairs of one launch: one for every 16 wavenumbers of the list, twice what full pairs take.  A list of short runs makes
// more, each with a full pair's scratch however few its wavenumbers: they follow one another through
// the same scratch.
static int field_pairs_max(int nk) { return std::max(1, (nk + FPG - 1) / FPG); }

// Scratch of field_mixed in bytes for nk wavenumbers at M points.
size_t field_mixed_scratch(bie_ctx* c, const double* hk, int nk, int64_t M, int nsm) {
  const size_t EQ = (size_t)(c->E * c->rule.Q);
  size_t values = 2 * (size_t)nk * EQ * sizeof(cf);  // P and P' at the quadrature points
  if (c->field_accurate_phase && c->field_variant == 2) {
    FieldPlan f;
    field_plan(hk, nk, M, nsm, f);
    values = (f.tails.empty() ? 0 : 2 * FPG * EQ * sizeof(cf)) + (size_t)std::min(field_pairs_max(nk), std::max(f.nuni, f.ngen)) * EQ * FPP * 2 * sizeof(cf);
  }
  return values + 512;
}

// Evaluates nk <= kMaxFieldBatch wavenumbers (hk on the host, kv the same on the device).
int field_mixed(bie_ctx* c, const double* hk, const double* kv, int nk, const cd* surf, const double* xp, int64_t M,
                const int32_t* foot_elem, const double* foot, cd* T, void* scratch, size_t scratch_bytes, int nsm) {
  BIE_TRY(ensure_mixed_tables(c));
  const int64_t EQ = c->E * c->rule.Q;
  if (nk > kMaxFieldBatch || field_mixed_scratch(c, hk, nk, M, nsm) > scratch_bytes)
    return fail(BIE_ERR_STATE, "field scratch too small");
  if (M <= 0) return BIE_OK;
  cf* Pq = (cf*)scratch;
  auto interp = [&](int start, int n) -> cf* {  // P at the quadrature points from Pq on, returns P'
    dim3 gi((unsigned)((EQ + 255) / 256), n);
    cf* Pnq = Pq + (int64_t)n * EQ;
    BIE_LAUNCH(k_interp_q32<<<gi, 256, 0, c->stream>>>(c->elems, c->N, c->E, c->rule.Q, c->qshape,
                                                       surf + (int64_t)start * 2 * c->N, Pq, Pnq));
    return Pnq;
  };
  TwoPi3f tp;
  const double two_pi = 2.0 * kPi;
  tp.c1 = (float)two_pi;
  tp.c2 = (float)(two_pi - (double)tp.c1);
  tp.c3 = (float)((two_pi - (double)tp.c1 - (double)tp.c2) + 2.4492935982947064e-16);
  tp.inv = (float)(1.0 / two_pi);
  if (!c->field_accurate_phase) {
    const cf* Pnq = interp(0, nk);
    dim3 gf((unsigned)((M + FT - 1) / FT), nk);
    BIE_LAUNCH(k_field32<false><<<gf, FT, 0, c->stream>>>(c->elems, c->N, EQ, c->qgeo32, Pq, Pnq, surf, xp, M, foot_elem,
                                                          foot, kv, T, tp));
  } else if (c->field_variant == 2) {
    FieldPlan f;
    field_plan(hk, nk, M, nsm, f);
    float4* PQ = (float4*)scratch;
    if (!f.tails.empty()) PQ = (float4*)(((uintptr_t)(Pq + 2 * FPG * EQ) + 255) & ~(uintptr_t)255);
    const int most = field_pairs_max(nk);
    for (int uni = 1; uni >= 0; --uni)
      for (int y0 = 0, np = uni ? f.nuni : f.ngen; y0 < np; y0 += most)
        BIE_TRY(launch_pairs(c, surf, xp, M, foot_elem, foot, kv, uni ? f.uni : f.gen, y0, std::min(most, np - y0), uni != 0, T,
                             uni ? f.zuni : f.zgen, PQ, nsm));
    for (const auto& t : f.tails) {
      const cf* Pnq = interp(t.start, t.n);
      bool zero = false;
      for (int j = 0; j < t.n; ++j) zero |= hk[t.start + j] == 0.0;
      launch_field32c<16, 128, 3, 32>(c, EQ, Pq, Pnq, surf + (int64_t)t.start * 2 * c->N, xp, M, foot_elem, foot,
                                      kv + t.start, t.n, T + (int64_t)t.start * M, tp, t.uniform, ff_from_double(t.dk), zero);
    }
  } else {
    const cf* Pnq = interp(0, nk);
    for (const auto& sg : field_segments(hk, nk)) {  // one launch each
      const int r0 = sg.first, n = sg.second > 0 ? sg.second : -sg.second;
      const int uniform = sg.second > 0 ? 1 : 0;
      const double dkv = uniform ? hk[r0 + 1] - hk[r0] : 0.0;
      // k = 0 (the zero-frequency term) takes f's limit inside the kernel; launches without it
      // keep that select out of the inner loop
      bool zero_s = false;
      for (int j = 0; j < n; ++j) zero_s |= hk[r0 + j] == 0.0;
      const ff dkf = ff_from_double(dkv);
      const double* kr = kv + r0;
      const cf *Pqr = Pq + (int64_t)r0 * EQ, *Pnqr = Pnq + (int64_t)r0 * EQ;
      const cd* sr = surf + (int64_t)r0 * 2 * c->N;
      cd* Tr = T + (int64_t)r0 * M;
      if (c->field_variant == 1) {
        launch_field32c<16, 64, 4, 64>(c, EQ, Pqr, Pnqr, sr, xp, M, foot_elem, foot, kr, n, Tr, tp, uniform, dkf, zero_s);
      } else {
        dim3 gb((unsigned)((M + FT - 1) / FT), (unsigned)((n + FKB - 1) / FKB));
        BIE_LAUNCH(k_field32b<<<gb, FT, 0, c->stream>>>(c->elems, c->N, EQ, c->qgeo32, Pqr, Pnqr, sr, xp, M, foot_elem,
                                                        foot, kr, n, Tr, tp, uniform, dkf));
      }
    }
  }
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

}  // namespace bie
