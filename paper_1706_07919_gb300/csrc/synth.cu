// synth.cu -- pulse spectra and space-time synthesis by the discrete Fourier transform with the
// sign of Eq. (inverseFourier) (exp(-i omega t)), evaluated by a radix-2 FFT (the last paragraph
// of Sec. 3 asks for the discrete fast Fourier transform).
//   spectrum:  S[p][m] = sum_n s[p][n] exp(+2 pi i m n / Nt) = conj(FFT(s))_m  (real s)
//   synthesis: out[p][x][n] = (1/Nt) Re sum_m c_m exp(-2 pi i m n / Nt),  c_m = w_m S[p][m] T[m][x],
//              w_0 = w_{Nt/2} = 1, else 2 (the m > Nt/2 half is the complex conjugate).
// Spectra, and the shortest or fewest signals: one CTA transforms one signal in shared memory with a Stockham
// (self-sorting) radix-2 FFT; others by k_synth_real.
#include <algorithm>
#include <mutex>

#include "bie_common.cuh"

namespace bie {

template <class S> struct C2 { S re, im; };

// tw[j] = exp(-2 pi i j / n), j < n/2, from sincospi (correctly rounded to ~1 ulp in FP64).
__global__ void k_twiddles(int n, double2* tw) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n / 2) return;
  double s, c;
  sincospi(2.0 * (double)j / (double)n, &s, &c);
  tw[j] = make_double2(c, -s);
}

// Forward FFT of buf (length n, power of two) in place, using tmp as the ping-pong partner.
// Returns the buffer that holds the result.
template <class S>
__device__ C2<S>* stockham(C2<S>* buf, C2<S>* tmp, int n, const double2* __restrict__ tw) {
  C2<S>* x = buf;
  C2<S>* y = tmp;
  for (int m = 1; m < n; m <<= 1) {
    const int twstep = n / (2 * m);
    for (int t = threadIdx.x; t < n / 2; t += blockDim.x) {
      const int j = t / m, kk = t - j * m;
      const double2 w2 = tw[kk * twstep];
      const C2<S> w = {(S)w2.x, (S)w2.y};
      const C2<S> a = x[j * m + kk], b = x[j * m + kk + n / 2];
      const C2<S> wb = {w.re * b.re - w.im * b.im, w.re * b.im + w.im * b.re};
      y[2 * j * m + kk] = {a.re + wb.re, a.im + wb.im};
      y[2 * j * m + kk + m] = {a.re - wb.re, a.im - wb.im};
    }
    __syncthreads();
    C2<S>* t = x;
    x = y;
    y = t;
  }
  return x;
}

template <class S>
__global__ void k_pulse_spectrum(const double* __restrict__ s, int n, const double2* __restrict__ tw,
                                 cd* __restrict__ Sout) {
  extern __shared__ unsigned char smem_raw[];
  C2<S>* buf = reinterpret_cast<C2<S>*>(smem_raw);
  C2<S>* tmp = buf + n;
  const double* sp = s + (int64_t)blockIdx.x * n;
  for (int t = threadIdx.x; t < n; t += blockDim.x) buf[t] = {(S)sp[t], (S)0};
  __syncthreads();
  C2<S>* X = stockham<S>(buf, tmp, n, tw);
  cd* o = Sout + (int64_t)blockIdx.x * (n / 2 + 1);
  for (int t = threadIdx.x; t <= n / 2; t += blockDim.x) o[t] = {(double)X[t].re, -(double)X[t].im};
}

// Synthesis of the shortest or fewest signals (synth_radix2); grid: (M, P), one signal per CTA.
template <class S, class O>
__global__ void k_synth(const cd* __restrict__ T, const int64_t* __restrict__ midx, int nk, int64_t M,
                        const cd* __restrict__ Sp, int n, const double2* __restrict__ tw, O* __restrict__ out) {
  extern __shared__ unsigned char smem_raw[];
  C2<S>* buf = reinterpret_cast<C2<S>*>(smem_raw);
  C2<S>* tmp = buf + n;
  const int64_t x = blockIdx.x;
  const int p = blockIdx.y;
  for (int t = threadIdx.x; t < n; t += blockDim.x) buf[t] = {(S)0, (S)0};
  __syncthreads();
  const cd* Srow = Sp + (int64_t)p * (n / 2 + 1);
  for (int r = threadIdx.x; r < nk; r += blockDim.x) {
    const int m = (int)midx[r];
    const double w = (m == 0 || 2 * m == n) ? 1.0 : 2.0;
    const cd a = cmul(Srow[m], T[(int64_t)r * M + x]);
    buf[m] = {(S)(w * a.re), (S)(w * a.im)};
  }
  __syncthreads();
  C2<S>* X = stockham<S>(buf, tmp, n, tw);
  O* o = out + ((int64_t)p * M + x) * n;
  const S inv = (S)1 / (S)n;
  for (int t = threadIdx.x; t < n; t += blockDim.x) o[t] = (O)(X[t].re * inv);
}

// ---- synthesis of many or long signals ------------------------------------------------
// A real signal of n samples is one complex transform of h = n / 2 values,
//   out[2 j] + i out[2 j + 1] = sum_k Z_k exp(-2 pi i j k / h),
//   Z_k = H_k (1 + i w_k) + conj(H_{h-k} (1 - i w_{h-k})),  w_k = exp(-2 pi i k / n),
// H_m = S_m T_m / n for 0 < m < h, H_0 and H_h the real parts of theirs; a frequency thus adds to Z_m and to
// Z_{h-m}.  h / 16 threads take a signal, 16 values each in registers: one pass of radix 2, 4 or 8
// where log2 h leaves a remainder, then radix-16 passes (Stockham order), exchanging through shared memory
// between passes -- two exchanges for n = 4096, where the radix-2 kernel had twelve round trips through
// shared memory, each with a division and a twiddle converted from FP64.  A CTA of up to 256 threads
// holds SB neighbouring points, so that T is read in whole sectors, and takes PG pulses one
// after the other with the points' T kept in shared memory.  FP32: S (1 + i w) / n and S (1 - i w) / n
// (`sp`, once per call) and T (once per point) enter as float-float and their products round once, as
// the FP64 product rounded to FP32 did: eight FP64 operations a frequency, point and pulse would cost 0.4 ms
// below on this GPU's narrow FP64 pipe.  Without `sp` the products are formed in FP64.
// Bound: shared memory and the transforms' arithmetic in about equal parts (DRAM: 1.1 GB written).
// Measured, the call for 8 pulses x 8192 points x 4096 samples from 512 frequencies in FP32: 7.2 -> 0.67 ms
// (with the factors 1 +- i w taken in the first pass, from rounded H, 0.84; with the passes' factors read
// out of the plain table and that, 1.6); without `sp` 1.43.
// Relative error against FP64 of 4096 / 512 samples, every frequency: 1.22e-7 / 1.03e-7 before (radix 2), 1.16e-7
// / 0.98e-7 here; an eighth of the frequencies: 1.10e-7 / 0.89e-7 and 1.09e-7 / 0.90e-7 (at 64 samples 0.67e-7
// and 0.70e-7: radix 2 adds exact zeros there).  That takes the products rounded once into Z and the fixed
// factors with their rests: 1.25e-7 / 1.08e-7 without.
template <class S> __device__ __forceinline__ C2<S> c2mul(C2<S> a, C2<S> b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <class S> __device__ __forceinline__ C2<S> c2add(C2<S> a, C2<S> b) { return {a.re + b.re, a.im + b.im}; }
template <class S> __device__ __forceinline__ C2<S> c2sub(C2<S> a, C2<S> b) { return {a.re - b.re, a.im - b.im}; }

// a transform's fixed factors, each as a value of its type and the rest: rounded alone they would add an error
// of the size of the products' own
template <class S> struct Fix {
  S hi, lo;
  __host__ __device__ constexpr Fix(double v, double rest) : hi((S)v), lo((S)((v - (double)(S)v) + rest)) {}
  __device__ __forceinline__ S operator()(S x) const { return fma(x, hi, x * lo); }
};
template <class S> __device__ __forceinline__ C2<S> c2fix(C2<S> a, Fix<S> c, Fix<S> s) {  // a (c + i s)
  return {fma(a.re, c.hi, fma(-a.im, s.hi, fma(a.re, c.lo, -(a.im * s.lo)))),
          fma(a.re, s.hi, fma(a.im, c.hi, fma(a.re, s.lo, a.im * c.lo)))};
}

template <class S> __device__ __forceinline__ void fft2(C2<S>& a, C2<S>& b) {
  const C2<S> t = c2sub(a, b);
  a = c2add(a, b);
  b = t;
}
template <class S> __device__ __forceinline__ void fft4(C2<S>& a, C2<S>& b, C2<S>& c, C2<S>& d) {
  const C2<S> t0 = c2add(a, c), t1 = c2sub(a, c), t2 = c2add(b, d), u = c2sub(b, d), t3 = {u.im, -u.re};
  a = c2add(t0, t2);
  b = c2add(t1, t3);
  c = c2sub(t0, t2);
  d = c2sub(t1, t3);
}
// Transforms of v[0 .. R-1]; output k is left at v[fft_at<R>(k)].
template <int R, class S> __device__ __forceinline__ void fft_small(C2<S>* v) {
  if constexpr (R == 2) {
    fft2(v[0], v[1]);
  } else if constexpr (R == 4) {
    fft4(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 8) {
    constexpr Fix<S> h(0.70710678118654752440, -4.833646656726457e-17);  // sqrt(1/2)
    fft4(v[0], v[2], v[4], v[6]);
    fft4(v[1], v[3], v[5], v[7]);
    v[3] = C2<S>{h(v[3].re + v[3].im), h(v[3].im - v[3].re)};
    v[5] = C2<S>{v[5].im, -v[5].re};
    v[7] = C2<S>{h(v[7].im - v[7].re), -h(v[7].re + v[7].im)};
#pragma unroll
    for (int q = 0; q < 4; ++q) fft2(v[2 * q], v[2 * q + 1]);
  } else {
    constexpr Fix<S> h(0.70710678118654752440, -4.833646656726457e-17);
    constexpr Fix<S> c(0.92387953251128675613, 1.7645047084336677e-17), mc(-0.92387953251128675613, -1.7645047084336677e-17);
    constexpr Fix<S> s(0.38268343236508977173, -1.0050772696461588e-17), ms(-0.38268343236508977173, 1.0050772696461588e-17);
#pragma unroll
    for (int i = 0; i < 4; ++i) fft4(v[i], v[i + 4], v[i + 8], v[i + 12]);
    v[5] = c2fix(v[5], c, ms);  // cos and sin of pi / 8
    v[9] = C2<S>{h(v[9].re + v[9].im), h(v[9].im - v[9].re)};
    v[13] = c2fix(v[13], s, mc);
    v[6] = C2<S>{h(v[6].re + v[6].im), h(v[6].im - v[6].re)};
    v[10] = C2<S>{v[10].im, -v[10].re};
    v[14] = C2<S>{h(v[14].im - v[14].re), -h(v[14].re + v[14].im)};
    v[7] = c2fix(v[7], s, mc);
    v[11] = C2<S>{h(v[11].im - v[11].re), -h(v[11].re + v[11].im)};
    v[15] = c2fix(v[15], mc, s);
#pragma unroll
    for (int q = 0; q < 4; ++q) fft4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  }
}
template <int R> __device__ __forceinline__ constexpr int fft_at(int k) {
  return R == 16 ? 4 * (k & 3) + (k >> 2) : R == 8 ? 2 * (k & 3) + (k >> 2) : k;
}
// element i of a signal's buffer: one spare element after every 16 keeps the passes' strided writes
// off the same banks
__device__ __forceinline__ int fft_pad(int i) { return i + (i >> 4); }
inline int fft_pad_len(int h) { return h + 1 + ((h + 1) >> 4) + 1; }

// tw[j] = exp(-2 pi i j / n), j < n / 2, in the transform's own type (rounded from FP64).  With
// `count` > n / 2 the radix-16 passes' factors follow in the order in which they are read: for a
// pass after Ns values (Ns = R0, 16 R0, ... < h) the 16 Ns factors exp(-2 pi i r t / (16 Ns)) at
// r Ns + t -- read from tw itself a warp's factors lie in up to 32 lines.
inline int pass_radix0(int L) { return (L & 3) ? 1 << (L & 3) : 16; }
inline int twiddle_count(int n) {  // table entries, pass factors included
  int L = 0;
  while ((2 << L) < n) ++L;
  const int h = n / 2;
  int c = h;
  for (int Ns = pass_radix0(L); Ns < h; Ns <<= 4) c += 16 * Ns;
  return c;
}
__device__ __forceinline__ double2 half_twiddle(int m, int n) {  // exp(-2 pi i m / n)
  double s, c;
  sincospi(2.0 * (double)m / (double)n, &s, &c);
  return make_double2(c, -s);
}
template <class S> __device__ __forceinline__ C2<S> twiddle(const C2<S>* __restrict__ tw, int i, int h) {
  const C2<S> w = tw[i & (h - 1)];  // i < 2 h = n: the second half is the first negated
  return (i & h) ? C2<S>{-w.re, -w.im} : w;
}

// (hi, lo) of a complex value: re hi, re lo, im hi, im lo
__device__ __forceinline__ float4 split_cd(cd v) {
  const ff r = ff_from_double(v.re), i = ff_from_double(v.im);
  return make_float4(r.hi, r.lo, i.hi, i.lo);
}
// a frequency's factors (1 +- i w) of an FP64 value a
__device__ __forceinline__ cd plus_iw(cd a, double2 w) {
  return {fma(-w.x, a.im, fma(-w.y, a.re, a.re)), fma(w.x, a.re, fma(-w.y, a.im, a.im))};
}
__device__ __forceinline__ cd minus_iw(cd a, double2 w) {
  return {fma(w.x, a.im, fma(w.y, a.re, a.re)), fma(-w.x, a.re, fma(w.y, a.im, a.im))};
}
// What a call prepares, in one launch: `count` entries of tw; w64 (unless NULL) [h]; and of `ns` values of
// Sp, spectra [..][h + 1], the factors sp[..][2] = S (1 + i w) / n, S (1 - i w) / n -- for m = 0 and h: S / n, 0.
template <class S>
__global__ void k_synth_tables(int n, int R0, int count, C2<S>* __restrict__ tw, double2* __restrict__ w64,
                               const cd* __restrict__ Sp, int64_t ns, float4* __restrict__ sp) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int h = n / 2;
  if (i < count) {
    int m = (int)i, N = n, at = (int)i - h, Ns = R0;
    while (at >= 16 * Ns) {
      at -= 16 * Ns;
      Ns <<= 4;
    }
    if (at >= 0) {
      m = (at / Ns) * (at % Ns);
      N = 16 * Ns;
    }
    const double2 w = half_twiddle(m, N);
    tw[i] = {(S)w.x, (S)w.y};
    return;
  }
  i -= count;
  if (w64) {
    if (i < h) {
      w64[i] = half_twiddle((int)i, n);
      return;
    }
    i -= h;
  }
  if (i >= ns) return;
  const int m = (int)(i % (h + 1));
  const double inv = 1.0 / n;  // a power of two
  const cd a = {Sp[i].re * inv, Sp[i].im * inv};
  const bool end = m == 0 || m == h;
  const double2 w = half_twiddle(m, n);
  sp[2 * i] = split_cd(end ? a : plus_iw(a, w));
  sp[2 * i + 1] = end ? make_float4(0.f, 0.f, 0.f, 0.f) : split_cd(minus_iw(a, w));
}
// a b - c d or a b + c d from float-float factors, rounded once
__device__ __forceinline__ float ff_dot2(float ah, float al, float bh, float bl, float ch, float cl, float dh, float dl) {
  const float p = __fmul_rn(ah, bh), q = __fmul_rn(ch, dh);
  const float e = __fmaf_rn(ah, bl, __fmaf_rn(al, bh, __fmaf_rn(ah, bh, -p)));
  const float f = __fmaf_rn(ch, dl, __fmaf_rn(cl, dh, __fmaf_rn(ch, dh, -q)));
  const ff t = ff_two_sum(p, q);
  return __fadd_rn(t.hi, __fadd_rn(t.lo, __fadd_rn(e, f)));
}
__device__ __forceinline__ C2<float> ff_cmul(float4 s, float4 t) {
  return {ff_dot2(s.x, s.y, t.x, t.y, -s.z, -s.w, t.z, t.w), ff_dot2(s.x, s.y, t.z, t.w, s.z, s.w, t.x, t.y)};
}

// First pass of radix R0 (inputs Z in buf), then radix-16 passes; the last one leaves
// its outputs in v (output fft_at<16>(r) of butterfly j is z[j + r Ns]).
template <int L, class S>
__device__ __forceinline__ void real_fft(C2<S>* __restrict__ buf, const C2<S>* __restrict__ tw, bool passes, int j,
                                         C2<S>* v) {
  constexpr int h = 1 << L, R0 = (L & 3) ? 1 << (L & 3) : 16, NT = h / 16;
#pragma unroll
  for (int b = 0; b < 16 / R0; ++b)
#pragma unroll
    for (int q = 0; q < R0; ++q) {
      const int k = j + b * NT + q * (h / R0);
      v[b * R0 + q] = buf[fft_pad(k)];
    }
#pragma unroll
  for (int b = 0; b < 16 / R0; ++b) fft_small<R0, S>(v + b * R0);
#pragma unroll
  for (int Ns = R0; Ns < h; Ns <<= 4) {  // (Ns: product of the radices so far)
    const int Np = Ns == R0 ? 1 : Ns >> 4;  // the previous pass's
    __syncthreads();
    if (Ns == R0) {
#pragma unroll
      for (int b = 0; b < 16 / R0; ++b)
#pragma unroll
        for (int r = 0; r < R0; ++r) buf[fft_pad((j + b * NT) * R0 + r)] = v[b * R0 + fft_at<R0>(r)];
    } else {
      const int at = (j / Np) * Np * 16 + (j & (Np - 1));
#pragma unroll
      for (int r = 0; r < 16; ++r) buf[fft_pad(at + r * Np)] = v[fft_at<16>(r)];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = buf[fft_pad(j + r * NT)];
    if (passes) {
      const C2<S>* pw = tw + h + (Ns == R0 ? 0 : 16 * R0 * ((Ns / R0 - 1) / 15)) + (j & (Ns - 1));
#pragma unroll
      for (int r = 1; r < 16; ++r) v[r] = c2mul(v[r], pw[r * Ns]);
    } else {
      const int step = (j & (Ns - 1)) * (2 * h / (Ns * 16));
#pragma unroll
      for (int r = 1; r < 16; ++r) v[r] = c2mul(v[r], twiddle<S>(tw, r * step, h));
    }
    fft_small<16, S>(v);
  }
}

// grid (ceil(M / SB), ceil(P / PG)), block SB h / 16.  Dynamic shared memory: SB fft_pad_len(h)
// values, then (KEEP: PG > 1) the points' T, [nk][SB] as float4 (FP32) or C2<double>.
template <int L, class S, bool KEEP>
__global__ void __launch_bounds__(256, sizeof(S) == 4 ? 3 : 1) k_synth_real(const cd* __restrict__ T, const int64_t* __restrict__ midx, int nk,
                                                    int low, int64_t M, const cd* __restrict__ Sp, const float4* __restrict__ sp,
                                                    const double2* __restrict__ w64, int P, int PG, int SB, const C2<S>* __restrict__ tw, bool passes,
                                                    S* __restrict__ out, int wide) {
  constexpr int h = 1 << L, n = 2 * h, NT = h / 16;
  constexpr bool F32 = sizeof(S) == 4;
  extern __shared__ float4 synth_smem[];
  const int len = h + 1 + ((h + 1) >> 4) + 1;
  C2<S>* bufs = reinterpret_cast<C2<S>*>(synth_smem);
  float4* kept = reinterpret_cast<float4*>(reinterpret_cast<unsigned char*>(synth_smem) +
                                           (((size_t)SB * len * sizeof(C2<S>) + 15) & ~(size_t)15));
  const int tid = threadIdx.x, pt = tid / NT, j = tid - pt * NT;
  const int64_t x0 = (int64_t)blockIdx.x * SB;
  C2<S>* buf = bufs + pt * len;
  if (KEEP)
    for (int e = tid; e < nk * SB; e += SB * NT) {
      const int r = e / SB, q = e - r * SB;
      const cd t = x0 + q < M ? T[(int64_t)r * M + x0 + q] : cd{0.0, 0.0};
      if constexpr (F32) kept[e] = split_cd(t);
      else reinterpret_cast<cd*>(kept)[e] = t;
    }
  const int p1 = min(P, (int)(blockIdx.y + 1) * PG);
  for (int p = blockIdx.y * PG; p < p1; ++p) {
    __syncthreads();  // the kept values; the previous pulse's last reads of the buffers
    for (int e = tid; e < SB * len; e += SB * NT) bufs[e] = {(S)0, (S)0};
    __syncthreads();
    const cd* Srow = Sp + (int64_t)p * (h + 1);
    // the frequencies below h / 2 store their shares of Z_m and Z_{h-m}, then those from h / 2 on add theirs
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      const int e0 = half ? low * SB : 0, e1 = half ? nk * SB : low * SB;
      for (int e = e0 + tid; e < e1; e += SB * NT) {
        const int r = e / SB, q = e - r * SB;
        if (x0 + q >= M) continue;
        const int m = (int)midx[r];
        const bool end = m == 0 || m == h;
        C2<S> za, zb;  // H (1 + i w), H (1 - i w); at the ends H
        bool fp64 = true;
        if constexpr (F32) {
          if (sp) {
            const float4 sa = sp[2 * ((int64_t)p * (h + 1) + m)], sb = sp[2 * ((int64_t)p * (h + 1) + m) + 1];
            float4 t4;
            if (KEEP) t4 = kept[e];
            else t4 = split_cd(T[(int64_t)r * M + x0 + q]);
            za = ff_cmul(sa, t4);
            zb = ff_cmul(sb, t4);
            // outside a safe range of FP32 (zero there, tiny, huge, not finite): the product in FP64
            const float tm = fmaxf(fabsf(t4.x), fabsf(t4.z)), sm = fmaxf(fabsf(sa.x), fabsf(sa.z));
            fp64 = !(tm >= 1e-25f && tm <= 1e25f && sm >= 1e-25f && sm <= 1e25f);
          }
        }
        if (fp64) {
          cd t;
          if constexpr (KEEP && !F32) t = reinterpret_cast<cd*>(kept)[e];
          else t = T[(int64_t)r * M + x0 + q];
          const cd a = cmul(Srow[m], t);
          cd u = a, d = {0.0, 0.0};
          if (!end) {
            const double2 w = w64[m];
            u = plus_iw(a, w);
            d = minus_iw(a, w);
          }
          constexpr S inv = (S)1 / (S)n;
          za = {(S)u.re * inv, (S)u.im * inv};
          zb = {(S)d.re * inv, (S)d.im * inv};
        }
        if (end) za = C2<S>{za.re, m == 0 ? za.re : -za.re};
        C2<S>* z = bufs + q * len;
        C2<S>& lo = z[fft_pad(m == h ? 0 : m)];
        lo = half ? c2add(lo, za) : za;
        if (!end && 2 * m != h) {  // (at h / 2, w = -i: 1 - i w = 0)
          C2<S>& hi = z[fft_pad(h - m)];
          const C2<S> b = {zb.re, -zb.im};
          hi = half ? c2add(hi, b) : b;
        }
      }
      __syncthreads();
    }
    C2<S> v[16];
    real_fft<L, S>(buf, tw, passes, j, v);
    if (x0 + pt < M) {
      S* o = out + ((int64_t)p * M + x0 + pt) * n;
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const C2<S> z = v[fft_at<16>(r)];
        const int i = 2 * (j + r * NT);
        if (wide) {  // the output is aligned to pairs
          if constexpr (F32) *reinterpret_cast<float2*>(o + i) = make_float2(z.re, z.im);
          else *reinterpret_cast<double2*>(o + i) = make_double2(z.re, z.im);
        } else {
          o[i] = z.re;
          o[i + 1] = z.im;
        }
      }
    }
  }
}

// Whether `signals` of n samples take the radix-2 kernel: fewer than 32 samples, which k_synth_real does not
// hold, or so few short ones that the latency of one signal counts: with 16 values a thread its warps take
// longer than radix 2 over n / 2 threads.  400 signals of 64 samples, the kernel: 5.4 us here, 9.5 there (FP64
// 6.7 and 20.2); of 512 samples 9.3 and 10.6 (21.7 and 27.9); one of 1024 and more is no faster here.
static bool synth_radix2(int n, int64_t signals, int nsm) { return n < 32 || (n <= 512 && signals <= 4 * nsm); }

// Tables of a transform of n samples (k_synth_tables): tw, with the pass factors too if `passes`; for the
// radix-2 kernel FP64 pairs in tw and nothing else.
template <class S>
static void launch_tables(int n, bool radix2, void* tw, bool passes, double2* w64, const cd* Sp, int64_t ns, float4* sp,
                          cudaStream_t st) {
  if (radix2) {
    if (tw) BIE_LAUNCH(k_twiddles<<<(n / 2 + 255) / 256, 256, 0, st>>>(n, (double2*)tw));
    return;
  }
  int L = 0;
  while ((2 << L) < n) ++L;
  const int count = !tw ? 0 : passes ? twiddle_count(n) : n / 2;
  const int64_t all = count + (w64 ? n / 2 : 0) + ns;
  BIE_LAUNCH(k_synth_tables<S><<<(unsigned)((all + 127) / 128), 128, 0, st>>>(n, pass_radix0(L), count, (C2<S>*)tw, w64, Sp, ns, sp));
}

// low: how many of the frequencies lie below h / 2 = n / 4; sp: the spectra's factors in float-float
// (k_synth_tables; FP32 only; NULL: products in FP64); w64: exp(-2 pi i m / n), m < n / 2, in FP64.
template <class S>
static int launch_synth(const cd* T, const int64_t* midx, int nk, int low, int64_t M, const cd* Sp, const float4* sp,
                        const double2* w64, int64_t P, int n, bool radix2, const void* tw, bool passes, S* out, int nsm,
                        cudaStream_t st) {
  if (radix2) {
    const dim3 g((unsigned)M, (unsigned)P);
    const size_t smem = 2 * (size_t)n * sizeof(C2<S>);
    BIE_LAUNCH(k_synth<S, S><<<g, std::max(32, n / 2), smem, st>>>(T, midx, nk, M, Sp, n, (const double2*)tw, out));
    return BIE_OK;
  }
  const int h = n / 2, wide = ((uintptr_t)out % (2 * sizeof(S))) == 0;
  // points per CTA: 256 threads' worth, fewer (down to a warp, or two points for whole sectors of T)
  // while the signals would not give every SM two CTAs
  int SB = 4096 / h;
  while (SB > 2 && SB * (h / 16) > 32 && (M + SB - 1) / SB * P < 2 * nsm) SB >>= 1;
  const int64_t bx = (M + SB - 1) / SB;
  if (bx > 0x7fffffff) return fail(BIE_ERR_INVALID_ARG, "too many observation points");
  const size_t bufs = ((size_t)SB * fft_pad_len(h) * sizeof(C2<S>) + 15) & ~(size_t)15;
  const size_t kept = (size_t)nk * SB * 16;
  // Pulses per CTA: all, with T kept, once the points alone give every SM a few CTAs; else one
  // (more CTAs; T is read once per pulse).  The kept T must leave room for two CTAs.
  const bool keep = P > 1 && bx >= 4 * nsm && bufs + kept <= 100 * 1024;
  const int PG = keep ? (int)P : 1;
  const dim3 g((unsigned)bx, (unsigned)(keep ? 1 : P));
  auto go = [&](auto kernel) -> int {
    BIE_TRY(set_smem_max(kernel));
    BIE_LAUNCH(kernel<<<g, SB * (h / 16), bufs + (keep ? kept : 0), st>>>(T, midx, nk, low, M, Sp, sp, w64, (int)P, PG, SB,
                                                                          (const C2<S>*)tw, passes, out, wide));
    return BIE_OK;
  };
  switch (h) {
#define BIE_SYNTH(L) \
  case 1 << L: return keep ? go(k_synth_real<L, S, true>) : go(k_synth_real<L, S, false>)
    BIE_SYNTH(4);
    BIE_SYNTH(5);
    BIE_SYNTH(6);
    BIE_SYNTH(7);
    BIE_SYNTH(8);
    BIE_SYNTH(9);
    BIE_SYNTH(10);
    BIE_SYNTH(11);
#undef BIE_SYNTH
  }
  return fail(BIE_ERR_INVALID_ARG, "Nt out of range");
}

static int twiddle_table(bie_ctx* c, int n, double2** tw) {
  BIE_TRY(ensure_buf(c, c->work2, (size_t)(n / 2 + 1) * sizeof(double2)));
  *tw = (double2*)c->work2.p;
  BIE_LAUNCH(k_twiddles<<<(n / 2 + 255) / 256, 256, 0, c->stream>>>(n, *tw));
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int pulse_spectrum(bie_ctx* c, const double* s, int64_t P, int n, cd* Sout) {
  double2* tw;
  BIE_TRY(twiddle_table(c, n, &tw));
  size_t smem = 2 * (size_t)n * sizeof(C2<double>);
  BIE_TRY((set_smem_max(k_pulse_spectrum<double>)));
  BIE_LAUNCH(k_pulse_spectrum<double><<<(unsigned)P, std::min(512, n / 2), smem, c->stream>>>(s, n, tw, Sout));
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

// Frequencies below a quarter of n samples in the ascending host list midx.
int low_frequencies(const int64_t* midx, int64_t nk, int64_t n) {
  return (int)(std::lower_bound(midx, midx + nk, (n + 3) / 4) - midx);
}

int synthesize(bie_ctx* c, const cd* T, const int64_t* midx_dev, int nk, int low, int64_t M, const cd* Sp, int64_t P, int n,
               void* out, int out_dtype) {
  // twiddles (at most FP64 pairs; FP32: theirs and FP64 ones), then the spectra in float-float (FP32), of so
  // many pulses at a time that they stay within 32 MB (511 pulses of 4096 samples)
  const size_t twb = (size_t)(twiddle_count(n) + n / 2 + 16) * sizeof(double2);
  const int64_t nm = n / 2 + 1;
  const bool f32 = out_dtype != 0;
  const int64_t pc = f32 ? std::min(P, std::max<int64_t>(1, (int64_t)(32 << 20) / (nm * 2 * (int64_t)sizeof(float4)))) : P;
  BIE_TRY(ensure_buf(c, c->work2, twb + (f32 ? (size_t)(2 * pc * nm) * sizeof(float4) : 0)));
  void* tw = c->work2.p;
  int nsm = 0;
  BIE_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device));
  const bool radix2 = synth_radix2(n, P * M, nsm);
  if (f32) {
    float4* sp = (float4*)((char*)tw + twb);
    double2* w64 = (double2*)tw + twiddle_count(n) + 16;
    for (int64_t p0 = 0; p0 < P; p0 += pc) {
      const int64_t np = std::min(pc, P - p0);
      const cd* S0 = Sp + p0 * nm;
      launch_tables<float>(n, radix2, p0 == 0 ? tw : nullptr, true, p0 == 0 ? w64 : nullptr, S0, np * nm, sp, c->stream);
      BIE_TRY(launch_synth<float>(T, midx_dev, nk, low, M, S0, sp, w64, np, n, radix2, tw, true, (float*)out + p0 * M * n, nsm, c->stream));
    }
  } else {
    launch_tables<double>(n, radix2, tw, true, nullptr, nullptr, 0, nullptr, c->stream);
    BIE_TRY(launch_synth<double>(T, midx_dev, nk, low, M, Sp, nullptr, (const double2*)tw, P, n, radix2, tw, true, (double*)out, nsm, c->stream));
  }
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

// ------------------------------------------------------------------------------------------
// Dominant frequencies (Sec. 4, Table I; Sec. 5): the space-time field is accurate already from
// the wavenumbers at which the incident spectrum is largest, so only those need a frequency
// solve.  One CTA ranks m = 0 .. nm-1 by max over the pulses of |S[p][m]|^2 (ties: the lower m
// first) with a bitonic sort in shared memory, keeps the first K and sorts them ascending.
// ------------------------------------------------------------------------------------------
constexpr int kTopMax = 4096;  // padded sort length (nm = Nt/2 + 1 <= 2049)

__global__ void __launch_bounds__(1024) k_top_frequencies(const cd* __restrict__ S, int64_t P, int nm, int K,
                                                          int64_t* __restrict__ midx_out) {
  extern __shared__ unsigned char smem_raw[];
  double* key = reinterpret_cast<double*>(smem_raw);     // [kTopMax]
  int32_t* idx = reinterpret_cast<int32_t*>(key + kTopMax);  // [kTopMax]
  int L = 1;
  while (L < nm) L <<= 1;
  for (int m = threadIdx.x; m < L; m += blockDim.x) {
    double a = -1.0;  // padding sorts last
    if (m < nm) {
      a = 0.0;
      for (int64_t p = 0; p < P; ++p) {
        const cd v = S[p * nm + m];
        a = fmax(a, v.re * v.re + v.im * v.im);
      }
    }
    key[m] = a;
    idx[m] = m;
  }
  __syncthreads();
  // descending by key, ascending by index on ties
  for (int size = 2; size <= L; size <<= 1)
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int t = threadIdx.x; t < L / 2; t += blockDim.x) {
        const int i = 2 * t - (t & (stride - 1)), j = i + stride;
        const bool up = (i & size) == 0;  // this run ends in the wanted order
        const bool j_first = key[j] > key[i] || (key[j] == key[i] && idx[j] < idx[i]);
        if (j_first == up) {
          const double tk = key[i]; key[i] = key[j]; key[j] = tk;
          const int32_t ti = idx[i]; idx[i] = idx[j]; idx[j] = ti;
        }
      }
      __syncthreads();
    }
  // the K selected indices in ascending order
  int LK = 1;
  while (LK < K) LK <<= 1;
  for (int t = threadIdx.x; t < LK; t += blockDim.x) key[t] = t < K ? (double)idx[t] : 1e300;
  __syncthreads();
  for (int size = 2; size <= LK; size <<= 1)
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int t = threadIdx.x; t < LK / 2; t += blockDim.x) {
        const int i = 2 * t - (t & (stride - 1)), j = i + stride;
        const bool up = (i & size) == 0;
        if ((key[j] < key[i]) == up) {
          const double tk = key[i]; key[i] = key[j]; key[j] = tk;
        }
      }
      __syncthreads();
    }
  for (int t = threadIdx.x; t < K; t += blockDim.x) midx_out[t] = (int64_t)key[t];
}

int top_frequencies(bie_ctx* c, const cd* S, int64_t P, int nm, int K, int64_t* midx_dev) {
  if (nm > kTopMax) return fail(BIE_ERR_INVALID_ARG, "too many frequencies to rank");
  const size_t smem = kTopMax * (sizeof(double) + sizeof(int32_t));
  BIE_TRY((set_smem_max(k_top_frequencies)));
  BIE_LAUNCH(k_top_frequencies<<<1, 1024, smem, c->stream>>>(S, P, nm, K, midx_dev));
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

// ------------------------------------------------------------------------------------------
// Allocation-free synthesis.  Some callers cannot allocate device memory while they run: a host
// framework that hands out a fixed device-memory budget through its own pool, or a latency-bound
// pipeline in which cudaMalloc/cudaFree would synchronise the device.  For them the synthesis's
// scratch (the FFT twiddle table and the device copy of the frequency indices) lives in one
// file-scope device array instead of context buffers, and no context is needed.
// ------------------------------------------------------------------------------------------
constexpr size_t kNoAllocScratchBytes = 64 * 1024;  // FP64 twiddles <= 32 KB (Nt <= 4096) + indices <= 32 KB
constexpr size_t kNoAllocTwiddle32Bytes = 16 * 1024;  // and the FP32 ones
constexpr int kNoAllocMaxDevices = 64;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes + kNoAllocTwiddle32Bytes];
static std::mutex g_noalloc_mu;
static void* g_noalloc_ptr[kNoAllocMaxDevices] = {};

// Device address of the array on the current device, looked up once per device (the host-side
// name of a __device__ variable is not a device address).
static int noalloc_scratch(void** out) {
  int dev = 0;
  BIE_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kNoAllocMaxDevices) return fail(BIE_ERR_INVALID_ARG, "device index too large");
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) return cuda_fail(e == cudaSuccess ? cudaErrorInvalidSymbol : e, "cudaGetSymbolAddress");
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return BIE_OK;
}

}  // namespace bie

extern "C" int bie_synthesize_noalloc(const void* T, const int64_t* midx, int64_t Nk, int64_t M, const void* S,
                                      int64_t P, int64_t Nt, void* out, int out_dtype, void* stream) {
  using namespace bie;
  if (P < 0 || M < 0 || Nk < 0 || Nt < 2 || Nt > 4096 || (Nt & (Nt - 1)))
    return fail(BIE_ERR_INVALID_ARG, "need P, M, Nk >= 0 and Nt a power of two in [2, 4096]");
  if (out_dtype != 0 && out_dtype != 1) return fail(BIE_ERR_INVALID_ARG, "out_dtype must be 0 (f64) or 1 (f32)");
  if (P > 65535) return fail(BIE_ERR_INVALID_ARG, "P > 65535");
  if ((size_t)Nk * sizeof(int64_t) > kNoAllocScratchBytes / 2)
    return fail(BIE_ERR_INVALID_ARG, "Nk = " + std::to_string(Nk) + " exceeds the fixed scratch (at most " +
                                         std::to_string(kNoAllocScratchBytes / 2 / sizeof(int64_t)) + ")");
  if (P == 0 || M == 0) return BIE_OK;
  if ((Nk > 0 && (!T || !midx)) || !S || !out) return fail(BIE_ERR_INVALID_ARG, "NULL pointer");
  for (int64_t r = 0; r < Nk; ++r) {
    if (midx[r] < 0 || midx[r] > Nt / 2) return fail(BIE_ERR_INVALID_ARG, "midx out of [0, Nt/2]");
    if (r > 0 && midx[r] <= midx[r - 1]) return fail(BIE_ERR_INVALID_ARG, "midx must be strictly increasing");
  }
  const int low = low_frequencies(midx, Nk, Nt);
  void* base = nullptr;
  BIE_TRY(noalloc_scratch(&base));
  cudaStream_t st = (cudaStream_t)stream;
  const int n = (int)Nt;
  double2* tw = (double2*)base;  // n/2 entries, rewritten by every call
  int64_t* md = (int64_t*)((char*)base + kNoAllocScratchBytes / 2);
  if (Nk > 0) BIE_CUDA_TRY(cudaMemcpyAsync(md, midx, Nk * sizeof(int64_t), cudaMemcpyHostToDevice, st));
  int dev = 0, nsm = 0;
  BIE_CUDA_TRY(cudaGetDevice(&dev));
  BIE_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const bool radix2 = synth_radix2(n, P * M, nsm);
  if (out_dtype == 0) {
    launch_tables<double>(n, radix2, tw, false, nullptr, nullptr, 0, nullptr, st);
    BIE_TRY(launch_synth<double>((const cd*)T, md, (int)Nk, low, M, (const cd*)S, nullptr, tw, P, n, radix2, tw, false, (double*)out, nsm, st));
  } else {
    void* tw32 = (char*)base + kNoAllocScratchBytes;
    if (radix2) tw32 = tw;
    launch_tables<float>(n, radix2, tw32, false, tw, nullptr, 0, nullptr, st);
    BIE_TRY(launch_synth<float>((const cd*)T, md, (int)Nk, low, M, (const cd*)S, nullptr, tw, P, n, radix2, tw32, false, (float*)out, nsm, st));
  }
  BIE_CUDA_TRY(cudaGetLastError());
  // the host index array must outlive its asynchronous copy
  BIE_CUDA_TRY(cudaStreamSynchronize(st));
  return BIE_OK;
}
