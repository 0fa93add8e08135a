// lu.cu -- batched dense complex LU with partial pivoting and triangular solves (the direct solver
// of Sec. 4), right-looking and blocked:
//   for each panel of width nb:  factor the panel (pivot = largest modulus, lowest row on ties),
//   apply its row swaps to the other columns, U12 = L11^{-1} A12, A22 -= L21 U12.
// Matrices are row-major with leading dimension ld, batched with stride `bstride` elements.
// This file holds the panel, swap/TRSM and SIMT-GEMM kernels in FP64 and FP32; the tensor-core
// (tcgen05, TF32) trailing update lives in lu_tc.cu.
#include "bie_common.cuh"

namespace bie {

template <class S> struct Cx { S re, im; };
template <class S> __device__ __forceinline__ Cx<S> cx_mul(Cx<S> a, Cx<S> b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <class S> __device__ __forceinline__ Cx<S> cx_div(Cx<S> a, Cx<S> b) {
  S d = b.re * b.re + b.im * b.im;
  return {(a.re * b.re + a.im * b.im) / d, (a.im * b.re - a.re * b.im) / d};
}

// a -= l u: in FP32 rounded as the one-CTA leaf does, in FP64 every product fused (four instructions of
// the narrow FP64 pipe instead of six).
__device__ __forceinline__ void cx_msub(Cx<float>& a, Cx<float> l, Cx<float> u) {
  a.re -= l.re * u.re - l.im * u.im;
  a.im -= l.re * u.im + l.im * u.re;
}
__device__ __forceinline__ void cx_msub(Cx<double>& a, Cx<double> l, Cx<double> u) {
  a.re = fma(-l.re, u.re, fma(l.im, u.im, a.re));
  a.im = fma(-l.re, u.im, fma(-l.im, u.re, a.im));
}

// x / d from y = 1 / d: one correction of the rounded product by its residual (Markstein's division), the
// quotient rounded once as by a division; plain division where the residual could leave FP64's range.
__device__ __forceinline__ bool quotient_safe(double d) { return d >= 0x1p-900 && d <= 0x1p900; }
__device__ __forceinline__ double quotient(double x, double d, double y, bool safe) {
  if (!safe) return x / d;
  const double q = x * y;
  return fma(fma(-q, d, x), y, q);
}
__device__ __forceinline__ Cx<double> cx_div_by(Cx<double> a, Cx<double> b, double bb, double y, bool safe) {  // bb = |b|^2
  return {quotient(fma(a.re, b.re, a.im * b.im), bb, y, safe), quotient(fma(a.im, b.re, -(a.re * b.im)), bb, y, safe)};
}

// ---- panel factorisation: one CTA per matrix, columns p0 .. p0+nb-1, rows p0 .. n-1 ----------
template <class S>
__global__ void __launch_bounds__(512) k_panel(Cx<S>* __restrict__ A, int64_t bstride, int n, int ld, int p0,
                                               int nb, int32_t* __restrict__ piv, int32_t* __restrict__ info) {
  Cx<S>* M = A + (int64_t)blockIdx.x * bstride;
  int32_t* pv = piv + (int64_t)blockIdx.x * n;
  __shared__ S red_v[32];
  __shared__ int red_i[32];
  __shared__ int s_piv;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int pend = min(p0 + nb, n);
  for (int c = p0; c < pend; ++c) {
    // pivot: largest |a_rc|^2 over r >= c, lowest row on ties
    S best = -1;
    int bi = n;
    for (int r = c + tid; r < n; r += nt) {
      Cx<S> v = M[(int64_t)r * ld + c];
      S m = v.re * v.re + v.im * v.im;
      if (m > best) { best = m; bi = r; }
    }
    for (int o = 16; o > 0; o >>= 1) {
      S ob = __shfl_xor_sync(0xffffffffu, best, o);
      int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    if (lane == 0) { red_v[warp] = best; red_i[warp] = bi; }
    __syncthreads();
    if (warp == 0) {
      best = lane < nw ? red_v[lane] : (S)-1;
      bi = lane < nw ? red_i[lane] : n;
      for (int o = 16; o > 0; o >>= 1) {
        S ob = __shfl_xor_sync(0xffffffffu, best, o);
        int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (lane == 0) {
        s_piv = bi;
        pv[c] = bi;
        if (!(best > 0) && info) atomicOr(info + blockIdx.x, 1);
      }
    }
    __syncthreads();
    const int p = s_piv;
    if (p != c && p < n)  // swap rows c and p inside the panel columns
      for (int j = p0 + tid; j < pend; j += nt) {
        Cx<S> t = M[(int64_t)c * ld + j];
        M[(int64_t)c * ld + j] = M[(int64_t)p * ld + j];
        M[(int64_t)p * ld + j] = t;
      }
    __syncthreads();
    const Cx<S> d = M[(int64_t)c * ld + c];
    const bool ok = (d.re != 0 || d.im != 0);
    // scale the column and update the rest of the panel (rank-1), one row per thread
    for (int r = c + 1 + tid; r < n; r += nt) {
      Cx<S> l = M[(int64_t)r * ld + c];
      if (ok) l = cx_div(l, d);
      M[(int64_t)r * ld + c] = l;
      for (int j = c + 1; j < pend; ++j) {
        Cx<S> u = M[(int64_t)c * ld + j];
        Cx<S> a = M[(int64_t)r * ld + j];
        a.re -= l.re * u.re - l.im * u.im;
        a.im -= l.re * u.im + l.im * u.re;
        M[(int64_t)r * ld + j] = a;
      }
    }
    __syncthreads();
  }
}

// ---- leaf-recursive panel: a leaf of `lw` columns factored in shared memory ------------------
// One CTA (1024 threads) per matrix holds rows c0..n-1 of columns c0..c0+lw-1, factors them with
// partial pivoting (largest modulus, lowest row on ties), writes them back, applies the leaf's
// row swaps to the other columns of the panel [p0, p0+w) and solves the leaf's U block for the
// panel columns right of the leaf, then updates the panel columns right of the leaf in the rows
// below it.  The leaf is stored column by column in shared memory (element (r, c) at
// c * rows + r), so that threads walking the rows touch consecutive words.
template <class S>
__global__ void __launch_bounds__(1024) k_leaf(Cx<S>* __restrict__ A, int64_t bstride, int n, int ld, int p0, int w,
                                               int c0, int lw, int32_t* __restrict__ piv, int32_t* __restrict__ info,
                                               int fuse) {
  extern __shared__ unsigned char smem_raw[];
  Cx<S>* L = reinterpret_cast<Cx<S>*>(smem_raw);  // [lw][rows]
  __shared__ S red_v[32];
  __shared__ int red_i[32];
  __shared__ int s_piv[16];
  Cx<S>* M = A + (int64_t)blockIdx.x * bstride;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int rows = n - c0;
  // global-memory loops are unrolled so that several loads per thread are in flight
  // 16-byte accesses need an even element index: even ld, batch stride, c0 and leaf width (the
  // last also keeps the U block below, at element rows * lw of the shared array, 16-byte aligned)
  const bool pairs = sizeof(S) == 4 && ((ld | bstride | c0 | lw) & 1) == 0;
  if (pairs) {  // FP32: 16-byte loads of column pairs
    const int hl = lw >> 1;
#pragma unroll 4
    for (int t = tid; t < rows * hl; t += nt) {
      const int r = t / hl, c = 2 * (t - r * hl);
      const float4 v = *reinterpret_cast<const float4*>(&M[(int64_t)(c0 + r) * ld + c0 + c]);
      L[c * rows + r] = Cx<S>{(S)v.x, (S)v.y};
      L[(c + 1) * rows + r] = Cx<S>{(S)v.z, (S)v.w};
    }
  } else {
#pragma unroll 4
    for (int t = tid; t < rows * lw; t += nt) {
      const int r = t / lw, c = t - r * lw;
      L[c * rows + r] = M[(int64_t)(c0 + r) * ld + c0 + c];
    }
  }
  __syncthreads();
  for (int c = 0; c < lw; ++c) {
    S best = -1;
    int bi = rows;
    for (int r = c + tid; r < rows; r += nt) {
      const Cx<S> v = L[c * rows + r];
      const S m = v.re * v.re + v.im * v.im;
      if (m > best) { best = m; bi = r; }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const S ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    if (lane == 0) { red_v[warp] = best; red_i[warp] = bi; }
    __syncthreads();
    if (warp == 0) {
      best = lane < nw ? red_v[lane] : (S)-1;
      bi = lane < nw ? red_i[lane] : rows;
      for (int o = 16; o > 0; o >>= 1) {
        const S ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (lane == 0) {
        if (bi >= rows) bi = c;
        s_piv[c] = bi;
        piv[(int64_t)blockIdx.x * n + c0 + c] = c0 + bi;
        if (!(best > 0) && info) atomicOr(info + blockIdx.x, 1);
      }
    }
    __syncthreads();
    const int p = s_piv[c];
    if (p != c && tid < lw) {
      const Cx<S> t = L[tid * rows + c];
      L[tid * rows + c] = L[tid * rows + p];
      L[tid * rows + p] = t;
    }
    __syncthreads();
    const Cx<S> d = L[c * rows + c];
    const bool ok = (d.re != 0 || d.im != 0);
    for (int r = c + 1 + tid; r < rows; r += nt) {
      Cx<S> l = L[c * rows + r];
      if (ok) l = cx_div(l, d);
      L[c * rows + r] = l;
      for (int j = c + 1; j < lw; ++j) {
        const Cx<S> u = L[j * rows + c];
        Cx<S> a = L[j * rows + r];
        a.re -= l.re * u.re - l.im * u.im;
        a.im -= l.re * u.im + l.im * u.re;
        L[j * rows + r] = a;
      }
    }
    __syncthreads();
  }
  for (int t = tid; t < rows * lw; t += nt) {
    const int r = t / lw, c = t - r * lw;
    M[(int64_t)(c0 + r) * ld + c0 + c] = L[c * rows + r];
  }
  // other panel columns: their rows c0 .. c0+lw-1 are staged in shared memory (X, [lw][wall]),
  // where each column's thread applies the leaf's swaps in order (rows below the leaf are swapped
  // in global memory) and solves the U block right of the leaf; then X is written back.  The
  // dependent chains of a column run on shared memory, not on global-memory round trips.
  const int pend = min(p0 + w, n);
  const int wall = pend - p0;
  Cx<S>* X = L + (size_t)rows * lw;  // [lw][wall]
  for (int t = tid; t < lw * wall; t += nt) {
    const int s = t / wall, jj = t - s * wall, j = p0 + jj;
    if (j >= c0 && j < c0 + lw) continue;
    X[t] = M[(int64_t)(c0 + s) * ld + j];
  }
  __syncthreads();
  for (int jj = tid; jj < wall; jj += nt) {
    const int j = p0 + jj;
    if (j >= c0 && j < c0 + lw) continue;
    for (int s = 0; s < lw; ++s) {
      const int p = s_piv[s];  // leaf-relative row, p >= s
      if (p != s) {
        const Cx<S> t = X[s * wall + jj];
        if (p < lw) {
          X[s * wall + jj] = X[p * wall + jj];
          X[p * wall + jj] = t;
        } else {
          Cx<S>& g = M[(int64_t)(c0 + p) * ld + j];
          X[s * wall + jj] = g;
          g = t;
        }
      }
    }
    if (j >= c0 + lw)
      for (int s = 1; s < lw; ++s) {
        Cx<S> v = X[s * wall + jj];
        for (int t = 0; t < s; ++t) {
          const Cx<S> l = L[t * rows + s];
          const Cx<S> xt = X[t * wall + jj];
          v.re -= l.re * xt.re - l.im * xt.im;
          v.im -= l.re * xt.im + l.im * xt.re;
        }
        X[s * wall + jj] = v;
      }
    for (int s = 0; s < lw; ++s) M[(int64_t)(c0 + s) * ld + j] = X[s * wall + jj];
  }
  // rows below the leaf, panel columns right of it: A -= L_leaf U_leaf, with the leaf's L and its
  // just-solved U block (in X) from shared memory; consecutive threads take consecutive columns
  // of a row (coalesced read-modify-write)
  const int cs = c0 + lw, wr = pend - cs;
  if (fuse && wr > 0 && rows > lw) {
    __syncthreads();  // every column's U block is complete in X
    const Cx<S>* U = X + (cs - p0);  // U[s * wall + j]: row c0 + s, column cs + j
    if (pairs && (wr & 1) == 0 && (wall & 1) == 0) {  // cs = c0 + lw and cs - p0 are even too
      // FP32: a thread takes two adjacent columns (one 16-byte load and store), several in flight
      const int hw = wr >> 1;
#pragma unroll 4
      for (int t = tid; t < (rows - lw) * hw; t += nt) {
        const int rr = t / hw, j = 2 * (t - rr * hw), r = lw + rr;
        float4* mp = reinterpret_cast<float4*>(&M[(int64_t)(c0 + r) * ld + cs + j]);
        float4 a = *mp;
        for (int s2 = 0; s2 < lw; ++s2) {
          const Cx<S> l = L[s2 * rows + r];
          const float4 u = *reinterpret_cast<const float4*>(&U[s2 * wall + j]);
          a.x -= l.re * u.x - l.im * u.y;
          a.y -= l.re * u.y + l.im * u.x;
          a.z -= l.re * u.z - l.im * u.w;
          a.w -= l.re * u.w + l.im * u.z;
        }
        *mp = a;
      }
    } else {
#pragma unroll 4
      for (int t = tid; t < (rows - lw) * wr; t += nt) {
        const int rr = t / wr, j = t - rr * wr, r = lw + rr;
        Cx<S>& m = M[(int64_t)(c0 + r) * ld + cs + j];
        Cx<S> a = m;
        for (int s2 = 0; s2 < lw; ++s2) {
          const Cx<S> l = L[s2 * rows + r], u = U[s2 * wall + j];
          a.re -= l.re * u.re - l.im * u.im;
          a.im -= l.re * u.im + l.im * u.re;
        }
        m = a;
      }
    }
  }
}

// Rows below the leaf, panel columns right of it: A -= L_leaf U_leaf (K = lw <= 16), as its own
// launch for small batches (the leaf kernel has one CTA per matrix).  One warp per row, lanes over the (<= 64) columns so that the read-modify-write of A coalesces;
// the row's lw entries of L are broadcast.  grid (any, batch), block 256: 8 warps, a row each at a time.
template <class S>
__global__ void __launch_bounds__(256) k_leaf_update(Cx<S>* __restrict__ A, int64_t bstride, int n, int ld, int p0,
                                                     int w, int c0, int lw) {
  __shared__ Cx<S> U[16 * 64];
  Cx<S>* M = A + (int64_t)blockIdx.y * bstride;
  const int cs = c0 + lw, ce = min(p0 + w, n), wr = ce - cs;
  if (wr <= 0) return;
  for (int t = threadIdx.x; t < lw * wr; t += blockDim.x) {
    const int s = t / wr, j = t - s * wr;
    U[s * 64 + j] = M[(int64_t)(c0 + s) * ld + cs + j];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int r = c0 + lw + blockIdx.x * 8 + warp; r < n; r += gridDim.x * 8) {
    const Cx<S>* lrow = M + (int64_t)r * ld + c0;
    Cx<S> l[16];
#pragma unroll
    for (int s = 0; s < 16; ++s)
      if (s < lw) l[s] = lrow[s];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = lane + 32 * h;
      if (j < wr) {
        S ar = 0, ai = 0;
#pragma unroll
        for (int s = 0; s < 16; ++s)
          if (s < lw) {
            const Cx<S> u = U[s * 64 + j];
            if constexpr (sizeof(S) == 4) {
              ar += l[s].re * u.re - l[s].im * u.im;
              ai += l[s].re * u.im + l[s].im * u.re;
            } else {
              ar = fma(l[s].re, u.re, fma(-l[s].im, u.im, ar));
              ai = fma(l[s].re, u.im, fma(l[s].im, u.re, ai));
            }
          }
        Cx<S>& m = M[(int64_t)r * ld + cs + j];
        m.re -= ar;
        m.im -= ai;
      }
    }
  }
}

// ---- cluster panel: one panel of each matrix by a thread-block cluster ------------------------
// The CTAs of a cluster (up to 16) share a matrix: CTA j holds rows [p0 + j ch, p0 + (j + 1) ch)
// of a leaf of up to 16 columns in shared memory, column by column.  Per column each CTA finds its best
// candidate row (largest modulus, lowest row on ties) during the rank-1 update of the column before,
// one warp stores the candidate and its leaf entries (the holder of row c also row c's) into every
// CTA's shared memory, and one cluster barrier later every warp picks the same winner p from its own
// copy; the holders of rows c and p exchange them, every CTA scales column c of its rows and applies
// the rank-1 update.  The records of consecutive columns alternate between two buffers: a CTA stores
// column c + 2's only after the barrier of column c + 1, at which every CTA has read column c's.
// After a leaf, CTA 0 (its chunk holds the panel's diagonal rows: ch >= 64) applies the leaf's
// interchanges, as one gather of the at most 32 rows they touch, to the panel's other columns and
// solves the leaf's U block L11^{-1} A12 for the panel columns right of the leaf; one barrier later
// every CTA updates its rows of those columns, A -= L U.  Global data written by another CTA of the
// cluster is read with L2-coherent loads after a cluster barrier (release / acquire).
// Bound: the latency of a column (a CTA barrier, the remote stores, a cluster barrier); in FP64 the
// rows' FP64 instructions.  N = 2884, two systems in FP64: 72.6 ms of one-CTA leaves and their updates ->
// 17.1 ms, the panels' other columns updated over all SMs (29.3 ms inside the cluster).
// The pivots and the factor do not depend on the cluster.  In FP32 every entry goes through the operations of
// the one-CTA leaf (k_leaf) in its order, so that for panels of up to 1536 rows (leaf, where that kernel
// takes 16 columns) the factor is its bit for bit; in FP64 the pivots are chosen as there, the products
// fused.  sum_first: A -= (sum of L U), as k_leaf_update forms it
// for small batches, instead of product by product.  (Taller panels of small batches fix the other
// order of the U block's fused products, leaf 0.)  The refinement's result moves by up to 1e-9 with
// the factor's rounding: which of the forms a panel takes depends on the batch, the rows and the
// number of SMs alone (panel_cluster), not on the cluster; so does the width of the leaves.
// The key of a candidate is |a|^2's bits plus one, 0 for none.  In FP64 the record also carries 1 / |a|^2, formed
// by the candidate's warp alone (every warp of every CTA would take the division's FP64 instructions
// otherwise); the quotients take one correction each and round once.  Two FP64 solves of N = 2884 in all:
// 72.1 ms with the keys' upper halves alone and 1 / |a|^2 by every warp, 69.0 this way.
namespace pcl {
constexpr int NT = 512, LW = 16, PW = 64, MAXC = 16;
template <class S> struct alignas(16) RecHead {
  unsigned long long head;  // key << 32 | row
};
template <> struct alignas(16) RecHead<double> {
  unsigned long long head, row;  // key; row
  double inv, mag;               // 1 / |a|^2, |a|^2
};
template <class S> struct alignas(16) Rec : RecHead<S> {
  alignas(16) Cx<S> v[LW];  // the candidate's leaf entries
};
template <class S> __host__ __device__ constexpr size_t smem_bytes(int lw, int ch) {
  // leaf, gathered rows of the other columns (32 x 64), U block (16 x 64)
  return ((size_t)lw * ch + 2 * LW * PW + LW * PW) * sizeof(Cx<S>);
}
__device__ __forceinline__ unsigned key_of(float m) { return __float_as_uint(m) + 1u; }
__device__ __forceinline__ unsigned long long key_of(double m) { return (unsigned long long)__double_as_longlong(m) + 1ull; }
__device__ __forceinline__ unsigned warp_max(unsigned k) { return __reduce_max_sync(0xffffffffu, k); }
__device__ __forceinline__ unsigned long long warp_max(unsigned long long k) {
  const unsigned hi = (unsigned)(k >> 32), H = __reduce_max_sync(0xffffffffu, hi);
  return ((unsigned long long)H << 32) | __reduce_max_sync(0xffffffffu, hi == H ? (unsigned)k : 0u);
}
template <class S> struct KeyOf { typedef unsigned type; };
template <> struct KeyOf<double> { typedef unsigned long long type; };
__device__ __forceinline__ uint32_t mapa(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_remote(uint32_t a, unsigned long long v) {
  asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t a, Cx<float> v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.re), "f"(v.im) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t a, Cx<double> v) {
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.re), "d"(v.im) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ Cx<float> ldcg(const Cx<float>* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return {v.x, v.y};
}
__device__ __forceinline__ Cx<double> ldcg(const Cx<double>* p) {
  return {__ldcg(&p->re), __ldcg(&p->im)};
}
}  // namespace pcl


template <class S>
__global__ void __launch_bounds__(pcl::NT, 1) k_panel_cluster(Cx<S>* __restrict__ A, int64_t bstride, int n, int ld,
                                                              int p0, int w, int c_lo, int c_hi, int lw, int ch,
                                                              int sum_first, int leaf, int update,
                                                              int32_t* __restrict__ piv, int32_t* __restrict__ info) {
  using namespace pcl;
  extern __shared__ float4 pcl_smem[];
  Cx<S>* L = reinterpret_cast<Cx<S>*>(pcl_smem);  // [lw][ch]: leaf entry (r, t) at t * ch + r - r_lo
  Cx<S>* X = L + (size_t)lw * ch;                 // [2 LW][PW]: gathered rows (CTA 0)
  Cx<S>* Ub = X + 2 * LW * PW;                    // [LW][PW]: the leaf's U block
  __shared__ Rec<S> rec[2][MAXC];
  __shared__ alignas(16) Cx<S> drow[2][LW];       // row c's leaf entries (vector stores, as rec)
  typedef typename KeyOf<S>::type Key;
  constexpr bool F64 = sizeof(S) == 8;
  __shared__ Key red_k[NT / 32];
  __shared__ unsigned red_r[NT / 32];
  __shared__ int s_piv[LW], s_rows[2 * LW], s_src[2 * LW], s_m;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t cl, rank;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(cl));
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int z = blockIdx.x / cl;
  Cx<S>* M = A + (int64_t)z * bstride;
  const int r_lo = p0 + (int)rank * ch, r_hi = min(n, r_lo + ch);  // empty when r_lo >= n
  const int pend = min(p0 + w, n);
  const uint32_t rec_a = (uint32_t)__cvta_generic_to_shared(&rec[0][0]);
  const uint32_t drow_a = (uint32_t)__cvta_generic_to_shared(&drow[0][0]);
  cluster_sync();  // every CTA of the cluster runs before the first remote store
  for (int c0 = c_lo; c0 < c_hi; c0 += lw) {
    const int l = min(lw, pend - c0);
    const int a = max(r_lo, c0);  // first leaf row held here
    const int nr = max(0, r_hi - a);
#pragma unroll 4
    for (int e = tid; e < nr * l; e += NT) {
      const int rr = e / l, t = e - rr * l;
      L[t * ch + a - r_lo + rr] = ldcg(M + (int64_t)(a + rr) * ld + c0 + t);
    }
    __syncthreads();
    // this thread's candidate for the leaf's first column
    S best = -1;
    int bi = n;
    for (int r = a + tid; r < r_hi; r += NT) {
      const Cx<S> v = L[r - r_lo];
      const S m = v.re * v.re + v.im * v.im;
      if (m > best) { best = m; bi = r; }
    }
    for (int cc = 0; cc < l; ++cc) {
      const int c = c0 + cc, buf = c & 1;
      {
        const Key k = bi < n ? key_of(best) : (Key)0;
        const Key K = warp_max(k);
        const unsigned R = __reduce_min_sync(0xffffffffu, k == K ? (unsigned)bi : 0xffffffffu);
        if (lane == 0) { red_k[warp] = K; red_r[warp] = R; }
      }
      __syncthreads();
      if (warp == 0) {
        const Key k = lane < NT / 32 ? red_k[lane] : (Key)0, K = warp_max(k);
        const unsigned r = lane < NT / 32 ? red_r[lane] : 0xffffffffu;
        const unsigned R = __reduce_min_sync(0xffffffffu, k == K ? r : 0xffffffffu);
        const int t = lane & 15;
        const bool mine = c >= r_lo && c < r_hi;
        const Cx<S> v = (K != 0 && t < l) ? L[t * ch + (int)R - r_lo] : Cx<S>{0, 0};
        const Cx<S> d = (mine && t < l) ? L[t * ch + c - r_lo] : Cx<S>{0, 0};
        double mag = 0.0, y = 0.0;
        if constexpr (F64) {
          if (K != 0) mag = __longlong_as_double((long long)(K - 1ull));
          y = 1.0 / mag;
        }
        const uint32_t ra = rec_a + (uint32_t)((buf * MAXC + (int)rank) * sizeof(Rec<S>));
        for (uint32_t q = lane >> 4; q < cl; q += 2) {
          const uint32_t rq = mapa(ra, q);
          st_remote(rq + (uint32_t)sizeof(RecHead<S>) + (uint32_t)(t * sizeof(Cx<S>)), v);
          if constexpr (F64) {
            if (t == 0) {
              st_remote(rq, K);
              st_remote(rq + 8u, (unsigned long long)R);
              st_remote(rq + 16u, Cx<double>{y, mag});
            }
          } else {
            if (t == 0) st_remote(rq, ((unsigned long long)K << 32) | R);
          }
          if (mine) st_remote(mapa(drow_a, q) + (uint32_t)((buf * LW + t) * sizeof(Cx<S>)), d);
        }
      }
      cluster_sync();
      // the winner, from this CTA's copy of the records
      const unsigned long long h = lane < (int)cl ? rec[buf][lane].head : 0ull;
      Key hk;
      unsigned hr;
      if constexpr (F64) {
        hk = h;
        hr = lane < (int)cl ? (unsigned)rec[buf][lane].row : 0u;
      } else {
        hk = (unsigned)(h >> 32);
        hr = (unsigned)h;
      }
      const Key K = warp_max(hk);
      const unsigned R = __reduce_min_sync(0xffffffffu, hk == K ? hr : 0xffffffffu);
      const unsigned who = __ballot_sync(0xffffffffu, hk == K && hr == R);
      const bool found = K != 0;  // (else no candidate is a number: nor is row c's)
      const int p = found ? (int)R : c;
      const Rec<S>& win = rec[buf][found ? __ffs(who) - 1 : 0];
      const Cx<S>* u = found ? win.v : drow[buf];  // the pivot row
      const Cx<S> d = u[cc];
      S dd = d.re * d.re + d.im * d.im;
      bool safe = false;
      double y = 0.0;
      if constexpr (F64) {
        dd = found ? win.mag : 0.0;
        safe = quotient_safe(dd);
        y = win.inv;
      }
      const bool okd = dd > 0;
      if (tid == 0) {
        s_piv[cc] = p;
        if (rank == 0) {
          piv[(int64_t)z * n + c] = p;
          if (!okd && info) atomicOr(info + z, 1);
        }
      }
      // row c takes the pivot row; the thread of row p, below, restores the former row c into it
      if (p != c && tid < l && c >= r_lo && c < r_hi) L[tid * ch + c - r_lo] = u[tid];
      best = -1;
      bi = n;
      for (int r = max(a, c + 1) + tid; r < r_hi; r += NT) {
        Cx<S>* x = L + r - r_lo;
        if (r == p)
          for (int t = 0; t < l; ++t) x[t * ch] = drow[buf][t];
        Cx<S> lv = x[cc * ch];
        if constexpr (sizeof(S) == 4) {
          if (okd) lv = cx_div(lv, d);
        } else {
          if (okd) lv = cx_div_by(lv, d, dd, y, safe);
        }
        x[cc * ch] = lv;
        if (cc + 1 < l) {
          Cx<S> y = x[(cc + 1) * ch];
          cx_msub(y, lv, u[cc + 1]);
          x[(cc + 1) * ch] = y;
          const S m = y.re * y.re + y.im * y.im;
          if (m > best) { best = m; bi = r; }
#pragma unroll 4
          for (int t = cc + 2; t < l; ++t) cx_msub(x[t * ch], lv, u[t]);
        }
      }
      // (the next column's __syncthreads orders these updates before any other thread reads them)
    }
    __syncthreads();
#pragma unroll 4
    for (int e = tid; e < nr * l; e += NT) {
      const int rr = e / l, t = e - rr * l;
      M[(int64_t)(a + rr) * ld + c0 + t] = L[t * ch + a - r_lo + rr];
    }
    const int wall = pend - p0;
    if (rank == 0 && wall > l) {
      // net effect of the leaf's interchanges on the rows they touch: row s_rows[i] receives the
      // former row s_src[i]; the leaf's own rows c0 .. c0+l-1 come first
      if (tid == 0) {
        int m = 0;
        for (int t = 0; t < l; ++t) { s_rows[m] = c0 + t; s_src[m] = c0 + t; ++m; }
        for (int t = 0; t < l; ++t) {
          const int pr = s_piv[t];
          if (pr == c0 + t) continue;
          int ip = -1;
          if (pr < c0 + l) ip = pr - c0;
          else
            for (int i = l; i < m; ++i)
              if (s_rows[i] == pr) { ip = i; break; }
          if (ip < 0) { s_rows[m] = pr; s_src[m] = pr; ip = m++; }
          const int tmp = s_src[t];
          s_src[t] = s_src[ip];
          s_src[ip] = tmp;
        }
        s_m = m;
      }
      __syncthreads();
      const int m = s_m;
#pragma unroll 4
      for (int e = tid; e < m * PW; e += NT) {
        const int i = e / PW, jj = e - i * PW, col = p0 + jj;
        if (jj < wall && (col < c0 || col >= c0 + l)) X[i * PW + jj] = ldcg(M + (int64_t)s_src[i] * ld + col);
      }
      __syncthreads();
      for (int jj = tid; jj < wall; jj += NT)  // U block: forward substitution with the unit lower L11
        if (p0 + jj >= c0 + l) {
          Cx<S> x[LW];
#pragma unroll
          for (int s = 0; s < LW; ++s) x[s] = s < l ? X[s * PW + jj] : Cx<S>{0, 0};
#pragma unroll
          for (int t = 0; t < LW - 1; ++t)
#pragma unroll
            for (int s = t + 1; s < LW; ++s)
              if (s < l) {
                const Cx<S> lv = L[t * ch + c0 + s - r_lo];
                if constexpr (sizeof(S) == 4) {
                  x[s].re -= fma(lv.re, x[t].re, -__fmul_rn(lv.im, x[t].im));
                  x[s].im -= leaf ? fma(lv.im, x[t].re, __fmul_rn(lv.re, x[t].im))
                                  : fma(lv.re, x[t].im, __fmul_rn(lv.im, x[t].re));
                } else {
                  cx_msub(x[s], lv, x[t]);
                }
              }
#pragma unroll
          for (int s = 0; s < LW; ++s)
            if (s < l) X[s * PW + jj] = x[s];
        }
      __syncthreads();
#pragma unroll 4
      for (int e = tid; e < m * PW; e += NT) {
        const int i = e / PW, jj = e - i * PW, col = p0 + jj;
        if (jj < wall && (col < c0 || col >= c0 + l)) M[(int64_t)s_rows[i] * ld + col] = X[i * PW + jj];
      }
    }
    if (!update) continue;  // (one leaf per launch: its update is another kernel's)
    cluster_sync();
    const int cs = c0 + l, wr = pend - cs;
    if (wr > 0) {  // rows below the leaf, panel columns right of it: A -= L_leaf U_leaf
      for (int e = tid; e < l * wr; e += NT) {
        const int t = e / wr, jj = e - t * wr;
        Ub[t * PW + jj] = ldcg(M + (int64_t)(c0 + t) * ld + cs + jj);
      }
      __syncthreads();
      const int rb = max(r_lo, cs);
      const int nrow = max(0, r_hi - rb);
      bool pairs = false;
      if constexpr (sizeof(S) == 4) pairs = ((wr | ld | cs) & 1) == 0 && (bstride & 1) == 0;
      if (pairs) {  // FP32: two columns per thread, 16-byte accesses
        const int hw = wr >> 1;
#pragma unroll 2
        for (int e = tid; e < nrow * hw; e += NT) {
          const int rr = e / hw, jj = 2 * (e - rr * hw), r = rb + rr;
          float4* mp = reinterpret_cast<float4*>(M + (int64_t)r * ld + cs + jj);
          float4 acc = __ldcg(mp);
          if (sum_first) {
            float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int t = 0; t < l; ++t) {
              const Cx<S> lv = L[t * ch + r - r_lo];
              const float4 uu = *reinterpret_cast<const float4*>(Ub + t * PW + jj);
              sum.x += lv.re * uu.x - lv.im * uu.y;
              sum.y += lv.re * uu.y + lv.im * uu.x;
              sum.z += lv.re * uu.z - lv.im * uu.w;
              sum.w += lv.re * uu.w + lv.im * uu.z;
            }
            acc.x -= sum.x; acc.y -= sum.y; acc.z -= sum.z; acc.w -= sum.w;
          } else {
            for (int t = 0; t < l; ++t) {
              const Cx<S> lv = L[t * ch + r - r_lo];
              const float4 uu = *reinterpret_cast<const float4*>(Ub + t * PW + jj);
              acc.x -= lv.re * uu.x - lv.im * uu.y;
              acc.y -= lv.re * uu.y + lv.im * uu.x;
              acc.z -= lv.re * uu.z - lv.im * uu.w;
              acc.w -= lv.re * uu.w + lv.im * uu.z;
            }
          }
          *mp = acc;
        }
      } else {
#pragma unroll 2
        for (int e = tid; e < nrow * wr; e += NT) {
          const int rr = e / wr, jj = e - rr * wr, r = rb + rr;
          Cx<S>* mp = M + (int64_t)r * ld + cs + jj;
          Cx<S> acc = ldcg(mp);
          if (sum_first) {
            S ar = 0, ai = 0;
            for (int t = 0; t < l; ++t) {
              const Cx<S> lv = L[t * ch + r - r_lo], uu = Ub[t * PW + jj];
              ar += lv.re * uu.re - lv.im * uu.im;
              ai += lv.re * uu.im + lv.im * uu.re;
            }
            acc.re -= ar;
            acc.im -= ai;
          } else {
            for (int t = 0; t < l; ++t) cx_msub(acc, L[t * ch + r - r_lo], Ub[t * PW + jj]);
          }
          *mp = acc;
        }
      }
      __syncthreads();
    }
  }
  cluster_sync();  // no CTA leaves while another may still store into its shared memory
}

// Leaf width for a panel whose rows start at p0: the widest power of two <= 16 whose leaf and U
// block (lw x 64) fit in 200 KB of shared memory (fewer, wider leaves re-read the panel fewer
// times); 0 if even one column does not fit (then the global-memory panel runs).
template <class S>
static int leaf_width(int n, int p0) {
  const size_t rows = (size_t)(n - p0);
  for (int lw = 16; lw >= 1; lw >>= 1)
    if ((rows + 64) * lw * sizeof(Cx<S>) <= 200 * 1024) return lw;
  return 0;
}

template <class S>
static int panel_factor(bie_ctx* c, Cx<S>* A, int batch, int n, int ld, int64_t bstride, int p0, int w,
                        int32_t* piv, int32_t* info) {
  const int lw = leaf_width<S>(n, p0);
  if (lw == 0 || w > 64) {
    BIE_LAUNCH(k_panel<S><<<batch, 512, 0, c->stream>>>(A, bstride, n, ld, p0, w, piv, info));
    return BIE_OK;
  }
  BIE_TRY((set_smem_max(k_leaf<S>)));
  // With a large batch the leaf kernel (one CTA per matrix) also updates the panel right of the
  // leaf; with a small one that update runs as its own launch over all rows of every matrix.
  const int fuse = batch >= 64 ? 1 : 0;
  for (int c0 = p0; c0 < p0 + w; c0 += lw) {
    const int l = std::min(lw, p0 + w - c0);
    const int wr = std::max(0, std::min(p0 + w, n) - c0 - l);  // panel columns right of the leaf
    const size_t smem = ((size_t)(n - c0) * l + (size_t)l * std::min(w, n - p0)) * sizeof(Cx<S>);
    BIE_LAUNCH(k_leaf<S><<<batch, 1024, smem, c->stream>>>(A, bstride, n, ld, p0, w, c0, l, piv, info, fuse));
    const int rows = n - c0 - l;
    if (!fuse && rows > 0 && wr > 0) {
      dim3 g((unsigned)((rows + 63) / 64), batch);
      BIE_LAUNCH(k_leaf_update<S><<<g, 256, 0, c->stream>>>(A, bstride, n, ld, p0, w, c0, l));
    }
  }
  return BIE_OK;
}

// ---- row swaps outside the panel, then U12 = L11^{-1} A12 ----------------------------------
// grid: (ceil((n - jlo) / 128), batch), block 128: one column j >= jlo per thread.  With swaps != 0
// the panel's row swaps are applied (in order) to every column outside the panel; the forward
// substitution with the unit lower L11 runs for the columns in [p0 + nb, tend).
template <class S>
__global__ void __launch_bounds__(128) k_swap_trsm(Cx<S>* __restrict__ A, int64_t bstride, int n, int ld, int p0,
                                                   int nb, const int32_t* __restrict__ piv, int jlo, int tend,
                                                   int swaps) {
  Cx<S>* M = A + (int64_t)blockIdx.y * bstride;
  const int32_t* pv = piv + (int64_t)blockIdx.y * n;
  extern __shared__ unsigned char smem_raw[];
  Cx<S>* L11 = reinterpret_cast<Cx<S>*>(smem_raw);  // [nb][nb]
  const int pend = min(p0 + nb, n);
  const int w = pend - p0;
  if (tend > pend) {  // some column is solved: stage L11
    for (int t = threadIdx.x; t < w * w; t += blockDim.x) {
      int r = t / w, cc = t % w;
      L11[t] = M[(int64_t)(p0 + r) * ld + p0 + cc];
    }
    __syncthreads();
  }
  const int j = jlo + blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n || (j >= p0 && j < pend)) return;
  if (swaps)
    for (int s = p0; s < pend; ++s) {
      int p = pv[s];
      if (p != s) {
        Cx<S> t = M[(int64_t)s * ld + j];
        M[(int64_t)s * ld + j] = M[(int64_t)p * ld + j];
        M[(int64_t)p * ld + j] = t;
      }
    }
  if (j < pend || j >= tend) return;  // columns left of the panel (or past tend) only get the swaps
  // forward substitution with the unit lower L11; solved entries are re-read from the column
  for (int s = 1; s < w; ++s) {
    Cx<S> v = M[(int64_t)(p0 + s) * ld + j];
    for (int t = 0; t < s; ++t) {
      const Cx<S> l = L11[s * w + t];
      const Cx<S> xt = M[(int64_t)(p0 + t) * ld + j];
      v.re -= l.re * xt.re - l.im * xt.im;
      v.im -= l.re * xt.im + l.im * xt.re;
    }
    M[(int64_t)(p0 + s) * ld + j] = v;
  }
}

// ---- U = L11^{-1} A for a full 64-row panel, FP32 --------------------------------------------
// grid (ceil((j1 - j0) / 64), batch), block 64, dynamic smem 64 KB: one column j in [j0, j1) per
// thread, solved in four blocks of 16 rows.  A block's 16 entries live in registers: first the
// products with the solved entries of the earlier blocks (a loop over t that reads x_t from this
// thread's shared-memory column and L11's column t as 16-byte broadcasts), then the solve inside
// the block (unrolled).  Each x_s receives its updates in increasing t, the order of the row-by-row
// substitution of k_swap_trsm.  (A fully unrolled 64-entry register version ran from the
// instruction cache's misses.)
// With bt.ub set, each solved column also goes, rounded to TF32, into the B^T buffer of the
// tensor-core update (the real embedding: B^T rows 2 (j - bt.cb) and 2 (j - bt.cb) + 1 get, at
// floats bt.koff + 2 s, [ur, -ui] and [ui, ur]; rows bt.krow floats long, bt.stride per matrix),
// which saves the separate build pass over U.
struct BtOut {
  float* ub;
  int64_t stride;
  int krow, koff, cb;
};
__device__ __forceinline__ float round_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}
constexpr size_t kTrsmSmem = 2 * 64 * 64 * sizeof(Cx<float>);  // L11^T and the solved columns
__global__ void __launch_bounds__(64) k_trsm64(Cx<float>* __restrict__ A, int64_t bstride, int n, int ld, int p0,
                                               int j0, int j1, BtOut bt) {
  extern __shared__ float4 trsm_smem[];
  Cx<float>* LT = reinterpret_cast<Cx<float>*>(trsm_smem);  // LT[t * 64 + s] = L11[s][t]
  Cx<float>(*X)[64] = reinterpret_cast<Cx<float>(*)[64]>(LT + 64 * 64);  // X[s][thread]: the solved column
  Cx<float>* M = A + (int64_t)blockIdx.y * bstride;
  const int tid = threadIdx.x;
#pragma unroll 8
  for (int e = tid; e < 64 * 64; e += 64) {
    const int r = e >> 6, c = e & 63;  // coalesced read of row r
    LT[c * 64 + r] = M[(int64_t)(p0 + r) * ld + p0 + c];
  }
  __syncthreads();
  const int j = j0 + blockIdx.x * blockDim.x + tid;
  const bool act = j < j1 && j < n;
#pragma unroll 1
  for (int b0 = 0; b0 < 64; b0 += 16) {
    Cx<float> xb[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) xb[r] = act ? M[(int64_t)(p0 + b0 + r) * ld + j] : Cx<float>{0.f, 0.f};
#pragma unroll 2
    for (int t = 0; t < b0; ++t) {  // earlier blocks
      const Cx<float> xt = X[t][tid];
      const float4* l4 = reinterpret_cast<const float4*>(&LT[t * 64 + b0]);
#pragma unroll
      for (int r = 0; r < 16; r += 2) {
        const float4 l = l4[r >> 1];  // L11[b0 + r][t], L11[b0 + r + 1][t]
        xb[r].re -= l.x * xt.re - l.y * xt.im;
        xb[r].im -= l.x * xt.im + l.y * xt.re;
        xb[r + 1].re -= l.z * xt.re - l.w * xt.im;
        xb[r + 1].im -= l.z * xt.im + l.w * xt.re;
      }
    }
#pragma unroll
    for (int t = 0; t < 15; ++t) {  // inside the block
      const Cx<float> xt = xb[t];
#pragma unroll
      for (int r = t + 1; r < 16; ++r) {
        const Cx<float> l = LT[(b0 + t) * 64 + b0 + r];
        xb[r].re -= l.re * xt.re - l.im * xt.im;
        xb[r].im -= l.re * xt.im + l.im * xt.re;
      }
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      X[b0 + r][tid] = xb[r];
      if (act && (b0 + r) > 0) M[(int64_t)(p0 + b0 + r) * ld + j] = xb[r];
    }
  }
  if (bt.ub && act) {  // this thread's column is complete in X
    float* o = bt.ub + (int64_t)blockIdx.y * bt.stride + (int64_t)2 * (j - bt.cb) * bt.krow + bt.koff;
#pragma unroll 4
    for (int s2 = 0; s2 < 64; s2 += 2) {
      const Cx<float> u0 = X[s2][tid], u1 = X[s2 + 1][tid];
      const float a0 = round_tf32(u0.re), b0 = round_tf32(u0.im), a1 = round_tf32(u1.re), b1 = round_tf32(u1.im);
      *reinterpret_cast<float4*>(o + 2 * s2) = make_float4(a0, -b0, a1, -b1);
      *reinterpret_cast<float4*>(o + bt.krow + 2 * s2) = make_float4(b0, a0, b1, a1);
    }
  }
}

// The same for FP64: 32 columns (lanes) per CTA, their 64 rows in the registers of four warps, four rows of
// every 16 each: the owner of the next four rows solves them and leaves them in shared memory, then
// every warp subtracts their products from its later rows.  Each SM quarter has its own FP64 lanes: one
// warp alone reaches a quarter of the rate.  grid (ceil((j1 - j0) / 32), batch), block 128.
// N = 2884, two systems (45 launches): 12.6 ms by k_swap_trsm<double>'s substitution through global
// memory, 18.1 ms one warp per 32 columns, 4.7 ms this way.
constexpr size_t kTrsm64dSmem = (64 * 64 + 4 * 32) * sizeof(Cx<double>);
__global__ void __launch_bounds__(128) k_trsm64d(Cx<double>* __restrict__ A, int64_t bstride, int n, int ld, int p0, int j0,
                                                 int j1) {
  extern __shared__ double2 trsmd_smem[];
  Cx<double>* LT = reinterpret_cast<Cx<double>*>(trsmd_smem);            // LT[t * 64 + s] = L11[s][t]
  Cx<double>(*X)[32] = reinterpret_cast<Cx<double>(*)[32]>(LT + 64 * 64);  // the four rows just solved
  Cx<double>* M = A + (int64_t)blockIdx.y * bstride;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll 8
  for (int e = threadIdx.x; e < 64 * 64; e += 128) {
    const int r = e >> 6, c = e & 63;
    LT[c * 64 + r] = M[(int64_t)(p0 + r) * ld + p0 + c];
  }
  const int j = j0 + blockIdx.x * 32 + lane;
  const bool act = j < j1 && j < n;
  Cx<double> x[4][4];  // rows 16 b + 4 warp + r
#pragma unroll
  for (int b = 0; b < 4; ++b)
#pragma unroll
    for (int r = 0; r < 4; ++r)
      x[b][r] = act ? M[(int64_t)(p0 + 16 * b + 4 * warp + r) * ld + j] : Cx<double>{0.0, 0.0};
  __syncthreads();
#pragma unroll
  for (int b = 0; b < 4; ++b)
#pragma unroll 1
    for (int w = 0; w < 4; ++w) {
      const int t0 = 16 * b + 4 * w;
      if (warp == w) {
#pragma unroll
        for (int t = 0; t < 3; ++t)
#pragma unroll
          for (int r = t + 1; r < 4; ++r) cx_msub(x[b][r], LT[(t0 + t) * 64 + t0 + r], x[b][t]);
#pragma unroll
        for (int r = 0; r < 4; ++r) X[r][lane] = x[b][r];
      }
      __syncthreads();
#pragma unroll
      for (int b2 = b; b2 < 4; ++b2)
        if (b2 > b || warp > w)
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const Cx<double> xt = X[t][lane];
#pragma unroll
            for (int r = 0; r < 4; ++r) cx_msub(x[b2][r], LT[(t0 + t) * 64 + 16 * b2 + 4 * warp + r], xt);
          }
      __syncthreads();
    }
  if (act)
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int r = 0; r < 4; ++r) M[(int64_t)(p0 + 16 * b + 4 * warp + r) * ld + j] = x[b][r];
}

// ---- SIMT trailing update A22 -= L21 U12 (64 x 64 complex tile per CTA, 256 threads) ---------
template <class S>
__global__ void __launch_bounds__(256) k_gemm_update(Cx<S>* __restrict__ A, int64_t bstride, int n, int ld,
                                                     int p0, int nb) {
  Cx<S>* M = A + (int64_t)blockIdx.z * bstride;
  const int r0 = p0 + nb + blockIdx.y * 64, c0 = p0 + nb + blockIdx.x * 64;
  if (r0 >= n || c0 >= n) return;
  __shared__ Cx<S> Ls[16][64 + 1];  // [k][row]
  __shared__ Cx<S> Us[16][64 + 1];  // [k][col]
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  Cx<S> acc[4][4];
  for (int a = 0; a < 4; ++a)
    for (int b = 0; b < 4; ++b) acc[a][b] = {0, 0};
  for (int k0 = p0; k0 < p0 + nb; k0 += 16) {
    for (int t = threadIdx.x; t < 16 * 64; t += 256) {
      int kk = t & 15, rr = t >> 4;
      int gr = r0 + rr, gk = k0 + kk;
      Ls[kk][rr] = (gr < n && gk < p0 + nb) ? M[(int64_t)gr * ld + gk] : Cx<S>{0, 0};
      int cc = t & 63, k2 = t >> 6;
      int gc = c0 + cc, gk2 = k0 + k2;
      Us[k2][cc] = (gc < n && gk2 < p0 + nb) ? M[(int64_t)gk2 * ld + gc] : Cx<S>{0, 0};
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < 16; ++kk) {
      Cx<S> l[4], u[4];
      for (int a = 0; a < 4; ++a) l[a] = Ls[kk][ty + 16 * a];
      for (int b = 0; b < 4; ++b) u[b] = Us[kk][tx + 16 * b];
      for (int a = 0; a < 4; ++a)
        for (int b = 0; b < 4; ++b) {
          acc[a][b].re += l[a].re * u[b].re - l[a].im * u[b].im;
          acc[a][b].im += l[a].re * u[b].im + l[a].im * u[b].re;
        }
    }
    __syncthreads();
  }
  for (int a = 0; a < 4; ++a)
    for (int b = 0; b < 4; ++b) {
      int gr = r0 + ty + 16 * a, gc = c0 + tx + 16 * b;
      if (gr < n && gc < n) {
        Cx<S>& m = M[(int64_t)gr * ld + gc];
        m.re -= acc[a][b].re;
        m.im -= acc[a][b].im;
      }
    }
}

// ---- solves with the factor: x = U^{-1} L^{-1} P b; one CTA per (matrix) -------------------
template <class S, class SB>
__global__ void __launch_bounds__(256) k_lu_solve(const Cx<S>* __restrict__ LU, int64_t bstride, int n, int ld,
                                                  const int32_t* __restrict__ piv, Cx<SB>* __restrict__ b,
                                                  int64_t bstride_b) {
  const Cx<S>* M = LU + (int64_t)blockIdx.x * bstride;
  const int32_t* pv = piv + (int64_t)blockIdx.x * n;
  Cx<SB>* x = b + (int64_t)blockIdx.x * bstride_b;
  __shared__ SB red[2][8];
  __shared__ Cx<SB> xr;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0)
    for (int s = 0; s < n; ++s) {
      int p = pv[s];
      if (p != s) { Cx<SB> t = x[s]; x[s] = x[p]; x[p] = t; }
    }
  __syncthreads();
  for (int pass = 0; pass < 2; ++pass) {
    for (int ii = 0; ii < n; ++ii) {
      const int r = pass == 0 ? ii : n - 1 - ii;
      SB sr = 0, si = 0;
      const int lo = pass == 0 ? 0 : r + 1, hi = pass == 0 ? r : n;
      for (int cc = lo + tid; cc < hi; cc += blockDim.x) {
        Cx<S> l = M[(int64_t)r * ld + cc];
        Cx<SB> v = x[cc];
        sr += (SB)l.re * v.re - (SB)l.im * v.im;
        si += (SB)l.re * v.im + (SB)l.im * v.re;
      }
      for (int o = 16; o > 0; o >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        si += __shfl_xor_sync(0xffffffffu, si, o);
      }
      if (lane == 0) { red[0][warp] = sr; red[1][warp] = si; }
      __syncthreads();
      if (tid == 0) {
        SB tr = 0, ti = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { tr += red[0][w]; ti += red[1][w]; }
        Cx<SB> v = {x[r].re - tr, x[r].im - ti};
        if (pass == 1) {
          Cx<S> d = M[(int64_t)r * ld + r];
          Cx<SB> dd = {(SB)d.re, (SB)d.im};
          SB den = dd.re * dd.re + dd.im * dd.im;
          v = {(v.re * dd.re + v.im * dd.im) / den, (v.im * dd.re - v.re * dd.im) / den};
        }
        x[r] = v;
      }
      __syncthreads();
    }
  }
}

// The same in FP64 over all SMs: y = P b gathered, then for each 64-row block its triangular solve by
// one CTA per system (k_solve_block) and the product with the rest of its columns by a warp per row
// (k_solve_rows).  N = 2884, two systems: 35.6 ms of one CTA per system, row by row -> 2.5 ms.
__global__ void k_gather_perm(const Cx<double>* __restrict__ b, int64_t bstride_b, int n, const int32_t* __restrict__ perm,
                              Cx<double>* __restrict__ y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[(int64_t)blockIdx.y * n + i] = b[(int64_t)blockIdx.y * bstride_b + perm[(int64_t)blockIdx.y * n + i]];
}
__global__ void k_copy_back(const Cx<double>* __restrict__ y, int n, Cx<double>* __restrict__ b, int64_t bstride_b) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[(int64_t)blockIdx.y * bstride_b + i] = y[(int64_t)blockIdx.y * n + i];
}
template <bool LOWER>
__global__ void __launch_bounds__(256) k_solve_block(const Cx<double>* __restrict__ LU, int64_t bstride, int n, int ld,
                                                     int j0, Cx<double>* __restrict__ yv) {
  extern __shared__ double2 sblk_smem[];
  Cx<double>* D = reinterpret_cast<Cx<double>*>(sblk_smem);  // [64][65], column t at t * 65
  Cx<double>* x = D + 64 * 65;
  const int bs = min(64, n - j0), tid = threadIdx.x;
  const Cx<double>* M = LU + (int64_t)blockIdx.x * bstride + (int64_t)j0 * ld + j0;
  Cx<double>* y = yv + (int64_t)blockIdx.x * n + j0;
#pragma unroll 8
  for (int e = tid; e < bs * 64; e += 256) {
    const int r = e >> 6, t = e & 63;
    if (t < bs) D[t * 65 + r] = M[(int64_t)r * ld + t];
  }
  if (tid < bs) x[tid] = y[tid];
  __syncthreads();
  if (tid >= 64) return;
  Cx<double> v = tid < bs ? x[tid] : Cx<double>{0.0, 0.0};  // thread r holds row r
  Cx<double> d = {1.0, 0.0};
  double dd = 1.0, inv = 1.0;  // |U_rr|^2 and its reciprocal, once
  if (!LOWER && tid < bs) {
    d = D[tid * 65 + tid];
    dd = d.re * d.re + d.im * d.im;
    inv = 1.0 / dd;
  }
  const bool safe = quotient_safe(dd);
  for (int k = 0; k < bs; ++k) {
    const int s = LOWER ? k : bs - 1 - k;
    if (tid == s) {
      if (!LOWER) v = cx_div_by(v, d, dd, inv, safe);
      x[s] = v;
    }
    asm volatile("bar.sync 1, 64;" ::: "memory");
    if (tid < bs && (LOWER ? tid > s : tid < s)) cx_msub(v, D[s * 65 + tid], x[s]);
  }
  if (tid < bs) y[tid] = v;
}
// y[r] -= sum over the block's columns of LU[r][c] y[c], rows [rlo, rhi): grid (ceil(rows / 8), batch), block 256
__global__ void __launch_bounds__(256) k_solve_rows(const Cx<double>* __restrict__ LU, int64_t bstride, int n, int ld, int j0,
                                                    int rlo, int rhi, Cx<double>* __restrict__ yv) {
  const int lane = threadIdx.x & 31, r = rlo + blockIdx.x * 8 + (threadIdx.x >> 5);
  if (r >= rhi) return;
  const Cx<double>* M = LU + (int64_t)blockIdx.y * bstride + (int64_t)r * ld + j0;
  Cx<double>* y = yv + (int64_t)blockIdx.y * n;
  const int bs = min(64, n - j0);
  Cx<double> a = {0.0, 0.0};
  for (int c = lane; c < bs; c += 32) cx_msub(a, M[c], y[j0 + c]);
  for (int o = 16; o > 0; o >>= 1) {
    a.re += __shfl_xor_sync(0xffffffffu, a.re, o);
    a.im += __shfl_xor_sync(0xffffffffu, a.im, o);
  }
  if (lane == 0) {
    y[r].re += a.re;
    y[r].im += a.im;
  }
}

// ---- host drivers -----------------------------------------------------------------------------
template <class S>
int lu_factor_simt(bie_ctx* c, Cx<S>* A, int batch, int n, int ld, int64_t bstride, int32_t* piv, int32_t* info,
                   int nb) {
  if (nb > 64) nb = 64;
  for (int p0 = 0; p0 < n; p0 += nb) {
    const int w = std::min(nb, n - p0);
    BIE_TRY(panel_factor<S>(c, A, batch, n, ld, bstride, p0, w, piv, info));
    dim3 gs((unsigned)((n + 127) / 128), batch);
    BIE_LAUNCH(k_swap_trsm<S><<<gs, 128, (size_t)w * w * sizeof(Cx<S>), c->stream>>>(A, bstride, n, ld, p0, w, piv,
                                                                                     0, n, 1));
    const int rem = n - p0 - w;
    if (rem > 0) {
      dim3 gg((unsigned)((rem + 63) / 64), (unsigned)((rem + 63) / 64), batch);
      BIE_LAUNCH(k_gemm_update<S><<<gg, 256, 0, c->stream>>>(A, bstride, n, ld, p0, w));
    }
  }
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

// The cluster panel (k_panel_cluster) for the panel at p0 when it applies; *used tells whether it
// ran.  The largest cluster of which as many as matrices are resident at once, or in the fewest
// rounds (the time of a column falls with its rows per CTA until the barrier's latency is left).
// Measured, factorisation
// phase with 16 / 8 / 4 / 2 CTAs a matrix and with one-CTA leaves (k_leaf): two systems of N = 10 272
// 46.8 / 55.8 / 76.7 / 140 / 141 ms, 24 of N = 3086 30.7 / 20.9 / 16.7 / 20.5 / 23.2, 64 of N = 2884 67.6 /
// 44.9 / 31.4 / 27.6 / 32.1, one of N = 362 0.86 / 0.87 / 0.87 / 0.90 / 1.09.  Where only one CTA a matrix
// fits (128 systems: 51.3 against 47.6 ms) the leaves of k_leaf remain, except for a panel that one
// CTA holds anyway.
template <class S>
static int panel_cluster(bie_ctx* c, Cx<S>* A, int batch, int n, int ld, int64_t bstride, int p0, int w, int32_t* piv,
                         int32_t* info, bool* used) {
  *used = false;
  const int rows = n - p0;
  if (!c->lu_coop || w > pcl::PW) return BIE_OK;
  BIE_TRY((set_smem_max(k_panel_cluster<S>)));
  BIE_CUDA_TRY(cudaFuncSetAttribute((const void*)k_panel_cluster<S>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaFuncAttributes fa;
  BIE_CUDA_TRY(cudaFuncGetAttributes(&fa, (const void*)k_panel_cluster<S>));
  const size_t limit = (size_t)smem_optin() - fa.sharedSizeBytes;
  // The form of the roundings: panels of up to 1536 rows and of batches above half the SMs as
  // k_leaf; else 16-column leaves, narrower where a matrix's share of the SMs, taken as one CTA each with
  // at least 256 rows, would hold no more of its rows in shared memory.
  int nsm = 0;
  BIE_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device));
  const int share = std::min(nsm / batch, (rows + 255) / 256);
  const int leaf = rows <= 1536 || share < 2 ? 1 : 0, sum_first = leaf && batch < 64 ? 1 : 0;
  int lw_max = pcl::LW;
  if (sizeof(S) == 8) {  // FP64: the widest leaf that 16 CTAs hold
    const int ch16 = std::max(pcl::PW, ((rows + 15) / 16 + 31) / 32 * 32);
    while (lw_max > 4 && pcl::smem_bytes<S>(lw_max, ch16) > limit) lw_max >>= 1;
  } else if (!leaf) {
    const size_t held = ((rows + share - 1) / share + 63) / 64 * 64;
    while (lw_max > 4 && (lw_max * held + pcl::LW * pcl::PW) * sizeof(Cx<S>) > 231 * 1024 - 4096) lw_max >>= 1;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(pcl::NT);
  cfg.stream = c->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  // the cluster: fewest rounds of resident clusters, then the most CTAs; sizes between the powers of two
  // only where those take two rounds (a cluster stays within one group of SMs, which leaves some of them
  // idle beside 8 or 16 CTAs): 40 systems of N = 5010 72.0 -> 66.8 ms
  int best_cl = 0, best_ch = 0, best_lw = 0, best_rounds = 0;
  auto consider = [&](int cl, int lw) -> int {
    const int ch = std::max(pcl::PW, ((rows + cl - 1) / cl + 31) / 32 * 32);
    if (cl > 1 && (int64_t)(cl / 2) * ch >= rows) return BIE_OK;  // half as many CTAs hold the rows
    if (cl == 1 && rows > pcl::PW) return BIE_OK;
    if (pcl::smem_bytes<S>(lw, ch) > limit) return BIE_OK;
    cfg.gridDim = dim3((unsigned)(batch * cl));
    cfg.dynamicSmemBytes = pcl::smem_bytes<S>(lw, ch);
    at[0].val.clusterDim.x = (unsigned)cl;
    int active = 0;
    BIE_CUDA_TRY(cudaOccupancyMaxActiveClusters(&active, k_panel_cluster<S>, &cfg));
    if (active < 1) return BIE_OK;
    const int rounds = (batch + active - 1) / active;
    if (best_cl == 0 || rounds < best_rounds) {
      best_cl = cl;
      best_ch = ch;
      best_lw = lw;
      best_rounds = rounds;
    }
    return BIE_OK;
  };
  for (const int cl : {16, 8, 4, 2, 1}) BIE_TRY(consider(cl, lw_max));
  if (best_rounds != 1)
    for (const int cl : {12, 9, 7, 6, 5, 3}) BIE_TRY(consider(cl, lw_max));
  // FP32 panels in two rounds: one round of clusters that hold eight columns of their rows costs less (a
  // leaf's own costs, twice as often, are 5 % of a panel's time): 9 / 18 systems of N = 20 544, whose sixteen
  // columns only 13 CTAs and more hold, 509 / 1019 -> 493 / 985 ms; 14 of N = 16 050 375.9 -> 373.6
  if (sizeof(S) == 4 && !leaf && best_rounds > 1 && lw_max > 8)
    for (const int cl : {12, 10, 9, 8, 7, 6, 5, 4, 3}) {
      if (best_rounds == 1) break;
      BIE_TRY(consider(cl, 8));
    }
  if (best_cl == 0 || best_rounds > (share >= 2 ? 2 : 1)) return BIE_OK;
  cfg.gridDim = dim3((unsigned)(batch * best_cl));
  cfg.dynamicSmemBytes = pcl::smem_bytes<S>(best_lw, best_ch);
  at[0].val.clusterDim.x = (unsigned)best_cl;
  const int lw = std::min(best_lw, w), pend = std::min(p0 + w, n);
  if (sizeof(S) == 4) {
    count_launch();
    BIE_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_panel_cluster<S>, A, bstride, n, ld, p0, w, p0, pend, lw, best_ch, sum_first,
                                    leaf, 1, piv, info));
  } else {
    // FP64: a launch per leaf, and the update of the panel's other columns over all SMs (the
    // clusters' few SMs would take longer for its FP64 arithmetic than for the leaf)
    for (int c0 = p0; c0 < pend; c0 += lw) {
      const int l = std::min(lw, pend - c0), below = n - c0 - l;
      count_launch();
      BIE_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_panel_cluster<S>, A, bstride, n, ld, p0, w, c0, c0 + l, lw, best_ch,
                                      sum_first, leaf, 0, piv, info));
      if (below > 0 && c0 + l < pend)
        BIE_LAUNCH(k_leaf_update<S><<<dim3((unsigned)((below + 7) / 8), batch), 256, 0, c->stream>>>(A, bstride, n, ld, p0, w,
                                                                                                  c0, l));
    }
  }
  *used = true;
  return BIE_OK;
}

// Panel factorisation plus row swaps (all columns) and the U12 solve of the columns in
// [p0 + w, tend) for one block column (FP32); the trailing update is left to the caller (the
// tensor-core kernels of lu_tc.cu).
int lu_panel_steps32(bie_ctx* c, cf* A, int batch, int n, int ld, int64_t bstride, int p0, int w, int32_t* piv,
                     int32_t* info, int tend, float* ub, int64_t ub_stride, int krow, int koff, bool* emitted) {
  if (emitted) *emitted = false;
  Cx<float>* M = reinterpret_cast<Cx<float>*>(A);
  bool used = false;
  BIE_TRY(panel_cluster<float>(c, M, batch, n, ld, bstride, p0, w, piv, info, &used));
  if (!used) BIE_TRY(panel_factor<float>(c, M, batch, n, ld, bstride, p0, w, piv, info));
  dim3 gs((unsigned)((n + 127) / 128), batch);
  if (w == 64) {  // swaps here, the solve with the register-resident kernel
    BIE_LAUNCH(k_swap_trsm<float><<<gs, 128, 0, c->stream>>>(M, bstride, n, ld, p0, w, piv, 0, p0 + w, 1));
    if (tend > p0 + w) {
      BIE_TRY((set_smem_max(k_trsm64)));
      dim3 gt((unsigned)((tend - p0 - w + 63) / 64), batch);
      const BtOut bt{ub, ub_stride, krow, koff, p0 + w};
      BIE_LAUNCH(k_trsm64<<<gt, 64, kTrsmSmem, c->stream>>>(M, bstride, n, ld, p0, p0 + w, tend, bt));
      if (emitted) *emitted = ub != nullptr;
    }
  } else {
    BIE_LAUNCH(k_swap_trsm<float><<<gs, 128, (size_t)w * w * sizeof(Cx<float>), c->stream>>>(M, bstride, n, ld, p0, w,
                                                                                            piv, 0, tend, 1));
  }
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

// U = L11^{-1} A for rows [p0, p0 + w) and the columns [jlo, n), L11 the unit lower diagonal block
// at (p0, p0) (FP32; no swaps).
int lu_trsm_rows32(bie_ctx* c, cf* A, int batch, int n, int ld, int64_t bstride, int p0, int w, int jlo, float* ub,
                   int64_t ub_stride, int krow, int koff, bool* emitted) {
  if (emitted) *emitted = false;
  if (jlo >= n) return BIE_OK;
  Cx<float>* M = reinterpret_cast<Cx<float>*>(A);
  dim3 gs((unsigned)((n - jlo + 127) / 128), batch);
  if (w == 64) {
    BIE_TRY((set_smem_max(k_trsm64)));
    dim3 gt((unsigned)((n - jlo + 63) / 64), batch);
    const BtOut bt{ub, ub_stride, krow, koff, jlo};
    BIE_LAUNCH(k_trsm64<<<gt, 64, kTrsmSmem, c->stream>>>(M, bstride, n, ld, p0, jlo, n, bt));
    if (emitted) *emitted = ub != nullptr;
  }
  else
    BIE_LAUNCH(k_swap_trsm<float><<<gs, 128, (size_t)w * w * sizeof(Cx<float>), c->stream>>>(M, bstride, n, ld, p0, w,
                                                                                            nullptr, jlo, n, 0));
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

size_t lu_split_scratch_bytes(int batch, int n);
int lu_update_split64(bie_ctx* c, cd* A, int batch, int n, int ld, int64_t bstride, int p0, void* scratch, int32_t* err);

// Bytes of c->work6 for the FP64 assembly, factorisation and solves of `batch` systems of n rows (the
// assembly's n may be the larger quadratic image's of a linear mesh: it is of the context's elements).
size_t fp64_scratch_bytes(bie_ctx* c, int batch, int n) {
  const size_t known = (size_t)batch * c->E * c->rule.Q * sizeof(cd);
  const size_t solve = (size_t)batch * n * (sizeof(cd) + sizeof(int32_t));
  return std::max(std::max(known, solve), n > 128 ? lu_split_scratch_bytes(batch, n) : (size_t)0);
}

// FP64 LU: 64-column panels (clusters, else one CTA per matrix), their row swaps and U blocks, and the
// trailing update: split into digits on the tensor cores (lu_split.cu), or on the FP64 pipe for matrices
// of at most two panels.  Its callers size c->work6 with their batch (fp64_scratch_bytes); only where one
// system alone fills the device's memory do the digits not fit beside it, and the FP64 pipe takes over.  info: zero pivots, per system; *err
// (device, cleared by the caller): a bounded wait gave up, every factor of the batch is void.
int lu_factor64(bie_ctx* c, cd* A, int batch, int n, int ld, int64_t bstride, int32_t* piv, int32_t* info, int32_t* err) {
  Cx<double>* M = reinterpret_cast<Cx<double>*>(A);
  const bool split = n > 128 && ensure_buf(c, c->work6, lu_split_scratch_bytes(batch, n)) == BIE_OK;
  for (int p0 = 0; p0 < n; p0 += 64) {
    const int w = std::min(64, n - p0);
    bool used = false;
    BIE_TRY(panel_cluster<double>(c, M, batch, n, ld, bstride, p0, w, piv, info, &used));
    if (!used) BIE_TRY(panel_factor<double>(c, M, batch, n, ld, bstride, p0, w, piv, info));
    dim3 gs((unsigned)((n + 127) / 128), batch);
    BIE_LAUNCH(k_swap_trsm<double><<<gs, 128, 0, c->stream>>>(M, bstride, n, ld, p0, w, piv, 0, p0 + w, 1));
    const int rem = n - p0 - w;
    if (rem > 0) {
      BIE_TRY((set_smem_max(k_trsm64d)));
      BIE_LAUNCH(k_trsm64d<<<dim3((unsigned)((rem + 31) / 32), batch), 128, kTrsm64dSmem, c->stream>>>(M, bstride, n, ld, p0,
                                                                                                     p0 + w, n));
      if (split) {
        BIE_TRY(lu_update_split64(c, A, batch, n, ld, bstride, p0, c->work6.p, err));
        continue;
      }
      dim3 gg((unsigned)((rem + 63) / 64), (unsigned)((rem + 63) / 64), batch);
      BIE_LAUNCH(k_gemm_update<double><<<gg, 256, 0, c->stream>>>(M, bstride, n, ld, p0, w));
    }
  }
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

__global__ void k_piv_to_perm(const int32_t* __restrict__ piv, int n, int32_t* __restrict__ perm);

int lu_solve64(bie_ctx* c, const cd* LU, int batch, int n, int ld, int64_t bstride, const int32_t* piv, cd* b,
               int64_t bstride_b) {
  const Cx<double>* M = reinterpret_cast<const Cx<double>*>(LU);
  Cx<double>* rhs = reinterpret_cast<Cx<double>*>(b);
  if ((size_t)n * sizeof(int32_t) > 200 * 1024) {  // the permutation is formed in shared memory
    BIE_LAUNCH(k_lu_solve<double, double><<<batch, 256, 0, c->stream>>>(M, bstride, n, ld, piv, rhs, bstride_b));
    BIE_CUDA_TRY(cudaGetLastError());
    return BIE_OK;
  }
  const size_t ysz = (size_t)batch * n * sizeof(Cx<double>);
  BIE_TRY(ensure_buf(c, c->work6, ysz + (size_t)batch * n * sizeof(int32_t)));
  Cx<double>* y = (Cx<double>*)c->work6.p;
  int32_t* perm = (int32_t*)((char*)c->work6.p + ysz);
  BIE_TRY((set_smem_max(k_piv_to_perm)));
  BIE_LAUNCH(k_piv_to_perm<<<batch, 256, (size_t)n * sizeof(int32_t), c->stream>>>(piv, n, perm));
  const dim3 gv((unsigned)((n + 255) / 256), batch);
  BIE_LAUNCH(k_gather_perm<<<gv, 256, 0, c->stream>>>(rhs, bstride_b, n, perm, y));
  const size_t smem = (64 * 65 + 64) * sizeof(Cx<double>);
  BIE_TRY((set_smem_max(k_solve_block<true>)));
  BIE_TRY((set_smem_max(k_solve_block<false>)));
  const int nblk = (n + 63) / 64;
  for (int pass = 0; pass < 2; ++pass)
    for (int bi = 0; bi < nblk; ++bi) {
      const int j0 = (pass == 0 ? bi : nblk - 1 - bi) * 64;
      if (pass == 0) BIE_LAUNCH(k_solve_block<true><<<batch, 256, smem, c->stream>>>(M, bstride, n, ld, j0, y));
      else BIE_LAUNCH(k_solve_block<false><<<batch, 256, smem, c->stream>>>(M, bstride, n, ld, j0, y));
      const int rlo = pass == 0 ? j0 + 64 : 0, rhi = pass == 0 ? n : j0;
      if (rhi > rlo)
        BIE_LAUNCH(k_solve_rows<<<dim3((unsigned)((rhi - rlo + 7) / 8), batch), 256, 0, c->stream>>>(M, bstride, n, ld, j0,
                                                                                                  rlo, rhi, y));
    }
  BIE_LAUNCH(k_copy_back<<<gv, 256, 0, c->stream>>>(y, n, rhs, bstride_b));
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}
// FP32 LU without tensor cores for systems the TF32 factor cannot refine: 64-column panels, their
// row swaps and U blocks, and the trailing update A22 -= L21 U12 in FP32 on the CUDA cores
// (k_gemm_update).
int lu_factor32_panels(bie_ctx* c, cf* A, int batch, int n, int ld, int64_t bstride, int32_t* piv, int32_t* info) {
  Cx<float>* M = reinterpret_cast<Cx<float>*>(A);
  for (int p0 = 0; p0 < n; p0 += 64) {
    const int w = std::min(64, n - p0);
    BIE_TRY(lu_panel_steps32(c, A, batch, n, ld, bstride, p0, w, piv, info, n, nullptr, 0, 0, 0, nullptr));
    const int rem = n - p0 - w;
    if (rem > 0) {
      dim3 gg((unsigned)((rem + 63) / 64), (unsigned)((rem + 63) / 64), batch);
      BIE_LAUNCH(k_gemm_update<float><<<gg, 256, 0, c->stream>>>(M, bstride, n, ld, p0, w));
    }
  }
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

int lu_factor32(bie_ctx* c, cf* A, int batch, int n, int ld, int64_t bstride, int32_t* piv, int32_t* info) {
  return lu_factor_simt<float>(c, reinterpret_cast<Cx<float>*>(A), batch, n, ld, bstride, piv, info, 32);
}
int lu_solve32(bie_ctx* c, const cf* LU, int batch, int n, int ld, int64_t bstride, const int32_t* piv, cf* b,
               int64_t bstride_b) {
  BIE_LAUNCH(k_lu_solve<float, float><<<batch, 256, 0, c->stream>>>(reinterpret_cast<const Cx<float>*>(LU), bstride, n, ld, piv,
                                                         reinterpret_cast<Cx<float>*>(b), bstride_b));
  BIE_CUDA_TRY(cudaGetLastError());
  return BIE_OK;
}

}  // namespace bie
