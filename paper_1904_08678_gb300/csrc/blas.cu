// BLAS-1 kernels and the device-side Arnoldi/Givens bookkeeping of the Krylov
// solvers (Sec. 2.1: MR, GMRES, FGMRES).  Fields are batches [nrhs][n] of
// complex numbers; every per-rhs scalar stays in device memory so the solver
// loops issue no host round trip except their stopping tests.
// Reductions are two-stage with fixed block counts and fixed summation trees:
// results are bitwise reproducible run to run.
#include <algorithm>

#include <cooperative_groups.h>

#include "kernels.h"

namespace wcmg {

constexpr int RED_T = 256;
// Blocks along the vector of a two-stage reduction: about 8 elements per thread
// for long vectors, but never fewer CTAs (over all `others` = rhs x chunks) than
// ~4 per SM while every thread still has an element: short coarse vectors are
// spread over the GPU instead of a dozen CTAs.  At most 608 (partial buffers).
static inline int red_blocks(long long n, long long others = 1) {
  const long long per8 = (n + 8 * RED_T - 1) / (8 * RED_T);
  const long long per1 = (n + RED_T - 1) / RED_T;
  const long long want = (4 * 152 + others - 1) / others;
  long long b = std::min(std::max(per8, want), per1);
  return (int)(b < 1 ? 1 : (b > 608 ? 608 : b));
}

template <typename A, typename B>
__global__ void k_convert(cplx<B>* __restrict__ out, const cplx<A>* __restrict__ in, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) out[i] = from_c64<B>(to_c64(in[i]));
}
template <typename A, typename B>
void launch_convert(cplx<B>* out, const cplx<A>* in, long long n, cudaStream_t st) {
  k_convert<A, B><<<nblk(n, 256), 256, 0, st>>>(out, in, n);
  WCMG_LAUNCH_CHECK();
}

// ---- dot / norm ----
template <typename R>
__global__ void __launch_bounds__(RED_T) k_dot_partial(double2* __restrict__ partial, const cplx<R>* __restrict__ a,
                                                       const cplx<R>* __restrict__ b, long long n) {
  __shared__ double2 scratch[RED_T / 32];
  __shared__ double2 red[1];
  const int r = blockIdx.y;
  a += (long long)r * n;
  b += (long long)r * n;
  cplx<R> acc = czero<R>();
  for (long long i = blockIdx.x * (long long)RED_T + threadIdx.x; i < n; i += (long long)gridDim.x * RED_T)
    cjmac(acc, a[i], b[i]);
  const R v[2] = {acc.x, acc.y};
  double* sd = reinterpret_cast<double*>(scratch);
  double* rd = reinterpret_cast<double*>(red);
  block_sum_mixed<R, 2>(v, sd, rd);
  if (threadIdx.x == 0) partial[(long long)r * gridDim.x + blockIdx.x] = make_double2(rd[0], rd[1]);
}
template <typename R>
__global__ void __launch_bounds__(RED_T) k_norm_partial(double* __restrict__ partial, const cplx<R>* __restrict__ a,
                                                        long long n) {
  __shared__ double scratch[RED_T / 32];
  __shared__ double red[1];
  const int r = blockIdx.y;
  a += (long long)r * n;
  R acc = 0;
  for (long long i = blockIdx.x * (long long)RED_T + threadIdx.x; i < n; i += (long long)gridDim.x * RED_T)
    acc += cnorm2(a[i]);
  const R v[1] = {acc};
  block_sum_mixed<R, 1>(v, scratch, red);
  if (threadIdx.x == 0) partial[(long long)r * gridDim.x + blockIdx.x] = red[0];
}
// out[r * ldo + i] = sum_{b < count} partial[r * pr + i * pi + b]  (grid: r = x, i = y)
// lim (nullable): rows i >= *lim + ladd are skipped (a device-side Arnoldi step count).
template <typename T>
__global__ void __launch_bounds__(RED_T) k_final(T* __restrict__ out, const T* __restrict__ partial, int count,
                                                 long long pr, long long pi, int ldo, const int* __restrict__ lim = nullptr,
                                                 int ladd = 0) {
  __shared__ T scratch[RED_T / 32];
  __shared__ T red[1];
  const int r = blockIdx.x, i = blockIdx.y;
  if (lim && i >= *lim + ladd) return;  // uniform per block
  const T* p = partial + r * pr + i * pi;
  T acc;
  memset(&acc, 0, sizeof(T));
  for (int b = threadIdx.x; b < count; b += RED_T) acc += p[b];
  block_sum_many<T>(&acc, 1, scratch, red);
  if (threadIdx.x == 0) out[(long long)r * ldo + i] = red[0];
}

template <typename R>
void launch_dot(double2* out, const cplx<R>* a, const cplx<R>* b, long long n, int nrhs, double2* partial,
                cudaStream_t st) {
  const int nb = red_blocks(n, nrhs);
  k_dot_partial<R><<<dim3(nb, nrhs), RED_T, 0, st>>>(partial, a, b, n);
  k_final<double2><<<dim3(nrhs, 1), RED_T, 0, st>>>(out, partial, nb, nb, 0, 1);
  ++launch_counter();
  WCMG_LAUNCH_CHECK();
}
template <typename R>
void launch_norm2(double* out, const cplx<R>* a, long long n, int nrhs, double* partial, cudaStream_t st) {
  const int nb = red_blocks(n, nrhs);
  k_norm_partial<R><<<dim3(nb, nrhs), RED_T, 0, st>>>(partial, a, n);
  k_final<double><<<dim3(nrhs, 1), RED_T, 0, st>>>(out, partial, nb, nb, 0, 1);
  ++launch_counter();
  WCMG_LAUNCH_CHECK();
}

// ---- Gram-Schmidt of an Arnoldi step: classical, twice ----
// h1 = V^dag w, w1 = w - V h1, h2 = V^dag w1, w2 = w1 - V h2 and ||w2||^2: four sweeps over the
// basis, bound by HBM.  The second projection has to be formed from w1 itself: what the first
// pass leaves of V in w1 is mostly the rounding of h1 and of the update, u |w| of |w1|, which
// h1 - (V^dag V) h1 (two sweeps fewer) does not contain.  With |w1| / |w| = 0.03 in FP32 that
// form left 7e-6 to 1e-4 of V in the new basis vector, two explicit passes 1e-7.
constexpr int MD_K = 8;
constexpr int GS_MAXK = 80;  // basis vectors (restart <= 64)
// <V_i, w> in chunks of 8 basis vectors
template <typename R>
__global__ void __launch_bounds__(RED_T) k_multidot_partial(double2* __restrict__ partial,
                                                            const cplx<R>* __restrict__ basis, long long bstride,
                                                            int k, const cplx<R>* __restrict__ w, long long n,
                                                            int nchunk, const int* __restrict__ kdev, int kadd,
                                                            int vec2) {
  __shared__ double2 scratch[(RED_T / 32) * MD_K];
  // chunks of basis vectors fastest in the grid: CTAs running together read the same w
  const int i0 = (blockIdx.x % nchunk) * MD_K, blk = blockIdx.x / nchunk, nblk_ = gridDim.x / nchunk;
  const int r = blockIdx.y, kpad = nchunk * MD_K;
  if (kdev) k = *kdev + kadd;
  if (i0 >= k) return;  // uniform per block
  const long long off = (long long)r * n;
  cplx<R> acc[MD_K];
#pragma unroll
  for (int q = 0; q < MD_K; ++q) acc[q] = czero<R>();
  if constexpr (sizeof(R) == 4) {
    if (vec2) {  // two complex entries per 16-byte load (n, bstride even; 16-byte aligned fields)
      const float4* w4 = reinterpret_cast<const float4*>(w + off);
      const long long n2 = n >> 1;
      for (long long e = blk * (long long)RED_T + threadIdx.x; e < n2; e += (long long)nblk_ * RED_T) {
        const float4 x = w4[e];
#pragma unroll
        for (int q = 0; q < MD_K; ++q)
          if (i0 + q < k) {
            const float4 v = reinterpret_cast<const float4*>(basis + (i0 + q) * bstride + off)[e];
            cjmac(acc[q], make_float2(v.x, v.y), make_float2(x.x, x.y));
            cjmac(acc[q], make_float2(v.z, v.w), make_float2(x.z, x.w));
          }
      }
    }
  }
  if (sizeof(R) == 8 || !vec2)
    for (long long e = blk * (long long)RED_T + threadIdx.x; e < n; e += (long long)nblk_ * RED_T) {
      const cplx<R> x = w[off + e];
#pragma unroll
      for (int q = 0; q < MD_K; ++q)
        if (i0 + q < k) cjmac(acc[q], basis[(i0 + q) * bstride + off + e], x);
    }
  // warp sums in the working precision (one transposing butterfly for the 8 values),
  // then FP64 across the warps of the CTA and across CTAs
  static_assert(MD_K == 8, "transposing warp reduction of 8 values");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  warp_sum8_transposed(acc, lane);
  if ((lane & 3) == 0) scratch[warp * MD_K + warp_sum8_index(lane)] = to_c64(acc[0]);
  __syncthreads();
  if (threadIdx.x < MD_K && i0 + threadIdx.x < k) {
    double2 t = scratch[threadIdx.x];
    for (int u = 1; u < RED_T / 32; ++u) t += scratch[u * MD_K + threadIdx.x];
    partial[((long long)r * kpad + i0 + threadIdx.x) * nblk_ + blk] = t;
  }
}
// 16-byte accesses to the basis and w
template <typename R>
static int basis_vec2(const cplx<R>* basis, long long bstride, const cplx<R>* w, long long n) {
  return sizeof(R) == 4 && n % 2 == 0 && bstride % 2 == 0 && reinterpret_cast<uintptr_t>(basis) % 16 == 0 &&
         reinterpret_cast<uintptr_t>(w) % 16 == 0;
}
template <typename R>
static void multidot(double2* out, const cplx<R>* basis, long long bstride, int k, int ldo, const cplx<R>* w,
                     long long n, int nrhs, double2* partial, cudaStream_t st, const int* kdev, int kadd) {
  const int nchunk = (k + MD_K - 1) / MD_K, kpad = nchunk * MD_K;
  const int nb = red_blocks(n, nrhs);  // independent of k: a captured graph sums in the same order
  k_multidot_partial<R><<<dim3(nb * nchunk, nrhs), RED_T, 0, st>>>(partial, basis, bstride, k, w, n, nchunk, kdev,
                                                                   kadd, basis_vec2<R>(basis, bstride, w, n));
  WCMG_LAUNCH_CHECK();
  k_final<double2><<<dim3(nrhs, k), RED_T, 0, st>>>(out, partial, nb, (long long)kpad * nb, nb, ldo, kdev, kadd);
  WCMG_LAUNCH_CHECK();
}

// w -= V h and ||w||^2 in one pass: AN_T threads x at most 608 CTAs per rhs stride over the
// field (two entries per 16-byte access when vec2), four basis vectors in flight.
constexpr int AN_T = 512;
template <typename R>
__global__ void __launch_bounds__(AN_T) k_project_norm(cplx<R>* __restrict__ w, const cplx<R>* __restrict__ basis,
                                                       long long bstride, int k, const double2* __restrict__ h, int ld,
                                                       long long n, double* __restrict__ partial,
                                                       const int* __restrict__ kdev, int kadd, int vec2) {
  __shared__ cplx<R> cf[GS_MAXK];
  __shared__ double scratch[AN_T / 32];
  __shared__ double red[1];
  const int r = blockIdx.y;
  if (kdev) k = min(*kdev + kadd, k);
  for (int i = threadIdx.x; i < k; i += AN_T) {
    const double2 c = h[(long long)r * ld + i];
    cf[i] = cmk(R(-c.x), R(-c.y));
  }
  __syncthreads();
  w += (long long)r * n;
  basis += (long long)r * n;
  R nn = 0;
  if (sizeof(R) == 4 && vec2) {
    const long long n2 = n >> 1;
    for (long long e = blockIdx.x * (long long)AN_T + threadIdx.x; e < n2; e += (long long)gridDim.x * AN_T) {
      float4 x = reinterpret_cast<float4*>(w)[e];
      float2 lo = make_float2(x.x, x.y), hi = make_float2(x.z, x.w);
#pragma unroll 4
      for (int i = 0; i < k; ++i) {
        const float4 v = reinterpret_cast<const float4*>(basis + i * bstride)[e];
        const float2 c = make_float2((float)cf[i].x, (float)cf[i].y);
        cmac(lo, c, make_float2(v.x, v.y));
        cmac(hi, c, make_float2(v.z, v.w));
      }
      reinterpret_cast<float4*>(w)[e] = make_float4(lo.x, lo.y, hi.x, hi.y);
      nn += (R)(cnorm2(lo) + cnorm2(hi));
    }
  } else {
    for (long long e = blockIdx.x * (long long)AN_T + threadIdx.x; e < n; e += (long long)gridDim.x * AN_T) {
      cplx<R> x = w[e];
#pragma unroll 4
      for (int i = 0; i < k; ++i) cmac(x, cf[i], basis[i * bstride + e]);
      w[e] = x;
      nn += cnorm2(x);
    }
  }
  const R v[1] = {nn};
  block_sum_mixed<R, 1>(v, scratch, red);
  if (threadIdx.x == 0) partial[(long long)r * gridDim.x + blockIdx.x] = red[0];
}
template <typename R>
static int project_norm(double* partial, cplx<R>* w, const cplx<R>* basis, long long bstride, int k, const double2* h,
                        int ld, long long n, int nrhs, cudaStream_t st, const int* kdev, int kadd) {
  const int vec2 = basis_vec2<R>(basis, bstride, w, n);
  const long long per = (long long)AN_T * (vec2 ? 2 : 1);
  const int nb = (int)std::max(1LL, std::min(608LL, (n + per - 1) / per));
  k_project_norm<R><<<dim3(nb, nrhs), AN_T, 0, st>>>(w, basis, bstride, k, h, ld, n, partial, kdev, kadd, vec2);
  WCMG_LAUNCH_CHECK();
  return nb;
}

template <typename R>
__global__ void k_multiaxpy(cplx<R>* __restrict__ w, const cplx<R>* __restrict__ basis, long long bstride, int k,
                           const double2* __restrict__ coef, int ldc, double sign, long long n,
                           const int* __restrict__ kdev, int kadd) {
  __shared__ cplx<R> cf[GS_MAXK];
  const int r = blockIdx.y;
  if (kdev) k = min(*kdev + kadd, k);
  for (int i = threadIdx.x; i < k; i += blockDim.x) {
    const double2 c = coef[(long long)r * ldc + i];
    cf[i] = cmk(R(sign * c.x), R(sign * c.y));
  }
  __syncthreads();
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const long long off = (long long)r * n + e;
  cplx<R> acc = w[off];
  for (int i = 0; i < k; ++i) cmac(acc, cf[i], basis[i * bstride + off]);
  w[off] = acc;
}
template <typename R>
void launch_multiaxpy(cplx<R>* w, const cplx<R>* basis, long long bstride, int k, const double2* coef, int ldc,
                      double sign, long long n, int nrhs, cudaStream_t st, const int* kdev, int kadd) {
  if (k <= 0) return;
  if (k > GS_MAXK) throw Error(-1, "multiaxpy supports k <= 80");
  k_multiaxpy<R><<<dim3(nblk(n, 256), nrhs), 256, 0, st>>>(w, basis, bstride, k, coef, ldc, sign, n, kdev, kadd);
  WCMG_LAUNCH_CHECK();
}

template <typename R>
int launch_gram_schmidt(double2* h1, double2* h2, double* norm_partial, cplx<R>* w, const cplx<R>* basis,
                        long long bstride, int k, int ld, long long n, int nrhs, double2* partial, cudaStream_t st,
                        const int* kdev, int kadd) {
  if (k > GS_MAXK) throw Error(-1, "Gram-Schmidt supports k <= 80");
  multidot<R>(h1, basis, bstride, k, ld, w, n, nrhs, partial, st, kdev, kadd);
  launch_multiaxpy<R>(w, basis, bstride, k, h1, ld, -1.0, n, nrhs, st, kdev, kadd);
  multidot<R>(h2, basis, bstride, k, ld, w, n, nrhs, partial, st, kdev, kadd);
  return project_norm<R>(norm_partial, w, basis, bstride, k, h2, ld, n, nrhs, st, kdev, kadd);
}

template <typename R>
__global__ void k_axpby(cplx<R>* __restrict__ y, R a, const cplx<R>* __restrict__ x, R b, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) y[i] = a * x[i] + b * y[i];
}
template <typename R>
void launch_axpby(cplx<R>* y, double a, const cplx<R>* x, double b, long long n, int nrhs, cudaStream_t st) {
  const long long N = n * nrhs;
  k_axpby<R><<<nblk(N, 256), 256, 0, st>>>(y, (R)a, x, (R)b, N);
  WCMG_LAUNCH_CHECK();
}

template <typename R>
__global__ void k_scale_dev(cplx<R>* y, const cplx<R>* x, const double* __restrict__ s,
                            int inv_sqrt, long long n, const int* __restrict__ ydev, int yadd, long long ystride,
                            cplx<R>* __restrict__ y2) {
  __shared__ R f_s;
  const int r = blockIdx.y;
  if (ydev) y += (long long)(*ydev + yadd) * ystride;
  if (threadIdx.x == 0) {
    double f = s[r];
    if (inv_sqrt) f = f > 0.0 ? 1.0 / sqrt(f) : 0.0;
    f_s = (R)f;
  }
  __syncthreads();
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= n) return;
  const cplx<R> v = f_s * x[(long long)r * n + e];
  y[(long long)r * n + e] = v;
  if (y2) y2[(long long)r * n + e] = v;
}
template <typename R>
void launch_scale_dev(cplx<R>* y, const cplx<R>* x, const double* s, int inv_sqrt, long long n, int nrhs,
                      cudaStream_t st, const int* ydev, int yadd, long long ystride, cplx<R>* y2) {
  k_scale_dev<R><<<dim3(nblk(n, 256), nrhs), 256, 0, st>>>(y, x, s, inv_sqrt, n, ydev, yadd, ystride, y2);
  WCMG_LAUNCH_CHECK();
}

// ---- minimal-residual updates ----
// Bound by HBM: what counts is how often the fields are read and written.  A pair of steps
// k, k + 1 shares one update of x: x += alpha_k r_k + alpha_{k+1} r_{k+1}, with r_{k+1}
// written over p_k so that r_k survives.  Four steps from x = 0 then move 15 fields (17
// with one update of x per step), and 16 when they are added to a given x (18, and 3 more
// for a separate addition).  16-byte accesses: n is even on every level and the fields
// start on 16 bytes, so an FP32 thread takes two entries.
template <typename R> struct MrVec;
template <> struct MrVec<double> { using type = double2; static constexpr int n = 1; };
template <> struct MrVec<float> { using type = float4; static constexpr int n = 2; };
__device__ __forceinline__ void vmac(double2& a, double2 s, double2 v) { cmac(a, s, v); }
__device__ __forceinline__ void vmac(float4& a, float2 s, float4 v) {
  float2 lo = make_float2(a.x, a.y), hi = make_float2(a.z, a.w);
  cmac(lo, s, make_float2(v.x, v.y));
  cmac(hi, s, make_float2(v.z, v.w));
  a = make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ double2 vsub(double2 a, double2 s, double2 v) { return a - cmul(s, v); }
__device__ __forceinline__ float4 vsub(float4 a, float2 s, float4 v) {
  const float2 lo = make_float2(a.x, a.y) - cmul(s, make_float2(v.x, v.y));
  const float2 hi = make_float2(a.z, a.w) - cmul(s, make_float2(v.z, v.w));
  return make_float4(lo.x, lo.y, hi.x, hi.y);
}
template <typename V> __device__ __forceinline__ V vzero() {
  V v;
  memset(&v, 0, sizeof(V));
  return v;
}
template <typename R>
__device__ __forceinline__ cplx<R> mr_alpha(const double2* pr, const double* pp, int q) {
  const double d = pp[q];
  return d != 0.0 ? cmk((R)(pr[q].x / d), (R)(pr[q].y / d)) : czero<R>();
}

template <typename R, bool X_ZERO, bool R_NEXT>
__global__ void k_mr_update(cplx<R>* __restrict__ x, cplx<R>* __restrict__ r, const cplx<R>* __restrict__ p,
                            const double2* __restrict__ pr, const double* __restrict__ pp, long long nv) {
  using V = typename MrVec<R>::type;
  __shared__ cplx<R> a_s;
  const int q = blockIdx.y;
  if (threadIdx.x == 0) a_s = mr_alpha<R>(pr, pp, q);
  __syncthreads();
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= nv) return;
  const long long o = (long long)q * nv + e;
  const V rv = reinterpret_cast<V*>(r)[o];
  V xv = X_ZERO ? vzero<V>() : reinterpret_cast<V*>(x)[o];
  vmac(xv, a_s, rv);
  reinterpret_cast<V*>(x)[o] = xv;
  if (R_NEXT) reinterpret_cast<V*>(r)[o] = vsub(rv, a_s, reinterpret_cast<const V*>(p)[o]);
}
template <typename R>
__global__ void k_mr_residual(cplx<R>* __restrict__ p, const cplx<R>* __restrict__ r, const double2* __restrict__ pr,
                              const double* __restrict__ pp, long long nv) {
  using V = typename MrVec<R>::type;
  __shared__ cplx<R> a_s;
  const int q = blockIdx.y;
  if (threadIdx.x == 0) a_s = mr_alpha<R>(pr, pp, q);
  __syncthreads();
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= nv) return;
  const long long o = (long long)q * nv + e;
  V* pv = reinterpret_cast<V*>(p) + o;
  *pv = vsub(reinterpret_cast<const V*>(r)[o], a_s, *pv);
}
template <typename R, bool X_ZERO, bool R_NEXT>
__global__ void k_mr_pair(cplx<R>* __restrict__ x, const cplx<R>* __restrict__ r0, cplx<R>* __restrict__ r1,
                          const cplx<R>* __restrict__ p1, const double2* __restrict__ pr0,
                          const double* __restrict__ pp0, const double2* __restrict__ pr1,
                          const double* __restrict__ pp1, long long nv) {
  using V = typename MrVec<R>::type;
  __shared__ cplx<R> a_s[2];
  const int q = blockIdx.y;
  if (threadIdx.x == 0) a_s[0] = mr_alpha<R>(pr0, pp0, q);
  if (threadIdx.x == 32) a_s[1] = mr_alpha<R>(pr1, pp1, q);
  __syncthreads();
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= nv) return;
  const long long o = (long long)q * nv + e;
  const V rv = reinterpret_cast<V*>(r1)[o];
  V xv = X_ZERO ? vzero<V>() : reinterpret_cast<V*>(x)[o];
  vmac(xv, a_s[0], reinterpret_cast<const V*>(r0)[o]);
  vmac(xv, a_s[1], rv);
  reinterpret_cast<V*>(x)[o] = xv;
  if (R_NEXT) reinterpret_cast<V*>(r1)[o] = vsub(rv, a_s[1], reinterpret_cast<const V*>(p1)[o]);
}

template <typename R>
static long long mr_vectors(long long n) {
  if (n % MrVec<R>::n) throw Error(-1, "MR update: odd field length");
  return n / MrVec<R>::n;
}
template <typename R>
void launch_mr_update(cplx<R>* x, cplx<R>* r, const cplx<R>* p, const double2* pr, const double* pp, long long n,
                      int nrhs, cudaStream_t st, bool x_zero, bool r_next) {
  const long long nv = mr_vectors<R>(n);
  const dim3 grid(nblk(nv, 256), nrhs);
  if (x_zero && r_next) k_mr_update<R, true, true><<<grid, 256, 0, st>>>(x, r, p, pr, pp, nv);
  else if (x_zero) k_mr_update<R, true, false><<<grid, 256, 0, st>>>(x, r, p, pr, pp, nv);
  else if (r_next) k_mr_update<R, false, true><<<grid, 256, 0, st>>>(x, r, p, pr, pp, nv);
  else k_mr_update<R, false, false><<<grid, 256, 0, st>>>(x, r, p, pr, pp, nv);
  WCMG_LAUNCH_CHECK();
}
template <typename R>
void launch_mr_residual(cplx<R>* p, const cplx<R>* r, const double2* pr, const double* pp, long long n, int nrhs,
                        cudaStream_t st) {
  const long long nv = mr_vectors<R>(n);
  k_mr_residual<R><<<dim3(nblk(nv, 256), nrhs), 256, 0, st>>>(p, r, pr, pp, nv);
  WCMG_LAUNCH_CHECK();
}
template <typename R>
void launch_mr_pair(cplx<R>* x, const cplx<R>* r0, cplx<R>* r1, const cplx<R>* p1, const double2* pr0,
                    const double* pp0, const double2* pr1, const double* pp1, long long n, int nrhs, cudaStream_t st,
                    bool x_zero, bool r_next) {
  const long long nv = mr_vectors<R>(n);
  const dim3 grid(nblk(nv, 256), nrhs);
#define WCMG_MP(XZ, RN) k_mr_pair<R, XZ, RN><<<grid, 256, 0, st>>>(x, r0, r1, p1, pr0, pp0, pr1, pp1, nv)
  if (x_zero && r_next) WCMG_MP(true, true);
  else if (x_zero) WCMG_MP(true, false);
  else if (r_next) WCMG_MP(false, true);
  else WCMG_MP(false, false);
#undef WCMG_MP
  WCMG_LAUNCH_CHECK();
}

__global__ void k_add_widened(double2* __restrict__ y, const float2* __restrict__ x, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) y[i] += to_c64(x[i]);
}
void launch_add_widened(double2* y, const float2* x, long long n, cudaStream_t st) {
  k_add_widened<<<nblk(n, 256), 256, 0, st>>>(y, x, n);
  WCMG_LAUNCH_CHECK();
}

template <typename R>
__global__ void k_mask_rhs(cplx<R>* __restrict__ x, const int* __restrict__ mask, long long n) {
  const int r = blockIdx.y;
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e < n && mask[r]) x[(long long)r * n + e] = czero<R>();
}
template <typename R>
void launch_mask_rhs(cplx<R>* x, const int* mask, long long n, int nrhs, cudaStream_t st) {
  k_mask_rhs<R><<<dim3(nblk(n, 256), nrhs), 256, 0, st>>>(x, mask, n);
  WCMG_LAUNCH_CHECK();
}

// dst[o * dmul + i] = src[o * smul + i], o = *idx (0 when idx is null): the copy of
// one Krylov basis slot selected on the device.
template <typename R>
__global__ void k_copy_idx(cplx<R>* __restrict__ dst, const cplx<R>* __restrict__ src, long long n,
                           const int* __restrict__ idx, long long dmul, long long smul) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const long long o = idx ? *idx : 0;
  dst[o * dmul + i] = src[o * smul + i];
}
template <typename R>
void launch_copy_idx(cplx<R>* dst, const cplx<R>* src, long long n, const int* idx, long long dmul, long long smul,
                     cudaStream_t st) {
  if (n <= 0) return;
  k_copy_idx<R><<<nblk(n, 256), 256, 0, st>>>(dst, src, n, idx, dmul, smul);
  WCMG_LAUNCH_CHECK();
}
template <typename R>
__global__ void k_fill_zero(cplx<R>* x, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) x[i] = czero<R>();
}
template <typename R>
void launch_fill_zero(cplx<R>* x, long long n, cudaStream_t st) {
  if (n <= 0) return;
  k_fill_zero<R><<<nblk(n, 256), 256, 0, st>>>(x, n);
  WCMG_LAUNCH_CHECK();
}

// ---- (F)GMRES bookkeeping (K8), one thread per rhs, FP64 ----
// Complex Givens rotation G = [[c, s], [-conj(s), c]], c real, with
// G [a, b]^T = [rho, 0]^T.
__device__ void givens(double2 a, double2 b, double& c, double2& s, double2& rho) {
  const double aa = sqrt(cnorm2(a));
  if (aa == 0.0) { c = 0.0; s = make_double2(1, 0); rho = b; return; }
  const double r = sqrt(cnorm2(a) + cnorm2(b));
  const double2 ph = make_double2(a.x / aa, a.y / aa);
  c = aa / r;
  s = (1.0 / r) * cmul(ph, conjg(b));
  rho = r * ph;
}

// init: the first cycle from x = 0, whose residual is b: also bnorm = beta and done = 0
__global__ void k_gmres_start(GmresState S, const double* __restrict__ nrm2, double tol, int nrhs,
                              double* __restrict__ inv_beta, bool init) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nrhs) return;
  const double beta = sqrt(nrm2[r]);
  const int m = S.m;
  if (init) {
    S.bnorm[r] = beta;
    S.done[r] = 0;
  }
  for (int i = 0; i <= m; ++i) S.g[(long long)r * (m + 1) + i] = make_double2(0, 0);
  S.g[(long long)r * (m + 1)] = make_double2(beta, 0);
  S.resid[r] = beta;
  S.jdone[r] = 0;
  const bool go = (init || !S.done[r]) && beta > tol * S.bnorm[r] && beta > 0.0;
  S.active[r] = go ? 1 : 0;
  inv_beta[r] = go ? 1.0 / beta : 0.0;
}
// bnorm = sqrt(nrm2), done = 0 (before the restart loop)
__global__ void k_gmres_init(GmresState S, const double* __restrict__ nrm2, int nrhs) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nrhs) return;
  S.bnorm[r] = sqrt(nrm2[r]);
  S.done[r] = 0;
}

// the state of one rhs
__device__ __forceinline__ GmresState gmres_of(GmresState S, int r) {
  const long long m = S.m;
  S.H += r * (m + 1) * m;
  S.cs += r * m;
  S.sn += r * m;
  S.g += r * (m + 1);
  S.y += r * m;
  S.hnorm += r;
  S.bnorm += r;
  S.resid += r;
  S.active += r;
  S.jdone += r;
  S.done += r;
  return S;
}

// Column j of the Hessenberg matrix of one rhs: the earlier rotations on hcol (j + 1 entries,
// overwritten; cs, sn: the rotations of columns 0 .. j - 1, all in shared memory), a new
// complex Givens rotation that removes ||w|| = sqrt(hn2), and the recurrence residual.
__device__ void gmres_rotate(GmresState S, int j, double2* hcol, const double* cs, const double2* sn, double hn2,
                             double tol, int final_done) {
  const int m = S.m;
  for (int i = 0; i < j; ++i) {
    const double2 a = hcol[i], b = hcol[i + 1];
    S.H[i * m + j] = cs[i] * a + cmul(sn[i], b);
    hcol[i + 1] = cs[i] * b - cmul(conjg(sn[i]), a);
  }
  double c; double2 s, rho;
  givens(hcol[j], make_double2(sqrt(hn2), 0), c, s, rho);
  S.cs[j] = c; S.sn[j] = s;
  S.H[j * m + j] = rho;
  S.H[(j + 1) * m + j] = make_double2(0, 0);
  const double2 gj = S.g[j];
  S.g[j + 1] = -cmul(conjg(s), gj);
  S.g[j] = c * gj;
  const double res = sqrt(cnorm2(S.g[j + 1]));
  S.resid[0] = res;
  S.jdone[0] = j + 1;
  if (res <= tol * S.bnorm[0]) {
    S.active[0] = 0;
    if (final_done) S.done[0] = 1;
  }
}

// One CTA per rhs: ||w||^2 from the `count` partials of k_project_norm, then the rotation with
// the column and the earlier rotations fetched in parallel (12 us, a launch of 4 us for the final
// sum less than the rotation by one thread from global memory, which took 12 us as well).
__global__ void __launch_bounds__(RED_T) k_gmres_step(GmresState S, int j, const double2* __restrict__ h1,
                                                      const double2* __restrict__ h2,
                                                      const double* __restrict__ partial, int count, double tol,
                                                      int final_done, double* __restrict__ inv_h,
                                                      const int* __restrict__ jdev) {
  __shared__ double2 hcol[65], sn[65];
  __shared__ double cs[65], scratch[RED_T / 32], red[1];
  const int r = blockIdx.x;
  if (jdev) j = *jdev;
  S = gmres_of(S, r);
  const bool act = S.active[0] != 0;
  if (threadIdx.x <= j) {
    const long long i = (long long)r * (S.m + 1) + threadIdx.x;
    hcol[threadIdx.x] = h1[i] + h2[i];
  }
  if (threadIdx.x < j) {
    cs[threadIdx.x] = S.cs[threadIdx.x];
    sn[threadIdx.x] = S.sn[threadIdx.x];
  }
  double acc = 0.0;
  for (int b = threadIdx.x; b < count; b += RED_T) acc += partial[(long long)r * count + b];
  block_sum_many<double>(&acc, 1, scratch, red);
  if (threadIdx.x == 0) {
    const double hn2 = red[0], nrm = sqrt(hn2);
    inv_h[r] = act && nrm > 0.0 ? 1.0 / nrm : 0.0;
    if (act) gmres_rotate(S, j, hcol, cs, sn, hn2, tol, final_done);
  }
}

// ---- fused Arnoldi step for short vectors (one rhs) ----
// Everything of one (F)GMRES Arnoldi step after the operator application, for
// vectors short enough that a single thread-block cluster streams them from L2:
// both classical Gram-Schmidt passes h1 = V^dag w, w -= V h1, h2 = V^dag w,
// w -= V h2, the norm ||w||^2, the Givens update of Hessenberg column j and
// V_{j+1} = w / ||w||.  CTA c of the C-CTA cluster owns a contiguous range of the
// vector.  Bound by latency, so: the warps share the basis vectors of a sweep evenly (warp
// sums only, no block barrier per chunk of vectors), the updated elements stay in registers
// until the norm is known (and in w for the second sweep), the rotations are requested before
// the first sweep, remote sums are read all at once, FP64 work is left to as few warps as it
// has values (a warp's FP64 instruction takes 16 cycles of the SM's unit), and the new
// rotation runs from shared memory while the cluster writes V_{j+1}.  Partial sums are
// exchanged through distributed shared memory and every CTA adds the C partials in the same
// order, so all CTAs hold identical coefficients.  24.6k entries, 16 CTAs, in a solve under ncu:
// 36 us with one warp per basis vector and every thread adding the remote norms in FP64, 20 us
// now (registers for one CTA per SM: under the default 64 the elements spilled).
constexpr int AC_T = 512, AC_MAXK = 65, AC_W = AC_T / 32;
constexpr int AC_EL = 16;  // most elements per thread

// sum over the cluster's ranks of one shared double2, all remote reads in flight
__device__ __forceinline__ double2 ac_cluster_sum(cooperative_groups::cluster_group& cl, double2* p, int C) {
  double2 v[16];
#pragma unroll
  for (int c = 0; c < 16; ++c) v[c] = c < C ? *cl.map_shared_rank(p, c) : make_double2(0, 0);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
#pragma unroll
    for (int c = 0; c < o; ++c) v[c] += v[c + o];
  return v[0];
}

// out[i] = this CTA's part of <V_i, w>, i < k: the 16 warps split into one group of P per basis
// vector (P = 16, 8, .. 1: as many as there are vectors for), each warp a P-th of the range.
// pw: scratch, one sum per warp.  Complete after the next barrier of the cluster.
template <typename R>
__device__ __forceinline__ void ac_sweep(double2* out, cplx<R>* pw, const cplx<R>* V, long long bstride,
                                         const cplx<R>* w, int cnt, int k) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int P = k == 1 ? 16 : k == 2 ? 8 : k <= 4 ? 4 : k <= 8 ? 2 : 1;
  for (int i = warp / P; i < k; i += AC_W / P) {
    const cplx<R>* vi = V + (long long)i * bstride;
    cplx<R> acc = czero<R>();
#pragma unroll 8
    for (int e = lane + 32 * (warp % P); e < cnt; e += 32 * P) cjmac(acc, vi[e], w[e]);
    const cplx<R> t = warp_sum(acc);
    if (lane == 0) {
      if (P == 1) out[i] = to_c64(t);
      else pw[warp] = t;
    }
  }
  if (P > 1) {
    __syncthreads();
    if (threadIdx.x < k) {
      double2 t = to_c64(pw[threadIdx.x * P]);
      for (int u = 1; u < P; ++u) t += to_c64(pw[threadIdx.x * P + u]);
      out[threadIdx.x] = t;
    }
  }
}

// x -= V c over the CTA's range, a thread's elements in registers: its loads of all elements
// per basis vector are in flight together
template <typename R, int NE>
__device__ __forceinline__ void ac_update(cplx<R> (&x)[NE], const cplx<R>* V, long long bstride, const cplx<R>* cf,
                                          int cnt, int k) {
  constexpr int UI = NE >= 8 ? 1 : 8 / NE;
#pragma unroll UI
  for (int i = 0; i < k; ++i) {
    const cplx<R>* v = V + (long long)i * bstride;
    const cplx<R> c = cf[i];
#pragma unroll
    for (int u = 0; u < NE; ++u) {
      const int e = threadIdx.x + u * AC_T;
      if (e < cnt) cnmac(x[u], c, v[e]);
    }
  }
}

// NE: elements per thread (power of two; the vector has at most C x AC_T x NE entries)
template <typename R, int NE>
__global__ void __launch_bounds__(AC_T, 1) k_arnoldi_cluster(cplx<R>* Vb, long long bstride, cplx<R>* w, long long n,
                                                          GmresState S, int j, const int* __restrict__ jdev,
                                                          double tol, int final_done, cplx<R>* __restrict__ vnext) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), crank = (int)cl.block_rank();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ double2 pA[2][AC_MAXK];  // this CTA's sums of the two passes (read by the whole cluster)
  __shared__ double2 pN;
  __shared__ cplx<R> pw[AC_W], cf[AC_MAXK];
  __shared__ double2 hcol[AC_MAXK], snn[AC_MAXK];
  __shared__ double csn[AC_MAXK];
  __shared__ R wsum[AC_W];
  __shared__ double hn_s;
  __shared__ R inv_s;
  if (jdev) j = *jdev;
  const int k = j + 1;
  const bool act = S.active[0] != 0;  // before this step (CTA 0 may change it below)
  const int per = (int)((n + C - 1) / C);
  const int e0 = crank * per, cnt = max(0, min(per, (int)n - e0));
  if (crank == 0)
    for (int i = threadIdx.x; i < j; i += AC_T) {
      csn[i] = S.cs[i];
      snn[i] = S.sn[i];
    }
  const cplx<R>* V = Vb + e0;
  cplx<R>* wv = w + e0;
  cplx<R> x[NE];
#pragma unroll
  for (int u = 0; u < NE; ++u) {
    const int e = threadIdx.x + u * AC_T;
    x[u] = e < cnt ? wv[e] : czero<R>();
  }
  for (int pass = 0; pass < 2; ++pass) {
    ac_sweep<R>(pA[pass], pw, V, bstride, wv, cnt, k);
    cl.sync();
    if (threadIdx.x < k) {
      const double2 h = ac_cluster_sum(cl, pA[pass] + threadIdx.x, C);
      cf[threadIdx.x] = cmk(R(h.x), R(h.y));
      hcol[threadIdx.x] = pass == 0 ? h : hcol[threadIdx.x] + h;
    }
    __syncthreads();
    ac_update<R, NE>(x, V, bstride, cf, cnt, k);
    if (pass == 0) {
#pragma unroll
      for (int u = 0; u < NE; ++u) {
        const int e = threadIdx.x + u * AC_T;
        if (e < cnt) wv[e] = x[u];
      }
      __syncthreads();  // w is complete for every warp, and cf and pw are free
    }
  }
  // the norm: warp sums in R, the warps' in FP64
  R nn = 0;
#pragma unroll
  for (int u = 0; u < NE; ++u) nn += cnorm2(x[u]);
  nn = warp_sum(nn);
  if (lane == 0) wsum[warp] = nn;
  __syncthreads();
  if (warp == 0) {
    double t = lane < AC_W ? (double)wsum[lane] : 0.0;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) pN = make_double2(t, 0);
  }
  cl.sync();
  if (threadIdx.x == 0) {  // one thread: FP64 runs at two lanes per cycle on an SM
    const double hn2 = ac_cluster_sum(cl, &pN, C).x, h = sqrt(hn2);
    hn_s = hn2;
    inv_s = (R)(act && h > 0.0 ? 1.0 / h : 0.0);
  }
  __syncthreads();
  cl.barrier_arrive();  // done with the others' shared memory
  if (crank == 0 && threadIdx.x == AC_T - 32 && act) gmres_rotate(S, j, hcol, csn, snn, hn_s, tol, final_done);
  const R inv = inv_s;
  cplx<R>* vn = Vb + (long long)(j + 1) * bstride + e0;
#pragma unroll
  for (int u = 0; u < NE; ++u) {
    const int e = threadIdx.x + u * AC_T;
    if (e < cnt) {
      const cplx<R> t = inv * x[u];
      vn[e] = t;
      if (vnext) vnext[e0 + e] = t;
    }
  }
  cl.barrier_wait();  // no CTA leaves while another may still read its shared memory
}

static int arnoldi_cluster_size() {
  static int cached = -1;
  if (cached >= 0) return cached;
  cached = 0;
  for (int C : {16, 8}) {
    auto kern = k_arnoldi_cluster<float, AC_EL>;
    if (C > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(AC_T);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) == cudaSuccess && nclusters > 0) {
      cached = C;
      break;
    }
    cudaGetLastError();
  }
  return cached;
}

// The 16-CTA cluster reads the basis through 16 SMs only: it beats the seven
// whole-GPU launches it replaces for short vectors (the coarsest levels: 10^4 - 4 x 10^4
// entries) but not for fine-level ones (a 16^4 lattice, 7.9 x 10^5 entries: 300 us per
// step against about 60 us), so it takes vectors of at most 2^17 entries.
bool arnoldi_fused_ok(long long n, int nrhs, int m) {
  return nrhs == 1 && m + 1 <= AC_MAXK && n <= (1LL << 17) && arnoldi_cluster_size() > 0 &&
         (n + arnoldi_cluster_size() - 1) / arnoldi_cluster_size() <= AC_EL * AC_T;
}

template <typename R>
void launch_arnoldi_fused(cplx<R>* Vb, long long bstride, cplx<R>* w, long long n, const GmresState& S, int j,
                          const int* jdev, double tol, int final_done, cudaStream_t st, cplx<R>* vnext) {
  const int C = arnoldi_cluster_size();
  if (C <= 0) throw Error(-1, "no thread-block cluster available for the fused Arnoldi step");
  const long long per = ((n + C - 1) / C + AC_T - 1) / AC_T;  // elements per thread
  auto kern = per <= 1   ? k_arnoldi_cluster<R, 1>
              : per <= 2 ? k_arnoldi_cluster<R, 2>
              : per <= 4 ? k_arnoldi_cluster<R, 4>
              : per <= 8 ? k_arnoldi_cluster<R, 8>
                         : k_arnoldi_cluster<R, AC_EL>;
  if (C > 8) WCMG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(AC_T);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  WCMG_CUDA(cudaLaunchKernelEx(&cfg, kern, Vb, bstride, w, n, S, j, jdev, tol, final_done, vnext));
  WCMG_LAUNCH_CHECK();
}
template void launch_arnoldi_fused<float>(float2*, long long, float2*, long long, const GmresState&, int, const int*,
                                          double, int, cudaStream_t, float2*);
template void launch_arnoldi_fused<double>(double2*, long long, double2*, long long, const GmresState&, int,
                                           const int*, double, int, cudaStream_t, double2*);

// y = R^-1 g by columns, one warp per rhs: lane i holds the right-hand sides i and i + 32, R
// (its columns from the diagonal up) lies in shared memory, and the diagonal's reciprocals
// are formed at once (m = 20: 11 us with one thread walking through global memory, 8.6 us now).
__global__ void __launch_bounds__(32) k_gmres_solve_y(GmresState S) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* Rs = reinterpret_cast<double2*>(smem_raw);  // column k at k (k + 1) / 2
  S = gmres_of(S, blockIdx.x);
  const int m = S.m, jd = S.jdone[0], lane = threadIdx.x;
  for (int k = 0; k < jd; ++k)
    for (int i = lane; i <= k; i += 32) Rs[k * (k + 1) / 2 + i] = S.H[i * m + k];
  double2 t[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) t[u] = lane + 32 * u < jd ? S.g[lane + 32 * u] : make_double2(0, 0);
  __syncwarp();
  double2 inv[2];  // conj(d) / |d|^2, or 0
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int k = lane + 32 * u;
    const double2 d = k < jd ? Rs[k * (k + 1) / 2 + k] : make_double2(0, 0);
    const double dd = cnorm2(d);
    inv[u] = dd > 0.0 ? (1.0 / dd) * conjg(d) : make_double2(0, 0);
  }
  for (int k = jd - 1; k >= 0; --k) {
    const double2* col = Rs + k * (k + 1) / 2;
    double2 y = k < 32 ? cmul(inv[0], t[0]) : cmul(inv[1], t[1]);
    y = make_double2(__shfl_sync(0xffffffffu, y.x, k & 31), __shfl_sync(0xffffffffu, y.y, k & 31));
    if (lane == 0) S.y[k] = y;
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (lane + 32 * u < k) cnmac(t[u], col[lane + 32 * u], y);
  }
  for (int i = jd + lane; i < m; i += 32) S.y[i] = make_double2(0, 0);
}

__global__ void k_gmres_mark_done(GmresState S, const double* __restrict__ nrm2, double tol, int nrhs) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nrhs) return;
  const double lim = tol * S.bnorm[r];
  if (sqrt(nrm2[r]) <= lim) S.done[r] = 1;
}

void launch_gmres_start(const GmresState& s, const double* nrm2, double tol, int nrhs, double* inv_beta,
                        cudaStream_t st, bool init) {
  k_gmres_start<<<nblk(nrhs, 64), 64, 0, st>>>(s, nrm2, tol, nrhs, inv_beta, init);
  WCMG_LAUNCH_CHECK();
}
void launch_gmres_init(const GmresState& s, const double* nrm2, int nrhs, cudaStream_t st) {
  k_gmres_init<<<nblk(nrhs, 64), 64, 0, st>>>(s, nrm2, nrhs);
  WCMG_LAUNCH_CHECK();
}
void launch_gmres_step(const GmresState& s, int j, const double2* h1, const double2* h2, const double* partial,
                       int count, double tol, int final_done, int nrhs, double* inv_h, cudaStream_t st,
                       const int* jdev) {
  k_gmres_step<<<nrhs, RED_T, 0, st>>>(s, j, h1, h2, partial, count, tol, final_done, inv_h, jdev);
  WCMG_LAUNCH_CHECK();
}
void launch_gmres_solve_y(const GmresState& s, int nrhs, cudaStream_t st) {
  k_gmres_solve_y<<<nrhs, 32, s.m * (s.m + 1) / 2 * sizeof(double2), st>>>(s);
  WCMG_LAUNCH_CHECK();
}
void launch_gmres_mark_done(const GmresState& s, const double* nrm2, double tol, int nrhs, cudaStream_t st) {
  k_gmres_mark_done<<<nblk(nrhs, 64), 64, 0, st>>>(s, nrm2, tol, nrhs);
  WCMG_LAUNCH_CHECK();
}

// ---- counter-based Gaussian fields (the generator of the seeded inputs) ----
// Element j of field i (stream stream0 + i): the counter c = seed * 0x9E3779B97F4A7C15
// + stream * 0xD1B54A32D192ED03 + k (mod 2^64) for k = 2j, 2j+1 goes through the
// SplitMix64 finaliser (Steele, Lea, Flood, OOPSLA 2014); u = (out >> 11) 2^-53 exactly;
// Box-Muller: re = sqrt(-2 log(1 - u_2j)) cos(2 pi u_2j+1), im = the same with sin.  The
// transform runs in FP32 (1 - u is formed exactly in FP64 first, so it never rounds to
// 0): FP64 transcendentals on this part would cost more than copying the fields in.
__device__ __forceinline__ double counter_uniform(unsigned long long base, unsigned long long k) {
  unsigned long long z = base + k;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  z = z ^ (z >> 31);
  return (double)(z >> 11) * 0x1.0p-53;
}
__global__ void k_counter_gaussian(double2* __restrict__ out, long long n, unsigned long long seed,
                                   unsigned long long stream0) {
  const long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (j >= n) return;
  const unsigned long long stream = stream0 + blockIdx.y;
  const unsigned long long base = seed * 0x9E3779B97F4A7C15ULL + stream * 0xD1B54A32D192ED03ULL;
  const double u1 = counter_uniform(base, 2ULL * j), u2 = counter_uniform(base, 2ULL * j + 1);
  const float r = sqrtf(-2.0f * logf((float)(1.0 - u1)));
  float sn, cs;
  sincospif((float)(2.0 * u2), &sn, &cs);
  out[(long long)blockIdx.y * n + j] = make_double2((double)(r * cs), (double)(r * sn));
}
void launch_counter_gaussian(double2* out, long long n, int nfields, unsigned long long seed,
                             unsigned long long stream0, cudaStream_t st) {
  k_counter_gaussian<<<dim3(nblk(n, 256), nfields), 256, 0, st>>>(out, n, seed, stream0);
  WCMG_LAUNCH_CHECK();
}

#define WCMG_INST(R)                                                                                             \
  template void launch_dot<R>(double2*, const cplx<R>*, const cplx<R>*, long long, int, double2*, cudaStream_t); \
  template void launch_norm2<R>(double*, const cplx<R>*, long long, int, double*, cudaStream_t);                 \
  template int launch_gram_schmidt<R>(double2*, double2*, double*, cplx<R>*, const cplx<R>*, long long, int, int, \
                                      long long, int, double2*, cudaStream_t, const int*, int);                  \
  template void launch_multiaxpy<R>(cplx<R>*, const cplx<R>*, long long, int, const double2*, int, double,       \
                                    long long, int, cudaStream_t, const int*, int);                              \
  template void launch_copy_idx<R>(cplx<R>*, const cplx<R>*, long long, const int*, long long, long long,        \
                                   cudaStream_t);                                                                \
  template void launch_axpby<R>(cplx<R>*, double, const cplx<R>*, double, long long, int, cudaStream_t);         \
  template void launch_scale_dev<R>(cplx<R>*, const cplx<R>*, const double*, int, long long, int, cudaStream_t,  \
                                    const int*, int, long long, cplx<R>*);                                       \
  template void launch_mr_update<R>(cplx<R>*, cplx<R>*, const cplx<R>*, const double2*, const double*, long long, \
                                    int, cudaStream_t, bool, bool);                                              \
  template void launch_mr_residual<R>(cplx<R>*, const cplx<R>*, const double2*, const double*, long long, int,   \
                                      cudaStream_t);                                                             \
  template void launch_mr_pair<R>(cplx<R>*, const cplx<R>*, cplx<R>*, const cplx<R>*, const double2*,            \
                                  const double*, const double2*, const double*, long long, int, cudaStream_t,    \
                                  bool, bool);                                                                   \
  template void launch_mask_rhs<R>(cplx<R>*, const int*, long long, int, cudaStream_t);                          \
  template void launch_fill_zero<R>(cplx<R>*, long long, cudaStream_t);
WCMG_INST(double)
WCMG_INST(float)
#undef WCMG_INST
template void launch_convert<double, float>(float2*, const double2*, long long, cudaStream_t);
template void launch_convert<float, double>(double2*, const float2*, long long, cudaStream_t);
template void launch_convert<double, double>(double2*, const double2*, long long, cudaStream_t);
template void launch_convert<float, float>(float2*, const float2*, long long, cudaStream_t);

}  // namespace wcmg
