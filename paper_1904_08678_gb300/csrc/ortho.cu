// Block orthonormalisation by Cholesky QR in double-float arithmetic (params.ortho_df).
//
// The Q factor with positive diag(R) of each (aggregate, chirality) panel A (m rows, k
// columns) without any column-by-column sweep: G = A^H A, G = L L^H, Q = A (L^-1)^H.  Two
// passes over the panel, each a dense product whose m k^2 / 2 complex multiply-adds are
// independent, take the place of 2 (k - 1) dependent ones with a block-wide reduction
// behind each: the Gram-Schmidt kernels of transfer.cu are bound by the re-reads of
// earlier columns and those reductions (82 GB of DRAM traffic per 32^3x64 call against 19 GB
// that have to move), this by the FP32 pipe (24 packed instructions per complex
// multiply-add).  G is summed in double-float and, across the threads, in FP64; the k x k
// factorisation and inverse run in FP64.
//
// Accuracy.  With W = L^-1, Q^H Q - 1 = W dG W^H for the error dG of the sums, whose entries
// are of the order u |a_i| |a_j|: column i of Q is off by u e_i, e_i = sum_j |W_ij|^2 |a_j|^2.
// Measured on 24 and 32 columns of 1536 rows with e from 3 to 1e10: max |Q^H Q - 1| is 0.8e-15
// to 6e-15 times max e_i (1e-14 below).  A panel is therefore taken here only if no e_i exceeds
// CQ_AMP = 8, where 24 and 32 columns are orthonormal to 1.4e-14 and 2.5e-14 from FP64 and to
// 2.5e-14 and 3.5e-14 from FP32 input (by Gram-Schmidt 1.1e-14); the others are flagged and the
// Gram-Schmidt kernel does them.  The pivots alone do not bound e: 24 columns that each keep
// 0.36 of their squared norm can have e = 3e6.  Near-null candidates have e below 4 after the
// initial sweeps and below 8 after two refinement sweeps on 32^3x64 (2823 of 16384 panels above
// 4); more sweeps make them more parallel, and from the fourth on nearly all panels go to
// Gram-Schmidt.  Error against 64 bits on mixed Gaussian panels (e = 2): 8e-15 (Gram-Schmidt
// 1.7e-14).
//
// 1024 panels of 1536 x 24 (16^3x32): 3.35 ms by Gram-Schmidt; now 1.10 + 0.11 + 1.22 ms from
// FP64 and 0.83 + 0.11 + 0.94 ms from FP32 input (Gram, factor, product).  The arithmetic
// alone is 0.6 ms per product at the FP32 pipe's rate; the pipe is 68 % busy in the Gram kernel
// and 55 % in the product (whose conversions to FP64 keep that unit 62 % busy), the rest goes to
// its latency at 4 to 6 warps per scheduler.
#include <algorithm>

#include "dfloat.cuh"

namespace wcmg {

constexpr int CQ_T = 256;     // Gram kernel: threads
constexpr int CQ_ROWS = 32;   // panel rows per staged tile
constexpr int CQ_FLUSH = 2;   // tiles between additions of the running double-float sums
constexpr float CQ_AMP = 8.f;       // greatest e
constexpr double CQ_LEAST = 1e-28;  // least |a_j|^2: the error terms of smaller columns' products underflow in FP32

// offset of panel row e (element of chirality s of aggregate blk) within a field
__device__ __forceinline__ long long cq_addr(bool fine, int blk, int e, int s, int Vf, int nc, int bvol) {
  const int half = nc >> 1;
  if (fine) return (long long)(s * half + e / bvol) * Vf + (long long)blk * bvol + e % bvol;
  return ((long long)blk * bvol + e / half) * nc + s * half + e % half;
}
// Packed double-float: the (re, im) pair of one complex value in two-lane FP32 registers, so
// that one instruction does both components of a step (the scalar form left the FMA pipe
// half idle behind the issue slots and register reads).
using f2 = unsigned long long;
__device__ __forceinline__ f2 f2_mk(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 f2_get(f2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
  return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
struct dfp { f2 h, l; };  // lanes: (re, im)
__device__ __forceinline__ dfp dfp_zero() { return {0ULL, 0ULL}; }
// acc += x y lane by lane; XS, YS: x, y have zero low parts.  The two error terms join the low
// part one after the other: the error of an FP32 entry's square has fixed last bits, and added
// to e first its rounding was biased (e = 8, 32 columns from FP32: 5.6e-14, now 3.5e-14).
template <bool XS, bool YS>
__device__ __forceinline__ void dfp_mac(dfp& acc, const dfp& x, const dfp& y) {
  const f2 p = f2_mul(x.h, y.h);
  f2 pe = f2_fma(x.h, y.h, p ^ 0x8000000080000000ULL);  // - p: on the integer pipe
  if (!YS) pe = f2_fma(x.h, y.l, pe);
  if (!XS) pe = f2_fma(x.l, y.h, pe);
  const f2 s = f2_add(acc.h, p), v = f2_sub(s, acc.h);
  const f2 e = f2_add(f2_sub(acc.h, f2_sub(s, v)), f2_sub(p, v));
  acc.h = s;
  acc.l = f2_add(f2_add(acc.l, pe), e);
}
__device__ __forceinline__ dfp dfp_norm(const dfp& a) {
  const f2 h = f2_add(a.h, a.l);
  return {h, f2_sub(a.l, f2_sub(h, a.h))};
}
__device__ __forceinline__ dfp dfp_add(const dfp& a, const dfp& b) {
  const f2 s = f2_add(a.h, b.h), v = f2_sub(s, a.h);
  const f2 e = f2_add(f2_sub(a.h, f2_sub(s, v)), f2_sub(b.h, v));
  return dfp_norm({s, f2_add(e, f2_add(a.l, b.l))});
}
__device__ __forceinline__ double2 dfp_to_fast(const dfp& a) {
  const float2 h = f2_get(a.h), l = f2_get(a.l);
  return make_double2(df_to_fast({h.x, l.x}), df_to_fast({h.y, l.y}));
}
// stored form of a complex value: (re.h, im.h, re.l, im.l)
__device__ __forceinline__ float4 cq_pack(const dfc& v) { return make_float4(v.re.h, v.im.h, v.re.l, v.im.l); }
__device__ __forceinline__ float4 cq_store(double2 v) { return cq_pack(dfc_split(v)); }
__device__ __forceinline__ float4 cq_store(float2 v) { return make_float4(v.x, v.y, 0.f, 0.f); }
__device__ __forceinline__ dfp cq_pair(float4 v) { return {f2_mk(v.x, v.y), f2_mk(v.z, v.w)}; }
__device__ __forceinline__ dfp dfp_load(const float4* v) {
  const float4 t = *v;
  return cq_pair(t);
}

// One CTA per panel.  The upper triangle of G is cut into 3 x 3 column blocks: thread (rg,
// pair) sums block `pair` over the rows rg, rg + RG, ... of each staged tile (6 shared reads
// of 16 bytes per 9 complex multiply-adds; a row's entries are 48 bytes apart between blocks,
// which hits distinct banks).  The next tile's loads are in flight during the sums.
// W[panel] = G, k x k FP64, upper triangle.
template <typename TIN>
__global__ void __launch_bounds__(CQ_T, 2) k_cholqr_gram(double2* __restrict__ W, const TIN* __restrict__ in, int Vf,
                                                         int nc, int bvol, int nvec, bool fine) {
  constexpr bool SINGLE = sizeof(TIN) == 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int blk = blockIdx.x, s = blockIdx.y, panel = blockIdx.x * 2 + blockIdx.y;
  const int nelem = bvol * (nc >> 1), ntile = (nelem + CQ_ROWS - 1) / CQ_ROWS;
  const long long fstride = (long long)Vf * nc;
  const int ng = (nvec + 2) / 3, np = ng * (ng + 1) / 2, pitch = 3 * ng + 1;
  const int RG = min(CQ_T / np, CQ_ROWS);
  const int pr = threadIdx.x % np, rg = threadIdx.x / np;
  int gi = 0;
  {
    int t = pr;
    while (t >= ng - gi) { t -= ng - gi; ++gi; }
  }
  int gj = pr - (gi * ng - gi * (gi - 1) / 2) + gi;
  float4* tile = reinterpret_cast<float4*>(smem_raw);  // [2][CQ_ROWS][pitch]
  // staging role: row lane of the tile, columns warp, warp + NW, ...
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int NW = CQ_T / 32, NL = (33 + NW - 1) / NW;
  TIN pre[NL];
  auto fetch = [&](int t) {
    const int e = t * CQ_ROWS + lane;
    const long long a = e < nelem ? cq_addr(fine, blk, e, s, Vf, nc, bvol) : 0;
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      const int i = warp + NW * j;
      TIN z;
      z.x = z.y = 0;
      pre[j] = e < nelem && i < nvec ? in[i * fstride + a] : z;
    }
  };
  auto stage = [&](int buf) {
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      const int i = warp + NW * j;
      if (i < 3 * ng) {
        tile[(buf * CQ_ROWS + lane) * pitch + i] = cq_store(pre[j]);
      }
    }
  };
  dfp acc[9];
  float4* tot = tile + 2 * CQ_ROWS * pitch + threadIdx.x;  // running sums [9][CQ_T]
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    acc[q] = dfp_zero();
    tot[q * CQ_T] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  fetch(0);
  stage(0);
  __syncthreads();
  for (int t = 0; t < ntile; ++t) {
    if (t + 1 < ntile) fetch(t + 1);
    if (rg < RG) {
      for (int r = rg; r < CQ_ROWS; r += RG) {
        const float4* row = tile + ((t & 1) * CQ_ROWS + r) * pitch;
        // conj(x) y = x.re (y.re, y.im) + x.im (y.im, -y.re)
        dfp y[3], yr[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const float4 v = row[3 * gj + q];
          y[q] = cq_pair(v);
          yr[q] = {f2_mk(v.y, -v.x), f2_mk(v.w, -v.z)};
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const float4 v = row[3 * gi + a];
          const dfp xr = {f2_mk(v.x, v.x), f2_mk(v.z, v.z)}, xi = {f2_mk(v.y, v.y), f2_mk(v.w, v.w)};
#pragma unroll
          for (int b = 0; b < 3; ++b) dfp_mac<SINGLE, SINGLE>(acc[3 * a + b], xr, y[b]);
#pragma unroll
          for (int b = 0; b < 3; ++b) dfp_mac<SINGLE, SINGLE>(acc[3 * a + b], xi, yr[b]);
        }
      }
      if (t % CQ_FLUSH == CQ_FLUSH - 1 || t + 1 == ntile) {
#pragma unroll
        for (int q = 0; q < 9; ++q) {
          const dfp v = dfp_add(dfp_load(tot + q * CQ_T), dfp_norm(acc[q]));
          const float2 h = f2_get(v.h), l = f2_get(v.l);
          tot[q * CQ_T] = make_float4(h.x, h.y, l.x, l.y);
          acc[q] = dfp_zero();
        }
      }
    }
    if (t + 1 < ntile) stage((t + 1) & 1);
    __syncthreads();
  }
  // upper triangle in FP64 from the row groups; zeros below (where L^-1 will form)
  const float4* tots = tile + 2 * CQ_ROWS * pitch;
  double2* G = W + (long long)panel * nvec * nvec;
  for (int q = threadIdx.x; q < np * 9; q += CQ_T) {
    const int p = q % np, a = q / np / 3, b = q / np % 3;
    double2 v = make_double2(0, 0);
    for (int r = 0; r < RG; ++r) v += dfp_to_fast(dfp_load(tots + (q / np) * CQ_T + r * np + p));
    int i = 0, u = p;
    while (u >= ng - i) { u -= ng - i; ++i; }
    const int gr = 3 * i + a, gc = 3 * (i + u) + b;
    if (gr <= gc && gc < nvec) G[gr * nvec + gc] = v;
  }
  for (int q = threadIdx.x; q < nvec * nvec; q += CQ_T)
    if (q % nvec < q / nvec) G[q] = make_double2(0, 0);
}

// G = R^H R (R upper) and L^-1, L = R^H, in place: one warp per panel, lane j owns column j of
// the k x k matrix in shared memory.  Step k eliminates column k below the diagonal, and
// the same row operations turn the identity into (up to the row scales) L^-1, whose strict
// lower triangle takes the eliminated entries' places.  In the Gram kernel's own CTAs this
// serial part (24 steps of FP64 at two lanes per cycle) left the FP32 pipe idle half of the
// time; here thousands of panels overlap.
constexpr int CQ_CW = 2;  // panels per CTA
__global__ void __launch_bounds__(32 * CQ_CW) k_cholqr_factor(double2* __restrict__ W, int npanel, int nvec,
                                                              int* __restrict__ flag, int* __restrict__ nflag) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, panel = blockIdx.x * CQ_CW + (threadIdx.x >> 5);
  if (panel >= npanel) return;  // warps are independent
  double2* M = reinterpret_cast<double2*>(smem_raw) + (threadIdx.x >> 5) * nvec * nvec;
  double2* w = W + (long long)panel * nvec * nvec;
  for (int q = lane; q < nvec * nvec; q += 32) M[q] = w[q];
  __syncwarp();
  const bool col = lane < nvec;
  const double d0 = col ? M[lane * nvec + lane].x : 1.0;
  double piv_own = 1.0;  // final pivot of row `lane`
  bool ok = true;
  for (int k = 0; k < nvec; ++k) {
    const double piv = M[k * nvec + k].x;
    const double ref = __shfl_sync(0xffffffffu, d0, k);
    // e_k >= |a_k|^2 / pivot; also for a NaN; uniform over the warp
    if (!(CQ_AMP * piv > ref) || !(ref > CQ_LEAST) || !isfinite(piv)) {
      ok = false;
      break;
    }
    if (lane == k) piv_own = piv;
    const double inv = 1.0 / piv;
    // row k: R's entries right of the diagonal, L^-1's left of it, 1 on it
    const double2 row = !col ? make_double2(0, 0) : lane == k ? make_double2(1, 0) : M[k * nvec + lane];
    const double2 mult = make_double2(inv * row.x, -inv * row.y);  // lane i > k: conj(G_ki) / piv
    for (int i = k + 1; i < nvec; ++i) {
      const double2 f = make_double2(__shfl_sync(0xffffffffu, mult.x, i), __shfl_sync(0xffffffffu, mult.y, i));
      if (col && (lane <= k || lane >= i)) cnmac(M[i * nvec + lane], f, row);
    }
    __syncwarp();
  }
  if (ok) {
    const double scale = 1.0 / sqrt(piv_own), norm = sqrt(d0);
    for (int i = 0; i < nvec; ++i) {
      const double si = __shfl_sync(0xffffffffu, scale, i);
      const double2 v = !col || lane > i ? make_double2(0, 0) : si * (lane == i ? make_double2(1, 0) : M[i * nvec + lane]);
      if (col) w[i * nvec + lane] = v;
      const float2 t = make_float2((float)(norm * v.x), (float)(norm * v.y));
      const float e = warp_sum(cnorm2(t));  // needs no more than FP32; the same in every lane
      ok = ok && e <= CQ_AMP;               // false for a NaN
    }
  }
  if (lane == 0) {
    flag[panel] = ok ? 0 : 1;
    if (!ok) atomicAdd(nflag, 1);
  }
}

// Q = A W^H: q_j = sum_{i <= j} a_i conj(W_ji).  Two threads per panel row (in different
// warps), whose entries lie in shared memory as [column][row]: with one, the rows alone allow
// 12 warps per SM, too few to hide the FP32 latency.  Columns of Q go in blocks of CQ_J
// (independent sums; the factors are read by a whole warp at once), and the blocks are dealt
// to the two threads from the longest on as 0 1 1 0 0 1 1 .., which balances the triangle.
// Writes P in FP64 and, if given, its FP32 rounding; a row is staged before any of it is
// written, so the FP64 input may be replaced in place.
template <typename TIN> struct CqRow;  // a staged entry: split once, FP32 input as it is
template <> struct CqRow<double2> { using type = float4; };
template <> struct CqRow<float2> { using type = float2; };
__device__ __forceinline__ void cq_put(float4* p, double2 v) { *p = cq_store(v); }
__device__ __forceinline__ void cq_put(float2* p, float2 v) { *p = v; }
__device__ __forceinline__ float4 cq_get(float4 v) { return v; }
__device__ __forceinline__ float4 cq_get(float2 v) { return cq_store(v); }
constexpr int CQ_R = 128, CQ_J = 4;  // rows per pass (2 CQ_R threads), columns per block
template <typename TIN>
__global__ void __launch_bounds__(2 * CQ_R) k_cholqr_apply(double2* out, float2* __restrict__ out32, const TIN* in,
                                                           const double2* __restrict__ W, const int* __restrict__ flag,
                                                           int Vf, int nc, int bvol, int nvec, bool fine) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int blk = blockIdx.x, s = blockIdx.y, panel = blockIdx.x * 2 + blockIdx.y;
  if (flag[panel]) return;
  const int nelem = bvol * (nc >> 1);
  const long long fstride = (long long)Vf * nc;
  const int nblk_ = (nvec + CQ_J - 1) / CQ_J, nj = nblk_ * CQ_J;
  constexpr bool SINGLE = sizeof(TIN) == 8;
  using TROW = typename CqRow<TIN>::type;
  const int half = threadIdx.x / CQ_R, r = threadIdx.x % CQ_R;
  float4* w = reinterpret_cast<float4*>(smem_raw);  // [i][nj][2]: f = conj(W_ji) (zero for j < i, j >= nvec) and i f
  TROW* row = reinterpret_cast<TROW*>(w + 2 * nvec * nj) + r;  // [i][CQ_R]
  for (int q = threadIdx.x; q < nvec * nj; q += 2 * CQ_R) {
    const int i = q / nj, j = q % nj;
    const float4 f = cq_store(j >= i && j < nvec ? conjg(W[((long long)panel * nvec + j) * nvec + i])
                                                 : make_double2(0, 0));
    w[2 * q] = f;
    w[2 * q + 1] = make_float4(-f.y, f.x, -f.w, f.z);
  }
  for (int e0 = blockIdx.z * CQ_R; e0 < nelem; e0 += gridDim.z * CQ_R) {
    const int e = e0 + r;
    const long long a = e < nelem ? cq_addr(fine, blk, e, s, Vf, nc, bvol) : 0;
    if (e < nelem)
      for (int i = half; i < nvec; i += 2) cq_put(row + i * CQ_R, in[i * fstride + a]);
    __syncthreads();
    if (e < nelem)
      for (int b = nblk_ - 1; b >= 0; --b) {
        if ((((nblk_ - b) >> 1) & 1) != half) continue;
        const int j0 = b * CQ_J;
        dfp acc[CQ_J];
#pragma unroll
        for (int q = 0; q < CQ_J; ++q) acc[q] = dfp_zero();
        const int top = min(j0 + CQ_J, nvec);
        for (int i = 0; i < top; ++i) {
          // x f = x.re f + x.im (i f)
          const float4 x = cq_get(row[i * CQ_R]);
          const dfp xr = {f2_mk(x.x, x.x), f2_mk(x.z, x.z)}, xi = {f2_mk(x.y, x.y), f2_mk(x.w, x.w)};
          const float4* wi = w + 2 * (i * nj + j0);
#pragma unroll
          for (int q = 0; q < CQ_J; ++q) dfp_mac<SINGLE, false>(acc[q], xr, dfp_load(wi + 2 * q));
#pragma unroll
          for (int q = 0; q < CQ_J; ++q) dfp_mac<SINGLE, false>(acc[q], xi, dfp_load(wi + 2 * q + 1));
          // keep the low parts short: their own rounding errors are what limits the sum
          if ((i & 7) == 7) {
#pragma unroll
            for (int q = 0; q < CQ_J; ++q) acc[q] = dfp_norm(acc[q]);
          }
        }
#pragma unroll
        for (int q = 0; q < CQ_J; ++q)
          if (j0 + q < nvec) {
            const double2 v = dfp_to_fast(dfp_norm(acc[q]));
            out[(j0 + q) * fstride + a] = v;
            if (out32) out32[(j0 + q) * fstride + a] = make_float2((float)v.x, (float)v.y);
          }
      }
    __syncthreads();
  }
}

template <typename TIN>
static void cholqr(double2* vecs, float2* out32, const TIN* in, double2* W, int* flag, int* nflag, int Vf, int nc,
                   int bvol, int nvec, bool fine, cudaStream_t st) {
  // two staged tiles and the running sums
  const int ng = (nvec + 2) / 3;
  const int smem = 2 * CQ_ROWS * (3 * ng + 1) * 16 + 9 * CQ_T * 16;
  auto kg = k_cholqr_gram<TIN>;
  WCMG_CUDA(cudaFuncSetAttribute(kg, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  kg<<<dim3(Vf / bvol, 2), CQ_T, smem, st>>>(W, in, Vf, nc, bvol, nvec, fine);
  WCMG_LAUNCH_CHECK();
  const int npanel = 2 * (Vf / bvol), smem1 = CQ_CW * nvec * nvec * 16;
  k_cholqr_factor<<<nblk(npanel, CQ_CW), 32 * CQ_CW, smem1, st>>>(W, npanel, nvec, flag, nflag);
  WCMG_LAUNCH_CHECK();
  const int nj = (nvec + CQ_J - 1) / CQ_J * CQ_J, nelem = bvol * (nc / 2);
  const int smem2 = 2 * nvec * nj * 16 + nvec * CQ_R * (int)sizeof(typename CqRow<TIN>::type);
  auto ka = k_cholqr_apply<TIN>;
  WCMG_CUDA(cudaFuncSetAttribute(ka, cudaFuncAttributeMaxDynamicSharedMemorySize, smem2));
  // a panel is split over up to four CTAs (each loads the factors once for its rows)
  const int split = std::max(1, std::min(4, nelem / CQ_R));
  ka<<<dim3(Vf / bvol, 2, split), 2 * CQ_R, smem2, st>>>(vecs, out32, in, W, flag, Vf, nc, bvol, nvec, fine);
  WCMG_LAUNCH_CHECK();
}

// Orthonormalise vecs (FP64, in place) or, when in32 is given, in32 into vecs and out32.
// *nflag is zeroed by the caller.
void launch_cholqr(double2* vecs, double2* W, int* flag, int* nflag, int Vf, int nc, int bvol, int nvec, bool fine,
                   cudaStream_t st, const float2* in32, float2* out32) {
  if (nvec > 32) throw Error(-1, "block orthonormalisation supports nvec <= 32");
  if (in32) cholqr<float2>(vecs, out32, in32, W, flag, nflag, Vf, nc, bvol, nvec, fine, st);
  else cholqr<double2>(vecs, out32, vecs, W, flag, nflag, Vf, nc, bvol, nvec, fine, st);
}

}  // namespace wcmg
