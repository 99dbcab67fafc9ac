// Gauge-equivariant parallel-transport convolution (PTC) network kernels: the
// learned coarse correction.  The paper has no learned component; the network
// maps a fine residual to an approximation of the multigrid coarse-grid
// correction P D_c^-1 P^dag r built from the operators of Sec. 2.1.
//
//   layer:  out_i(x) = sum_j sum_h W_{ijh} (T_h in_j)(x)
//   hops:   h = 0 identity, 1 + 2 mu: (T f)(x) = U_mu(x) f(x + mu),
//           2 + 2 mu: (T f)(x) = U_mu(x - mu)^dag f(x - mu);  T_{+-mu}^dag = T_{-+mu}
//   W_{ijh} complex 4x4 spin matrices (spin index), T_h acts on colour.
// Fields use the fine layout [12][V] (component 3 * spin + colour), FP32.
// The network's layers join one field to H = 12 fields, and both directions and the weight
// gradients move only the single field's side: the spin weights commute with the transport,
// so the expanding layer transports its one input 9 times and then mixes (12 x 9 mixings of
// 48 complex multiply-adds), the contracting one mixes at the neighbour first and transports
// the 9 sums.  Either way 9 transports per site (324 complex multiply-adds) join 5184
// for the mixing, where transporting every field's 9 hops costs 3888 more.  The backward
// passes are the same two kernels with the hops reversed and the weights conjugate-transposed
// (T_h^dag = T_{opp h}).  Bound by the FP32 pipe (22 k multiply-adds per site and
// layer; 43 to 55 % busy, its three-operand instructions' register reads allow 63 %).
// Forward and backward of four fields on 16^3x32, seven layer passes: 8.7 ms before, 5.6 ms
// now (per pass: expanding 0.69 ms, contracting 0.78, weight gradients 0.80 + 0.06; before:
// forward 0.68 and 0.85, backward 1.2, gradients 1.65 + 0.23).
#include "kernels.h"

namespace wcmg {

constexpr int PTC_NHOP = 9;

// t = (T_h f)(x), 12 complex, FP32
__device__ __forceinline__ void ptc_transport(float2 (&t)[12], const float2* __restrict__ f,
                                              const float2* __restrict__ U, const int* __restrict__ nbr, int V, int x,
                                              int h) {
  if (h == 0) {
#pragma unroll
    for (int c = 0; c < 12; ++c) t[c] = f[(long long)c * V + x];
    return;
  }
  const int mu = (h - 1) >> 1, back = (h - 1) & 1;
  const int y = nbr[(2 * mu + back) * V + x];
  const int ls = back ? y : x;
  float2 u[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) u[k] = U[((long long)mu * 9 + k) * V + ls];
  float2 g[12];
#pragma unroll
  for (int c = 0; c < 12; ++c) g[c] = f[(long long)c * V + y];
#pragma unroll
  for (int s = 0; s < 4; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float2 acc = make_float2(0.f, 0.f);
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        if (!back) cmac(acc, u[3 * a + b], g[3 * s + b]);
        else cjmac(acc, u[3 * b + a], g[3 * s + b]);
      }
      t[3 * s + a] = acc;
    }
}

// opposite hop: T_h^dag = T_{opp(h)}
__device__ __forceinline__ int ptc_opp(int h) { return h == 0 ? 0 : (((h - 1) & 1) ? h - 1 : h + 1); }

// Shared copy of one layer's weights [nf][9][16] as they act: row a, column b of the spin
// matrix applied to the field (adj: conj-transposed, for the backward pass).
__device__ __forceinline__ void ptc_load_weights(float2* Ws, const float2* __restrict__ W, int n, bool adj) {
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const int e = k & 15, a = e >> 2, b = e & 3;
    Ws[k] = adj ? conjg(W[(k & ~15) + 4 * b + a]) : W[k];
  }
  __syncthreads();
}
// acc += W t, a 4 x 4 spin matrix from shared memory.  The four products are summed before they
// join acc: one chain over all hops and fields (45 us less in the seven passes above) was half
// as much further from the FP64 result (2.8e-7, now 1.9e-7).
__device__ __forceinline__ void spin_mix(float2 (&acc)[12], const float2* __restrict__ w, const float2 (&t)[12]) {
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    float2 s[3];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const float2 wab = w[4 * a + b];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (b == 0) s[c] = cmul(wab, t[c]);
        else cmac(s[c], wab, t[3 * b + c]);
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[3 * a + c] += s[c];
  }
}

// Expanding layer (1 -> nf fields): out_i(x) = sum_h W_ih (T_h in)(x); each thread forms OG
// outputs at its site.
template <int OG>
__global__ void __launch_bounds__(128) k_ptc_expand(float2* __restrict__ out, const float2* __restrict__ in,
                                                    const float2* __restrict__ W, const float2* __restrict__ U,
                                                    const int* __restrict__ nbr, int V, int nf, int nrhs, bool adj) {
  extern __shared__ float2 Ws[];
  ptc_load_weights(Ws, W, nf * PTC_NHOP * 16, adj);
  const int ngrp = (nf + OG - 1) / OG;
  const int io0 = (blockIdx.y % ngrp) * OG, r = blockIdx.y / ngrp;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= V || r >= nrhs) return;
  const long long fs = 12LL * V;
  float2 acc[OG][12];
#pragma unroll
  for (int g = 0; g < OG; ++g)
#pragma unroll
    for (int c = 0; c < 12; ++c) acc[g][c] = make_float2(0.f, 0.f);
  const float2* f = in + (long long)r * fs;
  for (int h = 0; h < PTC_NHOP; ++h) {
    float2 t[12];
    ptc_transport(t, f, U, nbr, V, x, adj ? ptc_opp(h) : h);
#pragma unroll
    for (int g = 0; g < OG; ++g) {
      if (io0 + g >= nf) break;
      spin_mix(acc[g], Ws + ((io0 + g) * PTC_NHOP + h) * 16, t);
    }
  }
#pragma unroll
  for (int g = 0; g < OG; ++g) {
    if (io0 + g >= nf) break;
    float2* o = out + ((long long)r * nf + io0 + g) * fs;
#pragma unroll
    for (int c = 0; c < 12; ++c) o[(long long)c * V + x] = acc[g][c];
  }
}

// Contracting layer (nf -> 1 field): out(x) = sum_h T_h (sum_j W_jh in_j)(x), the spin sum
// formed at the site the hop reads from.
__global__ void __launch_bounds__(128) k_ptc_contract(float2* __restrict__ out, const float2* __restrict__ in,
                                                      const float2* __restrict__ W, const float2* __restrict__ U,
                                                      const int* __restrict__ nbr, int V, int nf, int nrhs, bool adj) {
  extern __shared__ float2 Ws[];
  ptc_load_weights(Ws, W, nf * PTC_NHOP * 16, adj);
  const int r = blockIdx.y;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= V) return;
  const long long fs = 12LL * V;
  const float2* f = in + (long long)r * nf * fs;
  float2 acc[12];
#pragma unroll
  for (int c = 0; c < 12; ++c) acc[c] = make_float2(0.f, 0.f);
  for (int h = 0; h < PTC_NHOP; ++h) {
    const int ho = adj ? ptc_opp(h) : h;
    const int mu = (ho - 1) >> 1, back = (ho - 1) & 1;
    const int y = ho == 0 ? x : nbr[(2 * mu + back) * V + x];
    float2 s[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) s[c] = make_float2(0.f, 0.f);
    // the next field is on its way while this one is mixed
    float2 t[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) t[c] = f[(long long)c * V + y];
    for (int j = 0; j < nf; ++j) {
      float2 n[12];
      const float2* fn = f + (long long)(j + 1 < nf ? j + 1 : j) * fs;
#pragma unroll
      for (int c = 0; c < 12; ++c) n[c] = fn[(long long)c * V + y];
      spin_mix(s, Ws + (j * PTC_NHOP + h) * 16, t);
#pragma unroll
      for (int c = 0; c < 12; ++c) t[c] = n[c];
    }
    if (ho == 0) {
#pragma unroll
      for (int c = 0; c < 12; ++c) acc[c] += s[c];
      continue;
    }
    const int ls = back ? y : x;
    float2 u[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) u[k] = U[((long long)mu * 9 + k) * V + ls];
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          if (!back) cmac(acc[3 * sp + a], u[3 * a + b], s[3 * sp + b]);
          else cjmac(acc[3 * sp + a], u[3 * b + a], s[3 * sp + b]);
        }
  }
  float2* o = out + (long long)r * fs;
#pragma unroll
  for (int c = 0; c < 12; ++c) o[(long long)c * V + x] = acc[c];
}

// Weight gradients as one small matrix product per tile of sites:
//   P[(i, a)][(h, b)] = sum_{x, c} m_i[a][c](x) conj(t_h[b][c](x)),
// m_i the nf-field side, t_h = T_h (or T_h^dag = T_{opp h}) of the single field: the expanding
// layer's gradient is P with m = its output gradients and t = T_h in; the contracting one's,
// sum_x g[a] conj((T_h in_j)[b]) = sum_y (T_h^dag g)[a] conj(in_j[b]), is P^dag with m = its
// inputs and t = T_h^dag g.  A CTA stages WG_S sites at a time in shared memory ([row][c, site]),
// and thread (c, ti, tj) sums a 4 x 6 tile (rows ti + TI q, columns tj + 6 p) over the sites of
// colour c, three columns at a time (14 shared reads per 24 complex multiply-adds, against one
// warp reduction of 16 values per 48 before).  The sums are in two levels, WG_CH sites and then
// the CTA's WG_TILES tiles: one chain over all of its 128 sites was twice as far from the FP64
// result (3.4e-7, now 1.75e-7).  Two CTAs per SM, one of which stages while the other multiplies:
// a quarter of the SM's registers holds five warps of 96, and three CTAs would put six on some
// of them, so the threads take 126 (96 spilled: 0.91 against 0.80 ms per gradient on the sizes
// above).  The colours are added in a fixed order and written as one partial per CTA;
// k_ptc_wgrad_sum and _final add the partials in FP64.
constexpr int WG_S = 32, WG_TILES = 4, WG_P = 3 * WG_S + 1;
constexpr int WG_CH = 16;    // sites per first-level sum
constexpr int WG_COLS = 36;  // 9 hops x 4 spins
constexpr int WG_T = 224;    // 3 colours x 12 x 6 threads multiply, all stage
__global__ void __launch_bounds__(WG_T, 2) k_ptc_wgrad_partial(float2* __restrict__ partial,
                                                               const float2* __restrict__ mf,
                                                               const float2* __restrict__ sf,
                                                               const float2* __restrict__ U,
                                                               const int* __restrict__ nbr, int V, int nf, int nrhs,
                                                               bool adj) {
  extern __shared__ float2 sm[];
  float2* Ms = sm;                   // [4 nf][WG_P]
  float2* Ts = sm + 4 * nf * WG_P;   // [36][WG_P]
  const long long fs = 12LL * V;
  const int tps = (V + WG_S - 1) / WG_S;  // tiles per rhs
  const int rows = 4 * nf, TI = nf;  // nf <= 12
  const int colour = threadIdx.x / 72, t = threadIdx.x % 72;
  const int ti = t / 6, tj = t % 6;
  float2 tot[4][6];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int p = 0; p < 6; ++p) tot[q][p] = make_float2(0.f, 0.f);
  for (int u = 0; u < WG_TILES; ++u) {
    const long long tile = (long long)blockIdx.x * WG_TILES + u;
    if (tile >= (long long)tps * nrhs) break;  // uniform
    const int r = (int)(tile / tps), x0 = (int)(tile % tps) * WG_S;
    // staging: lane = site, warp = (field, component) row or hop
    const int x = x0 + (threadIdx.x & 31), warp = threadIdx.x >> 5;
    const bool in = x < V;
    const float2* m = mf + (long long)r * nf * fs + x;
#pragma unroll 4
    for (int ic = warp; ic < 12 * nf; ic += WG_T / 32)  // 12 i + 3 a + c: row 4 i + a, colour c
      Ms[(ic / 3) * WG_P + (ic % 3) * WG_S + (threadIdx.x & 31)] = in ? m[(long long)ic * V] : make_float2(0.f, 0.f);
    for (int h = warp; h < PTC_NHOP; h += WG_T / 32) {
      float2 v[12];
#pragma unroll
      for (int c = 0; c < 12; ++c) v[c] = make_float2(0.f, 0.f);
      if (in) ptc_transport(v, sf + (long long)r * fs, U, nbr, V, x, adj ? ptc_opp(h) : h);
#pragma unroll
      for (int c = 0; c < 12; ++c) Ts[(4 * h + c / 3) * WG_P + (c % 3) * WG_S + (threadIdx.x & 31)] = v[c];
    }
    __syncthreads();
    if (ti < TI && colour < 3) {
#pragma unroll
      for (int half = 0; half < 6; half += 3)
        for (int k0 = colour * WG_S; k0 < (colour + 1) * WG_S; k0 += WG_CH) {
          float2 acc[4][3];
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int p = 0; p < 3; ++p) acc[q][p] = make_float2(0.f, 0.f);
#pragma unroll 2
          for (int k = k0; k < k0 + WG_CH; ++k) {
            float2 a[4], b[3];
#pragma unroll
            for (int q = 0; q < 4; ++q) a[q] = Ms[(ti + TI * q) * WG_P + k];
#pragma unroll
            for (int p = 0; p < 3; ++p) b[p] = Ts[(tj + 6 * (half + p)) * WG_P + k];
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
              for (int p = 0; p < 3; ++p) cjmac(acc[q][p], b[p], a[q]);  // m conj(t)
          }
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int p = 0; p < 3; ++p) tot[q][half + p] += acc[q][p];
        }
    }
    __syncthreads();
  }
  // colours in turn: 0 stores, 1 and 2 add
  float2* red = sm;  // [rows][36]
  for (int k = 0; k < 3; ++k) {
    if (colour == k && ti < TI) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int p = 0; p < 6; ++p) {
          float2* o = red + (ti + TI * q) * WG_COLS + tj + 6 * p;
          if (k == 0) *o = tot[q][p];
          else *o += tot[q][p];
        }
    }
    __syncthreads();
  }
  for (int k = threadIdx.x; k < rows * WG_COLS; k += WG_T) partial[(long long)blockIdx.x * rows * WG_COLS + k] = red[k];
}

// second stage, grid (entries / 32, slices): FP64 sums of the partials of a slice
constexpr int WF_SLICES = 16;
__global__ void __launch_bounds__(256) k_ptc_wgrad_sum(double2* __restrict__ part2, const float2* __restrict__ partial,
                                                       int npart, int nent) {
  __shared__ double2 sc[8][32];
  const int e = blockIdx.x * 32 + (threadIdx.x & 31), w = threadIdx.x >> 5;
  const int per = (npart + WF_SLICES - 1) / WF_SLICES;
  const int p0 = blockIdx.y * per, p1 = min(p0 + per, npart);
  double2 acc = make_double2(0, 0);
  if (e < nent) {
#pragma unroll 4
    for (int p = p0 + w; p < p1; p += 8) {
      const float2 v = partial[(long long)p * nent + e];
      acc.x += v.x;
      acc.y += v.y;
    }
  }
  sc[w][threadIdx.x & 31] = acc;
  __syncthreads();
  if (w == 0 && e < nent) {
    for (int k = 1; k < 8; ++k) acc += sc[k][threadIdx.x];
    part2[(long long)blockIdx.y * nent + e] = acc;
  }
}
// third stage: the slices, and from P's order to the weights' [field][hop][a][b]
__global__ void __launch_bounds__(128) k_ptc_wgrad_final(float2* __restrict__ gW, const double2* __restrict__ part2,
                                                         int nf, bool adj) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x, nent = nf * 4 * WG_COLS;
  if (k >= nent) return;
  const int b = k & 3, a = (k >> 2) & 3, h = (k >> 4) % PTC_NHOP, i = (k >> 4) / PTC_NHOP;
  // expanding: P[(i, a)][(h, b)]; contracting: conj(P[(i, b)][(h, a)])
  const int e = (4 * i + (adj ? b : a)) * WG_COLS + 4 * h + (adj ? a : b);
  double2 acc = make_double2(0, 0);
  for (int s = 0; s < WF_SLICES; ++s) acc += part2[(long long)s * nent + e];
  gW[k] = make_float2((float)acc.x, (float)(adj ? -acc.y : acc.y));
}

// Adam on the real and imaginary parts (real gradient = 2 x Wirtinger gradient).
__global__ void k_ptc_adam(float2* __restrict__ w, const float2* __restrict__ g, float2* __restrict__ m,
                           float2* __restrict__ v, int n, float lr, float b1, float b2, float eps, float bc1,
                           float bc2) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const float2 gr = make_float2(2.f * g[k].x, 2.f * g[k].y);
  float2 mk = m[k], vk = v[k];
  mk.x = b1 * mk.x + (1.f - b1) * gr.x;
  mk.y = b1 * mk.y + (1.f - b1) * gr.y;
  vk.x = b2 * vk.x + (1.f - b2) * gr.x * gr.x;
  vk.y = b2 * vk.y + (1.f - b2) * gr.y * gr.y;
  m[k] = mk;
  v[k] = vk;
  float2 wk = w[k];
  wk.x -= lr * (mk.x / bc1) / (sqrtf(vk.x / bc2) + eps);
  wk.y -= lr * (mk.y / bc1) / (sqrtf(vk.y / bc2) + eps);
  w[k] = wk;
}

// Counter-based Gaussian field (SplitMix64 finaliser on seed * phi + stream * c +
// index, uniform from the top 53 bits, Box-Muller), the same generator as the
// host-side input module, drawn on the device for training residuals.
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
__device__ __forceinline__ double u01(unsigned long long seed, unsigned long long stream, unsigned long long i) {
  const unsigned long long c = seed * 0x9E3779B97F4A7C15ULL + stream * 0xD1B54A32D192ED03ULL + i;
  return (double)(splitmix64(c) >> 11) * (1.0 / 9007199254740992.0);
}
__global__ void k_gaussian_field(float2* __restrict__ out, long long n, unsigned long long seed,
                                 unsigned long long stream) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double u1 = u01(seed, stream, 2 * i), u2 = u01(seed, stream, 2 * i + 1);
  const double rad = sqrt(-2.0 * log1p(-u1));
  double sv, cv;
  sincospi(2.0 * u2, &sv, &cv);
  out[i] = make_float2((float)(rad * cv), (float)(rad * sv));
}

// ---------------- launchers ----------------
void launch_ptc_expand(float2* out, const float2* in, const float2* W, const float2* U, const int* nbr, int V, int nf,
                       int nrhs, bool adj, cudaStream_t st) {
  const size_t smem = (size_t)nf * PTC_NHOP * 16 * sizeof(float2);
  k_ptc_expand<4><<<dim3(nblk(V, 128), ((nf + 3) / 4) * nrhs), 128, smem, st>>>(out, in, W, U, nbr, V, nf, nrhs, adj);
  WCMG_LAUNCH_CHECK();
}
void launch_ptc_contract(float2* out, const float2* in, const float2* W, const float2* U, const int* nbr, int V,
                         int nf, int nrhs, bool adj, cudaStream_t st) {
  const size_t smem = (size_t)nf * PTC_NHOP * 16 * sizeof(float2);
  k_ptc_contract<<<dim3(nblk(V, 128), nrhs), 128, smem, st>>>(out, in, W, U, nbr, V, nf, nrhs, adj);
  WCMG_LAUNCH_CHECK();
}
static long long wgrad_parts(int V, int nrhs) {
  const long long tiles = (long long)((V + WG_S - 1) / WG_S) * nrhs;
  return (tiles + WG_TILES - 1) / WG_TILES;
}
long long ptc_wgrad_partial_size(int V, int nf, int nrhs) {
  // the FP32 partials, then the slices' FP64 sums (two float2 each)
  return wgrad_parts(V, nrhs) * nf * 4 * WG_COLS + 2LL * WF_SLICES * nf * 4 * WG_COLS;
}
void launch_ptc_wgrad(float2* gW, float2* partial, const float2* mf, const float2* sf, const float2* U, const int* nbr,
                      int V, int nf, int nrhs, bool adj, cudaStream_t st) {
  const int rows = 4 * nf, nent = rows * WG_COLS;
  if (nf > 12) throw Error(-1, "PTC weight gradient: at most 12 fields");
  const long long np = wgrad_parts(V, nrhs);
  const int smem = (rows + WG_COLS) * WG_P * (int)sizeof(float2);
  WCMG_CUDA(cudaFuncSetAttribute(k_ptc_wgrad_partial, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  k_ptc_wgrad_partial<<<(unsigned)np, WG_T, smem, st>>>(partial, mf, sf, U, nbr, V, nf, nrhs, adj);
  WCMG_LAUNCH_CHECK();
  double2* part2 = reinterpret_cast<double2*>(partial + np * nent);
  k_ptc_wgrad_sum<<<dim3((nent + 31) / 32, WF_SLICES), 256, 0, st>>>(part2, partial, (int)np, nent);
  WCMG_LAUNCH_CHECK();
  k_ptc_wgrad_final<<<nblk(nent, 128), 128, 0, st>>>(gW, part2, nf, adj);
  WCMG_LAUNCH_CHECK();
}
void launch_ptc_adam(float2* w, const float2* g, float2* m, float2* v, int n, float lr, int t, cudaStream_t st) {
  const float b1 = 0.9f, b2 = 0.999f;
  k_ptc_adam<<<nblk(n, 256), 256, 0, st>>>(w, g, m, v, n, lr, b1, b2, 1e-8f, 1.f - powf(b1, (float)t),
                                           1.f - powf(b2, (float)t));
  WCMG_LAUNCH_CHECK();
}
void launch_gaussian_field(float2* out, long long n, unsigned long long seed, unsigned long long stream,
                           cudaStream_t st) {
  k_gaussian_field<<<nblk(n, 256), 256, 0, st>>>(out, n, seed, stream);
  WCMG_LAUNCH_CHECK();
}

}  // namespace wcmg
