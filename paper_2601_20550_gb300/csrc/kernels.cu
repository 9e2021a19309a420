// Non-template kernels: 2D Fourier sums / correlation spectrum and state conversion.
#include "fixed54.cuh"
#include "internal.h"

namespace heom {

__global__ void __launch_bounds__(256) dft_twiddle_kernel(double2 *__restrict__ tw, int n1, int n3) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n1 + n3) return;
  const int k = i < n1 ? i : i - n1, n = i < n1 ? n1 : n3;
  double s, c;
  sincospi(2.0 * (double)k / n, &s, &c);
  tw[i] = make_double2(c, s);
}

__global__ void __launch_bounds__(128) dft_rows_kernel(const double2 *__restrict__ RI, const double2 *__restrict__ RII,
                                                       const double2 *__restrict__ tw3, int n1, int n3,
                                                       double2 *__restrict__ F) {
  const int j = blockIdx.x, p = blockIdx.y * blockDim.x + threadIdx.x;
  if (p >= n3) return;
  const double2 *R = (blockIdx.z ? RII : RI) + (int64_t)j * n3;
  const double2 r0 = R[0];
  double re = 0.5 * r0.x, im = 0.5 * r0.y;
  int i = 0;
#pragma unroll 4
  for (int k = 1; k < n3; ++k) {
    i += p;
    i -= i >= n3 ? n3 : 0;
    const double2 r = R[k], t = tw3[i];
    re = fma(t.x, r.x, re);
    im = fma(t.x, r.y, im);
    re = fma(-t.y, r.y, re);
    im = fma(t.y, r.x, im);
  }
  F[((int64_t)blockIdx.z * n1 + j) * n3 + p] = make_double2(re, im);
}

__global__ void __launch_bounds__(128) dft_cols_kernel(const double2 *__restrict__ F, const double2 *__restrict__ tw1,
                                                       int n1, int n3, double dtau, double *__restrict__ SC) {
  const int q = blockIdx.x, p = blockIdx.y * blockDim.x + threadIdx.x;
  if (p >= n3) return;
  const double2 *FI = F + p, *FII = F + (int64_t)n1 * n3 + p;
  double s = 0.5 * (FI[0].y + FII[0].y), s2 = 0.0;
  int i = 0;
#pragma unroll 4
  for (int j = 1; j < n1; ++j) {
    i += q;
    i -= i >= n1 ? n1 : 0;
    const double2 a = FI[(int64_t)j * n3], b = FII[(int64_t)j * n3], t = tw1[i];
    // Im[conj(t) a] + Im[t b]: the rephasing part enters at -Omega1
    s = fma(t.x, a.y, s);
    s = fma(t.x, b.y, s);
    s2 = fma(t.y, b.x, s2);
    s2 = fma(-t.y, a.x, s2);
  }
  SC[(int64_t)q * n3 + p] = dtau * dtau * (s + s2);
}

void dft2d_sc(const double2 *RI, const double2 *RII, int n1, int n3, double dtau, double *SC, double2 *work,
              cudaStream_t st) {
  double2 *F = work, *tw1 = work + 2 * (int64_t)n1 * n3, *tw3 = tw1 + n1;
  const unsigned pb = (unsigned)((n3 + 127) / 128);
  dft_twiddle_kernel<<<(unsigned)((n1 + n3 + 255) / 256), 256, 0, st>>>(tw1, n1, n3);
  dft_rows_kernel<<<dim3((unsigned)n1, pb, 2), 128, 0, st>>>(RI, RII, tw3, n1, n3, F);
  dft_cols_kernel<<<dim3((unsigned)n1, pb), 128, 0, st>>>(F, tw1, n1, n3, dtau, SC);
  count_launch(3);
}

// Block = 32 x 32 entries of one item, 2 x 2 per thread; 16-wide slices of the contraction
// index in shared memory as fixed point against the slice's largest exponents, one FP64
// addition per slice and component.
template <bool kDagger>
static __global__ void __launch_bounds__(256, 3) kick64_kernel(const double2 *__restrict__ w, double2 *__restrict__ out,
                                                               const double *__restrict__ K, int d, int tiles) {
  constexpr int kTile = 32, kSlice = 16, kLd = kSlice + 1, kPer = kTile * kSlice / 256;
  // K[p][k], w[k][q], then -K[k][q], w[p][k]
  __shared__ __align__(16) int4 w1[2 * kTile * kLd];
  __shared__ __align__(16) int2 k1[2 * kTile * kLd];
  __shared__ int top[2][2];
  const int64_t item = blockIdx.x / (tiles * tiles);
  const int tile = (int)(blockIdx.x - item * tiles * tiles);
  const int p0 = (tile / tiles) * kTile, q0 = (tile % tiles) * kTile;
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const double2 *wi = w + item * d * d;
  auto at = [&](int r, int c) {
    if (!kDagger) return wi[(int64_t)r * d + c];
    const double2 v = wi[(int64_t)c * d + r];
    return make_double2(-v.x, v.y);
  };
  const double2 z = make_double2(0.0, 0.0);
  double2 sum[2][2] = {{z, z}, {z, z}};
  if (t < 4) top[t >> 1][t & 1] = 1;
  __syncthreads();
  int par = 0;
  for (int k0 = 0; k0 < d; k0 += kSlice, par ^= 1) {
    double2 x[2][kPer];
    double m[2][kPer];
    int ek = 1, ew = 1;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int e = t + 256 * i, k = k0 + e % kSlice, r = e / kSlice;       // along rows
      const int r2 = e % kTile, k2 = k0 + e / kTile;                        // along columns
      m[0][i] = k < d && p0 + r < d ? K[(int64_t)(p0 + r) * d + k] : 0.0;
      m[1][i] = k2 < d && q0 + r2 < d ? -K[(int64_t)k2 * d + q0 + r2] : 0.0;
      // the item is read along its own rows: w[k][q] by columns of the tile, or by rows of w^dagger
      x[0][i] = !kDagger ? (k2 < d && q0 + r2 < d ? at(k2, q0 + r2) : z) : (k < d && q0 + r < d ? at(k, q0 + r) : z);
      x[1][i] = !kDagger ? (k < d && p0 + r < d ? at(p0 + r, k) : z) : (k2 < d && p0 + r2 < d ? at(p0 + r2, k2) : z);
    }
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      ek = max(ek, max(exponent(make_double2(m[0][i], m[1][i])), 1));
      ew = max(ew, max(exponent(x[0][i]), exponent(x[1][i])));
    }
    ek = __reduce_max_sync(0xffffffffu, ek);
    ew = __reduce_max_sync(0xffffffffu, ew);
    if ((t & 31) == 0) {
      atomicMax(&top[par][0], ek);
      atomicMax(&top[par][1], ew);
    }
    __syncthreads();   // the last slice's sums are done too
    ek = top[par][0];
    ew = top[par][1];
    if (t < 2) top[par ^ 1][t] = 1;
    if (ek == 0x7ff || ew == 0x7ff) {   // infinities or NaN: as they are
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int p = p0 + ty + 16 * i, q = q0 + tx + 16 * j;
          if (p >= d || q >= d) continue;
          for (int k = k0; k < min(d, k0 + kSlice); ++k) {
            const double2 u = at(k, q), v = at(p, k);
            const double l = K[(int64_t)p * d + k], r = K[(int64_t)k * d + q];
            sum[i][j].x += l * u.x - v.x * r;
            sum[i][j].y += l * u.y - v.y * r;
          }
        }
      __syncthreads();
      continue;
    }
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int e = t + 256 * i, a = e / kSlice * kLd + e % kSlice, b = e % kTile * kLd + e / kTile;
      k1[a] = fixed54(m[0][i], ek);
      k1[kTile * kLd + b] = fixed54(m[1][i], ek);
      w1[kDagger ? a : b] = fixed54(x[0][i], ew);
      w1[kTile * kLd + (kDagger ? b : a)] = fixed54(x[1][i], ew);
    }
    __syncthreads();
    long long hh[2][2][2] = {}, hl[2][2][2] = {};
    auto mad = [&](int i, int j, const int2 &k, const int4 &x) {
      hh[i][j][0] += (long long)k.x * x.x;
      hl[i][j][0] += (long long)k.x * x.y;
      hl[i][j][0] += (long long)k.y * x.x;
      hh[i][j][1] += (long long)k.x * x.z;
      hl[i][j][1] += (long long)k.x * x.w;
      hl[i][j][1] += (long long)k.y * x.z;
    };
#pragma unroll 2
    for (int k = 0; k < kSlice; ++k) {
      const int2 kp[2] = {k1[ty * kLd + k], k1[(ty + 16) * kLd + k]};
      const int4 xq[2] = {w1[tx * kLd + k], w1[(tx + 16) * kLd + k]};
      const int2 kq[2] = {k1[(kTile + tx) * kLd + k], k1[(kTile + tx + 16) * kLd + k]};
      const int4 xp[2] = {w1[(kTile + ty) * kLd + k], w1[(kTile + ty + 16) * kLd + k]};
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          mad(i, j, kp[i], xq[j]);
          mad(i, j, kq[j], xp[i]);
        }
    }
    const Unit54 unit(ek, ew);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        sum[i][j].x = unit.add(hh[i][j][0], hl[i][j][0], sum[i][j].x);
        sum[i][j].y = unit.add(hh[i][j][1], hl[i][j][1], sum[i][j].y);
      }
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int p = p0 + ty + 16 * i, q = q0 + tx + 16 * j;
      if (p < d && q < d) out[(item * d + p) * d + q] = sum[i][j];
    }
}

void kick_tiled(const double2 *w, double2 *out, const double *K, int d, int64_t items, bool dagger, cudaStream_t st) {
  const int tiles = (d + 31) / 32;
  const unsigned blocks = grid_blocks(items * tiles * tiles);
  if (dagger)
    kick64_kernel<true><<<blocks, 256, 0, st>>>(w, out, K, d, tiles);
  else
    kick64_kernel<false><<<blocks, 256, 0, st>>>(w, out, K, d, tiles);
  count_launch(1);
}

__global__ void dft1d_kernel(const double2 *__restrict__ R, int n, double dtau, double *__restrict__ I) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  double s = 0;
  for (int k = 0; k < n; ++k) {
    double sn, cs;
    sincospi(2.0 * (double)((long long)p * k % n) / n, &sn, &cs);
    const double w = k == 0 ? 0.5 : 1.0;
    s += w * (sn * R[k].x + cs * R[k].y);
  }
  I[p] = dtau * s;
}

__global__ void __launch_bounds__(256) stage_kernel_vb(const float2 *__restrict__ w, const float2 *y, float2 *out,
                                                       float alpha, VbModel M, int64_t total) {
  const int d = M.d;
  const int64_t dd = (int64_t)d * d;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t el = e % dd;
    const int64_t bn = e / dd;
    const int n = (int)(bn % M.n_ado);
    const int64_t br = bn / M.n_ado;
    const int a = (int)(el / d), b = (int)(el % d);
    const float2 *wb = w + br * M.n_ado * dd;
    const float2 *wn = wb + (int64_t)n * dd;
    float re = 0.f, im = 0.f;
    const float *Ha = M.H + (int64_t)a * d;
    for (int c = 0; c < d; ++c) {
      const float h1 = Ha[c], h2 = M.H[(int64_t)c * d + b];
      const float2 x = wn[(int64_t)c * d + b], z = wn[(int64_t)a * d + c];
      re += h1 * x.x - z.x * h2;
      im += h1 * x.y - z.y * h2;
    }
    float ore = im, oim = -re;
    const float dec = (float)M.decay[n];
    const float2 self = wn[el];
    ore -= dec * self.x;
    oim -= dec * self.y;
    for (int s = 0; s < M.n_modes; ++s) {
      const int o0 = M.nb_off[n * M.n_modes + s], o1 = M.nb_off[n * M.n_modes + s + 1];
      if (o0 == o1) continue;
      const float la = M.lam[s * d + a], lb = M.lam[s * d + b];
      const float f = la - lb, g = la + lb;
      for (int q = o0; q < o1; ++q) {
        const float2 x = wb[(int64_t)M.nb_idx[q] * dd + el];
        const float p = M.nb_cB[q] * g, qq = M.nb_cA[q] * f;
        ore += p * x.x + qq * x.y;
        oim += p * x.y - qq * x.x;
      }
    }
    const float2 yv = y[e];
    out[e] = make_float2(yv.x + alpha * ore, yv.y + alpha * oim);
  }
}

// Tiled variant for larger bases: one block per 32 x 32 output tile of one item,
// 8 rows x 32 columns of threads with 4 rows each.  The commutator's contraction
// runs over 32-wide slices of H' and w_n staged in shared memory (each element
// reused 32 times instead of re-read per output); the decay and system-bath terms
// are the same elementwise code as stage_kernel_vb, in the same summation order.
__global__ void __launch_bounds__(256) stage_kernel_vb_tiled(const float2 *__restrict__ w, const float2 *y,
                                                             float2 *out, float alpha, VbModel M, int tiles) {
  __shared__ float sHa[32][33], sHb[32][33];
  __shared__ float2 sWa[32][33], sWb[32][33];
  const int d = M.d;
  const int64_t dd = (int64_t)d * d;
  const int64_t item = blockIdx.x / (tiles * tiles);
  const int tile = (int)(blockIdx.x - item * tiles * tiles);
  const int a0 = (tile / tiles) * 32, b0 = (tile % tiles) * 32;
  const int n = (int)(item % M.n_ado);
  const int64_t br = item / M.n_ado;
  const float2 *wb = w + br * M.n_ado * dd;
  const float2 *wn = wb + (int64_t)n * dd;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  float re[4] = {0.f, 0.f, 0.f, 0.f}, im[4] = {0.f, 0.f, 0.f, 0.f};
  for (int c0 = 0; c0 < d; c0 += 32) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = ty + 8 * i;                       // tile row / slice index
      const bool ca = c0 + tx < d, cr = c0 + r < d;
      sHa[r][tx] = (a0 + r < d && ca) ? M.H[(int64_t)(a0 + r) * d + c0 + tx] : 0.f;
      sWa[r][tx] = (a0 + r < d && ca) ? wn[(int64_t)(a0 + r) * d + c0 + tx] : make_float2(0.f, 0.f);
      sHb[r][tx] = (cr && b0 + tx < d) ? M.H[(int64_t)(c0 + r) * d + b0 + tx] : 0.f;
      sWb[r][tx] = (cr && b0 + tx < d) ? wn[(int64_t)(c0 + r) * d + b0 + tx] : make_float2(0.f, 0.f);
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      const float2 x = sWb[k][tx];
      const float h2 = sHb[k][tx];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = ty + 8 * i;
        const float h1 = sHa[r][k];
        const float2 z = sWa[r][k];
        re[i] += h1 * x.x - z.x * h2;
        im[i] += h1 * x.y - z.y * h2;
      }
    }
    __syncthreads();
  }
  const int b = b0 + tx;
  if (b >= d) return;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int a = a0 + ty + 8 * i;
    if (a >= d) continue;
    const int64_t el = (int64_t)a * d + b;
    float ore = im[i], oim = -re[i];
    const float dec = (float)M.decay[n];
    const float2 self = wn[el];
    ore -= dec * self.x;
    oim -= dec * self.y;
    for (int s = 0; s < M.n_modes; ++s) {
      const int o0 = M.nb_off[n * M.n_modes + s], o1 = M.nb_off[n * M.n_modes + s + 1];
      if (o0 == o1) continue;
      const float la = M.lam[s * d + a], lb = M.lam[s * d + b];
      const float f = la - lb, g = la + lb;
      for (int q = o0; q < o1; ++q) {
        const float2 xv = wb[(int64_t)M.nb_idx[q] * dd + el];
        const float p = M.nb_cB[q] * g, qq = M.nb_cA[q] * f;
        ore += p * xv.x + qq * xv.y;
        oim += p * xv.y - qq * xv.x;
      }
    }
    const int64_t e = item * dd + el;
    const float2 yv = y[e];
    out[e] = make_float2(yv.x + alpha * ore, yv.y + alpha * oim);
  }
}

// FP32 commutators K w - w K in register tiles: block = 64 x 64 entries of one item, 4 x 4
// per thread (a warp: 16 rows, 32 columns), 32-wide slices of the contraction index through
// a double buffer in shared memory (cp.async).  Along k the entries by row are read four
// (K) or two (w) at a time, the entries by column two columns at a time: 24 shared loads
// per 384 arithmetic instructions, against 10 per 24 with one column and four rows per
// thread; real and imaginary part take one packed instruction each time, which leaves half
// the issue slots (d = 125, 924 items: stage 715 to 646 us, kick 490 to 461; the FP32
// pipe's rate alone would take 340).  Every entry's operations and their order are those of stage_kernel_vb_tiled and
// kick_kernel<float> (per term a product, a multiply-add and an addition), so the bits are
// the same.
constexpr int kC32Tile = 64, kC32Slice = 32;
constexpr int kC32LdKr = 36, kC32LdWr = 68, kC32LdKc = 68, kC32LdWc = 132;   // in floats
constexpr int kC32Kr = 0, kC32Wr = kC32Kr + kC32Tile * kC32LdKr, kC32Kc = kC32Wr + kC32Tile * kC32LdWr;
constexpr int kC32Wc = kC32Kc + kC32Slice * kC32LdKc, kC32Buf = kC32Wc + kC32Slice * kC32LdWc;
constexpr int kC32Smem = 2 * kC32Buf * 4;

template <int kBytes>
__device__ __forceinline__ void cp_async(float *dst, const void *src, bool ok) {   // zeros if not ok
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "n"(kBytes), "r"(ok ? kBytes : 0));
}

// Two FP32 operations per instruction, each rounded as its scalar form.
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// kOp: 0 out = K w - w K; 1 the same of -w^dagger; 2 RK4 stage of stage_kernel_vb
template <int kOp>
__global__ void __launch_bounds__(256, 2) comm32_kernel(const float2 *__restrict__ w, const float2 *y, float2 *out,
                                                        const float *__restrict__ K, int d, int tiles, float alpha,
                                                        const __grid_constant__ VbModel M) {
  extern __shared__ __align__(16) float c32_smem[];
  const int64_t dd = (int64_t)d * d, item = blockIdx.x / (tiles * tiles);
  const int tile = (int)(blockIdx.x - item * tiles * tiles);
  const int p0 = (tile / tiles) * kC32Tile, q0 = (tile % tiles) * kC32Tile;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int wp = (warp >> 1) * 16 + (lane >> 3), wq = (warp & 1) * 32 + (lane & 7) * 2;   // rows wp + 4 i
  const float2 *wn = w + item * dd;
  // w by rows: w[p][k] (kOp 1: w[q][k]); w by columns: w[k][q] (kOp 1: w[k][p])
  const int r0 = kOp == 1 ? q0 : p0, c0 = kOp == 1 ? p0 : q0;
  auto load = [&](int k0, float *b) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = (t >> 5) + 8 * i, k = k0 + lane;
      const bool kp = p0 + r < d && k < d, wr = r0 + r < d && k < d;
      cp_async<4>(b + kC32Kr + r * kC32LdKr + lane, K + (kp ? (p0 + r) * d + k : 0), kp);
      cp_async<8>(b + kC32Wr + r * kC32LdWr + 2 * lane, wn + (wr ? (r0 + r) * d + k : 0), wr);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int c = t & 63, r = (t >> 6) + 4 * i, k = k0 + r;
      const bool kq = q0 + c < d && k < d, wc = c0 + c < d && k < d;
      cp_async<4>(b + kC32Kc + r * kC32LdKc + c, K + (kq ? k * d + q0 + c : 0), kq);
      cp_async<8>(b + kC32Wc + r * kC32LdWc + 2 * c, wn + (wc ? k * d + c0 + c : 0), wc);
    }
    asm volatile("cp.async.commit_group;");
  };
  unsigned long long sum[4][4] = {};   // complex, packed
  const bool idle = p0 + (warp >> 1) * 16 >= d || q0 + (warp & 1) * 32 >= d;
  load(0, c32_smem);
  for (int k0 = 0, par = 0; k0 < d; k0 += kC32Slice, par ^= 1) {
    asm volatile("cp.async.wait_group 0;");
    __syncthreads();   // this slice is there, and nobody reads the last one any more
    if (k0 + kC32Slice < d) load(k0 + kC32Slice, c32_smem + (par ^ 1) * kC32Buf);
    const float *b = c32_smem + par * kC32Buf;
    const int end = idle ? 0 : min(kC32Slice, d - k0);
    for (int k = 0; k < end; k += 4) {
      float h[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 v = *(const float4 *)(b + kC32Kr + (wp + 4 * i) * kC32LdKr + k);
        h[i][0] = v.x;
        h[i][1] = v.y;
        h[i][2] = v.z;
        h[i][3] = v.w;
      }
#pragma unroll
      for (int k2 = 0; k2 < 4; k2 += 2) {
        float4 wr[4];   // two k of the four rows (kOp 1: of the four columns)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = kOp == 1 ? wq + (i & 1) + 16 * (i >> 1) : wp + 4 * i;
          wr[i] = *(const float4 *)(b + kC32Wr + r * kC32LdWr + 2 * (k + k2));
        }
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
          const float *kc = b + kC32Kc + (k + k2 + kk) * kC32LdKc + wq;
          const float *wc = b + kC32Wc + (k + k2 + kk) * kC32LdWc;
          const float2 ga = *(const float2 *)kc, gb = *(const float2 *)(kc + 16);
          const float g[4] = {ga.x, ga.y, gb.x, gb.y};
          float2 v[4], u[4];   // by row, by column
#pragma unroll
          for (int i = 0; i < 4; ++i) v[i] = kk ? make_float2(wr[i].z, wr[i].w) : make_float2(wr[i].x, wr[i].y);
          if (kOp == 1) {
#pragma unroll
            for (int i = 0; i < 4; ++i) u[i] = *(const float2 *)(wc + 2 * (wp + 4 * i));
          } else {
            const float4 ua = *(const float4 *)(wc + 2 * wq), ub = *(const float4 *)(wc + 2 * wq + 32);
            u[0] = make_float2(ua.x, ua.y);
            u[1] = make_float2(ua.z, ua.w);
            u[2] = make_float2(ub.x, ub.y);
            u[3] = make_float2(ub.z, ub.w);
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float k1 = h[i][k2 + kk], k2_ = g[j];
              if (kOp == 1) {   // the real part's product is the other one
                float2 s = unpack2(sum[i][j]);
                s.x += __fmaf_rn(u[i].x, k2_, -__fmul_rn(k1, v[j].x));
                s.y += __fmaf_rn(k1, v[j].y, -__fmul_rn(u[i].y, k2_));
                sum[i][j] = pack2(s.x, s.y);
              } else {
                sum[i][j] = add2(sum[i][j], fma2(pack2(k1, k1), pack2(u[j].x, u[j].y),
                                                 mul2(pack2(v[i].x, v[i].y), pack2(-k2_, -k2_))));
              }
            }
        }
      }
    }
  }
  __syncthreads();
  // through shared memory, so that a warp's accesses to memory are along rows
  float2 *tilebuf = (float2 *)c32_smem;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      tilebuf[(wp + 4 * i) * kC32Tile + wq + (j & 1) + 16 * (j >> 1)] = unpack2(sum[i][j]);
  __syncthreads();
  const int b = q0 + (t & 63);
  if (b >= d) return;
  const int n = kOp == 2 ? (int)(item % M.n_ado) : 0;
  const float2 *wb = wn - n * dd;
  const float dec = kOp == 2 ? (float)M.decay[n] : 0.f;
  constexpr int kRows = 8;
  auto couple = [](float2 &o, float2 x, float p, float q) {
    o.x += p * x.x + q * x.y;
    o.y += p * x.y - q * x.x;
  };
#pragma unroll 1
  for (int g = 0; g < 64 / 4 / kRows; ++g) {
    const int row = (t >> 6) + 4 * kRows * g;   // rows row + 4 i
    if (p0 + row >= d) break;
    float2 o[kRows];
#pragma unroll
    for (int i = 0; i < kRows; ++i) o[i] = tilebuf[(row + 4 * i) * kC32Tile + (t & 63)];
    if (kOp == 2) {
      int el[kRows];
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        el[i] = min(p0 + row + 4 * i, d - 1) * d + b;
        const float2 self = wn[el[i]];
        o[i] = make_float2(o[i].y - dec * self.x, -o[i].x - dec * self.y);
      }
      for (int s = 0; s < M.n_modes; ++s) {
        const int o0 = M.nb_off[n * M.n_modes + s], o1 = M.nb_off[n * M.n_modes + s + 1];
        if (o0 == o1) continue;
        const float lb = M.lam[s * d + b];
        float f[kRows], gg[kRows];
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
          const float la = M.lam[s * d + min(p0 + row + 4 * i, d - 1)];
          f[i] = la - lb;
          gg[i] = la + lb;
        }
        int q = o0;
        for (; q + 1 < o1; q += 2) {
          const float2 *xn = wb + (int64_t)M.nb_idx[q] * dd, *xn2 = wb + (int64_t)M.nb_idx[q + 1] * dd;
          const float cA = M.nb_cA[q], cB = M.nb_cB[q], cA2 = M.nb_cA[q + 1], cB2 = M.nb_cB[q + 1];
          float2 xv[kRows], xv2[kRows];
#pragma unroll
          for (int i = 0; i < kRows; ++i) {
            xv[i] = xn[el[i]];
            xv2[i] = xn2[el[i]];
          }
#pragma unroll
          for (int i = 0; i < kRows; ++i) {
            couple(o[i], xv[i], cB * gg[i], cA * f[i]);
            couple(o[i], xv2[i], cB2 * gg[i], cA2 * f[i]);
          }
        }
        if (q < o1) {
          const float2 *xn = wb + (int64_t)M.nb_idx[q] * dd;
          const float cA = M.nb_cA[q], cB = M.nb_cB[q];
          float2 xv[kRows];
#pragma unroll
          for (int i = 0; i < kRows; ++i) xv[i] = xn[el[i]];
#pragma unroll
          for (int i = 0; i < kRows; ++i) couple(o[i], xv[i], cB * gg[i], cA * f[i]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int a = p0 + row + 4 * i;
      if (a >= d) break;
      const int64_t e = item * dd + (int64_t)a * d + b;
      if (kOp == 2) {
        const float2 yv = y[e];
        out[e] = make_float2(yv.x + alpha * o[i].x, yv.y + alpha * o[i].y);
      } else {
        out[e] = o[i];
      }
    }
  }
}

template <int kOp>
static void comm32(const float2 *w, const float2 *y, float2 *out, const float *K, int d, int64_t items, float alpha,
                   const VbModel &M, cudaStream_t st) {
  const int tiles = (d + kC32Tile - 1) / kC32Tile;
  CUDA_TRY(cudaFuncSetAttribute(comm32_kernel<kOp>, cudaFuncAttributeMaxDynamicSharedMemorySize, kC32Smem));
  comm32_kernel<kOp><<<grid_blocks(items * tiles * tiles), 256, kC32Smem, st>>>(w, y, out, K, d, tiles, alpha, M);
  count_launch(1);
}

void kick_tiled(const float2 *w, float2 *out, const float *K, int d, int64_t items, bool dagger, cudaStream_t st) {
  dagger ? comm32<1>(w, nullptr, out, K, d, items, 0.f, VbModel{}, st)
         : comm32<0>(w, nullptr, out, K, d, items, 0.f, VbModel{}, st);
}

void stage32(const float2 *w, const float2 *y, float2 *out, float alpha, const VbModel &M, int64_t items,
             cudaStream_t st) {
  const int64_t tiles = (M.d + kC32Tile - 1) / kC32Tile;
  if (M.d >= 36 && items * tiles * tiles >= 152) return comm32<2>(w, y, out, M.H, M.d, items, alpha, M, st);
  const int t32 = (M.d + 31) / 32;
  stage_kernel_vb_tiled<<<grid_blocks(items * t32 * t32), 256, 0, st>>>(w, y, out, alpha, M, t32);
  count_launch(1);
}

__global__ void convert_f64_to_f32(const double2 *__restrict__ x, float2 *__restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = make_float2((float)x[i].x, (float)x[i].y);
}

__global__ void convert_f32_to_f64(const float2 *__restrict__ x, double2 *__restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = make_double2((double)x[i].x, (double)x[i].y);
}

}  // namespace heom
