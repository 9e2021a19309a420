// Non-template kernels: 2D Fourier sums / correlation spectrum and state conversion.
#include "kernels.cuh"

namespace heom {

void count_launch(uint64_t n);

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

__global__ void convert_f64_to_f32(const double2 *__restrict__ x, float2 *__restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = make_float2((float)x[i].x, (float)x[i].y);
}

__global__ void convert_f32_to_f64(const float2 *__restrict__ x, double2 *__restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = make_double2((double)x[i].x, (double)x[i].y);
}

}  // namespace heom
