// Kernels of the discrete adjoint of the FP64 propagation (reverse mode through
// the RK4 stages, kicks and traces of Sec. II.C), used by heom_response_2d_grad.
//
// Inner product: <x, y> = Re sum conj(x) y over every entry of every ADO and
// branch.  For a complex-linear map y = A x the adjoint is the conjugate
// transpose; the gradient of a real loss with respect to a real model entry M is
// Re <ybar, (dA/dM) x>.  The RHS adjoint L^H has the structure of L itself
// (H -> -H, each coupling entry n <- m with (cA, cB) becomes m <- n with
// (-cA, cB)), so it runs through the FP64 stages with a second set of tables (f64_stage.h,
// in the coupling eigenbasis; stage_kernel<double> for models that it does not take);
// the kernels here only accumulate the model gradients and apply the trace and
// dagger adjoints.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

#include "f64_stage.h"
#include "fixed54.cuh"
#include "kernels.cuh"

namespace heom {

constexpr int kAdjMaxExp = 32;
constexpr int kAdjMaxVl = 4 * 16 * 16;   // sum_s n_s^2 (n_s <= 16)

// y += a x over n complex entries.
static __global__ void __launch_bounds__(256) axpy_kernel(double2 *__restrict__ y, const double2 *__restrict__ x, double a,
                                                   int64_t n) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const double2 v = x[e];
    y[e].x += a * v.x;
    y[e].y += a * v.y;
  }
}

// out_n = -(in_n)^dagger for every ADO matrix (the map that turns the R_I trunk
// into the R_II trunk; as a real-linear map it is its own adjoint).
static __global__ void __launch_bounds__(256) neg_dagger_kernel(const double2 *__restrict__ in, double2 *__restrict__ out,
                                                         int d, int64_t total) {
  const int64_t dd = (int64_t)d * d;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t el = e % dd, base = e - el;
    const int a = (int)(el / d), b = (int)(el % d);
    const double2 v = in[base + (int64_t)b * d + a];
    out[e] = make_double2(-v.x, v.y);
  }
}

// Commutator-type gradient: for every item (ADO matrix) i,
//   G[p][q] += alpha Re[ phase ( sum_b conj(g_i[p][b]) w_i[q][b] - sum_a w_i[a][p] conj(g_i[a][q]) ) ],
// the derivative of Re <g, phase^* ... > with respect to a matrix K in K^x w
// (phase = -i for the Hamiltonian term -i[H, w], 1 for a kick K^x w).  Only the
// component the phase selects is accumulated: the imaginary part for -i, the real
// part for 1 (half the arithmetic of the full complex product).
// GB300 issues 2 FP64 operations per clock and SM, on the FP64 tensor instruction too, but
// 32 multiply-adds of 32 x 32 + 64 bits, so the sums run in integers: the entries of a
// 16-wide slice as 54-bit fixed point against the slice's largest exponent, in limbs of 28
// and 26 bits, three products each (low x low, 2^-58 of the largest, dropped), 64 exact
// products per sum, then one FP64 addition.  Block = (16 T)^2 entries of G over a share of
// the (item, slice) units, T x T per thread.  At d = 64, 224 items: 649 us with one FP64
// sum per thread, 452 us in register tiles (the FP64 pipe's
// rate, also of its mma.m8n8k4 form), 133 us here; rms error 1.0e-16 of the largest entry,
// FP64 sums 3.9e-16.
constexpr int kCommSlice = 16, kCommLd = kCommSlice + 1;

constexpr int comm_smem(int T) { return 4 * 16 * T * kCommLd * 16 + 256 * T * T * 8; }

template <bool kImag, int T>
__global__ void __launch_bounds__(256, 2) comm_grad_kernel(const double2 *__restrict__ g,
                                                           const double2 *__restrict__ w, int64_t n_items, int d,
                                                           double alpha, double *__restrict__ G) {
  constexpr int kTile = 16 * T, kPer = kTile * kCommSlice / 256;
  extern __shared__ __align__(16) int4 comm_smem_[];
  // [entry row or column][slice index]: g and w along their columns, w and g along their rows
  int4 *g1 = comm_smem_, *w1 = g1 + kTile * kCommLd, *w2 = w1 + kTile * kCommLd, *g2 = w2 + kTile * kCommLd;
  double *sum = (double *)(g2 + kTile * kCommLd);   // [T * T][256]
  __shared__ int top[2][2];
  const int tiles = (d + kTile - 1) / kTile, slices = (d + kCommSlice - 1) / kCommSlice;
  const int tile = blockIdx.x % (tiles * tiles);
  const int chunk = blockIdx.x / (tiles * tiles), n_chunks = gridDim.x / (tiles * tiles);
  const int p0 = (tile / tiles) * kTile, q0 = (tile % tiles) * kTile;
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int64_t dd = (int64_t)d * d;
  const double2 z = make_double2(0.0, 0.0);
#pragma unroll
  for (int i = 0; i < T * T; ++i) sum[i * 256 + t] = 0.0;
  if (t < 4) top[t >> 1][t & 1] = 1;
  __syncthreads();
  int par = 0;
  for (int64_t u = chunk; u < n_items * slices; u += n_chunks, par ^= 1) {
    const int64_t item = u / slices;
    const int k0 = (int)(u - item * slices) * kCommSlice;
    const double2 *gi = g + item * dd, *wi = w + item * dd;
    double2 x[4][kPer];
    int eg = 1, ew = 1;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int e = t + 256 * i, k = k0 + e % kCommSlice, r = e / kCommSlice;
      const int r2 = e % kTile, k2 = k0 + e / kTile;
      x[0][i] = k < d && p0 + r < d ? gi[(int64_t)(p0 + r) * d + k] : z;
      x[1][i] = k < d && q0 + r < d ? wi[(int64_t)(q0 + r) * d + k] : z;
      x[2][i] = k2 < d && p0 + r2 < d ? wi[(int64_t)k2 * d + p0 + r2] : z;
      x[3][i] = k2 < d && q0 + r2 < d ? gi[(int64_t)k2 * d + q0 + r2] : z;
    }
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      eg = max(eg, max(exponent(x[0][i]), exponent(x[3][i])));
      ew = max(ew, max(exponent(x[1][i]), exponent(x[2][i])));
    }
    eg = __reduce_max_sync(0xffffffffu, eg);
    ew = __reduce_max_sync(0xffffffffu, ew);
    if ((t & 31) == 0) {
      atomicMax(&top[par][0], eg);
      atomicMax(&top[par][1], ew);
    }
    __syncthreads();   // the last unit's sums are done too
    eg = top[par][0];
    ew = top[par][1];
    if (t < 2) top[par ^ 1][t] = 1;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int e = t + 256 * i, a = e / kCommSlice * kCommLd + e % kCommSlice, b = e % kTile * kCommLd + e / kTile;
      // Im conj(g) w = (-g.im, g.re) . w and -Im w conj(g) = (-w.im, w.re) . g; or the real parts
      g1[a] = fixed54(kImag ? make_double2(-x[0][i].y, x[0][i].x) : x[0][i], eg);
      w1[a] = fixed54(x[1][i], ew);
      w2[b] = fixed54(make_double2(kImag ? -x[2][i].y : -x[2][i].x, kImag ? x[2][i].x : -x[2][i].y), ew);
      g2[b] = fixed54(x[3][i], eg);
    }
    __syncthreads();
    long long hh[T][T], hl[T][T];
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
      for (int j = 0; j < T; ++j) hh[i][j] = hl[i][j] = 0;
#pragma unroll 2
    for (int k = 0; k < 2 * kCommSlice; ++k) {
      const int o = k / kCommSlice * 2 * kTile * kCommLd + k % kCommSlice;   // g1 and w1, then w2 and g2
      int4 b[T];
#pragma unroll
      for (int j = 0; j < T; ++j) b[j] = w1[o + (tx + 16 * j) * kCommLd];
#pragma unroll
      for (int i = 0; i < T; ++i) {
        const int4 a = g1[o + (ty + 16 * i) * kCommLd];
#pragma unroll
        for (int j = 0; j < T; ++j) {
          hh[i][j] += (long long)a.x * b[j].x;
          hl[i][j] += (long long)a.x * b[j].y;
          hh[i][j] += (long long)a.z * b[j].z;
          hl[i][j] += (long long)a.y * b[j].x;
          hl[i][j] += (long long)a.z * b[j].w;
          hl[i][j] += (long long)a.w * b[j].z;
        }
      }
    }
    const Unit54 unit(eg, ew);
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
      for (int j = 0; j < T; ++j) {
        double *s = sum + (i * T + j) * 256 + t;
        *s = unit.add(hh[i][j], hl[i][j], *s);
      }
  }
#pragma unroll
  for (int i = 0; i < T; ++i)
#pragma unroll
    for (int j = 0; j < T; ++j) {
      const int p = p0 + ty + 16 * i, q = q0 + tx + 16 * j;
      if (p < d && q < d) atomicAdd(G + (int64_t)p * d + q, alpha * sum[(i * T + j) * 256 + t]);
    }
}

// Gradients of the system-bath and decay terms of L (Eq. HEOM_DB) for one pair
// (g, w) of an adjoint and a forward state, summed over branches and ADOs:
//   Gv[s][p][r]  += alpha d/dv_s[p][r]   Re <g, V X^L - X^R V>,  X^L = sum (-i cA + cB) w_m,
//                                                                X^R = sum (-i cA - cB) w_m
//   Gre[j], Gim[j] += alpha n_j Re <g_n, -i [V_s, w_{n-e_j}]>,  alpha n_j Re <g_n, {V_s, w_{n-e_j}}>
//   Gnu[j]       -= alpha n_j Re <g_n, w_n>
// (cA = n_j Re c_j and cB = n_j Im c_j on down-neighbours; up-neighbours carry
// constants).  One block per item; warps walk rows for the V X^L part (mode
// digit of the row uniform per warp) and columns for the X^R V part.
// entry_exp[q] = exponential j of a down-neighbour entry, -1 for up entries.
static __global__ void __launch_bounds__(256) coupling_grad_kernel(const double2 *__restrict__ g,
                                                            const double2 *__restrict__ w, DevModel<double> M,
                                                            const int *__restrict__ ado, int n_exp,
                                                            const int *__restrict__ entry_exp, int64_t n_items,
                                                            double alpha, double *__restrict__ Gv,
                                                            double *__restrict__ Gre, double *__restrict__ Gim,
                                                            double *__restrict__ Gnu) {
  __shared__ double s_v[kAdjMaxVl];
  __shared__ double s_re[kAdjMaxExp], s_im[kAdjMaxExp];
  __shared__ double s_dot;
  const int d = M.d, S = M.n_modes;
  const int64_t dd = (int64_t)d * d;
  int nvl = 0;
  for (int s = 0; s < S; ++s) nvl += M.dims[s] * M.dims[s];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
    for (int i = threadIdx.x; i < nvl; i += blockDim.x) s_v[i] = 0.0;
    for (int i = threadIdx.x; i < n_exp; i += blockDim.x) s_re[i] = s_im[i] = 0.0;
    if (threadIdx.x == 0) s_dot = 0.0;
    __syncthreads();
    const int n = (int)(item % M.n_ado);
    const double2 *gn = g + item * dd;
    const double2 *wb = w + (item - n) * dd;     // first ADO of this branch
    double dot = 0.0;
    // rows: V X^L part, decay, and the exponential gradients
    for (int a = warp; a < d; a += nwarps) {
      for (int c0 = 0; c0 < d; c0 += 32) {
        const int c = c0 + lane;
        const bool ok = c < d;
        const double2 gv = ok ? gn[(int64_t)a * d + c] : make_double2(0.0, 0.0);
        if (ok) {
          const double2 wv = wb[(int64_t)n * dd + (int64_t)a * d + c];
          dot += gv.x * wv.x + gv.y * wv.y;
        }
        for (int s = 0; s < S; ++s) {
          const int ns = M.dims[s], st = M.stride[s];
          const int as = (a / st) % ns, cs = ok ? (c / st) % ns : 0;
          const double *v = M.vloc + M.vloc_off[s];
          const int lo = M.nb_off[n * S + s], hi = M.nb_off[n * S + s + 1];
          for (int q = lo; q < hi; ++q) {
            const double2 *wm = wb + (int64_t)M.nb_idx[q] * dd;
            const double cA = M.nb_cA[q], cB = M.nb_cB[q];
            const int j = entry_exp[q];
            double vw_r = 0, vw_i = 0;
            for (int r = 0; r < ns; ++r) {
              const double2 x = ok ? wm[(int64_t)(a + (r - as) * st) * d + c] : make_double2(0.0, 0.0);
              // conj(g) (-i cA + cB) x, real part
              const double kr = cB, ki = -cA;
              const double xr = kr * x.x - ki * x.y, xi = kr * x.y + ki * x.x;
              double val = gv.x * xr + gv.y * xi;
              for (int o = 16; o > 0; o >>= 1) val += __shfl_xor_sync(0xffffffffu, val, o);
              if (lane == 0) atomicAdd(&s_v[M.vloc_off[s] + as * ns + r], val);
              if (j >= 0) {
                const double vv = v[as * ns + r];
                vw_r += vv * x.x;
                vw_i += vv * x.y;
              }
            }
            if (j >= 0) {   // (V w_m)[a][c] and (w_m V)[a][c]
              double wv_r = 0, wv_i = 0;
              for (int r = 0; r < ns; ++r) {
                const double2 x = ok ? wm[(int64_t)a * d + c + (r - cs) * st] : make_double2(0.0, 0.0);
                const double vv = v[r * ns + cs];
                wv_r += x.x * vv;
                wv_i += x.y * vv;
              }
              const double nj = (double)ado[(int64_t)n * n_exp + j];
              const double cm_r = vw_r - wv_r, cm_i = vw_i - wv_i;   // [V, w]
              const double ac_r = vw_r + wv_r, ac_i = vw_i + wv_i;   // {V, w}
              // Re conj(g) (-i [V, w]) = g.x * cm_i - g.y * cm_r
              double vre = nj * (gv.x * cm_i - gv.y * cm_r);
              double vim = nj * (gv.x * ac_r + gv.y * ac_i);
              for (int o = 16; o > 0; o >>= 1) {
                vre += __shfl_xor_sync(0xffffffffu, vre, o);
                vim += __shfl_xor_sync(0xffffffffu, vim, o);
              }
              if (lane == 0) {
                atomicAdd(&s_re[j], vre);
                atomicAdd(&s_im[j], vim);
              }
            }
          }
        }
      }
    }
    // columns: - X^R V part
    for (int c = warp; c < d; c += nwarps) {
      for (int a0 = 0; a0 < d; a0 += 32) {
        const int a = a0 + lane;
        const bool ok = a < d;
        const double2 gv = ok ? gn[(int64_t)a * d + c] : make_double2(0.0, 0.0);
        for (int s = 0; s < S; ++s) {
          const int ns = M.dims[s], st = M.stride[s];
          const int cs = (c / st) % ns;
          const int lo = M.nb_off[n * S + s], hi = M.nb_off[n * S + s + 1];
          for (int q = lo; q < hi; ++q) {
            const double2 *wm = wb + (int64_t)M.nb_idx[q] * dd;
            const double cA = M.nb_cA[q], cB = M.nb_cB[q];
            for (int p = 0; p < ns; ++p) {
              const double2 x = ok ? wm[(int64_t)a * d + c + (p - cs) * st] : make_double2(0.0, 0.0);
              // conj(g) (-i cA - cB) x, real part, with a minus sign
              const double kr = -cB, ki = -cA;
              const double xr = kr * x.x - ki * x.y, xi = kr * x.y + ki * x.x;
              double val = -(gv.x * xr + gv.y * xi);
              for (int o = 16; o > 0; o >>= 1) val += __shfl_xor_sync(0xffffffffu, val, o);
              if (lane == 0) atomicAdd(&s_v[M.vloc_off[s] + p * ns + cs], val);
            }
          }
        }
      }
    }
    for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    if (lane == 0) atomicAdd(&s_dot, dot);
    __syncthreads();
    for (int i = threadIdx.x; i < nvl; i += blockDim.x)
      if (s_v[i] != 0.0) atomicAdd(Gv + i, alpha * s_v[i]);
    for (int j = threadIdx.x; j < n_exp; j += blockDim.x) {
      const double nj = (double)ado[(int64_t)n * n_exp + j];
      if (s_re[j] != 0.0) atomicAdd(Gre + j, alpha * s_re[j]);
      if (s_im[j] != 0.0) atomicAdd(Gim + j, alpha * s_im[j]);
      if (nj != 0.0) atomicAdd(Gnu + j, -alpha * nj * s_dot);
    }
    __syncthreads();
  }
}

// The same gradients in the coupling eigenbasis, where V_s is diagonal: with
// A = sum cA w_m and B = sum cB w_m over the coupling list of (n, s) summed first,
//   Gv[s][p][r] += alpha Re <g, V X^L - X^R V>_{pr},  X^L = B - i A, X^R = -B - i A
// is a contraction over everything but the mode's digit, and the exponentials' terms are
// elementwise.  One block per (item, mode, side, 16 columns (left) or rows (right,
// transposed)): g and X in shared memory, n_s x n_s sums per thread.  Bound by the FP64
// pipe and, with few items, by one block's chain (hence the split over panels).  At
// d = 64, 224 items: 1284 us with a warp reduction per neighbour and digit, 166 us here;
// 28 items: 980 and 42 us (one block for all panels: 260 and 93 us).
constexpr int kGradPanel = 16, kGradLd = kGradPanel + 1, kGradMaxN = 6;
constexpr int kGradSmem = 226 * 1024;   // dynamic, beside 0.8 KB of static arrays

struct CouplingGradArgs {
  const double2 *g, *w;
  F64Ops O;
  const int *ado, *entry_exp;
  int n_exp, splits;
  double alpha;
  double *Gv, *Gre, *Gim, *Gnu;
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sums of v[0..M) over the warp, added to sums[0..M): a halving exchange, M additions per
// lane instead of 5 M.
template <int M, int O = 16, int kAll>
__device__ __forceinline__ void warp_halve(double (&v)[kAll]) {
  constexpr int kHalf = (M + 1) / 2;
  const bool up = M > 1 && (threadIdx.x & O);
#pragma unroll
  for (int i = 0; i < kHalf; ++i) {
    const double hi = i + kHalf < M ? v[i + kHalf] : 0.0;
    v[i] = (up ? hi : v[i]) + __shfl_xor_sync(0xffffffffu, M == 1 || up ? v[i] : hi, O);
  }
  if constexpr (O > 1) warp_halve<kHalf, O / 2>(v);
}

// Entry that slot e of this lane holds after warp_halve<M, O>, or -1
template <int M, int O = 16>
__device__ __forceinline__ int halved_entry(int e) {
  constexpr int kHalf = (M + 1) / 2;
  if constexpr (O > 1) e = halved_entry<kHalf, O / 2>(e);
  if (threadIdx.x & O) e = M > 1 && e >= 0 ? e + kHalf : -1;
  return e < M ? e : -1;
}

template <int M>
__device__ __forceinline__ void warp_sums(double (&v)[M], double *sums) {
  warp_halve<M>(v);
#pragma unroll
  for (int i = 0; i < (M + 31) / 32; ++i) {
    const int e = halved_entry<M>(i);
    if (e >= 0) atomicAdd(sums + e, v[i]);
  }
}

template <int N>
__device__ __forceinline__ void coupling_grad_unit(const CouplingGradArgs &P, int64_t item, int s, int split,
                                                   bool right, double *sums, double *ex) {
  extern __shared__ __align__(16) double2 grad_smem[];
  const F64Ops &O = P.O;
  const int d = O.d, S = O.n_modes, n = (int)(item % O.n_ado);
  const int64_t dd = (int64_t)d * d;
  double2 *gs = grad_smem, *xs = gs + d * kGradLd;
  const double2 *g = P.g + item * dd, *wb = P.w + (item - n) * dd;
  const int q0 = O.noff[n * S + s], q1 = O.noff[n * S + s + 1];
  const bool self = s == 0 && !right;
  if (q0 == q1 && !self) return;
  int str = 1;
  for (int t = s + 1; t < S; ++t) str *= O.dims[t];
  const int t = threadIdx.x, lane = t & 31;
  for (int i = t; i < 2 * P.n_exp + 1; i += blockDim.x) ex[i] = 0.0;
  if (t < N * N) sums[t] = 0.0;
  __syncthreads();
  const uint16_t *dig = O.dig + s * d;
  double acc[N * N], norm = 0.0;
#pragma unroll
  for (int i = 0; i < N * N; ++i) acc[i] = 0.0;
  for (int p0 = split * kGradPanel; p0 < d; p0 += P.splits * kGradPanel) {
    const int np = min(kGradPanel, d - p0);
    // entry i of the panel: left, column p0 + l, row c; right, row p0 + l, column c
    auto place = [&](int i, int &c, int &l) {
      if (right) {
        l = i / d;
        c = i - l * d;
      } else {
        c = i / kGradPanel;
        l = i % kGradPanel;
      }
      return l < np;
    };
    for (int i = t; i < d * kGradPanel; i += blockDim.x) {
      int c, l;
      if (!place(i, c, l)) continue;
      const int64_t el = right ? (int64_t)(p0 + l) * d + c : (int64_t)c * d + p0 + l;
      const double2 u = g[el];
      gs[c * kGradLd + l] = u;
      xs[c * kGradLd + l] = make_double2(0.0, 0.0);
      if (self) {
        const double2 v = wb[n * dd + el];
        norm = fma(u.y, v.y, fma(u.x, v.x, norm));
      }
    }
    for (int q = q0; q < q1; ++q) {
      const F64Entry en = O.nb[q];
      const double2 *xq = wb + (int64_t)en.idx * dd;
      // down-neighbours: Re <g, -i [V, w]> and Re <g, {V, w}>
      const int j = right ? -1 : P.entry_exp[q];
      const double cB = en.kind == 2 ? (right ? -en.cB : en.cB) : 0.0;
      double a = 0.0, b = 0.0;
      for (int i = t; i < d * kGradPanel; i += blockDim.x) {   // the same thread's entries every time
        int c, l;
        if (!place(i, c, l)) continue;
        const double2 v = xq[right ? (int64_t)(p0 + l) * d + c : (int64_t)c * d + p0 + l];
        double2 *px = xs + c * kGradLd + l;
        double2 x = *px;
        x.x = fma(en.cA, v.y, x.x);
        x.y = fma(-en.cA, v.x, x.y);
        if (en.kind == 2) {
          x.x = fma(cB, v.x, x.x);
          x.y = fma(cB, v.y, x.y);
        }
        *px = x;
        if (j >= 0) {
          const double2 u = gs[c * kGradLd + l], fg = O.fg[O.tab_off[s] + dig[c] * N + dig[p0 + l]];
          a = fma(fg.x, fma(u.x, v.y, -u.y * v.x), a);
          b = fma(fg.y, fma(u.x, v.x, u.y * v.y), b);
        }
      }
      if (j >= 0) {
        a = warp_sum(a);
        b = warp_sum(b);
        if (lane == 0) {
          atomicAdd(&ex[2 * j], a);
          atomicAdd(&ex[2 * j + 1], b);
        }
      }
    }
    __syncthreads();
    if (q0 < q1)
      for (int i = t; i < d / N * kGradPanel; i += blockDim.x) {
        const int l = i % kGradPanel, f = i / kGradPanel;
        if (l >= np) continue;
        const int base = (f / str) * str * N + f % str;
        double2 x[N];
  #pragma unroll
        for (int r = 0; r < N; ++r) x[r] = xs[(base + r * str) * kGradLd + l];
  #pragma unroll
        for (int p = 0; p < N; ++p) {
          const double2 v = gs[(base + p * str) * kGradLd + l];
  #pragma unroll
          for (int r = 0; r < N; ++r) {
            acc[p * N + r] = fma(v.x, x[r].x, acc[p * N + r]);
            acc[p * N + r] = fma(v.y, x[r].y, acc[p * N + r]);
          }
        }
      }
    __syncthreads();
  }
  if (self) {
    norm = warp_sum(norm);
    if (lane == 0) atomicAdd(&ex[2 * P.n_exp], norm);
  }
  if (q0 < q1) warp_sums(acc, sums);
  __syncthreads();
  // left: V's row digit from g, column digit from X; right: the other way, subtracted
  if (q0 < q1 && t < N * N) {
    const int p = t / N, r = t % N;
    atomicAdd(P.Gv + O.tab_off[s] + (right ? r * N + p : p * N + r), (right ? -P.alpha : P.alpha) * sums[t]);
  }
  if (right) return;
  for (int j = t; j < P.n_exp; j += blockDim.x) {
    const double nj = P.alpha * P.ado[(int64_t)n * P.n_exp + j];
    if (nj == 0.0) continue;
    if (ex[2 * j] != 0.0) atomicAdd(P.Gre + j, nj * ex[2 * j]);
    if (ex[2 * j + 1] != 0.0) atomicAdd(P.Gim + j, nj * ex[2 * j + 1]);
    if (self) atomicAdd(P.Gnu + j, -nj * ex[2 * P.n_exp]);
  }
}

// kMax: the largest mode basis of the model (fewer sums per thread, more blocks per SM)
template <int kMax>
__global__ void __launch_bounds__(256, kMax > 4 ? 2 : 4)
    coupling_grad_vb_kernel(const __grid_constant__ CouplingGradArgs P) {
  __shared__ double sums[kGradMaxN * kGradMaxN], ex[2 * kAdjMaxExp + 1];
  const int per = 2 * P.splits * P.O.n_modes;
  const int64_t item = blockIdx.x / per;
  const int u = (int)(blockIdx.x - item * per), split = (u >> 1) % P.splits, s = (u >> 1) / P.splits;
  const bool right = u & 1;
  switch (P.O.dims[s]) {
    case 1: return coupling_grad_unit<1>(P, item, s, split, right, sums, ex);
    case 2: return coupling_grad_unit<2>(P, item, s, split, right, sums, ex);
    case 3: return coupling_grad_unit<3>(P, item, s, split, right, sums, ex);
    case 4: return coupling_grad_unit<4>(P, item, s, split, right, sums, ex);
  }
  if constexpr (kMax > 4) {
    if (P.O.dims[s] == 5) return coupling_grad_unit<5>(P, item, s, split, right, sums, ex);
    coupling_grad_unit<6>(P, item, s, split, right, sums, ex);
  }
}

// Trace adjoint: R_b = c tr{mu rho_{b,0}} for every branch b, c = i^order.
// lam_{b,0} += conj(c) Rbar_b mu^T, and Gmu[p][q] += Re(conj(Rbar_b) c rho_{b,0}[q][p]).
static __global__ void __launch_bounds__(256) trace_adjoint_kernel(double2 *__restrict__ lam, const double2 *__restrict__ rho,
                                                            const double2 *__restrict__ rbar, int64_t rbar_stride,
                                                            const double *__restrict__ mu, int d, int64_t per_branch,
                                                            int branches, double c_re, double c_im,
                                                            double *__restrict__ Gmu) {
  const int64_t dd = (int64_t)d * d;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < dd; e += (int64_t)gridDim.x * blockDim.x) {
    const int a = (int)(e / d), b = (int)(e % d);
    const double m = mu[(int64_t)b * d + a];
    double gsum = 0.0;
    for (int br = 0; br < branches; ++br) {
      const double2 rb = rbar[(int64_t)br * rbar_stride];
      // conj(c) Rbar
      const double t_re = c_re * rb.x + c_im * rb.y, t_im = c_re * rb.y - c_im * rb.x;
      double2 &l = lam[(int64_t)br * per_branch + e];
      l.x += t_re * m;
      l.y += t_im * m;
      // Re(conj(Rbar) c rho[b][a]) for G[a][b]
      const double2 r = rho[(int64_t)br * per_branch + (int64_t)b * d + a];
      const double u_re = rb.x * c_re + rb.y * c_im, u_im = rb.x * c_im - rb.y * c_re;   // conj(Rbar) c
      gsum += u_re * r.x - u_im * r.y;
    }
    Gmu[e] += gsum;
  }
}

}  // namespace heom
