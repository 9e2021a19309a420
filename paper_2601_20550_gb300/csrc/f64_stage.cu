// FP64 stage out = y + alpha L(w) in the coupling eigenbasis (declared in f64_stage.h).
//
// What bounds it.  GB300 issues 2 FP64 operations per clock and SM, 1/64 of its FP32
// rate.  The commutator's 2 x 2 x d multiply-adds per element were nine tenths of the
// stage on that pipe.  Here they run as integer products on the IMAD pipe (32 IMAD.WIDE
// per clock and SM): w (per item, or per column and row) and H' are rounded to 57-bit fixed
// point and cut into two signed limbs, 31 bits above 26, and
//   sum_c h z = 2^52 sum h1 z1 + 2^26 sum (h1 z0 + h0 z1)   (+ 2^0 sum h0 z0, dropped: each
//   term at most 2^-62 of the largest value that the sum can take, so 2^-56.8 for the 37
//   products of a row at four levels, 2^-54 for the 250 that 57 bits allow)
// is accumulated without rounding in two 64-bit integers, three IMAD.WIDE per product;
// only H''s structural non-zeros are multiplied (37 of 64 columns at four levels, 61 of
// 125 at five).  The sums are rounded once when they turn back into FP64.  The
// elementwise rest takes ~38 FP64 operations per element and stage and shares the SM
// with the integer phase of other resident blocks.
//
// Accuracy is that of FP64 relative to the largest entry of an ADO (of a column or row of
// it in the panels of large bases), not entry by entry: the change of basis alone mixes an
// ADO's entries.  One mode of six levels, 40 steps from the ground state: the populations of
// levels 1 to 5, 2e-7 to 2e-10, have absolute errors near 1e-17, relative ones of 1e-10 to
// 6e-8 (2e-14 and less with stage_kernel<double> in the product basis).
#include "f64_stage.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <stdexcept>
#include <type_traits>

#include <cooperative_groups.h>

#include "internal.h"

namespace cg = cooperative_groups;

namespace heom {

namespace {

// Columns (rows) of a panel, and the most threads of its block.
constexpr int kPanel = 16;
__host__ __device__ constexpr int panel_threads(int R) { return R == 5 ? 320 : 384; }
__host__ __device__ constexpr int panel_blocks(int R) { return R == 4 ? 2 : 3; }   // per SM, of that many
constexpr int kF64MaxExp = 16;             // build_hierarchy's limit
constexpr int kRotPad = 33;
// Largest basis of f64_small_kernel and rotate_item_kernel (row and column in six bits).
// Two steps at d = 36, 7 ADOs: 142 us in one launch, 352 with a launch per stage; 84
// items: 324 and 441 us.
constexpr int kSmallD = 48;
constexpr size_t kMaxSmem = 227 * 1024;
// Bases whose items fit a block, two of them per SM (up to 83 states), take the items'
// arithmetic; larger ones always go by panels of columns and rows.
constexpr size_t kFusedSmem = 112 * 1024;

struct F64Set {
  F64Ops O;
  const double2 *w, *y;
  double2 *out, *tp;
  int64_t begin;      // first block of the set
  int64_t items;
  int per_block;      // fused: items per block; panels: panels per item
  int smem_t;         // fused: commutator part kept in shared memory
};

struct F64Args {
  F64Set one;
  const F64Set *many;
  int n;
  double alpha;
};

template <bool kMulti>
__device__ __forceinline__ const F64Set &pick(const F64Args &P) {
  if (!kMulti) return P.one;
  int k = 0;
  while (k + 1 < P.n && (int64_t)blockIdx.x >= P.many[k + 1].begin) ++k;
  return P.many[k];
}

__device__ __forceinline__ int exp_field(double2 v) {
  return max((__double2hiint(v.x) >> 20) & 0x7ff, (__double2hiint(v.y) >> 20) & 0x7ff);
}

// x (exponent field at most emax) as round(x 2^(1021 + bits - emax)), magnitude at most
// 2^(bits - 1), in two signed limbs hi 2^low + lo.  Integer operations only: a conversion
// instruction would take the FP64 pipe.
__device__ __forceinline__ int2 to_limbs(double x, int emax, int bits, int low) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  const long long m = ((b & 0xfffffffffffffLL) | (e > 0 ? 1LL << 52 : 0LL)) << (bits - 54);
  const int sh = min(emax - max(e, 1), 62);
  long long v = (m + ((1LL << sh) >> 1)) >> sh;
  v = b < 0 ? -v : v;
  int2 r;
  r.y = ((int)((unsigned)v << (32 - low))) >> (32 - low);
  r.x = (int)((v - r.y) >> low);
  return r;
}

// Factor alpha 2^k of a finished sum, k the exponent of its unit (see to_limbs, f64_build
// and finish), formed by adding to alpha's exponent field.  Below the normal range the
// sum takes 2^-64 of it (deep); NaN for a column that holds an infinity or a NaN.
struct Unit {
  double f;
  bool deep;
};

__device__ __forceinline__ Unit unit(int emax, int hexp, double alpha) {
  if (emax >= 0x7ff) return {__longlong_as_double(0x7ff8000000000000LL), false};
  const long long a = __double_as_longlong(alpha);
  const int k = emax + hexp - 1083, e = (int)((a >> 52) & 0x7ff) + k;
  if ((a << 1) == 0) return {0.0, false};
  if (e >= 0x7ff) return {alpha * __longlong_as_double(0x7ff0000000000000LL), false};
  if (e > 0) return {__longlong_as_double(a + ((long long)k << 52)), false};
  return {e > -64 ? __longlong_as_double(a + ((long long)(k + 64) << 52)) : 0.0, true};
}

__device__ __forceinline__ double sum_value(long long t, const Unit &u) {
  const double v = __ll2double_rn(t);
  return u.deep ? v * 5.421010862427522e-20 : v;   // 2^-64
}

template <int R>
struct Acc {
  long long h[R], x[R];
};

// Rows g R .. g R + R - 1 of H' times one real column of w (the real or imaginary parts
// of a complex one) at zl, elements stride apart.  One component per lane: ten 64-bit
// sums of five rows leave room for 1152 threads per SM.
template <int R>
__device__ __forceinline__ void group_product(const F64Ops &O, int g, const int2 *zl, int stride, Acc<R> &A) {
  constexpr int RP = (R + 1) / 2;
#pragma unroll
  for (int r = 0; r < R; ++r) A.h[r] = A.x[r] = 0;
  auto mac = [&](int r, int hx, int hy, const int2 &z) {
    A.h[r] += (long long)hx * z.x;
    A.x[r] += (long long)hx * z.y;
    A.x[r] += (long long)hy * z.x;
  };
  const int f1 = O.foff[g + 1];
  const int4 *fh = O.fh;
#pragma unroll 2
  for (int q = O.foff[g]; q < f1; ++q) {
    int4 h[RP];
#pragma unroll
    for (int p = 0; p < RP; ++p) h[p] = fh[q * RP + p];
    const int2 z = zl[(R % 2 ? h[RP - 1].z : O.fc[q]) * stride];
#pragma unroll
    for (int p = 0; p < RP; ++p) {
      mac(2 * p, h[p].x, h[p].y, z);
      if (2 * p + 1 < R) mac(2 * p + 1, h[p].z, h[p].w, z);
    }
  }
  // columns between states that differ in the two leading modes: the last digit stays,
  // so row r meets column c + r, all with one factor
  const int d1 = O.doff[g + 1];
  for (int q = O.doff[g]; q < d1; ++q) {
    const int4 h = O.dh[q];
    const int2 *zc = zl + h.z * stride;
#pragma unroll
    for (int r = 0; r < R; ++r) mac(r, h.x, h.y, zc[r * stride]);
  }
  if (!O.soff) return;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int s1 = O.soff[g * R + r + 1];
#pragma unroll 2
    for (int q = O.soff[g * R + r]; q < s1; ++q) {
      const int4 h = O.sh[q];
      mac(r, h.x, h.y, zl[h.z * stride]);
    }
  }
}

// A sum as a 62-bit integer, units of 2^(2 low - 1).
__device__ __forceinline__ long long finish(long long h, long long x, int low) {
  return (h << 1) + ((x + (1LL << (low - 2))) >> (low - 1));
}

template <int R>
__device__ __forceinline__ long long finish(const Acc<R> &A, int r, int low) {
  return finish(A.h[r], A.x[r], low);
}

// An ADO's coupling list in shared memory.
struct List {
  F64Entry e[2 * kF64MaxExp];
  int off[kF64MaxModes + 1];
};

// Dynamic shared memory that a launch may ask for, beside its kernel's own static arrays.
constexpr size_t kStageSmem = kMaxSmem - sizeof(List) - 256;   // whole items, panels
constexpr size_t kRotSmem = kMaxSmem - 512;
constexpr size_t kSmallSmem = kMaxSmem - 1024;

__device__ __forceinline__ void fill_list(const F64Ops &O, int n, List *L, int t, int nt) {
  const int *off = O.noff + n * O.n_modes;
  const int q0 = off[0], nq = off[O.n_modes] - q0;
  for (int i = t; i <= O.n_modes; i += nt) L->off[i] = off[i] - q0;
  for (int i = t; i < nq; i += nt) L->e[i] = O.nb[q0 + i];
}

// (alpha (lam_a - lam_b), alpha (lam_a + lam_b)) of every digit pair, mode after mode.
__device__ __forceinline__ void fill_tab(const F64Ops &O, double alpha, double2 *tab) {
  for (int i = threadIdx.x; i < O.tab; i += blockDim.x) {
    const double2 t = O.fg[i];
    tab[i] = make_double2(alpha * t.x, alpha * t.y);
  }
}

// Elementwise rest of element (a, b) (offset el) of the ADO at wn on top of acc:
//   acc - alpha gamma w + sum_s [ -i f_s A_s + g_s B_s ],  A_s = sum cA w_m, B_s = sum cB w_m,
// the neighbours' loads issued four at a time.
__device__ __forceinline__ double2 couple(const F64Ops &O, const double2 *tab, const List &L, const double2 *wb,
                                          const double2 *wn, int64_t dd, int a, int b, int el, double2 acc,
                                          double adec) {
  const double2 w = wn[el];
  acc.x = fma(-adec, w.x, acc.x);
  acc.y = fma(-adec, w.y, acc.y);
  for (int s = 0; s < O.n_modes; ++s) {
    const int q0 = L.off[s], q1 = L.off[s + 1];
    if (q0 == q1) continue;
    double2 A = make_double2(0.0, 0.0), B = A;
    bool both = false;
    for (int q = q0; q < q1; q += 4) {
      double2 x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (q + j < q1) x[j] = wb[(int64_t)L.e[q + j].idx * dd + el];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (q + j < q1) {
          const F64Entry &en = L.e[q + j];
          const bool first = q + j == q0;
          if (en.kind == 0) {
            A = first ? x[j] : make_double2(__dadd_rn(A.x, x[j].x), __dadd_rn(A.y, x[j].y));
          } else {
            const double c = en.cA;
            A = first ? make_double2(c * x[j].x, c * x[j].y) : make_double2(fma(c, x[j].x, A.x), fma(c, x[j].y, A.y));
            if (en.kind == 2) {
              const double e = en.cB;
              B = both ? make_double2(fma(e, x[j].x, B.x), fma(e, x[j].y, B.y)) : make_double2(e * x[j].x, e * x[j].y);
              both = true;
            }
          }
        }
    }
    const double2 fg = tab[O.tab_off[s] + O.dig[s * O.d + a] * O.dims[s] + O.dig[s * O.d + b]];
    acc.x = fma(fg.x, A.y, acc.x);
    acc.y = fma(-fg.x, A.x, acc.y);
    if (both) {
      acc.x = fma(fg.y, B.x, acc.x);
      acc.y = fma(fg.y, B.y, acc.y);
    }
  }
  return acc;
}

// y + alpha (L w)_{ab}: the elementwise rest (couple from zero, tab unscaled), the commutator
// from its integer sums c (units of f), then alpha.  Whole items, their panels and the
// small-hierarchy kernel compute an element with these operations in this order, on limbs
// scaled by the item's largest exponent, so its bits depend neither on the launch nor on
// what else is in the batch.
__device__ __forceinline__ double2 element(double2 rest, longlong2 c, const Unit &f, double2 y, double alpha) {
  return make_double2(fma(alpha, fma(f.f, sum_value(c.y, f), rest.x), y.x),
                      fma(alpha, fma(-f.f, sum_value(c.x, f), rest.y), y.y));
}

// ---------------------------------------------------------------------------
// Whole items per block: w's limbs (scaled per item) in shared memory with an odd row
// stride, so that a warp reads 32 columns of a row or 32 rows of a column without bank
// conflicts.  H' w with lanes along the columns, w H' (H' symmetric) with lanes along
// the rows, then the elementwise rest.
// ---------------------------------------------------------------------------
template <int R, bool kMulti>
__global__ void __launch_bounds__(256, 4) f64_item_kernel(const __grid_constant__ F64Args P) {
  extern __shared__ __align__(16) uint8_t smem[];
  const F64Set &S = pick<kMulti>(P);
  const F64Ops &O = S.O;
  const int d = O.d, ld = d | 1, m = S.per_block, dd = d * d, isz = d * ld;
  const int64_t i0 = ((int64_t)blockIdx.x - S.begin) * m;
  const int nm = (int)min((int64_t)m, S.items - i0);
  double2 *tab = reinterpret_cast<double2 *>(smem);
  int4 *zs = reinterpret_cast<int4 *>(tab + O.tab);
  double2 *ts = reinterpret_cast<double2 *>(zs + m * isz);
  List *lists = reinterpret_cast<List *>(ts + (S.smem_t ? m * isz : 0));
  int *iexp = reinterpret_cast<int *>(lists + m);
  for (int i = threadIdx.x; i < m; i += blockDim.x) iexp[i] = 1;
  fill_tab(O, 1.0, tab);
  __syncthreads();
  const double2 *w = S.w + i0 * dd;
  {
    int cur = -1, e = 0;
    for (int k = threadIdx.x; k < nm * dd; k += blockDim.x) {
      const int i = k / dd, el = k - i * dd, a = el / d;
      const double2 v = w[k];
      if (i != cur) {
        if (cur >= 0) atomicMax(iexp + cur, e);
        cur = i;
        e = 0;
      }
      e = max(e, exp_field(v));
      reinterpret_cast<double2 *>(zs)[i * isz + a * ld + el - a * d] = v;
    }
    if (cur >= 0) atomicMax(iexp + cur, e);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nm * dd; k += blockDim.x) {
    const int i = k / dd, el = k - i * dd, a = el / d;
    int4 *p = zs + i * isz + a * ld + el - a * d;
    const double2 v = *reinterpret_cast<double2 *>(p);
    const int2 re = to_limbs(v.x, iexp[i], O.bits, O.bits - 31), im = to_limbs(v.y, iexp[i], O.bits, O.bits - 31);
    *p = make_int4(re.x, re.y, im.x, im.y);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  for (int i = warp; i < nm; i += warps) fill_list(O, (int)((i0 + i) % O.n_ado), lists + i, lane, 32);
  const int cols = 2 * nm * d, chunks = (cols + 31) / 32, tasks = O.groups * chunks;
  // phase 0: t = H' w (lane = column); phase 1: t -= w H' (lane = row); still integers
  for (int ph = 0; ph < 2; ++ph) {
    for (int k = warp; k < tasks; k += warps) {
      const int ch = k / O.groups, g = k - ch * O.groups;
      const int q = min(ch * 32 + lane, cols - 1), col = q >> 1, comp = q & 1;
      const int i = col / d, l = col - i * d;
      Acc<R> A;
      group_product<R>(O, g, reinterpret_cast<const int2 *>(zs + i * isz + (ph == 0 ? l : l * ld)) + comp,
                       ph == 0 ? 2 * ld : 2, A);
      if (ch * 32 + lane < cols) {
        long long *t = reinterpret_cast<long long *>(S.smem_t ? ts + i * isz : S.tp + (i0 + i) * dd) + comp;
        const int tld = S.smem_t ? ld : d;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int x = g * R + r;
          if (x < d) {
            const long long v = finish(A, r, O.bits - 31);
            if (ph == 0)
              t[2 * (x * tld + l)] = v;
            else
              t[2 * (l * tld + x)] -= v;
          }
        }
      }
    }
    __syncthreads();
  }
  for (int k = threadIdx.x; k < nm * dd; k += blockDim.x) {
    const int i = k / dd, el = k - i * dd, a = el / d, b = el - a * d;
    const int64_t item = i0 + i;
    const int n = (int)(item % O.n_ado);
    const longlong2 c = *reinterpret_cast<const longlong2 *>(S.smem_t ? ts + i * isz + a * ld + b : S.tp + item * dd + el);
    const double2 zero = make_double2(0.0, 0.0);
    const double2 rest = couple(O, tab, lists[i], S.w + ado_offset(item - n, d), S.w + ado_offset(item, d), dd, a, b, el,
                                zero, O.decay[n]);
    S.out[item * dd + el] =
        element(rest, c, unit(iexp[i], O.hexp, O.hsign), S.y ? S.y[item * dd + el] : zero, P.alpha);
  }
}

// ---------------------------------------------------------------------------
// One panel per block: kPanel columns of w in the left kernel (tp = H' w), kPanel rows in
// the right one, which takes w H' off and adds the elementwise rest of those rows.  Half of
// the right kernel's blocks take the elementwise part first: it lives on the FP64 pipe and
// the products on the IMAD pipe, and blocks that start together would otherwise wait for
// the same pipe all the time.
//
// kItem: bases whose items fit a block (launches with few of them), with the arithmetic of
// f64_item_kernel: limbs scaled by the whole item's largest exponent, which every block
// finds for itself (d^2 loads that hit L2: 5 to 8 % of a launch of a few hundred items; one
// cluster per item that shares it: as fast for 10 items, 2 to 12 % slower from 80 on); the
// commutator's integers in tp; blocks that take the elementwise part first keep it in
// shared memory.
//
// Otherwise: limbs scaled per column (row), tp = -i alpha H' w in FP64, on which the right
// kernel adds in either order; ADO and panel decide, so that an element's additions have
// one order wherever its branch stands.  d = 125, 924 items: 830 us (IMAD pipe 74 % busy)
// and 1544 us (FP64 pipe 72 %, IMAD 52 %); one thread per element in the product basis took
// 17.4 ms.
// ---------------------------------------------------------------------------
template <int R, bool kRight, bool kMulti, bool kItem>
__global__ void __launch_bounds__(panel_threads(R), panel_blocks(R))
    f64_panel_kernel(const __grid_constant__ F64Args P) {
  extern __shared__ __align__(16) uint8_t smem[];
  const F64Set &S = pick<kMulti>(P);
  const F64Ops &O = S.O;
  const int d = O.d;
  const int64_t dd = (int64_t)d * d;
  const int64_t lb = (int64_t)blockIdx.x - S.begin;
  const int64_t item = lb / S.per_block;
  const int p0 = (int)(lb - item * S.per_block) * kPanel, np = min(kPanel, d - p0);
  constexpr int ld = kRight ? kPanel + 1 : kPanel;
  double2 *tab = reinterpret_cast<double2 *>(smem);
  int4 *zs = reinterpret_cast<int4 *>(tab + O.tab);      // [d][ld]
  double2 *rest = reinterpret_cast<double2 *>(zs + d * ld);   // kItem, early blocks: [kPanel][d | 1]
  __shared__ int lexp[kPanel], turn;
  __shared__ List list;
  const double alpha = P.alpha, ah = alpha * O.hsign;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  if (threadIdx.x < kPanel) lexp[threadIdx.x] = 1;
  const int n = (int)(item % O.n_ado);
  if (kRight) {
    if (threadIdx.x == 0) turn = (int)(((unsigned)n * (unsigned)d + (unsigned)p0) * 2654435761u >> 31);
    fill_tab(O, kItem ? 1.0 : alpha, tab);
    fill_list(O, n, &list, threadIdx.x, blockDim.x);
  }
  __syncthreads();
  const double2 *w = S.w + item * dd;
  const double2 zero = make_double2(0.0, 0.0);
  const int col_t = threadIdx.x & (kPanel - 1), row_t = threadIdx.x / kPanel, rows_t = blockDim.x / kPanel;
  if (!kRight) {
    int e = 0;
    for (int c = row_t; c < d; c += rows_t) {
      const double2 v = col_t < np ? w[(int64_t)c * d + p0 + col_t] : zero;
      e = max(e, exp_field(v));
      reinterpret_cast<double2 *>(zs)[c * ld + col_t] = v;
    }
    if (!kItem) atomicMax(lexp + col_t, e);
  } else {
    for (int a = warp; a < kPanel; a += warps) {
      int e = 0;
      for (int c = lane; c < d; c += 32) {
        const double2 v = a < np ? w[(int64_t)(p0 + a) * d + c] : zero;
        e = max(e, exp_field(v));
        reinterpret_cast<double2 *>(zs)[c * ld + a] = v;
      }
      if (!kItem) {
        e = __reduce_max_sync(0xffffffffu, e);
        if (lane == 0) lexp[a] = max(e, 1);
      }
    }
  }
  if (kItem) {
    int top = 0;
#pragma unroll 4
    for (int k = threadIdx.x; k < (int)dd; k += blockDim.x) top = max(top, exp_field(w[k]));
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) atomicMax(lexp, top);
  }
  __syncthreads();
  const int emax = lexp[kItem ? 0 : col_t];
  for (int c = row_t; c < d; c += rows_t) {
    int4 *p = zs + c * ld + col_t;
    const double2 v = *reinterpret_cast<double2 *>(p);
    const int2 re = to_limbs(v.x, emax, O.bits, O.bits - 31), im = to_limbs(v.y, emax, O.bits, O.bits - 31);
    *p = make_int4(re.x, re.y, im.x, im.y);
  }
  const bool early = kRight && turn;
  // the elementwise rest of the panel's rows: with the commutator in tp into out, or (kItem,
  // early) alone into shared memory
  auto elementwise = [&]() {
    const double2 *wb = S.w + (item - n) * dd, *from = S.tp + item * dd;
    const double2 *y = S.y ? S.y + item * dd : nullptr;
    const double dec = kItem ? O.decay[n] : alpha * O.decay[n];
    for (int k = threadIdx.x; k < np * d; k += blockDim.x) {
      const int ar = k / d, el = p0 * d + k;
      double2 acc = zero;
      if (!kItem) {
        acc = from[el];
        if (y) {
          const double2 yv = y[el];
          acc = make_double2(acc.x + yv.x, acc.y + yv.y);
        }
      }
      acc = couple(O, tab, list, wb, w, dd, p0 + ar, k - ar * d, el, acc, dec);
      if (kItem && early)
        rest[ar * (d | 1) + k - ar * d] = acc;
      else if (kItem)
        S.out[item * dd + el] = element(acc, *reinterpret_cast<const longlong2 *>(from + el),
                                        unit(emax, O.hexp, O.hsign), y ? y[el] : zero, alpha);
      else
        S.out[item * dd + el] = acc;
    }
  };
  if (early) elementwise();
  __syncthreads();
  // one task: a row group and the 16 complex columns, lane = (column, component)
  const int comp = lane & 1, col = lane >> 1;
  for (int g = warp; g < O.groups; g += warps) {
    Acc<R> A;
    group_product<R>(O, g, reinterpret_cast<const int2 *>(zs + col) + comp, 2 * ld, A);
    const int step = kRight ? 2 : 2 * d, live = col < np ? min(R, d - g * R) : 0;
    const int64_t at = 2 * (kRight ? (int64_t)(p0 + col) * d + g * R : (int64_t)g * R * d + p0 + col);
    if (kItem) {
      long long *o = reinterpret_cast<long long *>(S.tp + item * dd) + at + comp, v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = kRight && r < live ? o[r * step] : 0;
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = kRight ? v[r] - finish(A, r, O.bits - 31) : finish(A, r, O.bits - 31);
      if (early) {
        // element(): the real sum goes to the imaginary part, and out may be tp
        __syncwarp();
        const Unit f = unit(emax, O.hexp, comp ? O.hsign : -O.hsign);
        const double *e = reinterpret_cast<const double *>(rest + col * (d | 1) + g * R) + (comp ^ 1);
        const double *y = S.y ? reinterpret_cast<const double *>(S.y + item * dd) + at + (comp ^ 1) : nullptr;
        double *out = reinterpret_cast<double *>(S.out + item * dd) + at + (comp ^ 1), yv[R];
#pragma unroll
        for (int r = 0; r < R; ++r) yv[r] = y && r < live ? y[2 * r] : 0.0;
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (r < live) out[2 * r] = fma(alpha, fma(f.f, sum_value(v[r], f), e[2 * r]), yv[r]);
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (r < live) o[r * step] = v[r];
      }
    } else if (col < np) {
      // -i alpha (x + i y) = alpha (y - i x): the real sum goes to the imaginary part
      const Unit f = unit(lexp[col], O.hexp, comp == (kRight ? 1 : 0) ? -ah : ah);
      double *t = reinterpret_cast<double *>((early ? S.out : S.tp) + item * dd) + (comp ^ 1);
      double v[R], old[R];
      double *o = t + at;
#pragma unroll
      for (int r = 0; r < R; ++r) old[r] = kRight && r < live ? o[r * step] : 0.0;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        v[r] = sum_value(finish(A, r, O.bits - 31), f);
        v[r] = kRight ? fma(f.f, v[r], old[r]) : f.f * v[r];
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (r < live) o[r * step] = v[r];
    }
  }
  if (kRight && !early) {
    __syncthreads();
    elementwise();
  }
}

// ---------------------------------------------------------------------------
// Many RK4 steps of a small hierarchy in one launch.  A stage of such a hierarchy takes
// 1-3 us of the FP64 pipe of the SMs it spreads over, but 12-19 us as a launch of its
// own, which starts with a chain of dependent table loads; here the tables stay in
// shared memory and the blocks meet at a barrier after each stage.  Work is split into
// units (item, row range); kSync 0: one block per branch, 1: one cluster per branch, 2:
// the whole (cooperative) grid shares all branches' units.  The states are the caller's
// buffers, exchanged through L2.
// ---------------------------------------------------------------------------
struct F64SmallSet {
  F64Ops O;
  double2 *y, *wa, *wb;
  int branches;
  int parts;          // row ranges per item
  int units;          // units per block
  int bpb;            // blocks per branch (kSync 0, 1), or blocks of the grid (2)
  int begin;          // first block of the set
};

struct F64SmallArgs {
  F64SmallSet one;
  const F64SmallSet *many;   // kMulti: the sets' blocks follow one another (kSync 0, 1)
  int n;
  double alpha[4];           // dt / 4, dt / 3, dt / 2, dt
  int64_t steps;
};

constexpr int kSmallPre = 8;   // neighbours whose loads are issued ahead

// What a block of f64_small_kernel keeps in shared memory: everything the steps need
// besides the states, with the index arithmetic done once.
struct SmallItem {
  int64_t base, branch;   // element offsets of the item and of its branch
  double decay;
  int n_nb, off[kF64MaxModes + 1];
  F64Entry e[2 * kF64MaxExp];   // idx: element offset within the branch
};

// One thread per component of an element: the commutator's sum takes 6 IMAD.WIDE per
// column, the rest about ten FP64 operations, which have 67 cycles of latency each and
// so need the parallelism more than the shared loads.
template <int kSync, bool kMulti>
__global__ void __launch_bounds__(512) f64_small_kernel(const __grid_constant__ F64SmallArgs G) {
  extern __shared__ __align__(16) uint8_t smem[];
  int ks = 0;
  while (kMulti && ks + 1 < G.n && (int)blockIdx.x >= G.many[ks + 1].begin) ++ks;
  const F64SmallSet &P = kMulti ? G.many[ks] : G.one;
  const F64Ops &O = P.O;
  const int d = O.d, ld = d | 1, dd = d * d, isz = d * ld, low = O.bits - 31, nm = O.n_modes;
  // this block's units: consecutive in (item, part) order of its branch (kSync 2: of all)
  const int blk = (int)blockIdx.x - P.begin;
  const int n_units = (kSync == 2 ? P.branches : 1) * O.n_ado * P.parts;
  const int u0 = min(n_units, (blk % P.bpb) * P.units);
  const int nu = min(P.units, n_units - u0);
  const int64_t first = kSync == 2 ? 0 : (int64_t)(blk / P.bpb) * O.n_ado;   // first item of the branch
  const int64_t i0 = first + u0 / P.parts;
  const int ni = nu > 0 ? (u0 + nu - 1) / P.parts - u0 / P.parts + 1 : 0;      // items touched
  const int max_items = (P.units + P.parts - 1) / P.parts + (P.parts > 1 ? 1 : 0);
  double2 *tab = reinterpret_cast<double2 *>(smem);
  int4 *zs = reinterpret_cast<int4 *>(tab + O.tab);
  SmallItem *items = reinterpret_cast<SmallItem *>(zs + max_items * isz);
  int2 *hs = reinterpret_cast<int2 *>(items + max_items);       // H' limbs, dense
  int *iexp = reinterpret_cast<int *>(hs + dd);                 // [2][max_items], by stage parity
  int *dig = iexp + 2 * max_items;                              // [n_modes][2][d] table offsets of row and column
  int *elem = dig + 2 * nm * d;                                 // this block's elements: item, row, column
  int *place = elem + P.units * ((d + P.parts - 1) / P.parts) * d;   // its items' elements: item, offset in zs
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int rows = (d + P.parts - 1) / P.parts;   // rows per part
  for (int i = warp; i < ni; i += warps) {
    SmallItem &I = items[i];
    const int64_t item = i0 + i;
    const int n = (int)(item % O.n_ado);
    const int *off = O.noff + n * nm;
    const int q0 = off[0], nq = off[nm] - q0;
    if (lane == 0) {
      I.base = ado_offset(item, d);
      I.branch = ado_offset(item - n, d);
      I.decay = O.decay[n];
      I.n_nb = nq;
    }
    for (int m = lane; m <= nm; m += 32) I.off[m] = off[m] - q0;
    for (int q = lane; q < nq; q += 32) {
      I.e[q] = O.nb[q0 + q];
      I.e[q].idx *= dd;
    }
  }
  for (int i = threadIdx.x; i < dd; i += blockDim.x) hs[i] = O.hd[i];
  for (int i = threadIdx.x; i < O.tab; i += blockDim.x) tab[i] = O.fg[i];
  for (int i = threadIdx.x; i < 2 * ni; i += blockDim.x) iexp[i] = 1;
  for (int i = threadIdx.x; i < nm * d; i += blockDim.x) {
    const int s = i / d, a = i - s * d;
    dig[2 * s * d + a] = O.tab_off[s] + O.dig[i] * O.dims[s];
    dig[(2 * s + 1) * d + a] = O.dig[i];
  }
  for (int k = threadIdx.x; k < nu * rows * d; k += blockDim.x) {
    const int u = k / (rows * d), r = k - u * rows * d, ug = u0 + u;
    const int a = (ug % P.parts) * rows + r / d, b = r % d;
    elem[k] = (ug / P.parts - u0 / P.parts) << 12 | a << 6 | b;   // a may pass d in the last part: skipped
  }
  for (int k = threadIdx.x; k < ni * dd; k += blockDim.x) {
    const int i = k / dd, el = k - i * dd;
    place[k] = i << 20 | (i * isz + el / d * ld + el % d);
  }
  __syncthreads();
  const int work = 2 * nu * rows * d, nz = ni * dd;
  const int64_t z0 = ado_offset(i0, d);
  int parity = 0;
  for (int64_t s = 0; s < G.steps; ++s)
    for (int q = 0; q < 4; ++q, parity ^= 1) {
      const double2 *w = q == 0 ? P.y : q == 2 ? P.wb : P.wa;
      double2 *out = q == 3 ? P.y : q == 1 ? P.wb : P.wa;
      const double alpha = G.alpha[q];
      int *ie = iexp + parity * ni;
      // component k of this block: all its loads (y, w, the first neighbours) at once
      int el = 0, a = 0, b = 0;
      const SmallItem *I = items;
      double yv = 0.0, wv = 0.0;
      double2 x[kSmallPre];
      const int comp = threadIdx.x & 1;
      bool live = false;
      auto fetch = [&](int k) {
        live = false;
        if (k >= work) return;
        const int e = elem[k >> 1];
        a = (e >> 6) & 63;
        b = e & 63;
        if (a >= d) return;
        live = true;
        I = items + (e >> 12);
        el = a * d + b;
        yv = __ldcg(reinterpret_cast<const double *>(P.y + I->base + el) + comp);
        wv = __ldcg(reinterpret_cast<const double *>(w + I->base + el) + comp);
        const double2 *wb = w + I->branch + el;
        const int nq = I->n_nb;
#pragma unroll
        for (int j = 0; j < kSmallPre; ++j)
          if (j < nq) x[j] = __ldcg(wb + I->e[j].idx);
      };
      fetch(threadIdx.x);
      // limbs of the items' w
      for (int k = threadIdx.x; k < ((nz + 31) & ~31); k += blockDim.x) {
        int it = ni - 1, e = 0;
        if (k < nz) {
          const int p = place[k];
          const double2 v = __ldcg(w + z0 + k);
          it = p >> 20;
          e = exp_field(v);
          reinterpret_cast<double2 *>(zs)[p & 0xfffff] = v;
        }
        const int il = __shfl_sync(0xffffffffu, it, 0), ih = __shfl_sync(0xffffffffu, it, 31);
        if (il == ih) {
          e = __reduce_max_sync(0xffffffffu, e);
          if (lane == 0) atomicMax(ie + it, e);
        } else {
          atomicMax(ie + it, e);
        }
      }
      __syncthreads();
      for (int k = threadIdx.x; k < nz; k += blockDim.x) {
        const int p = place[k], e = ie[p >> 20];
        int4 *z = zs + (p & 0xfffff);
        const double2 v = *reinterpret_cast<double2 *>(z);
        const int2 re = to_limbs(v.x, e, O.bits, low), im = to_limbs(v.y, e, O.bits, low);
        *z = make_int4(re.x, re.y, im.x, im.y);
      }
      for (int k = threadIdx.x; k < ni; k += blockDim.x) iexp[(parity ^ 1) * ni + k] = 1;
      __syncthreads();
      for (int k = threadIdx.x; k < work; k += blockDim.x) {
        if (live) {
          // -i C: the real component takes the commutator's imaginary part, and back
          const int it = (int)(I - items);
          const int2 *zb = reinterpret_cast<const int2 *>(zs + it * isz + b) + (comp ^ 1);
          const int2 *za = reinterpret_cast<const int2 *>(zs + it * isz + a * ld) + (comp ^ 1);
          const int2 *ha = hs + a * d, *hb = hs + b * d;   // H' is symmetric
          long long h1 = 0, x1 = 0, h2 = 0, x2 = 0;
#pragma unroll 4
          for (int c = 0; c < d; ++c) {
            const int2 h = ha[c], g = hb[c], z = *zb, t = za[2 * c];
            zb += 2 * ld;
            h1 += (long long)h.x * z.x;
            x1 += (long long)h.x * z.y;
            x1 += (long long)h.y * z.x;
            h2 += (long long)g.x * t.x;
            x2 += (long long)g.x * t.y;
            x2 += (long long)g.y * t.x;
          }
          const Unit f = unit(ie[it], O.hexp, comp ? -O.hsign : O.hsign);
          const double cm = sum_value(finish(h1, x1, low) - finish(h2, x2, low), f);
          // acc = -gamma w + sum_s [ +- f_s A_s(other component) + g_s B_s ] +- f C, the
          // operations of stage_element in their order
          double acc = fma(-I->decay, wv, 0.0), A = 0.0, B = 0.0;
          int m = 0;
          bool any = false, both = false;
          auto close = [&]() {
            if (!any) return;
            const double2 fg = tab[dig[2 * m * d + a] + dig[(2 * m + 1) * d + b]];
            acc = fma(comp ? -fg.x : fg.x, A, acc);
            if (both) acc = fma(fg.y, B, acc);
            any = both = false;
          };
          auto entry = [&](int j, const double2 &v) {
            while (j >= I->off[m + 1]) {
              close();
              ++m;
            }
            const F64Entry &en = I->e[j];
            const double o = comp ? v.x : v.y;
            if (en.kind == 0) {
              A = any ? __dadd_rn(A, o) : o;
            } else {
              A = any ? fma(en.cA, o, A) : en.cA * o;
              if (en.kind == 2) {
                const double t = comp ? v.y : v.x;
                B = both ? fma(en.cB, t, B) : en.cB * t;
                both = true;
              }
            }
            any = true;
          };
          const int nq = I->n_nb;
#pragma unroll
          for (int j = 0; j < kSmallPre; ++j)
            if (j < nq) entry(j, x[j]);
          for (int j = kSmallPre; j < nq; ++j) entry(j, __ldcg(w + I->branch + I->e[j].idx + el));
          close();
          acc = fma(f.f, cm, acc);
          __stcg(reinterpret_cast<double *>(out + I->base + el) + comp, fma(alpha, acc, yv));
        }
        fetch(k + blockDim.x);
      }
      if (kSync == 0)
        __syncthreads();
      else if (kSync == 1)
        cg::this_cluster().sync();
      else
        cg::this_grid().sync();
    }
}

// ---------------------------------------------------------------------------
// Basis change along one index of every ADO, mode by mode, a panel of 32 columns
// (left: the row index) or rows (right) in shared memory; each thread transforms one
// fibre of n_s values in registers: 6 n_s products per element and side instead of the
// 2 d of a dense product.  In fixed point, 59 bits below the column's 2-norm (which the
// orthogonal factors keep, so nothing overflows) with 59-bit coefficients in 30-bit
// limbs: a state goes in and out of this basis in every call, and the roundings of the
// same products in FP64 (3.6e-16 of the norm for a round trip at four levels) would
// exceed a step's own; here the results' conversion to FP64 is what remains.
// ---------------------------------------------------------------------------
constexpr int kRotMaxN = 8;

__device__ __forceinline__ long long to_fixed59(double x, int emax) {
  const int2 l = to_limbs(x, emax, 60, 30);
  return ((long long)l.x << 30) + l.y;
}

// t 2^(e - 1081), in two factors where one would leave the exponent range; NaN if not finite.
__device__ __forceinline__ double2 from_fixed59(const longlong2 &t, int e, bool finite) {
  const double f = __longlong_as_double(finite ? (long long)(e > 58 ? e - 58 : e + 964) << 52 : 0x7ff8000000000000LL);
  double re = __ll2double_rn(t.x) * f, im = __ll2double_rn(t.y) * f;
  if (e <= 58) {
    re *= __longlong_as_double(1LL << 52);
    im *= __longlong_as_double(1LL << 52);
  }
  return make_double2(re, im);
}

// One fibre of N values, str apart.
template <int N>
__device__ __forceinline__ void rotate_fibre(longlong2 *p, const int2 *__restrict__ u, int str) {
  {
    int4 in[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const longlong2 t = p[k * str];
      const int re = ((int)((unsigned)t.x << 2)) >> 2, im = ((int)((unsigned)t.y << 2)) >> 2;
      in[k] = make_int4((int)((t.x - re) >> 30), re, (int)((t.y - im) >> 30), im);
    }
    for (int i = 0; i < N; ++i) {
      long long hr = 0, xr = 0, hi = 0, xi = 0;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const int2 c = u[k * N + i];
        hr += (long long)c.x * in[k].x;
        xr += (long long)c.x * in[k].y;
        xr += (long long)c.y * in[k].x;
        hi += (long long)c.x * in[k].z;
        xi += (long long)c.x * in[k].w;
        xi += (long long)c.y * in[k].z;
      }
      p[i * str] = make_longlong2((hr << 1) + ((xr + (1LL << 28)) >> 29), (hi << 1) + ((xi + (1LL << 28)) >> 29));
    }
  }
}

// Fibres f = warp, warp + warps, ... of one lane's column.
template <int N>
__device__ __forceinline__ void rotate_fibres(longlong2 *v, const int2 *__restrict__ u, int str, int d, int warp,
                                              int warps) {
  for (int f = warp; f < d / N; f += warps)
    rotate_fibre<N>(v + ((f / str) * str * N + f % str) * kRotPad, u, str * kRotPad);
}

template <bool kRight>
__global__ void __launch_bounds__(256) rotate_kernel(const double2 *x, double2 *out, const int2 *__restrict__ u, const __grid_constant__ RotOps r,
                                                     int panels) {
  extern __shared__ __align__(16) uint8_t smem[];
  longlong2 *v = reinterpret_cast<longlong2 *>(smem);   // [d][33], second index along the panel
  __shared__ int lexp[32];
  __shared__ unsigned lsum[32];
  const int d = r.d;
  const int64_t item = blockIdx.x / panels;
  const int p0 = (int)(blockIdx.x - item * panels) * 32, np = min(32, d - p0);
  const double2 *xi = x + item * d * d;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  if (threadIdx.x < 32) {
    lexp[lane] = 1;
    lsum[lane] = 0;
  }
  if (!kRight) {
    if (lane < np)
      for (int c = warp; c < d; c += warps)
        reinterpret_cast<double2 *>(v)[c * kRotPad + lane] = xi[(int64_t)c * d + p0 + lane];
  } else {
    for (int k = threadIdx.x; k < np * d; k += blockDim.x) {
      const int a = k / d;
      reinterpret_cast<double2 *>(v)[(k - a * d) * kRotPad + a] = xi[(int64_t)p0 * d + k];
    }
  }
  __syncthreads();
  // exponent of the column's largest component, then of (an upper bound of) its 2-norm,
  // from an integer sum of squares (the same whatever the order)
  if (lane < np) {
    int e = 0;
    for (int c = warp; c < d; c += warps) e = max(e, exp_field(reinterpret_cast<double2 *>(v)[c * kRotPad + lane]));
    atomicMax(lexp + lane, e);
  }
  __syncthreads();
  const int e1 = lexp[lane];
  if (lane < np) {
    unsigned q = 0;
    for (int c = warp; c < d; c += warps) {
      const double2 t = reinterpret_cast<double2 *>(v)[c * kRotPad + lane];
      const int2 re = to_limbs(t.x, e1, 60, 30), im = to_limbs(t.y, e1, 60, 30);
      // |component| / 2^29 < 1 up to the low limb's share
      const float a = (float)(abs(re.x) + 1) * (1.f / (1 << 29)), b = (float)(abs(im.x) + 1) * (1.f / (1 << 29));
      q += (unsigned)((a * a + b * b) * 262144.f) + 2u;
    }
    atomicAdd(lsum + lane, q);
  }
  __syncthreads();
  // norm <= 2^(e1 - 1022 + k), 4^k >= lsum / 2^18
  const int lg = 32 - __clz(lsum[lane]);
  const int en = e1 + (lg > 18 ? (lg - 17) / 2 : 0);
  if (lane < np)
    for (int c = warp; c < d; c += warps) {
      longlong2 *p = v + c * kRotPad + lane;
      const double2 t = *reinterpret_cast<double2 *>(p);
      *p = make_longlong2(to_fixed59(t.x, en), to_fixed59(t.y, en));
    }
  for (int s = 0; s < r.n_modes; ++s) {
    __syncthreads();
    const int n = r.dims[s], str = r.stride[s];
    const int2 *us = u + r.off[s];
    if (lane < np) {
      longlong2 *vl = v + lane;
      switch (n) {   // fibre lengths unrolled: the fibre stays in registers
        case 2: rotate_fibres<2>(vl, us, str, d, warp, warps); break;
        case 3: rotate_fibres<3>(vl, us, str, d, warp, warps); break;
        case 4: rotate_fibres<4>(vl, us, str, d, warp, warps); break;
        case 5: rotate_fibres<5>(vl, us, str, d, warp, warps); break;
        case 6: rotate_fibres<6>(vl, us, str, d, warp, warps); break;
        case 7: rotate_fibres<7>(vl, us, str, d, warp, warps); break;
        case 8: rotate_fibres<8>(vl, us, str, d, warp, warps); break;
        default: break;   // one level: the identity
      }
    }
  }
  __syncthreads();
  double2 *oi = out + item * d * d;
  auto store = [&](int64_t at, const longlong2 &t, int e, bool finite) { oi[at] = from_fixed59(t, e, finite); };
  if (!kRight) {
    if (lane < np)
      for (int c = warp; c < d; c += warps) store((int64_t)c * d + p0 + lane, v[c * kRotPad + lane], en, e1 < 0x7ff);
  } else {
    if (threadIdx.x < 32) lsum[lane] = (unsigned)en;
    __syncthreads();
    for (int k = threadIdx.x; k < np * d; k += blockDim.x) {
      const int a = k / d;
      store((int64_t)p0 * d + k, v[(k - a * d) * kRotPad + a], (int)lsum[a], lexp[a] < 0x7ff);
    }
  }
}

// Both sides at once for small bases: one item per block in shared memory, one scale
// for it (its Frobenius norm).  Two launches of the panel kernels are ~17 us however
// small the state is.
__global__ void __launch_bounds__(256) rotate_item_kernel(const double2 *x, double2 *out, const int2 *__restrict__ u,
                                                          const __grid_constant__ RotOps r) {
  extern __shared__ __align__(16) uint8_t smem[];
  longlong2 *v = reinterpret_cast<longlong2 *>(smem);   // [d][d | 1]
  __shared__ int s_exp;
  __shared__ unsigned s_sum;
  const int d = r.d, ld = d | 1, dd = d * d;
  const double2 *xi = x + (int64_t)blockIdx.x * dd;
  if (threadIdx.x == 0) {
    s_exp = 1;
    s_sum = 0;
  }
  __syncthreads();
  int e = 0;
  for (int k = threadIdx.x; k < dd; k += blockDim.x) {
    const double2 z = xi[k];
    e = max(e, exp_field(z));
    reinterpret_cast<double2 *>(v)[(k / d) * ld + k % d] = z;
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&s_exp, e);
  __syncthreads();
  const int e1 = s_exp;
  unsigned q = 0;
  for (int k = threadIdx.x; k < dd; k += blockDim.x) {
    const double2 t = reinterpret_cast<double2 *>(v)[(k / d) * ld + k % d];
    const int2 re = to_limbs(t.x, e1, 60, 30), im = to_limbs(t.y, e1, 60, 30);
    const float a = (float)(abs(re.x) + 1) * (1.f / (1 << 29)), b = (float)(abs(im.x) + 1) * (1.f / (1 << 29));
    q += (unsigned)((a * a + b * b) * 262144.f) + 2u;   // up to 2304 elements: below 2^31
  }
  atomicAdd(&s_sum, q);
  __syncthreads();
  const int lg = 32 - __clz(s_sum);
  const int en = e1 + (lg > 18 ? (lg - 17) / 2 : 0);
  for (int k = threadIdx.x; k < dd; k += blockDim.x) {
    longlong2 *p = v + (k / d) * ld + k % d;
    const double2 t = *reinterpret_cast<double2 *>(p);
    *p = make_longlong2(to_fixed59(t.x, en), to_fixed59(t.y, en));
  }
  for (int side = 0; side < 2; ++side)
    for (int s = 0; s < r.n_modes; ++s) {
      __syncthreads();
      const int n = r.dims[s], str = r.stride[s];
      const int2 *us = u + r.off[s];
      for (int k = threadIdx.x; k < dd / n; k += blockDim.x) {
        const int f = side == 0 ? k / d : k % (d / n), o = side == 0 ? k % d : k / (d / n);
        const int base = (f / str) * str * n + f % str;
        longlong2 *p = side == 0 ? v + base * ld + o : v + o * ld + base;
        const int ps = side == 0 ? str * ld : str;
        switch (n) {
          case 2: rotate_fibre<2>(p, us, ps); break;
          case 3: rotate_fibre<3>(p, us, ps); break;
          case 4: rotate_fibre<4>(p, us, ps); break;
          case 5: rotate_fibre<5>(p, us, ps); break;
          case 6: rotate_fibre<6>(p, us, ps); break;
          case 7: rotate_fibre<7>(p, us, ps); break;
          case 8: rotate_fibre<8>(p, us, ps); break;
          default: break;
        }
      }
    }
  __syncthreads();
  for (int k = threadIdx.x; k < dd; k += blockDim.x)
    out[(int64_t)blockIdx.x * dd + k] = from_fixed59(v[(k / d) * ld + k % d], en, e1 < 0x7ff);
}

template <typename T>
const T *up(const std::vector<T> &v, std::vector<void *> &allocs) {
  void *p = nullptr;
  const size_t bytes = std::max<size_t>(16, v.size() * sizeof(T));
  if (device_malloc(&p, bytes) != cudaSuccess) {
    (void)cudaGetLastError();
    throw DeviceOom();
  }
  allocs.push_back(p);
  if (!v.empty()) CUDA_TRY(cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
  return (const T *)p;
}

int digits_differ(const Model &M, int a, int c) {
  int k = 0;
  for (int s = 0; s < M.n_modes; ++s) k += (a / M.stride[s]) % M.dims[s] != (c / M.stride[s]) % M.dims[s];
  return k;
}

// Structural non-zeros in a row of H'.
int row_products(const Model &M) {
  int nz = 0;
  for (int c = 0; c < M.d; ++c) nz += digits_differ(M, 0, c) <= 2;
  return nz;
}

// Unevaluated sum of two doubles (about 32 digits), enough operations for the basis
// change of H.
struct DD {
  double h = 0.0, l = 0.0;
  void add_product(DD a, DD b) {
    const double p = a.h * b.h;
    const double e = std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h);
    const double s = h + p, v = s - h;
    const double r = ((h - (s - v)) + (p - v)) + l + e;
    h = s + r;
    l = r - (h - s);
  }
};

// X' = U^T X U, mode by mode, to about 32 digits.
std::vector<DD> coupling_matrix(const Model &M, const std::vector<double> &X) {
  const int d = M.d;
  std::vector<DD> A((size_t)d * d), v;
  for (size_t i = 0; i < A.size(); ++i) A[i].h = X[i];
  for (int side = 0; side < 2; ++side)
    for (int s = 0; s < M.n_modes; ++s) {
      const int n = M.dims[s], str = M.stride[s];
      v.resize(n);
      for (int f = 0; f < d / n; ++f) {
        const int base = (f / str) * str * n + f % str;
        for (int o = 0; o < d; ++o) {
          auto at = [&](int k) -> DD & {
            return side == 0 ? A[(size_t)(base + k * str) * d + o] : A[(size_t)o * d + base + k * str];
          };
          for (int k = 0; k < n; ++k) v[k] = at(k);
          for (int i = 0; i < n; ++i) {
            DD acc;
            for (int k = 0; k < n; ++k)
              acc.add_product(DD{M.cb_U[s][(size_t)k * n + i], M.cb_U_lo[s][(size_t)k * n + i]}, v[k]);
            at(i) = acc;
          }
        }
      }
    }
  return A;
}

int table_size(const Model &M) {
  int t = 0;
  for (int s = 0; s < M.n_modes; ++s) t += M.dims[s] * M.dims[s];
  return t;
}

size_t panel_smem(int d, int tab) { return (size_t)tab * 16 + (size_t)d * (kPanel + 1) * 16; }

size_t item_panel_smem(int d, int tab) { return panel_smem(d, tab) + (size_t)kPanel * (d | 1) * 16; }

size_t fused_smem(int d, int tab, int m, bool t) {
  return (size_t)tab * 16 + (size_t)m * d * (d | 1) * 16 * (t ? 2 : 1) + (size_t)m * (sizeof(List) + 4) + 64;
}

int sm_count() {
  int dev = 0, sms = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  return sms;
}

int row_group(const Model &M) {
  const int n = M.dims.back();
  return n % 5 == 0 ? 5 : n % 3 == 0 ? 6 : 4;
}

// Panels instead of whole items?  An item keeps one SM busy for 40 us at d = 36 and 160 us at
// d = 64, so a launch with few items spreads each over panels; from d = 69 on an SM holds two
// whole items at most, and panels, which an SM holds more of, are faster for any number.  Us
// per stage, items / panels (15 exponents' neighbours), by number of items: d = 36, 160
// items: 61 / 50, 240: 63 / 64, 480: 96 / 104; d = 45, 480: 139 / 131, 960: 224 / 221, 1280:
// 281 / 286; d = 48, 640: 189 / 187, 960: 248 / 259; d = 60, 1920: 822 / 818, 2560: 1058 /
// 1067; d = 64, 80: 172 / 69, 480: 355 / 257, 1920: 960 / 937, 2560: 1231 / 1233; d = 72,
// 3840: 3749 / 2523; d = 80, 80: 297 / 102, 3840: 3996 / 3338.
enum Variant { kItems = 0, kItemPanels = 1, kPanels = 2 };

Variant variant_of(int d, int tab, int64_t items) {
  const size_t one = fused_smem(d, tab, 1, false);
  if (one > kFusedSmem) return kPanels;
  if (d <= 32) return kItems;
  if (3 * (one + 1024) > kMaxSmem + 1024) return kItemPanels;
  // items per SM: 1.5 at d = 36, 4.6 at d = 48, 16.5 at d = 64
  const int64_t x = d - 30, per_sm_280 = std::max<int64_t>(70 * std::min<int64_t>(x, 15), 4 * x * x);
  return items * 280 < sm_count() * per_sm_280 ? kItemPanels : kItems;
}

// Threads of a panel block: small blocks are out of step with one another, so that the
// products of some (IMAD pipe) run beside the elementwise part of others (FP64 pipe), and
// the row groups divide evenly (25 at five levels, 16 at four); big ones where a launch
// has few blocks or a basis that leaves room for three.  d = 125, 924 items: 160 threads
// 827 + 1540 us, 320 854 + 1669 us; d = 64, both launches, 896 blocks: 256 threads 140
// us, 384 159 us; 112 blocks: 57 and 53 us; d = 216, 1920 blocks: 384 threads 460 + 596 us,
// 192 639 + 798 us.
int panel_shape(int R, int64_t blocks) {
  const int sms = sm_count();
  if (R == 5) return blocks >= 4 * sms ? 160 : 320;
  return R == 4 && blocks >= 2 * sms ? 256 : 384;
}

// Items per block of the whole-item kernel: enough columns for two to four warps of
// lanes, as long as the launch still has a few blocks per SM.
int items_per_block(int d, int tab, int64_t items) {
  int m = std::max(1, 128 / d);
  m = (int)std::min<int64_t>(m, std::max<int64_t>(1, items / (152 * 4)));
  while (m > 1 && fused_smem(d, tab, m, true) > 56 * 1024) --m;
  return m;
}

F64Set make_set(const F64Buf &b, int64_t begin, Variant *variant, size_t *smem, int64_t *blocks) {
  const F64Ops &O = *b.ops;
  F64Set s{};
  s.O = O;
  s.w = b.w;
  s.y = b.y;
  s.out = b.out;
  s.tp = b.tp;
  s.begin = begin;
  s.items = (int64_t)b.branches * O.n_ado;
  *variant = variant_of(O.d, O.tab, s.items);
  if (*variant == kItems) {
    s.per_block = items_per_block(O.d, O.tab, s.items);
    s.smem_t = fused_smem(O.d, O.tab, s.per_block, true) <= 56 * 1024;
    *smem = fused_smem(O.d, O.tab, s.per_block, s.smem_t);
    *blocks = (s.items + s.per_block - 1) / s.per_block;
  } else {
    s.per_block = (O.d + kPanel - 1) / kPanel;
    *smem = *variant == kItemPanels ? item_panel_smem(O.d, O.tab) : panel_smem(O.d, O.tab);
    *blocks = s.items * s.per_block;
  }
  return s;
}

// The limit belongs to the kernel in its context, for every thread that launches it: always
// the same value, never this launch's size.
template <typename K>
void allow_smem(K kernel, size_t smem, size_t most) {
  if (smem > 48 * 1024)
    CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
}

template <int R, bool kMulti, bool kItem>
void launch_panels(const F64Args &a, int64_t blocks, size_t smem, int threads, cudaStream_t st) {
  allow_smem(f64_panel_kernel<R, false, kMulti, kItem>, smem, kStageSmem);
  allow_smem(f64_panel_kernel<R, true, kMulti, kItem>, smem, kStageSmem);
  f64_panel_kernel<R, false, kMulti, kItem><<<(unsigned)blocks, threads, smem, st>>>(a);
  f64_panel_kernel<R, true, kMulti, kItem><<<(unsigned)blocks, threads, smem, st>>>(a);
  count_launch(2);
}

template <int R, bool kMulti>
void launch_r(const F64Args &a, Variant variant, int64_t blocks, size_t smem, int threads, cudaStream_t st) {
  if (variant == kItemPanels) return launch_panels<R, kMulti, true>(a, blocks, smem, threads, st);
  if (variant == kPanels) return launch_panels<R, kMulti, false>(a, blocks, smem, threads, st);
  allow_smem(f64_item_kernel<R, kMulti>, smem, kStageSmem);
  f64_item_kernel<R, kMulti><<<(unsigned)blocks, threads, smem, st>>>(a);
  count_launch(1);
}

void launch(const F64Args &a, int R, Variant variant, int64_t blocks, size_t smem, int threads, cudaStream_t st) {
  if (blocks == 0) return;
  (void)grid_blocks(blocks);   // refuses what one launch cannot hold
  auto with = [&](auto multi) {
    constexpr bool m = decltype(multi)::value;
    if (R == 4)
      launch_r<4, m>(a, variant, blocks, smem, threads, st);
    else if (R == 5)
      launch_r<5, m>(a, variant, blocks, smem, threads, st);
    else
      launch_r<6, m>(a, variant, blocks, smem, threads, st);
  };
  if (a.n > 0)
    with(std::true_type());
  else
    with(std::false_type());
}

}  // namespace

bool f64_supported(const Model &M) {
  const int tab = table_size(M);
  if (M.n_exp > kF64MaxExp || M.n_modes > kF64MaxModes || tab > kF64MaxTab || panel_smem(M.d, tab) > kStageSmem)
    return false;
  if (row_products(M) > 500) return false;   // the 64-bit sums stay exact
  for (double h : M.vb_H)
    if (!std::isfinite(h)) return false;
  return true;
}

std::vector<double> f64_matrix(const Model &M, const std::vector<double> &X) {
  const std::vector<DD> A = coupling_matrix(M, X);
  std::vector<double> r(A.size());
  for (size_t i = 0; i < r.size(); ++i) r[i] = A[i].h;
  return r;
}

F64Ops f64_build(const Model &M, const std::vector<int32_t> &nb_off, const std::vector<int32_t> &nb_idx,
                 const std::vector<double> &nb_cA, const std::vector<double> &nb_cB, double hsign,
                 std::vector<void *> &allocs) {
  F64Ops O;
  const int d = M.d, R = row_group(M);
  O.d = d;
  O.n_ado = M.n_ado;
  O.n_modes = M.n_modes;
  O.R = R;
  O.groups = (d + R - 1) / R;
  O.tab = table_size(M);
  O.hsign = hsign;
  // H' shifted by the middle of its diagonal (the commutator does not change; smaller
  // entries, smaller rounding of the limbs) and scaled by a power of two so that the
  // absolute sum of a row stays below 1: with |w| < 1 the integer sums cannot overflow.
  std::vector<DD> Hc = coupling_matrix(M, M.H);
  double lo = Hc[0].h, hi = lo;
  for (int a = 0; a < d; ++a) {
    lo = std::min(lo, Hc[(size_t)a * d + a].h);
    hi = std::max(hi, Hc[(size_t)a * d + a].h);
  }
  for (int a = 0; a < d; ++a) Hc[(size_t)a * d + a].add_product(DD{-0.5 * (lo + hi), 0.0}, DD{1.0, 0.0});
  auto h_at = [&](int a, int c) {
    if (digits_differ(M, a, c) > 2) return DD();
    return Hc[(size_t)std::min(a, c) * d + std::max(a, c)];
  };
  double norm = 0.0;
  for (int a = 0; a < d; ++a) {
    double s = 0.0;
    for (int c = 0; c < d; ++c) s += std::fabs(h_at(a, c).h);
    norm = std::max(norm, s);
  }
  std::frexp(norm > 0 ? norm * (1 + 1e-12) : 1.0, &O.hexp);
  // |h1|, |z1| <= 2^30 and |h0|, |z0| <= 2^(low - 1): the cross sum stays below
  // (products + 1) 2^(29 + low) < 2^63
  const int bits = row_products(M) <= 250 ? 57 : 56, low = bits - 31;
  O.bits = bits;
  auto limbs = [&](int a, int c) {
    const DD h = h_at(a, c);
    const double x = std::ldexp(h.h, bits - 1 - O.hexp);
    const long long v0 = std::llrint(x), v = v0 + std::llrint(x - (double)v0 + std::ldexp(h.l, bits - 1 - O.hexp));
    int2 r;
    r.y = (int)((unsigned)(unsigned long long)v << (32 - low)) >> (32 - low);
    r.x = (int)((v - r.y) >> low);
    return r;
  };
  std::vector<int> foff(1, 0), fc, doff(1, 0), soff(1, 0);
  std::vector<int2> hd(d <= kSmallD ? (size_t)d * d : 0);   // the same limbs, dense
  auto dense = [&](int a, int c, const int2 &v) {
    if (a < d && !hd.empty()) hd[(size_t)a * d + c] = v;
  };
  std::vector<int4> fh, dh, sh;
  const bool aligned = R == M.dims.back();   // a group is the last mode's digits
  auto last_digit_kept = [&](int a, int c) { return a % R == c % R; };
  for (int g = 0; g < O.groups; ++g) {
    const int a0 = g * R, a1 = std::min(d, a0 + R);
    std::vector<std::vector<int>> single(R);
    for (int c = 0; c < d; ++c) {
      int nz = 0;
      for (int a = a0; a < a1; ++a) nz += digits_differ(M, a, c) <= 2;
      // all rows together (one read of w, R products) or row by row
      if (2 * nz > R) {
        fc.push_back(c);
        for (int p = 0; p < (R + 1) / 2; ++p) {
          const int2 u = a0 + 2 * p < a1 ? limbs(a0 + 2 * p, c) : make_int2(0, 0);
          const int2 v = 2 * p + 1 >= R ? make_int2(c, 0) : a0 + 2 * p + 1 < a1 ? limbs(a0 + 2 * p + 1, c) : make_int2(0, 0);
          dense(a0 + 2 * p, c, u);
          if (2 * p + 1 < R) dense(a0 + 2 * p + 1, c, v);
          fh.push_back(make_int4(u.x, u.y, v.x, v.y));
        }
      } else {
        for (int a = a0; a < a1; ++a)
          if (digits_differ(M, a, c) <= 2) single[a - a0].push_back(c);
      }
    }
    foff.push_back((int)fc.size());
    if (aligned) {
      const std::vector<int> cand = single[0];
      for (int c : cand)
        if (last_digit_kept(a0, c)) {
          const int2 v = limbs(a0, c);
          dh.push_back(make_int4(v.x, v.y, c, 0));
          for (int r = 0; r < R; ++r) {
            single[r].erase(std::find(single[r].begin(), single[r].end(), c + r));
            dense(a0 + r, c + r, v);
          }
        }
    }
    doff.push_back((int)dh.size());
    for (int r = 0; r < R; ++r) {
      for (int c : single[r]) {
        const int2 v = limbs(a0 + r, c);
        sh.push_back(make_int4(v.x, v.y, c, 0));
        dense(a0 + r, c, v);
      }
      soff.push_back((int)sh.size());
    }
  }
  std::vector<F64Entry> nb(nb_idx.size());
  for (size_t q = 0; q < nb.size(); ++q)
    nb[q] = F64Entry{nb_idx[q], nb_cB[q] != 0.0 ? 2 : nb_cA[q] != 1.0 ? 1 : 0, nb_cA[q], nb_cB[q]};
  std::vector<double2> fg;
  std::vector<uint16_t> dig((size_t)M.n_modes * d);
  for (int s = 0; s < M.n_modes; ++s) {
    O.dims[s] = M.dims[s];
    O.tab_off[s] = (int)fg.size();
    for (int a = 0; a < M.dims[s]; ++a)
      for (int b = 0; b < M.dims[s]; ++b)   // lam_a -+ lam_b, rounded once
        fg.push_back(make_double2((M.cb_lam[s][a] - M.cb_lam[s][b]) + (M.cb_lam_lo[s][a] - M.cb_lam_lo[s][b]),
                                  (M.cb_lam[s][a] + M.cb_lam[s][b]) + (M.cb_lam_lo[s][a] + M.cb_lam_lo[s][b])));
    for (int a = 0; a < d; ++a) dig[(size_t)s * d + a] = (uint16_t)((a / M.stride[s]) % M.dims[s]);
  }
  if (!hd.empty()) O.hd = up(hd, allocs);
  O.foff = up(foff, allocs);
  O.fc = up(fc, allocs);
  O.fh = up(fh, allocs);
  O.doff = up(doff, allocs);
  O.dh = up(dh, allocs);
  if (!sh.empty()) {
    O.soff = up(soff, allocs);
    O.sh = up(sh, allocs);
  }
  O.noff = up(std::vector<int>(nb_off.begin(), nb_off.end()), allocs);
  O.nb = up(nb, allocs);
  O.decay = up(M.decay, allocs);
  O.fg = up(fg, allocs);
  O.dig = up(dig, allocs);
  O.ready = true;
  return O;
}

std::vector<std::pair<int, int>> f64_shapes(const F64Buf &b) {
  Variant variant = kItems;
  size_t smem = 0;
  int64_t blocks = 0;
  make_set(b, 0, &variant, &smem, &blocks);
  const int n = (int)std::min<int64_t>(blocks, 0x7fffffff);
  if (variant == kItems) return {{256, n}, {128, n}, {64, n}};
  const int t = panel_shape(b.ops->R, blocks);
  return b.ops->R == 5 ? std::vector<std::pair<int, int>>{{t, n}, {480 - t, n}}
                       : std::vector<std::pair<int, int>>{{t, n}, {640 - t, n}, {128, n}};
}

void f64_stage(const F64Buf &b, double alpha, int threads, cudaStream_t st) {
  Variant variant = kItems;
  size_t smem = 0;
  int64_t blocks = 0;
  F64Args a{};
  a.one = make_set(b, 0, &variant, &smem, &blocks);
  a.alpha = alpha;
  launch(a, b.ops->R, variant, blocks, smem, threads, st);
}

namespace {

struct SmallShape {
  int sync = 0, blocks = 0, threads = 0, cluster = 1;
  size_t smem = 0;
};

// Elements per block up to which a launch for all steps wins: beyond it a stage's own
// work (20-26 FP64 operations per element, two per clock and SM) exceeds what a launch
// per stage costs, and the whole-item kernel, which multiplies only H''s non-zeros over
// the whole GPU, takes over.
constexpr int kSmallElems = 1536;

bool small_fit(F64SmallSet &p, SmallShape &sh) {
  const F64Ops &O = p.O;
  const int dd = O.d * O.d;
  const int64_t n_units = (sh.sync == 2 ? p.branches : 1) * (int64_t)O.n_ado * p.parts;
  p.units = (int)std::min<int64_t>((n_units + p.bpb - 1) / p.bpb, 1 << 20);
  if (sh.sync == 2) p.bpb = (int)((n_units + p.units - 1) / p.units);
  const int64_t max_items = (p.units + p.parts - 1) / p.parts + (p.parts > 1 ? 1 : 0);
  const int64_t work = (int64_t)p.units * dd / p.parts;
  const int rows = (O.d + p.parts - 1) / p.parts;
  const int64_t smem = O.tab * 16 + max_items * ((int64_t)O.d * (O.d | 1) * 16 + sizeof(SmallItem) + 8 + dd * 4) + dd * 8 +
                       2 * O.n_modes * O.d * 4 + (int64_t)p.units * rows * O.d * 4;
  if (work > kSmallElems || smem > (int64_t)kSmallSmem || n_units * dd > (1 << 30)) return false;
  sh.smem = std::max(sh.smem, (size_t)smem);
  sh.threads = std::max(sh.threads, work <= 32 ? 64 : work <= 64 ? 128 : work <= 256 ? 256 : 512);
  sh.blocks += sh.sync == 2 ? p.bpb : p.branches * p.bpb;
  return true;
}

// How the steps of one hierarchy's branches run as one launch; false: they do not.
bool small_shape(F64SmallSet &p, SmallShape &sh) {
  if (!p.O.hd || p.branches < 1) return false;
  const int sms = sm_count(), B = p.branches;
  const int64_t elems = (int64_t)p.O.n_ado * p.O.d * p.O.d;
  p.parts = 1;
  int c = 1;
  while (c < 16 && 2 * c * (int64_t)B <= sms && c < p.O.n_ado) c *= 2;
  p.bpb = sh.cluster = c;
  sh.sync = c > 1 ? 1 : 0;
  // a cluster reaches 16 SMs; a few larger branches spread over the whole grid instead
  if (B * (int64_t)c * 3 < 2 * sms && elems / c > 256) {
    sh.sync = 2;
    const int64_t items = (int64_t)B * p.O.n_ado;
    p.parts = (int)std::max<int64_t>(1, std::min<int64_t>(4, sms / items));
    p.bpb = (int)std::min<int64_t>(sms, items * p.parts);
  }
  return small_fit(p, sh);
}

template <bool kMulti>
bool launch_small(const F64SmallArgs &a, const SmallShape &sh, cudaStream_t st) {
  auto kernel = sh.sync == 0 ? f64_small_kernel<0, kMulti> : f64_small_kernel<1, kMulti>;
  if constexpr (!kMulti)
    if (sh.sync == 2) kernel = f64_small_kernel<2, false>;
  allow_smem(kernel, sh.smem, kSmallSmem);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)sh.blocks);
  cfg.blockDim = dim3((unsigned)sh.threads);
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  cfg.attrs = &at;
  if (sh.sync == 1) {
    if (sh.cluster > 8) CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)sh.cluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n < 1) {
      (void)cudaGetLastError();
      return false;
    }
  } else if (sh.sync == 2) {
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cfg.numAttrs = 1;
  }
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, a);
  if (e == cudaErrorCooperativeLaunchTooLarge) {   // fewer SMs than the device's
    (void)cudaGetLastError();
    return false;
  }
  CUDA_TRY(e);
  count_launch(1);
  return true;
}

}  // namespace

bool f64_small_steps(const F64Ops &O, double2 *y, double2 *wa, double2 *wb, int branches, double dt, int64_t steps,
                     cudaStream_t st, std::pair<int, int> *shape) {
  F64SmallArgs a{};
  SmallShape sh;
  a.one.O = O;
  a.one.y = y;
  a.one.wa = wa;
  a.one.wb = wb;
  a.one.branches = branches;
  for (int q = 0; q < 4; ++q) a.alpha[q] = dt / (4 - q);
  a.steps = steps;
  if (!small_shape(a.one, sh) || !launch_small<false>(a, sh, st)) return false;
  if (shape) *shape = {sh.threads, sh.blocks};
  return true;
}

F64SmallPlan::~F64SmallPlan() {
  if (desc) cudaFree(desc);
}

void f64_small_plan(F64SmallPlan &p, const std::vector<F64SmallBuf> &sets, cudaStream_t st) {
  std::vector<F64SmallSet> v;
  SmallShape sh;
  const int sms = sm_count();
  int64_t total = 0;
  int least = 1 << 30;
  for (const F64SmallBuf &b : sets) {
    if (!b.ops->hd) return;
    total += b.branches;
    least = std::min(least, b.ops->n_ado);
  }
  // one cluster size for all sets; no row ranges and no grid-wide barrier here
  while (sh.cluster < 16 && 2 * sh.cluster * total <= sms && sh.cluster < least) sh.cluster *= 2;
  sh.sync = sh.cluster > 1 ? 1 : 0;
  for (const F64SmallBuf &b : sets) {
    F64SmallSet s{};
    s.O = *b.ops;
    s.y = b.y;
    s.wa = b.wa;
    s.wb = b.wb;
    s.branches = b.branches;
    s.parts = 1;
    s.bpb = sh.cluster;
    s.begin = sh.blocks;
    if (!small_fit(s, sh)) return;
    v.push_back(s);
  }
  if (device_malloc(&p.desc, v.size() * sizeof(F64SmallSet)) != cudaSuccess) {
    p.desc = nullptr;
    (void)cudaGetLastError();
    throw DeviceOom();
  }
  CUDA_TRY(cudaMemcpyAsync(p.desc, v.data(), v.size() * sizeof(F64SmallSet), cudaMemcpyHostToDevice, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  p.n = (int)v.size();
  p.sync = sh.sync;
  p.blocks = sh.blocks;
  p.threads = sh.threads;
  p.cluster = sh.cluster;
  p.smem = sh.smem;
}

bool f64_small_steps_plan(const F64SmallPlan &p, double dt, int64_t steps, cudaStream_t st) {
  if (!p.desc) return false;
  F64SmallArgs a{};
  a.many = (const F64SmallSet *)p.desc;
  a.n = p.n;
  for (int q = 0; q < 4; ++q) a.alpha[q] = dt / (4 - q);
  a.steps = steps;
  SmallShape sh;
  sh.sync = p.sync;
  sh.blocks = p.blocks;
  sh.threads = p.threads;
  sh.cluster = p.cluster;
  sh.smem = p.smem;
  return launch_small<true>(a, sh, st);
}

F64Plan::~F64Plan() {
  for (Class &c : classes)
    if (c.desc) cudaFree(c.desc);
}

void f64_plan(F64Plan &p, const std::vector<F64Buf> &sets, cudaStream_t st) {
  std::map<std::pair<int, int>, std::vector<F64Set>> by;
  std::map<std::pair<int, int>, std::pair<int64_t, size_t>> size;
  for (const F64Buf &b : sets) {
    Variant variant = kItems;
    size_t smem = 0;
    int64_t blocks = 0;
    F64Set s = make_set(b, 0, &variant, &smem, &blocks);
    const auto key = std::make_pair(b.ops->R, (int)variant);
    s.begin = size[key].first;
    size[key].first += blocks;
    size[key].second = std::max(size[key].second, smem);
    by[key].push_back(s);
  }
  for (auto &kv : by) {
    F64Plan::Class c{kv.first.first, kv.first.second, size[kv.first].first, size[kv.first].second,
                     (int)kv.second.size(), nullptr};
    if (device_malloc(&c.desc, kv.second.size() * sizeof(F64Set)) != cudaSuccess) {
      (void)cudaGetLastError();
      throw DeviceOom();
    }
    p.classes.push_back(c);
    CUDA_TRY(cudaMemcpyAsync(c.desc, kv.second.data(), kv.second.size() * sizeof(F64Set), cudaMemcpyHostToDevice, st));
  }
  CUDA_TRY(cudaStreamSynchronize(st));
}

void f64_stage_plan(const F64Plan &p, double alpha, cudaStream_t st) {
  for (const F64Plan::Class &c : p.classes) {
    F64Args a{};
    a.many = (const F64Set *)c.desc;
    a.n = c.n;
    a.alpha = alpha;
    launch(a, c.R, (Variant)c.variant, c.blocks, c.smem, c.variant == kItems ? 256 : panel_shape(c.R, c.blocks), st);
  }
}

bool rot_supported(const Model &M) {
  if (M.n_modes > kF64MaxModes || (size_t)M.d * kRotPad * 16 > kRotSmem) return false;
  for (int n : M.dims)
    if (n > kRotMaxN) return false;
  return true;
}

RotOps rot_build(const Model &M, std::vector<void *> &allocs) {
  RotOps r;
  r.d = M.d;
  r.n_modes = M.n_modes;
  std::vector<int2> f, b;
  for (int s = 0; s < M.n_modes; ++s) {
    const int n = M.dims[s];
    auto limbs = [&](int k, int i) {
      const double h = std::ldexp(M.cb_U[s][(size_t)k * n + i], 59), l = std::ldexp(M.cb_U_lo[s][(size_t)k * n + i], 59);
      const long long v0 = std::llrint(h), v = v0 + std::llrint(h - (double)v0 + l);
      int2 c;
      c.y = (int)((unsigned)(unsigned long long)v << 2) >> 2;
      c.x = (int)((v - c.y) >> 30);
      return c;
    };
    r.dims[s] = n;
    r.stride[s] = M.stride[s];
    r.off[s] = (int)f.size();
    for (int k = 0; k < n; ++k)
      for (int i = 0; i < n; ++i) {
        f.push_back(limbs(k, i));
        b.push_back(limbs(i, k));
      }
  }
  r.fwd = up(f, allocs);
  r.bwd = up(b, allocs);
  r.ready = true;
  return r;
}

void rotate(const RotOps &r, bool forward, const double2 *x, double2 *out, double2 *tmp, int64_t items, cudaStream_t st) {
  const int panels = (r.d + 31) / 32, dd = r.d * r.d;
  const int2 *u = forward ? r.fwd : r.bwd;
  const size_t smem = (size_t)r.d * (r.d <= kSmallD ? r.d | 1 : kRotPad) * 16;
  if (r.d > kSmallD) {
    allow_smem(rotate_kernel<false>, smem, kRotSmem);
    allow_smem(rotate_kernel<true>, smem, kRotSmem);
  }
  for (int64_t n = 0; items > 0; items -= n, x += ado_offset(n, r.d), out += ado_offset(n, r.d)) {
    if (r.d <= kSmallD) {
      n = launch_share(items, 1);
      rotate_item_kernel<<<grid_blocks(n), dd <= 64 ? 64 : dd <= 128 ? 128 : 256, smem, st>>>(x, out, u, r);
      count_launch(1);
      continue;
    }
    n = launch_share(items, panels);
    rotate_kernel<false><<<grid_blocks(n * panels), 256, smem, st>>>(x, tmp, u, r, panels);
    rotate_kernel<true><<<grid_blocks(n * panels), 256, smem, st>>>(tmp, out, u, r, panels);
    count_launch(2);
  }
}

}  // namespace heom
