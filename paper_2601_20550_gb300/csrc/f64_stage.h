// FP64 right-hand side of the hierarchy (Eq. HEOM_DB) in the coupling eigenbasis.
//
// An FP64 state is propagated in the orthogonal basis where every V_s is diagonal
// (rho' = U^T rho U, U the Kronecker product of the per-mode eigenvectors of V_s):
// the system-bath terms are elementwise there, and H' = U^T H_S' U keeps H_S''s
// structure (elements between states that differ in three or more modes vanish).
// The commutator [H', w] runs in 57-bit fixed point on the IMAD pipe, its sums in integers
// (see f64_stage.cu, also for the accuracy); everything else is FP64.  An item's result is
// the same bits in every kernel that takes its basis, so it does not depend on the batch.
#pragma once

#include <cstdint>
#include <utility>
#include <vector>

#include <cuda_runtime.h>

#include "model.h"

namespace heom {

constexpr int kF64MaxModes = 8;
constexpr int kF64MaxTab = 1024;   // sum_s n_s^2 of the (lam_a -+ lam_b) tables

// One entry of an ADO's coupling list: neighbour index and the kind of its
// coefficients (0: cA = 1, cB = 0; 1: cB = 0; 2: both).
struct F64Entry {
  int idx, kind;
  double cA, cB;
};

// Device tables of one right-hand side (the equation's, or its adjoint's).
struct F64Ops {
  bool ready = false;
  int d = 0, n_ado = 0, n_modes = 0;
  int R = 0, groups = 0;          // rows of H' per register group
  int tab = 0;                    // sum_s n_s^2
  double hsign = 1.0;             // -1: the adjoint's -H'
  int bits = 0, hexp = 0;
  int dims[kF64MaxModes] = {}, tab_off[kF64MaxModes] = {};
  // entries of H' as two signed limbs, h = (hi 2^(bits - 31) + lo) 2^(hexp + 1 - bits).  Per
  // group: columns where most rows are non-zero (all R rows' limbs, two per int4; for odd
  // R the spare half of the last holds the column), the columns that all rows meet with
  // one factor, shifted by the row (limbs and first column), then per row the remaining
  // columns (limbs and column; soff null if there are none).
  const int *foff = nullptr, *fc = nullptr, *doff = nullptr, *soff = nullptr;
  const int4 *fh = nullptr, *dh = nullptr, *sh = nullptr;
  const int *noff = nullptr;      // [n_ado * n_modes + 1]
  const F64Entry *nb = nullptr;
  const double *decay = nullptr;  // [n_ado]
  const double2 *fg = nullptr;    // (lam_a - lam_b, lam_a + lam_b) per digit pair, mode after mode
  const int2 *hd = nullptr;       // limbs of H', dense (small bases)
  const uint16_t *dig = nullptr;  // [n_modes][d] digit of mode s
};

// Buffers of one stage out = y + alpha L(w) over branches x n_ado items of ops'
// hierarchy.  y == nullptr: zero.  out may equal y, not w; tp (the commutator's
// part) may equal out, not y or w.
struct F64Buf {
  const F64Ops *ops;
  const double2 *w, *y;
  double2 *out, *tp;
  int branches;
};

// Whether the engine takes the model (table sizes, exactness of the integer sums,
// shared memory of a panel); other models stay on stage_kernel<double>.
bool f64_supported(const Model &M);
// Tables of the forward right-hand side; with nb_* given, those coupling lists and
// -H' instead (the adjoint's).  Allocations are appended to allocs.
F64Ops f64_build(const Model &M, const std::vector<int32_t> &nb_off, const std::vector<int32_t> &nb_idx,
                 const std::vector<double> &nb_cA, const std::vector<double> &nb_cB, double hsign,
                 std::vector<void *> &allocs);
// Launch shapes (threads per block, blocks) of one stage of one hierarchy, the default
// first, and the stage with one of them (the result does not depend on it).
std::vector<std::pair<int, int>> f64_shapes(const F64Buf &b);
void f64_stage(const F64Buf &b, double alpha, int threads, cudaStream_t st);

// steps RK4 steps (Horner form) of branches in one launch, for hierarchies small enough
// that a launch per stage would cost more than the stage; false if this one is not, or
// the launch is not possible (nothing has run then).  shape receives the launch's
// threads per block and blocks.
bool f64_small_steps(const F64Ops &O, double2 *y, double2 *wa, double2 *wb, int branches, double dt, int64_t steps,
                     cudaStream_t st, std::pair<int, int> *shape);

// The same for several hierarchies (empty desc: they do not all fit).
struct F64SmallBuf {
  const F64Ops *ops;
  double2 *y, *wa, *wb;
  int branches;
};
struct F64SmallPlan {
  void *desc = nullptr;
  int n = 0, sync = 0, blocks = 0, threads = 0, cluster = 1;
  size_t smem = 0;
  F64SmallPlan() = default;
  ~F64SmallPlan();
  F64SmallPlan(const F64SmallPlan &) = delete;
  F64SmallPlan &operator=(const F64SmallPlan &) = delete;
};
void f64_small_plan(F64SmallPlan &p, const std::vector<F64SmallBuf> &sets, cudaStream_t st);
bool f64_small_steps_plan(const F64SmallPlan &p, double dt, int64_t steps, cudaStream_t st);

// One stage of several hierarchies: a plan (device descriptors) per set of buffers.
struct F64Plan {
  struct Class {   // sets of one kernel variant
    int R, variant;
    int64_t blocks;
    size_t smem;
    int n;
    void *desc;
  };
  std::vector<Class> classes;
  F64Plan() = default;
  ~F64Plan();
  F64Plan(const F64Plan &) = delete;
  F64Plan &operator=(const F64Plan &) = delete;
};
void f64_plan(F64Plan &p, const std::vector<F64Buf> &sets, cudaStream_t st);
void f64_stage_plan(const F64Plan &p, double alpha, cudaStream_t st);

// Basis change of every ADO, mode by mode: out = U^T x U (forward) or U x U^T.
// fwd, bwd: the per-mode matrices u[k][i], out_i = sum_k u[k][i] x_k, scaled by 2^59 in
// two signed 30-bit limbs.
struct RotOps {
  bool ready = false;
  int d = 0, n_modes = 0;
  int dims[kF64MaxModes] = {}, stride[kF64MaxModes] = {}, off[kF64MaxModes] = {};
  const int2 *fwd = nullptr, *bwd = nullptr;
};
bool rot_supported(const Model &M);
RotOps rot_build(const Model &M, std::vector<void *> &allocs);
// tmp: scratch of the same element count; out may equal x.
void rotate(const RotOps &r, bool forward, const double2 *x, double2 *out, double2 *tmp, int64_t items, cudaStream_t st);
// U^T X U of a d x d matrix of the model, rounded once.
std::vector<double> f64_matrix(const Model &M, const std::vector<double> &X);

}  // namespace heom
