// The persistent Krylov cycle (cycle.cu): one cooperative launch runs all Arnoldi steps of a GMRES
// cycle, preconditioner included.
#pragma once

#include "solver.h"
#include "solver_dev.h"

namespace lfx {

// Grid, shape and shared memory of the cycle for one system on the current device.
struct CyclePlan {
  int rows_ctas = 0;      // CTAs that own block rows (one more runs the small dense algebra); 0: not eligible
  const CycleMap *map = nullptr;
  int lanes = 4;          // lanes per block row
  size_t smem = 0;
  size_t f_bytes = 0;     // of it: velocity records kept resident
  size_t vb_bytes = 0;    // of it: basis vectors' own rows
  int spill = 0;          // row data left in global memory (own_bytes)
  int device = -1;
};

// Words the CTAs meet at, and the partial sums they exchange.
struct CycleSync {
  unsigned arrived;       // arrivals at the grid barrier, all steps
  unsigned progress;      // 2 (steps decided) + (1 if the cycle has ended)
  unsigned solved;        // 1 once y = R^-1 g is in place
  unsigned product_ns[kMaxRestart];   // the slowest CTA's time in the product of each step (statistics)
  int error;              // a bounded wait gave up
  // statistics of the cycles since the last check: nanoseconds of plain F passes (from barrier to barrier) and
  // of products (the slowest CTA's, summed), and their numbers
  unsigned long long t_f, t_spmv;
  int n_f, n_spmv;
};

template <class S, class T>
struct CycleArgs {
  int64_t V;
  const int32_t *rowptr;
  const int32_t *row_off, *cta_seg, *seg_off;   // row range and segment of each CTA, CTA range of each segment
  int n_seg;
  KState *kseg;                        // [n_seg] status of the segments (n_seg > 1)
  const int32_t *halo_off, *halo;      // each CTA's neighbour rows
  const uint16_t *lcol;                // [nnzb] local index of each block's column
  const S *F, *G, *DC;
  const T *A;                          // [nnzb][16] the Krylov operator
  const T *dinvF, *dinvS;
  const SmoothCoef *cf;
  int f_steps;
  T *Q, *D0, *D1, *X, *W4;             // [V][4] vectors read at neighbours
  T *xp, *rr, *pf;                     // [V]
  T *wk, *t;                           // [V][4], [V]: the Krylov vector and Schur residual, if not in shared memory
  int L;                               // multigrid levels; 1: the dense inverse of S itself
  const CoarseArgs<T> *coarse;
  CsrV<T> R0, P0;
  T *b1;
  const T *x1, *coarse_inv;
  T alpha;
  T *Vb, *Zb, *x;
  KState *ks, *parent;                 // status; that of the flexible solve it preconditions, or null
  void *part, *part_n;                 // [kMaxRestart + 1][rows_ctas], [rows_ctas] partial sums
  CycleSync *sync;
  int m, maxit;
  int max_rows, max_loc;
  uint32_t f_bytes, vb_bytes, polls;   // polls: limit of every wait (0: kWaitPolls)
  unsigned unreachable;                // added to the arrivals that a barrier waits for (tests: it gives up)
  int spill;
};

// CTAs that share V rows of T values on the current device (0: no cooperative launches)
template <class T>
lfx_status cycle_ctas(int64_t V, int *ctas);
template <class S, class T>
lfx_status plan_cycle(int64_t V, int64_t nnzb, const CycleMap &map, CyclePlan *plan);
template <class S, class T>
lfx_status launch_cycle(cudaStream_t st, const CyclePlan &plan, const CycleArgs<S, T> &args);
// bytes of the partial sums of a plan, and where (in doubles) those of the norm start
size_t cycle_part_norm_offset(const CyclePlan &plan);
size_t cycle_part_bytes(const CyclePlan &plan);

}  // namespace lfx
