// One operation of the AMG cycle as a plain record.  The cycle (cycle.cu) is written
// against an emitter that launches the operations or records them as phases; recorded
// phases run in the cluster and persistent kernels (cycle.cu) and, on blocks of unit
// vectors, in the construction of the stored coarse-cycle matrix (coarse_map.cu).
#pragma once

#include <cstdint>
#include <vector>

struct amg_handle;

namespace amgp2 {

// kFirst: the colours of a Gauss-Seidel sweep from x = 0 on a row's lower-colour blocks
// (x_j = 0 on the others), x_i = omega D^{-1} s with s = b_i - (L x)_i; it also leaves
// p_i = (1 - omega) s, from which the residual after the sweep is p_i - (U x)_i: kResid with
// b = p on the row's higher-colour blocks (b - L x - D x = s - omega s).
enum RowMode { kApply = 0, kResid = 1, kGS = 2, kJacobi = 3, kFirst = 4 };

enum PhaseType : int {
  PH_ZERO = 0, PH_COPY, PH_ROWS, PH_RESTRICT, PH_PROLONG, PH_RESTRICT1, PH_PROLONG1,
  PH_COARSE, PH_BT_ADD, PH_PROWS, PH_SROWS, PH_VEC, PH_VANKA
};

// One operation of the cycle with its operands (a plain record, copied to the
// device for the cluster launch or passed by value to a single launch).
struct Phase {
  int type, mode, G, n;   // n: rows / nodes / entries
  const int* rows;
  const int* rowptr;      // PH_ROWS: blocks rowptr[g] .. rowend[g] of stored row g
  const int* rowend;
  const int* col;
  const void* val;
  int64_t nnz;
  const void* dinv;
  const void* x;
  const void* b;
  void* y;
  const int* crow;        // PH_PROWS: C; PH_ROWS: B^T (null: none), its nnz in n3, its p in
                          // sd; PH_RESTRICT, PH_PROLONG: m rows of H^T or H, the other
                          // level's nodes in n3
  const int* ccol;
  const void* cval;
  const void* sd;
  const void* p;          // pressure iterate (PH_PROWS); PH_ROWS, kFirst: output (1 - omega) s
  const double* X;
  int m, n3;
  double omega;
  const void* wt;         // the level's steps, weights included (null: omega, 1)
  int vbf;                // PH_ROWS: values stored as BF16 (FP32 arithmetic)
  int sctas;              // PH_ROWS, Gauss-Seidel: CTAs per SM of the streaming colour
                          // kernel (0: one group of lanes per row, k_gs_pdl)
  int tma;                // PH_ROWS, Gauss-Seidel, FP32: the TMA-staged colour kernel
  int* err;               // the handle's error word (bounded waits that gave up)
  const long long* off;   // PH_VANKA: offsets of the patch inverses
};

// The operations that coarse_map.cu tabulates from level l: on level 0 one whole
// preconditioner application, below it what the finer level calls from x = 0 (nu cycles).
template <typename T>
void record_map_phases(amg_handle* h, int l, std::vector<Phase>& ph);

}  // namespace amgp2
