// The transform plan (host planner state and device tables), shared by the
// single-pattern entry points (fft_plan.cu) and the many-pattern batch
// (batch.cu).
#pragma once
#include <cuda_runtime.h>

#include <vector>

#include "../../include/pfft.h"
#include "fft_mixed.hpp"
#include "fft_plan.hpp"
#include "lattice.hpp"
#include "plan_common.hpp"

// The stages of one kind of mixed-radix tile and their device tables.
struct MixStages {
  bool ready = false;
  std::vector<pfft::MixStage> st;  // sig, blk and the divisors of a tile are set with its T
  int ndirect = 0;                 // the first ones, run as direct sums
  void* stw = nullptr;
  int* gtab = nullptr;
  int ws_in = 0, ws_out = 0;  // row tiles: pad units of the workspace side
  int *psin = nullptr, *psout = nullptr;
};

struct pfft_plan_s {
  int d = 0;
  int64_t batch = 0;
  int dtype = 0;
  pfft::IMat M, H, G;
  pfft::i64 m = 0;
  std::vector<pfft::i64> eps;                 // all d elementary divisors
  int D = 0;                                  // non-trivial cycles
  std::vector<int> n;                         // their lengths, ascending
  std::vector<std::vector<pfft::i64>> LAM;    // D rows: lambda_j(y) = LAM_j . y mod n_j
  std::vector<std::vector<pfft::i64>> MU;     // D rows: mu_j(k) = MU_j . k mod n_j
  int nD = 1, LB = 1;       // row length and number of rows of the logical LB x nD array
  std::vector<int> pen;     // column-pass pencil axes (row-major), product LB
  int fs_na = 1;            // four-step split of a long last cycle: n = fs_na * nD
  pfft::i64 fs_N = 1;       // the full length of the last cycle
  void* fs_tab = nullptr;   // exp(-2 pi i t / fs_N), two-level table
  // options (set before plan_device)
  pfft::Arena* arena = nullptr;  // sub-allocate device tables here (batch plans)
  int max_threads = 1024;        // of a mixed-radix tile (complex128: 512 at most)
  bool generic_only = false;     // mixed-radix passes only (grouped launches)
  bool own_workspace = true;     // allocate the LB x nD workspace
  bool tc = false;               // split-precision tensor-core radix-16 / 32 stages
  int max2 = 16;                 // largest power-of-two radix of the mixed-radix passes (16 or 8)
  // device state
  int device = 0;
  int nsm = 0;  // multiprocessors
  int* dtab = nullptr;
  void* tw = nullptr;
  int col_n = 0;           // order of tw_col
  void* tw_col = nullptr;  // column-pass table when its axes do not divide nD (split last cycle)
  void* ws = nullptr;
  void* stw = nullptr;  // stage twiddle tables of the register-resident passes
  int* runs = nullptr;  // bulk-copy runs of the row pass
  int* status = nullptr;  // device status word
  pfft::PassArgs rowp{}, colp{};
  // mixed-radix passes (fft_mixed.cuh), by MixKind: which ones the plan runs
  // (a whole tile replaces both passes), their descriptors, and the stages for
  // max2 = 16 [0] and 8 [1]
  bool mixed[3] = {false, false, false};
  pfft::MixDesc mix[3]{};
  MixStages stages[2][3];
  std::vector<int> PIinv;  // element of each column position
  int* maps = nullptr;  // whole tiles: tile positions of the input box's slots, then of the output box's
  pfft::Profiler prof;
  // Transposed route.  Entry (k, y) of F(M) is entry (y, k) of F(M^T) in box
  // order (eq. (Fouriermatrix) read for M^T), so the forward transform of M
  // is the adjoint passes of M^T without their conjugations and the inverse
  // of M is the forward passes of M^T with conjugated input and output.  tr
  // is the plan of M^T (sharing this plan's workspace and status word);
  // tr_fwd / tr_inv: the direction runs through it.
  pfft_plan_s* tr = nullptr;
  bool tr_fwd = false, tr_inv = false;

  int alloc(void** p, size_t bytes) { return arena ? arena->alloc(p, bytes) : pfft::device_alloc(p, bytes); }
};

namespace pfft {
// Exact integer planning (HNF, SNF, cycle split); no device work.
pfft_status plan_host(pfft_plan_s& P, int d, const int64_t* M);
// Device tables and pass descriptors.
pfft_status plan_device(pfft_plan_s& P);
// Re-choose the tiles of both passes (pencils per CTA) under the given
// element budgets and the largest power-of-two radix (16 or 8); mixed-radix
// passes only.  The first call with another radix builds its stage tables on the
// default stream: the caller waits for them before a launch.
pfft_status plan_retile(pfft_plan_s& P, int row_budget, int col_budget, int max2);
void plan_release(pfft_plan_s* P);
}  // namespace pfft
