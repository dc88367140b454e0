// Device-side records of the batched personalised-PageRank kernel, shared by
// the one-shot batch call (ppr.cu, ppr_steps.cu) and the continuous-batching server
// (serve.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "gpr_internal.cuh"

namespace gpr {

constexpr int kPprCols = 64;  // columns per job

enum : int32_t { kColEmpty = 0, kColFresh = 1, kColRunning = 2, kColDone = 3 };

// One personalised-PageRank column (one seed).
struct PprCol {
  int32_t status;
  int32_t seed;       // original node id
  float damping;
  float tol;          // stop when d/(1-d) * ||x_k - x_{k-1}||_1 <= tol (0: never)
  int32_t max_iters;  // stop after this many steps in total
  int32_t iters;      // steps run so far
  double dangling;    // dangling mass of the current iterate
  double residual;    // last ||x_k - x_{k-1}||_1
  double best;        // smallest residual so far
  float* out;         // where the finished column goes: out[v * ldo], v = node id
  int32_t ldo;
  int32_t stall;      // steps since the residual last reached a new minimum
  float bused;        // seed coefficient (1 - d) + d D of the latest step (BF16 deltas recompute x from it)
};

// A column with tol > 0 also stops once its residual has not reached a new
// minimum for this many steps: the update contracts L1 distances by d per
// step, so a residual that stops shrinking has met the floor of the storage
// precision, and no further step brings the iterate closer.
constexpr int32_t kStallSteps = 8;

// One ppr_batch job: a graph and 64 column places; its state lives in the
// workspace of the cluster that runs it.
struct PprJob {
  const int32_t* col_ptr;  // relabelled CSC (execution layout)
  const int32_t* row_idx;
  const float* inv_deg;
  const int32_t* old2new;
  const int32_t* heavy_rows;  // ascending ids of the long rows (in-degree > heavy_deg)
  int32_t n_heavy;
  int32_t heavy_deg;
  int32_t n;
  int32_t n_cap;        // rows of the per-cluster workspace
  int32_t iters;        // steps to run at most
  PprCol* cols;         // 64 records
};

// ---- step-major execution (ppr_steps.cu) --------------------------------------
constexpr int kStWarps = 8;          // warps of a block
constexpr int64_t kPieceWork = 256;  // work of a piece: an edge counts 1, a row 3

struct StepState;

// One graph with up to 64 columns: a job of a batch, or a slot of the server.
struct StepJob {
  const int32_t* col_ptr;
  const int32_t* row_idx;
  const float* inv_deg;
  const int32_t* old2new;
  const int32_t* new2old;
  int64_t m;
  int32_t n, npieces, nitems;
  int32_t per;          // pieces of an item for each of its block's warps
  int32_t long_deg;     // rows of more edges are summed by chunks
  int32_t* prows;       // npieces + 1 row boundaries
  int32_t* long_base;   // a batch's: first chunk of each long row (n entries)
  float* X;             // n x W: x, or with BF16 deltas the running sums
  void* C[2];           // (n + 1) x W: contributions, and a row of zeros
  float* S;             // n x W: sent sums (BF16 deltas)
  float* chunk_sum;     // chunks x W
  // a slot's long rows and chunks are the graph plan's: long row i of
  // heavy_rows (ascending) sums chunks [hbeg, hend) then [cbeg, cend) of split
  // entry split0 + i
  const int32_t* heavy_rows;
  const int32_t* chunk_begin;
  const int32_t* chunk_end;
  const int32_t* split_hbeg;
  const int32_t* split_hend;
  const int32_t* split_cbeg;
  const int32_t* split_cend;
  int32_t n_heavy, split0, nchunks;
  int32_t parity;       // C[parity & 1] holds the contributions before step 0
  StepState* st;
  PprCol* cols;         // 64 records
};

// The state of a job's columns between two steps.
struct StepState {
  float d[kPprCols], b[kPprCols], bprev[kPprCols], tol[kPprCols];
  int32_t seed[kPprCols], status[kPprCols], iters[kPprCols], stall[kPprCols], max_iters[kPprCols];
  double res[kPprCols], best[kPprCols];
  unsigned long long acc[2][kPprCols];  // this step's dangling masses and residuals so far
  uint32_t arrived;                     // items that have added theirs
  int32_t live;                         // columns still running
};

// A chunk of a long row: edges [e0, e1) of job `slot`.
struct LongChunk {
  int32_t slot, e0, e1, pad;
};

struct StepItem {
  int32_t slot, part;
};

// Pieces of g's rows, of about kPieceWork work each.
int32_t ppr_pieces(const gpr_graph* g);
// The pieces' row boundaries (ppr_pieces(g) + 1).
void ppr_piece_bounds(const gpr_graph* g, int32_t* prows, cudaStream_t s);
// The long rows of g's plan (in-degree above *deg): *n ascending row ids, the
// first of them split entry *split0 of the plan's chunk lists.
void heavy_of(const gpr_graph* g, const int32_t** rows, int32_t* n, int32_t* deg, int32_t* split0);
// `steps` steps of the slots of `items`, (slot, q) for every kStWarps x per pieces:
// columns with status kColFresh in their records join first,
// finished ones go out by node id at the end, when the records are written.
// citems: (slot, q) for every kStWarps chunks of the slots.  scratch: a word.
void ppr_slot_steps(const StepJob* jobs, const StepItem* items, int nitems, const StepItem* citems, int ncitems,
                    int32_t steps, gpr_dtype dt, uint32_t* scratch, cudaStream_t s);

// One graph with k <= 64 columns, whose 64 records are in device memory: the
// outputs of columns 0..k-1 are consecutive floats of a row of x_out.
struct StepRequest {
  const gpr_graph* graph;
  int32_t k;
  PprCol* cols;
};
// Runs every request to its end on s (no synchronisation, but for every few
// steps' look at the stops when tol) and leaves status, iters and residual in
// the records.
void run_ppr_steps(const std::vector<StepRequest>& reqs, int32_t max_iters, bool tol, gpr_dtype dt, cudaStream_t s);

}  // namespace gpr
