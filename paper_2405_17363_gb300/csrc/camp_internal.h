// Internal declarations shared by the host layer and the kernel translation
// units of the batched BiCGSTAB library.  Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include "camp_solver.h"

namespace camp {

// SpMV schedule word of one slot (see build_schedule in solver.cu): 4 * col
// (bits 16-31) | 4 * row (bits 2-15) | end (bit 0): the slot multiplies the
// gathered vector's entry col; on the last slot of a row (end) the running
// sum is stored to row.  Four slots of a lane are one 16-byte load: slot j of
// lane sl lies at word_pos(j, sl).  Alongside, src (same places) is the entry
// of the cell's A row (pattern order) that slot uses, or -1 for padding; each
// cell's A is staged in slot order, two slots of a lane side by side
// (pair_pos), so a lane reads them with one 16-byte load.  Slots past the last
// whole block (pair) lie [slot][lane], so neither layout needs padding.
typedef unsigned int SchedWord;
constexpr unsigned kSlotEnd = 1u, kSlotRowMask = 0xfffcu;
constexpr int kSlotBlock = 4;  // slots per word block
// A dst map's second copy starts here: at an odd int, so that its entry 1 is
// 8-byte aligned (the map has dst_odd(nnz) + nnz ints).
__host__ __device__ inline int dst_odd(int nnz) { return nnz | 1; }
// Words of a launch's row-end mask, one bit per slot; slots past it are taken
// as row ends of some lane (what every slot of so long a product is anyway).
constexpr int kEndWords = 8;
__host__ __device__ inline SchedWord slot_word(int col, int row, bool end) {
  return ((SchedWord)col << 18) | ((SchedWord)row << 2) | (end ? kSlotEnd : 0u);
}
__host__ __device__ inline int word_pos(int j, int sl, int L, int Lc) {
  return j < (L & ~3) ? ((j >> 2) * Lc + sl) * 4 + (j & 3) : j * Lc + sl;
}
__host__ __device__ inline int pair_pos(int j, int sl, int L, int Lc) {
  return j < (L & ~1) ? ((j >> 1) * Lc + sl) * 2 + (j & 1) : j * Lc + sl;
}
// Bytes the plain launches reserve at the start of dynamic shared memory for
// nsch schedule words (rounded to 16); the host sizes the allocation and the
// kernels place their per-warp regions with this one function.
__host__ __device__ inline size_t sched_smem_bytes(int nsch) {
  return (((size_t)nsch * sizeof(SchedWord)) + 15) & ~(size_t)15;
}

// Tables of a mass-action mechanism for one lane count, read through L1.  A
// cell's chains (the Jacobian terms of a matrix entry, the rate terms of a row)
// may be summed by any lane, each in its order: they are sorted by length and
// taken in groups of Lc, one per lane, all lanes running as many steps as the
// group's longest (shorter chains start with steps that add zero), so the
// loops are uniform and the lanes balanced.  Offsets are bytes from the cell's
// matrix block; the two entries after it hold 1.0 and 0.0 while the tables
// are used, the third takes what idle lanes store.
struct MechTables {
  // Jacobian: runs of groups {steps, groups}; per group and lane {start value
  // of the chain (its leading constant terms summed on the host, in order),
  // place of the entry, high word of its identity part}; per step and lane
  // {coefficient, offset of its concentration or of 1.0}
  const int2 *jrun;
  const int4 *jhead, *jstep;
  int jruns;
  // rates f(y), in chunks of at most the matrix block's doubles: per chunk
  // {rounds of second-order reactions, rounds of first-order ones, runs of
  // row groups, 0}; per round and lane {rate constant, offsets of y_a | y_b
  // << 16 in units of 8 bytes, offset of the reaction's rate}; per group and
  // lane the row's offset in the rate vector's buffer; per step and lane the
  // reaction's rate offset | sign << 31
  const int4 *rchunk;
  int rchunks;
  const int4 *rate;
  const int2 *rrun;
  const int *rhead;
  const unsigned *rstep;
};

// Arguments of the warp-packed kernel: Lc lanes per cell, k = 32/Lc cells per
// warp ("segments"), E rows per lane (template), one group of k consecutive
// cells per warp at a time.
struct WarpArgs {
  int cells, n, nnz;
  int Lc, log2Lc, k;       // lanes per cell, log2, cells per warp
  int L;                   // schedule slots per lane
  int segA, segV;          // shared-memory doubles per cell: A block, one vector
  int segStride;           // doubles from one cell's block to the next (bank-spread)
  int ngroups;             // ceil(cells / k)
  const double *A, *b;     // [cells x nnz], [cells x n]
  double *x;               // [cells x n]
  int *iters;              // [cells]
  double *resid;           // [cells]
  int *status;             // [cells] or null
  const SchedWord *sched;  // [L x Lc] slot words (word_pos)
  const int *src;          // [L x Lc] A entry of each slot (word_pos; transposed view: permuted), -1 pad
  const int *dst;          // [nnz] place (pair_pos) of each A entry (pattern order), twice (dst_odd)
  const int *pads;         // [npads] places (pair_pos) of the padding slots; npads < 0: [Lc] each
  int npads;               // lane's first padding slot (all its later ones are padding too)
  unsigned ends[kEndWords];  // bit j: some lane ends a row in slot j
  const int *dslot;        // [n] place (pair_pos) of each row's diagonal entry
  const int *dentry;       // [n] A entry of each row's diagonal (A read from global memory)
  // Single-cell tickets (the plain launch at 16 lanes per cell): tickets t <
  // single_from solve the pair at positions 2t, 2t+1; tickets t >= single_from
  // solve the one cell at position 2 * single_from + (t - single_from) with
  // all 32 lanes, bit for bit as its pair would (split schedule below: each
  // 16-lane lane's rows divided between lanes v and v + 16, every row's
  // entries in the same order).  No single tickets when sched2 is null or
  // single_from >= ngroups.
  int single_from;
  int L2;                  // slots per lane of the split schedule
  const SchedWord *sched2; // [L2 x 32]
  const int *dst2;         // [nnz] split place of each A entry
  const int *pads2;        // [npads2] places of its padding slots
  int npads2;
  unsigned ends2[kEndWords];
  const int *dslot2;       // [n] split place of each row's diagonal entry
  double tol;
  int maxit;
  int x0_given;
  // Optional dynamic queue for the plain launch: [0] next group, [1] warps
  // finished.  The last warp to finish resets both to zero, so the pair is
  // ready for the next launch in stream order.  Null: static assignment.
  unsigned int *queue;
  // Optional cell order: group g's segment s solves cell order[g*k + s]
  // (cells sorted by an estimate of their iteration count), or null.  With
  // an order, each SM should get a mix of hard and easy groups in the first
  // wave.  ord_stride 0: every warp first solves group w*B + b (b its CTA
  // of B, w its warp in the CTA; b reversed for odd w), so each CTA, hence
  // each SM, takes one group from every stratum of B groups; the queue's
  // tickets then take groups ord_wave + t (ord_wave = all warps of the grid)
  // in order.  ord_stride > 0 (fewer groups than warps): ticket t takes
  // group (t * ord_stride) mod ord_wave (ord_wave = ngroups, ord_stride
  // coprime with it), so tickets taken together get mixed difficulty.
  const int *order;
  int ord_wave, ord_stride;
  // In-launch difficulty ordering (plain solve only; ord_ws null: off).  The
  // launch is cooperative: every CTA first classifies a contiguous share of
  // the cells by the largest |A_ii - 1| over the diagonal entries at pattern
  // positions ord_rows[0 .. ord_nrows) (the whole diagonal, or the rows where
  // the estimate peaked before), then, through two grid barriers, writes the
  // hardest-first order to ord_out (= order) before any warp solves.
  // ord_ws: kOrdWords ints (class totals, the barrier counter, the
  // time-out flag), zero on entry and cleared by the launch's last warp;
  // ord_cls: [cells] class | rank << 6 words; ord_hits (or null): per
  // sampled row, the CTAs whose hardest cell peaked there; ord_err: a
  // host-mapped word set to 1 (and left set for the host to read) when a
  // bounded wait ran out; ord_wait: the limit of every wait, in SM clock
  // cycles.  After a time-out the launch's last warp marks every cell of the
  // launch CAMP_CELL_INVALID (resid NaN) and clears the order entries.
  int *ord_out;
  int *ord_ws;
  int *ord_cls;
  const int *ord_rows;
  int ord_nrows;
  unsigned *ord_hits;
  int *ord_err;
  long long ord_wait;
  // Fused assembly (assemble_bicgstab_kernel and newton_bicgstab_kernel): the
  // cell's matrix is built in shared memory as A = I - gamma J(conc) instead of
  // read from A; mechanism tables, see MechTables.
  const double *conc;      // [cells x n]
  const double *gamma;     // [cells]
  // Newton corrector (newton_bicgstab_kernel only): the history term is read
  // from b, y (in: initial guess, out: solution) from x, the linear tolerance
  // and iteration cap from tol and maxit.
  MechTables mech;
  double newton_tol;
  int max_newton;
  int *newton_iters;       // [cells]
  double *upd;             // [cells] final ||d|| / ||y||
};

// Persistent launch over up to kMaxMech mechanisms: mechanism m owns work
// items [item_begin[m], item_begin[m+1]) (one item = one group of
// 32/m[m].Lc cells); counter is the queue head (reset to 0 before launch).
constexpr int kMaxMech = 8;
struct BatchArgs {
  int nmech;
  int total_items;
  int item_begin[kMaxMech + 1];
  int warp_doubles;            // shared-memory doubles per warp
  unsigned int *counter;
  WarpArgs m[kMaxMech];        // schedules in global memory
};

// Arguments of the block kernel (the paper's Block-cells(k) arrangement):
// cpb cells per CTA, one thread per row, rows of cell j at threads [j*n, j*n+n).
struct BlockArgs {
  int cells, n, nnz, cpb;
  const double *A, *b;
  double *x;
  int *iters;
  double *resid;
  int *status;
  const int *a_perm;
  const int *diag;
  const int *row_ptr, *col_idx;  // the view's CSR
  double tol;
  int maxit;
  int x0_given;
  int coupled;  // 1: the block's cells form one system (shared scalars, one test)
};

// per-cell grad kernel arguments
struct GradArgs {
  int cells, n, nnz;
  const int *row_of;   // [nnz] row index of entry k
  const int *col_idx;  // [nnz]
  const double *lambda, *x;
  double *gA;
};

// Launchers (each returns the launch error, cudaSuccess on success).
// plain solve; a cooperative launch when a.ord_ws is set (grid must then be
// co-resident: at most SMs x the occupancy of the launch shape)
cudaError_t launch_warp(int E, const WarpArgs &a, int warps_per_block,
                        int grid, size_t smem, cudaStream_t st);
// occupancies of the kernel a launch at Lc lanes per cell with those tickets
// (tk) runs
cudaError_t warp_occupancy(int E, int Lc, int tk, int warps_per_block, size_t smem, int *blocks);
// persistent batch kernel: E in {3,4,5,6,8}, A staged in shared memory or not
const void *batch_kernel(int E, bool a_smem);
cudaError_t batch_prepare(int E, bool a_smem, int warps_per_block, size_t smem,
                          int *blocks_per_sm);
cudaError_t launch_block(const BlockArgs &a, int threads, size_t smem,
                         cudaStream_t st);
cudaError_t block_set_smem(size_t smem);
// fused-assembly solve, E in 1..8
cudaError_t launch_assemble(int E, const WarpArgs &a, int warps_per_block,
                            int grid, size_t smem, cudaStream_t st);
cudaError_t assemble_occupancy(int E, int Lc, int tk, int warps_per_block, size_t smem, int *blocks);
// device Newton corrector around the fused assembly + solve, E in 1..8
cudaError_t launch_newton(int E, const WarpArgs &a, int warps_per_block,
                          int grid, size_t smem, cudaStream_t st);
cudaError_t newton_occupancy(int E, int Lc, int tk, int warps_per_block, size_t smem, int *blocks);
cudaError_t launch_grad(const GradArgs &a, cudaStream_t st);
// Difficulty ordering: cells binned by decreasing max_i |A_ii - 1| (half
// octaves), written to *order (inside the caller's scratch of
// difficulty_scratch_bytes(cells) bytes).
size_t difficulty_scratch_bytes(int cells);
cudaError_t launch_difficulty_order(const double *A, int cells, int n, int nnz,
                                    const int *diag, void *scratch, int **order,
                                    cudaStream_t st);

// Difficulty ordering of a persistent multi-mechanism batch (order.cu): one
// classify and one scatter launch over the concatenated cells of all
// mechanisms (cell_begin: offsets, cell_begin[nmech] = total); counts holds
// per mechanism kOrdClasses totals (zero on entry), cls and pos a cell's class
// and its place in it;
// order + cell_begin[m] receives mechanism m's cells, hardest class first.
struct BatchOrderArgs {
  int nmech;
  const double *A[kMaxMech];
  const int *diag[kMaxMech];
  int n[kMaxMech], nnz[kMaxMech];
  int cell_begin[kMaxMech + 1];
  unsigned char *cls;
  int *counts;
  int *order, *pos;
};
constexpr int kBatchOrderPiece = 64;  // cells a block of the classify launch takes
const void *batch_classify_kernel_fn();  // __global__ (const BatchOrderArgs)
const void *batch_scatter_kernel_fn();   // __global__ (const BatchOrderArgs), 1 thread per cell

constexpr int kMaxE = 16;  // rows per lane supported by the warp kernel
// Tickets of a plain launch: groups of k cells, single cells, or groups and
// then single cells (the last two at 16 lanes per cell).
constexpr int kTicketsPack = 0, kTicketsOne = 1, kTicketsBoth = 2;
inline int tickets_of(const WarpArgs &a) {
  if (!a.sched2 || a.single_from >= a.ngroups) return kTicketsPack;
  return a.single_from == 0 ? kTicketsOne : kTicketsBoth;
}

// Difficulty classes of the ordering (half octaves of max_i |A_ii - 1|) and
// the in-launch ordering's workspace: class totals, one barrier counter
// (word kOrdClasses) and one time-out flag (word kOrdFlag).
constexpr int kOrdClasses = 64;
constexpr int kOrdFlag = kOrdClasses + 1;
constexpr int kOrdWords = kOrdClasses + 2;
// Default limit of the in-launch ordering's waits (SM clock cycles, about a
// second at 2 GHz; a legitimate wait is microseconds).
constexpr long long kOrdWaitCycles = 1ll << 31;
// Cells one CTA classifies per pass of the in-launch ordering, and the
// shared-memory bytes that ordering borrows from the CTA's warp regions
// before they are used: histogram, class bases, the CTA's hardest key, and
// one 64-bit (estimate, row) key per cell of a pass.
constexpr int kOrdPiece = 256;
constexpr size_t kOrdKeyOffset = (2 * kOrdClasses + 4) * sizeof(int);
constexpr size_t kOrdSmemBytes = kOrdKeyOffset + kOrdPiece * sizeof(unsigned long long);
// Rows the ordering samples once it has seen where the estimate peaks, and
// how often (in ordered solves) it reads the whole diagonal again to re-pick.
constexpr int kOrdSample = 8;
constexpr unsigned kOrdRecalibrate = 64;
constexpr int kOrdBatch = 8;  // diagonal loads a thread keeps in flight

// Raise a kernel's dynamic shared-memory limit to the device maximum once per
// (kernel, device): setting the attribute on every launch serialises
// otherwise-concurrent work on some drivers.
cudaError_t ensure_max_smem(const void *kernel);
// Vectors of n (padded) doubles per cell in the warp kernel's shared memory
// for E rows per lane: the gathered vector and the two products; up to
// kRegVecMaxE rows per lane the shadow residual and the Jacobi reciprocals
// stay in registers (freeing shared memory for more resident warps), beyond
// it they take two more vectors.  The Newton launch adds one vector.
constexpr int kRegVecMaxE = 5;
__host__ __device__ constexpr int warp_vectors(int E) { return E <= kRegVecMaxE ? 3 : 5; }

}  // namespace camp

namespace camp {
// Arguments of the FP32-inner / FP64-outer refinement kernel (warp-packed
// layout as WarpArgs).
struct MixedArgs {
  int cells, n, nnz;
  int Lc, log2Lc, k, L;
  int segA, segV;
  int ngroups;
  const double *A, *b;
  double *x;
  int *iters;     // total inner FP32 iterations
  int *sweeps;    // outer sweeps (or null)
  double *resid;  // final FP64 true relative residual
  int *status;    // or null
  const SchedWord *sched;
  const int *src;
  const int *dst;      // [nnz] place (pair_pos) of each A entry in the FP64 copy
  const int *dst32;    // [nnz] place (word_pos) of each A entry in the FP32 copy
  const int *pads, *pads32;  // [npads] places of the padding slots in either copy
  int npads;
  const int *dslot32;  // [n] place (word_pos) of each row's diagonal entry
  double tol;
  int max_sweeps;
  float tol_in;
  int maxit_in;
  int a64_smem;   // 1: FP64 A staged in shared memory; 0: read through L1 from A
  // dynamic group queue and difficulty ordering, as in WarpArgs
  unsigned int *queue;
  const int *order;
  int ord_wave, ord_stride;
  int *ord_out;
  int *ord_ws;
  int *ord_cls;
  const int *ord_rows;
  int ord_nrows;
  unsigned *ord_hits;
  int *ord_err;
  long long ord_wait;
};
// Shared-memory bytes per cell of the refinement kernel: FP32 A, FP64 A when
// staged, and two FP64 vectors, whose space the three FP32 vectors of the
// inner iteration share; rounded to 16 and, with several cells per warp, to Lc
// four-byte banks modulo the 32 (at least 16 bytes), so that the warp's cells
// gather from different banks (24 species, 8 lanes: a multiple of 128 bytes
// put all four cells of a warp on the same ones, 254 us against 211 for 88,758
// cells).
__host__ __device__ inline size_t mixed_cell_bytes(int segA, int segV, bool a64_smem, int Lc) {
  const size_t need = ((size_t)(a64_smem ? 12 : 4) * segA + (size_t)16 * segV + 15) & ~(size_t)15;
  if (Lc >= 32) return need;
  const size_t want = Lc < 4 ? 16 : 4 * (size_t)Lc;
  return need + (want + 128 - need % 128) % 128;
}
// a cooperative launch when a.ord_ws is set (grid at most SMs x occupancy)
cudaError_t launch_mixed(int E, const MixedArgs &a, int warps_per_block,
                         int grid, size_t smem, cudaStream_t st);
cudaError_t mixed_occupancy(int E, int Lc, int warps_per_block, size_t smem, int *blocks);
}  // namespace camp
