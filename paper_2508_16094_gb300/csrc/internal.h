// Internal data structures of the solver library (host + device).
#pragma once

#include <cmath>
#include <cstdint>
#include <string>
#include <vector>

#include <cuda_runtime.h>

namespace gipm {

// ---------------------------------------------------------------------------
// Symbolic analysis (host). Final numbering = given ordering + etree postorder.
// ---------------------------------------------------------------------------
struct Symbolic {
  int32_t n = 0;
  std::vector<int32_t> perm, iperm;       // final new->old, old->new
  std::vector<int32_t> parent, colcount;  // elimination tree, column counts (incl. diagonal)
  // lower CSC pattern of K in the ORIGINAL numbering (export order)
  std::vector<int64_t> kop;
  std::vector<int32_t> koi;
  // supernodes
  int32_t nsuper = 0, nlevels = 0;
  std::vector<int32_t> super, sparent, slevel;
  std::vector<int64_t> srp;  // row structure of each supernode (rows below its columns)
  std::vector<int32_t> sri;
  int64_t nnz_l = 0;
  double flops = 0.0;
};

// Per-supernode layout of the frontal matrices (device-visible, 64 bytes).
// Front of supernode s: order nf = ncol + nrow; local index p < ncol is column
// first + p, p >= ncol is row sri[rows_off + p - ncol]. The first ncol columns
// live in the panel (row-major, nf rows x ld), the trailing nrow x nrow block
// (the update matrix handed to the parent) lives in U storage (row-major, uld).
// Front assembly tiles: kBuildTile rows x at most kBuildTile columns.
constexpr int kBuildTile = 64;

struct FrontInfo {
  int64_t loff;      // panel offset in the factor storage (elements)
  int64_t uoff;      // update matrix offset in the update storage (elements)
  int64_t rows_off;  // offset of the row structure in sri
  int64_t inv_off;   // offset of this front's map into its parent's front (length nf(parent))
  int32_t first, ncol, nrow, ld;
  int32_t uld, child_begin, child_end, parent;
};
static_assert(sizeof(FrontInfo) == 64, "FrontInfo layout");

// A unit of work of a batched kernel: meaning of a/b depends on the kernel.
struct Task {
  int32_t front, a, b, c;
};

// One task of the persistent solve with everything it reads of its front,
// so a CTA fetches what its next task needs in a single 112-byte copy.
struct SolveRec {
  Task task;
  FrontInfo front;
  int64_t toff;   // the front's update vector
  int64_t pbase;  // its first partial-sum row of the backward sweep
  int32_t slot0;  // slot of its first diagonal block
  int32_t kid_chunks;     // below-front chunks of all its children
  int32_t parent_blocks;  // diagonal blocks of its parent (0 at a root)
  int32_t word0;          // its first column among the published entries
};
static_assert(sizeof(SolveRec) == 112 && sizeof(SolveRec) % 16 == 0, "SolveRec layout");

// A task of a persistent solve. Tasks run in the order of the plan
// (a ticket taken from a global counter), and a task waits only for tasks
// earlier in that order (flags and counters in device memory), so the solve
// needs no grid barrier and cannot deadlock. (Sizes below: FP32, 128-wide blocks.)
enum SolveTaskKind : int32_t {
  WS_FWD_DIAG = 0,   // (front, a = block i): gather the children's update entries for
                     // the block's rows, subtract L_ij y_j for j < i as each y_j is
                     // published, y_i = L_ii^{-1} (.) (explicit inverse), publish y_i
  WS_FWD_BELOW = 1,  // (front, a = first row below the front of a 128-row chunk): gather,
                     // add L_rj y_j for every block j, store the front's update vector
  WS_FWD_NARROW = 2, // (front): both of the above for a narrow front (narrow_front) in one task
  WS_BWD_PART = 3,   // (front, b = first row below of a 128-row chunk): partial sums
                     // L_{r,cb}^T x_r of every column block cb, last first, once the
                     // parent front is done
  WS_BWD_DIAG = 4,   // (front, a = column block cb): the partial sums, L_{i,cb}^T x_i for
                     // i > cb as each x_i is published, x_cb = L_cc^{-T} (.), publish x_cb
  WS_BWD_NARROW = 5  // (front): both of the above for a narrow front in one task
};

// Work of one level of the supernodal tree, as ranges into the task arrays.
//
// Panel solves and trailing updates of the FMA-pipe factor are numbered by
// block: a launch's entries [b, e) hold one Task {front, a = number of the
// front's first block of the launch, b = first column of the step} per front,
// and a block finds its front by bisection, so a front's O((nf / tile)^2)
// update tiles need no list.
constexpr int64_t kSms = 152;  // SMs the schedules are made for
// Rows per batch of a panel solve's blocks, for `rows` rows in the launch: as few as give
// every block an SM of its own (a batch of 16, 8 or 4 rows takes 10, 6 or 4 us of an
// SM's FP64 units and latencies). Batches per block: one while every block has an SM of
// its own, up to four beyond that, which read the diagonal block once per 64 rows.
constexpr int kTrsmRows = 16;
inline int trsm_rows(int64_t rows) { return rows <= 4 * kSms ? 4 : rows <= 8 * kSms ? 8 : kTrsmRows; }
inline int trsm_batches(int64_t rows) {
  const int64_t b = (rows + kTrsmRows * kSms - 1) / (kTrsmRows * kSms);
  return (int)(b < 1 ? 1 : b > 4 ? 4 : b);
}
// Update tile, FP64: 32, and 16 where the launch has at most two blocks of 32 per SM: a
// 32 x 32 tile of 64 columns is 16 us of an SM's FP64 units, a 16 x 16 tile 4 us, so the
// last wave is shorter (31 launches of 3 to 438 tiles: 20.2 us each with 32 throughout;
// with 16 up to half a block per SM a direction takes 2.48 ms, up to two 2.39).
constexpr int kUpdTile64 = 32, kUpdTileSmall64 = 16;
constexpr int kUpdTile32 = 64;  // update tile, FP32
// One trailing-update launch: columns from min(c0, ncol) to min(clim, ncol) of
// the panels, and with_u the update matrices, by the columns [k0, min(k1, ncol)).
struct UpdRange {
  int32_t b = 0, e = 0, n = 0;  // entries, blocks
  int32_t k0 = 0, k1 = 0, c0 = 0, clim = 0, with_u = 0, ts = 0;
};
struct StepRange {
  int32_t potrf_b = 0, potrf_e = 0, trsm_b = 0, trsm_e = 0, trsm_n = 0, trsm_bat = 1, trsm_rows = kTrsmRows;
  UpdRange next64, rest64;  // FP64: the next step's columns (with look-ahead), everything past them
  UpdRange upd32, sup32;  // FP32: the rest of the super-step; at its end everything past it
};

// Tiles of a front's trailing update (TS x TS; see UpdRange): panel column tiles
// from c0 = min(k1, ncol), each with the row tiles from its own first column
// down, then the lower triangle of the update matrix's tiles.
struct UpdTile {
  int32_t r, c, cend;  // first row and column (front-local), end of its columns
};
#ifdef __CUDACC__
#define GIPM_HD __host__ __device__
#else
#define GIPM_HD
#endif
GIPM_HD inline int64_t upd_tiles(int ncol, int nrow, int k1, int clim, int with_u, int TS) {
  const int c0 = k1 < ncol ? k1 : ncol, lim = clim < ncol ? clim : ncol;
  const int64_t A = (ncol + nrow - c0 + TS - 1) / TS, J = lim > c0 ? (lim - c0 + TS - 1) / TS : 0;
  const int64_t B = with_u ? (nrow + TS - 1) / TS : 0;
  return J * A - J * (J - 1) / 2 + B * (B + 1) / 2;
}
GIPM_HD inline UpdTile upd_decode(int ncol, int nrow, int k1, int clim, int with_u, int TS, int t) {
  const int c0 = k1 < ncol ? k1 : ncol, lim = clim < ncol ? clim : ncol;
  const int A = (ncol + nrow - c0 + TS - 1) / TS, J = lim > c0 ? (lim - c0 + TS - 1) / TS : 0;
  const int64_t np = (int64_t)J * A - (int64_t)J * (J - 1) / 2;
  if (t < np) {  // column tile j holds A - j row tiles: first of j is j A - j (j - 1) / 2
    const double h = A + 0.5;
    double disc = h * h - 2.0 * t;
    int j = (int)(h - sqrt(disc > 0.0 ? disc : 0.0));
    if (j > J - 1) j = J - 1;
    if (j < 0) j = 0;
    while (j > 0 && (int64_t)j * A - (int64_t)j * (j - 1) / 2 > t) j--;
    while (j + 1 < J && (int64_t)(j + 1) * A - (int64_t)(j + 1) * j / 2 <= t) j++;
    const int i = j + (int)(t - ((int64_t)j * A - (int64_t)j * (j - 1) / 2));
    return UpdTile{c0 + TS * i, c0 + TS * j, lim};
  }
  const int u = (int)(t - np);  // row tile i of the lower triangle holds i + 1 tiles
  int i = (int)((sqrt(8.0 * u + 1.0) - 1.0) * 0.5);
  while (i > 0 && (int64_t)i * (i + 1) / 2 > u) i--;
  while ((int64_t)(i + 1) * (i + 2) / 2 <= u) i++;
  const int j = u - (int)((int64_t)i * (i + 1) / 2);
  (void)with_u;
  return UpdTile{ncol + TS * i, ncol + TS * j, ncol + nrow};
}
struct LevelPlan {
  int32_t front_b = 0, front_e = 0;  // into the level-ordered front list
  int32_t build_b = 0, build_e = 0;  // front-assembly tiles
  int64_t build_k = -1;              // where the level's ranges start in Plan::build_k (-1: K by its own launch)
  int64_t k_b = 0, k_e = 0;          // K entries of this level's fronts
  int32_t gath_b = 0, gath_e = 0;    // solve gather tasks
  int32_t rg_b = 0, rg_e = 0;        // backward-solve tasks on the rows below the block
  int32_t sdiag_b = 0, sdiag_e = 0;  // solve diagonal-block tasks, by step: see solve_steps
  std::vector<StepRange> steps;      // factor steps (block columns)
  bool ahead64 = false;              // FP64: look-ahead (see factor_steps64)
  std::vector<int32_t> sstep_b;      // solve steps: [sstep_b[j], sstep_b[j+1]) in stasks
  std::vector<int32_t> sgemv_b;      // solve update tasks per step
  int32_t max_ncol = 0;
};

// Persistent solve over blocks of `B` columns and chunks of `B` rows: inverses of
// the diagonal blocks (slot s: jb rows of jb rounded up to 16 bytes at
// dinv_off[s]; the slots of a front are consecutive from first_slot[front]) and
// the task list, forward tasks first. Flags (32-bit words): [0, 32) tickets, then
// per slot "partial sums done", per front "update-vector chunks of its children
// done", "column blocks done".
constexpr int kSolveB32 = 128, kSolveB64 = 64;  // block widths, FP32 and FP64
// A front that one task solves in each sweep: its chunks of rows below hold less work
// than a task costs.
constexpr int kNarrowCols = 32, kNarrowRows = 512;
inline bool narrow_front(const FrontInfo &F) { return F.ncol <= kNarrowCols && F.nrow <= kNarrowRows; }
struct SolvePlan {
  int B = 0;
  std::vector<Task> inv;                  // (front, first column, slot)
  std::vector<int32_t> first_slot;        // per front: slot of block 0
  std::vector<int64_t> dinv_off;
  int64_t dinv_entries = 0;
  std::vector<Task> tasks;                // (front, a, b, kind)
  int32_t fwd_tasks = 0;
  std::vector<int64_t> pbase;             // per front: first partial-sum row (B values each)
  std::vector<SolveRec> recs;             // per task: the task and its front's data
  std::vector<int32_t> kid_chunks;        // per front: below-front chunks of all its children
  std::vector<int32_t> parent_blocks;     // per front: diagonal blocks of its parent (0 at roots)
  int64_t part_entries = 0;               // values of partial sums
  int64_t flag_words = 0;
  int64_t words = 0;                      // 8-byte words of published entries, y or x (FP64: two per value)
};

// Numeric plan: everything the kernels need, built on the host by analysis.
struct Plan {
  static constexpr int kSuper32 = 256;  // columns per super-step of the FP32 FMA-pipe factor
  int nb = 64;                       // factor block width
  int nbs = 64;                      // solve block width
  std::vector<FrontInfo> fronts;     // by supernode index
  std::vector<int32_t> sched;        // schedule level of each supernode (parent = child + 1)
  std::vector<int32_t> level_fronts; // supernodes sorted by (schedule level, index)
  std::vector<int32_t> children;     // child lists (ascending), ranges in FrontInfo
  std::vector<int32_t> inv;          // child -> parent-front inverse maps
  std::vector<int32_t> relpos;       // child row -> position in parent's front (by sri offset)
  std::vector<LevelPlan> levels;
  std::vector<Task> build_tasks, potrf_tasks, trsm_ents, upd_ents;
  std::vector<Task> gath_tasks, sdiag_tasks, sgemv_tasks, rgemv_tasks;
  std::vector<int64_t> toff;         // per front: offset of its solve update vector (length nrow)
  int64_t t_entries = 0;
  SolvePlan s32, s64;  // persistent solves (s64: when the storage is sized for FP64)
  // K entries in level-major order
  std::vector<int64_t> k_slot;   // element offset of L(i, j) in the factor storage
  std::vector<int64_t> build_k;  // per assembly tile of a level with fuse_k: K entries of its rows, [first, end)
  std::vector<int64_t> k_poff;   // products [k_poff[q], k_poff[q+1])
  std::vector<int32_t> k_pa, k_pb;  // CSR positions of the two J factors of each product
  std::vector<int64_t> k_w;      // W value index or -1
  std::vector<int32_t> k_diag;   // original variable index for a diagonal entry, else -1
  std::vector<int64_t> k_orig;   // original lower-CSC entry index (export order)
  int64_t l_entries = 0, u_entries = 0;
  int32_t max_front = 0, max_ncol = 0;
};

// Problem description kept by the context (host copies).
struct Problem {
  int32_t n = 0, m = 0;
  std::vector<int64_t> jp;
  std::vector<int32_t> ji;
  std::vector<int32_t> jrow;         // row of each CSR position
  std::vector<int64_t> jtp;          // CSC of J: column pointers
  std::vector<int32_t> jtpos;        // CSR position of each CSC entry
  std::vector<int64_t> wp;
  std::vector<int32_t> wi;
  std::vector<double> l, u;
  int32_t nl = 0, nu = 0;
  int64_t mt = 0;
  std::vector<int32_t> lidx, uidx;   // variables with a finite lower/upper bound
  std::vector<int32_t> lpos, upos;   // per variable: row of its bound in g (or -1)
};

void analyze_symbolic(const Problem &P, const int32_t *perm, Symbolic &S);
void build_plan(const Problem &P, const Symbolic &S, Plan &plan, int nb, int nbs);
void validate_plan(const Problem &P, const Symbolic &S, const Plan &plan);
// Task lists of a persistent solve with blocks of B columns (128 FP32, 64 FP64).
void build_fused_solve(const Plan &plan, int B, SolvePlan &sp);

}  // namespace gipm
