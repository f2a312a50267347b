// Host launchers of the device kernels (one stream, no synchronisation inside).
#pragma once

#include "dev.cuh"
#include "side_stream.h"

namespace gipm {

// K = W + J^T diag(D_J) J + diag(D_bounds) + delta_p I into the compact FP64
// array kval (level-major order of the plan).
void launch_assemble(const DevPlan &dp, const double *jv, const double *D, const double *wv,
                     double delta_p, double *kval, cudaStream_t st);

struct CudaApi {
  using Stream = cudaStream_t;
  using Event = cudaEvent_t;
  static bool current_device(int &dev) { return cudaGetDevice(&dev) == cudaSuccess; }
  static bool create(bool high, Stream &s) {
    int lo = 0, hi = 0;
    return cudaDeviceGetStreamPriorityRange(&lo, &hi) == cudaSuccess &&
           cudaStreamCreateWithPriority(&s, cudaStreamNonBlocking, high ? hi : lo) == cudaSuccess;
  }
  static bool create(Event &e) { return cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess; }
  static void destroy(Stream s) { cudaStreamDestroy(s); }
  static void destroy(Event e) { cudaEventDestroy(e); }
};
using SideStream = SideStreamOf<CudaApi>;

// Multifrontal factorisation of all levels with SIMT FMA kernels. status must
// be initialised by the caller (ST_FAIL_COL = INT32_MAX, ST_PERTURBED = 0). chain: the
// highest-priority stream of the FP64 factor's look-ahead (one per context; see factor_steps64).
template <typename T>
void launch_factor_simt(const DevPlan &dp, const Plan &plan, const double *kval, T *L, T *U,
                        int32_t *status, bool perturb, const SideStream &chain, cudaStream_t st);

// Pieces of a level of the factorisation, shared with the tensor-core path:
// front assembly (+ K entries), diagonal-block Cholesky (64 wide) and the
// triangular solve of the rows below of one block step.
template <typename T>
void launch_build_level(const DevPlan &dp, const LevelPlan &LP, const double *kval, T *L, T *U,
                        cudaStream_t st);
template <typename T>
void launch_potrf(const DevPlan &dp, const StepRange &S, T *L, int32_t *status, bool perturb,
                  cudaStream_t st);
template <typename T>
void launch_trsm(const DevPlan &dp, const StepRange &S, T *L, cudaStream_t st);

// Triangular solves with the factor: y (final numbering, length n) is
// overwritten by L^{-T} L^{-1} y (L^{-T} S L^{-1} y for a signed factor,
// dp.sgn). t: update-vector scratch (plan.t_entries).
template <typename T, typename V>
void launch_solve(const DevPlan &dp, const Plan &plan, const T *L, V *y, V *t, cudaStream_t st);

// y <- S y with the pivot signs of a signed factor (no-op without dp.sgn).
template <typename V>
void launch_sign(const DevPlan &dp, V *y, cudaStream_t st);

// Loads the level-solve kernels (FP64 and FP32) so that a later first launch
// commits no device memory (lazy module loading); used by the allocation-free solve.
cudaError_t preload_level_solve();

// The vectors of a persistent solve: right-hand sides, forward results, solutions,
// update vectors, partial sums, flags and published entries of up to kSolveRhs right-hand sides,
// each kind `sd` apart from one to the next (t in values of T). The entries wy, wx handed from
// block to block carry the tag of their launch: zeroed before the first one, and no two launches
// between have the same tag `epoch` (not 0). A solve is bound by its
// chain of diagonal blocks, so right-hand sides side by side cost little until they
// fill the chip: 56^3 TF32x3, eight right-hand sides with PCG: 27.4 ms one by one,
// 16.6 in fours, 15.2 as eight.
constexpr int kSolveRhs = 8;
struct SolveStride {
  int64_t n = 0, t = 0, part = 0, flags = 0, words = 0;
};
template <typename T> struct SolveBufs {
  T *a = nullptr, *b = nullptr, *x = nullptr, *t = nullptr, *part = nullptr;
  unsigned *flags = nullptr;
  uint2 *wy = nullptr, *wx = nullptr;
  unsigned epoch = 0;
  SolveStride sd;
};

// Persistent solve: inverses of the diagonal blocks (after each factorisation
// that does not write them itself), then x = L^{-T} L^{-1} a in one launch, with b
// the forward result and t the update vectors. fwd/bwd select the sweeps: forward
// only maps a to b = L^{-1} a; backward only maps b to x = L^{-T} b. part:
// part_entries values of scratch; flags: flag_words words (zeroed by the launch),
// both from the solve plan of the storage type. A wait that runs out sets
// status[ST_SOLVE_TIMEOUT] and the launch drains. test_spins (0: the default of
// seconds) bounds each wait; test_withhold >= 0 abandons the task of that ticket
// (tests of the bounded wait).
void launch_dinv(const DevPlan &dp, const Plan &plan, const float *L, float *Dinv, cudaStream_t st);
void launch_dinv(const DevPlan &dp, const Plan &plan, const double *L, double *Dinv, cudaStream_t st);
template <typename T>
void launch_psolve(const DevPlan &dp, const Plan &plan, const T *L, const T *Dinv, const SolveBufs<T> &v,
                   int nrhs, int32_t *status, bool fwd, bool bwd, cudaStream_t st, unsigned test_spins = 0,
                   int test_withhold = -1);

// Sampled entries of L (final numbering).
template <typename T>
void launch_factor_entries(const DevPlan &dp, const T *L, const int32_t *col2s, int64_t count,
                           const int32_t *rows, const int32_t *cols, double *out,
                           cudaStream_t st);

}  // namespace gipm
