// Persistent supernodal triangular solves (FP32 storage: TF32/TF32x3/BF16/FP32
// factors, 128-wide blocks; FP64 storage: 64-wide blocks, so a lane reads 16
// bytes of a row either way and a tile holds as many loads in flight).
//
// After each factorisation one launch inverts every diagonal block of L (explicit
// inverse, rows padded to 16 bytes). A solve is then ONE launch of a persistent kernel
// whose CTAs take the tasks of the plan in order from a global ticket counter (forward
// sweep leaves -> root, backward sweep root -> leaves), for one right-hand side or for
// up to kSolveRhs side by side. Instead of grid barriers between phases, each task
// waits only for the results it reads. Along the diagonal blocks of a front, whose
// chain is the time of a solve, the entries of y and x carry their own flag: each
// 32-bit half is stored with the launch's tag in one 8-byte word, and a
// consumer reads the words until all of them have the tag, so a block costs one
// trip through L2 and no fence (a counter behind a release, polled and
// acquired before the values are read, takes three: 2.6 us a block of the root
// against 1.8; a whole solve, TF32x3: 834 -> 666 us at 48^3, 1845 -> 1548 at
// 64^3). The words lie in the order of the columns, each front on lines of its own. A
// diagonal block of the forward sweep subtracts L_ij y_j as each y_j of its front
// appears (a wavefront down the front's blocks), rows below a front take every
// y_j and then count towards the front's update vector, which the parent's gathers
// wait for; the backward sweep mirrors this with partial sums over the rows below
// a front (waiting for the parent front) and x_i published block by block. A task
// waits only for earlier tasks, so the schedule cannot deadlock, and every wait is
// bounded: on expiry the status word is set and the whole launch drains.
// Three vectors keep reads disjoint from writes: a (right-hand side), b
// (forward result) and x (solution); t holds the fronts' update vectors.
// Vectors written inside the launch are read through L2 (ld.global.cg), and
// the loads of L for a block are issued before its wait.
#include <algorithm>
#include <stdexcept>
#include <string>

#include "launch.h"

namespace gipm {

namespace {

constexpr int kT = 256;                     // threads per CTA
constexpr unsigned kBarrierSpins = 1u << 24;  // polls of >= 0.3 us each: seconds before giving up

// Shapes of a solve over values of type T: blocks of B columns and chunks of B
// rows, a warp takes RW rows and a lane the VW columns of one 16-byte load.
template <typename T> struct Ps {
  static constexpr int VW = 16 / (int)sizeof(T), B = 32 * VW, RW = B / (kT / 32);
};
static_assert(Ps<float>::B == kSolveB32 && Ps<double>::B == kSolveB64, "block widths of the plan");
template <typename T> struct alignas(16) Vec {
  T v[Ps<T>::VW];
};
template <typename T> __device__ __forceinline__ Vec<T> vzero() {
  Vec<T> z;
#pragma unroll
  for (int h = 0; h < Ps<T>::VW; h++) z.v[h] = T(0);
  return z;
}
// 16 bytes as one load or store (a copy of the struct is split into its members).
__device__ __forceinline__ Vec<float> from16(float4 f) { return Vec<float>{{f.x, f.y, f.z, f.w}}; }
__device__ __forceinline__ Vec<double> from16(double2 f) { return Vec<double>{{f.x, f.y}}; }
__device__ __forceinline__ Vec<float> ldg16(const float *p) { return from16(__ldg(reinterpret_cast<const float4 *>(p))); }
__device__ __forceinline__ Vec<double> ldg16(const double *p) { return from16(__ldg(reinterpret_cast<const double2 *>(p))); }
__device__ __forceinline__ Vec<float> ld16(const float *p) { return from16(*reinterpret_cast<const float4 *>(p)); }
__device__ __forceinline__ Vec<double> ld16(const double *p) { return from16(*reinterpret_cast<const double2 *>(p)); }
__device__ __forceinline__ void st16(float *p, const Vec<float> &v) {
  *reinterpret_cast<float4 *>(p) = make_float4(v.v[0], v.v[1], v.v[2], v.v[3]);
}
__device__ __forceinline__ void st16(double *p, const Vec<double> &v) {
  *reinterpret_cast<double2 *>(p) = make_double2(v.v[0], v.v[1]);
}
// acc + <a, b>, the last component first
template <typename T>
__device__ __forceinline__ T vdot(const Vec<T> &a, const Vec<T> &b, T acc) {
#pragma unroll
  for (int h = Ps<T>::VW - 1; h >= 0; h--) acc = fma(a.v[h], b.v[h], acc);
  return acc;
}
template <typename T> __device__ __forceinline__ Vec<T> vfma(const Vec<T> &l, T y, Vec<T> acc) {
#pragma unroll
  for (int h = 0; h < Ps<T>::VW; h++) acc.v[h] = fma(l.v[h], y, acc.v[h]);
  return acc;
}

void ck(cudaError_t e, const char *what) {
  if (e != cudaSuccess) throw std::runtime_error(std::string(what) + ": " + cudaGetErrorString(e));
}

// Inverse of one diagonal block (jb <= 128): column c of X = L_jj^{-1} by
// forward substitution in thread c; stored as jb rows of ldi = round_up(jb, 4)
// floats with zeros above the diagonal and in the padding.
__global__ void __launch_bounds__(128) dinv_kernel(DevPlan dp, const float *__restrict__ L,
                                                   float *__restrict__ Dinv) {
  constexpr int LS = 129, kB = Ps<float>::B;
  const Task tk = dp.s32.inv[blockIdx.x];
  const FrontInfo F = dp.fronts[tk.front];
  const int j = tk.a, jb = min(kB, F.ncol - j), ldi = (jb + 3) & ~3, tid = threadIdx.x;
  extern __shared__ float smd[];
  float *A = smd;             // [128][129]
  float *X = smd + 128 * LS;  // [128][129]
  const float *g = L + F.loff + (int64_t)j * F.ld + j;
  for (int e = tid; e < jb * jb; e += 128) {
    const int r = e / jb, c = e % jb;
    A[r * LS + c] = (c <= r) ? g[(int64_t)r * F.ld + c] : 0.f;
  }
  __syncthreads();
  if (tid < jb) {
    const int c = tid;
    for (int i = c; i < jb; i++) {
      float s = (i == c) ? 1.f : 0.f;
      for (int m = c; m < i; m++) s = fmaf(-A[i * LS + m], X[m * LS + c], s);
      X[i * LS + c] = s / A[i * LS + i];
    }
  }
  __syncthreads();
  float *out = Dinv + dp.s32.dinv_off[tk.b];
  for (int e = tid; e < jb * ldi; e += 128) {
    const int r = e / ldi, c = e % ldi;
    out[e] = (c <= r && c < jb) ? X[r * LS + c] : 0.f;
  }
}

// FP64: inverse of one diagonal block (jb <= 64), right-looking in panels of eight rows:
// a thread per column finishes the panel's rows, then every row below takes their
// multiples, two warps per quarter SM (an FP64 instruction occupies the quarter's unit
// for 64 cycles whatever its active lanes). A 64-column block is 288 warp instructions on
// the panels' warp and 336 on each quarter after them; with a thread per column down all
// the rows it was 2080 on one, which a 64-column block took 70 us for wherever it stood,
// and the last one of a factor waits for nothing else (augmented system of 1716 + 1716
// unknowns: 78 -> 36 us).
constexpr int kDinvThreads = 256;
__global__ void __launch_bounds__(kDinvThreads) dinv64_kernel(DevPlan dp, const double *__restrict__ L,
                                                              double *__restrict__ Dinv) {
  constexpr int kB = Ps<double>::B, LS = kB + 1, Q = 4;
  const Task tk = dp.s64.inv[blockIdx.x];
  const FrontInfo F = dp.fronts[tk.front];
  const int j = tk.a, jb = min(kB, F.ncol - j), ldi = (jb + 1) & ~1, rows = (jb + 7) & ~7, tid = threadIdx.x;
  extern __shared__ __align__(16) double smd64[];
  double *A = smd64, *X = smd64 + kB * LS;  // L[i][m] at A[m LS + i] (zero past jb), X[i][c] at X[i kB + c]
  __shared__ double rd[kB];
  const double *g = L + F.loff + (int64_t)j * F.ld + j;
  for (int e = tid; e < rows * kB; e += kDinvThreads) {
    const int i = e / kB, c = e % kB;
    const double v = (i < jb && c <= i) ? g[(int64_t)i * F.ld + c] : 0.0;
    A[c * LS + i] = v;
    X[e] = i == c ? 1.0 : 0.0;
    if (i == c) rd[i] = i < jb ? 1.0 / v : 0.0;
  }
  __syncthreads();
  for (int r0 = 0; r0 < rows; r0 += 8) {
    const int nc = r0 + 8;  // columns that are not zero in these rows
    if (tid < ((nc + 31) & ~31)) {
      double x[8];
#pragma unroll
      for (int i = 0; i < 8; i++) x[i] = X[(r0 + i) * kB + tid];
#pragma unroll
      for (int m = 0; m < 8; m++) {
        x[m] *= rd[r0 + m];
#pragma unroll
        for (int i = m + 1; i < 8; i++) x[i] = fma(-x[m], A[(r0 + m) * LS + r0 + i], x[i]);
      }
#pragma unroll
      for (int i = 0; i < 8; i++) X[(r0 + i) * kB + tid] = x[i];
    }
    __syncthreads();
    const int nout = (rows - nc) * nc;
    if (tid < nout) {  // (at most 32 x 32 outputs: Q per thread)
      double s[Q];
      int at[Q], row[Q], col[Q];
#pragma unroll
      for (int q = 0; q < Q; q++) {
        const int e = min(tid + kDinvThreads * q, nout - 1), i = e / nc;
        row[q] = nc + i;
        col[q] = e - nc * i;
        at[q] = row[q] * kB + col[q];
        s[q] = X[at[q]];
      }
      const int n = (nout - (tid & ~31) + kDinvThreads - 1) / kDinvThreads;  // of this warp
#pragma unroll
      for (int m = 0; m < 8; m++)
#pragma unroll
        for (int q = 0; q < Q; q++)
          if (q < n) s[q] = fma(-X[(r0 + m) * kB + col[q]], A[(r0 + m) * LS + row[q]], s[q]);
#pragma unroll
      for (int q = 0; q < Q; q++)
        if (tid + kDinvThreads * q < nout) X[at[q]] = s[q];
    }
    __syncthreads();
  }
  double *out = Dinv + dp.s64.dinv_off[tk.b];
  for (int e = tid; e < jb * (ldi / 2); e += kDinvThreads) {
    const int i = e / (ldi / 2), c = 2 * (e % (ldi / 2));
    st16(out + i * ldi + c, Vec<double>{{c <= i ? X[i * kB + c] : 0.0, c + 1 <= i ? X[i * kB + c + 1] : 0.0}});
  }
}

template <typename T> struct PsArgs {
  DevPlan dp;
  DevSolve sv;
  const T *L, *Dinv;
  T *a, *b, *x, *t, *part;
  int32_t q0, q1;    // tasks [q0, q1) of the plan
  unsigned *ticket;  // ticket counter, and the solve plan's flag words, zeroed before the launch
  unsigned *flags;
  uint2 *ly, *lx;    // published entries of y and x, one word each (FP64: two)
  unsigned epoch;    // tag of this launch's entries
  int32_t *status;   // ST_SOLVE_TIMEOUT
  unsigned spins;    // polls before a wait gives up
  int32_t withhold;  // test of the bounded wait: the task of this ticket is abandoned (-1: none)
  int32_t nslot, nfr;
  int32_t fwd_here;  // the forward sweep runs in this launch: backward blocks wait for their y
  int32_t nrhs;      // right-hand sides; ticket k is task k / nrhs of right-hand side k % nrhs
  SolveStride sd;    // from one right-hand side's vectors, flags and words to the next
};

// The vectors, flags and words of right-hand side k.
template <typename T> __device__ __forceinline__ void shift_rhs(PsArgs<T> &A, int k) {
  A.a += k * A.sd.n;
  A.b += k * A.sd.n;
  A.x += k * A.sd.n;
  A.t += k * A.sd.t;
  A.part += k * A.sd.part;
  A.flags += k * A.sd.flags;
  A.ly += k * A.sd.words;
  A.lx += k * A.sd.words;
}

constexpr int kMaxKids = 32;  // children staged in shared memory for the gathers
constexpr long long kCopySpinCycles = 2000000000ll;  // bounded wait on a staging copy (~1 s)

template <typename T> __device__ __forceinline__ T ldcg(const T *p) { return __ldcg(p); }

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Flag words (see SolvePlan): tickets, then per slot partial sums done, per front
// update-vector chunks and column blocks done.
template <typename T>
__device__ __forceinline__ unsigned *f_part(const PsArgs<T> &A, int slot) {
  return A.flags + 32 + slot;
}
// per front: chunks of rows below its children that are done (the children's
// update vectors are complete once it reaches the record's kid_chunks)
template <typename T>
__device__ __forceinline__ unsigned *f_tvec(const PsArgs<T> &A, int front) {
  return A.flags + 32 + A.nslot + front;
}
template <typename T>
__device__ __forceinline__ unsigned *f_front(const PsArgs<T> &A, int front) {
  return A.flags + 32 + A.nslot + A.nfr + front;
}

constexpr int kLbStride = 72;  // FP64, row stride of PsShared::lb: two rows of a quarter warp's reads side by side

// Shared scratch of one CTA (dynamic shared memory).
template <typename T> struct PsShared {
  static constexpr int B = Ps<T>::B;
  T di[B * B];                  // staged inverse of a diagonal block (TMA bulk copy)
  alignas(16) T lb[sizeof(T) == 8 ? B * kLbStride : 2];  // FP64: its block of L, lower triangle
  alignas(16) T sv[B];          // values handed to the diagonal-block solve
  T xs[B];                      // solution entries of the rows below a front
  alignas(16) T ys[sizeof(T) == 8 ? kT / 32 : 1][B];  // FP64: a warp's copy of the running y block
  alignas(16) T red4[kT / 32][B];  // per-row-group column sums
  unsigned long long mbar;      // completion of the staging copy
  uint32_t parity;              // its phase
  int tk;                       // this CTA's current task
  int rhs;                      // and its right-hand side
  int ok;                       // outcome of the last wait
  int nkids;                    // children of the task's front staged below
  int64_t kid_inv[kMaxKids];    // their child -> front map offsets
  int64_t kid_toff[kMaxKids];   // their update-vector offsets
  alignas(16) SolveRec rec[2];  // the running task's record and the next one's
};

// Start the copies of a diagonal block's inverse into S.di (thread 0: a bulk copy) and, FP64, of
// its block of L (column j on, zero above the diagonal) into S.lb; wait_dinv ends both.
template <typename T>
__device__ __forceinline__ void stage_dinv(const PsArgs<T> &A, PsShared<T> &S, const FrontInfo &F, int j, int slot) {
  constexpr int VW = Ps<T>::VW, B = Ps<T>::B;
  const int jb = min(B, F.ncol - j);
  if constexpr (sizeof(T) == 8) {
    const T *g = A.L + F.loff + (int64_t)j * F.ld + j;
    for (int e = threadIdx.x; e < jb * (B / 2); e += kT) {
      const int r = e / (B / 2), c = 2 * (e % (B / 2));
      T *dst = S.lb + r * kLbStride + c;
      if (c <= r)  // (the factor holds a zero beside an even row's diagonal entry)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(g + (int64_t)r * F.ld + c)
                     : "memory");
      else if (c < (r | 7))  // up to the end of the diagonal's group of eight
        st16(dst, vzero<T>());
    }
  }
  if (threadIdx.x != 0) return;
  const uint32_t bytes = (uint32_t)(jb * ((jb + VW - 1) & ~(VW - 1)) * (int)sizeof(T));
  const T *src = A.Dinv + A.sv.dinv_off[slot];
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&S.mbar)),
               "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(S.di)),
      "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(&S.mbar))
      : "memory");
}

// All threads: bounded wait for the staging copy; false after a timeout (the
// status word is set, and a second bounded wait lets the copy land first) or if
// ok_in was false in any thread.
template <typename T>
__device__ bool wait_dinv(const PsArgs<T> &A, PsShared<T> &S, bool ok_in) {
  const uint32_t par = S.parity;
  if constexpr (sizeof(T) == 8) asm volatile("cp.async.wait_all;" ::: "memory");  // (the barrier below shares it)
  auto try_wait = [&]() {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(&S.mbar)), "r"(par)
        : "memory");
    return done != 0;
  };
  bool ok = true;
  long long t0 = clock64();
  while (!try_wait()) {
    if (clock64() - t0 > kCopySpinCycles) {
      ok = false;
      atomicExch(A.status + ST_SOLVE_TIMEOUT, 1);
      t0 = clock64();
      while (!try_wait() && clock64() - t0 < kCopySpinCycles) {
      }
      break;
    }
  }
  ok = __syncthreads_and(ok && ok_in) != 0;  // one outcome for the whole CTA
  if (threadIdx.x == 0) S.parity = par ^ 1u;
  return ok;
}

// Words of published entries: value bits and the launch's tag in one 8-byte access
// (FP64: two words, low and high half), so a word with the tag holds its value.
__device__ __forceinline__ uint2 split_word(unsigned long long w) { return make_uint2((unsigned)w, (unsigned)(w >> 32)); }
__device__ __forceinline__ unsigned long long make_word(unsigned bits, unsigned tag) {
  return (unsigned long long)tag << 32 | bits;
}
__device__ __forceinline__ uint4 ld_words(const uint2 *p) {
  unsigned long long a, b;
  asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
  const uint2 u = split_word(a), v = split_word(b);
  return make_uint4(u.x, u.y, v.x, v.y);
}
__device__ __forceinline__ uint2 ld_word(const uint2 *p) {
  unsigned long long a;
  asm volatile("ld.volatile.global.u64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
  return split_word(a);
}
__device__ __forceinline__ void publish(uint2 *slot, int r, float v, unsigned tag) {
  asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(slot + r), "l"(make_word(__float_as_uint(v), tag)) : "memory");
}
__device__ __forceinline__ void publish(uint2 *slot, int r, double v, unsigned tag) {
  asm volatile("st.volatile.global.v2.u64 [%0], {%1, %2};" ::"l"(slot + 2 * r),
               "l"(make_word((unsigned)__double2loint(v), tag)), "l"(make_word((unsigned)__double2hiint(v), tag))
               : "memory");
}
__device__ __forceinline__ double word_double(unsigned lo, unsigned hi) { return __hiloint2double((int)hi, (int)lo); }
// The words of block j of a record's front.
template <typename T> __device__ __forceinline__ uint2 *block_words(uint2 *base, const SolveRec &R, int j) {
  return base + ((int64_t)R.word0 + Ps<T>::B * j) * (int)(sizeof(T) / 4);
}

// One warp: until load() holds in every lane (it reads the lane's words and tells
// whether they carry the tag), at most A.spins polls and only while no other wait
// of the launch has run out. The block next in a chain (critical) polls all its
// words; the others watch the block's first word, to leave L2 to the chain.
template <typename T, typename Load>
__device__ __forceinline__ bool wait_words(const PsArgs<T> &A, const uint2 *first, bool critical, Load load) {
  if (__all_sync(0xffffffffu, load())) return true;
  const int lane = threadIdx.x % 32;
  for (unsigned spins = 0;; spins++) {
    bool look = true;
    if (!critical) {
      unsigned seen = 0;
      if (lane == 0) seen = ld_word(first).y == A.epoch;
      look = __shfl_sync(0xffffffffu, seen, 0) != 0;
      if (!look) __nanosleep(64);
    }
    if (look && __all_sync(0xffffffffu, load())) return true;
    int stop = 0;
    if (lane == 0 && (spins & 63u) == 0) stop = *(volatile int32_t *)(A.status + ST_SOLVE_TIMEOUT) != 0;
    if (lane == 0 && spins >= A.spins) {
      atomicExch(A.status + ST_SOLVE_TIMEOUT, 1);
      stop = 1;
    }
    if (__shfl_sync(0xffffffffu, stop, 0)) return false;
  }
}

// Row sums of 16 consecutive rows per warp: p[k] = <row k, v> for the lane's
// columns; returns the full sum of row lane / 2 (each lane keeps half of its rows
// at every exchange).
__device__ __forceinline__ float rows_reduce(const float (&p)[16]) {
  const int lane = threadIdx.x % 32;
  float a[8], b[4], c[2], d;
  const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4, h1 = lane & 2;
#pragma unroll
  for (int k = 0; k < 8; k++) a[k] = (h4 ? p[k + 8] : p[k]) + __shfl_xor_sync(0xffffffffu, h4 ? p[k] : p[k + 8], 16);
#pragma unroll
  for (int k = 0; k < 4; k++) b[k] = (h3 ? a[k + 4] : a[k]) + __shfl_xor_sync(0xffffffffu, h3 ? a[k] : a[k + 4], 8);
#pragma unroll
  for (int k = 0; k < 2; k++) c[k] = (h2 ? b[k + 2] : b[k]) + __shfl_xor_sync(0xffffffffu, h2 ? b[k] : b[k + 2], 4);
  d = (h1 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, h1 ? c[0] : c[1], 2);
  return d + __shfl_xor_sync(0xffffffffu, d, 1);
}
// Entry r of a published block; false while its words lack the tag.
__device__ __forceinline__ bool read_word(const uint2 *slot, int r, unsigned tag, float &v) {
  const uint2 w = ld_word(slot + r);
  v = __uint_as_float(w.x);
  return w.y == tag;
}
__device__ __forceinline__ bool read_word(const uint2 *slot, int r, unsigned tag, double &v) {
  const uint4 w = ld_words(slot + 2 * r);
  v = word_double(w.x, w.z);
  return w.y == tag && w.w == tag;
}

// Sum over the four neighbouring lanes (valid in all of them).
template <typename T> __device__ __forceinline__ T quad_sum(T v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// Product of a B x B tile's rows (row stride ld) with a block of the forward
// result, accumulated over tiles. The loads of a tile are issued by load(),
// before the block's words are waited for (wait_y, per warp).
//  FP32: warp w takes rows 16w .. 16w + 15, lane: columns 4 lane ..; the row sums
//  are reduced across the warp once, after the last tile.
//  FP64: an addition costs as much as a multiply-add (64 cycles per warp on a
//  quarter SM), so the cross-lane reduction is kept short: four threads share a
//  row (thread h: columns 8m + 2h, 8m + 2h + 1) and y comes from shared memory.
template <typename T> struct FwdTile;

template <> struct FwdTile<float> {
  static constexpr int RW = Ps<float>::RW;
  float4 l[RW];
  float acc[RW];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < RW; k++) acc[k] = 0.f;
  }
  // FULL: the block has all B columns
  template <bool FULL>
  __device__ __forceinline__ void load(const float *P, int64_t ld, int nr, int nc) {
    const int c = 4 * (threadIdx.x % 32), rw = RW * (threadIdx.x / 32);
    const float *row = P + (int64_t)rw * ld + c;
#pragma unroll
    for (int k = 0; k < RW; k++)
      l[k] = ((FULL || c < nc) && rw + k < nr) ? __ldg(reinterpret_cast<const float4 *>(row + (int64_t)k * ld))
                                               : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // y: block of nc values; columns past nc (padding of a last block) never enter
  uint4 w0, w1;
  __device__ __forceinline__ bool wait_y(const PsArgs<float> &A, const uint2 *words, int nc, bool critical) {
    const int c = 4 * (threadIdx.x % 32);
    return wait_words(A, words, critical, [&]() {
      if (c >= nc) return true;
      w0 = ld_words(words + c);
      w1 = ld_words(words + c + 2);
      return w0.y == A.epoch && (c + 1 >= nc || w0.w == A.epoch) && (c + 2 >= nc || w1.y == A.epoch) &&
             (c + 3 >= nc || w1.w == A.epoch);
    });
  }
  template <bool FULL>
  __device__ __forceinline__ void mul(PsShared<float> &, int nc) {
    const int c = 4 * (threadIdx.x % 32);
    const float4 y4 = make_float4(FULL || c < nc ? __uint_as_float(w0.x) : 0.f,
                                  FULL || c + 1 < nc ? __uint_as_float(w0.z) : 0.f,
                                  FULL || c + 2 < nc ? __uint_as_float(w1.x) : 0.f,
                                  FULL || c + 3 < nc ? __uint_as_float(w1.z) : 0.f);
#pragma unroll
    for (int k = 0; k < RW; k++) {
      float4 v = l[k];
      if (!FULL) {
        if (c + 1 >= nc) v.y = 0.f;
        if (c + 2 >= nc) v.z = 0.f;
        if (c + 3 >= nc) v.w = 0.f;
      }
      acc[k] = fmaf(v.x, y4.x, fmaf(v.y, y4.y, fmaf(v.z, y4.z, fmaf(v.w, y4.w, acc[k]))));
    }
  }
  // f(row, sum) once per row
  template <typename F> __device__ __forceinline__ void finish(int nr, F f) {
    const float s = rows_reduce(acc);
    const int lane = threadIdx.x % 32, r = RW * (threadIdx.x / 32) + lane / 2;
    if (lane % 2 == 0 && r < nr) f(r, s);
  }
};
template <> struct FwdTile<double> {
  static constexpr int NL = 8;
  Vec<double> l[NL];
  double acc;
  __device__ __forceinline__ void clear() { acc = 0.0; }
  template <bool FULL>
  __device__ __forceinline__ void load(const double *P, int64_t ld, int nr, int nc) {
    const int r = threadIdx.x / 4, c = 2 * (threadIdx.x % 4);
    const double *row = P + (int64_t)r * ld + c;
#pragma unroll
    for (int m = 0; m < NL; m++)
      l[m] = (r < nr && (FULL || 8 * m + c < nc)) ? ldg16(row + 8 * m) : vzero<double>();
  }
  uint4 w0, w1;  // the lane's two entries of y
  __device__ __forceinline__ bool wait_y(const PsArgs<double> &A, const uint2 *words, int nc, bool critical) {
    const int v = 2 * (threadIdx.x % 32);
    return wait_words(A, words, critical, [&]() {
      if (v >= nc) return true;
      w0 = ld_words(words + 2 * v);
      w1 = ld_words(words + 2 * v + 2);
      return w0.y == A.epoch && w0.w == A.epoch && (v + 1 >= nc || (w1.y == A.epoch && w1.w == A.epoch));
    });
  }
  template <bool FULL>
  __device__ __forceinline__ void mul(PsShared<double> &S, int nc) {
    const int v = 2 * (threadIdx.x % 32);
    double *ys = S.ys[threadIdx.x / 32];
    __syncwarp();  // the previous block has been read
    st16(ys + v, Vec<double>{{FULL || v < nc ? word_double(w0.x, w0.z) : 0.0,
                              FULL || v + 1 < nc ? word_double(w1.x, w1.z) : 0.0}});
    __syncwarp();
    const int c = 2 * (threadIdx.x % 4);
#pragma unroll
    for (int m = 0; m < NL; m++) {
      Vec<double> x = l[m];
      if (!FULL && 8 * m + c + 1 >= nc) x.v[1] = 0.0;
      acc = vdot(x, ld16(ys + 8 * m + c), acc);
    }
  }
  template <typename F> __device__ __forceinline__ void finish(int nr, F f) {
    const double s = quad_sum(acc);
    const int r = threadIdx.x / 4;
    if (threadIdx.x % 4 == 0 && r < nr) f(r, s);
  }
};

// y = b[first + j + r] = sum_c Dinv[r][c] v[c]  (Dinv staged in S.di, v = S.sv
// zero past jb), published in the slot's words and kept at `keep` if given; a warp's rows
// stop at their diagonal.
// FP32: warp w takes rows 16w .. 16w + 15
__device__ void diag_fwd(const PsArgs<float> &A, PsShared<float> &S, const FrontInfo &F, int j, uint2 *words,
                         float *keep = nullptr) {
  constexpr int B = Ps<float>::B, RW = Ps<float>::RW;
  const int jb = min(B, F.ncol - j), ldi = (jb + 3) & ~3;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, c = 4 * lane, rw = RW * warp;
  if (rw >= jb) return;  // whole warp idle (uniform per warp)
  const float4 v4 = *reinterpret_cast<const float4 *>(S.sv + c);
  float p[RW];
#pragma unroll
  for (int k = 0; k < RW; k++) {
    p[k] = 0.f;
    if (c <= rw + k && rw + k < jb) {  // (zero above the diagonal)
      const float4 d = *reinterpret_cast<const float4 *>(S.di + (rw + k) * ldi + c);
      p[k] = d.x * v4.x + d.y * v4.y + d.z * v4.z + d.w * v4.w;
    }
  }
  const float s = rows_reduce(p);
  const int r = rw + lane / 2;
  if (lane % 2 == 0 && r < jb) {
    publish(words, r, s, A.epoch);
    A.b[F.first + j + r] = s;
    if (keep) keep[r] = s;
  }
}
// Row (forward) or column (backward) of a diagonal block for this quad of lanes, eight a warp.
// Warps w and w + 4 share a quarter SM's FP64 unit: theirs are paired so that the triangle gives
// each quarter the same work.
__device__ __forceinline__ int quad_row() {
  const int w = threadIdx.x / 32;
  return 8 * (w < 4 ? w : 11 - w) + threadIdx.x % 32 / 4;
}
// FP64: four threads per row. A product with the inverse alone leaves a residual of |L| |L^-1|
// |v| u where substitution leaves |L| |y| u (a thousand times as much for a block with entries of
// either sign and condition 1e6), so its result is corrected once: y += Dinv (v - L y). That
// is three triangular products a block on the FP64 unit instead of one (a solve at 40^3 takes
// 1675 us, 1195 with the product alone; 2632 and 1915 at 48^3); a chain of 64 exchanges and
// multiply-adds, as substitution has, would be longer still.
__device__ void diag_fwd(const PsArgs<double> &A, PsShared<double> &S, const FrontInfo &F, int j, uint2 *words,
                         double *keep = nullptr) {
  constexpr int B = Ps<double>::B;
  const int jb = min(B, F.ncol - j), ldi = (jb + 1) & ~1, r = quad_row(), h = threadIdx.x % 4, c = 2 * h;
  const int last = 8 * (r / 8) < jb ? r / 8 : -1;  // column groups of this warp's rows (uniform per warp)
  double *y0 = S.red4[0], *rs = S.red4[1], s = 0.0;
  auto product = [&](const double *row, int end, const double *v) {  // both triangles are zero past r
    double a = 0.0;
#pragma unroll 4
    for (int m = 0; m <= last; m++)
      if (r < jb && 8 * m + c < end) a = vdot(ld16(row + 8 * m + c), ld16(v + 8 * m + c), a);
    return quad_sum(a);
  };
  if (last >= 0) {
    s = product(S.di + r * ldi, ldi, S.sv);
    if (h == 0) y0[r] = s;
  }
  __syncthreads();
  if (last >= 0) {
    const double t = product(S.lb + r * kLbStride, B, y0);
    if (h == 0) rs[r] = S.sv[r] - t;
  }
  __syncthreads();
  if (last < 0) return;
  s += product(S.di + r * ldi, ldi, rs);
  if (h == 0 && r < jb) {
    publish(words, r, s, A.epoch);
    A.b[F.first + j + r] = s;
    if (keep) keep[r] = s;
  }
}

// Column sums over the row groups of S.red4: FP32 on the first warp, f(first of
// four columns, their sums); FP64 with four threads per column, f(column, its sum).
template <typename Fn> __device__ __forceinline__ void groups_sum(const PsShared<float> &S, Fn f) {
  if (threadIdx.x >= 32) return;
  const int q = threadIdx.x;
  Vec<float> s = ld16(S.red4[0] + 4 * q);
#pragma unroll
  for (int g = 1; g < kT / 32; g++) {
    const Vec<float> o = ld16(S.red4[g] + 4 * q);
#pragma unroll
    for (int h = 0; h < 4; h++) s.v[h] += o.v[h];
  }
  f(4 * q, s);
}
template <typename Fn> __device__ __forceinline__ void groups_sum(const PsShared<double> &S, Fn f) {
  const int c = threadIdx.x / 4, g = 2 * (threadIdx.x % 4);
  const double s = quad_sum(S.red4[g][c] + S.red4[g + 1][c]);
  if (threadIdx.x % 4 == 0) f(c, s);
}
// f(column, sum) for each of them, and the store of all of them to a row
template <typename Fn> __device__ __forceinline__ void each_sum(int c, const Vec<float> &s, Fn f) {
#pragma unroll
  for (int h = 0; h < 4; h++) f(c + h, s.v[h]);
}
template <typename Fn> __device__ __forceinline__ void each_sum(int c, double s, Fn f) { f(c, s); }
__device__ __forceinline__ void put_sum(float *row, int c, const Vec<float> &s) {
  st16(row + c, s);
}
__device__ __forceinline__ void put_sum(double *row, int c, double s) { row[c] = s; }

// x[first + j + c] = sum_{r >= c} Dinv[r][c] v[r]  (Dinv staged in S.di, zero above the
// diagonal; v = S.sv), published in the slot's words. FP32: thread (g, q) takes columns
// 4q .. and rows 16g ..; FP64: four threads per column, a warp's eight columns start
// at their diagonal, and the result is corrected as in diag_fwd.
__device__ void diag_bwd(const PsArgs<float> &A, PsShared<float> &S, const FrontInfo &F, int j, uint2 *words) {
  constexpr int B = Ps<float>::B, RW = Ps<float>::RW;
  const int jb = min(B, F.ncol - j), ldi = (jb + 3) & ~3;
  const int q = threadIdx.x % 32, g = threadIdx.x / 32, c = 4 * q;
  Vec<float> acc = vzero<float>();
  if (c < ldi && c < RW * (g + 1)) {  // (zero above the diagonal)
#pragma unroll
    for (int k = 0; k < RW; k++) {
      const int r = RW * g + k;
      if (r < jb) acc = vfma(ld16(S.di + r * ldi + c), S.sv[r], acc);
    }
  }
  st16(S.red4[g] + 4 * q, acc);
  __syncthreads();
  float *xo = A.x + F.first + j;
  groups_sum(S, [&](int c0, auto s) {
    each_sum(c0, s, [&](int cc, float v) {
      if (cc >= jb) return;
      publish(words, cc, v, A.epoch);
      xo[cc] = v;
    });
  });
}
__device__ void diag_bwd(const PsArgs<double> &A, PsShared<double> &S, const FrontInfo &F, int j, uint2 *words) {
  constexpr int B = Ps<double>::B;
  const int jb = min(B, F.ncol - j), ldi = (jb + 1) & ~1, c = quad_row(), h = threadIdx.x % 4;
  const int m0 = 2 * (c / 8), m1 = (jb + 3) / 4;  // row groups of this warp's columns (uniform per warp)
  double *x0 = S.red4[0], *rs = S.red4[1], s = 0.0;
  auto product = [&](const double *M, int ld, const double *v) {
    double a = 0.0;
#pragma unroll 4
    for (int m = m0; m < m1; m++) {
      const int r = 4 * m + h;
      if (r < jb && c < jb) a = fma(M[r * ld + c], v[r], a);
    }
    return quad_sum(a);
  };
  if (m0 < m1) {
    s = product(S.di, ldi, S.sv);
    if (h == 0) x0[c] = s;
  }
  __syncthreads();
  if (m0 < m1) {
    const double t = product(S.lb, kLbStride, x0);
    if (h == 0) rs[c] = S.sv[c] - t;
  }
  __syncthreads();
  if (m0 >= m1) return;
  s += product(S.di, ldi, rs);
  if (h == 0 && c < jb) {
    publish(words, c, s, A.epoch);
    A.x[F.first + j + c] = s;
  }
}

// Thread 0 polls *w until it reaches target (acquire), at most A.spins times
// and only while no other wait of the launch has run out; the CTA then shares
// the outcome. On expiry the status word is set, and every later wait of the
// launch gives up at once.
template <typename T>
__device__ bool wait_flag(const PsArgs<T> &A, PsShared<T> &S, const unsigned *w, unsigned target) {
  __syncthreads();  // every thread has read the previous outcome
  if (threadIdx.x == 0) {
    unsigned v, spins = 0;
    int ok = 1;
    while (true) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(w) : "memory");
      if (v >= target) break;
      if ((spins & 63u) == 0 && *(volatile int32_t *)(A.status + ST_SOLVE_TIMEOUT) != 0) {
        ok = 0;
        break;
      }
      if (++spins > A.spins) {
        atomicExch(A.status + ST_SOLVE_TIMEOUT, 1);
        ok = 0;
        break;
      }
      __nanosleep(32);
    }
    S.ok = ok;
  }
  __syncthreads();
  return S.ok != 0;
}

// After this CTA's writes: count one more on *w. The barrier orders every
// thread's writes before thread 0's release add, and a release is cumulative,
// so a consumer that acquires the count sees all of them.
__device__ void signal(unsigned *w) {
  __syncthreads();
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(w) : "memory");
}

// Wait until the update vectors of all children of front s are complete (one
// counter per front), and stage the children's map and vector offsets.
template <typename T>
__device__ bool wait_children(const PsArgs<T> &A, PsShared<T> &S, const FrontInfo &F, const SolveRec &R) {
  const DevPlan &dp = A.dp;
  const int nk = F.child_end - F.child_begin;
  if (threadIdx.x < min(nk, kMaxKids)) {
    const int32_t ch = dp.children[F.child_begin + threadIdx.x];
    S.kid_inv[threadIdx.x] = dp.fronts[ch].inv_off;
    S.kid_toff[threadIdx.x] = dp.toff[ch];
  }
  if (threadIdx.x == 0) S.nkids = nk;
  if (nk == 0) {
    __syncthreads();
    return true;
  }
  return wait_flag(A, S, f_tvec(A, R.task.front), (unsigned)R.kid_chunks);  // (syncs first)
}

// Sum of the children's update entries at front position p (after
// wait_children), in child order; the map entries of two children are loaded
// together, then their update entries.
template <typename T>
__device__ __forceinline__ T gather_children(const PsArgs<T> &A, const PsShared<T> &S,
                                                 const FrontInfo &F, int p) {
  const DevPlan &dp = A.dp;
  auto offs = [&](int k, int64_t &io, int64_t &to) {
    if (k < kMaxKids) {
      io = S.kid_inv[k];
      to = S.kid_toff[k];
    } else {
      const int32_t ch = dp.children[F.child_begin + k];
      io = dp.fronts[ch].inv_off;
      to = dp.toff[ch];
    }
  };
  T v = T(0);
  const int nk = S.nkids;
  int k = 0;
  for (; k + 1 < nk; k += 2) {
    int64_t io0, to0, io1, to1;
    offs(k, io0, to0);
    offs(k + 1, io1, to1);
    const int32_t q0 = dp.inv[io0 + p], q1 = dp.inv[io1 + p];
    const T t0 = q0 >= 0 ? ldcg(A.t + to0 + q0) : T(0);
    const T t1 = q1 >= 0 ? ldcg(A.t + to1 + q1) : T(0);
    if (q0 >= 0) v += t0;
    if (q1 >= 0) v += t1;
  }
  if (k < nk) {
    int64_t io, to;
    offs(k, io, to);
    const int32_t q = dp.inv[io + p];
    if (q >= 0) v += ldcg(A.t + to + q);
  }
  return v;
}

// The CTA's next ticket and its task record (registers of thread 32), taken
// once the running task has passed its last wait: the atomic and the load of
// the record then overlap the task's remaining work, and no CTA ever holds a
// ticket while it waits, so the smallest unfinished ticket is always running.
struct Next {
  int q;  // ticket
  bool have;
};

template <typename T>
__device__ __forceinline__ void take_next(const PsArgs<T> &A, Next &N) {
  if (threadIdx.x == 32 && !N.have) {
    N.q = (int)atomicAdd(A.ticket, 1u);  // the result is first read after the task
    N.have = true;
  }
}

// Thread 32: start the asynchronous copy of record q into S.rec[buf], and
// warm L2 with the record one grid further on.
template <typename T>
__device__ __forceinline__ void fetch_rec(const PsArgs<T> &A, PsShared<T> &S, int q, int buf) {
  if (q >= A.q1) return;
  const char *src = reinterpret_cast<const char *>(A.sv.recs + q);
  const uint32_t dst = smem_u32(&S.rec[buf]);
#pragma unroll
  for (int k = 0; k < (int)(sizeof(SolveRec) / 16); k++)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * k), "l"(src + 16 * k)
                 : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
  const int ahead = min(q + (int)gridDim.x, A.q1 - 1);
  asm volatile("prefetch.global.L2 [%0];" ::"l"(A.sv.recs + ahead));
}

// Forward, diagonal block i of front s: rows j0 .. j0 + jb of the front (the
// loads of block j are issued before y_j is waited for).
template <typename T>
__device__ void fwd_diag(const PsArgs<T> &A, PsShared<T> &S, const SolveRec &R, Next &N) {
  constexpr int B = Ps<T>::B;
  const Task &tk = R.task;
  const FrontInfo &F = R.front;
  const int i = tk.a, j0 = B * i, jb = min(B, F.ncol - j0), slot0 = R.slot0;
  stage_dinv(A, S, F, j0, slot0 + i);
  bool ok = wait_children(A, S, F, R);
  if (ok && threadIdx.x < B)
    S.sv[threadIdx.x] = threadIdx.x < jb
                            ? ldcg(A.a + F.first + j0 + threadIdx.x) - gather_children(A, S, F, j0 + threadIdx.x)
                            : T(0);
  FwdTile<T> tile;
  tile.clear();
  __syncthreads();  // S.sv is written
  const T *row = A.L + F.loff + (int64_t)j0 * F.ld;
  for (int j = 0; j < i && ok; j++) {  // block j < i is a full block
    tile.template load<true>(row + B * j, F.ld, jb, B);
    ok = tile.wait_y(A, block_words<T>(A.ly, R, j), B, j == i - 1);
    if (ok) tile.template mul<true>(S, B);
  }
  take_next(A, N);
  tile.finish(ok ? jb : 0, [&](int r, T v) { S.sv[r] -= v; });
  // the staged copy always lands before S.di is reused; the wait ends with a
  // barrier, after which every row of S.sv is final
  if (wait_dinv(A, S, ok)) diag_fwd(A, S, F, j0, block_words<T>(A.ly, R, i));
}

// Forward, rows r0 .. r0 + nr below front s: the children's entries plus
// L_rj y_j over every block j of the front, into the front's update vector.
template <typename T>
__device__ void fwd_below(const PsArgs<T> &A, PsShared<T> &S, const SolveRec &R, Next &N) {
  constexpr int B = Ps<T>::B;
  const Task &tk = R.task;
  const FrontInfo &F = R.front;
  const int r0 = tk.a, nr = min(B, F.nrow - r0), nb = (F.ncol + B - 1) / B;
  const int slot0 = R.slot0;
  bool ok = wait_children(A, S, F, R);
  if (ok && threadIdx.x < nr) S.xs[threadIdx.x] = gather_children(A, S, F, F.ncol + r0 + threadIdx.x);
  FwdTile<T> tile;
  tile.clear();
  __syncthreads();  // S.xs is written
  const T *row = A.L + F.loff + (int64_t)(F.ncol + r0) * F.ld;
  for (int j = 0; j < nb && ok; j++) {
    const int jbj = min(B, F.ncol - B * j);
    const T *P = row + B * j;
    if (jbj == B) tile.template load<true>(P, F.ld, nr, B);
    else tile.template load<false>(P, F.ld, nr, jbj);
    ok = tile.wait_y(A, block_words<T>(A.ly, R, j), jbj, false);
    if (!ok) break;
    if (jbj == B) tile.template mul<true>(S, B);
    else tile.template mul<false>(S, jbj);
  }
  take_next(A, N);
  tile.finish(ok ? nr : 0, [&](int r, T v) { A.t[R.toff + r0 + r] = S.xs[r] + v; });
  if (__syncthreads_and(ok)) signal(f_tvec(A, F.parent));  // rows below a front exist only below a parent
}

// Backward, rows r0 .. r0 + nr below front s: once the parent front (and so
// every ancestor holding those rows) is solved, the partial sums
// part[cb][c] = sum_r L[ncol + r0 + r, B cb + c] x[row r] of every column
// block, last block first (the order of the front's backward chain), each
// published as it is written. Thread (g, q): columns VW q .., rows RW g ..;
// the loads of the next block are issued before the reduction of the current
// one.
template <typename T>
__device__ void bwd_part(const PsArgs<T> &A, PsShared<T> &S, const SolveRec &R, Next &N) {
  constexpr int B = Ps<T>::B, VW = Ps<T>::VW, RW = Ps<T>::RW;
  const Task &tk = R.task;
  const FrontInfo &F = R.front;
  const DevPlan &dp = A.dp;
  const int r0 = tk.b, nr = min(B, F.nrow - r0), nb = (F.ncol + B - 1) / B;
  const int nbl = (F.nrow + B - 1) / B;
  const int q = threadIdx.x % 32, g = threadIdx.x / 32;
  const T *P = A.L + F.loff + (int64_t)(F.ncol + r0 + RW * g) * F.ld + VW * q;
  Vec<T> l[RW];
  auto load = [&](int cb) {
    const int c = B * cb + VW * q;
#pragma unroll
    for (int k = 0; k < RW; k++)
      l[k] = (c < F.ncol && RW * g + k < nr) ? ldg16(P + (int64_t)k * F.ld + B * cb) : vzero<T>();
  };
  load(nb - 1);
  const int32_t xrow = threadIdx.x < nr ? dp.sri[F.rows_off + r0 + threadIdx.x] : 0;
  if (F.parent >= 0 && !wait_flag(A, S, f_front(A, F.parent), (unsigned)R.parent_blocks))
    return;
  take_next(A, N);
  if (threadIdx.x < nr) S.xs[threadIdx.x] = ldcg(A.x + xrow);
  __syncthreads();
  for (int cb = nb - 1; cb >= 0; cb--) {
    Vec<T> acc = vzero<T>();
#pragma unroll
    for (int k = 0; k < RW; k++)
      if (RW * g + k < nr) acc = vfma(l[k], S.xs[RW * g + k], acc);
    if (cb > 0) load(cb - 1);
    st16(S.red4[g] + VW * q, acc);
    __syncthreads();
    T *row = A.part + (R.pbase + (int64_t)cb * nbl + r0 / B) * B;
    groups_sum(S, [&](int c, auto s) { put_sum(row, c, s); });
    signal(f_part(A, R.slot0 + cb));  // (its barrier also frees S.red4)
  }
}

// Brings a warp's RW rows of a tile (512 bytes each; nr rows in the tile) into L2
// ahead of their loads: a tile's registers allow one in flight, and DRAM's latency
// is as long as a chain's step.
template <typename T> __device__ __forceinline__ void prefetch_tile(const T *P, int64_t ld, int nr) {
  constexpr int RW = Ps<T>::RW, PER = RW / 8, EL = 128 / (int)sizeof(T);  // lines per lane, values per line
  const int lane = threadIdx.x % 32, r = RW * (threadIdx.x / 32) + lane * PER / 4;
  if (r >= nr) return;
#pragma unroll
  for (int h = 0; h < PER; h++)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(P + (int64_t)r * ld + (lane * PER % 4 + h) * EL));
}

// Backward, column block cb of front s: the partial sums in chunk order, then
// L[block i, block cb]^T x_i for i > cb as each x_i is published, then
// x_cb = L_cc^{-T} (.) with the staged inverse.
template <typename T>
__device__ void bwd_diag(const PsArgs<T> &A, PsShared<T> &S, const SolveRec &R, Next &N) {
  constexpr int B = Ps<T>::B, VW = Ps<T>::VW, RW = Ps<T>::RW;
  const Task &tk = R.task;
  const FrontInfo &F = R.front;
  const int cb = tk.a, c0 = B * cb, jb = min(B, F.ncol - c0), nb = (F.ncol + B - 1) / B;
  const int nbl = (F.nrow + B - 1) / B, slot0 = R.slot0;
  stage_dinv(A, S, F, c0, slot0 + cb);
  bool ok = true;
  if (nbl > 0) ok = wait_flag(A, S, f_part(A, slot0 + cb), nbl);  // implies the parent is done
  else if (ok && F.parent >= 0)
    ok = wait_flag(A, S, f_front(A, F.parent), (unsigned)R.parent_blocks);
  // b of this block is the forward result: the words of this launch's forward
  // task of the block, or complete before a backward-only launch
  if (ok) {
    // FP64: four threads per column (see quad_sum), the first holds the result
    constexpr int TPC = sizeof(T) == 8 ? 4 : 1;
    const int cc = threadIdx.x / TPC;
    const bool mine = threadIdx.x % TPC == 0 && cc < jb;
    T bv = T(0);
    const uint2 *words = block_words<T>(A.ly, R, cb);
    if (A.fwd_here)
      ok = wait_words(A, words, false, [&]() { return !mine || read_word(words, cc, A.epoch, bv); });
    else if (mine)
      bv = ldcg(A.b + F.first + c0 + cc);
    T ps = T(0);
    const T *pp = A.part + (R.pbase + (int64_t)cb * nbl) * B + cc;
    for (int k = threadIdx.x % TPC; k < nbl && cc < jb; k += TPC) ps += ldcg(pp + (int64_t)k * B);
    if (TPC == 4) ps = quad_sum(ps);
    if (threadIdx.x % TPC == 0 && cc < B) S.sv[cc] = bv - ps;  // (zero past jb)
  }
  const int q = threadIdx.x % 32, g = threadIdx.x / 32, c = c0 + VW * q;
  Vec<T> acc = vzero<T>();
  const bool wide = c0 + B <= F.ncol;  // (a block with blocks after it is a whole one)
  if (wide && nb - 2 > cb) prefetch_tile(A.L + F.loff + (int64_t)(B * (nb - 2)) * F.ld + c0, F.ld, B);
  for (int i = nb - 1; i > cb && ok; i--) {
    const int jbi = min(B, F.ncol - B * i);
    if (wide && i - 2 > cb) prefetch_tile(A.L + F.loff + (int64_t)(B * (i - 2)) * F.ld + c0, F.ld, B);
    Vec<T> l[RW];
    const T *P = A.L + F.loff + (int64_t)(B * i + RW * g) * F.ld + c;
#pragma unroll
    for (int k = 0; k < RW; k++)
      l[k] = (c < F.ncol && RW * g + k < jbi) ? ldg16(P + (int64_t)k * F.ld) : vzero<T>();
    // lane k < RW reads x of row RW g + k of block i; the warp shares them
    T xv = T(0);
    const bool mine = q < RW && RW * g + q < jbi;
    const uint2 *words = block_words<T>(A.lx, R, i);
    ok = wait_words(A, words, i == cb + 1, [&]() { return !mine || read_word(words, RW * g + q, A.epoch, xv); });
    if (!ok) break;
#pragma unroll
    for (int k = 0; k < RW; k++) acc = vfma(l[k], __shfl_sync(0xffffffffu, xv, k), acc);
  }
  take_next(A, N);
  st16(S.red4[g] + VW * q, acc);
  ok = __syncthreads_and(ok) != 0;
  if (ok)
    groups_sum(S, [&](int k0, auto s) {
      each_sum(k0, s, [&](int k, T v) {
        if (k < jb) S.sv[k] -= v;
      });
    });
  if (wait_dinv(A, S, ok)) {  // (ends with a barrier)
    diag_bwd(A, S, F, c0, block_words<T>(A.lx, R, cb));
    signal(f_front(A, tk.front));
  }
}

// A narrow front in one task (narrow_front: at most 32 columns and 512 rows below). The
// lower half of a nested-dissection tree is thousands of such fronts, and a task costs 3
// to 4 us whatever its size (ticket, record, the children's flag, two dependent gathers,
// its own flag): one task a front and sweep instead of one per block and chunk of rows,
// which also hands y to the rows below through shared memory. One solve, TF32x3: 666 ->
// 574 us at 48^3, 1548 -> 1320 at 64^3; eight right-hand
// sides at 56^3 with PCG 15.2 -> 12.6 ms. (64 columns in FP32: 12.0 ms, nothing for one
// right-hand side.)
// Forward: a thread per row below (its L row in registers before the wait), the
// diagonal block as in fwd_diag.
template <typename T>
__device__ void fwd_narrow(const PsArgs<T> &A, PsShared<T> &S, const SolveRec &R, Next &N) {
  constexpr int B = Ps<T>::B, VW = Ps<T>::VW, NV = kNarrowCols / VW;
  const FrontInfo &F = R.front;
  const int nc = F.ncol, nr = F.nrow, tid = threadIdx.x;
  stage_dinv(A, S, F, 0, R.slot0);
  const T *rows = A.L + F.loff + (int64_t)nc * F.ld;
  Vec<T> l[NV];
  auto load = [&](int r) {
#pragma unroll
    for (int m = 0; m < NV; m++)
      l[m] = (r < nr && VW * m < nc) ? ldg16(rows + (int64_t)r * F.ld + VW * m) : vzero<T>();
  };
  load(tid);
  const bool ok = wait_children(A, S, F, R);
  T g = T(0);
  if (ok) {
    if (tid < B) S.sv[tid] = tid < nc ? ldcg(A.a + F.first + tid) - gather_children(A, S, F, tid) : T(0);
    if (tid < nr) g = gather_children(A, S, F, nc + tid);
  }
  if (tid >= nc && tid < kNarrowCols) S.xs[tid] = T(0);
  take_next(A, N);
  if (!wait_dinv(A, S, ok)) return;  // (a barrier: S.sv is written)
  diag_fwd(A, S, F, 0, block_words<T>(A.ly, R, 0), S.xs);
  __syncthreads();
  for (int r0 = 0; r0 < nr; r0 += kT) {
    const int r = r0 + tid;
    if (r0 > 0) {
      load(r);
      g = r < nr ? gather_children(A, S, F, nc + r) : T(0);
    }
    T s = T(0);
#pragma unroll
    for (int m = 0; m < NV; m++)
      if (VW * m < nc) {
        Vec<T> v = l[m];
#pragma unroll
        for (int h = 1; h < VW; h++)
          if (VW * m + h >= nc) v.v[h] = T(0);  // (padding of the row)
        s = vdot(v, ld16(S.xs + VW * m), s);
      }
    if (r < nr) A.t[R.toff + r] = g + s;
  }
  if (nr > 0) signal(f_tvec(A, F.parent));
}

// Backward: 2^lg threads per row, each the VW columns of a 16-byte load, down the rows
// below; sums across a warp's rows by shuffles and across the warps through shared
// memory, then the diagonal block as in bwd_diag. The solution at the rows below sits in
// the part of S.di past the staged inverse.
template <typename T>
__device__ void bwd_narrow(const PsArgs<T> &A, PsShared<T> &S, const SolveRec &R, Next &N) {
  constexpr int VW = Ps<T>::VW, NL = 8;
  static_assert(kNarrowCols * kNarrowCols + kNarrowRows <= Ps<T>::B * Ps<T>::B, "room past the staged inverse");
  static_assert(kNarrowRows <= 2 * kT && kNarrowCols / VW <= 16 && kNarrowCols <= 32, "rows and columns per thread");
  const FrontInfo &F = R.front;
  const int nc = F.ncol, nr = F.nrow, tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  stage_dinv(A, S, F, 0, R.slot0);
  int lg = 0;
  while ((VW << lg) < nc) lg++;
  const int cg = 1 << lg, c = VW * (tid & (cg - 1)), rr = tid >> lg, rp = kT >> lg;
  const T *P = A.L + F.loff + (int64_t)nc * F.ld + c;
  T *xs = S.di + kNarrowCols * kNarrowCols;
  Vec<T> l[NL];
  auto load = [&](int r0) {
#pragma unroll
    for (int k = 0; k < NL; k++) {
      const int r = r0 + rr + k * rp;
      l[k] = (c < nc && r < nr) ? ldg16(P + (int64_t)r * F.ld) : vzero<T>();
    }
  };
  load(0);
  const int32_t *ri = A.dp.sri + F.rows_off;
  const int32_t i0 = tid < nr ? ri[tid] : 0, i1 = tid + kT < nr ? ri[tid + kT] : 0;
  bool ok = F.parent < 0 || wait_flag(A, S, f_front(A, F.parent), (unsigned)R.parent_blocks);
  take_next(A, N);
  T bv = T(0);
  if (ok) {
    if (tid < nr) xs[tid] = ldcg(A.x + i0);
    if (tid + kT < nr) xs[tid + kT] = ldcg(A.x + i1);
    const uint2 *words = block_words<T>(A.ly, R, 0);
    if (A.fwd_here) ok = wait_words(A, words, false, [&]() { return tid >= nc || read_word(words, tid, A.epoch, bv); });
    else if (tid < nc) bv = ldcg(A.b + F.first + tid);
  }
  __syncthreads();
  Vec<T> acc = vzero<T>();
  for (int r0 = 0; r0 < nr && ok; r0 += NL * rp) {
    if (r0 > 0) load(r0);
#pragma unroll
    for (int k = 0; k < NL; k++) {
      const int r = r0 + rr + k * rp;
      if (r < nr) acc = vfma(l[k], xs[r], acc);
    }
  }
  for (int o = cg; o < 32; o <<= 1)
#pragma unroll
    for (int h = 0; h < VW; h++) acc.v[h] += __shfl_xor_sync(0xffffffffu, acc.v[h], o);
  if (lane < cg) st16(S.red4[warp] + c, acc);
  __syncthreads();
  if (tid < nc) {
    T s = S.red4[0][tid];
#pragma unroll
    for (int w = 1; w < kT / 32; w++) s += S.red4[w][tid];
    S.sv[tid] = bv - s;
  }
  if (wait_dinv(A, S, ok)) {  // (ends with a barrier)
    diag_bwd(A, S, F, 0, block_words<T>(A.lx, R, 0));
    signal(f_front(A, R.task.front));
  }
}

template <typename T>
__device__ __forceinline__ void run_task(const PsArgs<T> &A, PsShared<T> &S, const SolveRec &R, Next &N) {
  switch (R.task.c) {
    case WS_FWD_DIAG: fwd_diag(A, S, R, N); break;
    case WS_FWD_BELOW: fwd_below(A, S, R, N); break;
    case WS_FWD_NARROW: fwd_narrow(A, S, R, N); break;
    case WS_BWD_PART: bwd_part(A, S, R, N); break;
    case WS_BWD_NARROW: bwd_narrow(A, S, R, N); break;
    default: bwd_diag(A, S, R, N); break;
  }
}

// Persistent solve: every CTA takes tasks in plan order from the global ticket
// counter until the range is exhausted. With several right-hand sides (MANY) each
// task comes once per right-hand side, next to each other: their chains of blocks,
// which leave most of the chip waiting, run side by side, and a tile of L is read
// from DRAM once for all of them.
template <typename T, bool MANY> __global__ void __launch_bounds__(kT, 2) psolve_kernel(PsArgs<T> A) {
  extern __shared__ __align__(128) unsigned char ps_smem[];
  PsShared<T> &S = *reinterpret_cast<PsShared<T> *>(ps_smem);
  // Thread 32 takes the tickets: the first here, each next one inside the
  // running task once it has passed its last wait (take_next), or right after
  // a task that ended early; the next task's record is copied into the other
  // shared buffer while the CTA finishes the current one.
  Next N{0, false};
  int cur = 0;
  auto fetch = [&](int ticket, int buf) {  // thread 32: the ticket's task
    const int q = A.q0 + (MANY ? ticket / A.nrhs : ticket);
    fetch_rec(A, S, q, buf);
    asm volatile("cp.async.wait_all;" ::: "memory");
    S.tk = q;
    if (MANY) S.rhs = ticket % A.nrhs;
  };
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&S.mbar)), "r"(1u));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    S.parity = 0;
  }
  if (threadIdx.x == 32) fetch((int)atomicAdd(A.ticket, 1u), 0);
  __syncthreads();
  while (true) {
    const int qt = S.tk;
    if (qt >= A.q1) break;
    const SolveRec &R = S.rec[cur];
    N.have = false;
    if (qt == A.withhold) {
      // abandoned (test of the bounded waits): the tasks that need its result
      // run out of time
    } else if (MANY) {
      PsArgs<T> Ak = A;
      shift_rhs(Ak, S.rhs);
      run_task(Ak, S, R, N);
    } else {
      run_task(A, S, R, N);
    }
    take_next(A, N);  // a task that gave up early
    if (threadIdx.x == 32) fetch(N.q, cur ^ 1);
    __syncthreads();  // the next record has landed; the shared scratch is free
    cur ^= 1;
  }
}

template <typename T, bool MANY> int psolve_grid(int64_t ntask) {
  static int per_device[64] = {0};
  int dev = 0;
  ck(cudaGetDevice(&dev), "cudaGetDevice");
  int &g = per_device[dev & 63];
  if (g == 0) {
    int sms = 0, nb = 0;
    auto kernel = psolve_kernel<T, MANY>;
    ck(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PsShared<T>)),
       "solve shared-memory attribute");
    ck(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev), "SM count");
    ck(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, kT, sizeof(PsShared<T>)), "occupancy");
    g = std::max(1, sms * std::min(nb, 2));
  }
  return (int)std::max<int64_t>(1, std::min<int64_t>(g, ntask));
}

}  // namespace

// Allow a kernel this much shared memory on the current device (`once`: the kernel's).
template <typename K> static void allow_smem(K kernel, int smem, DeviceOnce &once) {
  int dev = 0;
  ck(cudaGetDevice(&dev), "cudaGetDevice");
  if (!once.needed(dev)) return;
  ck(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem), "dinv attribute");
  once.done(dev);
}

void launch_dinv(const DevPlan &dp, const Plan &plan, const float *L, float *Dinv,
                 cudaStream_t st) {
  const int n = (int)plan.s32.inv.size();
  if (n == 0) return;
  const int smem = 2 * 128 * 129 * (int)sizeof(float);
  static DeviceOnce once;
  allow_smem(dinv_kernel, smem, once);
  note_launch();
  dinv_kernel<<<n, 128, smem, st>>>(dp, L, Dinv);
}

void launch_dinv(const DevPlan &dp, const Plan &plan, const double *L, double *Dinv,
                 cudaStream_t st) {
  const int n = (int)plan.s64.inv.size();
  if (n == 0) return;
  constexpr int smem = kSolveB64 * (2 * kSolveB64 + 1) * (int)sizeof(double);
  static DeviceOnce once;
  allow_smem(dinv64_kernel, smem, once);
  note_launch();
  dinv64_kernel<<<n, kDinvThreads, smem, st>>>(dp, L, Dinv);
}

template <typename T>
void launch_psolve(const DevPlan &dp, const Plan &plan, const T *L, const T *Dinv, const SolveBufs<T> &v,
                   int nrhs, int32_t *status, bool fwd, bool bwd, cudaStream_t st,
                   unsigned test_spins, int test_withhold) {
  const SolvePlan &sp = sizeof(T) == 8 ? plan.s64 : plan.s32;
  const int32_t q0 = fwd ? 0 : sp.fwd_tasks;
  const int32_t q1 = bwd ? (int32_t)sp.tasks.size() : sp.fwd_tasks;
  if (q1 <= q0) return;
  ck(cudaMemsetAsync(v.flags, 0, (size_t)(nrhs * v.sd.flags) * sizeof(unsigned), st), "solve flags");
  PsArgs<T> A{dp, sizeof(T) == 8 ? dp.s64 : dp.s32, L, Dinv, v.a, v.b, v.x, v.t, v.part, q0, q1, v.flags, v.flags,
              v.wy, v.wx, v.epoch, status, test_spins ? test_spins : kBarrierSpins, test_withhold,
              (int32_t)sp.dinv_off.size(), (int32_t)plan.fronts.size(), fwd && bwd ? 1 : 0, nrhs, v.sd};
  const int64_t tickets = (int64_t)(q1 - q0) * nrhs;
  note_launch();
  if (nrhs == 1) psolve_kernel<T, false><<<psolve_grid<T, false>(tickets), kT, sizeof(PsShared<T>), st>>>(A);
  else psolve_kernel<T, true><<<psolve_grid<T, true>(tickets), kT, sizeof(PsShared<T>), st>>>(A);
  ck(cudaGetLastError(), "solve launch");
}
template void launch_psolve<float>(const DevPlan &, const Plan &, const float *, const float *,
                                   const SolveBufs<float> &, int, int32_t *, bool, bool, cudaStream_t, unsigned,
                                   int);
template void launch_psolve<double>(const DevPlan &, const Plan &, const double *, const double *,
                                    const SolveBufs<double> &, int, int32_t *, bool, bool, cudaStream_t, unsigned,
                                    int);

}  // namespace gipm
