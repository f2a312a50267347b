// Assembly of the primal condensed matrix (Eq. 5) and the level-scheduled
// multifrontal supernodal Cholesky (Sec. 2: pivoting-free factorisation with
// elimination-tree parallelism), SIMT FMA path for FP64 and FP32.
//
// Per level of the supernodal tree: build every frontal matrix of the level
// (gather of the children's update matrices, each entry written once) and add the
// K entries owned by the level, then factor the fronts block column by block
// column: Cholesky of the diagonal block, triangular solve of the rows below,
// right-looking update of the rest of the panel and of the update matrix
// U = F22 - L21 L21^T. No atomics on values: results are bit-reproducible.
#include <cfloat>
#include <climits>
#include <stdexcept>

#include "launch.h"
#include "ptx.cuh"

namespace gipm {

namespace {

__global__ void assemble_kernel(DevPlan dp, const double *__restrict__ jv,
                                const double *__restrict__ D, const double *__restrict__ wv,
                                double delta_p, double *__restrict__ kval) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < dp.nk;
       q += (int64_t)gridDim.x * blockDim.x) {
    double v = 0.0;
    const int64_t p1 = dp.k_poff[q + 1];
    for (int64_t p = dp.k_poff[q]; p < p1; p++) {
      const int32_t a = dp.k_pa[p], b = dp.k_pb[p];
      v = fma(jv[a] * D[dp.jrow[a]], jv[b], v);
    }
    const int64_t w = dp.k_w[q];
    if (w >= 0 && wv) v += wv[w];
    const int32_t i = dp.k_diag[q];
    if (i >= 0) {
      double d = delta_p;
      if (dp.lpos[i] >= 0) d += D[dp.lpos[i]];
      if (dp.upos[i] >= 0) d += D[dp.upos[i]];
      v += d;
    }
    kval[q] = v;
  }
}

// Four consecutive entries at a 16-byte aligned address.
__device__ __forceinline__ void store4(float *p, float a, float b, float c, float d) {
  *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void store4(double *p, double a, double b, double c, double d) {
  reinterpret_cast<double2 *>(p)[0] = make_double2(a, b);
  reinterpret_cast<double2 *>(p)[1] = make_double2(c, d);
}

// Front assembly: one tile of 64 rows x (at most) 64 columns of a front's
// lower triangle per block of 128 threads; thread (row group g, column group
// q) owns rows r0 + g + 8i (i < 8) and columns c0 + 4q .. c0 + 4q + 3. Each
// entry is the sum, over the children in ascending order, of the matching
// entry of the child's update matrix (through the child->front inverse map);
// then, in levels of few tiles (FUSED), the K entries of the tile's rows that
// fall in its columns are added to what the block has stored.
// The maps of up to four children are staged together (one memory round
// trip), and a child none of whose rows or none of whose columns fall in the
// tile is skipped by the whole block. Panel tiles start at multiples of 64
// columns and update-matrix tiles at ncol + multiples of 64, so every
// 4-column group is one aligned vector store (entries above the diagonal and
// padding past ncol or nf are written as zeros). 32 entries per thread keep
// enough bytes in flight per block for the chain of dependent loads
// (task, front, children, maps) a tile starts with.
constexpr int kBuildThreads = 128, kBuildGroup = 4;
template <typename T, bool FUSED>
__global__ void __launch_bounds__(kBuildThreads) build_front_kernel(DevPlan dp, int32_t task0, int64_t build_k,
                                                                    const double *__restrict__ kval,
                                                                    T *__restrict__ L,
                                                                    T *__restrict__ U) {
  constexpr int BT = kBuildTile, RS = kBuildThreads / (BT / 4), NR = BT / RS;  // 8 row groups, 8 rows each
  const Task tk = dp.build[task0 + blockIdx.x];
  longlong2 kr = make_longlong2(0, 0);  // K entries of the tile's rows
  if (FUSED) kr = *reinterpret_cast<const longlong2 *>(dp.build_k + build_k + 2 * (int64_t)blockIdx.x);
  const FrontInfo F = dp.fronts[tk.front];
  const int nf = F.ncol + F.nrow;
  const int r0 = tk.a, c0 = tk.b, w = tk.c;
  __shared__ __align__(16) int32_t map[kBuildGroup][2 * BT];  // row maps, then column maps
  __shared__ int32_t hit[kBuildGroup][2 * BT / 32];  // per 32 maps: some entry maps into the child
  __shared__ int64_t uoff[kBuildGroup];
  __shared__ int32_t uld[kBuildGroup];
  const int tid = threadIdx.x, lane = tid % 32, g = tid / (BT / 4), q4 = 4 * (tid % (BT / 4));
  T acc[NR][4];
#pragma unroll
  for (int i = 0; i < NR; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) acc[i][j] = T(0);
  for (int cg = F.child_begin; cg < F.child_end; cg += kBuildGroup) {
    const int nc = min(kBuildGroup, F.child_end - cg);
    __syncthreads();
    // a warp's 32 entries are half of one child's row maps or column maps
    for (int e = tid; e < nc * 2 * BT; e += kBuildThreads) {
      const int q = e / (2 * BT), m = e % (2 * BT);
      const FrontInfo C = dp.fronts[dp.children[cg + q]];
      const int idx = m < BT ? r0 + m : c0 + m - BT;
      const bool inside = m < BT ? idx < nf : m - BT < w;
      const int32_t t = inside ? dp.inv[C.inv_off + idx] : -1;
      map[q][m] = t;
      const unsigned any = __ballot_sync(0xffffffffu, t >= 0);
      if (lane == 0) hit[q][m / 32] = any != 0u;
      if (m == 0) {
        uoff[q] = C.uoff;
        uld[q] = C.uld;
      }
    }
    __syncthreads();
    for (int q = 0; q < nc; q++) {
      if (!(hit[q][0] | hit[q][1]) || !(hit[q][2] | hit[q][3])) continue;
      const int4 b = *reinterpret_cast<const int4 *>(&map[q][BT + q4]);
      const int bb[4] = {b.x, b.y, b.z, b.w};
      const T *Uc = U + uoff[q];
      const int64_t ldq = uld[q];
#pragma unroll
      for (int i = 0; i < NR; i++) {
        const int rr = g + RS * i;
        const int a = map[q][rr];
        const T *row = Uc + a * ldq;
        T v[4];
#pragma unroll
        for (int j = 0; j < 4; j++)
          v[j] = (a >= 0 && bb[j] >= 0 && r0 + rr >= c0 + q4 + j) ? row[bb[j]] : T(0);
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] += v[j];
      }
    }
  }
  if (!FUSED && q4 >= w) return;
  const int c = c0 + q4;
  const bool panel = c0 < F.ncol;
  const int lim = panel ? F.ncol : nf;  // columns past lim are padding
#pragma unroll
  for (int i = 0; i < NR; i++) {
    const int r = r0 + g + RS * i;
    if (r >= nf || (FUSED && q4 >= w)) continue;
    T o[4];
#pragma unroll
    for (int j = 0; j < 4; j++) o[j] = (c + j <= r && c + j < lim) ? acc[i][j] : T(0);
    T *dst = panel ? L + F.loff + (int64_t)r * F.ld + c
                   : U + F.uoff + (int64_t)(r - F.ncol) * F.uld + (c - F.ncol);
    if (panel || r >= F.ncol) store4(dst, o[0], o[1], o[2], o[3]);
  }
  if (!FUSED || kr.x == kr.y) return;
  __syncthreads();  // the tile is stored
  for (int64_t q = kr.x + tid; q < kr.y; q += kBuildThreads) {
    const int64_t s = dp.k_slot[q], at = s - F.loff;
    const int col = F.ncol > BT ? (int)(at % F.ld) : c0;
    if (col >= c0 && col < c0 + w) L[s] = T((double)L[s] + kval[q]);
  }
}

template <typename T>
__global__ void kadd_kernel(DevPlan dp, int64_t q0, int64_t q1, const double *__restrict__ kval,
                            T *__restrict__ L) {
  for (int64_t q = q0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < q1;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = dp.k_slot[q];
    L[s] = T((double)L[s] + kval[q]);
  }
}

// 16 bytes as one load or store (a copy of the struct is split into its members).
template <typename T> struct Vec16 {
  T v[16 / sizeof(T)];
};
__device__ __forceinline__ Vec16<float> ld16(const float *p) {
  const float4 f = *reinterpret_cast<const float4 *>(p);
  return Vec16<float>{{f.x, f.y, f.z, f.w}};
}
__device__ __forceinline__ Vec16<double> ld16(const double *p) {
  const double2 f = *reinterpret_cast<const double2 *>(p);
  return Vec16<double>{{f.x, f.y}};
}
__device__ __forceinline__ void st16(float *p, const Vec16<float> &v) {
  *reinterpret_cast<float4 *>(p) = make_float4(v.v[0], v.v[1], v.v[2], v.v[3]);
}
__device__ __forceinline__ void st16(double *p, const Vec16<double> &v) {
  *reinterpret_cast<double2 *>(p) = make_double2(v.v[0], v.v[1]);
}

// Trailing update of a level's fronts by the finished columns [k0, k1) (C -= A S
// B^T, A and B rows of a front's panel, S = diag(pivot signs), nullptr: I): one
// TS x TS tile of the columns [min(c0, ncol), min(clim, ncol)) of a panel, or,
// with_u, also of the update matrix, per block (tile numbering: upd_decode).
//
// FP64 (32 x 32 tiles, 64 columns per launch, right-looking): GB300's FP64 pipe
// starts two multiply-adds a cycle per SM, so a 32 x 32 x 64 tile is 16 us of pipe
// time for 48 KB of L2 traffic, and nothing but spreading the tiles over all SMs
// matters. A left-looking form (one block column at a time, K = all columns before
// it) has 47 blocks of 64 x 64 for 152 SMs on a 3008-column front: 118 ms of updates
// on the 32^3 grid LP against 37 ms (32 ms at the nominal FP64 rate). FP32 (64 x 64 tiles): the pipe
// is 64 times faster, so the tile's reads and writes are spread over a longer K
// (columns of a super-step: see Plan::kSuper32).
template <typename T, int TS, int NT, int BK>
__global__ void __launch_bounds__(NT, sizeof(T) == 8 ? 3 : 2) upd_kernel(DevPlan dp, const Task *__restrict__ ents, int nent,
                                                 int k0, int k1, int c0, int clim, int with_u,
                                                 T *__restrict__ L, T *__restrict__ U) {
  constexpr int TY = NT / 16, MI = TS / TY, NJ = TS / 16;
  constexpr int VW = 16 / (int)sizeof(T), LD = BK + VW, NV = BK / VW;  // rows of BK values, 16-byte padded
  constexpr int PER = 2 * TS * NV / NT;                                // 16-byte loads per thread and chunk
  static_assert(sizeof(T) == 4 || BK >= 64, "an FP64 launch has at most 64 columns");
  static_assert(2 * TS * NV % NT == 0 && TS * NV % NT == 0, "loader shape");
  __shared__ __align__(16) T sA[TS * LD], sB[TS * LD];
  int lo = 0, hi = nent - 1;  // the front this block's tile belongs to
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (ents[mid].a <= (int)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const Task tk = ents[lo];
  const FrontInfo F = dp.fronts[tk.front];
  const int nf = F.ncol + F.nrow, K = min(k1, F.ncol) - k0;
  const UpdTile tl = upd_decode(F.ncol, F.nrow, c0, clim, with_u, TS, (int)blockIdx.x - tk.a);
  const int M = min(TS, nf - tl.r), N = min(TS, tl.cend - tl.c);
  T *P = L + F.loff;
  const T *A = P + (int64_t)tl.r * F.ld + k0, *B = P + (int64_t)tl.c * F.ld + k0;
  T *C;
  int64_t ldc;
  if (tl.c < F.ncol) {
    ldc = F.ld;
    C = P + (int64_t)tl.r * ldc + tl.c;
  } else {
    ldc = F.uld;
    C = U + F.uoff + (int64_t)(tl.r - F.ncol) * ldc + (tl.c - F.ncol);
  }
  const int8_t *sk = dp.sgn ? dp.sgn + F.first + k0 : nullptr;
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  using V = Vec16<T>;
  V reg[PER];
  auto load = [&](int kc) {  // chunk [kc, kc + BK) of both operands (zero past K, M, N)
#pragma unroll
    for (int q = 0; q < PER; q++) {
      const bool isb = q >= PER / 2;
      const int e = tid + NT * (isb ? q - PER / 2 : q), r = e / NV, kk = kc + VW * (e % NV);
      V x;
#pragma unroll
      for (int h = 0; h < VW; h++) x.v[h] = T(0);
      if (r < (isb ? N : M) && kk < K) {
        x = ld16((isb ? B : A) + (int64_t)r * F.ld + kk);
#pragma unroll
        for (int h = 0; h < VW; h++) {
          if (kk + h >= K) x.v[h] = T(0);
          else if (isb && sk && sk[kk + h] < 0) x.v[h] = -x.v[h];
        }
      }
      reg[q] = x;
    }
  };
  load(0);
  T acc[MI][NJ], cv[MI][NJ];  // the products' sum, the target's values
#pragma unroll
  for (int i = 0; i < MI; i++)
#pragma unroll
    for (int j = 0; j < NJ; j++) {
      const int r = ty + TY * i, c = tx + 16 * j;
      acc[i][j] = T(0);
      cv[i][j] = (r < M && c < N) ? C[(int64_t)r * ldc + c] : T(0);
    }
  for (int kc = 0; kc < K; kc += BK) {
    if (kc > 0) __syncthreads();
#pragma unroll
    for (int q = 0; q < PER; q++) {
      const bool isb = q >= PER / 2;
      const int e = tid + NT * (isb ? q - PER / 2 : q);
      st16((isb ? sB : sA) + (e / NV) * LD + VW * (e % NV), reg[q]);
    }
    __syncthreads();
    if (sizeof(T) == 4 && kc + BK < K) load(kc + BK);  // (FP64: one chunk)
    const int kn = min(BK, K - kc);
#pragma unroll (sizeof(T) == 8 ? 4 : 1)
    for (int kk = 0; kk < kn; kk += VW) {
      V a[MI], b[NJ];
#pragma unroll
      for (int i = 0; i < MI; i++) a[i] = ld16(sA + (ty + TY * i) * LD + kk);
#pragma unroll
      for (int j = 0; j < NJ; j++) b[j] = ld16(sB + (tx + 16 * j) * LD + kk);
#pragma unroll
      for (int h = 0; h < VW; h++)
#pragma unroll
        for (int i = 0; i < MI; i++)
#pragma unroll
          for (int j = 0; j < NJ; j++) acc[i][j] = fma(a[i].v[h], b[j].v[h], acc[i][j]);
    }
  }
#pragma unroll
  for (int i = 0; i < MI; i++)
#pragma unroll
    for (int j = 0; j < NJ; j++) {
      const int r = ty + TY * i, c = tx + 16 * j;
      if (r < M && c < N) C[(int64_t)r * ldc + c] = cv[i][j] - acc[i][j];
    }
}

template <typename T> __device__ __forceinline__ T big_pivot();
template <> __device__ __forceinline__ float big_pivot<float>() { return 1e30f; }
template <> __device__ __forceinline__ double big_pivot<double>() { return 1e64; }

// Out of line, so that the division is not evaluated beside the usual path.
template <typename T> __device__ __noinline__ T slow_div(T a, T b) { return a / b; }

// Estimates of 1 / d and 1 / sqrt(d) in FP32 for a double d > 0 within FP32's
// normal range (in_fp32), converted by moving bits: GB300's FP64 unit takes about
// 90 cycles for a conversion or a comparison, as for a multiply-add.
__device__ __forceinline__ bool in_fp32(double d) {  // 2^-119 <= d < 2^120
  return ((unsigned)__double2hiint(d) >> 20) - 904u < 239u;  // (false for d < 0 and NaN)
}
__device__ __forceinline__ float low_float(double d) {  // d cut to 24 bits
  return __int_as_float(((__double2hiint(d) - (896 << 20)) << 3) | ((unsigned)__double2loint(d) >> 29));
}
__device__ __forceinline__ double widen(float f) {  // normal f > 0
  const int b = __float_as_int(f);
  return __hiloint2double((b >> 3) + (896 << 20), b << 29);
}
// 1 / sqrt(d): one third-order step from the estimate, r (1 + e/2 + 3 e^2 / 8) with e =
// 1 - d r^2 (|e| < 2^-20: the step's own error is below 2^-58).
__device__ __forceinline__ double inv_sqrt(double d) {
  if (!in_fp32(d)) return slow_div(1.0, sqrt(d));
  const double r = widen(rsqrtf(low_float(d)));
  const double e = fma(-(d * r), r, 1.0);
  return fma(r * e, fma(0.375, e, 0.5), r);
}
__device__ __forceinline__ float inv_sqrt(float d) {
  if (!(d > 1e-30f && d < 1e30f)) return 1.f / sqrtf(d);
  const float r = rsqrtf(d);
  return fmaf(0.5f * r, fmaf(-d * r, r, 1.f), r);
}
// 1 / d is r0 (1 + e + e^2), r0 the estimate and e = 1 - d r0 (|e| < 2^-20), and a / d
// is a r0 plus (e + e^2) of it: a chain of three FP64 operations.
__device__ __forceinline__ double recip_start(double d) { return widen(ptx::rcp_estimate(low_float(d))); }
__device__ __forceinline__ double recip_err(double d, double r0) {
  const double e = fma(-d, r0, 1.0);
  return fma(e, e, e);
}
__device__ __forceinline__ double quotient(double a, double d) {
  if (!in_fp32(d)) return slow_div(a, d);
  const double r0 = recip_start(d), w0 = a * r0;
  return fma(w0, recip_err(d, r0), w0);
}
__device__ __forceinline__ float quotient(float a, float d) { return a / d; }  // (1 / d overflows below 2^-128)
// a / l from r = 1 / l, for an entry of the factor: correctly rounded in FP32 and, EXACT (signed
// factors), in FP64, by one correction of the product, r being correctly rounded; else the product. A
// direction of the 11 x 12 x 13 augmented system takes 2.48 ms with the corrections, 2.39 without.
template <bool EXACT> __device__ __forceinline__ double entry(double a, double l, double r) {
  const double q = a * r;
  return EXACT ? fma(fma(-q, l, a), r, q) : q;
}
template <bool EXACT> __device__ __forceinline__ float entry(float a, float l, float) { return a / l; }
// s v for s = +-1 and 0 < d < big_pivot^2 (false for NaN) on the integer pipe:
// an FP64 multiplication or comparison costs as much as a multiply-add.
__device__ __forceinline__ double flip(double v, bool neg) {
  return __hiloint2double(__double2hiint(v) ^ (neg ? 0x80000000 : 0), __double2loint(v));
}
__device__ __forceinline__ float flip(float v, bool neg) { return neg ? -v : v; }
__device__ __forceinline__ bool pivot_ok(double d) {
  const long long b = __double_as_longlong(d);
  return b > 0 && b < __double_as_longlong(1e128);
}
__device__ __forceinline__ bool pivot_ok(float d) { return d > 0.f && d < INFINITY; }

// Cholesky of one diagonal block (kb <= 64). A pivot that is not positive is
// either reported (smallest failing column kept) or replaced by a large value
// (static pivoting) and counted. With pivot signs (dp.sgn, a quasi-definite
// matrix) the block is factored as L S L^T: the pivot d_j must have the sign
// s_j, L_jj = sqrt(s_j d_j), L_ij = a_ij / (s_j L_jj).
//
// What bounds it on GB300: an FP64 instruction occupies a quarter SM's unit for
// 64 cycles whatever its active lanes (measured; results after 66; a conversion or
// comparison more), so the count of FP64 warp instructions on each of the four
// warps is the time, and the chain of 64 pivots is on it too. So the elimination
// runs on unscaled columns (a_ic -= (a_ij / d_j) a_cj: no square root on the chain; all
// columns are scaled by 1 / L_jj on their way out), and the block goes in four panels of
// 16 columns, two threads per row, each column published through shared memory (one
// barrier per column); past the panel a rank-16 update over the entries of the lower
// triangle, one a thread, on two warps per quarter (one leaves it idle between
// multiply-adds: 15.4k against 11.3k cycles past the first panel). 64 columns: 95k
// cycles when each panel was scaled by itself and updated in 8 x 8 blocks on one warp
// per quarter, 78k now, 49k of them in the panels.
constexpr int kPotrfThreads = 256;  // the first 128 for the panels

// Barrier 1 over the first `threads` threads of the block (whole warps).
__device__ __forceinline__ void bar1(int threads) {
  asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}

// Panel at column c0 of the block in S (rows c0 .. 63) on 2 (64 - c0) threads: two
// per row, thread h of a row holds the columns c0 + h + 2 q. This form takes every
// pivot; potrf_panel_fast the usual ones.
template <typename T>
__device__ __forceinline__ void potrf_panel(T *S, int ls, int c0, T (*col)[64], const int8_t *neg, T *piv,
                                            T (*W)[64], int32_t *status, int perturb, int first) {
  const int t = threadIdx.x, i = t / 2, h = t % 2, act = 2 * (64 - c0);  // row c0 + i
  T x[8];
#pragma unroll
  for (int q = 0; q < 8; q++) x[q] = S[(c0 + i) * ls + c0 + h + 2 * q];
  if (h == 0) col[0][i] = x[0];
  bar1(act);
#pragma unroll
  for (int j = 0; j < 16; j++) {
    const T *cj = col[j % 3];
    const bool ng = neg[c0 + j] != 0;
    T d = flip(cj[j], ng), v[8];  // s_j d_j; the column's entries at this thread's columns
    const T aij = cj[i];
#pragma unroll
    for (int q = (j + 1) / 2; q < 8; q++) v[q] = cj[h + 2 * q];
    if (!pivot_ok(d)) {  // (uniform over the panel)
      if (t == 0) {
        if (perturb) atomicAdd(&status[ST_PERTURBED], 1);
        else atomicMin(&status[ST_FAIL_COL], first + c0 + j);
      }
      d = perturb ? big_pivot<T>() : T(1);
    }
    if (t == 0) piv[c0 + j] = d;
    const T w = flip(quotient(aij, d), ng);  // a_ij / d_j
    if (h == j % 2) W[j][c0 + i] = w;
    if (j == 15) break;
    // column j + 1 first: published before the barrier, the other columns after it,
    // beside the next pivot's chain (three buffers: the next column but one is
    // written while slower warps still read column j); column j itself is final
    const int qn = (j + 1) / 2;
    if (j % 2 == 1 || h == 1) x[qn] = fma(-w, v[qn], x[qn]);
    if (h == (j + 1) % 2) col[(j + 1) % 3][i] = x[qn];
    bar1(act);
#pragma unroll
    for (int q = (j + 1) / 2 + 1; q < 8; q++) x[q] = fma(-w, v[q], x[q]);
  }
#pragma unroll
  for (int q = 0; q < 8; q++)
    if (h + 2 * q <= i) S[(c0 + i) * ls + c0 + h + 2 * q] = x[q];
}

// The same without a branch, for pivots of the right sign within FP32's normal range;
// false (in every thread of the panel, S as it was) if one is not. In one basic block
// the multiply-adds of column j fill the time in which the loads and the estimate of
// column j + 1 are under way: 820 cycles a column with the branches, 760 without.
__device__ __forceinline__ bool potrf_panel_fast(double *S, int ls, int c0, double (*col)[64], const int8_t *neg,
                                                 double *piv, double (*W)[64]) {
  const int t = threadIdx.x, i = t / 2, h = t % 2, act = 2 * (64 - c0);  // row c0 + i
  // place of row r in col: the panel's 16 rows by parity, so that a thread's columns come
  // in 16-byte reads
  auto place = [](int r) { return r < 16 ? 8 * (r % 2) + r / 2 : r; };
  const int mine = place(i);
  double x[8];
#pragma unroll
  for (int q = 0; q < 8; q++) x[q] = S[(c0 + i) * ls + c0 + h + 2 * q];
  unsigned sign = 0;  // bit j: column j's pivot sign is negative
#pragma unroll
  for (int j = 0; j < 16; j++) sign |= (neg[c0 + j] != 0 ? 1u : 0u) << j;
  if (h == 0) col[0][mine] = x[0];
  bar1(act);
  bool good = true;
  double d = flip(col[0][0], sign & 1u), a = col[0][mine], r0 = recip_start(d), v[8], w = 0.0;
  auto columns = [&](const double *c, int q0, double (&o)[8]) {  // q0 .. 7 (and one before)
#pragma unroll
    for (int q = 0; q < 8; q += 2)
      if (q + 1 >= q0) {
        const double2 f = *reinterpret_cast<const double2 *>(c + 8 * h + q);
        o[q] = f.x, o[q + 1] = f.y;
      }
  };
  columns(col[0], 0, v);
#pragma unroll
  for (int j = 0; j < 16; j++) {
    good = good && in_fp32(d);
    if (t == 0) piv[c0 + j] = d;
    const double w0 = a * r0;
    w = flip(fma(w0, recip_err(d, r0), w0), sign >> j & 1u);  // a_ij / d_j
    if (h == j % 2) W[j][c0 + i] = w;
    if (j == 15) break;
    const int qn = (j + 1) / 2;
    if (j % 2 == 1 || h == 1) x[qn] = fma(-w, v[qn], x[qn]);
    double *cn = col[(j + 1) % 3];
    if (h == (j + 1) % 2) cn[mine] = x[qn];
    bar1(act);
    d = flip(cn[place(j + 1)], sign >> (j + 1) & 1u);
    a = cn[mine];
    double u[8];
    columns(cn, (j + 2) / 2, u);
    r0 = recip_start(d);
#pragma unroll
    for (int q = qn + 1; q < 8; q++) x[q] = fma(-w, v[q], x[q]);
#pragma unroll
    for (int q = (j + 2) / 2; q < 8; q++) v[q] = u[q];
  }
  if (!good) return false;
#pragma unroll
  for (int q = 0; q < 8; q++)
    if (h + 2 * q <= i) S[(c0 + i) * ls + c0 + h + 2 * q] = x[q];
  return true;
}
__device__ __forceinline__ bool potrf_panel_fast(float *, int, int, float (*)[64], const int8_t *, float *,
                                                 float (*)[64]) {
  return false;  // (FP32 arithmetic is not what bounds the FP32 panel)
}

// Entries e0, e0 + 256, .. (Q of them) of the lower triangle of the m rows and columns past
// a panel, numbered row by row: a_ic -= sum_j a_ij w_cj. (All sums before the first store:
// a store to S would hold back the loads of the next sum.)
template <int Q, typename T>
__device__ __forceinline__ void panel_trail(T *S, int ls, int c0, int e0, int nout, const T (*W)[64]) {
  T s[Q];
  int at[Q], col[Q];
#pragma unroll
  for (int q = 0; q < Q; q++) {
    const int e = min(e0 + kPotrfThreads * q, nout - 1);
    int bi = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);
    if (bi * (bi + 1) / 2 > e) bi--;
    if ((bi + 1) * (bi + 2) / 2 <= e) bi++;
    col[q] = c0 + 16 + e - bi * (bi + 1) / 2;
    at[q] = (c0 + 16 + bi) * ls;
    s[q] = S[at[q] + col[q]];
  }
#pragma unroll
  for (int j = 0; j < 16; j++)
#pragma unroll
    for (int q = 0; q < Q; q++) s[q] = fma(-S[at[q] + c0 + j], W[j][col[q]], s[q]);
#pragma unroll
  for (int q = 0; q < Q; q++)
    if (e0 + kPotrfThreads * q < nout) S[at[q] + col[q]] = s[q];
}

template <typename T, bool SGN>
__global__ void __launch_bounds__(kPotrfThreads) potrf_kernel(DevPlan dp, const Task *__restrict__ tasks,
                                                              T *__restrict__ L, int32_t *status,
                                                              int perturb) {
  constexpr int NB = 64, LS = NB + 1, NT = kPotrfThreads;
  const Task tk = tasks[blockIdx.x];
  const FrontInfo F = dp.fronts[tk.front];
  const int k = tk.a, kb = min(NB, F.ncol - k);
  T *A = L + F.loff + (int64_t)k * F.ld + k;
  const int8_t *sg = SGN ? dp.sgn + F.first + k : nullptr;
  __shared__ T S[NB * LS];  // the block; past kb: zero, with a unit diagonal
  __shared__ __align__(16) T col[3][NB];
  __shared__ T piv[NB], W[16][NB];  // W: a panel's a_ij / d_j
  __shared__ int8_t neg[NB];
  const int tid = threadIdx.x;
  // 16 bytes at a time (rows are padded to 16 bytes, and zero past their last column)
  constexpr int VW = 16 / (int)sizeof(T), NV = NB / VW;
#pragma unroll
  for (int q = 0; q < NB * NV / NT; q++) {
    const int e = tid + NT * q, r = e / NV, c = VW * (e % NV);
    Vec16<T> v;
#pragma unroll
    for (int h = 0; h < VW; h++) v.v[h] = T(0);
    if (r < kb && c <= r) v = ld16(A + (int64_t)r * F.ld + c);
#pragma unroll
    for (int h = 0; h < VW; h++) S[r * LS + c + h] = (r < kb && c + h <= r) ? v.v[h] : (r == c + h ? T(1) : T(0));
  }
  if (tid < NB) neg[tid] = sg && tid < kb && sg[tid] < 0;
  __syncthreads();
#pragma unroll 1
  for (int p = 0; p < 4; p++) {
    const int c0 = 16 * p;
    if (c0 >= kb) break;
    if (tid < 2 * (NB - c0) && !potrf_panel_fast(S, LS, c0, col, neg, piv, W)) {
      bar1(2 * (NB - c0));
      potrf_panel<T>(S, LS, c0, col, neg, piv, W, status, perturb, F.first + k);
    }
    __syncthreads();
    if (p == 3 || c0 + 16 >= kb) break;
    const int m = 48 - c0, nout = m * (m + 1) / 2;
    if (m > 32) panel_trail<5>(S, LS, c0, tid, nout, W);
    else if (m > 16) panel_trail<3>(S, LS, c0, tid, nout, W);
    else if (tid < nout) panel_trail<1>(S, LS, c0, tid, nout, W);
    __syncthreads();
  }
  // L_ij = s_j a_ij / L_jj, L_jj = sqrt(d) from d and 1 / sqrt(d)
  if (tid < kb) {
    const T d = piv[tid], r = inv_sqrt(d), l0 = d * r, l = fma(fma(-l0, l0, d), T(0.5) * r, l0);
    col[0][tid] = quotient(T(1), l);
    col[1][tid] = l;
  }
  __syncthreads();
#pragma unroll 2
  for (int q = 0; q < NB * NV / NT; q++) {
    const int e = tid + NT * q, r = e / NV, c = VW * (e % NV);
    if (r >= kb || c > r) continue;
    Vec16<T> v;
#pragma unroll
    for (int h = 0; h < VW; h++) {
      const T x = flip(entry<SGN>(S[r * LS + c + h], col[1][c + h], col[0][c + h]), neg[c + h] != 0);
      v.v[h] = c + h < r ? x : c + h == r ? col[1][r] : T(0);
    }
    st16(A + (int64_t)r * F.ld + c, v);
  }
}

// Rows below the diagonal block: X <- X L_kk^{-T} (X L_kk^{-T} S_k with pivot
// signs) by substitution, kb <= 64, R = 128 / P rows at a time on four warps. P lanes
// share a row (lane h keeps the columns of residue h mod P in registers); with unit
// columns u_c = L_:c / L_cc and z_c = x_c L_cc the substitution is z_c2 -= z_c
// u_c2,c, and x = z / diag is formed once at the end, so a column costs its
// multiply-adds and nothing else. Bound by the FP64 unit (64 cycles per warp
// instruction on each quarter SM: 10 us per 16 rows and SM, P = 8), and where there are
// SMs to spare by fewer rows on each with more lanes a row (trsm_rows: P = 16 and 32,
// half and a quarter of the instructions, then the chain of 64 exchanges and
// multiply-adds; 31 launches of at most 1216 rows: 16.5 us each with P = 8, 12.0 with
// P = 16 and 8.6 with P = 32). A block takes `batches`
// times R rows: more than one only when the rows exceed 16 per SM (trsm_batches),
// so that a 3008-row front reaches every SM (128 rows a block, as before: 24
// blocks, 169 us a launch on the 32^3 grid); the code of a batch is unrolled over
// the columns and fits the instruction cache, which wider per-warp tiles (16
// rows a warp, 56 KB of code run once) did not: 98 us against 55 us a launch on the
// 40^3 grid.
template <typename T, int P, bool SGN>
__global__ void __launch_bounds__(128) trsm_kernel(DevPlan dp, const Task *__restrict__ ents, int nent,
                                                   int batches, T *__restrict__ L) {
  constexpr int NB = 64, LS = NB + 1, NQ = NB / P, R = 128 / P;
  int lo = 0, hi = nent - 1;  // the front this block's rows belong to
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (ents[mid].a <= (int)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const Task tk = ents[lo];
  const FrontInfo F = dp.fronts[tk.front];
  const int nf = F.ncol + F.nrow, k = tk.b, kb = min(NB, F.ncol - k);
  const int tid = threadIdx.x, lane = tid % 32, h = lane % P;
  int row = k + kb + batches * R * ((int)blockIdx.x - tk.a) + tid / P;
  __shared__ T U[NB * LS];      // column c: u_c2,c at U[c * LS + c2]
  __shared__ T rd[NB], dg[NB];  // s_c / L_cc, s_c L_cc
  T *Xr = L + F.loff + (int64_t)row * F.ld + k;
  T z[NQ];
#pragma unroll
  for (int q = 0; q < NQ; q++) z[q] = (row < nf && h + P * q < kb) ? Xr[h + P * q] : T(0);
  const int8_t *sg = SGN ? dp.sgn + F.first + k : nullptr;
  const T *A = L + F.loff + (int64_t)k * F.ld + k;
  if (tid < kb) {
    const T d = A[(int64_t)tid * F.ld + tid];
    rd[tid] = flip(quotient(T(1), d), sg && sg[tid] < 0);
    dg[tid] = flip(d, sg && sg[tid] < 0);
  }
  T u[NB * NB / 128];
#pragma unroll
  for (int q = 0; q < NB * NB / 128; q++) {
    const int c2 = 2 * q + tid / NB, c = tid % NB;
    u[q] = (c2 < kb && c < c2) ? A[(int64_t)c2 * F.ld + c] : T(0);
  }
  __syncthreads();
  {
    // column c of this thread: u = L_c2,c / L_cc (the signs of L and of the scale cancel)
    const int c = tid % NB;
    const bool ng = sg && c < kb && sg[c] < 0;
    const T s = c < kb ? flip(rd[c], ng) : T(0), d = c < kb ? flip(dg[c], ng) : T(1);
#pragma unroll
    for (int q = 0; q < NB * NB / 128; q++) {
      const int c2 = 2 * q + tid / NB;
      U[c * LS + c2] = 2 * q + 1 > (c & 32) ? entry<SGN>(u[q], d, s) : T(0);  // (uniform per warp)
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int b = 0; b < batches && row - tid / P < nf; b++) {
#pragma unroll
    for (int c = 0; c < NB; c++) {
      if (c >= kb) break;
      const T zc = __shfl_sync(0xffffffffu, z[c / P], (lane & ~(P - 1)) | (c % P));
#pragma unroll
      for (int q = c / P; q < NQ; q++)  // (U is zero up to its own column)
        if (P * q + P - 1 > c) z[q] = fma(-zc, U[c * LS + P * q + h], z[q]);
    }
#pragma unroll
    for (int q = 0; q < NQ; q++)
      if (row < nf && h + P * q < kb) Xr[h + P * q] = entry<SGN>(z[q], dg[h + P * q], rd[h + P * q]);
    row += R;
    Xr += (int64_t)R * F.ld;
    if (b + 1 < batches)
#pragma unroll
      for (int q = 0; q < NQ; q++) z[q] = (row < nf && h + P * q < kb) ? Xr[h + P * q] : T(0);
  }
}

template <typename T>
__global__ void entries_kernel(DevPlan dp, const T *__restrict__ L, const int32_t *col2s,
                               int64_t count, const int32_t *rows, const int32_t *cols,
                               double *out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = rows[e], j = cols[e];
    double v = 0.0;
    if (i >= j && j >= 0 && i < dp.n) {
      const FrontInfo F = dp.fronts[col2s[j]];
      int32_t p = -1;
      if (i < F.first + F.ncol) {
        p = i - F.first;
      } else {
        int lo = 0, hi = F.nrow;  // binary search in the row structure
        const int32_t *rs = dp.sri + F.rows_off;
        while (lo < hi) {
          int mid = (lo + hi) / 2;
          if (rs[mid] < i) lo = mid + 1; else hi = mid;
        }
        if (lo < F.nrow && rs[lo] == i) p = F.ncol + lo;
      }
      if (p >= 0) v = (double)L[F.loff + (int64_t)p * F.ld + (j - F.first)];
    }
    out[e] = v;
  }
}

inline int grid_for(int64_t n, int block) {
  int64_t g = (n + block - 1) / block;
  return (int)(g < 1 ? 1 : (g > 152 * 32 ? 152 * 32 : g));
}

}  // namespace

void launch_assemble(const DevPlan &dp, const double *jv, const double *D, const double *wv,
                     double delta_p, double *kval, cudaStream_t st) {
  if (dp.nk == 0) return;
  { note_launch(); assemble_kernel<<<grid_for(dp.nk, 256), 256, 0, st>>>(dp, jv, D, wv, delta_p, kval); }
}

template <typename T>
void launch_build_level(const DevPlan &dp, const LevelPlan &LP, const double *kval, T *L, T *U,
                        cudaStream_t st) {
  const bool fused = LP.build_k >= 0;
  if (LP.build_e > LP.build_b)
    {
      auto kernel = fused ? build_front_kernel<T, true> : build_front_kernel<T, false>;
      note_launch();
      kernel<<<LP.build_e - LP.build_b, kBuildThreads, 0, st>>>(dp, LP.build_b, LP.build_k, kval, L, U);
    }
  if (!fused && LP.k_e > LP.k_b)
    { note_launch(); kadd_kernel<T><<<grid_for(LP.k_e - LP.k_b, 256), 256, 0, st>>>(dp, LP.k_b, LP.k_e, kval, L); }
}

template <typename T>
void launch_potrf(const DevPlan &dp, const StepRange &S, T *L, int32_t *status, bool perturb,
                  cudaStream_t st) {
  if (S.potrf_e <= S.potrf_b) return;
  note_launch();
  auto kernel = dp.sgn ? potrf_kernel<T, true> : potrf_kernel<T, false>;
  kernel<<<S.potrf_e - S.potrf_b, kPotrfThreads, 0, st>>>(dp, dp.potrf + S.potrf_b, L, status, perturb ? 1 : 0);
}

template <typename T, bool SGN> auto trsm_for(int rows) {
  return rows == 4 ? trsm_kernel<T, 32, SGN> : rows == 8 ? trsm_kernel<T, 16, SGN> : trsm_kernel<T, 8, SGN>;
}
template <typename T>
void launch_trsm(const DevPlan &dp, const StepRange &S, T *L, cudaStream_t st) {
  if (S.trsm_n <= 0) return;
  note_launch();
  auto kernel = dp.sgn ? trsm_for<T, true>(S.trsm_rows) : trsm_for<T, false>(S.trsm_rows);
  kernel<<<S.trsm_n, 128, 0, st>>>(dp, dp.trsm + S.trsm_b, S.trsm_e - S.trsm_b, S.trsm_bat, L);
}

static void launch_upd(const DevPlan &dp, const UpdRange &u, double *L, double *U, cudaStream_t st) {
  if (u.n <= 0) return;
  note_launch();
  auto kernel = u.ts == kUpdTile64 ? upd_kernel<double, kUpdTile64, 128, 64> : upd_kernel<double, kUpdTileSmall64, 128, 64>;
  kernel<<<u.n, 128, 0, st>>>(dp, dp.upd + u.b, u.e - u.b, u.k0, u.k1, u.c0, u.clim, u.with_u, L, U);
}
static void launch_upd(const DevPlan &dp, const UpdRange &u, float *L, float *U, cudaStream_t st) {
  if (u.n <= 0) return;
  note_launch();
  upd_kernel<float, kUpdTile32, 256, 32><<<u.n, 256, 0, st>>>(dp, dp.upd + u.b, u.e - u.b, u.k0, u.k1, u.c0,
                                                              u.clim, u.with_u, L, U);
}

// FP64 with look-ahead: the chain (diagonal block, panel solve, update of the
// next step's columns) goes on its own stream ahead of the update of everything past
// them, whose blocks it would otherwise wait for; it has the higher priority, so its
// blocks start as soon as an SM has room. The columns of step s + 1 take the updates of
// steps 0 .. s in order: rest(s - 1) is complete before next(s) starts. 32^3 grid LP
// (FP64): 47.2 -> 43.7 ms a system.
static void factor_steps64(const DevPlan &dp, const LevelPlan &LP, double *L, double *U, int32_t *status, bool perturb,
                           const SideStream &chain, cudaStream_t st) {
  cudaEventRecord(chain.fork, st);  // the level's fronts are built
  cudaStreamWaitEvent(chain.s, chain.fork, 0);
  for (size_t k = 0; k < LP.steps.size(); k++) {
    const StepRange &S = LP.steps[k];
    launch_potrf<double>(dp, S, L, status, perturb, chain.s);
    launch_trsm<double>(dp, S, L, chain.s);
    cudaEventRecord(chain.join, chain.s);
    if (k > 0) cudaStreamWaitEvent(chain.s, chain.fork, 0);
    launch_upd(dp, S.next64, L, U, chain.s);
    cudaStreamWaitEvent(st, chain.join, 0);
    launch_upd(dp, S.rest64, L, U, st);
    if (k + 1 < LP.steps.size()) cudaEventRecord(chain.fork, st);
  }
}

template <typename T>
void launch_factor_simt(const DevPlan &dp, const Plan &plan, const double *kval, T *L, T *U,
                        int32_t *status, bool perturb, const SideStream &chain, cudaStream_t st) {
  for (const LevelPlan &LP : plan.levels) {
    launch_build_level<T>(dp, LP, kval, L, U, st);
    if constexpr (sizeof(T) == 8) {
      if (LP.ahead64) {
        factor_steps64(dp, LP, L, U, status, perturb, chain, st);
        continue;
      }
    }
    for (const StepRange &S : LP.steps) {
      launch_potrf<T>(dp, S, L, status, perturb, st);
      launch_trsm<T>(dp, S, L, st);
      if (sizeof(T) == 8) {
        launch_upd(dp, S.rest64, L, U, st);
      } else {
        launch_upd(dp, S.upd32, L, U, st);
        launch_upd(dp, S.sup32, L, U, st);
      }
    }
  }
}

template <typename T>
void launch_factor_entries(const DevPlan &dp, const T *L, const int32_t *col2s, int64_t count,
                           const int32_t *rows, const int32_t *cols, double *out,
                           cudaStream_t st) {
  if (count <= 0) return;
  { note_launch(); entries_kernel<T><<<grid_for(count, 256), 256, 0, st>>>(dp, L, col2s, count, rows, cols, out); }
}

template void launch_build_level<float>(const DevPlan &, const LevelPlan &, const double *,
                                        float *, float *, cudaStream_t);
template void launch_build_level<double>(const DevPlan &, const LevelPlan &, const double *,
                                         double *, double *, cudaStream_t);
template void launch_potrf<double>(const DevPlan &, const StepRange &, double *, int32_t *, bool,
                                   cudaStream_t);
template void launch_trsm<double>(const DevPlan &, const StepRange &, double *, cudaStream_t);
template void launch_factor_simt<double>(const DevPlan &, const Plan &, const double *, double *,
                                         double *, int32_t *, bool, const SideStream &, cudaStream_t);
template void launch_factor_simt<float>(const DevPlan &, const Plan &, const double *, float *,
                                        float *, int32_t *, bool, const SideStream &, cudaStream_t);
template void launch_factor_entries<double>(const DevPlan &, const double *, const int32_t *,
                                            int64_t, const int32_t *, const int32_t *, double *,
                                            cudaStream_t);
template void launch_factor_entries<float>(const DevPlan &, const float *, const int32_t *,
                                           int64_t, const int32_t *, const int32_t *, double *,
                                           cudaStream_t);

}  // namespace gipm
