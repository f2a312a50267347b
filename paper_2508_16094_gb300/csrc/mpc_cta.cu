// Batched MPC QPs in FP64: one CTA of four warps per instance (Sec. 6, batch
// solvers; the method of mpc_batch.cu: KKT conditions (2), Newton system (3)
// condensed to (5), block tridiagonal with 16 x 16 blocks over the stages).
//
// What bounds it: an FP64 instruction occupies a quarter SM for 64 cycles whatever
// its active lanes, so the kernel is the count of FP64 warp instructions, and for a
// small batch the chain over the stages. With 16 lanes per instance (as the FP32
// variant still runs) the two instances of a warp diverge and every 16 x 16 block
// was assembled and factored by rows with most lanes idle. Here
//  - elementwise work runs over (stage, variable) pairs, eight stages at a time;
//  - the blocks use J's structure: with M_k = [B_k A_k] and Dbar_k = D+ + D- of the
//    dynamics pairs, K's blocks are sums of G_k = M_k^T Dbar_k M_k and Dbar_k M_k, one
//    entry of the lower triangle per thread;
//  - a block is factored as U Delta U^T (U unit lower): no square roots, one
//    quotient per column, and the couplings Y = K_{k,k-1} U^{-T} keep their 12
//    non-zero columns;
//  - multipliers of a dynamics pair enter J^T only through their difference, kept as
//    one vector.
// One warp runs the pivot chain and the substitutions; the SM's other CTAs fill the
// FP64 unit meanwhile (five a SM: 46.1 ms for 4096 instances of 10 to 100 stages; four,
// without register spills, 49.7; three 58.5). 16 lanes per instance took 180 ms with
// the default shape (120 with the autotuned one), and 68 ms against 10.4 for 96 instances.
#include <cmath>
#include <stdexcept>
#include <type_traits>

#include "mpc_batch.h"

namespace gipm {

namespace {

constexpr int NX = 12, NU = 4, NS = 16, SLOT = 64, kThreads = 128;
constexpr int kRing = 4, kRingStage = 256 + 192 + 16;  // U, Y and a vector of one stage

struct Shared {
  double M[NX][NS];      // M_{k+1}
  double DM[2][NX][NS];  // Dbar M of stages k + 1 and k (by parity)
  double S[NS][NS + 1];
  double U[NS][NS + 1];       // of the stage just factored (strictly lower)
  double di[NS];              // 1 / Delta
  double Y[NS][NX + 1], Ys[NS][NX + 1];  // coupling to the stage before, and Y / Delta
  double Ko[NU][NX];          // rows u of the next coupling block
  double db[2][NX], col[3][NS], piv[NS];
  alignas(16) double ring[kRing][kRingStage];
  double xs[NS];
  double red[4][6];
  int inst, ok;
};

// Vectors of one instance in the workspace (16 doubles per stage, or SLOT with slot
// 16 * kind + i; kinds: dynamics h >= 0 and -h >= 0 (i < 12), lower bound, upper bound).
struct Inst {
  int T;
  const double *A, *B, *Q, *R, *x0;
  double *z, *dz, *rhs, *q, *lamd, *td;  // lamd, td: differences over the dynamics pairs
  double *s, *lam, *D, *aux, *ds, *dl, *il;
  double *U, *Y;  // 256 per stage: U row-major with 1 / Delta on its diagonal; Y 16 x 12
};
// aux: h (0 .. 11), Dbar (16 .. 27), diagonal of K without delta_p (32 .. 47), scratch (48 .. 63)

__device__ Inst make_inst(const MpcArgs &a, int inst) {
  Inst I;
  const int64_t s0 = a.soff[inst];
  I.T = a.T[inst];
  I.A = a.A + s0 * NX * NX;
  I.B = a.B + s0 * NX * NU;
  I.Q = a.Q + (int64_t)inst * NX;
  I.R = a.R + (int64_t)inst * NU;
  I.x0 = a.x0 + (int64_t)inst * NX;
  const int64_t T = I.T;
  double *p = a.work + s0 * kMpcStageDoubles;
  auto take = [&](int64_t per) {
    double *r = p;
    p += T * per;
    return r;
  };
  I.z = take(NS);
  I.dz = take(NS);
  I.rhs = take(NS);
  I.q = take(NS);
  I.lamd = take(NS);
  I.td = take(NS);
  I.s = take(SLOT);
  I.lam = take(SLOT);
  I.D = take(SLOT);
  I.aux = take(SLOT);
  I.ds = take(SLOT);
  I.dl = take(SLOT);
  I.il = take(SLOT);
  take(SLOT);
  I.U = take(256);
  I.Y = take(256);
  return I;
}

__device__ __forceinline__ long long bits(double v) { return __double_as_longlong(v); }
// |v|, NaN as zero (the maxima skip NaN, the sums do not), and comparisons of
// non-negative values, on the integer pipe
__device__ __forceinline__ double abs_or_zero(double v) {
  const long long b = bits(v) & 0x7FFFFFFFFFFFFFFFll;
  return b > 0x7FF0000000000000ll ? 0.0 : __longlong_as_double(b);
}
__device__ __forceinline__ double max_pos(double a, double b) { return bits(a) > bits(b) ? a : b; }
__device__ __forceinline__ double min_pos(double a, double b) { return bits(a) < bits(b) ? a : b; }
__device__ __forceinline__ double neg(double v) { return __longlong_as_double(bits(v) ^ (1ll << 63)); }

// 1 / d for d > 0: FP32 estimate (converted by moving bits) and a second-order
// step, r0 (1 + e + e^2), e = 1 - d r0; values outside FP32's normal range divide.
__device__ __noinline__ double slow_recip(double d) { return 1.0 / d; }
__device__ __forceinline__ bool in_fp32(double d) {
  return ((unsigned)__double2hiint(d) >> 20) - 904u < 239u;  // 2^-119 <= d < 2^120
}
__device__ __forceinline__ double recip_estimate(double d) {
  const float f = __int_as_float(((__double2hiint(d) - (896 << 20)) << 3) | ((unsigned)__double2loint(d) >> 29));
  const int b = __float_as_int(__fdividef(1.f, f));
  return __hiloint2double((b >> 3) + (896 << 20), b << 29);
}
__device__ __forceinline__ double recip(double d) {
  if (!in_fp32(d)) return slow_recip(d);
  const double r0 = recip_estimate(d), e = fma(-d, r0, 1.0);
  return fma(r0, fma(e, e, e), r0);
}
__device__ __noinline__ double slow_div(double a, double d) { return a / d; }
__device__ __forceinline__ double quotient(double a, double d) {
  if (!in_fp32(d) || !in_fp32(a)) return slow_div(a, d);  // (an infinite a stays infinite)
  const double r0 = recip_estimate(d), w0 = a * r0, e = fma(-d, r0, 1.0);
  return fma(w0, fma(e, e, e), w0);
}

// a / b < c / d of values >= 0 by cross products, by division where one of them may have left
// FP64's range
__device__ __noinline__ bool slow_less(double a, double b, double c, double d) { return a / b < c / d; }
__device__ __forceinline__ bool ratio_less(double a, double b, double c, double d) {
  const double p = a * d, q = c * b;
  auto ordinary = [](double v) { return ((unsigned)__double2hiint(v) >> 20) - 100u < 1800u; };
  if (!ordinary(p) || !ordinary(q)) return slow_less(a, b, c, d);
  return bits(p) < bits(q);
}

constexpr int R_SUM = 0, R_MAX = 1, R_MIN = 2;  // max and min of non-negative values
template <int OP> __device__ __forceinline__ double combine(double a, double b) {
  return OP == R_SUM ? a + b : (OP == R_MAX ? max_pos(a, b) : min_pos(a, b));
}
template <int OP> __device__ __forceinline__ double warp_reduce(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = combine<OP>(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}
// Reductions over the CTA, the results in every thread.
template <int... OPS> __device__ __forceinline__ void cta_reduce(Shared &S, double (&v)[sizeof...(OPS)]) {
  {
    int k = 0;
    ((v[k] = warp_reduce<OPS>(v[k]), k++), ...);
  }
  __syncthreads();  // (the previous results have been read)
  if (threadIdx.x % 32 == 0)
#pragma unroll
    for (int k = 0; k < (int)sizeof...(OPS); k++) S.red[threadIdx.x / 32][k] = v[k];
  __syncthreads();
  {
    int k = 0;
    auto all = [&](auto op) {
      constexpr int OP = decltype(op)::value;
      v[k] = combine<OP>(combine<OP>(S.red[0][k], S.red[1][k]), combine<OP>(S.red[2][k], S.red[3][k]));
      k++;
    };
    (all(std::integral_constant<int, OPS>{}), ...);
  }
}

__device__ __forceinline__ double wdiag(const Inst &I, int i) { return i < NU ? I.R[i] : I.Q[i - NU]; }

// (J v)_h of row i < 12 of stage k: v_{x_{k+1}} - A_k v_{x_k} - B_k v_{u_k} (x0: x_0, or
// nullptr for a direction)
__device__ __forceinline__ double dyn_row(const Inst &I, const double *v, const double *x0, int k, int i) {
  const double *vk = v + k * NS, *Ar = I.A + (int64_t)k * NX * NX + i * NX, *Br = I.B + (int64_t)k * NX * NU + i * NU;
  double h0 = vk[NU + i], h1 = 0.0;
  const double *xp = k > 0 ? vk - NS + NU : x0;
  if (xp)
#pragma unroll
    for (int j = 0; j < NX; j += 2) {
      h0 = fma(-Ar[j], xp[j], h0);
      h1 = fma(-Ar[j + 1], xp[j + 1], h1);
    }
#pragma unroll
  for (int j = 0; j < NU; j += 2) {
    h0 = fma(-Br[j], vk[j], h0);
    h1 = fma(-Br[j + 1], vk[j + 1], h1);
  }
  return h0 + h1;
}
// -(coefficients of variable i of stage k in the dynamics rows it enters other than as
// x_{k+1}) . d: B_k's column i, or A_{k+1}'s column i - 4 with stage k + 1's values (d: 16
// per stage, 12 used)
__device__ __forceinline__ double dyn_col(const Inst &I, const double *d, int k, int i) {
  const bool u = i < NU;
  if (!u && k + 1 >= I.T) return 0.0;
  const double *c = u ? I.B + (int64_t)k * NX * NU + i : I.A + (int64_t)(k + 1) * NX * NX + (i - NU);
  const double *r = d + (u ? k : k + 1) * NS;
  const int st = u ? NU : NX;
  double a0 = 0.0, a1 = 0.0;
#pragma unroll
  for (int j = 0; j < NX; j += 2) {
    a0 = fma(-c[j * st], r[j], a0);
    a1 = fma(-c[(j + 1) * st], r[j + 1], a1);
  }
  return a0 + a1;
}

// K's block factorisation (see the head of the file) with regularisation delta_p;
// false if a pivot is not in (0, 1e64).
__device__ __noinline__ bool factor(Shared &S, const Inst &I, double delta_p) {
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32, T = I.T;
  // this thread's entry of the lower triangle: 120 off-diagonal, then two diagonal ones
  int ei, ej, ei2 = -1;
  if (tid < 120) {
    ei = 1;
    ej = tid;
    while (ej >= ei) ej -= ei++;
  } else {
    ei = ej = 2 * (tid - 120);
    ei2 = ei + 1;
  }
  double m[2], d[2];                       // prefetched entries of M and Dbar
  double bnext[2] = {0.0, 0.0}, bcur[2];   // K's diagonal (the last eight threads)
  auto fetch = [&](int k) {  // stage k's M and Dbar, entries tid and tid + 128 of 192
    if (k >= T) return;
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int e = tid + kThreads * h, r = e / NS, c = e % NS;
      if (e < NX * NS) {
        m[h] = c < NU ? I.B[(int64_t)k * NX * NU + r * NU + c] : I.A[(int64_t)k * NX * NX + r * NX + c - NU];
        d[h] = I.aux[k * SLOT + 16 + r];
      }
    }
    if (tid >= 120) {
      bnext[0] = I.aux[k * SLOT + 32 + ei];
      bnext[1] = I.aux[k * SLOT + 32 + ei2];
    }
  };
  fetch(0);
  if (tid == 0) S.ok = 1;
  double g_old[2] = {0.0, 0.0};  // G_k's entries of columns u
  for (int k = -1; k < T; k++) {
    const int par = (k + 1) & 1;
    const bool next = k + 1 < T;
    if (next) {
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int e = tid + kThreads * h, r = e / NS, c = e % NS;
        if (e < NX * NS) {
          S.M[r][c] = m[h];
          S.DM[par][r][c] = d[h] * m[h];
          if (c == 0) S.db[par][r] = d[h];
        }
      }
    }
    bcur[0] = bnext[0];
    bcur[1] = bnext[1];
    __syncthreads();
    // G_{k+1}'s entry and with it the entry of stage k's block, K_kk - Y Delta^{-1} Y^T
    auto entry = [&](int i, int j, int w) {
      double g = 0.0, g1 = 0.0;
      if (next)
#pragma unroll
        for (int r = 0; r < NX; r += 2) {
          g = fma(S.M[r][i], S.DM[par][r][j], g);
          g1 = fma(S.M[r + 1][i], S.DM[par][r + 1][j], g1);
        }
      g += g1;
      if (k >= 0) {
        double v = j >= NU ? g : (i < NU ? g_old[w] : neg(S.DM[par ^ 1][i - NU][j]));
        if (i == j) {
          v += S.piv[i] + delta_p;
          if (i >= NU) v += S.db[par ^ 1][i - NU];
        }
        if (k > 0) {
          double a0 = 0.0, a1 = 0.0;
#pragma unroll
          for (int c = 0; c < NX; c += 2) {
            a0 = fma(S.Y[i][c], S.Ys[j][c], a0);
            a1 = fma(S.Y[i][c + 1], S.Ys[j][c + 1], a1);
          }
          v -= a0 + a1;
        }
        S.S[i][j] = v;
      }
      if (j < NU) {
        g_old[w] = g;
        if (i >= NU && next) S.Ko[j][i - NU] = g;
      }
    };
    entry(ei, ej, 0);
    if (ei2 >= 0) entry(ei2, ei2, 1);
    __syncthreads();
    if (tid >= 120) {  // the diagonal of stage k + 1, read in the next pass
      S.piv[ei] = bcur[0];
      S.piv[ei2] = bcur[1];
    }
    fetch(k + 2);
    if (k < 0) continue;
    // S = U Delta U^T on one warp: lane (row lane / 2, columns lane % 2 + 2 q)
    if (warp == 0) {
      const int i = lane / 2, h = lane % 2;
      double x[8], u[8], r_i = 0.0;
#pragma unroll
      for (int q = 0; q < 8; q++) x[q] = h + 2 * q <= i ? S.S[i][h + 2 * q] : 0.0;
      if (h == 0) S.col[0][i] = x[0];
      __syncwarp();
      bool good = true;
#pragma unroll
      for (int j = 0; j < NS; j++) {
        const double *cj = S.col[j % 3];
        double p = cj[j], v[8];
        const double aij = cj[i];
#pragma unroll
        for (int q = (j + 1) / 2; q < 8; q++) v[q] = cj[h + 2 * q];
        if (!(bits(p) > 0 && bits(p) < bits(1e64))) {  // (uniform)
          good = false;
          p = 1.0;
        }
        double w;  // a_ij / p, and 1 / p on the pivot's own row
        if (in_fp32(p)) {
          const double r0 = recip_estimate(p), a = i == j ? 1.0 : aij, w0 = a * r0, e = fma(-p, r0, 1.0);
          w = fma(w0, fma(e, e, e), w0);
        } else {
          w = (i == j ? 1.0 : aij) * slow_recip(p);
        }
        if (i == j) r_i = w;
        if (h == j % 2) u[j / 2] = i > j ? w : 0.0;
        if (j + 1 < NS) {
          const int qn = (j + 1) / 2;
          if (j % 2 == 1 || h == 1) x[qn] = fma(-w, v[qn], x[qn]);
          if (h == (j + 1) % 2) S.col[(j + 1) % 3][i] = x[qn];
          __syncwarp();
#pragma unroll
          for (int q = (j + 1) / 2 + 1; q < 8; q++) x[q] = fma(-w, v[q], x[q]);
        }
      }
      double *out = I.U + (int64_t)k * 256 + i * NS;
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const int c = h + 2 * q;
        S.U[i][c] = u[q];
        out[c] = c == i ? r_i : u[q];
      }
      if (h == 0) S.di[i] = r_i;
      if (!good && lane == 0) S.ok = 0;
    }
    __syncthreads();
    if (!S.ok) return false;
    // Y_{k+1} = K_{k+1,k} U^{-T} on columns x: row tid / 4, columns tid % 4 + 4 q
    if (next && tid < 64) {
      const int i = tid / 4, h = tid % 4;
      double y[3];
#pragma unroll
      for (int q = 0; q < 3; q++) y[q] = i < NU ? S.Ko[i][h + 4 * q] : neg(S.DM[par][i - NU][NU + h + 4 * q]);
#pragma unroll
      for (int c = 0; c < NX; c++) {
        const double yc = __shfl_sync(0xffffffffu, y[c / 4], (lane & ~3) | (c % 4));
#pragma unroll
        for (int q = c / 4; q < 3; q++)  // (U is zero on and above its diagonal)
          if (4 * q + 3 > c) y[q] = fma(-yc, S.U[NU + h + 4 * q][NU + c], y[q]);
      }
      double *out = I.Y + (int64_t)(k + 1) * 256 + i * NX;
#pragma unroll
      for (int q = 0; q < 3; q++) {
        const int c = h + 4 * q;
        S.Y[i][c] = y[q];
        S.Ys[i][c] = y[q] * S.di[NU + c];
        out[c] = y[q];
      }
    }
    // (the barrier of the next pass orders Y, Ys before their use)
  }
  __syncthreads();
  return true;
}

// Copies U, Y and one vector of stage k into the ring (16-byte asynchronous copies).
__device__ __forceinline__ void ring_load(Shared &S, const Inst &I, const double *vec, int k) {
  double *dst = S.ring[k & (kRing - 1)];
  for (int e = threadIdx.x; e < kRingStage / 2; e += kThreads) {
    const double *src = e < 128 ? I.U + (int64_t)k * 256 + 2 * e
                        : e < 224 ? I.Y + (int64_t)k * 256 + 2 * (e - 128)
                                  : vec + k * NS + 2 * (e - 224);
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst + 2 * e);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N> __device__ __forceinline__ void ring_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
  __syncthreads();
}

// dz = K^{-1} rhs with the block factor: q_k = Delta^{-1} U^{-1} (r_k - Y_k q_{k-1}), then
// x_k = U^{-T} (q_k - Delta^{-1} Y_{k+1}^T x_{k+1}). The substitutions run on warp 0, lane
// (row lane / 2, half lane % 2); all warps keep the ring filled.
__device__ __noinline__ void solve(Shared &S, const Inst &I) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, i = lane / 2, h = lane % 2, T = I.T;
#pragma unroll
  for (int k = 0; k < kRing - 1; k++) {
    if (k < T) ring_load(S, I, I.rhs, k);
    else asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int k = 0; k < T; k++) {
    ring_wait<kRing - 2>();  // stage k has landed; every thread is done with stage k - 1
    if (k + kRing - 1 < T) ring_load(S, I, I.rhs, k + kRing - 1);
    else asm volatile("cp.async.commit_group;" ::: "memory");
    if (warp != 0) continue;
    const double *U = S.ring[k & (kRing - 1)], *Y = U + 256, *r = Y + 192;
    double u[15];
#pragma unroll
    for (int c = 0; c < 15; c++) u[c] = i > c ? U[i * NS + c] : 0.0;
    const double di = U[i * NS + i];
    double t = h == 0 ? r[i] : 0.0, t1 = 0.0;
    if (k > 0)
#pragma unroll
      for (int m = 0; m < 6; m += 2) {
        t = fma(-Y[i * NX + 2 * m + h], S.xs[NU + 2 * m + h], t);
        t1 = fma(-Y[i * NX + 2 * m + 2 + h], S.xs[NU + 2 * m + 2 + h], t1);
      }
    t += t1;
    t += __shfl_xor_sync(0xffffffffu, t, 1);
#pragma unroll
    for (int c = 0; c < 15; c++) t = fma(-u[c], __shfl_sync(0xffffffffu, t, 2 * c), t);
    t *= di;
    __syncwarp();  // the previous stage's values have been read
    if (h == 0) {
      S.xs[i] = t;
      I.q[k * NS + i] = t;
    }
    __syncwarp();
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __threadfence_block();
  __syncthreads();  // q is complete
#pragma unroll
  for (int g = 0; g < 2; g++) {
    const int k = T - 1 - g;
    if (k >= 0) ring_load(S, I, I.q, k);
    else asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int k = T - 1; k >= 0; k--) {
    ring_wait<1>();  // stage k has landed; stage k + 1 is still in the ring
    if (k - 2 >= 0) ring_load(S, I, I.q, k - 2);
    else asm volatile("cp.async.commit_group;" ::: "memory");
    if (warp != 0) continue;
    const double *U = S.ring[k & (kRing - 1)], *q = U + 448;
    double u[15];
#pragma unroll
    for (int c = 1; c < NS; c++) u[c - 1] = i < c ? U[c * NS + i] : 0.0;
    double t = q[i];
    if (k + 1 < T) {
      const double *Y = S.ring[(k + 1) & (kRing - 1)] + 256;
      double a0 = 0.0, a1 = 0.0;
      if (i >= NU)
#pragma unroll
        for (int m = 0; m < 8; m += 2) {
          a0 = fma(Y[(2 * m + h) * NX + i - NU], S.xs[2 * m + h], a0);
          a1 = fma(Y[(2 * m + 2 + h) * NX + i - NU], S.xs[2 * m + 2 + h], a1);
        }
      a0 += a1;
      a0 += __shfl_xor_sync(0xffffffffu, a0, 1);
      t = fma(-U[i * NS + i], a0, t);
    }
#pragma unroll
    for (int c = NS - 1; c >= 1; c--) t = fma(-u[c - 1], __shfl_sync(0xffffffffu, t, 2 * c), t);
    __syncwarp();
    if (h == 0) {
      S.xs[i] = t;
      I.dz[k * NS + i] = t;
    }
    __syncwarp();
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
}

// rhs = -(W z + J^T t) from td (differences over the dynamics pairs) and the bounds'
// part of J^T t in aux's scratch
__device__ __forceinline__ void make_rhs(const Inst &I, int i, int k0) {
  for (int k = k0; k < I.T; k += kThreads / NS) {
    double a = fma(wdiag(I, i), I.z[k * NS + i], I.aux[k * SLOT + 48 + i]) + dyn_col(I, I.td, k, i);
    if (i >= NU) a += I.td[k * NS + i - NU];
    I.rhs[k * NS + i] = neg(a);
  }
}

// Recovery of d_lambda, d_s from dz (rows 2-3 of (3)) and the step lengths to the
// boundary (before tau): w = sig_mu - ds dl of the predictor (corrector) or 0. The
// smallest ratio v / (-dv) of a thread is kept as a fraction, compared by cross products.
__device__ __forceinline__ void recover(Shared &S, const Inst &I, int i, int k0, double umax, double xmax,
                                        bool corrector, double sig_mu, double &mp, double &md) {
  double pn = 1e30, pd = 1.0, dn = 1e30, dd = 1.0;  // (a ratio above 1 bounds no step)
  const double lim = i < NU ? umax : xmax;
  for (int k = k0; k < I.T; k += kThreads / NS) {
    const double zi = I.z[k * NS + i], dzi = I.dz[k * NS + i];
    double h = 0.0, jh = 0.0;
    if (i < NX) {
      h = I.aux[k * SLOT + i];
      jh = dyn_row(I, I.dz, nullptr, k, i);
    }
#pragma unroll
    for (int kind = 0; kind < 4; kind++) {
      if (kind < 2 && i >= NX) continue;
      const int q = k * SLOT + 16 * kind + i;
      // g + J dz of the row
      const double gj = kind == 0 ? h + jh : (kind == 1 ? neg(h + jh) : (kind == 2 ? (zi + lim) + dzi : (lim - zi) - dzi));
      const double s = I.s[q], lam = I.lam[q], il = I.il[q];
      const double wl = corrector ? (sig_mu - I.ds[q] * I.dl[q]) * il : 0.0;
      const double d = I.D[q] * (wl - gj);
      const double e = fma(-(s * il), d, wl - s);
      I.dl[q] = d;
      I.ds[q] = e;
      // e < 0 and s / -e below the smallest so far
      if (bits(e) < 0 && ratio_less(s, neg(e), pn, pd)) { pn = s; pd = neg(e); }
      if (bits(d) < 0 && ratio_less(lam, neg(d), dn, dd)) { dn = lam; dd = neg(d); }
    }
  }
  double v[2] = {quotient(pn, pd), quotient(dn, dd)};
  cta_reduce<R_MIN, R_MIN>(S, v);
  mp = v[0];
  md = v[1];
}

__device__ void solve_instance(Shared &S, const MpcArgs &a, int inst) {
  const Inst I = make_inst(a, inst);
  const int tid = threadIdx.x, i = tid % NS, k0 = tid / NS, T = I.T;
  constexpr int KS = kThreads / NS;
  const double mt = (double)T * 56.0, inv_mt = recip(mt);
  const double lim = i < NU ? a.umax : a.xmax;
  // starting point: z at the middle of its box (0), s = max(g, 1), lambda = 1
  for (int k = k0; k < T; k += KS) I.z[k * NS + i] = 0.0;
  __syncthreads();
  for (int k = k0; k < T; k += KS) {
    const double h = i < NX ? dyn_row(I, I.z, I.x0, k, i) : 0.0;
    for (int kind = 0; kind < 4; kind++) {
      const int q = k * SLOT + 16 * kind + i;
      const bool v = kind >= 2 || i < NX;
      I.s[q] = v ? fmax(kind == 0 ? h : (kind == 1 ? -h : lim), 1.0) : 1.0;
      I.lam[q] = v ? 1.0 : 0.0;
    }
    I.lamd[k * NS + i] = 0.0;
  }
  // scale of the primal residual: bfull = [A_0 x_0 (dynamics), bounds]
  double bs = fmax(a.umax, a.xmax);
  {
    double v[1] = {0.0};
    if (tid < NX) {
      double h = 0.0;
      for (int j = 0; j < NX; j++) h = fma(I.A[tid * NX + j], I.x0[j], h);
      v[0] = abs_or_zero(h);
    }
    cta_reduce<R_MAX>(S, v);
    bs = recip(fmax(1.0, fmax(bs, v[0])));
  }
  double delta_p = a.delta_p;
  int status = 7, it = 0;
  double kkt = 0.0, fx = 0.0;
  for (it = 0; it <= a.max_iter; it++) {
    __syncthreads();  // z, s, lambda are up to date
    // g, the residuals, D, 1 / lambda, and the predictor's row values t = D g - lambda
    double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};  // sums s lambda, f; maxima |g - s|, |s lambda|, |rd|
    for (int k = k0; k < T; k += KS) {
      const double zi = I.z[k * NS + i];
      const double h = i < NX ? dyn_row(I, I.z, I.x0, k, i) : 0.0;
      double D[4] = {0.0, 0.0, 0.0, 0.0}, lm[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int kind = 0; kind < 4; kind++) {
        if (kind < 2 && i >= NX) continue;
        const int q = k * SLOT + 16 * kind + i;
        const double g = kind == 0 ? h : (kind == 1 ? neg(h) : (kind == 2 ? zi + lim : lim - zi));
        const double s = I.s[q], l = I.lam[q], sl = s * l;
        v[0] += sl;
        v[2] = max_pos(v[2], abs_or_zero(g - s));
        v[3] = max_pos(v[3], abs_or_zero(sl));
        // one reciprocal per row: with t = delta_d lambda + s and r = 1 / (lambda t), 1 /
        // lambda = t r and D = 1 / (delta_d + s / lambda) = lambda^2 r
        const double t = fma(a.delta_d, l, s), r = recip(l * t);
        I.il[q] = t * r;
        D[kind] = (l * l) * r;
        I.D[q] = D[kind];
        lm[kind] = l;
      }
      const double wz = wdiag(I, i) * zi, db = D[0] + D[1];
      double rd = dyn_col(I, I.lamd, k, i) + (lm[2] - lm[3]);  // (J^T lambda)_i
      if (i >= NU) rd += I.lamd[k * NS + i - NU];
      v[4] = max_pos(v[4], abs_or_zero(wz - rd));
      v[1] = fma(0.5 * wz, zi, v[1]);
      if (i < NX) {
        I.aux[k * SLOT + i] = h;
        I.aux[k * SLOT + 16 + i] = db;
        I.td[k * NS + i] = fma(db, h, neg(I.lamd[k * NS + i]));
      }
      I.aux[k * SLOT + 32 + i] = wdiag(I, i) + (D[2] + D[3]);
      I.aux[k * SLOT + 48 + i] = fma(D[2], zi + lim, neg(lm[2])) - fma(D[3], lim - zi, neg(lm[3]));
    }
    cta_reduce<R_SUM, R_SUM, R_MAX, R_MAX, R_MAX>(S, v);
    fx = v[1];
    const double mu = v[0] * inv_mt;
    kkt = fmax(v[2] * bs, fmax(v[4], quotient(v[3], fmax(1.0, fabs(fx)))));
    if (!(kkt == kkt) || !(fx == fx) || !(mu == mu)) { status = 6; break; }
    if (kkt <= a.tol) { status = 0; break; }
    if (it == a.max_iter) break;
    bool fok = false;
    for (int tries = 0; tries < 12 && !fok; tries++) {
      fok = factor(S, I, delta_p);
      __syncthreads();
      if (!fok) delta_p *= 100.0;
    }
    if (!fok) { status = 5; break; }
    make_rhs(I, i, k0);
    __syncthreads();
    solve(S, I);
    double mp, md;
    recover(S, I, i, k0, a.umax, a.xmax, false, 0.0, mp, md);
    const double apa = fmin(1.0, mp), ada = fmin(1.0, md);
    double m1[1] = {0.0};
    for (int k = k0; k < T; k += KS)
#pragma unroll
      for (int kind = 0; kind < 4; kind++) {
        if (kind < 2 && i >= NX) continue;
        const int q = k * SLOT + 16 * kind + i;
        m1[0] = fma(fma(apa, I.ds[q], I.s[q]), fma(ada, I.dl[q], I.lam[q]), m1[0]);
      }
    cta_reduce<R_SUM>(S, m1);
    const double ratio = quotient(m1[0] * inv_mt, mu), sig_mu = ratio * ratio * ratio * mu;
    // the corrector's row values: the predictor's minus D w / lambda
    for (int k = k0; k < T; k += KS) {
      double e[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int kind = 0; kind < 4; kind++) {
        if (kind < 2 && i >= NX) continue;
        const int q = k * SLOT + 16 * kind + i;
        e[kind] = I.D[q] * ((sig_mu - I.ds[q] * I.dl[q]) * I.il[q]);
      }
      if (i < NX) I.td[k * NS + i] -= e[0] - e[1];
      I.aux[k * SLOT + 48 + i] -= e[2] - e[3];
    }
    __syncthreads();
    make_rhs(I, i, k0);
    __syncthreads();
    solve(S, I);
    recover(S, I, i, k0, a.umax, a.xmax, true, sig_mu, mp, md);
    const double tau = fmax(0.99, 1.0 - mu), ap = fmin(1.0, tau * mp), ad = fmin(1.0, tau * md);
    for (int k = k0; k < T; k += KS) {
      I.z[k * NS + i] = fma(ap, I.dz[k * NS + i], I.z[k * NS + i]);
      double l[2] = {0.0, 0.0};
#pragma unroll
      for (int kind = 0; kind < 4; kind++) {
        if (kind < 2 && i >= NX) continue;
        const int q = k * SLOT + 16 * kind + i;
        I.s[q] = fma(ap, I.ds[q], I.s[q]);
        const double ln = fma(ad, I.dl[q], I.lam[q]);
        I.lam[q] = ln;
        if (kind < 2) l[kind] = ln;
      }
      I.lamd[k * NS + i] = l[0] - l[1];
    }
  }
  if (tid == 0) {
    a.obj[inst] = fx;
    a.kkt[inst] = kkt;
    a.iters[inst] = it;
    a.status[inst] = status;
    if (a.fp64_used) a.fp64_used[inst] = 0;
  }
  __syncthreads();
  if (a.zout)
    for (int k = k0; k < T; k += KS) a.zout[(a.soff[inst] + k) * NS + i] = I.z[k * NS + i];
}

__global__ void __launch_bounds__(kThreads, 5) mpc_cta_kernel(MpcArgs a) {
  __shared__ Shared S;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) S.inst = atomicAdd(a.counter, 1);
    __syncthreads();
    const int q = S.inst;
    if (q >= a.count) break;
    solve_instance(S, a, a.order[q]);
  }
}

}  // namespace

int mpc_cta_slots() {
  static int per_device[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 152;
  int &g = per_device[dev & 63];
  if (g == 0) {
    int sms = 0, nb = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 152;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, mpc_cta_kernel, kThreads, 0) != cudaSuccess) return sms;
    g = sms * (nb > 0 ? nb : 1);
  }
  return g;
}

void launch_mpc_cta(const MpcArgs &a, int ctas, cudaStream_t st) {
  note_launch();
  mpc_cta_kernel<<<ctas, kThreads, 0, st>>>(a);
}

}  // namespace gipm
