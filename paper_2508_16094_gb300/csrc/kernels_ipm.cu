// FP64 map/reduce kernels of the interior-point iteration (Sec. 1: line search
// and barrier updates are map or reduce operations) and of the matrix-free
// residual used by iterative refinement. A reduction's grid depends on the length
// alone and its partial results are combined in block order, so every result is
// bit-reproducible.
#include <cfloat>
#include <type_traits>

#include "ipm_kernels.h"

namespace gipm {

namespace {

constexpr int kRedBlock = 256;

// |v| and the larger of two of them on the integer pipe: an FP64 comparison
// occupies GB300's FP64 unit as long as a multiply-add. The bits of a NaN compare above
// those of infinity, so a maximum over values with a NaN among them is NaN; the comparison
// leaves the sign bit out, which the compiler's |v| may leave set on a NaN.
__device__ __forceinline__ double abs_bits(double v) {
  return __longlong_as_double(__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFll);
}
__device__ __forceinline__ double max_nonneg(double a, double b) {
  return (unsigned long long)__double_as_longlong(a) << 1 > (unsigned long long)__double_as_longlong(b) << 1 ? a : b;
}
// RED_MAX combines values >= 0 or NaN (identity 0)
template <int OP> __device__ __forceinline__ double red_combine(double a, double b) {
  return OP == RED_SUM ? a + b : (OP == RED_MAX ? max_nonneg(a, b) : fmin(a, b));
}
template <int OP> __device__ __forceinline__ double red_identity() { return OP == RED_MIN ? DBL_MAX : 0.0; }

template <int OP> __device__ __forceinline__ double warp_reduce(double x, int from) {
  for (int o = from; o > 0; o >>= 1) x = red_combine<OP>(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}
// Reduction over a block, the result in thread 0.
template <int OP> __device__ __forceinline__ double block_reduce(double x, double *sh) {
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  x = warp_reduce<OP>(x, 16);
  if (lane == 0) sh[warp] = x;
  __syncthreads();
  if (warp == 0) x = warp_reduce<OP>(lane < kRedBlock / 32 ? sh[lane] : red_identity<OP>(), 4);
  return x;
}

// Reduction over the grid in one launch: every block stores its partial results,
// the last one to finish combines them (in block order, so results do not
// depend on which block that is) and calls fin(results) on one thread. `ticket`
// is zero before the launch and zero again after it. A second launch whose one
// thread added 256 values, as before, took 17 us.
template <int... OPS, typename Fin>
__device__ __forceinline__ void grid_reduce(double (&v)[sizeof...(OPS)], double *partial, unsigned *ticket,
                                            Fin fin) {
  constexpr int NS = sizeof...(OPS);
  __shared__ double sh[NS][kRedBlock / 32];
  __shared__ bool last;
  {
    int k = 0;
    ((v[k] = block_reduce<OPS>(v[k], sh[k]), k++), ...);
  }
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NS; k++) partial[blockIdx.x * NS + k] = v[k];
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  {
    int k = 0;
    auto one = [&](auto op) {
      constexpr int OP = decltype(op)::value;
      double x = red_identity<OP>();
      for (int b = threadIdx.x; b < (int)gridDim.x; b += kRedBlock)
        x = red_combine<OP>(x, __ldcg(partial + b * NS + k));
      v[k] = block_reduce<OP>(x, sh[k]);
      k++;
    };
    (one(std::integral_constant<int, OPS>{}), ...);
  }
  if (threadIdx.x == 0) {
    fin(v);
    *ticket = 0u;
  }
}

#define GRID_STRIDE(i, n)                                                              \
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n);             \
       i += (int64_t)gridDim.x * blockDim.x)

// Blocks of a reduction over n values: at most kRedBlocks, a function of n alone.
inline int red_grid(int64_t n) {
  const int64_t g = (n + kRedBlock - 1) / kRedBlock;
  return (int)(g < 1 ? 1 : (g > kRedBlocks ? kRedBlocks : g));
}
inline int grid_of(int64_t n) {
  int64_t g = (n + 255) / 256;
  return (int)(g < 1 ? 1 : (g > 152 * 16 ? 152 * 16 : g));
}

// ---------------------------------------------------------------------------
__global__ void jv_kernel(DevPlan dp, const double *__restrict__ jv, const double *__restrict__ x,
                          double *__restrict__ out) {
  GRID_STRIDE(r, dp.m) {
    double a = 0.0;
    for (int64_t e = dp.jp[r]; e < dp.jp[r + 1]; e++) a = fma(jv[e], x[dp.ji[e]], a);
    out[r] = a;
  }
}

// out[j] = base_j + sgn * (J^T v)_j + (W x)_j  (v has length m_tot: general rows,
// then lower-bound rows (+e_i), then upper-bound rows (-e_i))
__global__ void jtv_kernel(DevPlan dp, const double *__restrict__ jv, const double *__restrict__ v,
                           double sgn, const double *__restrict__ wv, const double *__restrict__ x,
                           const double *__restrict__ base, double *__restrict__ out) {
  GRID_STRIDE(j, dp.n) {
    double a = 0.0;
    for (int64_t t = dp.jtp[j]; t < dp.jtp[j + 1]; t++) {
      const int32_t e = dp.jtpos[t];
      a = fma(jv[e], v[dp.jrow[e]], a);
    }
    if (dp.lpos[j] >= 0) a += v[dp.lpos[j]];
    if (dp.upos[j] >= 0) a -= v[dp.upos[j]];
    a = sgn * a + (base ? base[j] : 0.0);
    if (wv && x)
      for (int64_t e = dp.wfp[j]; e < dp.wfp[j + 1]; e++) a = fma(wv[dp.wfsrc[e]], x[dp.wfi[e]], a);
    out[j] = a;
  }
}
__global__ void init_slack_kernel(int64_t mt, const double *__restrict__ g, double *__restrict__ s,
                                  double *__restrict__ lam) {
  GRID_STRIDE(k, mt) {
    s[k] = fmax(g[k], 1.0);
    lam[k] = 1.0;
  }
}

// (J x) for all m_tot rows: general rows from jx, bound rows +-x
__global__ void jfull_kernel(DevPlan dp, const double *__restrict__ jx, const double *__restrict__ x,
                             double *__restrict__ out) {
  GRID_STRIDE(k, dp.mt) {
    double v;
    if (k < dp.m) v = jx[k];
    else if (k < dp.m + dp.nl) v = x[dp.lidx[k - dp.m]];
    else v = -x[dp.uidx[k - dp.m - dp.nl]];
    out[k] = v;
  }
}

// residual r = b - K x with K = W + J_A^T D_A J_A + diag(D_l + D_u) + delta_p I
__global__ void resid_rows_kernel(DevPlan dp, const double *__restrict__ jv,
                                  const double *__restrict__ D, const double *__restrict__ x,
                                  double *__restrict__ tA) {
  GRID_STRIDE(r, dp.m) {
    double a = 0.0;
    for (int64_t e = dp.jp[r]; e < dp.jp[r + 1]; e++) a = fma(jv[e], x[dp.ji[e]], a);
    tA[r] = D[r] * a;
  }
}
// (K x)_j from tA = D_A J x
__device__ __forceinline__ double kx_col(const DevPlan &dp, const double *jv, const double *D,
                                         const double *wv, double delta_p, const double *tA,
                                         const double *x, int64_t j) {
  double a = 0.0;
  for (int64_t t = dp.jtp[j]; t < dp.jtp[j + 1]; t++) {
    const int32_t e = dp.jtpos[t];
    a = fma(jv[e], tA[dp.jrow[e]], a);
  }
  double d = delta_p;
  if (dp.lpos[j] >= 0) d += D[dp.lpos[j]];
  if (dp.upos[j] >= 0) d += D[dp.upos[j]];
  a = fma(d, x[j], a);
  if (wv)
    for (int64_t e = dp.wfp[j]; e < dp.wfp[j + 1]; e++) a = fma(wv[dp.wfsrc[e]], x[dp.wfi[e]], a);
  return a;
}
// 1 / m, the scale that keeps a right-hand side of largest entry m in FP32's range
__device__ __forceinline__ double scale_of(double m) { return (m > 0.0 && m < DBL_MAX) ? 1.0 / m : 1.0; }

// r = b - K x, and its largest entry and scale (`flag`: a status word copied out beside them)
__global__ void __launch_bounds__(kRedBlock) resid_cols_kernel(
    DevPlan dp, const double *__restrict__ jv, const double *__restrict__ D, const double *__restrict__ wv,
    double delta_p, const double *__restrict__ tA, const double *__restrict__ x,
    const double *__restrict__ b, double *__restrict__ r, const int32_t *flag, double *out,
    double *partial, unsigned *ticket) {
  double m[1] = {0.0};
  GRID_STRIDE(j, dp.n) {
    const double v = b[j] - kx_col(dp, jv, D, wv, delta_p, tA, x, j);
    r[j] = v;
    m[0] = max_nonneg(m[0], abs_bits(v));
  }
  grid_reduce<RED_MAX>(m, partial, ticket, [&](double (&v)[1]) {
    out[0] = v[0];
    out[1] = scale_of(v[0]);
    if (flag) out[2] = (double)*flag;
  });
}
// q = K p, p . q and the step length alpha = rz / (p . q) (0 if that is 0)
__global__ void __launch_bounds__(kRedBlock) kp_dot_kernel(
    DevPlan dp, const double *__restrict__ jv, const double *__restrict__ D, const double *__restrict__ wv,
    double delta_p, const double *__restrict__ tA, const double *__restrict__ p, double *__restrict__ q,
    const double *rz, double *alpha, double *partial, unsigned *ticket) {
  double s[1] = {0.0};
  GRID_STRIDE(j, dp.n) {
    const double v = kx_col(dp, jv, D, wv, delta_p, tA, p, j);
    q[j] = v;
    s[0] = fma(p[j], v, s[0]);
  }
  grid_reduce<RED_SUM>(s, partial, ticket,
                       [&](double (&v)[1]) { alpha[0] = v[0] != 0.0 ? rz[0] / v[0] : 0.0; });
}
__global__ void kx_kernel(DevPlan dp, const double *__restrict__ jv, const double *__restrict__ D,
                          const double *__restrict__ wv, double delta_p, const double *__restrict__ tA,
                          const double *__restrict__ x, double *__restrict__ q) {
  GRID_STRIDE(j, dp.n) q[j] = kx_col(dp, jv, D, wv, delta_p, tA, x, j);
}

// row sums of |K|: |W| 1 + |J_A|^T D_A |J_A| 1 + D_l + D_u + delta_p (D >= 0)
__global__ void absk_rows_kernel(DevPlan dp, const double *__restrict__ jv,
                                 const double *__restrict__ D, double *__restrict__ tA) {
  GRID_STRIDE(r, dp.m) {
    double a = 0.0;
    for (int64_t e = dp.jp[r]; e < dp.jp[r + 1]; e++) a += fabs(jv[e]);
    tA[r] = D[r] * a;
  }
}
__global__ void absk_cols_kernel(DevPlan dp, const double *__restrict__ jv,
                                 const double *__restrict__ D, const double *__restrict__ wv,
                                 double delta_p, const double *__restrict__ tA,
                                 double *__restrict__ out) {
  GRID_STRIDE(j, dp.n) {
    double a = 0.0;
    for (int64_t t = dp.jtp[j]; t < dp.jtp[j + 1]; t++) {
      const int32_t e = dp.jtpos[t];
      a = fma(fabs(jv[e]), tA[dp.jrow[e]], a);
    }
    double d = fabs(delta_p);
    if (dp.lpos[j] >= 0) d += D[dp.lpos[j]];
    if (dp.upos[j] >= 0) d += D[dp.upos[j]];
    a += d;
    if (wv)
      for (int64_t e = dp.wfp[j]; e < dp.wfp[j + 1]; e++) a += fabs(wv[dp.wfsrc[e]]);
    out[j] = a;
  }
}
template <typename V>
__global__ void permute_in_kernel(int32_t n, const int32_t *__restrict__ perm,
                                  const double *__restrict__ b, const double *__restrict__ scale,
                                  V *__restrict__ y) {
  const double s = scale ? scale[0] : 1.0;
  GRID_STRIDE(k, n) y[k] = (V)(b[perm[k]] * s);
}
template <typename V>
__global__ void permute_out_kernel(int32_t n, const int32_t *__restrict__ perm,
                                   const V *__restrict__ y, const double *__restrict__ scale,
                                   double *__restrict__ x, int accumulate) {
  const double s = scale ? 1.0 / scale[0] : 1.0;
  GRID_STRIDE(k, n) {
    const double v = (double)y[k] * s;
    if (accumulate) x[perm[k]] += v;
    else x[perm[k]] = v;
  }
}

// z = P^T y / scale, r . z, and beta = (r . z) / rz_old (without it: only r . z)
template <typename V>
__global__ void __launch_bounds__(kRedBlock) permute_out_dot_kernel(
    int32_t n, const int32_t *__restrict__ perm, const V *__restrict__ y, const double *__restrict__ scale,
    const double *__restrict__ r, double *__restrict__ z, const double *rz_old, double *rz, double *beta,
    double *partial, unsigned *ticket) {
  const double s = scale ? 1.0 / scale[0] : 1.0;
  double d[1] = {0.0};
  GRID_STRIDE(k, n) {
    const int32_t i = perm[k];
    const double v = (double)y[k] * s;
    z[i] = v;
    d[0] = fma(r[i], v, d[0]);
  }
  grid_reduce<RED_SUM>(d, partial, ticket, [&](double (&v)[1]) {
    if (rz_old) beta[0] = rz_old[0] != 0.0 ? v[0] / rz_old[0] : 0.0;
    rz[0] = v[0];
  });
}

// ---- reductions -----------------------------------------------------------
// out[0] = max |v|, out[1] = its scale (see scale_of)
__global__ void __launch_bounds__(kRedBlock) absmax_kernel(int64_t n, const double *__restrict__ v, double *out,
                                                           int with_scale, double *partial, unsigned *ticket) {
  double a[1] = {0.0};
  GRID_STRIDE(i, n) a[0] = max_nonneg(a[0], abs_bits(v[i]));
  grid_reduce<RED_MAX>(a, partial, ticket, [&](double (&m)[1]) {
    out[0] = m[0];
    if (with_scale) out[1] = scale_of(m[0]);
  });
}
__global__ void __launch_bounds__(kRedBlock) dot_kernel(int64_t n, const double *__restrict__ a,
                                                        const double *__restrict__ b, double *out,
                                                        double *partial, unsigned *ticket) {
  double v[1] = {0.0};
  GRID_STRIDE(i, n) v[0] = fma(a[i], b[i], v[0]);
  grid_reduce<RED_SUM>(v, partial, ticket, [&](double (&d)[1]) { out[0] = d[0]; });
}

// KKT quantities: sum s.lambda, max|g - s|, max|s.lambda|, max|rd|, f(x)
__global__ void __launch_bounds__(kRedBlock) kkt_reduce_kernel(
    DevPlan dp, const double *__restrict__ g, const double *__restrict__ s, const double *__restrict__ lam,
    const double *__restrict__ rd, const double *__restrict__ c, const double *__restrict__ wx,
    const double *__restrict__ x, IpmScalars *sc, double *partial, unsigned *ticket) {
  double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  GRID_STRIDE(i, dp.mt + dp.n) {
    if (i < dp.mt) {
      const double sl = s[i] * lam[i];
      v[0] += sl;
      v[1] = max_nonneg(v[1], abs_bits(g[i] - s[i]));
      v[2] = max_nonneg(v[2], abs_bits(sl));
    } else {
      const int64_t j = i - dp.mt;
      v[3] = max_nonneg(v[3], abs_bits(rd[j]));
      v[4] = fma(c[j] + (wx ? 0.5 * wx[j] : 0.0), x[j], v[4]);
    }
  }
  const int64_t mt = dp.mt;
  grid_reduce<RED_SUM, RED_MAX, RED_MAX, RED_MAX, RED_SUM>(v, partial, ticket, [&](double (&red)[5]) {
    sc->mu = red[0] / (double)(mt > 0 ? mt : 1);
    sc->primal_inf = red[1];
    sc->compl_inf = red[2];
    sc->dual_inf = red[3];
    sc->fx = red[4];
  });
}

// fraction to the boundary: min over ds<0 of -s/ds, min over dl<0 of -lam/dl
__global__ void __launch_bounds__(kRedBlock) ftb_kernel(
    int64_t mt, const double *__restrict__ s, const double *__restrict__ ds, const double *__restrict__ lam,
    const double *__restrict__ dl, IpmScalars *sc, int affine, double *partial, unsigned *ticket) {
  double v[2] = {DBL_MAX, DBL_MAX};
  GRID_STRIDE(i, mt) {
    if (ds[i] < 0.0) v[0] = fmin(v[0], -s[i] / ds[i]);
    if (dl[i] < 0.0) v[1] = fmin(v[1], -lam[i] / dl[i]);
  }
  grid_reduce<RED_MIN, RED_MIN>(v, partial, ticket, [&](double (&red)[2]) {
    if (affine) {
      sc->alpha_aff_p = fmin(1.0, red[0]);
      sc->alpha_aff_d = fmin(1.0, red[1]);
    } else {
      const double tau = fmax(0.99, 1.0 - sc->mu);
      sc->alpha_p = fmin(1.0, tau * red[0]);
      sc->alpha_d = fmin(1.0, tau * red[1]);
    }
  });
}

__global__ void __launch_bounds__(kRedBlock) muaff_kernel(
    int64_t mt, const double *__restrict__ s, const double *__restrict__ ds, const double *__restrict__ lam,
    const double *__restrict__ dl, IpmScalars *sc, double *partial, unsigned *ticket) {
  const double ap = sc->alpha_aff_p, ad = sc->alpha_aff_d;
  double v[1] = {0.0};
  GRID_STRIDE(i, mt) v[0] = fma(fma(ap, ds[i], s[i]), fma(ad, dl[i], lam[i]), v[0]);
  grid_reduce<RED_SUM>(v, partial, ticket,
                       [&](double (&red)[1]) { sc->mu_aff = red[0] / (double)(mt > 0 ? mt : 1); });
}

// ---- elementwise steps ---------------------------------------------------
// g = J x - bfull from (J x) of the general rows
__global__ void g_kernel(DevPlan dp, const double *__restrict__ jx, const double *__restrict__ x,
                         const double *__restrict__ b, const double *__restrict__ l,
                         const double *__restrict__ u, double *__restrict__ g) {
  GRID_STRIDE(k, dp.mt) {
    double v;
    if (k < dp.m) v = jx[k] - b[k];
    else if (k < dp.m + dp.nl) { const int32_t i = dp.lidx[k - dp.m]; v = x[i] - l[i]; }
    else { const int32_t i = dp.uidx[k - dp.m - dp.nl]; v = u[i] - x[i]; }
    g[k] = v;
  }
}
__global__ void scaling_kernel(int64_t mt, const double *__restrict__ s,
                               const double *__restrict__ lam, double delta_d,
                               double *__restrict__ D) {
  GRID_STRIDE(k, mt) D[k] = 1.0 / (delta_d + s[k] / lam[k]);
}
// t = D (g - w/lambda) - lambda   (w may be NULL: zero)
__global__ void rhs_rows_kernel(int64_t mt, const double *__restrict__ D, const double *__restrict__ g,
                                const double *__restrict__ w, const double *__restrict__ lam,
                                double *__restrict__ t) {
  GRID_STRIDE(k, mt) {
    const double wl = w ? w[k] / lam[k] : 0.0;
    t[k] = D[k] * (g[k] - wl) - lam[k];
  }
}
__global__ void negate_kernel(int64_t n, double *__restrict__ v) {
  GRID_STRIDE(i, n) v[i] = -v[i];
}
// d_lambda = D (w/lambda - g - J d_x);  d_s = -s + w/lambda - (s/lambda) d_lambda
__global__ void recover_kernel(int64_t mt, const double *__restrict__ D, const double *__restrict__ g,
                               const double *__restrict__ w, const double *__restrict__ s,
                               const double *__restrict__ lam, const double *__restrict__ jdx,
                               double *__restrict__ ds, double *__restrict__ dl) {
  GRID_STRIDE(k, mt) {
    const double wl = w ? w[k] / lam[k] : 0.0;
    const double d = D[k] * (wl - g[k] - jdx[k]);
    dl[k] = d;
    ds[k] = -s[k] + wl - (s[k] / lam[k]) * d;
  }
}
// w = sigma mu - ds_aff .* dl_aff, with sigma = (mu_aff / mu)^3 computed here
__global__ void corrector_target_kernel(int64_t mt, const double *__restrict__ ds,
                                        const double *__restrict__ dl, IpmScalars *sc,
                                        double *__restrict__ w) {
  const double mu = sc->mu, ratio = sc->mu_aff / mu;
  const double sm = ratio * ratio * ratio * mu;
  if (blockIdx.x == 0 && threadIdx.x == 0) sc->sigma = ratio * ratio * ratio;
  GRID_STRIDE(k, mt) w[k] = sm - ds[k] * dl[k];
}
__global__ void update_kernel(int64_t n, int64_t mt, const IpmScalars *sc, double *__restrict__ x,
                              const double *__restrict__ dx, double *__restrict__ s,
                              const double *__restrict__ ds, double *__restrict__ lam,
                              const double *__restrict__ dl) {
  const double ap = sc->alpha_p, ad = sc->alpha_d;
  GRID_STRIDE(i, n + mt) {
    if (i < n) x[i] = fma(ap, dx[i], x[i]);
    else {
      const int64_t k = i - n;
      s[k] = fma(ap, ds[k], s[k]);
      lam[k] = fma(ad, dl[k], lam[k]);
    }
  }
}
// ---- vector updates used by refinement / PCG ------------------------------
// x += alpha p, r -= alpha q, and the largest entry of the new r with its scale
__global__ void __launch_bounds__(kRedBlock) cg_step_kernel(
    int64_t n, const double *alpha, const double *__restrict__ p, const double *__restrict__ q,
    double *__restrict__ x, double *__restrict__ r, double *out, double *partial, unsigned *ticket) {
  const double a = alpha[0];
  double m[1] = {0.0};
  GRID_STRIDE(i, n) {
    x[i] = fma(a, p[i], x[i]);
    const double v = fma(-a, q[i], r[i]);
    r[i] = v;
    m[0] = max_nonneg(m[0], abs_bits(v));
  }
  grid_reduce<RED_MAX>(m, partial, ticket, [&](double (&v)[1]) {
    out[0] = v[0];
    out[1] = scale_of(v[0]);
  });
}
// p = z + beta p
__global__ void cg_direction_kernel(int64_t n, const double *beta, const double *__restrict__ z,
                                    double *__restrict__ p) {
  const double b = beta[0];
  GRID_STRIDE(i, n) p[i] = fma(b, p[i], z[i]);
}

}  // namespace

// ---------------------------------------------------------------------------
// Load the kernels of the allocation-free solve now (a function query loads a
// lazily loaded kernel), so that its later launches commit no device memory.
cudaError_t preload_vec_kernels() {
  cudaFuncAttributes a;
  cudaError_t e = cudaSuccess;
  auto q = [&](const void *f) { if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, f); };
  q((const void *)permute_in_kernel<double>);
  q((const void *)permute_in_kernel<float>);
  q((const void *)permute_out_kernel<double>);
  q((const void *)permute_out_kernel<float>);
  q((const void *)absmax_kernel);
  return e;
}

void VecOps::absmax(int64_t n, const double *v, double *out, bool with_scale) const {
  note_launch();
  absmax_kernel<<<red_grid(n), kRedBlock, 0, st>>>(n, v, out, with_scale ? 1 : 0, partial, ticket);
}
void VecOps::dot(int64_t n, const double *a, const double *b, double *out) const {
  note_launch();
  dot_kernel<<<red_grid(n), kRedBlock, 0, st>>>(n, a, b, out, partial, ticket);
}
void VecOps::jv(const double *jvals, const double *x, double *out) const {
  if (dp.m > 0) { note_launch(); jv_kernel<<<grid_of(dp.m), 256, 0, st>>>(dp, jvals, x, out); }
}
void VecOps::jfull(const double *jx, const double *x, double *out) const {
  if (dp.mt > 0) { note_launch(); jfull_kernel<<<grid_of(dp.mt), 256, 0, st>>>(dp, jx, x, out); }
}
void VecOps::jtv(const double *jvals, const double *v, double sgn, const double *wv,
                 const double *x, const double *base, double *out) const {
  { note_launch(); jtv_kernel<<<grid_of(dp.n), 256, 0, st>>>(dp, jvals, v, sgn, wv, x, base, out); }
}
void VecOps::init_slack(const double *gv, double *s, double *lam) const {
  if (dp.mt > 0) { note_launch(); init_slack_kernel<<<grid_of(dp.mt), 256, 0, st>>>(dp.mt, gv, s, lam); }
}
void VecOps::rows_product(const double *jvals, const double *D, const double *x, double *tA) const {
  if (dp.m > 0) { note_launch(); resid_rows_kernel<<<grid_of(dp.m), 256, 0, st>>>(dp, jvals, D, x, tA); }
}
void VecOps::residual(const double *jvals, const double *D, const double *wv, double delta_p,
                      const double *x, const double *b, double *r, double *tA, double *out,
                      const int32_t *flag) const {
  rows_product(jvals, D, x, tA);
  note_launch();
  resid_cols_kernel<<<red_grid(dp.n), kRedBlock, 0, st>>>(dp, jvals, D, wv, delta_p, tA, x, b, r, flag, out,
                                                          partial, ticket);
}
void VecOps::kx(const double *jvals, const double *D, const double *wv, double delta_p, const double *x,
                double *q, double *tA) const {
  rows_product(jvals, D, x, tA);
  note_launch();
  kx_kernel<<<grid_of(dp.n), 256, 0, st>>>(dp, jvals, D, wv, delta_p, tA, x, q);
}
void VecOps::kp_dot(const double *jvals, const double *D, const double *wv, double delta_p, const double *p,
                    double *q, double *tA, const double *rz, double *alpha) const {
  rows_product(jvals, D, p, tA);
  note_launch();
  kp_dot_kernel<<<red_grid(dp.n), kRedBlock, 0, st>>>(dp, jvals, D, wv, delta_p, tA, p, q, rz, alpha, partial,
                                                      ticket);
}
void VecOps::cg_step(int64_t n, const double *alpha, const double *p, const double *q, double *x, double *r,
                     double *out) const {
  note_launch();
  cg_step_kernel<<<red_grid(n), kRedBlock, 0, st>>>(n, alpha, p, q, x, r, out, partial, ticket);
}
void VecOps::cg_direction(int64_t n, const double *beta, const double *z, double *p) const {
  note_launch();
  cg_direction_kernel<<<grid_of(n), 256, 0, st>>>(n, beta, z, p);
}
void VecOps::abs_rowsum(const double *jvals, const double *D, const double *wv, double delta_p,
                        double *out, double *tA) const {
  if (dp.m > 0) { note_launch(); absk_rows_kernel<<<grid_of(dp.m), 256, 0, st>>>(dp, jvals, D, tA); }
  { note_launch(); absk_cols_kernel<<<grid_of(dp.n), 256, 0, st>>>(dp, jvals, D, wv, delta_p, tA, out); }
}
template <typename V>
void VecOps::permute_in(const double *b, const double *scale, V *y) const {
  { note_launch(); permute_in_kernel<V><<<grid_of(dp.n), 256, 0, st>>>(dp.n, dp.perm, b, scale, y); }
}
template <typename V>
void VecOps::permute_out(const V *y, const double *scale, double *x, bool accumulate) const {
  { note_launch(); permute_out_kernel<V><<<grid_of(dp.n), 256, 0, st>>>(dp.n, dp.perm, y, scale, x, accumulate); }
}
template <typename V>
void VecOps::permute_out_dot(const V *y, const double *scale, const double *r, double *z, const double *rz_old,
                             double *rz, double *beta) const {
  note_launch();
  permute_out_dot_kernel<V><<<red_grid(dp.n), kRedBlock, 0, st>>>(dp.n, dp.perm, y, scale, r, z, rz_old, rz, beta,
                                                                  partial, ticket);
}
template void VecOps::permute_out_dot<double>(const double *, const double *, const double *, double *,
                                              const double *, double *, double *) const;
template void VecOps::permute_out_dot<float>(const float *, const double *, const double *, double *,
                                             const double *, double *, double *) const;
template void VecOps::permute_in<double>(const double *, const double *, double *) const;
template void VecOps::permute_in<float>(const double *, const double *, float *) const;
template void VecOps::permute_out<double>(const double *, const double *, double *, bool) const;
template void VecOps::permute_out<float>(const float *, const double *, double *, bool) const;

void VecOps::kkt(const double *g, const double *s, const double *lam, const double *rd,
                 const double *c, const double *wx, const double *x, IpmScalars *sc) const {
  note_launch();
  kkt_reduce_kernel<<<red_grid(dp.mt + dp.n), kRedBlock, 0, st>>>(dp, g, s, lam, rd, c, wx, x, sc, partial, ticket);
}
void VecOps::g(const double *jx, const double *x, const double *b, const double *l,
               const double *u, double *gout) const {
  if (dp.mt > 0) { note_launch(); g_kernel<<<grid_of(dp.mt), 256, 0, st>>>(dp, jx, x, b, l, u, gout); }
}
void VecOps::scaling(const double *s, const double *lam, double delta_d, double *D) const {
  if (dp.mt > 0) { note_launch(); scaling_kernel<<<grid_of(dp.mt), 256, 0, st>>>(dp.mt, s, lam, delta_d, D); }
}
void VecOps::rhs_rows(const double *D, const double *gv, const double *w, const double *lam,
                      double *t) const {
  if (dp.mt > 0) { note_launch(); rhs_rows_kernel<<<grid_of(dp.mt), 256, 0, st>>>(dp.mt, D, gv, w, lam, t); }
}
void VecOps::negate(int64_t n, double *v) const {
  { note_launch(); negate_kernel<<<grid_of(n), 256, 0, st>>>(n, v); }
}
void VecOps::recover(const double *D, const double *gv, const double *w, const double *s,
                     const double *lam, const double *jdx, double *ds, double *dl) const {
  if (dp.mt > 0)
    { note_launch(); recover_kernel<<<grid_of(dp.mt), 256, 0, st>>>(dp.mt, D, gv, w, s, lam, jdx, ds, dl); }
}
void VecOps::ftb(const double *s, const double *ds, const double *lam, const double *dl, IpmScalars *sc,
                 bool affine) const {
  note_launch();
  ftb_kernel<<<red_grid(dp.mt), kRedBlock, 0, st>>>(dp.mt, s, ds, lam, dl, sc, affine ? 1 : 0, partial, ticket);
}
void VecOps::muaff(const double *s, const double *ds, const double *lam, const double *dl,
                   IpmScalars *sc) const {
  note_launch();
  muaff_kernel<<<red_grid(dp.mt), kRedBlock, 0, st>>>(dp.mt, s, ds, lam, dl, sc, partial, ticket);
}
void VecOps::corrector_target(const double *ds, const double *dl, IpmScalars *sc,
                              double *w) const {
  { note_launch(); corrector_target_kernel<<<grid_of(dp.mt), 256, 0, st>>>(dp.mt, ds, dl, sc, w); }
}
void VecOps::update(const IpmScalars *sc, double *x, const double *dx, double *s,
                    const double *ds, double *lam, const double *dl) const {
  { note_launch(); update_kernel<<<grid_of(dp.n + dp.mt), 256, 0, st>>>(dp.n, dp.mt, sc, x, dx, s, ds, lam, dl); }
}

}  // namespace gipm
