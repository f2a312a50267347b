// Launchers of the FP64 vector kernels (interior-point step, residuals, reductions).
#pragma once

#include "dev.cuh"

namespace gipm {

enum RedOp : int { RED_SUM = 0, RED_MAX = 1, RED_MIN = 2 };

// Scalars of one interior-point iteration, kept in device memory so that the
// iteration needs no host round trip except the convergence test.
struct IpmScalars {
  double mu, mu_aff, sigma;
  double alpha_aff_p, alpha_aff_d, alpha_p, alpha_d;
  double primal_inf, dual_inf, compl_inf, fx;
  double pad[5];
};

// Loads the vector kernels the allocation-free solve launches (see capi.cu).
cudaError_t preload_vec_kernels();

constexpr int kRedBlocks = 304;  // largest grid of a reduction (2 blocks per SM)

struct VecOps {
  DevPlan dp;
  cudaStream_t st;
  double *partial;   // kRedBlocks * 8 doubles
  unsigned *ticket;  // one word, zero between launches (a reduction counts its finished blocks)

  // out[0] = max |v| (NaN if one of them is); with_scale: out[1] = 1 / out[0] (1 if that is 0 or
  // not finite)
  void absmax(int64_t n, const double *v, double *out, bool with_scale = false) const;
  void dot(int64_t n, const double *a, const double *b, double *out) const;
  void jv(const double *jvals, const double *x, double *out) const;
  void jfull(const double *jx, const double *x, double *out) const;
  // out = base + sgn J^T v (+ W x)
  void jtv(const double *jvals, const double *v, double sgn, const double *wv, const double *x,
           const double *base, double *out) const;
  // s = max(g, 1), lambda = 1
  void init_slack(const double *gv, double *s, double *lam) const;
  // tA = D_A J x (scratch of length m of the products below)
  void rows_product(const double *jvals, const double *D, const double *x, double *tA) const;
  // r = b - K x (matrix-free), out[0] = max |r|, out[1] = its scale (as absmax), with
  // flag: out[2] = *flag
  void residual(const double *jvals, const double *D, const double *wv, double delta_p,
                const double *x, const double *b, double *r, double *tA, double *out,
                const int32_t *flag = nullptr) const;
  // q = K x
  void kx(const double *jvals, const double *D, const double *wv, double delta_p, const double *x, double *q,
          double *tA) const;
  // one conjugate-gradient iteration around the preconditioner: q = K p and alpha = rz /
  // (p . q); x += alpha p, r -= alpha q with out[0..1] as residual's; z = P^T y / scale with
  // rz = r . z and beta = rz / rz_old; p = z + beta p
  void kp_dot(const double *jvals, const double *D, const double *wv, double delta_p, const double *p, double *q,
              double *tA, const double *rz, double *alpha) const;
  void cg_step(int64_t n, const double *alpha, const double *p, const double *q, double *x, double *r,
               double *out) const;
  template <typename V>
  void permute_out_dot(const V *y, const double *scale, const double *r, double *z, const double *rz_old,
                       double *rz, double *beta) const;
  void cg_direction(int64_t n, const double *beta, const double *z, double *p) const;
  // out_j = sum_i |K_ji| (matrix-free, D >= 0); tA: scratch of length m
  void abs_rowsum(const double *jvals, const double *D, const double *wv, double delta_p,
                  double *out, double *tA) const;
  template <typename V> void permute_in(const double *b, const double *scale, V *y) const;
  template <typename V>
  void permute_out(const V *y, const double *scale, double *x, bool accumulate) const;
  void kkt(const double *g, const double *s, const double *lam, const double *rd, const double *c,
           const double *wx, const double *x, IpmScalars *sc) const;
  void g(const double *jx, const double *x, const double *b, const double *l, const double *u,
         double *gout) const;
  void scaling(const double *s, const double *lam, double delta_d, double *D) const;
  void rhs_rows(const double *D, const double *gv, const double *w, const double *lam,
                double *t) const;
  void negate(int64_t n, double *v) const;
  void recover(const double *D, const double *gv, const double *w, const double *s,
               const double *lam, const double *jdx, double *ds, double *dl) const;
  void ftb(const double *s, const double *ds, const double *lam, const double *dl, IpmScalars *sc,
           bool affine) const;
  void muaff(const double *s, const double *ds, const double *lam, const double *dl, IpmScalars *sc) const;
  void corrector_target(const double *ds, const double *dl, IpmScalars *sc, double *w) const;
  void update(const IpmScalars *sc, double *x, const double *dx, double *s, const double *ds,
              double *lam, const double *dl) const;
};

}  // namespace gipm
