// HDCR solve (Section 4): flexible GCR(m) on H in FP64, preconditioned by the
// two-level V-cycle
//     z1 = S r;   z2 = z1 + P A^{-1} P^dag (r - H z1);   z = z2 + S (r - H z2)
// with S a fixed number of CR steps from zero and A^{-1} a CR solve on the
// coarse operator to a loose tolerance.  For a fixed linear S and an exact
// coarse solve this equals M_outer = S P_L + P_R S + Q - S P_L H S.  The
// preconditioner is nonlinear (CR), which is why the outer iteration is the
// flexible variant.  The preconditioner runs in FP64 or FP32 (inner_dtype);
// the outer orthogonalisation, updates and the true residual are FP64.
// Smoother: CR steps from zero (nonlinear) or the Chebyshev polynomial
// S = H p(H^2) of Section 4 (linear).  Coarse solve: CR on the coarse operator
// or its dense inverse.
#include <chrono>
#include <mutex>
#include <vector>

#include "host_io.cuh"
#include "level2.cuh"
#include "chebyshev.cuh"
#include "coarse.cuh"

namespace hdcr {

// ------------------------------------------------------------------ kernels
template <typename R>
__global__ void sub_kernel(const cpx<R>* __restrict__ a, const cpx<R>* __restrict__ b, cpx<R>* __restrict__ out,
                           long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    st(out + i, ld(a + i) - ld(b + i));
}

template <typename R>
__global__ void add_kernel(cpx<R>* __restrict__ y, const cpx<R>* __restrict__ x, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    st(y + i, ld(y + i) + ld(x + i));
}

// The outer flexible GCR keeps its directions as the preconditioner left them and its images
// w_i orthogonal but not normalised: with beta_ji = <w_j, w> / |w_j|^2 of the i-th image,
//     H z_i = w_i + sum_j<i beta_ji w_j,   r -= a_i w_i,   a_i = <w_i, r> / |w_i|^2,
// and at the end of a cycle x += sum_i y_i z_i with y_i + sum_k>i beta_ik y_k = a_i.  The
// modified Gram-Schmidt steps are those of the normalised form; the z updates (as many
// as the w updates: half of the outer iteration's FP64 work), the scaling of both and
// the x update of every iteration are not made.  A step's update and the next one's inner
// product share a pass: at 16^3 x 32 x 16 the vector work of an iteration with 3.5
// earlier images took 3.5 ms of FP64 pipe and memory in seven kinds of pass.

// beta <- <u, v> / n2, into the double pair ``out``
__device__ __forceinline__ void store_ratio(double re, double im, double n2, double* out) {
  const double s = n2 > 0.0 ? 1.0 / n2 : 0.0;
  out[0] = re * s;
  out[1] = im * s;
}

__global__ void __launch_bounds__(RED_THREADS) gs_dot_kernel(const cpx<double>* __restrict__ u,
                                                             const cpx<double>* __restrict__ v, long long n,
                                                             const double* __restrict__ n2, RedScratch rs,
                                                             double* beta) {
  double acc[2] = {0.0, 0.0};
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const cpx<double> a = ld(u + i), b = ld(v + i);
    acc[0] = fma(a.re, b.re, fma(a.im, b.im, acc[0]));
    acc[1] = fma(a.re, b.im, fma(-a.im, b.re, acc[1]));
  }
  double tot[2];
  if (grid_reduce<2>(acc, rs, tot)) store_ratio(tot[0], tot[1], *n2, beta);
}

// w -= beta wj (wj null: w as it is), then
//   LAST = false: beta_next <- <wn, w> / *n2n
//   LAST = true:  *n2 <- |w|^2,  a <- <w, r> / |w|^2     (wn = r)
template <bool LAST>
__global__ void __launch_bounds__(RED_THREADS) gs_step_kernel(cpx<double>* __restrict__ w,
                                                              const cpx<double>* __restrict__ wj,
                                                              const double* __restrict__ beta,
                                                              const cpx<double>* __restrict__ wn, long long n,
                                                              double* n2, RedScratch rs, double* out) {
  const double br = wj ? beta[0] : 0.0, bi = wj ? beta[1] : 0.0;
  double acc[3] = {0.0, 0.0, 0.0};
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    cpx<double> u = w[i];
    if (wj) {
      const cpx<double> a = ld(wj + i);
      u.re = fma(-br, a.re, fma(bi, a.im, u.re));
      u.im = fma(-br, a.im, fma(-bi, a.re, u.im));
      w[i] = u;
    }
    const cpx<double> q = ld(wn + i);
    if (LAST) {  // <w, r>
      acc[0] = fma(u.re, q.re, fma(u.im, q.im, acc[0]));
      acc[1] = fma(u.re, q.im, fma(-u.im, q.re, acc[1]));
      acc[2] = fma(u.re, u.re, fma(u.im, u.im, acc[2]));
    } else {
      acc[0] = fma(q.re, u.re, fma(q.im, u.im, acc[0]));
      acc[1] = fma(q.re, u.im, fma(-q.im, u.re, acc[1]));
    }
  }
  double tot[3];
  if (grid_reduce<3>(acc, rs, tot)) {
    if (LAST) *n2 = tot[2];
    store_ratio(tot[0], tot[1], *n2, out);
  }
}

// r -= a w;  |r|^2 -> *rr
__global__ void __launch_bounds__(RED_THREADS) fgcr_residual_kernel(cpx<double>* __restrict__ r,
                                                                    const cpx<double>* __restrict__ w, long long n,
                                                                    const double* __restrict__ a, RedScratch rs,
                                                                    double* rr) {
  const double ar = a[0], ai = a[1];
  double acc[1] = {0.0};
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const cpx<double> wv = ld(w + i);
    cpx<double> rv = r[i];
    rv.re = fma(-ar, wv.re, fma(ai, wv.im, rv.re));
    rv.im = fma(-ar, wv.im, fma(-ai, wv.re, rv.im));
    r[i] = rv;
    acc[0] = fma(rv.re, rv.re, fma(rv.im, rv.im, acc[0]));
  }
  double tot[1];
  if (grid_reduce<1>(acc, rs, tot)) *rr = tot[0];
}

// y from a by back substitution over the first m columns; beta_ji at B[2 (i restart + j)]
__global__ void fgcr_coef_kernel(const double* __restrict__ B, const double* __restrict__ a, double* y, int m,
                                 int restart) {
  for (int i = m - 1; i >= 0; --i) {
    double re = a[2 * i], im = a[2 * i + 1];
    for (int k = i + 1; k < m; ++k) {
      const double br = B[2 * (k * restart + i)], bi = B[2 * (k * restart + i) + 1];
      re -= br * y[2 * k] - bi * y[2 * k + 1];
      im -= br * y[2 * k + 1] + bi * y[2 * k];
    }
    y[2 * i] = re;
    y[2 * i + 1] = im;
  }
}

// x += sum_i<m y_i z_i, z_i at Z + i n
__global__ void fgcr_solution_kernel(cpx<double>* __restrict__ x, const cpx<double>* __restrict__ Z, long long n,
                                     const double* __restrict__ y, int m) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    cpx<double> v = x[i];
    for (int k = 0; k < m; ++k) v = cmadd(v, cpx<double>(y[2 * k], y[2 * k + 1]), ld(Z + k * n + i));
    x[i] = v;
  }
}

// ------------------------------------------------------------------ workspace
struct SolveCache {
  int restart = 0;
  int inner = -1;
  long long fs = 0, cs = 0;
  void* mem = nullptr;
  // FP64 outer
  cpx<double>* Z = nullptr;  // restart fields
  cpx<double>* W = nullptr;  // restart fields
  cpx<double>* r = nullptr;
  cpx<double>* tmp = nullptr;
  // inner precision (R): r_in, z_in, t1, t2, e; coarse rhs / solution
  void* r_in = nullptr;
  void* z_in = nullptr;
  void* t1 = nullptr;
  void* t2 = nullptr;
  void* e = nullptr;
  void* c_rhs = nullptr;
  void* c_sol = nullptr;
  void* U_in = nullptr;  // links in the inner precision (FP32 mode)
  void* sw = nullptr;    // CRWork<R> of the smoother
  void* cw = nullptr;    // CRWork<R> of the coarse solve
  void* chw = nullptr;   // ChebWork<R> of the Chebyshev smoother
  std::vector<double> cheb_c;
  double* B = nullptr;   // restart^2 complex beta, then restart each of complex a, complex y, |w|^2
  RedBuffers rb{};       // outer reductions and scalars
  cudaEvent_t ev[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
  FxCtx fx;              // encoded links and fields of the FP64 applications
  CRGraph cgraph;        // the coarse CR's iterations between host checks, replayed every V-cycle
};

template <typename R>
static void free_inner(SolveCache* c) {
  if (c->sw) {
    crwork_free<R>((CRWork<R>*)c->sw);
    delete (CRWork<R>*)c->sw;
  }
  if (c->cw) {
    crwork_free<R>((CRWork<R>*)c->cw);
    delete (CRWork<R>*)c->cw;
  }
  if (c->chw) {
    cheb_work_free<R>((ChebWork<R>*)c->chw);
    delete (ChebWork<R>*)c->chw;
  }
  c->sw = c->cw = c->chw = nullptr;
}

void solve_cache_free(SolveCache* c) {
  if (!c) return;
  if (c->inner == HDCR_C128) free_inner<double>(c);
  if (c->inner == HDCR_C64) free_inner<float>(c);
  cr_graph_free(&c->cgraph);
  fx_ctx_free(&c->fx);
  if (c->mem) cudaFree(c->mem);
  red_buffers_free(&c->rb);
  for (int i = 0; i < 6; ++i)
    if (c->ev[i]) cudaEventDestroy(c->ev[i]);
  delete c;
}

template <typename R>
static int alloc_cache(const hdcr_coarse* co, int restart, SolveCache** out) {
  SolveCache* c = new SolveCache();
  c->restart = restart;
  c->inner = sizeof(R) == 8 ? HDCR_C128 : HDCR_C64;
  c->fs = co->g.V5 * 12;
  c->cs = (long long)co->bg.Vc * co->nvec;
  const size_t f64 = sizeof(cpx<double>) * c->fs, fin = sizeof(cpx<R>) * c->fs, cin = sizeof(cpx<R>) * c->cs;
  // the fields' places, laid out twice: for their total size (base null), then in the memory
  auto lay_out = [&](char* base) {
    size_t at = 0;
    auto take = [&](size_t b) {
      void* q = base + at;
      at += (b + 255) & ~(size_t)255;
      return q;
    };
    c->Z = (cpx<double>*)take(f64 * restart);
    c->W = (cpx<double>*)take(f64 * restart);
    c->r = (cpx<double>*)take(f64);
    c->tmp = (cpx<double>*)take(f64);
    c->r_in = take(fin);
    c->z_in = take(fin);
    c->t1 = take(fin);
    c->t2 = take(fin);
    c->e = take(fin);
    c->c_rhs = take(cin);
    c->c_sol = take(cin);
    c->U_in = take(sizeof(cpx<R>) * (size_t)co->g.V4 * 36);
    c->B = (double*)take(sizeof(double) * restart * (2 * restart + 5));
    return at;
  };
  const size_t bytes = lay_out(nullptr);
  cudaError_t e = dev_malloc(&c->mem, bytes);
  if (e != cudaSuccess) {
    delete c;
    set_error("HDCR workspace: cudaMalloc(%zu) failed: %s", bytes, cudaGetErrorString(e));
    return HDCR_ERR_NO_MEMORY;
  }
  lay_out((char*)c->mem);
  int s = red_buffers_alloc(&c->rb, 192);
  CRWork<R>* sw = new CRWork<R>();
  CRWork<R>* cw = new CRWork<R>();
  ChebWork<R>* chw = new ChebWork<R>();
  c->sw = sw;
  c->cw = cw;
  c->chw = chw;
  if (s == HDCR_OK) s = crwork_alloc<R>(sw, c->fs);
  if (s == HDCR_OK) s = crwork_alloc<R>(cw, c->cs);
  if (s == HDCR_OK) s = cheb_work_alloc<R>(chw, c->fs);
  for (int i = 0; i < 6 && s == HDCR_OK; ++i) {
    if (cudaEventCreate(&c->ev[i]) != cudaSuccess) s = HDCR_ERR_CUDA;
  }
  if (s != HDCR_OK) {
    solve_cache_free(c);  // frees whatever part was allocated
    return s;
  }
  if (!co->cf) fx_ctx_alloc(&c->fx, co->g, 1, sizeof(R) == 8 ? 2 : 1);  // (FP32 V-cycle: the outer H alone)
  *out = c;
  return HDCR_OK;
}

struct VStats {
  int fine = 0;          // inner-precision fine applies
  int coarse = 0;        // coarse stencil applies
  int coarse_dense = 0;  // dense coarse solves
  int coarse_fail = 0;
};

// out = S r (out must not alias r or the workspaces)
template <typename R>
static int smooth(const FineOp<R>& H, SolveCache* c, const hdcr_solve_params* prm, const cpx<R>* r, cpx<R>* out,
                  VStats* vs, cudaStream_t st) {
  if (prm->smoother_kind == HDCR_SMOOTHER_CHEBYSHEV)
    return cheb_smoother<R>(H, r, out, c->cheb_c, prm->cheb_lo, prm->cheb_hi, *(ChebWork<R>*)c->chw, st, &vs->fine);
  CRWork<R>& sw = *(CRWork<R>*)c->sw;
  CRConfig cfg;
  cfg.fixed_iters = prm->smoother_order;
  cfg.x_zero = true;
  CRResult res;
  HDCR_CUDA_TRY(cudaMemsetAsync(out, 0, sizeof(cpx<R>) * c->fs, st));
  HDCR_TRY(cr_run<R>(H, r, out, sw, cfg, &res, st));
  vs->fine += res.matvecs;
  return HDCR_OK;
}

// c_sol = A^{-1} c_rhs (coarse vectors in R)
template <typename R>
static int coarse_solve(const hdcr_coarse* co, SolveCache* c, const hdcr_solve_params* prm, VStats* vs,
                        cudaStream_t st) {
  if (prm->coarse_solver == HDCR_COARSE_RECURSIVE) {
    int it = 0;
    HDCR_TRY(level2_solve<R>(co, (const cpx<R>*)c->c_rhs, (cpx<R>*)c->c_sol, prm->coarse_tol, prm->coarse_max, &it,
                             st));
    vs->coarse += it;
    return HDCR_OK;
  }
  if (prm->coarse_solver == HDCR_COARSE_DENSE) {
    vs->coarse_dense++;
    return launch_dense_solve<R>(co, (const cpx<R>*)c->c_rhs, (cpx<R>*)c->c_sol, 1, st);
  }
  CRWork<R>& cw = *(CRWork<R>*)c->cw;
  HDCR_CUDA_TRY(cudaMemsetAsync(c->c_sol, 0, sizeof(cpx<R>) * c->cs, st));
  CRConfig ccfg;
  ccfg.tol = prm->coarse_tol;
  ccfg.max_iter = prm->coarse_max;
  ccfg.x_zero = true;
  ccfg.check_every = 8;
  ccfg.graph = &c->cgraph;
  CoarseOp<R> A{co};
  CRResult res;
  HDCR_TRY(cr_run<R>(A, (const cpx<R>*)c->c_rhs, (cpx<R>*)c->c_sol, cw, ccfg, &res, st));
  vs->coarse += res.matvecs;
  if (!res.converged) vs->coarse_fail++;
  return HDCR_OK;
}

// out = r - H z (its encoded form left in e1 when ``enc``); in FP64 without the FP64 pipe z is
// encoded first unless ``zin`` holds it already, and the subtraction rides in the application
template <typename R>
static int residual(const FineOp<R>& H, SolveCache* c, const cpx<R>* r, const cpx<R>* z, const FxField* zin, bool enc,
                    cpx<R>* out, cudaStream_t st) {
  if constexpr (sizeof(R) == 8) {
    if (H.fixed()) {
      const FxField in = fx_of(zin ? *zin : H.fx->e0, z);
      if (!zin) HDCR_TRY(launch_fx_encode(H.g, z, H.nrhs, in, nullptr, H.fx->u, st));
      int slot;
      stencil_timer_begin(0, H.g.V5 * H.nrhs, st, &slot);
      const int s = launch_fx_g5dwf_res(H.g, H.M5, H.mf, H.fx->u, in, r, out, enc ? &H.fx->e1 : nullptr, H.nrhs, st);
      stencil_timer_end(slot, st);
      return s;
    }
  }
  cpx<R>* t1 = (cpx<R>*)c->t1;
  HDCR_TRY(H.apply(z, t1, st));
  sub_kernel<R><<<num_blocks(c->fs, 256, 4096), 256, 0, st>>>(r, t1, out, c->fs); count_launch();
  HDCR_LAUNCH_CHECK();
  return HDCR_OK;
}

// e = S t2 after residual(..., enc = true, t2): from its encoded form where there is one
template <typename R>
static int smooth_residual(const FineOp<R>& H, SolveCache* c, const hdcr_solve_params* prm, const cpx<R>* t2, cpx<R>* e,
                           VStats* vs, cudaStream_t st) {
  if constexpr (sizeof(R) == 8)
    if (H.fixed() && prm->smoother_kind == HDCR_SMOOTHER_CHEBYSHEV)
      return cheb_smoother_fx(H, fx_of(H.fx->e1, t2), H.fx->e0, e, c->cheb_c, prm->cheb_lo, prm->cheb_hi,
                              *(ChebWork<double>*)c->chw, st, &vs->fine);
  return smooth<R>(H, c, prm, t2, e, vs, st);
}

// z = B r in precision R (r, z in R)
template <typename R>
static int vcycle(const hdcr_coarse* co, const FineOp<R>& H, SolveCache* c, const hdcr_solve_params* prm,
                  const cpx<R>* r, cpx<R>* z, VStats* vs, cudaStream_t st) {
  const long long fs = c->fs;
  cpx<R>* t2 = (cpx<R>*)c->t2;
  cpx<R>* e = (cpx<R>*)c->e;
  const int nb = num_blocks(fs, 256, 4096);
  if (prm->cycle == HDCR_CYCLE_POST) {
    // z1 = P A^{-1} P^dag r;  z = z1 + S (r - H z1)
    HDCR_CUDA_TRY(cudaEventRecord(c->ev[0], st));
    HDCR_CUDA_TRY(cudaEventRecord(c->ev[1], st));
    HDCR_CUDA_TRY(cudaEventRecord(c->ev[2], st));
    HDCR_TRY(launch_restrict<R>(co->sub, r, (cpx<R>*)c->c_rhs, 1, st));
    HDCR_TRY(coarse_solve<R>(co, c, prm, vs, st));
    HDCR_TRY(launch_prolong<R>(co->sub, (const cpx<R>*)c->c_sol, (const cpx<R>*)nullptr, z, 1, st));
    HDCR_CUDA_TRY(cudaEventRecord(c->ev[3], st));
    HDCR_TRY(residual<R>(H, c, r, z, nullptr, true, t2, st));
    vs->fine++;
    HDCR_CUDA_TRY(cudaEventRecord(c->ev[4], st));
    HDCR_TRY(smooth_residual<R>(H, c, prm, t2, e, vs, st));
    add_kernel<R><<<nb, 256, 0, st>>>(z, e, fs); count_launch();
    HDCR_LAUNCH_CHECK();
    HDCR_CUDA_TRY(cudaEventRecord(c->ev[5], st));
    return HDCR_OK;
  }
  // z1 = S r
  HDCR_CUDA_TRY(cudaEventRecord(c->ev[0], st));
  HDCR_TRY(smooth<R>(H, c, prm, r, z, vs, st));
  HDCR_CUDA_TRY(cudaEventRecord(c->ev[1], st));
  // r1 = r - H z1;  z2 = z1 + P A^{-1} P^dag r1
  // (the Chebyshev smoother leaves z encoded in e1)
  const FxField* zin = H.fixed() && prm->smoother_kind == HDCR_SMOOTHER_CHEBYSHEV ? &H.fx->e1 : nullptr;
  HDCR_TRY(residual<R>(H, c, r, z, zin, false, t2, st));
  vs->fine++;
  HDCR_CUDA_TRY(cudaEventRecord(c->ev[2], st));
  HDCR_TRY(launch_restrict<R>(co->sub, t2, (cpx<R>*)c->c_rhs, 1, st));
  HDCR_TRY(coarse_solve<R>(co, c, prm, vs, st));
  HDCR_TRY(launch_prolong<R>(co->sub, (const cpx<R>*)c->c_sol, z, z, 1, st));
  HDCR_CUDA_TRY(cudaEventRecord(c->ev[3], st));
  // r2 = r - H z2;  z = z2 + S r2
  HDCR_TRY(residual<R>(H, c, r, z, nullptr, true, t2, st));
  vs->fine++;
  HDCR_CUDA_TRY(cudaEventRecord(c->ev[4], st));
  HDCR_TRY(smooth_residual<R>(H, c, prm, t2, e, vs, st));
  add_kernel<R><<<nb, 256, 0, st>>>(z, e, fs); count_launch();
  HDCR_LAUNCH_CHECK();
  HDCR_CUDA_TRY(cudaEventRecord(c->ev[5], st));
  return HDCR_OK;
}

template <typename R>
static int solve_impl(const hdcr_coarse* co, SolveCache* c, const void* U, const cpx<double>* b, cpx<double>* x,
                      const hdcr_solve_params* prm, hdcr_solve_stats* stats, cudaStream_t st) {
  const auto t0 = std::chrono::steady_clock::now();
  const long long fs = c->fs;
  const int nb = num_blocks(fs, 256, 4096);
  FineOp<double> H64{co->g, co->M5, co->mf, (const cpx<double>*)U};
  H64.cf = co->cf;
  H64.fx = &c->fx;
  HDCR_TRY(fx_ctx_links(c->fx, co->g, (const cpx<double>*)U, st));
  const cpx<R>* Uin = (const cpx<R>*)U;
  if (sizeof(R) != 8) {
    HDCR_TRY(launch_convert(U, HDCR_C128, c->U_in, HDCR_C64, (long long)co->g.V4 * 36, st));
    Uin = (const cpx<R>*)c->U_in;
  }
  FineOp<R> Hin{co->g, co->M5, co->mf, Uin};
  Hin.cf = co->cf;
  Hin.fx = &c->fx;
  if (prm->smoother_kind == HDCR_SMOOTHER_CHEBYSHEV)
    c->cheb_c = cheb_inverse_coeffs(prm->cheb_lo, prm->cheb_hi, prm->smoother_order);
  double* scal = c->rb.scal;    // 132: |r|^2; 133: |b|^2
  const int m = c->restart;     // columns that the workspace holds (at least prm->restart)
  double* B = c->B;
  double* ac = B + 2 * m * m;
  double* yc = ac + 2 * m;
  double* wn2 = yc + 2 * m;
  RedScratch rs = c->rb.rs;
  double* ring = pinned_ring();
  if (!ring) {
    set_error("pinned host buffer unavailable");
    return HDCR_ERR_NO_MEMORY;
  }
  // r = b - H x, |b|^2
  HDCR_TRY(H64.apply(x, c->tmp, st));
  sub_kernel<double><<<nb, 256, 0, st>>>(b, c->tmp, c->r, fs); count_launch();
  HDCR_LAUNCH_CHECK();
  HDCR_TRY(launch_norm2<double>(b, fs, rs, scal + 133, st));
  HDCR_TRY(launch_norm2<double>(c->r, fs, rs, scal + 132, st));
  HDCR_CUDA_TRY(cudaMemcpyAsync(ring, scal + 132, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
  HDCR_CUDA_TRY(cudaStreamSynchronize(st));
  const double bb = ring[1];
  double rr = ring[0];
  int fine64 = 1, iters = 0, restarts = 0, status = HDCR_OK;
  VStats vs;
  double t_smooth = 0.0, t_coarse = 0.0;
  if (!(bb == bb) || !(rr == rr) || bb > 1e300) {
    set_error("hdcr_solve: non-finite right-hand side or initial residual");
    return HDCR_ERR_NONFINITE;
  }
  const double tol2 = prm->tol * prm->tol * bb;
  bool converged = bb == 0.0 || rr <= tol2;
  while (!converged && iters < prm->max_outer) {
    int done = 0;  // iterations of this cycle that x takes
    for (int i = 0; i < prm->restart && iters < prm->max_outer; ++i) {
      cpx<double>* z = c->Z + (long long)i * fs;
      cpx<double>* w = c->W + (long long)i * fs;
      // z = B r
      if (sizeof(R) == 8) {
        HDCR_TRY(vcycle<R>(co, Hin, c, prm, (const cpx<R>*)c->r, (cpx<R>*)z, &vs, st));
      } else {
        HDCR_TRY(launch_convert(c->r, HDCR_C128, c->r_in, HDCR_C64, fs, st));
        HDCR_TRY(vcycle<R>(co, Hin, c, prm, (const cpx<R>*)c->r_in, (cpx<R>*)c->z_in, &vs, st));
        HDCR_TRY(launch_convert(c->z_in, HDCR_C64, z, HDCR_C128, fs, st));
      }
      // w = H z, orthogonalised against the earlier w_j;  r -= a w
      HDCR_TRY(H64.apply(z, w, st));
      fine64++;
      const int nr = red_blocks(fs);
      double* col = B + 2 * (size_t)i * m;
      if (i > 0) {
        gs_dot_kernel<<<nr, RED_THREADS, 0, st>>>(c->W, w, fs, wn2, rs, col); count_launch();
      }
      for (int j = 0; j + 1 < i; ++j) {
        gs_step_kernel<false><<<nr, RED_THREADS, 0, st>>>(w, c->W + (long long)j * fs, col + 2 * j,
                                                          c->W + (long long)(j + 1) * fs, fs, wn2 + j + 1, rs,
                                                          col + 2 * (j + 1)); count_launch();
      }
      gs_step_kernel<true><<<nr, RED_THREADS, 0, st>>>(w, i > 0 ? c->W + (long long)(i - 1) * fs : nullptr,
                                                       col + 2 * (i - 1), c->r, fs, wn2 + i, rs, ac + 2 * i); count_launch();
      fgcr_residual_kernel<<<nr, RED_THREADS, 0, st>>>(c->r, w, fs, ac + 2 * i, rs, scal + 132); count_launch();
      HDCR_LAUNCH_CHECK();
      HDCR_CUDA_TRY(cudaMemcpyAsync(ring, scal + 132, sizeof(double), cudaMemcpyDeviceToHost, st));
      HDCR_CUDA_TRY(cudaStreamSynchronize(st));
      float ms = 0.f;
      if (cudaEventElapsedTime(&ms, c->ev[0], c->ev[1]) == cudaSuccess) t_smooth += ms * 1e-3;
      if (cudaEventElapsedTime(&ms, c->ev[4], c->ev[5]) == cudaSuccess) t_smooth += ms * 1e-3;
      if (cudaEventElapsedTime(&ms, c->ev[2], c->ev[3]) == cudaSuccess) t_coarse += ms * 1e-3;
      ++iters;
      rr = ring[0];
      if (!(rr == rr) || rr > 1e300) {
        set_error("hdcr_solve: non-finite residual at outer iteration %d", iters);
        status = HDCR_ERR_NONFINITE;
        break;
      }
      done = i + 1;
      if (rr <= tol2) break;
    }
    // x += Z y over the cycle's iterations (the one that met a non-finite residual left out)
    if (done > 0) {
      fgcr_coef_kernel<<<1, 1, 0, st>>>(B, ac, yc, done, m); count_launch();
      fgcr_solution_kernel<<<nb, 256, 0, st>>>(x, c->Z, fs, yc, done); count_launch();
      HDCR_LAUNCH_CHECK();
    }
    if (status != HDCR_OK) break;
    // true residual (restart or convergence check)
    HDCR_TRY(H64.apply(x, c->tmp, st));
    fine64++;
    sub_kernel<double><<<nb, 256, 0, st>>>(b, c->tmp, c->r, fs); count_launch();
    HDCR_LAUNCH_CHECK();
    HDCR_TRY(launch_norm2<double>(c->r, fs, rs, scal + 132, st));
    HDCR_CUDA_TRY(cudaMemcpyAsync(ring, scal + 132, sizeof(double), cudaMemcpyDeviceToHost, st));
    HDCR_CUDA_TRY(cudaStreamSynchronize(st));
    rr = ring[0];
    ++restarts;
    if (!(rr == rr)) {
      status = HDCR_ERR_NONFINITE;
      set_error("hdcr_solve: non-finite true residual");
      break;
    }
    converged = rr <= tol2;
  }
  if (status == HDCR_OK && !converged) {
    set_error("hdcr_solve: not converged after %d outer iterations (|r|/|b| = %g)", iters,
              bb > 0 ? sqrt(rr / bb) : 0.0);
    status = HDCR_ERR_NOT_CONVERGED;
  }
  if (stats) {
    stats->status = status;
    stats->iters = iters;
    stats->fine_matvecs = fine64 + (sizeof(R) == 8 ? vs.fine : 0);
    stats->fine_matvecs_lo = sizeof(R) == 8 ? 0 : vs.fine;
    stats->coarse_matvecs = vs.coarse + vs.coarse_dense;
    stats->restarts = restarts;
    stats->true_resid = bb > 0 ? sqrt(rr / bb) : 0.0;
    stats->t_total = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    stats->t_smoother = t_smooth;
    stats->t_coarse = t_coarse;
  }
  return status;
}

}  // namespace hdcr

using namespace hdcr;

// The solve workspace is cached per coarse handle (created on first use,
// released by hdcr_coarse_destroy).  Solves on one handle must not overlap.
static std::mutex g_cache_mutex;
static std::vector<std::pair<const hdcr_coarse*, SolveCache*>> g_cache;

static SolveCache** cache_slot(const hdcr_coarse* co) {
  for (auto& p : g_cache)
    if (p.first == co) return &p.second;
  g_cache.push_back({co, nullptr});
  return &g_cache.back().second;
}

namespace hdcr {
void solve_cache_release(const hdcr_coarse* co) {
  std::lock_guard<std::mutex> lock(g_cache_mutex);
  for (size_t i = 0; i < g_cache.size(); ++i)
    if (g_cache[i].first == co) {
      solve_cache_free(g_cache[i].second);
      g_cache.erase(g_cache.begin() + i);
      return;
    }
}
}  // namespace hdcr

static int solve_entry(hdcr_coarse* co, const void* U, const void* b, void* x, const hdcr_solve_params* prm,
                       hdcr_solve_stats* stats, void* stream) {
  HDCR_TRY(coarse_check(co));
  if (!U || !b || !x || !prm || b == x) {
    set_error("hdcr_solve: null pointer or b == x");
    return HDCR_ERR_BAD_ARG;
  }
  if (!(prm->tol > 0.0) || prm->max_outer < 1 || prm->restart < 1 || prm->restart > 64 ||
      prm->smoother_order < 0 || !(prm->coarse_tol > 0.0) || prm->coarse_max < 1 ||
      (prm->smoother_kind != HDCR_SMOOTHER_CR && prm->smoother_kind != HDCR_SMOOTHER_CHEBYSHEV) ||
      (prm->coarse_solver != HDCR_COARSE_CR && prm->coarse_solver != HDCR_COARSE_DENSE &&
       prm->coarse_solver != HDCR_COARSE_RECURSIVE) ||
      (prm->cycle != HDCR_CYCLE_SYMMETRIC && prm->cycle != HDCR_CYCLE_POST)) {
    set_error("hdcr_solve: bad parameters");
    return HDCR_ERR_BAD_ARG;
  }
  if (prm->smoother_kind == HDCR_SMOOTHER_CHEBYSHEV &&
      (prm->smoother_order < 1 || !(prm->cheb_lo > 0.0) || !(prm->cheb_hi > prm->cheb_lo))) {
    set_error("hdcr_solve: Chebyshev smoother needs order >= 1 and 0 < cheb_lo < cheb_hi");
    return HDCR_ERR_BAD_ARG;
  }
  if (prm->inner_dtype != HDCR_C128 && prm->inner_dtype != HDCR_C64) {
    set_error("hdcr_solve: unknown inner dtype %d", prm->inner_dtype);
    return HDCR_ERR_BAD_ARG;
  }
  if (co->dtype != prm->inner_dtype || co->sub->dtype != prm->inner_dtype) {
    set_error("hdcr_solve: basis (%d) and coarse operator (%d) must be stored in the inner dtype %d",
              co->sub->dtype, co->dtype, prm->inner_dtype);
    return HDCR_ERR_BAD_ARG;
  }
  if (prm->coarse_solver == HDCR_COARSE_DENSE && !co->Ainv) HDCR_TRY(coarse_invert(co, as_stream(stream)));
  if (prm->coarse_solver == HDCR_COARSE_RECURSIVE && !co->l2) {
    set_error("hdcr_solve: the recursive coarse solve needs a third level (hdcr_coarse_build_level2)");
    return HDCR_ERR_BAD_ARG;
  }
  cudaStream_t st = as_stream(stream);
  SolveCache* cache = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_cache_mutex);
    SolveCache** slot = cache_slot(co);
    if (*slot && ((*slot)->inner != prm->inner_dtype || (*slot)->restart < prm->restart)) {
      solve_cache_free(*slot);
      *slot = nullptr;
    }
    if (!*slot) {
      int s = prm->inner_dtype == HDCR_C128 ? alloc_cache<double>(co, prm->restart, slot)
                                            : alloc_cache<float>(co, prm->restart, slot);
      if (s != HDCR_OK) return s;
    }
    cache = *slot;
  }
  if (prm->inner_dtype == HDCR_C128)
    return solve_impl<double>(co, cache, U, (const cpx<double>*)b, (cpx<double>*)x, prm, stats, st);
  return solve_impl<float>(co, cache, U, (const cpx<double>*)b, (cpx<double>*)x, prm, stats, st);
}

extern "C" int hdcr_solve(hdcr_coarse* co, const void* U, const void* b, void* x,
                          const hdcr_solve_params* prm, hdcr_solve_stats* stats, void* stream) {
  HDCR_TRY(coarse_check(co));
  if (!U || !b || !x || b == x) {
    set_error("hdcr_solve: null pointer or b == x");
    return HDCR_ERR_BAD_ARG;
  }
  // links, source and solution given in host memory are staged through the device
  cudaStream_t st = as_stream(stream);
  const size_t field = (size_t)co->g.V5 * 12 * 16;
  Staged su, sb, sx;
  HDCR_TRY(su.in(U, (size_t)co->g.V4 * 36 * 16, st));
  HDCR_TRY(sb.in(b, field, st));
  HDCR_TRY(sx.out(x, field, st, true));
  const int s = solve_entry(co, su.ptr(), sb.ptr(), sx.ptr(), prm, stats, stream);
  HDCR_TRY(sx.finish());
  if (sx.ptr() != x) HDCR_CUDA_TRY(cudaStreamSynchronize(st));
  return s;
}
