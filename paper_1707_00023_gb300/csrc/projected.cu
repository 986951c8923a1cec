// FP64 projected (small, dense) work of the Krylov path:
//  * matrix exponentials on a cluster of thread blocks (kx_cdense.cuh),
//  * time sub-step control from Lemma 1's residual (eq. (resid)),
//  * projected solutions with a sine source (eq. (corr2), Corollary 1),
//  * shifted Hessenberg solves of the multi-shift FOM.
#include <atomic>

#include "kx_cdense.cuh"
#include "kx_internal.cuh"

namespace kx {

// ---------------------------------------------------------------------------
// Time sub-step control (restart in time, Sect. 3.3): with the Arnoldi
// decomposition of the current restart, u(t) = exp(-t H_m) beta e_1 is
// tabulated at t_k = k * tau / K, and Lemma 1 gives the residual norm
// ||r_m(t_k)|| = h_{m+1,m} |e_m^T u(t_k)| (||v_{m+1}|| = 1).  The largest t_k
// whose integrated residual (trapezoid rule, an error bound for a
// contractive exp(-tA)) stays below tol_rate * t_k is accepted; if none,
// tau shrinks 4x and the table is rebuilt.
//
// One cluster a slot: the exponential of one step of the table as in
// kx_cdense.cuh, then the table itself, each block multiplying its rows (16
// lanes a row: four products and four sums of the slow double-precision pipe
// in each of two warps) and storing its entries of u into every block's
// shared memory, one cluster barrier a step.  Every block follows the same
// values, so all take the same decisions; block 0 records them.
constexpr int TAB_LANES = 16;
constexpr int TAB_ROWS = MMAX / CD_PORTABLE;   // most rows of a block
constexpr int TAB_STEPS = 32;              // K: steps of the table, one a lane in the check
static_assert(TAB_ROWS * TAB_LANES <= CD_THREADS && MMAX / CD_WIDE * TAB_LANES % 32 == 0, "whole warps");
static_assert(CD_WIDE <= TAB_LANES, "a lane stores to each block");
static_assert((TAB_STEPS + 1) * MMAX <= CD_MAT, "the table fits the right operand's place");

__global__ void __launch_bounds__(CD_THREADS) k_substep(SlotSet<float> ss, int ldh, double* ws) {
  constexpr int K = TAB_STEPS;
  const int C = cl_size(), slot = blockIdx.x / C, rank = cl_rank();
  const Slot<float> sl = slot_at(ss, slot);
  const double* H = sl.H;
  SlotState* st = sl.st;
  extern __shared__ __align__(16) double sm[];
  __shared__ double red[32];
  __shared__ double s_err;
  __shared__ int s_kacc;
  const CdShared sh = cd_shared(sm);
  double* g = ws + (size_t)slot * CD_WS;
  const SlotState s0 = *st;   // block 0 rewrites it at the end, past the last barrier
  if (s0.finished || s0.status || s0.retired) return;
  const int tid = threadIdx.x;
  const int m = s0.m_done;
  if (m <= 0 || s0.beta == 0.0) {
    cl_sync();
    if (rank == 0) {
      for (int i = tid; i < ldh - 1; i += CD_THREADS) sl.u[i] = 0.0;
      if (tid == 0) {
        st->t_now = s0.T;
        st->finished = 1;
      }
    }
    return;
  }
  const CdRows w = cd_rows(m, rank);
  const double hnext = s0.done ? 0.0 : H[m + (int64_t)(m - 1) * ldh];
  const double remaining = s0.T - s0.t_now;
  auto entry = [&](int r, int c) { return r <= c + 1 ? H[r + (int64_t)c * ldh] : 0.0; };
  const double nrm = cd_norm1(m, red, entry);
  double tol_abs = s0.tol_abs;
  if (s0.tol_mode == 0 && !(tol_abs > 0.0)) tol_abs = s0.rtol * s0.beta / s0.T;
  const double tol_rate = s0.tol_mode ? s0.rtol * s0.beta / s0.T : tol_abs;
  // first trial: Krylov dimension over the 1-norm of H_m
  double tau = s0.tau_try > 0.0 ? s0.tau_try : (nrm > 0.0 ? 0.5 * m / nrm : remaining);
  tau = fmin(tau, remaining);
  int evals = 0, kacc = 0;
  double err = 0.0, uacc = 0.0;
  bool bad = false;
  for (int attempt = 0; attempt < 40; ++attempt) {
    const double dt = tau / K;
    int q = 0, s = 0;
    ++evals;
    if (!cd_plan(dt * nrm, 1, &q, &s)) {
      bad = true;
      break;
    }
    const double sc = -ldexp(dt, -s);
    const double* E = cd_expm(sh, g, m, w, q, s, [&](int r, int c) { return sc * entry(r, c); });
    // table of u(t_k), k = 0 .. K, over the (now free) right operand
    double* U = sh.B;
    for (int i = tid; i < m; i += CD_THREADS) U[i] = (i == 0) ? s0.beta : 0.0;
    cl_sync();   // every block past its exponential before another one's stores arrive
    const int row = tid / TAB_LANES, lane = tid % TAB_LANES;
    for (int k = 1; k <= K; ++k) {
      if (tid < MMAX / C * TAB_LANES) {
        const double* u = U + (k - 1) * MMAX;
        double x = 0.0;
        if (row < w.R)
          for (int c = lane; c < m; c += TAB_LANES) x = fma(E[row * CD_LD + c], u[c], x);
#pragma unroll
        for (int o = TAB_LANES / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (row < w.R && lane < C) cl_store(&U[k * MMAX + w.r0 + row], lane, x);
      }
      cl_sync();
    }
    // lane k - 1 of the first warp: the integrated residual up to t_k; the
    // accepted steps are the leading ones within the tolerance
    if (tid < 32) {
      const int k = tid + 1;
      const double rp = k <= K && k >= 2 ? fabs(hnext * U[(k - 1) * MMAX + m - 1]) : 0.0;
      const double rk = k <= K ? fabs(hnext * U[k * MMAX + m - 1]) : 0.0;
      double e = 0.5 * dt * (rp + rk);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, e, o);
        if (tid >= o) e += v;
      }
      const unsigned okm = __ballot_sync(0xffffffffu, k <= K && isfinite(e) && e <= tol_rate * (k * dt));
      const int n = __ffs(~okm) - 1;   // leading accepted steps (32: none refused)
      if (tid == 0) s_kacc = n < 0 ? 32 : n;
      const double ea = __shfl_sync(0xffffffffu, e, max(0, (n < 0 ? 32 : n) - 1));
      if (tid == 0) s_err = ea;
    }
    __syncthreads();
    kacc = s_kacc;
    err = s_err;
    if (kacc > 0 && tid < m) uacc = U[kacc * MMAX + tid];
    cl_sync();   // the table is read: its buffers may be rewritten, a block may end
    if (kacc > 0) break;
    tau *= 0.25;
  }
  if (rank != 0) return;
  if (kacc > 0 && tid < m) sl.u[tid] = uacc;
  if (tid == 0) {
    if (s0.tol_mode == 0) st->tol_abs = tol_abs;
    if (bad) {
      // a failed slot stops: the later kernels of queued sub-steps skip it
      st->status = KX_ENONFINITE;
      st->done = 1;
      return;
    }
    st->expm_evals = s0.expm_evals + evals;
    if (kacc == 0) {
      st->status = KX_ENOCONV;
      st->done = 1;
      return;
    }
    const double dt = tau / K;
    const bool to_end = (tau >= remaining);
    const double tacc = (kacc == K && to_end) ? remaining : kacc * dt;
    const double t_now = (kacc == K && to_end) ? s0.T : s0.t_now + tacc;
    st->t_now = t_now;
    st->t_acc = tacc;
    st->err_acc = s0.err_acc + err;
    st->k_acc = kacc;
    st->substeps = s0.substeps + 1;
    if (kacc == K) st->tau_try = to_end ? s0.tau_try : tau * 1.5;
    else st->tau_try = tacc * 1.1;
    st->finished = (t_now >= s0.T) ? 1 : 0;
  }
}

kx_status launch_substep_control(kx_ctx* c, int slot, int ns) {
  const int m = c->m;
  static ClusterOptIn attr{};
  int blocks = 0;
  const kx_status so = cluster_opt_in(c, attr, (const void*)k_substep, CD_SMEM, &blocks);
  if (so != KX_OK) return so;
  time_begin(c);
  launch_cluster(k_substep, blocks, ns, CD_SMEM, c->stream, make_slotset<float>(c, slot), m + 1, c->d_cd_ws);
  time_end(c, KX_K_PROJ, 0.0);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

// ---------------------------------------------------------------------------
// Projected solutions:
//   nfreq == 0:  u = exp(-tau H_m) beta e_1
//   otherwise :  u_f = [exp(tau N_f)]_{0..m-1, m+1},
//                N_f = [[-H_m, beta e_1, 0], [0, 0, W_f], [0, -W_f, 0]],
// the exact solution of u' = -H_m u + sin(W_f t) beta e_1, u(0) = 0, whose
// two extra states carry sin and cos of W_f t (eq. (corr2)).
//
// N_f = [[A, B], [0, J_f]] is block triangular with the same A for every
// frequency, so one cluster carries X = exp(A) once and, beside it, only the
// two columns Y_f of the upper right block of every exp(N_f):
//   series   : N^k has the upper right block B_k = sum_{i<k} A^{k-1-i} B J^i,
//              a combination of e_1, A e_1, .., A^3 e_1 for k <= 4, so the
//              Horner step P <- P A^4 + C, Y <- P B_4 + Y J^4 + D takes the
//              four extra columns P A^i e_1, whatever nfreq;
//   squaring : X <- X^2, Y <- X Y + Y exp(J).
// Against one exponential of order m + 2 a frequency, each on one block (32
// frequencies, m = 64, tau ||H|| = 40: 1337 us) now 155 us.
constexpr int PHI_YLD = 2 * MAXF;                       // row stride of the Y block
constexpr int PHI_SMEM = CD_SMEM + (2 * CD_RMAX + MMAX) * PHI_YLD * (int)sizeof(double);
static_assert(CD_WS_MATS * CD_MAT + 2 * MMAX * PHI_YLD <= 2 * CD_WS, "the workspace of two clusters holds it");

// The solutions of nfreq frequencies om[sel[f]] (none: the plain exponential),
// series degree 4 q and s squarings for all.  exp of the 2 x 2 rotation generator
// [[0, w], [-w, 0]] acts on a row (a, b) from the right as (a cos w - b sin w,
// a sin w + b cos w).  Every thread of the cluster calls it.
__device__ void phi_group(const double* H, int ldh, int m, double beta, double tau, const double* om, const int* sel,
                          int nfreq, int q, int s, double* u_out, double* sm, double* ws) {
  __shared__ double wd[MAXF];          // W_f d
  __shared__ double pa[CD_RMAX][4];
  const int rank = cl_rank(), tid = threadIdx.x;
  const CdShared sh = cd_shared(sm);
  double* Ya = sm + CD_SMEM / sizeof(double);   // own rows of Y, two in turn
  double* Yb = Ya + CD_RMAX * PHI_YLD;
  double* Yf = Yb + CD_RMAX * PHI_YLD;          // Y whole
  double* gY = ws + CD_WS_MATS * CD_MAT;
  const CdRows w = cd_rows(m, rank);
  const int ny = 2 * nfreq;
  auto entry = [&](int r, int c) { return H[r + (int64_t)c * ldh]; };
  const double d = ldexp(tau, -s);
  for (int f = tid; f < nfreq; f += CD_THREADS) wd[f] = om[sel[f]] * d;
  // a_p = A^p e_1, p < 4, A = -d H: exchanged below
  auto xe = [&](int r, int c) { return -d * entry(r, c); };
  cd_powers(sh, ws, m, w, xe);
  for (int r = tid; r < w.R; r += CD_THREADS)
    for (int p = 0; p < 3; ++p) gY[MMAX * PHI_YLD + (w.r0 + r) * 4 + p] = sh.S[p][r * CD_LD];
  cl_sync();
  cd_load(sh.B, ws, m, m);
  __syncthreads();
  // a_0 .. a_3 beside A^4 in the right operand (columns m .. m + 3)
  for (int o = tid; o < 4 * m; o += CD_THREADS) {
    const int r = o >> 2, p = o & 3;
    sh.B[r * CD_LD + m + p] = p == 0 ? (r == 0 ? 1.0 : 0.0) : __ldcg(gY + MMAX * PHI_YLD + r * 4 + p - 1);
  }
  __syncthreads();
  // B_k of frequency f at own row r: d sum_{i<k} a_{k-1-i}(r) (e_1^T J^i),
  // e_1^T J^i = (1,0), (0,w), (-w^2,0), (0,-w^3)
  auto bk = [&](int k, int r, double x, double* o0, double* o1) {
    const double* a = sh.B + (w.r0 + r) * CD_LD + m;
    double p0 = a[k - 1], p1 = 0.0;
    if (k >= 2) p1 = x * a[k - 2];
    if (k >= 3) p0 = fma(-x * x, a[k - 3], p0);
    if (k >= 4) p1 = fma(-x * x * x, a[k - 4], p1);
    *o0 = d * p0;
    *o1 = d * p1;
  };
  double cf[4];
  const double top = c_rfact[4 * q];
  for (int i = 0; i < 4; ++i) cf[i] = c_rfact[4 * q - 4 + i];
  for (int o = tid; o < w.R * m; o += CD_THREADS) {
    const int r = o / m, c = o - r * m;
    sh.S[4][r * CD_LD + c] = fma(top, sh.S[3][r * CD_LD + c], cd_poly(sh, cf, w, r, c));
  }
  for (int o = tid; o < w.R * nfreq; o += CD_THREADS) {
    const int r = o / nfreq, f = o - r * nfreq;
    const double x = wd[f];
    double y0 = 0.0, y1 = 0.0, b0, b1;
    for (int i = 1; i <= 4; ++i) {
      bk(i, r, x, &b0, &b1);
      const double ci = i == 4 ? top : cf[i];
      y0 = fma(ci, b0, y0);
      y1 = fma(ci, b1, y1);
    }
    Ya[r * PHI_YLD + 2 * f] = y0;
    Ya[r * PHI_YLD + 2 * f + 1] = y1;
  }
  __syncthreads();
  double *P = sh.S[4], *Q = sh.S[3], *Y = Ya, *Z = Yb;
  for (int b = q - 2; b >= 0; --b) {
    for (int i = 0; i < 4; ++i) cf[i] = c_rfact[4 * b + i];
    cd_mm(P, sh.B, w.R, m, m + 4, [&](int r, int c, double v) {
      if (c < m) Q[r * CD_LD + c] = v + cd_poly(sh, cf, w, r, c);
      else pa[r][c - m] = v;
    });
    __syncthreads();
    for (int o = tid; o < w.R * nfreq; o += CD_THREADS) {
      const int r = o / nfreq, f = o - r * nfreq;
      const double x = wd[f], x2 = x * x;
      const double* pv = pa[r];   // P B_4 = d (P a_3 - w^2 P a_1, w P a_2 - w^3 P a_0)
      const double p0 = d * fma(-x2, pv[1], pv[3]), p1 = d * x * fma(-x2, pv[0], pv[2]);
      // J^4 = w^4 I
      double y0 = fma(x2 * x2, Y[r * PHI_YLD + 2 * f], p0), y1 = fma(x2 * x2, Y[r * PHI_YLD + 2 * f + 1], p1);
      double b0, b1;
      for (int i = 1; i < 4; ++i) {
        bk(i, r, x, &b0, &b1);
        y0 = fma(cf[i], b0, y0);
        y1 = fma(cf[i], b1, y1);
      }
      Z[r * PHI_YLD + 2 * f] = y0;
      Z[r * PHI_YLD + 2 * f + 1] = y1;
    }
    __syncthreads();
    double* t = P; P = Q; Q = t;
    t = Y; Y = Z; Z = t;
  }
  // nfreq == 0: the column exp(A) e_1 beta itself takes Y's place at the end
  for (int k = 0; k < s; ++k) {
    double* gk = ws + ((k & 1) ? 0 : 1) * CD_MAT;
    double* gy = gY + (size_t)(k & 1) * MMAX * PHI_YLD;
    for (int o = tid; o < w.R * m; o += CD_THREADS) {
      const int r = o / m, c = o - r * m;
      gk[(w.r0 + r) * CD_LD + c] = P[r * CD_LD + c];
    }
    for (int o = tid; o < w.R * ny; o += CD_THREADS) {
      const int r = o / ny, c = o - r * ny;
      gy[(size_t)(w.r0 + r) * PHI_YLD + c] = Y[r * PHI_YLD + c];
    }
    cl_sync();
    const bool last = k == s - 1;
    if (!last || ny == 0) cd_load(sh.B, gk, m, m);
    for (int o = tid; o < m * nfreq; o += CD_THREADS) {
      const int r = o / nfreq, f = o - r * nfreq;
      *reinterpret_cast<double2*>(Yf + r * PHI_YLD + 2 * f) =
          __ldcg(reinterpret_cast<const double2*>(gy + (size_t)r * PHI_YLD + 2 * f));
    }
    __syncthreads();
    // Y <- X Y + Y exp(J): own rows of X times the whole Y (two columns a
    // thread: one load of X's entry serves both)
    const double2* Yf2 = reinterpret_cast<const double2*>(Yf);
    for (int o = tid; o < w.R * nfreq; o += CD_THREADS) {
      const int r = o / nfreq, f = o - r * nfreq;
      double v0 = 0.0, v1 = 0.0;
      for (int i = 0; i < m; ++i) {
        const double x = P[r * CD_LD + i];
        const double2 yv = Yf2[i * (PHI_YLD / 2) + f];
        v0 = fma(x, yv.x, v0);
        v1 = fma(x, yv.y, v1);
      }
      double sn, cs;
      sincos(ldexp(wd[f], k), &sn, &cs);
      const double a = Y[r * PHI_YLD + 2 * f], b = Y[r * PHI_YLD + 2 * f + 1];
      Z[r * PHI_YLD + 2 * f] = v0 + (a * cs - b * sn);
      Z[r * PHI_YLD + 2 * f + 1] = v1 + (a * sn + b * cs);
    }
    // the last level needs X^2 only where no frequency is asked for, and then
    // its first column alone
    if (!last) cd_mm(P, sh.B, w.R, m, m, [&](int r, int c, double v) { Q[r * CD_LD + c] = v; });
    else if (ny == 0) cd_mm(P, sh.B, w.R, m, 1, [&](int r, int c, double v) { Q[r * CD_LD + c] = v; });
    __syncthreads();
    double* t = P; P = Q; Q = t;
    t = Y; Y = Z; Z = t;
  }
  if (nfreq == 0) {
    for (int r = tid; r < w.R; r += CD_THREADS) u_out[w.r0 + r] = beta * P[r * CD_LD];
  } else {
    for (int o = tid; o < w.R * nfreq; o += CD_THREADS) {
      const int f = o / w.R, r = o - f * w.R;
      u_out[(int64_t)sel[f] * m + w.r0 + r] = beta * Y[r * PHI_YLD + 2 * f + 1];
    }
  }
}

__global__ void __launch_bounds__(CD_THREADS) k_expm_project(const double* H, int ldh, int m, double beta,
                                                             double tau, const double* om, int nfreq,
                                                             double* u_out, int* status, double* ws) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double red[32], pnorm[MAXF];
  __shared__ int pq[MAXF], ps[MAXF], sel[MAXF];
  const int tid = threadIdx.x, nf = max(nfreq, 1);
  const double hn = cd_norm1(m, red, [&](int r, int c) { return H[r + (int64_t)c * ldh]; });
  // Each frequency's norm of tau N_f with beta = 1 (u is linear in beta, which
  // scales the result at the end) and the plan for it.  Below ||H|| = 1 the
  // source's column, whose size is arbitrary, counts as ||H||: the terms of the
  // upper right block are bounded by powers of ||H|| + W.
  if (tid < nf) {
    pnorm[tid] = fabs(tau) * (nfreq > 0 ? fmax(hn, fabs(om[tid]) + fmin(1.0, hn)) : hn);
    if (!cd_plan(pnorm[tid], nfreq > 0 ? 2 : 1, &pq[tid], &ps[tid])) ps[tid] = -1;
  }
  __syncthreads();
  for (int f = 0; f < nf; ++f)
    if (ps[f] < 0) {
      if (cl_rank() == 0 && tid == 0) *status = KX_ENONFINITE;
      return;
    }
  // One group, the rule, unless the squarings differ by more than one: under a
  // larger scaling than its own a frequency loses a bit a squaring (W = 0.4
  // beside 300, tau = 10: 1.4e-14 off instead of 4e-16).
  uint64_t todo = nf < 64 ? (1ull << nf) - 1ull : ~0ull;
  static_assert(MAXF <= 64, "a bit a frequency");
  for (;;) {
    int lead = -1, count = 0;
    for (int f = 0; f < nf; ++f)
      if ((todo >> f) & 1u && (lead < 0 || pnorm[f] > pnorm[lead])) lead = f;
    for (int f = 0; f < nf; ++f)
      if ((todo >> f) & 1u && ps[f] >= ps[lead] - 1) {
        todo &= ~(1ull << f);
        if (tid == 0) sel[count] = f;
        ++count;
      }
    __syncthreads();
    phi_group(H, ldh, m, beta, tau, om, sel, nfreq > 0 ? count : 0, pq[lead], ps[lead], u_out, sm, ws);
    if (!todo) return;
    cl_sync();   // the exchanged matrices are read by every block
  }
}

kx_status launch_expm_project(kx_ctx* c, const double* dH, int ldh, int m, double beta, double tau,
                              const double* d_om, int nfreq, double* d_u) {
  static ClusterOptIn attr{};
  int blocks = 0;
  const kx_status so = cluster_opt_in(c, attr, (const void*)k_expm_project, PHI_SMEM, &blocks);
  if (so != KX_OK) return so;
  int* status = reinterpret_cast<int*>(c->d_small + 64);
  time_begin(c);
  launch_cluster(k_expm_project, blocks, 1, PHI_SMEM, c->stream, dH, ldh, m, beta, tau, d_om, nfreq, d_u, status,
                 c->d_cd_ws);
  time_end(c, KX_K_PROJ, 0.0);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

// ---------------------------------------------------------------------------
// Shifted Hessenberg solves of the restarted multi-shift FOM (one warp per
// shift f):  (H_m + i W_f I) c_f = rho_f e_1,  then
//   coef_f = scale .* c_f  (real and imaginary parts, for z_f += V_m c_f),
//   rho_f <- -h_{m+1,m} e_m^T c_f   (the new residual is rho_f v_{m+1}).
// Gaussian elimination with partial pivoting between the two candidate
// rows of each column keeps the Hessenberg structure; the upper factor is
// kept in shared memory for the back substitution.  A chain of 2 m dependent
// double-precision steps, so what counts is the dependent operations in each:
// magnitudes by |re| + |im| (LAPACK's choice for pivots) instead of hypot, and
// the back substitution by columns (no sum over the lanes), its right-hand
// side carried with its rounding errors: in plain double precision the
// columns' order gave solutions 1.1e-15 from exact ones where the rows' sums
// gave 0.75e-15 (carried: 0.75e-15).  A stationary solve of ten cycles, m = 64,
// 8 shifts, 45 x 38 x 52 in double precision: 77.3 -> 76.5 ms.
struct cplx { double r, i; };
__device__ __forceinline__ cplx cmul(cplx a, cplx b) { return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r}; }
__device__ __forceinline__ cplx csub(cplx a, cplx b) { return {a.r - b.r, a.i - b.i}; }
__device__ __forceinline__ double cabs1(cplx a) { return fabs(a.r) + fabs(a.i); }
__device__ __forceinline__ cplx cdiv(cplx a, cplx b) {
  const double n2 = b.r * b.r + b.i * b.i;
  if (n2 > 1e-280 && n2 < 1e280) {
    const cplx t = cmul(a, cplx{b.r, -b.i});
    return {t.r / n2, t.i / n2};
  }
  // Smith's algorithm where the squares leave the range
  if (fabs(b.r) >= fabs(b.i)) {
    const double q = b.i / b.r, d = b.r + b.i * q;
    return {(a.r + a.i * q) / d, (a.i - a.r * q) / d};
  }
  const double q = b.r / b.i, d = b.r * q + b.i;
  return {(a.r * q + a.i) / d, (a.i * q - a.r) / d};
}

template <typename T>
__global__ void k_shifted(const double* H, int ldh, int m, const double* scale, const double* om,
                          double* rho, T* coef, int* status) {
  extern __shared__ double smx[];
  cplx* U = reinterpret_cast<cplx*>(smx);          // m x m upper factor, row stride m + 1
  const int f = blockIdx.x, ldu = m + 1;
  const int lane = threadIdx.x;
  const double W = om[f];
  auto Hc = [&](int r, int c) -> cplx {
    cplx v = {0.0, 0.0};
    if (r < m && c < m && r <= c + 1) v.r = H[r + (int64_t)c * ldh];
    if (r == c) v.i = W;
    return v;
  };
  auto bcast = [&](cplx v, int l) -> cplx {
    return {__shfl_sync(0xffffffffu, v.r, l), __shfl_sync(0xffffffffu, v.i, l)};
  };
  // current pivot-candidate row (columns k..m-1) held across lanes; the next
  // one is loaded a step ahead
  cplx cur[2], ahead[2], y[2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int q = 0; q < 2; ++q) {
    cur[q] = Hc(0, lane + 32 * q);
    ahead[q] = Hc(1, lane + 32 * q);
  }
  cplx rcur = {rho[2 * f], rho[2 * f + 1]};
  bool ok = true;
  for (int k = 0; k < m; ++k) {
    cplx nxt[2];
    for (int q = 0; q < 2; ++q) {
      nxt[q] = ahead[q];
      ahead[q] = Hc(k + 2, lane + 32 * q);
    }
    cplx rnxt = {0.0, 0.0};
    // diagonal entries at column k
    const int ll = k & 31;
    cplx dk = bcast(k < 32 ? cur[0] : cur[1], ll), nk = bcast(k < 32 ? nxt[0] : nxt[1], ll);
    const bool swap = (k + 1 < m) && (cabs1(nk) > cabs1(dk));
    if (swap) {
      for (int q = 0; q < 2; ++q) { const cplx t = cur[q]; cur[q] = nxt[q]; nxt[q] = t; }
      const cplx t = rcur; rcur = rnxt; rnxt = t;
      const cplx t2 = dk; dk = nk; nk = t2;
    }
    if (!(cabs1(dk) > 0.0)) ok = false;
    // pivot row is U's row k
    for (int q = 0; q < 2; ++q) { const int c = lane + 32 * q; if (c < m) U[k * ldu + c] = cur[q]; }
    if (lane == ll) y[k >> 5] = rcur;
    if (k + 1 < m && ok) {
      const cplx l = cdiv(nk, dk);
      for (int q = 0; q < 2; ++q) cur[q] = csub(nxt[q], cmul(l, cur[q]));
      rcur = csub(rnxt, cmul(l, rcur));
    }
  }
  __syncwarp();
  if (!ok) {
    if (lane == 0) *status = KX_ENONFINITE;
    return;
  }
  // back substitution by columns: lane holds rows lane and lane + 32
  cplx dg[2];
  for (int q = 0; q < 2; ++q) {
    const int r = lane + 32 * q;
    dg[q] = r < m ? U[r * ldu + r] : cplx{1.0, 0.0};
  }
  // t - a b with its rounding error added to e (exact for t and the result
  // within a factor 2)
  auto sub = [](double& t, double& e, double a, double b) {
    const double n = fma(-a, b, t);
    e += fma(-a, b, t - n);
    t = n;
  };
  cplx lo[2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int k = m - 1; k >= 0; --k) {
    const int h = k >> 5;
    const cplx yk = h ? cplx{y[1].r + lo[1].r, y[1].i + lo[1].i} : cplx{y[0].r + lo[0].r, y[0].i + lo[0].i};
    const cplx x = bcast(cdiv(yk, h ? dg[1] : dg[0]), k & 31);
    for (int q = 0; q < 2; ++q) {
      const int r = lane + 32 * q;
      if (r < k) {
        const cplx u = U[r * ldu + k];
        sub(y[q].r, lo[q].r, u.r, x.r);
        sub(y[q].r, lo[q].r, -u.i, x.i);
        sub(y[q].i, lo[q].i, u.r, x.i);
        sub(y[q].i, lo[q].i, u.i, x.r);
      } else if (r == k) {
        y[q] = x;
      }
    }
  }
  for (int q = 0; q < 2; ++q) {
    const int i = lane + 32 * q;
    const double sc = (i < m) ? scale[i] : 0.0;
    coef[(2 * f) * MMAX + i] = (T)(i < m ? y[q].r * sc : 0.0);
    coef[(2 * f + 1) * MMAX + i] = (T)(i < m ? y[q].i * sc : 0.0);
    if (i == m - 1) {
      const double h = H[m + (int64_t)(m - 1) * ldh];
      rho[2 * f] = -h * y[q].r;
      rho[2 * f + 1] = -h * y[q].i;
    }
  }
}

kx_status launch_shifted_solve(kx_ctx* c, int slot, int nfreq, int m) {
  Slot<double> s = make_slot<double>(c, slot);
  int* status = reinterpret_cast<int*>(c->d_small + 64);
  const size_t sm = (size_t)m * (m + 1) * sizeof(cplx);
  static SmemOptIn attr_f{}, attr_d{};
  kx_status so = smem_opt_in(c, attr_f, (const void*)k_shifted<float>, MMAX * (MMAX + 1) * sizeof(cplx));
  if (so == KX_OK) so = smem_opt_in(c, attr_d, (const void*)k_shifted<double>, MMAX * (MMAX + 1) * sizeof(cplx));
  if (so != KX_OK) return so;
  time_begin(c);
  struct End { kx_ctx* c; ~End() { time_end(c, KX_K_PROJ, 0.0); } } end{c};
  if (c->d.precision == KX_FP64)
    k_shifted<double><<<nfreq, 32, sm, c->stream>>>(s.H, c->m + 1, m, s.scale, c->d_omegas, c->d_rho,
                                                     c->d_coefd, status);
  else
    k_shifted<float><<<nfreq, 32, sm, c->stream>>>(s.H, c->m + 1, m, s.scale, c->d_omegas, c->d_rho,
                                                    c->d_coef, status);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

}  // namespace kx
