// Adjoint of the frequency responses: gradient of the summed output-plane
// intensity L = sum_f sum_plane |E_f(T)|^2 with respect to the per-cell
// permittivity.  (The paper has no gradient; this follows from eq. (ode).)
//
//   dL/deps_c = -sum_f int_0^T lambda_f(t)^T (dA/deps_c) y_f(t) dt,
//   lambda_f(t) = exp(-(T - t) A^T) lambda_f(T),  lambda_f(T) = 2 P^T P y_f(T),
//   (dA/deps_c) y |_e = -(1 / (4 eps_e)) (A y)_e   for the E nodes e around c,
// so dL/deps_c = (1/4) sum_{e around c} Q_e with
//   Q_e = sum_f int_0^T lambda_e(t) (A y)_e(t) / eps_e dt.
//
// Per time sub-step [t_k, t_k + tau_k] of the forward solution (restarted
// in time), y(t_k + s) = V u(s) from the forward basis recomputed from the
// checkpoint y(t_k), (A y) = V_{m+1} H u + sin(W t) g from its Arnoldi
// relation, and lambda(t_k + s) = W w(tau_k - s) from an Arnoldi basis of A^T
// started at lambda(t_k + tau_k).  The integral over the sub-step is
// composite Gauss-Legendre quadrature; the projected coefficients u, w at the
// nodes are exact exponentials of the projected matrices.
#include <algorithm>
#include <cmath>
#include <vector>

#include <atomic>

#include "kx_cdense.cuh"
#include "kx_eft.cuh"
#include "kx_internal.cuh"

namespace kx {

constexpr int GAUSS_P = 8;          // Gauss-Legendre nodes per sub-interval
constexpr double QUAD_DELTA = 0.4;  // longest sub-interval (time units)

// lambda(T) = 2 P^T P y: plane values of the E components, zero elsewhere.
template <typename T>
__global__ void k_adj_seed(Geo g, int axis, int idx, const T* __restrict__ y, T* __restrict__ lam) {
  const int nE = g.ne;
  int na, nb;
  if (g.dim == 2) {
    na = axis == 0 ? g.ny : g.nx;
    nb = 1;
  } else {
    na = axis == 0 ? g.ny : g.nx;
    nb = axis == 2 ? g.ny : g.nz;
  }
  const int64_t np = (int64_t)na * nb;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nE * np;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int q = (int)(t / np);
    const int64_t p = t % np;
    const int a = (int)(p % na), b = (int)(p / na);
    int i, j, k;
    if (g.dim == 2) {
      k = 0;
      if (axis == 0) { i = idx; j = a; } else { i = a; j = idx; }
    } else if (axis == 0) { i = idx; j = a; k = b; }
    else if (axis == 1) { i = a; j = idx; k = b; }
    else { i = a; j = b; k = idx; }
    const int64_t e = (int64_t)(g.nh + q) * g.ncell + ((int64_t)k * g.ny + j) * g.nx + i;
    lam[e] = (T)(2.0 * (double)y[e]);
  }
}

// exp(-delta H_m) of the forward basis (cluster 0, slot 0) and the adjoint
// basis (cluster 1, slot 1), rows with stride CD_LD in the cluster's global
// matrix ADJ_E (kx_cdense.cuh).
constexpr int ADJ_E = 2 * CD_MAT;

__global__ void __launch_bounds__(CD_THREADS) k_adj_expm(SlotSet<float> ss, int ldh, double delta, double* ws,
                                                         int* status) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double red[32];
  const int which = blockIdx.x / cl_size(), rank = cl_rank();
  const Slot<float> sl = slot_at(ss, which);
  const double* H = sl.H;
  const int m = sl.st->m_done;
  if (m <= 0 || sl.st->beta == 0.0) return;   // zero state: no coefficients are formed
  auto entry = [&](int r, int c) { return r <= c + 1 ? H[r + (int64_t)c * ldh] : 0.0; };
  int q = 0, s = 0;
  if (!cd_plan(delta * cd_norm1(m, red, entry), 1, &q, &s)) {
    if (rank == 0 && threadIdx.x == 0) *status = KX_ENONFINITE;
    return;
  }
  const CdRows w = cd_rows(m, rank);
  const double sc = -ldexp(delta, -s);
  double* g = ws + (size_t)which * CD_WS;
  const double* E = cd_expm(cd_shared(sm), g, m, w, q, s, [&](int r, int c) { return sc * entry(r, c); });
  for (int o = threadIdx.x; o < w.R * m; o += CD_THREADS) {
    const int r = o / m, c = o - r * m;
    g[ADJ_E + (w.r0 + r) * CD_LD + c] = E[r * CD_LD + c];
  }
}

// M x with M's entries in registers, four threads a row (columns part + 4 k);
// the sum in every lane of the row's four.
__device__ __forceinline__ double adj_row(const double* Mr, const double* x, int part) {
  double a = 0.0, b = 0.0;
#pragma unroll
  for (int k = 0; k < 16; k += 2) {
    a = fma(Mr[k], x[part + 4 * k], a);
    b = fma(Mr[k + 1], x[part + 4 * k + 4], b);
  }
  a += b;
  a += __shfl_xor_sync(0xffffffffu, a, 1);
  a += __shfl_xor_sync(0xffffffffu, a, 2);
  return a;
}

// Projected quadrature coefficients of one sub-step, one block for each
// Gauss node j (blockIdx.x) and basis (blockIdx.y: 0 forward, slot 0; 1
// adjoint, slot 1).
//   nodes s_q = (i + x_j) delta, q = i * P + j, delta = tau / nsub
//   alpha[q][r] = scale_V[r] (H_V u(s_q))_r,  r <= m_V   (A y at s_q)
//   alpha[q][MMAX + 1] = sin(W (t_k + s_q))              (the source's factor)
//   omg[q][r]   = scale_W[r] w(tau - s_q)_r,  r < m_W    (lambda at s_q)
//   cw[q] = delta * wg[j]
//   block (P, 1): slot 1's u = w(tau)   (lambda at t_k, for the next sub-step)
// The start exp(-x_j delta H) beta e_1 by its Taylor series, then nsub
// products with E = exp(-delta H).  Marching the eight nodes one after the
// other on one block, with the exponential before them, took 2.0 ms at m =
// 64, tau = 12; each product is bound by the double-precision pipe (1.2 us).
constexpr int ADJ_A = MMAX + 2;   // stored alpha rows a node

__global__ void __launch_bounds__(256) k_adj_march(SlotSet<float> ss, int ldh, double tau, int nsub,
                                                   const double* __restrict__ xg, const double* __restrict__ wg,
                                                   double omega, double tk, const double* __restrict__ ws,
                                                   double* __restrict__ alpha, double* __restrict__ omg,
                                                   double* __restrict__ cw) {
  const int which = blockIdx.y, j = blockIdx.x, tid = threadIdx.x;
  const bool end = j == GAUSS_P;
  if (end && which == 0) return;
  __shared__ double z[2][MMAX], scl[MMAX + 1], red[32];
  const Slot<float> sl = slot_at(ss, which);
  const double* H = sl.H;
  const int m = sl.st->m_done;
  const double beta = sl.st->beta;
  const double delta = tau / nsub;
  const bool zero = m <= 0 || beta == 0.0;
  if (!end && which == 0)
    for (int i = tid; i < nsub; i += blockDim.x) {
      cw[i * GAUSS_P + j] = delta * wg[j];
      alpha[(size_t)(i * GAUSS_P + j) * ADJ_A + MMAX + 1] = sin(omega * (tk + (i + xg[j]) * delta));
    }
  if (zero) {
    // zero state: every coefficient vanishes
    if (end) {
      if (tid < ldh - 1) sl.u[tid] = 0.0;
      return;
    }
    for (int i = 0; i < nsub; ++i) {
      const size_t q = (size_t)i * GAUSS_P + j;
      if (which == 0 && tid <= MMAX) alpha[q * ADJ_A + tid] = 0.0;
      if (which == 1 && tid < MMAX) omg[q * MMAX + tid] = 0.0;
    }
    return;
  }
  const int r = tid >> 2, part = tid & 3;
  const double* E = ws + (size_t)which * CD_WS + ADJ_E;
  double Er[16], Hr[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int c = part + 4 * k;
    Er[k] = r < m && c < m ? E[r * CD_LD + c] : 0.0;
    Hr[k] = r < m && c < m && r <= c + 1 ? H[r + (int64_t)c * ldh] : 0.0;
  }
  if (tid < MMAX) z[0][tid] = tid == 0 ? beta : 0.0;
  if (tid <= m) scl[tid] = sl.scale[tid];
  double hn = 0.0;   // ||H||_inf bounds the Taylor terms
  {
    double a = 0.0;
#pragma unroll
    for (int k = 0; k < 16; ++k) a += fabs(Hr[k]);
    a += __shfl_xor_sync(0xffffffffu, a, 1);
    a += __shfl_xor_sync(0xffffffffu, a, 2);
    for (int o = 16; o > 2; o >>= 1) a = fmax(a, __shfl_xor_sync(0xffffffffu, a, o));
    if ((tid & 31) == 0) red[tid >> 5] = a;
    __syncthreads();
    for (int q = 0; q < 8; ++q) hn = fmax(hn, red[q]);
  }
  int cur = 0;
  if (!end) {
    const double h = -xg[j] * delta;
    int terms = 0;
    for (double t = 1.0; t > 1e-18 && terms < 60; t *= fabs(h) * hn / terms) ++terms;
    double acc = r == 0 ? beta : 0.0;
    for (int kk = 1; kk <= terms; ++kk) {
      const double v = adj_row(Hr, z[cur], part) * (h / kk);
      acc += v;
      if (part == 0) z[cur ^ 1][r] = v;
      __syncthreads();
      cur ^= 1;
    }
    if (part == 0) z[cur ^ 1][r] = acc;   // rows past m stay zero
    __syncthreads();
    cur ^= 1;
  }
  const double hnext = H[m + (int64_t)(m - 1) * ldh];
  // value at (i + x_j) delta is E^i z
  for (int i = 0; i < nsub; ++i) {
    if (!end) {
      const double* u = z[cur];
      if (which == 0) {
        // alpha = scale .* (Hbar u), Hbar the (m+1) x m Hessenberg matrix
        double* al = alpha + (size_t)(i * GAUSS_P + j) * ADJ_A;
        const double v = adj_row(Hr, u, part);
        if (part == 0) al[r] = r < m ? scl[r] * v : (r == m ? scl[m] * hnext * u[m - 1] : 0.0);
        if (tid == 0) al[MMAX] = m == MMAX ? scl[m] * hnext * u[m - 1] : 0.0;
      } else if (tid < MMAX) {
        // lambda at t_k + s_q needs w(tau - s_q): tau - s_q = (nsub-1-i + x_{P-1-j}) delta
        omg[(size_t)((nsub - 1 - i) * GAUSS_P + (GAUSS_P - 1 - j)) * MMAX + tid] = tid < m ? scl[tid] * u[tid] : 0.0;
      }
      if (i == nsub - 1) break;
    }
    const double v = adj_row(Er, z[cur], part);
    if (part == 0) z[cur ^ 1][r] = v;
    __syncthreads();
    cur ^= 1;
  }
  // w(tau) = E^nsub beta e_1 for the update lambda(t_k) = W w(tau)
  if (end && tid < m) sl.u[tid] = z[cur][tid];
}

// The quadrature over the sub-step's nodes, done once on the coefficients:
//   M_{i,k} = sum_q cw_q alpha_{q,i} omg_{q,k}
// (row MMAX + 1: the source's factor), as float pairs hi + lo.  One block a row.
__global__ void __launch_bounds__(256) k_adj_moments(const double* __restrict__ alpha, const double* __restrict__ omg,
                                                     const double* __restrict__ cw, int nq, float* __restrict__ M) {
  extern __shared__ __align__(16) double wq[];   // nq
  __shared__ double part[4][MMAX];
  const int i = blockIdx.x, tid = threadIdx.x, k = tid & (MMAX - 1), g = tid / MMAX;
  for (int q = tid; q < nq; q += blockDim.x) wq[q] = cw[q] * alpha[(size_t)q * ADJ_A + i];
  __syncthreads();
  double a = 0.0;
  for (int q = g; q < nq; q += 4) a = fma(wq[q], omg[(size_t)q * MMAX + k], a);
  part[g][k] = a;
  __syncthreads();
  if (g == 0) {
    a = (part[0][k] + part[1][k]) + (part[2][k] + part[3][k]);
    const float hi = (float)a;
    M[i * MMAX + k] = hi;
    M[(ADJ_A + i) * MMAX + k] = (float)(a - (double)hi);
  }
}

// Q_e += (sum_{i,k} V_{i,e} M_{i,k} W_{k,e} + g_e sum_k M_{MMAX+1,k} W_{k,e}) / eps_e
// over the E nodes e: the quadrature of (A y)_e lambda_e on the sub-step.  One
// thread a node, W's column of the node in registers, M in shared memory.
// With M formed first a node costs 66 x 64 products whatever the number of
// quadrature nodes; evaluating both factors at every node took 129 FMAs a
// node and quadrature point (240 of them at tau = 12: 667 us at 48^3).
// In double-precision contexts the sums carry their rounding errors (hi + lo,
// kx_eft.cuh) and M is a float pair, five packed operations for two products:
// the entries of M cancel where the factors at a node did not, and plain sums
// missed that path's accuracy (1.07e-7 on a gradient held to 1e-7).  In
// single-precision contexts, whose bases are off by as much, plain packed sums
// do (48^3: 320 -> 115 us).
template <typename T>
__global__ void __launch_bounds__(128) k_adj_accum(Geo g, const T* __restrict__ V, const T* __restrict__ W,
                                                  int64_t ld, int mV, int mW, const T* __restrict__ gsrc,
                                                  const T* __restrict__ ie, const float* __restrict__ M,
                                                  double* __restrict__ Q) {
  constexpr bool COMP = sizeof(T) == 8;
  __shared__ __align__(16) float sM[(COMP ? 2 : 1) * ADJ_A * MMAX];
  for (int o = threadIdx.x; o < (COMP ? 2 : 1) * ADJ_A * MMAX; o += blockDim.x) sM[o] = M[o];
  __syncthreads();
  const int64_t nE = (int64_t)g.ne * g.ncell;
  const int64_t off = (int64_t)g.nh * g.ncell;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nE; e += (int64_t)gridDim.x * blockDim.x) {
    float2 w[MMAX / 2];
#pragma unroll
    for (int k = 0; k < MMAX / 2; ++k) {
      w[k].x = 2 * k < mW ? (float)W[(int64_t)(2 * k) * ld + off + e] : 0.f;
      w[k].y = 2 * k + 1 < mW ? (float)W[(int64_t)(2 * k + 1) * ld + off + e] : 0.f;
    }
    float qh = 0.f, ql = 0.f;
#pragma unroll(COMP ? 1 : 2)
    for (int i = 0; i <= mV + 1; ++i) {
      const int row = i <= mV ? i : MMAX + 1;
      const float v = i <= mV ? (float)V[(int64_t)i * ld + off + e] : (float)gsrc[off + e];
      const float4* mh = reinterpret_cast<const float4*>(sM + row * MMAX);
      float2 h0 = make_float2(0.f, 0.f), h1 = h0, l0 = h0, l1 = h0;
      if constexpr (COMP) {
        const float4* ml = reinterpret_cast<const float4*>(sM + (ADJ_A + row) * MMAX);
#pragma unroll
        for (int k = 0; k < MMAX / 4; ++k) {
          const float4 x = mh[k], y = ml[k];
          l0 = __ffma2_rn(make_float2(y.x, y.y), w[2 * k], l0);
          l1 = __ffma2_rn(make_float2(y.z, y.w), w[2 * k + 1], l1);
          sub_fma2(h0, l0, make_float2(x.x, x.y), w[2 * k]);
          sub_fma2(h1, l1, make_float2(x.z, x.w), w[2 * k + 1]);
        }
        // t = h + l: the four partial sums added with their errors
        float th = 0.f, tl = (l0.x + l0.y) + (l1.x + l1.y);
        sub_fma(th, tl, 1.f, h0.x);
        add_two(th, tl, h0.y);
        add_two(th, tl, h1.x);
        add_two(th, tl, h1.y);
        ql = fmaf(v, tl, ql);
        sub_fma(qh, ql, v, th);
      } else {
#pragma unroll
        for (int k = 0; k < MMAX / 4; k += 2) {
          const float4 x = mh[k], y = mh[k + 1];
          h0 = __ffma2_rn(make_float2(x.x, x.y), w[2 * k], h0);
          h1 = __ffma2_rn(make_float2(x.z, x.w), w[2 * k + 1], h1);
          l0 = __ffma2_rn(make_float2(y.x, y.y), w[2 * k + 2], l0);
          l1 = __ffma2_rn(make_float2(y.z, y.w), w[2 * k + 3], l1);
        }
        h0 = __fadd2_rn(__fadd2_rn(h0, h1), __fadd2_rn(l0, l1));
        sub_fma(qh, ql, v, h0.x + h0.y);
      }
    }
    Q[e] += ((double)qh + (double)ql) * (double)ie[e];
  }
}

// grad_c = (1/4) sum of Q over the E nodes whose closure holds cell c.
__global__ void k_adj_cells(Geo g, const double* __restrict__ Q, double* __restrict__ grad) {
  for (int64_t cell = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; cell < g.ncell;
       cell += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(cell % g.nx);
    const int64_t r = cell / g.nx;
    const int j = (int)(r % g.ny), k = (int)(r / g.ny);
    const int ip = i + 1 == g.nx ? 0 : i + 1, jp = j + 1 == g.ny ? 0 : j + 1;
    const int kp = (g.dim == 3 && k + 1 == g.nz) ? 0 : k + 1;
    const int64_t nx = g.nx, nxy = (int64_t)g.nx * g.ny, nc = g.ncell;
    double s = 0.0;
    if (g.dim == 2) {
      s = Q[j * nx + i] + Q[j * nx + ip] + Q[jp * nx + i] + Q[jp * nx + ip];
    } else {
      // Ex nodes (i, j or j+1, k or k+1); Ey (i or i+1, j, k or k+1); Ez (i or i+1, j or j+1, k)
      s += Q[k * nxy + j * nx + i] + Q[k * nxy + jp * nx + i] + Q[kp * nxy + j * nx + i] +
           Q[kp * nxy + jp * nx + i];
      s += Q[nc + k * nxy + j * nx + i] + Q[nc + k * nxy + j * nx + ip] + Q[nc + kp * nxy + j * nx + i] +
           Q[nc + kp * nxy + j * nx + ip];
      s += Q[2 * nc + k * nxy + j * nx + i] + Q[2 * nc + k * nxy + j * nx + ip] +
           Q[2 * nc + k * nxy + jp * nx + i] + Q[2 * nc + k * nxy + jp * nx + ip];
    }
    grad[cell] = 0.25 * s;
  }
}

// ---------------------------------------------------------------------------
kx_status launch_adj_seed(kx_ctx* c, const void* y, void* lam, int axis, int idx) {
  if (c->d.precision == KX_FP64)
    k_adj_seed<double><<<c->nblk, NTHREADS, 0, c->stream>>>(c->geo, axis, idx, (const double*)y, (double*)lam);
  else
    k_adj_seed<float><<<c->nblk, NTHREADS, 0, c->stream>>>(c->geo, axis, idx, (const float*)y, (float*)lam);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

kx_status launch_adj_substep(kx_ctx* c, double tau, double omega, double tk, const void* g) {
  const int nsub = std::max(1, (int)std::ceil(tau / QUAD_DELTA));
  if (nsub * GAUSS_P > c->adj_nq_max) {
    snprintf(c->err, sizeof(c->err), "adjoint: sub-step %.3g needs more than %d quadrature nodes", tau,
             c->adj_nq_max);
    return KX_EINVAL;
  }
  const int m = c->m;
  static ClusterOptIn attr{};
  int cl = 0;
  const kx_status so = cluster_opt_in(c, attr, (const void*)k_adj_expm, CD_SMEM, &cl);
  if (so != KX_OK) return so;
  int* status = reinterpret_cast<int*>(c->d_small + 64);
  const SlotSet<float> ss = make_slotset<float>(c, 0);
  const int nq = nsub * GAUSS_P;
  time_begin(c);
  launch_cluster(k_adj_expm, cl, 2, CD_SMEM, c->stream, ss, m + 1, tau / nsub, c->d_cd_ws, status);
  KX_CHECK_LAUNCH(c);
  k_adj_march<<<dim3(GAUSS_P + 1, 2), 256, 0, c->stream>>>(ss, m + 1, tau, nsub, c->d_gauss, c->d_gauss + GAUSS_P,
                                                           omega, tk, c->d_cd_ws, c->d_adj_alpha, c->d_adj_omg,
                                                           c->d_adj_cw);
  KX_CHECK_LAUNCH(c);
  k_adj_moments<<<ADJ_A, 256, nq * sizeof(double), c->stream>>>(c->d_adj_alpha, c->d_adj_omg, c->d_adj_cw, nq,
                                                               c->d_adj_M);
  time_end(c, KX_K_PROJ, 0.0);
  KX_CHECK_LAUNCH(c);
  const int64_t nE = (int64_t)c->geo.ne * c->geo.ncell;
  const int blocks = (int)std::min<int64_t>((nE + 127) / 128, (int64_t)c->nsm * 8);
  const int64_t sV = (int64_t)(m + 1) * c->ld;
  // the basis sizes are read back by the host after each Arnoldi run
  const int mV = c->h_state[0].m_done, mW = c->h_state[1].m_done;
  time_begin(c);
  if (c->d.precision == KX_FP64) {
    k_adj_accum<double><<<blocks, 128, 0, c->stream>>>(
        c->geo, (const double*)c->d_V, (const double*)c->d_V + sV, c->ld, mV, mW, (const double*)g,
        (const double*)c->d_inv_eps, c->d_adj_M, c->d_adj_Q);
  } else {
    k_adj_accum<float><<<blocks, 128, 0, c->stream>>>(
        c->geo, (const float*)c->d_V, (const float*)c->d_V + sV, c->ld, mV, mW, (const float*)g,
        (const float*)c->d_inv_eps, c->d_adj_M, c->d_adj_Q);
  }
  time_end(c, KX_K_ZUPDATE, (double)(mV + 1 + mW) * nE * c->esize);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

kx_status launch_adj_cells(kx_ctx* c, double* grad) {
  k_adj_cells<<<c->nblk, NTHREADS, 0, c->stream>>>(c->geo, c->d_adj_Q, grad);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

// Gauss-Legendre nodes and weights on [0, 1] by Newton's method on P_n.
void gauss_legendre01(int n, double* x, double* w) {
  for (int i = 0; i < n; ++i) {
    double t = std::cos(M_PI * (i + 0.75) / (n + 0.5));
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = t;
      for (int k = 2; k <= n; ++k) {
        const double p2 = ((2 * k - 1) * t * p1 - (k - 1) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      const double dp = n * (t * p1 - p0) / (t * t - 1.0);
      const double dt = p1 / dp;
      t -= dt;
      if (std::fabs(dt) < 1e-16) break;
    }
    double p0 = 1.0, p1 = t;
    for (int k = 2; k <= n; ++k) {
      const double p2 = ((2 * k - 1) * t * p1 - (k - 1) * p0) / k;
      p0 = p1;
      p1 = p2;
    }
    const double dp = n * (t * p1 - p0) / (t * t - 1.0);
    // node on [-1, 1] -> [0, 1], ascending
    x[n - 1 - i] = 0.5 * (t + 1.0);
    w[n - 1 - i] = 1.0 / ((1.0 - t * t) * dp * dp);
  }
}

int gauss_points() { return GAUSS_P; }

}  // namespace kx
