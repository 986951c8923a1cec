// Residual-based restarting in Krylov dimension for many frequencies at
// once (Sect. 3.4, eq. (rst), Corollary 2, Fig. alg:rst; regular Krylov
// variant).  The Krylov basis of every restart comes from the Arnoldi
// passes (stencil.cu, linalg.cu) and serves all frequencies; this file holds
// the per-frequency projected work and the accumulation of the responses.
//
// Restart k, basis V_m, Hessenberg H_m, h = h_{m+1,m}:
//   u_j' = -H_m u_j + alpha_j(t) e_1,  u_j(0) = 0       (eq. (corr2))
//   y_j(T) += V_m u_j(T)                                (eq. (upd1))
//   alpha_j <- alphahat_j = -h e_m^T u_j(t)              (eqs. (resid), (rst))
// alpha_j is held on a uniform grid t_i = i d (i = 0..Nt, d = T / Nt) as
// the quintic Hermite interpolant of its value and first two derivatives
// at the grid points (Fig. alg:rst step 2(b) stores the samples), i.e. as
// six coefficients b_0..b_5 per interval, p(theta) = sum_j b_j theta^j,
// theta = (t - t_i) / d.  For that source the projected problem has the
// exact interval map
//   u(t_{i+1}) = E u(t_i) + sum_j b_j W_j,
//   E = exp(-d H_m),  W_j = d j! phi_{j+1}(-d H_m) e_1,
// and the derivatives of alphahat follow from the projected equation:
//   alphahat'  = -h e_m^T (-H_m u + alpha e_1),
//   alphahat'' = -h e_m^T (H_m^2 u - alpha H_m e_1 + alpha' e_1).
//
//   k_rst_source   restart 1's source ||g|| sin(W t) as interval coefficients.
//   k_rst_setup    one cluster: E and the W_j from one exponential of the
//                  (m+6)-square matrix [[-d H_m, e_1 e_1^T], [0, J]] (J the
//                  6x6 shift; its top right block holds phi_1..phi_6 (-d H_m) e_1),
//                  and the tables that advance a chunk of 16 intervals at once.
//   k_rst_drive, k_rst_march, k_rst_sample
//                  the Nt interval maps in chunks; alphahat and its first two
//                  derivatives at every grid point.
//   k_rst_coef     the next restart's interval coefficients from those
//                  samples (all intervals in parallel).
//   k_rst_plane    y_j += V_m u_j(T) on the output plane, FP64 accumulators.
//   k_rst_full     the same on the full field (optional).
#include <atomic>
#include <cmath>

#include "kx_cdense.cuh"
#include "kx_internal.cuh"
#include "kx_reduce.cuh"

namespace kx {

// Coefficients of p(theta) = sum_j b_j theta^j on an interval of length d
// with p, dp/dt, d2p/dt2 given at both ends (quintic Hermite interpolation).
__device__ __forceinline__ void hermite5(double a0, double da0, double dda0, double a1, double da1,
                                         double dda1, double d, double* b) {
  b[0] = a0;
  b[1] = d * da0;
  b[2] = 0.5 * d * d * dda0;
  const double R0 = a1 - (b[0] + b[1] + b[2]);
  const double R1 = d * da1 - (b[1] + 2.0 * b[2]);
  const double R2 = d * d * dda1 - 2.0 * b[2];
  b[3] = 10.0 * R0 - 4.0 * R1 + 0.5 * R2;
  b[4] = -15.0 * R0 + 7.0 * R1 - R2;
  b[5] = 6.0 * R0 - 3.0 * R1 + 0.5 * R2;
}

// ---------------------------------------------------------------------------
__global__ void k_rst_source(const double* __restrict__ om, double beta, int Nt, double d,
                             double* __restrict__ b) {
  const int f = blockIdx.y;
  const double W = om[f];
  double* bf = b + (int64_t)f * Nt * RST_P;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Nt; i += gridDim.x * blockDim.x) {
    double s0, c0, s1, c1;
    sincos(W * (i * d), &s0, &c0);
    sincos(W * ((i + 1) * d), &s1, &c1);
    double bb[RST_P];
    hermite5(beta * s0, beta * W * c0, -beta * W * W * s0, beta * s1, beta * W * c1, -beta * W * W * s1, d, bb);
#pragma unroll
    for (int j = 0; j < RST_P; ++j) bf[(int64_t)i * RST_P + j] = bb[j];
  }
}

kx_status launch_rst_source(kx_ctx* c, cudaStream_t st, int nfreq, double beta, int Nt, double d, double* b) {
  const int gx = std::min((Nt + 255) / 256, 64);
  k_rst_source<<<dim3(gx, nfreq), 256, 0, st>>>(c->d_omegas, beta, Nt, d, b);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

// ---------------------------------------------------------------------------
// Set-up of one restart, one cluster (kx_cdense.cuh): E and the W_j from one
// exponential of order m + 6, then the chunk tables by doubling.  With G =
// E^P known (P = 1, 2, 4, 8), the blocks hold their rows of G and stage all of
// it:  E^2P = G G,  Z_{P+l} = G Z_l (Z_l = E^l W, l < P),  R_{P+l} = R_l G
// (R_l = C E^l, C the three sampling rows); one cluster barrier a doubling.
// On one block (the exponential alone, 64 dependent pivots of its solve) the
// set-up took 1060 us at m = 64.
constexpr int RST_ZC = RST_L * RST_P;                   // columns of [Z_0 .. Z_{L-1}]
constexpr int RST_O = 3 * RST_L;                        // sampled values of a chunk
constexpr int RST_SMEM = CD_SMEM + MMAX * CD_LD * (int)sizeof(double);
static_assert(RST_L == 16, "four doublings");
static_assert(RST_ZC / 2 <= CD_LD && RST_O <= MMAX && RST_O / 2 <= CD_RMAX * CD_PORTABLE, "the half-filled tables fit the shared operands");

__global__ void __launch_bounds__(CD_THREADS) k_rst_setup(const double* __restrict__ H, int ldh, const SlotState* st,
                                                          double d, double* mats, double* ws, int* status) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double red[32];
  const int C = cl_size(), rank = cl_rank(), tid = threadIdx.x;
  const int md = st->m_done;
  const int n = md + RST_P;
  // (m+6)-square [[-d H_m, e_1 e_1^T], [0, J]], J the shift
  auto entry = [&](int r, int c) {
    if (r < md && c < md) return r <= c + 1 ? -d * H[r + (int64_t)c * ldh] : 0.0;
    return (r == 0 && c == md) || (r >= md && c == r + 1) ? 1.0 : 0.0;
  };
  int q = 0, s = 0;
  const bool ok = md >= 1 && !st->status;
  if (!ok || !cd_plan(cd_norm1(n, red, entry), 1, &q, &s)) {
    // the Arnoldi process's own status (a non-finite value, a bounded wait
    // that ran out), else no step completed or a non-finite matrix
    if (rank == 0 && tid == 0) *status = st->status ? st->status : KX_ENONFINITE;
    return;
  }
  const CdShared sh = cd_shared(sm);
  double* Zs = sm + CD_SMEM / sizeof(double);
  const CdRows w = cd_rows(n, rank);
  const int R = max(0, min(w.R, md - w.r0));   // own rows among the first md
  const double sc = ldexp(1.0, -s);
  double* P = cd_expm(sh, ws, n, w, q, s, [&](int r, int c) { return sc * entry(r, c); });
  double* Q = P == sh.S[3] ? sh.S[4] : sh.S[3];
  double* gE = ws + 2 * CD_MAT;                // E^P, two in turn
  double* gZ = ws + 4 * CD_MAT;                // Z, row stride RST_ZC
  double* gR = gZ + MMAX * RST_ZC;             // R, row stride MMAX
  static_assert(4 * CD_MAT + MMAX * RST_ZC + RST_O * MMAX <= CD_WS, "the workspace holds the tables");
  // C: last rows of -h I, h H_m and -h H_m^2 (nonzero in the last three columns)
  const double h = st->done ? 0.0 : H[md + (int64_t)(md - 1) * ldh];
  const int lr = md - 1;
  auto crow = [&](int comp, int c) {
    if (c < lr - 2) return 0.0;
    if (comp == 0) return c == lr ? -h : 0.0;
    if (comp == 1) return c >= lr - 1 ? h * H[lr + (int64_t)c * ldh] : 0.0;
    double v = 0.0;
    for (int k = max(0, lr - 1); k < md; ++k)
      if (k <= c + 1) v += H[lr + (int64_t)k * ldh] * H[k + (int64_t)c * ldh];
    return -h * v;
  };
  for (int o = tid; o < R * md; o += CD_THREADS) {
    const int r = o / md, c = o - r * md;
    gE[(w.r0 + r) * CD_LD + c] = P[r * CD_LD + c];
  }
  for (int o = tid; o < R * RST_P; o += CD_THREADS) {
    const int r = o / RST_P, j = o - r * RST_P;
    double f = d;
    for (int k = 2; k <= j; ++k) f *= k;
    gZ[(w.r0 + r) * RST_ZC + j] = f * P[r * CD_LD + md + j];
  }
  if (rank == 0)
    for (int o = tid; o < 3 * md; o += CD_THREADS) {
      const int comp = o / md, c = o - comp * md;
      gR[comp * MMAX + c] = crow(comp, c);
    }
  cl_sync();
  for (int k = 0; (1 << k) < RST_L; ++k) {
    const int half = 1 << k;
    const double* cur = gE + (k & 1) * CD_MAT;
    double* nxt = gE + ((k & 1) ^ 1) * CD_MAT;
    cd_load(sh.B, cur, md, md);
    for (int o = tid; o < md * half * (RST_P / 2); o += CD_THREADS) {
      const int r = o / (half * (RST_P / 2)), c = 2 * (o - r * (half * (RST_P / 2)));
      *reinterpret_cast<double2*>(Zs + r * CD_LD + c) = __ldcg(reinterpret_cast<const double2*>(gZ + r * RST_ZC + c));
    }
    // this block's share of the sampling rows
    const int per = (3 * half + C - 1) / C;
    const int s0 = min(3 * half, rank * per), ns = min(3 * half, s0 + per) - s0;
    for (int o = tid; o < ns * md; o += CD_THREADS) {
      const int r = o / md, c = o - r * md;
      sh.S[0][r * CD_LD + c] = __ldcg(gR + (s0 + r) * MMAX + c);
    }
    __syncthreads();
    cd_mm(P, sh.B, R, md, md, [&](int r, int c, double v) {
      Q[r * CD_LD + c] = v;
      nxt[(w.r0 + r) * CD_LD + c] = v;
    });
    cd_mm(P, Zs, R, md, half * RST_P,
          [&](int r, int c, double v) { gZ[(w.r0 + r) * RST_ZC + half * RST_P + c] = v; });
    cd_mm(sh.S[0], sh.B, ns, md, md, [&](int r, int c, double v) { gR[(3 * half + s0 + r) * MMAX + c] = v; });
    cl_sync();
    double* t = P;
    P = Q;
    Q = t;
  }
  // the tables of the marching kernels, zero past the basis' size
  const double* EL = gE;                       // E^16 after four doublings
  const int t0 = rank * CD_THREADS + tid, nt = C * CD_THREADS;
  for (int o = t0; o < MMAX * MMAX; o += nt) {
    const int r = o / MMAX, c = o % MMAX;
    mats[o] = r < md && c < md ? __ldcg(EL + r * CD_LD + c) : 0.0;
  }
  for (int o = t0; o < RST_ZC * MMAX; o += nt) {
    const int k = o / MMAX, r = o % MMAX, qq = k / RST_P, j = k % RST_P;
    mats[RST_OFF_Z + o] = r < md ? __ldcg(gZ + r * RST_ZC + (RST_L - 1 - qq) * RST_P + j) : 0.0;
  }
  const double hm0 = lr <= 1 ? H[lr] : 0.0, del = md == 1 ? 1.0 : 0.0;
  for (int o = t0; o < (MMAX + RST_ZC) * RST_O; o += nt) {
    const int k = o / RST_O, c = o % RST_O, r = c / 3, comp = c % 3;
    double v = 0.0;
    if (k < MMAX) {
      if (k < md) v = __ldcg(gR + c * MMAX + k);
    } else {
      const int qq = (k - MMAX) / RST_P, j = (k - MMAX) % RST_P;
      if (qq < r) {
        for (int i = max(0, lr - 2); i <= lr; ++i)
          v = fma(crow(comp, i), __ldcg(gZ + i * RST_ZC + (r - 1 - qq) * RST_P + j), v);
      } else if (qq == r) {
        // alphahat' and alphahat'' carry the source and its slope (b_1 = d alpha')
        if (j == 0) v = comp == 1 ? -h * del : (comp == 2 ? h * hm0 : 0.0);
        if (j == 1 && comp == 2) v = -h * del / d;
      }
    }
    mats[RST_OFF_R + o] = v;
  }
}

kx_status launch_rst_setup(kx_ctx* c, cudaStream_t st, int slot, double d) {
  Slot<float> s = make_slot<float>(c, slot);
  int* status = reinterpret_cast<int*>(c->d_small + 64);
  static ClusterOptIn attr{};
  int blocks = 0;
  const kx_status so = cluster_opt_in(c, attr, (const void*)k_rst_setup, RST_SMEM, &blocks);
  if (so != KX_OK) return so;
  time_begin(c);
  launch_cluster(k_rst_setup, blocks, 1, RST_SMEM, st, (const double*)s.H, c->m + 1, (const SlotState*)s.st, d, c->d_rst_mats,
                 c->d_cd_ws, status);
  time_end(c, KX_K_PROJ, 0.0);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

// ---------------------------------------------------------------------------
// The march over the Nt intervals, in chunks of L = RST_L.  Done interval by
// interval it is Nt dependent products with E, one block a frequency: 4.5k
// double-precision FMAs an interval on one SM's slow pipe, 3.2 ms for Nt =
// 2160.  Over a chunk starting at u_c,
//   u_{c+1}        = E^L u_c + F_c,   F_c = sum_q Z_{L-1-q} b_q,
//   s_r (r < L)    = R_r u_c + sum_{q<r} C Z_{r-1-q} b_q + D b_r
// (s the samples alphahat, alphahat', alphahat''; D the source's own share),
// so only the short recursion over chunks is serial:
//   k_rst_drive    F_c of every chunk and frequency (a 64 x 6L product)
//   k_rst_march    u_{c+1} = E^L u_c + F_c, one block a frequency
//   k_rst_sample   the samples of every chunk (a 3L x (64 + 6L) product)
// about 860 FMAs an interval, all but 256 of them spread over the GPU.  L = 16
// balances the serial part (64^2 / L an interval) against the samples' share
// (grows with L) and the tables' set-up (log L products).
// The first chunk may be short: it starts pad = Nt_chunks L - Nt intervals
// early with u = 0 and no source, so every chunk is treated alike.
constexpr int RST_CB = 4;   // chunks a block of the parallel kernels

__device__ __forceinline__ int rst_chunks(int Nt) { return (Nt + RST_L - 1) / RST_L; }

// The source coefficients of chunks c0 .. c0 + RST_CB - 1 to shared memory.
__device__ __forceinline__ void rst_load_b(double* sb, const double* __restrict__ bf, int c0, int nch, int pad) {
  for (int o = threadIdx.x; o < RST_CB * RST_ZC; o += blockDim.x) {
    const int64_t k = (int64_t)c0 * RST_ZC + o - (int64_t)pad * RST_P;
    sb[o] = (c0 + o / RST_ZC < nch && k >= 0) ? bf[k] : 0.0;
  }
}

__global__ void __launch_bounds__(RST_CB * MMAX) k_rst_drive(const double* __restrict__ mats,
                                                            const double* __restrict__ b, double* __restrict__ fu,
                                                            int Nt, const int* __restrict__ fstate) {
  const int f = blockIdx.y;
  if (fstate[f] != 0) return;
  __shared__ double sb[RST_CB * RST_ZC];
  const int nch = rst_chunks(Nt), c0 = blockIdx.x * RST_CB;
  rst_load_b(sb, b + (int64_t)f * Nt * RST_P, c0, nch, nch * RST_L - Nt);
  __syncthreads();
  const int r = threadIdx.x % MMAX, ci = threadIdx.x / MMAX;
  const double* z = mats + RST_OFF_Z + r;
  const double* x = sb + ci * RST_ZC;
  double a0 = 0.0, a1 = 0.0;
#pragma unroll 8
  for (int k = 0; k < RST_ZC; k += 2) {
    a0 = fma(z[k * MMAX], x[k], a0);
    a1 = fma(z[(k + 1) * MMAX], x[k + 1], a1);
  }
  if (c0 + ci < nch) fu[((int64_t)f * nch + c0 + ci) * MMAX + r] = a0 + a1;
}

// Two threads a row, E^L's entries in registers (2048 issue clocks of the
// double-precision pipe a chunk, which is what bounds it); the next F's are
// loaded RST_AHEAD chunks before their use.  F_c is replaced by u_c.
constexpr int RST_MV = 2 * MMAX;
constexpr int RST_AHEAD = 4;

__global__ void __launch_bounds__(RST_MV) k_rst_march(const double* __restrict__ mats, double* __restrict__ fu, int Nt,
                                                     int* fstate, double* resid, unsigned* cnt, double* u_out) {
  const int f = blockIdx.x;
  const int tid = threadIdx.x;
  __shared__ int s_state;
  __shared__ double u[2][MMAX];
  if (tid == 0) s_state = fstate[f];
  if (tid < MMAX) u[0][tid] = 0.0;
  __syncthreads();
  if (s_state != 0) {
    if (tid == 0 && s_state == 1) fstate[f] = 2;
    return;
  }
  if (tid == 0) {
    resid[f] = 0.0;
    cnt[f] = 0u;
  }
  const int nch = rst_chunks(Nt);
  const int r = tid >> 1, q = tid & 1;
  double* ff = fu + (int64_t)f * nch * MMAX + r;
  double Er[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) Er[k] = mats[r * MMAX + q + 2 * k];
  double fn[RST_AHEAD];
#pragma unroll
  for (int t = 0; t < RST_AHEAD; ++t) fn[t] = (q == 0 && t < nch) ? ff[t * MMAX] : 0.0;
  double mine = 0.0;
  for (int c0 = 0; c0 < nch; c0 += RST_AHEAD) {
#pragma unroll
    for (int t = 0; t < RST_AHEAD; ++t) {
      const int c = c0 + t;
      if (c < nch) {
        const double* uc = u[t & 1];
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int k = 0; k < 32; k += 2) {
          s0 = fma(Er[k], uc[q + 2 * k], s0);
          s1 = fma(Er[k + 1], uc[q + 2 * k + 2], s1);
        }
        double sum = s0 + s1;
        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        if (q == 0) {
          sum += fn[t];
          ff[(int64_t)c * MMAX] = mine;
          if (c + RST_AHEAD < nch) fn[t] = ff[(int64_t)(c + RST_AHEAD) * MMAX];
          u[(t & 1) ^ 1][r] = sum;
          mine = sum;
        }
        __syncthreads();
      }
    }
  }
  static_assert(RST_AHEAD % 2 == 0, "the buffer of u alternates with t");
  if (q == 0) u_out[(int64_t)f * MMAX + r] = mine;
}

// One thread a sampled value of a chunk; the warp stops at its latest
// sample's sources.  The last block of a frequency to finish takes the
// stopping test from the maximum (of non-negative doubles, whose bits order
// as integers: the same whatever the blocks' order).
__global__ void __launch_bounds__(RST_CB * RST_O) k_rst_sample(const double* __restrict__ mats,
                                                              const double* __restrict__ b,
                                                              const double* __restrict__ fu, double* __restrict__ smp,
                                                              int Nt, double tol_abs, int* fstate, double* resid,
                                                              unsigned* cnt, const double* __restrict__ u_end) {
  const int f = blockIdx.y;
  if (fstate[f] != 0) return;
  __shared__ double sb[RST_CB * RST_ZC], su[RST_CB * MMAX];
  __shared__ double red[RST_CB * RST_O / 32];
  const int tid = threadIdx.x;
  const int nch = rst_chunks(Nt), c0 = blockIdx.x * RST_CB, pad = nch * RST_L - Nt;
  const double* bf = b + (int64_t)f * Nt * RST_P;
  double* sf = smp + (int64_t)f * (Nt + 1) * 3;
  rst_load_b(sb, bf, c0, nch, pad);
  for (int o = tid; o < RST_CB * MMAX; o += blockDim.x)
    su[o] = c0 + o / MMAX < nch ? fu[((int64_t)f * nch + c0) * MMAX + o] : 0.0;
  __syncthreads();
  const int o = tid % RST_O, ci = tid / RST_O, r = o / 3, comp = o % 3;
  const double* t = mats + RST_OFF_R + o;
  const double* x = su + ci * MMAX;
  double a0 = 0.0, a1 = 0.0;
#pragma unroll 8
  for (int k = 0; k < MMAX; k += 2) {
    a0 = fma(t[k * RST_O], x[k], a0);
    a1 = fma(t[(k + 1) * RST_O], x[k + 1], a1);
  }
  t += MMAX * RST_O;
  x = sb + ci * RST_ZC;
  const int lim = (__reduce_max_sync(0xffffffffu, r) + 1) * RST_P;
#pragma unroll 6
  for (int k = 0; k < lim; k += 2) {
    a0 = fma(t[k * RST_O], x[k], a0);
    a1 = fma(t[(k + 1) * RST_O], x[k + 1], a1);
  }
  const int i = (c0 + ci) * RST_L - pad + r;
  double mx = 0.0;
  if (c0 + ci < nch && i >= 0) {
    const double v = a0 + a1;
    sf[(int64_t)i * 3 + comp] = v;
    if (comp == 0) mx = fabs(v);
  }
  if (blockIdx.x == gridDim.x - 1 && tid < 3) {
    // t = T: source value and d-scaled slope from the last interval's
    // polynomial at theta = 1 (the rows of r = 0 give C and D)
    const double* last = bf + (int64_t)(Nt - 1) * RST_P;
    double al = 0.0, dal = 0.0;
    for (int j = 0; j < RST_P; ++j) {
      al += last[j];
      dal += j * last[j];
    }
    const double* tc = mats + RST_OFF_R + tid;
    double v = 0.0;
    for (int k = 0; k < MMAX; ++k) v = fma(tc[k * RST_O], u_end[(int64_t)f * MMAX + k], v);
    v = fma(tc[MMAX * RST_O], al, v);
    v = fma(tc[(MMAX + 1) * RST_O], dal, v);
    sf[(int64_t)Nt * 3 + tid] = v;
    if (tid == 0) mx = fabs(v) > mx || !(v == v) ? fabs(v) : mx;
  }
  // the largest bits (a NaN's order above every number's)
  unsigned long long m = (unsigned long long)__double_as_longlong(mx);
  for (int s = 16; s > 0; s >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, m, s);
    m = y > m ? y : m;
  }
  if ((tid & 31) == 0) red[tid >> 5] = __longlong_as_double((long long)m);
  __syncthreads();
  if (tid != 0) return;
  for (int wq = 0; wq < RST_CB * RST_O / 32; ++wq) {
    const unsigned long long y = (unsigned long long)__double_as_longlong(red[wq]);
    m = y > m ? y : m;
  }
  unsigned long long* rb = reinterpret_cast<unsigned long long*>(resid) + f;
  atomicMax(rb, m);
  __threadfence();
  if (atomicAdd(cnt + f, 1u) != gridDim.x - 1) return;
  __threadfence();
  const double all = __longlong_as_double((long long)atomicMax(rb, 0ull));
  if (!isfinite(all)) fstate[f] = 3;            // reported by the host
  else if (all <= tol_abs) fstate[f] = 1;       // stops after this restart's combination
}

kx_status launch_rst_cascade(kx_ctx* c, cudaStream_t st, int nfreq, const double* b, int Nt, double d,
                             double tol_abs) {
  (void)d;
  const int nch = (Nt + RST_L - 1) / RST_L;
  const dim3 grid((nch + RST_CB - 1) / RST_CB, nfreq);
  time_begin(c);
  k_rst_drive<<<grid, RST_CB * MMAX, 0, st>>>(c->d_rst_mats, b, c->d_rst_fu, Nt, c->d_rst_state);
  KX_CHECK_LAUNCH(c);
  k_rst_march<<<nfreq, RST_MV, 0, st>>>(c->d_rst_mats, c->d_rst_fu, Nt, c->d_rst_state, c->d_rst_res, c->d_rst_cnt,
                                       c->d_rst_u);
  KX_CHECK_LAUNCH(c);
  k_rst_sample<<<grid, RST_CB * RST_O, 0, st>>>(c->d_rst_mats, b, c->d_rst_fu, c->d_rst_smp, Nt, tol_abs,
                                               c->d_rst_state, c->d_rst_res, c->d_rst_cnt, c->d_rst_u);
  time_end(c, KX_K_CASCADE, 0.0);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

// The next restart's interval coefficients from the samples (frequencies
// still running only).
__global__ void k_rst_coef(const double* __restrict__ smp, double* __restrict__ b, int Nt, double d,
                           const int* __restrict__ fstate) {
  const int f = blockIdx.y;
  if (fstate[f] != 0) return;
  const double* sf = smp + (int64_t)f * (Nt + 1) * 3;
  double* bf = b + (int64_t)f * Nt * RST_P;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Nt; i += gridDim.x * blockDim.x) {
    double bb[RST_P];
    hermite5(sf[3 * i], sf[3 * i + 1], sf[3 * i + 2], sf[3 * i + 3], sf[3 * i + 4], sf[3 * i + 5], d, bb);
#pragma unroll
    for (int j = 0; j < RST_P; ++j) bf[(int64_t)i * RST_P + j] = bb[j];
  }
}

kx_status launch_rst_coef(kx_ctx* c, cudaStream_t st, int nfreq, double* b, int Nt, double d) {
  const int gx = std::min((Nt + 255) / 256, 64);
  k_rst_coef<<<dim3(gx, nfreq), 256, 0, st>>>(c->d_rst_smp, b, Nt, d, c->d_rst_state);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

// v_{m+1} of one basis slot (stored unnormalised in column m_done) becomes
// column 0 of another; m_done is read on the device.
template <typename T>
__global__ void k_rst_nextvec(Slot<T> from, Slot<T> to, int64_t n, int64_t ld) {
  const int md = from.st->m_done;
  const T* __restrict__ src = from.V + (int64_t)md * ld;
  T* __restrict__ dst = to.V;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    dst[e] = src[e];
}

kx_status launch_rst_nextvec(kx_ctx* c, cudaStream_t st, int from, int to) {
  if (c->d.precision == KX_FP64)
    k_rst_nextvec<double><<<c->nblk, NTHREADS, 0, st>>>(make_slot<double>(c, from), make_slot<double>(c, to), c->n,
                                                        c->ld);
  else
    k_rst_nextvec<float><<<c->nblk, NTHREADS, 0, st>>>(make_slot<float>(c, from), make_slot<float>(c, to), c->n,
                                                       c->ld);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

// ---------------------------------------------------------------------------
// y_j += V_m u_j(T) on the output plane (FP64), for frequencies not stopped
// before this restart.  Stored basis columns are unnormalised: v_i = scale_i V_i.
template <typename T>
__global__ void __launch_bounds__(NTHREADS) k_rst_plane(Slot<T> s, int64_t ld, Geo g, int axis, int idx,
                                                       int64_t P, const int* __restrict__ fstate,
                                                       const double* __restrict__ u, double* yp) {
  const int f = blockIdx.y;
  const int sf = fstate[f];
  if (sf == 2 || sf == 3) return;
  __shared__ double cf[MMAX];
  const int md = s.st->m_done;
  for (int q = threadIdx.x; q < md; q += blockDim.x) cf[q] = u[(int64_t)f * MMAX + q] * s.scale[q];
  __syncthreads();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < P; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = plane_node(g, axis, idx, t);
    double acc = 0.0;
    for (int j = 0; j < md; ++j) acc = fma(cf[j], (double)s.V[(int64_t)j * ld + e], acc);
    yp[(int64_t)f * P + t] += acc;
  }
}

kx_status launch_rst_plane(kx_ctx* c, cudaStream_t st, int slot, int nfreq, int axis, int idx, int64_t P) {
  const int gx = (int)std::max<int64_t>(1, std::min<int64_t>((P + NTHREADS - 1) / NTHREADS, 64));
  time_begin(c);
  if (c->d.precision == KX_FP64)
    k_rst_plane<double><<<dim3(gx, nfreq), NTHREADS, 0, st>>>(make_slot<double>(c, slot), c->ld, c->geo,
                                                                   axis, idx, P, c->d_rst_state, c->d_rst_u,
                                                                   c->d_rst_yp);
  else
    k_rst_plane<float><<<dim3(gx, nfreq), NTHREADS, 0, st>>>(make_slot<float>(c, slot), c->ld, c->geo,
                                                                  axis, idx, P, c->d_rst_state, c->d_rst_u,
                                                                  c->d_rst_yp);
  time_end(c, KX_K_RESTART, 0.0);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

// ---------------------------------------------------------------------------
// y_j += V_m u_j(T) on the full field.  FP64: plain accumulation into Y.
// FP32: every coefficient is split into a float pair hi + lo, the
// combination is summed error-free (two-product by FMA, Knuth's two-sum) and
// added to the float-pair accumulator (Y_j, lo_j) by a two-sum, so the
// accumulated response keeps about twice float precision over the restarts.
// One thread a field value, its basis row in registers; the coefficients'
// float pairs are formed once a block (formed at every use, in double
// precision on this GPU's slow pipe, they were most of this kernel's time:
// 36^3, 4 frequencies 855 us).  FP32 takes two values a thread: the packed
// operations serve both and each pair of coefficients is loaded once for them.
__device__ __forceinline__ void rst_acc2(float2& s, float2& c, float2 hi, float2 lo, float2 v) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const float2 p = __fmul2_rn(hi, v);
  const float2 np = __fmul2_rn(p, m1);
  const float2 e = __ffma2_rn(lo, v, __ffma2_rn(hi, v, np));
  const float2 t = __fadd2_rn(s, p);
  const float2 z = __ffma2_rn(s, m1, t);                       // t - s
  const float2 d = __ffma2_rn(z, m1, t);                       // t - z
  c = __fadd2_rn(c, __fadd2_rn(__fadd2_rn(__ffma2_rn(d, m1, s), __ffma2_rn(z, m1, p)), e));
  s = t;
}

__global__ void __launch_bounds__(128) k_rst_full32(Slot<float> s, int64_t ld, int64_t n, int nfreq,
                                                   const int* __restrict__ fstate, const double* __restrict__ u,
                                                   float* __restrict__ Y, float* __restrict__ lo_acc) {
  extern __shared__ __align__(16) float4 cf4[];   // per frequency and column: hi, hi, lo, lo
  __shared__ int act[MAXF];
  const int md = s.st->m_done;
  for (int q = threadIdx.x; q < nfreq * MMAX; q += blockDim.x) {
    const int j = q % MMAX;
    const double c = j < md ? u[q] * s.scale[j] : 0.0;
    const float hi = (float)c, lo = (float)(c - (double)hi);
    cf4[q] = make_float4(hi, hi, lo, lo);
  }
  for (int f = threadIdx.x; f < nfreq; f += blockDim.x) act[f] = !(fstate[f] == 2 || fstate[f] == 3);
  __syncthreads();
  const int64_t half = (n + 1) >> 1;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < half; e += (int64_t)gridDim.x * blockDim.x) {
    // values e and e + half (the last may not exist)
    const int64_t e2 = e + half < n ? e + half : e;
    float2 v[MMAX];
#pragma unroll
    for (int j = 0; j < MMAX; ++j)
      v[j] = j < md ? make_float2(s.V[(int64_t)j * ld + e], s.V[(int64_t)j * ld + e2]) : make_float2(0.f, 0.f);
    for (int f = 0; f < nfreq; ++f) {
      if (!act[f]) continue;
      float2 sx = make_float2(0.f, 0.f), cx = sx;
      const float4* cf = cf4 + f * MMAX;
#pragma unroll
      for (int j = 0; j < MMAX; ++j) {
        const float4 c = cf[j];
        rst_acc2(sx, cx, make_float2(c.x, c.y), make_float2(c.z, c.w), v[j]);
      }
      // (Y, lo) += sx + cx
      auto fold = [&](int64_t i, float sv, float cv) {
        float& yh = Y[(int64_t)f * n + i];
        float& yl = lo_acc[(int64_t)f * n + i];
        const float t = yh + sv;
        const float z = t - yh;
        const float err = (yh - (t - z)) + (sv - z);
        yh = t;
        yl += err + cv;
      };
      fold(e, sx.x, cx.x);
      if (e2 != e) fold(e2, sx.y, cx.y);
    }
  }
}

__global__ void __launch_bounds__(NTHREADS) k_rst_full64(Slot<double> s, int64_t ld, int64_t n, int nfreq,
                                                        const int* __restrict__ fstate,
                                                        const double* __restrict__ u, double* __restrict__ Y) {
  extern __shared__ __align__(16) double cf[];    // nfreq x MMAX
  __shared__ int act[MAXF];
  const int md = s.st->m_done;
  for (int q = threadIdx.x; q < nfreq * MMAX; q += blockDim.x) {
    const int j = q % MMAX;
    cf[q] = j < md ? u[q] * s.scale[j] : 0.0;
  }
  for (int f = threadIdx.x; f < nfreq; f += blockDim.x) act[f] = !(fstate[f] == 2 || fstate[f] == 3);
  __syncthreads();
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double v[MMAX];
#pragma unroll
    for (int j = 0; j < MMAX; ++j) v[j] = j < md ? s.V[(int64_t)j * ld + e] : 0.0;
    for (int f = 0; f < nfreq; ++f) {
      if (!act[f]) continue;
      double acc = 0.0;
#pragma unroll
      for (int j = 0; j < MMAX; ++j) acc = fma(cf[f * MMAX + j], v[j], acc);
      Y[(int64_t)f * n + e] += acc;
    }
  }
}

kx_status launch_rst_full(kx_ctx* c, cudaStream_t st, int slot, int nfreq, void* Y) {
  static SmemOptIn attr{};
  const kx_status so = smem_opt_in(c, attr, (const void*)k_rst_full32, MAXF * MMAX * sizeof(float4));
  if (so != KX_OK) return so;
  time_begin(c);
  if (c->d.precision == KX_FP64) {
    k_rst_full64<<<c->nblk, NTHREADS, nfreq * MMAX * sizeof(double), st>>>(make_slot<double>(c, slot), c->ld, c->n,
                                                                           nfreq, c->d_rst_state, c->d_rst_u,
                                                                           (double*)Y);
  } else {
    const int64_t blocks = std::min<int64_t>(((c->n + 1) / 2 + 127) / 128, (int64_t)c->nsm * 8);
    k_rst_full32<<<(int)blocks, 128, nfreq * MMAX * sizeof(float4), st>>>(make_slot<float>(c, slot), c->ld, c->n,
                                                                          nfreq, c->d_rst_state, c->d_rst_u,
                                                                          (float*)Y, (float*)c->d_zre);
  }
  time_end(c, KX_K_RESTART, (c->m + 3.0 * nfreq) * c->n * c->esize);
  KX_CHECK_LAUNCH(c);
  return KX_OK;
}

// ---------------------------------------------------------------------------
// Outputs: plane values in the context's precision and the summed |E|^2 per
// frequency (one CTA each); the full field's float pair folded to one float.
template <typename T>
__global__ void k_rst_out(const double* __restrict__ yp, int64_t P, T* __restrict__ E_plane, double* intensity) {
  const int f = blockIdx.x;
  double acc = 0.0;
  for (int64_t t = threadIdx.x; t < P; t += blockDim.x) {
    const double v = yp[(int64_t)f * P + t];
    if (E_plane) E_plane[(int64_t)f * P + t] = (T)v;
    acc += v * v;
  }
  __shared__ double red[32];
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    intensity[f] = s;
  }
}

__global__ void k_rst_fold(int64_t total, float* __restrict__ Y, const float* __restrict__ lo) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x)
    Y[e] += lo[e];
}

kx_status launch_rst_out(kx_ctx* c, cudaStream_t st, int nfreq, int64_t P, void* E_plane, double* d_intensity,
                         void* Y) {
  if (c->d.precision == KX_FP64)
    k_rst_out<double><<<nfreq, 1024, 0, st>>>(c->d_rst_yp, P, (double*)E_plane, d_intensity);
  else
    k_rst_out<float><<<nfreq, 1024, 0, st>>>(c->d_rst_yp, P, (float*)E_plane, d_intensity);
  KX_CHECK_LAUNCH(c);
  if (Y && c->d.precision == KX_FP32) {
    k_rst_fold<<<c->nblk, NTHREADS, 0, st>>>((int64_t)nfreq * c->n, (float*)Y, (const float*)c->d_zre);
    KX_CHECK_LAUNCH(c);
  }
  return KX_OK;
}

}  // namespace kx
