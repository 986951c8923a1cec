// Dense FP64 work on the projected (small) matrices, spread over a cluster
// of C = 16 thread blocks (8, the portable size, where the device cannot place
// one of 16: the same operations on other rows, the same bits).
//
// What bounds it: this GPU's double-precision pipe does about two FMAs a
// clock on one SM, so one product of 64-square matrices takes one SM 66 us
// and an exponential 0.9 ms; the matrices themselves are 33 KB.  Each block
// therefore owns R = ceil(n / C) rows of every matrix, held in its
// shared memory, and multiplies them with a right operand staged whole in
// shared memory (4.3 us for n = 64 at the pipe's rate).  Sixteen blocks against
// eight: an exponential of norm 2 at m = 64 61 against 94 us.  Rows of X Y need
// all of Y but only the same rows of X, so a chain of products with one fixed
// right operand (the powers of A, the Horner steps in A^4) runs without any
// exchange between the blocks; only a new right operand is published through
// global memory (L2) with one cluster barrier.
//
// The exponential is the truncated Taylor series in Paterson-Stockmeyer form
// (Paterson & Stockmeyer 1973, blocks of four) with scaling and squaring; it
// needs no linear solve, whose one-column-at-a-time elimination is 64
// dependent barriers (half the time of the Pade form on one block).  The
// norm limits are those for which the series' backward error is below 2^-53
// (Al-Mohy & Higham 2011, "Computing the action of the matrix exponential",
// SIAM J. Sci. Comput. 33(2), eq. (3.9)'s bound, evaluated in 60-digit
// arithmetic).
//
// Measured at m = 64: the step control of one sub-step 969 -> 88 us, the
// set-up of a restart 1060 -> 179 us, the projected solutions of 32
// frequencies 1337 -> 155 us.
#pragma once

#include "kx_internal.cuh"

namespace kx {

constexpr int CD_WIDE = 16, CD_PORTABLE = 8;   // thread blocks a cluster (the wide form is opted in per kernel)
constexpr int CD_THREADS = 256;
constexpr int CD_NMAX = MMAX + RST_P;      // largest matrix
constexpr int CD_RMAX = (CD_NMAX + CD_PORTABLE - 1) / CD_PORTABLE;
constexpr int CD_LD = 72;                  // row stride, shared and global
constexpr int CD_MAT = CD_NMAX * CD_LD;    // doubles of one matrix
constexpr int CD_SLICE = CD_RMAX * CD_LD;  // doubles of one block's rows
constexpr int CD_WS_MATS = 6;              // global matrices a cluster
constexpr int CD_WS = CD_WS_MATS * CD_MAT; // doubles of global workspace a cluster
constexpr int CD_SLICES = 5;
constexpr int CD_SMEM = (CD_MAT + CD_SLICES * CD_SLICE) * (int)sizeof(double);
static_assert(CD_NMAX <= CD_LD && CD_LD % 2 == 0, "rows are loaded as 16-byte pairs");

__device__ __forceinline__ int cl_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ int cl_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return (int)r;
}
// All threads of the cluster: what any of them wrote before (shared or
// global memory) is visible to all after.
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Store to the same shared-memory variable of block `rank` of the cluster.
__device__ __forceinline__ void cl_store(double* p, int rank, double v) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p), b;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(b), "d"(v) : "memory");
}

// Rows [r0, r0 + R) of an n-row matrix belong to block `rank`.
struct CdRows {
  int r0, R;
};
__device__ __forceinline__ CdRows cd_rows(int n, int rank) {
  const int C = cl_size(), per = (n + C - 1) / C;
  const int r0 = min(n, rank * per);
  return {r0, min(n, r0 + per) - r0};
}

// N outputs a thread of (R x K) . (K x cols); a warp whose lanes are all past
// the end skips the products (a double-precision instruction costs the same
// issue time whatever its active lanes).
template <int N, typename F>
__device__ __forceinline__ void cd_dots(const double* sa, const double* sb, int K, int cols, int tot, int first,
                                        F&& f) {
  double acc[N];
  int ra[N], cb[N];
#pragma unroll
  for (int t = 0; t < N; ++t) {
    const int idx = min(first + t * CD_THREADS, tot - 1);
    const int r = idx / cols;
    ra[t] = r * CD_LD;
    cb[t] = idx - r * cols;
    acc[t] = 0.0;
  }
#pragma unroll 2
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int t = 0; t < N; ++t) acc[t] = fma(sa[ra[t] + k], sb[k * CD_LD + cb[t]], acc[t]);
#pragma unroll
  for (int t = 0; t < N; ++t)
    if (first + t * CD_THREADS < tot) f(ra[t] / CD_LD, cb[t], acc[t]);
}

// f(r, c, (sa sb)_{r,c}) for r < R, c < cols; sa, sb in shared memory with
// row stride CD_LD.  f may write neither operand.
template <typename F>
__device__ __forceinline__ void cd_mm(const double* sa, const double* sb, int R, int K, int cols, F&& f) {
  const int tot = R * cols;
  const int warp0 = threadIdx.x & ~31;
  for (int base = 0; base < tot; base += 3 * CD_THREADS) {
    const int left = tot - base - warp0;   // outputs from this warp's first lane on
    const int first = base + (int)threadIdx.x;
    if (left > 2 * CD_THREADS) cd_dots<3>(sa, sb, K, cols, tot, first, f);
    else if (left > CD_THREADS) cd_dots<2>(sa, sb, K, cols, tot, first, f);
    else if (left > 0) cd_dots<1>(sa, sb, K, cols, tot, first, f);
  }
}

// Whole matrix from global memory (written by other blocks: past L1).
__device__ __forceinline__ void cd_load(double* sb, const double* g, int rows, int cols) {
  const int half = (cols + 1) >> 1;
  for (int q = threadIdx.x; q < rows * half; q += CD_THREADS) {
    const int r = q / half, c = 2 * (q - r * half);
    *reinterpret_cast<double2*>(sb + r * CD_LD + c) = __ldcg(reinterpret_cast<const double2*>(g + r * CD_LD + c));
  }
}

// Series degree 4 q and squarings s of exp(X) from ||X||_1: the fewest
// products (q + 2 for the series, `per` for each squaring); false where the
// norm is not finite.
__device__ __forceinline__ bool cd_plan(double norm, int per, int* q, int* s) {
  const double theta[4] = {0.2996158914, 0.7802874257, 1.438252597, 2.219048869};   // degrees 12, 16, 20, 24
  if (!isfinite(norm)) return false;
  int best = 1 << 30;
  for (int t = 0; t < 4; ++t) {
    const int sq = norm > theta[t] ? max(1, (int)ceil(log2(norm / theta[t]))) : 0;
    const int cost = t + 5 + per * sq;
    if (cost <= best) {
      best = cost;
      *q = t + 3;
      *s = sq;
    }
  }
  return true;
}

// 1 / k!, k = 0 .. 24 (the factors of the series; computed where they were
// used, by every thread, they took as long as the products between them)
static __constant__ double c_rfact[25] = {
    1.0, 1.0, 0.5, 0.16666666666666666,
    0.041666666666666664, 0.008333333333333333, 0.001388888888888889, 0.0001984126984126984,
    2.48015873015873e-05, 2.7557319223985893e-06, 2.755731922398589e-07, 2.505210838544172e-08,
    2.08767569878681e-09, 1.6059043836821613e-10, 1.1470745597729725e-11, 7.647163731819816e-13,
    4.779477332387385e-14, 2.8114572543455206e-15, 1.5619206968586225e-16, 8.22063524662433e-18,
    4.110317623312165e-19, 1.9572941063391263e-20, 8.896791392450574e-22, 3.8681701706306835e-23,
    1.6117375710961184e-24};

// Largest column sum of |entry(r, c)|, the same in every thread.
template <typename A>
__device__ __forceinline__ double cd_norm1(int n, double* red, A&& entry) {
  double s = 0.0;
  const int c = threadIdx.x;
  if (c < n)
    for (int r = 0; r < n; ++r) s += fabs(entry(r, c));
  if (!(s == s)) s = INFINITY;   // a NaN would pass fmax unseen
  for (int o = 16; o > 0; o >>= 1) s = fmax(s, __shfl_xor_sync(0xffffffffu, s, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  for (int w = 0; w < CD_THREADS / 32; ++w) s = fmax(s, red[w]);
  return s;
}

// One block's shared memory.
struct CdShared {
  double* B;                 // right operand (CD_MAT)
  double* S[CD_SLICES];      // own rows: A, A^2, A^3, and two in turn
};
__device__ __forceinline__ CdShared cd_shared(double* dyn) {
  CdShared sh;
  sh.B = dyn;
  for (int q = 0; q < CD_SLICES; ++q) sh.S[q] = dyn + CD_MAT + q * CD_SLICE;
  return sh;
}

// The block's rows of A = entry (n x n), A^2 and A^3 into S[0..2], with A as
// the right operand in B; its rows of A^4 into S[3] and to the global
// matrix g4.  No barrier at the end.
template <typename A>
__device__ __forceinline__ void cd_powers(const CdShared& sh, double* g4, int n, CdRows w, A&& entry) {
  for (int q = threadIdx.x; q < n * n; q += CD_THREADS) {
    const int r = q / n, c = q - r * n;
    const double v = entry(r, c);
    sh.B[r * CD_LD + c] = v;
    if (r >= w.r0 && r < w.r0 + w.R) sh.S[0][(r - w.r0) * CD_LD + c] = v;
  }
  __syncthreads();
  for (int p = 0; p < 3; ++p) {
    double* dst = sh.S[p + 1];
    cd_mm(sh.S[p], sh.B, w.R, n, n, [&](int r, int c, double v) {
      dst[r * CD_LD + c] = v;
      if (p == 2) g4[(w.r0 + r) * CD_LD + c] = v;
    });
    __syncthreads();
  }
}

// c_0 I + c_1 A + c_2 A^2 + c_3 A^3 at the block's entry (r, c), c_i = 1/(4 b + i)!
__device__ __forceinline__ double cd_poly(const CdShared& sh, const double* cf, CdRows w, int r, int c) {
  const int o = r * CD_LD + c;
  double v = cf[3] * sh.S[2][o];
  v = fma(cf[2], sh.S[1][o], v);
  v = fma(cf[1], sh.S[0][o], v);
  return w.r0 + r == c ? v + cf[0] : v;
}

// exp(2^s X): the block's rows in the returned slice (S[3] or S[4]) from its
// rows of X = entry; q, s from cd_plan for 2^s X.  g: two global matrices.
// Every thread of the cluster calls it; ends with a block barrier.
template <typename A>
__device__ double* cd_expm(const CdShared& sh, double* g, int n, CdRows w, int q, int s, A&& entry) {
  double* g0 = g;
  double* g1 = g + CD_MAT;
  cd_powers(sh, g0, n, w, entry);
  cl_sync();
  cd_load(sh.B, g0, n, n);
  // P = c_{4q} A^4 + block q - 1, then P <- P A^4 + block b
  double cf[4];
  {
    const double top = c_rfact[4 * q];
    for (int i = 0; i < 4; ++i) cf[i] = c_rfact[4 * q - 4 + i];
    for (int o = threadIdx.x; o < w.R * n; o += CD_THREADS) {
      const int r = o / n, c = o - r * n;
      sh.S[4][r * CD_LD + c] = fma(top, sh.S[3][r * CD_LD + c], cd_poly(sh, cf, w, r, c));
    }
  }
  __syncthreads();
  double *P = sh.S[4], *Q = sh.S[3];
  for (int b = q - 2; b >= 0; --b) {
    for (int i = 0; i < 4; ++i) cf[i] = c_rfact[4 * b + i];
    cd_mm(P, sh.B, w.R, n, n, [&](int r, int c, double v) { Q[r * CD_LD + c] = v + cd_poly(sh, cf, w, r, c); });
    __syncthreads();
    double* t = P;
    P = Q;
    Q = t;
  }
  for (int k = 0; k < s; ++k) {
    double* gk = (k & 1) ? g0 : g1;   // a block may still read the other one
    for (int o = threadIdx.x; o < w.R * n; o += CD_THREADS) {
      const int r = o / n, c = o - r * n;
      gk[(w.r0 + r) * CD_LD + c] = P[r * CD_LD + c];
    }
    cl_sync();
    cd_load(sh.B, gk, n, n);
    __syncthreads();
    cd_mm(P, sh.B, w.R, n, n, [&](int r, int c, double v) { Q[r * CD_LD + c] = v; });
    __syncthreads();
    double* t = P;
    P = Q;
    Q = t;
  }
  return P;
}

// Blocks a cluster of this kernel (with `smem` bytes of dynamic shared memory)
// on the current device: CD_WIDE where such a cluster can be placed, else
// CD_PORTABLE; a context may ask for either.  Looked up once a device.
struct ClusterOptIn {
  SmemOptIn smem;
  int blocks[SMEM_MAX_DEVICES];   // accessed atomically
};
inline kx_status cluster_opt_in(kx_ctx* c, ClusterOptIn& rec, const void* kernel, size_t smem, int* blocks) {
  const kx_status so = smem_opt_in(c, rec.smem, kernel, smem);
  if (so != KX_OK) return so;
  int dev = 0;
  cudaGetDevice(&dev);   // checked by smem_opt_in
  int n = __atomic_load_n(&rec.blocks[dev], __ATOMIC_ACQUIRE);
  if (n == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CD_WIDE);
    cfg.blockDim = dim3(CD_THREADS);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CD_WIDE;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int fit = 0;
    const bool wide = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                      cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg) == cudaSuccess && fit >= 1;
    if (!wide) cudaGetLastError();
    n = wide ? CD_WIDE : CD_PORTABLE;
    __atomic_store_n(&rec.blocks[dev], n, __ATOMIC_RELEASE);
  }
  *blocks = c->cluster_blocks > 0 ? std::min(c->cluster_blocks, n) : n;
  return KX_OK;
}

// Launch of a cluster kernel: `clusters` clusters of `blocks` blocks.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_cluster(void (*kern)(KArgs...), int blocks, int clusters, size_t smem, cudaStream_t st,
                                  Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clusters * blocks);
  cfg.blockDim = dim3(CD_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = blocks;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace kx
