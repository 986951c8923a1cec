// The two-pass Arnoldi process (Sect. 3.2, eqs. (Arn), (Arn1)) of a small
// grid in one cooperative launch.
//
// What bounds it: on grids whose basis lives in L2 a step moves little (a
// 36^3 vector is 1.1 MB) and its time is latency: three launches (pass A, its
// finalisation, pass B) with their start-up loads cost about 20 us a step,
// whatever the columns.  Here every thread keeps one item (a quad of x-cells,
// or one cell) for the whole process, the new vector stays in its registers
// between the dots and the update (it is never written before it is
// orthogonal), and a step has two grid barriers: after the partial dots, and
// after the partial norms, which also orders the new column before its
// neighbours' reads (double precision: a third, after the dots' totals).  Every block sums the same partials in the same order,
// so all reach the same coefficients and decisions; block 0 records them.
//   phase A: w = A v_j, partial dots V_i . w (i <= j) and ||w||^2
//   phase B: v_{j+1} = w - sum_i h_ij v_i (compensated in FP32), partial norm
// A thread always reads the same part of every column.  The first columns,
// those read most often, are held in its SM's shared memory (the barrier's
// acquire drops L1; m = 64, us with and without: 64^3 3758 and 3951 (4
// columns), 48^3 1551 and 1725 (8), 36^3 1118 and 1184 (16), 2D 64^2 in double
// precision 908 and 946 (all)); the others stay in its die's L2, phase A
// taking them upwards and phase B downwards, each starting on those the other
// ended on.
// Where a block's items fill less than half of it, its warps split the
// columns as well (CS groups; the groups' shares of the update are added
// through shared memory).
//
// Only data another block wrote is read past L1 (the stencil's neighbours,
// the partials); a thread's own columns are plain loads.
// Every barrier wait is bounded: when one runs out the block records
// KX_ETIMEOUT and returns, and so do the others.
// One slot's blocks take nearly every SM, for the shortest process; contexts of
// several slots, or driven beside others, may take fewer (coop_run).
#include <atomic>

#include "kx_eft.cuh"
#include "kx_internal.cuh"
#include "kx_reduce.cuh"
#include "kx_stencil.cuh"

namespace kx {

namespace {

constexpr int CO_GROUPT = 256;             // threads a block may have by splitting the columns
// Shared memory a block may take: past 196 KB the next carve-out leaves 28 KB
// of L1, too few for the loads in flight (64^3 with 4 columns held 3758 us,
// with 5 4430; 45^3 cells with 8 1585, with 16 1737).
constexpr size_t CO_SMEM = 195 * 1024;

// Barrier over the `blocks` blocks of a slot: the counter reaches `target`
// (blocks times the barriers so far; zeroed by the kernel that normalises
// column 0).  False when the wait runs out: after `limit` polls (a cooperative
// grid starts all its blocks or none, measured beside a kernel that held half of
// the SMs, so other kernels' blocks are never waited for here).  Four polls a
// round of the loop: with one the double-precision process took 1.3 % longer
// (32^3 2845 us, 2811).  The release on the arrival covers the writes of the
// whole block (ordered before it by the block barrier), and the acquire on the
// poll the reads after it.
__device__ __forceinline__ bool grid_barrier(unsigned* cnt, unsigned target, unsigned limit) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(cnt) : "memory");
    int good = 0;
#pragma unroll 4
    for (unsigned k = 0; k < limit; ++k) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
      if ((int)(v - target) >= 0) {
        good = 1;
        break;
      }
    }
    ok = good;
  }
  __syncthreads();
  return ok != 0;
}

// Sums over warps and blocks.  Single precision: an unevaluated pair hi + lo
// (Knuth's TwoSum at every addition, 2^-48 of the terms), because a chain of
// double-precision additions is what these reductions would wait for on this
// GPU (tens of clocks each; every block sums up to 65 columns of partials).
// The terms are a warp's float sums, good to 2^-24, so the five bits fewer than
// in double precision are not seen: fields of the plain method against a
// double-precision context, geometric means over 48 media of 24^3 to 64^3,
// 3.61e-7 with the per-step launches (which sum in double precision), 3.61e-7
// with pairs, 3.63e-7 with triples (2^-72; 45^3 1585 -> 1880 us a process).
// Double precision: double.
struct Pair {
  float h, l;
};
__device__ __forceinline__ Pair add(Pair a, Pair b) {
  Pair r;
  r.h = a.h + b.h;
  const float z = r.h - a.h;
  r.l = (a.l + b.l) + ((a.h - (r.h - z)) + (b.h - z));
  return r;
}
__device__ __forceinline__ Pair add(Pair a, float b) {
  Pair r;
  r.h = a.h + b;
  const float z = r.h - a.h;
  r.l = a.l + ((a.h - (r.h - z)) + (b - z));
  return r;
}
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ Pair shfl(Pair a, int o) {
  return {__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
}
__device__ __forceinline__ double shfl(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ double value(Pair a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ double value(double a) { return a; }
template <typename T> struct SumOf;
template <> struct SumOf<float> {
  using S = Pair;
  static __device__ __forceinline__ S of(float x) { return {x, 0.f}; }
  static __device__ __forceinline__ S get(const double* p) {
    const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
    return {v.x, v.y};
  }
  static __device__ __forceinline__ void put(double* p, S v) { *reinterpret_cast<float2*>(p) = make_float2(v.h, v.l); }
};
template <> struct SumOf<double> {
  using S = double;
  static __device__ __forceinline__ S of(double x) { return x; }
  static __device__ __forceinline__ S get(const double* p) { return __ldcg(p); }
  static __device__ __forceinline__ void put(double* p, S v) { *p = v; }
};
template <typename S>
__device__ __forceinline__ S warp_total(S x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = add(x, shfl(x, o));
  return x;
}
// warp_sum8 over these sums
template <typename S>
__device__ __forceinline__ S warp_total8(S* p, int lane) {
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
#pragma unroll
  for (int t = 0; t < 4; ++t) p[t] = add(b4 ? p[t + 4] : p[t], shfl(b4 ? p[t] : p[t + 4], 16));
#pragma unroll
  for (int t = 0; t < 2; ++t) p[t] = add(b3 ? p[t + 2] : p[t], shfl(b3 ? p[t] : p[t + 2], 8));
  S x = add(b2 ? p[1] : p[0], shfl(b2 ? p[0] : p[1], 4));
  x = add(x, shfl(x, 2));
  return add(x, shfl(x, 1));
}
constexpr int TOT_COL = PCOLS - 2;   // partial column that holds the totals (double precision)

__device__ __forceinline__ float ldcg_w(const float* p, int idx, unsigned w, int c) {
  return (w >> c) & 1u ? 0.f : __ldcg(p + idx);
}
__device__ __forceinline__ float4 ldcg_w4(const float* p, int idx, unsigned w0, unsigned w1, int c) {
  float4 r = __ldcg(reinterpret_cast<const float4*>(p + idx));
  if ((w0 >> c) & 1u) r.x = 0.f;
  if ((w1 >> c) & 1u) {
    r.y = 0.f;
    r.z = 0.f;
    r.w = 0.f;
  }
  return r;
}
__device__ __forceinline__ float4 mul4(const float4& a, const float4& b) {
  return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w);
}

// Items of four x-cells, 3D FP32 lossy layer (nx % 4 == 0): stencil_quad32's
// operations, field loads past L1.
template <int AUG, int TR, int MT>
struct QuadItem {
  using T = float;
  using V = float4;
  static constexpr int NC = 6;
  // columns in flight in the dots and the update (what the registers hold)
  static constexpr int BATCH = MT <= 384 ? 4 : 2, MAXT = MT;
  static __device__ __forceinline__ int64_t count(const Geo& g) { return g.ncell >> 2; }
  static __device__ __forceinline__ int64_t first(int64_t item) { return item << 2; }
  static __device__ __forceinline__ V zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ V load(const T* p) { return *reinterpret_cast<const float4*>(p); }
  static __device__ __forceinline__ void store(T* p, const V& v) { *reinterpret_cast<float4*>(p) = v; }
  static __device__ __forceinline__ T dot(const V& a, const V& b) { return dot4(a, b); }
  static __device__ __forceinline__ void sub(V& hi, V& lo, T c, const V& v) { sub_fma4(hi, lo, -c, v); }
  static __device__ __forceinline__ V fold(const V& h, const V& l) {
    return make_float4(h.x + l.x, h.y + l.y, h.z + l.z, h.w + l.w);
  }
  static __device__ __forceinline__ void join(V& h, V& l, const V& a, const V& b) {
    add_two(h.x, l.x, a.x);
    add_two(h.y, l.y, a.y);
    add_two(h.z, l.z, a.z);
    add_two(h.w, l.w, a.w);
    l = fold(l, b);
  }
  // o = s A v (+ gco g), s = tsj
  static __device__ __forceinline__ void apply(const Geo& g, const T* v, const T* __restrict__ ie,
                                               const T* __restrict__ sig2, const T* __restrict__ gsrc, T tsj, T gco,
                                               int64_t item, V* o) {
    const int nc = (int)g.ncell;
    const int c0 = (int)(item << 2);
    const int nx = g.nx, ny = g.ny, nz = g.nz, nxy = nx * ny;
    const unsigned r = (unsigned)c0 / (unsigned)nx;
    const int i0 = c0 - (int)r * nx;
    const unsigned kq = r / (unsigned)ny;
    const int jj = (int)r - (int)kq * ny, kk = (int)kq;
    const int jp = (jj + 1 == ny) ? 0 : jj + 1, jm = (jj == 0) ? ny - 1 : jj - 1;
    const int kp = (kk + 1 == nz) ? 0 : kk + 1, km = (kk == 0) ? nz - 1 : kk - 1;
    const int cjp = c0 + (jp - jj) * nx, cjm = c0 + (jm - jj) * nx;
    const int ckp = c0 + (kp - kk) * nxy, ckm = c0 + (km - kk) * nxy;
    const int ixp = (i0 + 4 == nx) ? 0 : i0 + 4, ixm = (i0 == 0) ? nx - 1 : i0 - 1;
    const int cxp = c0 - i0 + ixp, cxm = c0 - i0 + ixm;
    const unsigned xm = wall_bits(g, 0), ym = wall_bits(g, 1), zm = wall_bits(g, 2);
    const unsigned wx0 = i0 == 0 ? xm : 0u, wy = jj == 0 ? ym : 0u, wz = kk == 0 ? zm : 0u;
    const unsigned wyp = jp == 0 ? ym : 0u, wym = jm == 0 ? ym : 0u, wzp = kp == 0 ? zm : 0u;
    const unsigned wzm = km == 0 ? zm : 0u;
    const unsigned o0 = wx0 | wy | wz, o1 = wy | wz;
    const T *vHx = v, *vHy = v + nc, *vHz = v + 2 * (int64_t)nc;
    const T *vEx = v + 3 * (int64_t)nc, *vEy = v + 4 * (int64_t)nc, *vEz = v + 5 * (int64_t)nc;
    const T *ie1p = ie + nc, *ie2p = ie + 2 * (int64_t)nc;
    const float4 Hx = ldcg_w4(vHx, c0, o0, o1, 0), Hy = ldcg_w4(vHy, c0, o0, o1, 1), Hz = ldcg_w4(vHz, c0, o0, o1, 2);
    float4 Ex = ldcg_w4(vEx, c0, o0, o1, 3), Ey = ldcg_w4(vEy, c0, o0, o1, 4), Ez = ldcg_w4(vEz, c0, o0, o1, 5);
    float4 Ez_jp = ldcg_w4(vEz, cjp, wx0 | wyp | wz, wyp | wz, 5), Ex_jp = ldcg_w4(vEx, cjp, wx0 | wyp | wz, wyp | wz, 3);
    float4 Ey_kp = ldcg_w4(vEy, ckp, wx0 | wy | wzp, wy | wzp, 4), Ex_kp = ldcg_w4(vEx, ckp, wx0 | wy | wzp, wy | wzp, 3);
    const float4 Hz_jm = ldcg_w4(vHz, cjm, wx0 | wym | wz, wym | wz, 2), Hx_jm = ldcg_w4(vHx, cjm, wx0 | wym | wz, wym | wz, 0);
    const float4 Hy_km = ldcg_w4(vHy, ckm, wx0 | wy | wzm, wy | wzm, 1), Hx_km = ldcg_w4(vHx, ckm, wx0 | wy | wzm, wy | wzm, 0);
    const unsigned wxp = (ixp == 0 ? xm : 0u) | wy | wz, wxm = (ixm == 0 ? xm : 0u) | wy | wz;
    float Ez_n = ldcg_w(vEz, cxp, wxp, 5), Ey_n = ldcg_w(vEy, cxp, wxp, 4);
    const float Hz_p = ldcg_w(vHz, cxm, wxm, 2), Hy_p = ldcg_w(vHy, cxm, wxm, 1);
    const float4 ie0 = ld4(ie + c0), ie1 = ld4(ie1p + c0), ie2 = ld4(ie2p + c0);
    if (TR) {
      // A^T: the curl of E / eps, then plain E rows
      Ex = mul4(Ex, ie0);
      Ey = mul4(Ey, ie1);
      Ez = mul4(Ez, ie2);
      Ez_jp = mul4(Ez_jp, ld4(ie2p + cjp));
      Ex_jp = mul4(Ex_jp, ld4(ie + cjp));
      Ey_kp = mul4(Ey_kp, ld4(ie1p + ckp));
      Ex_kp = mul4(Ex_kp, ld4(ie + ckp));
      Ez_n *= ie2p[cxp];
      Ey_n *= ie1p[cxp];
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int li = g.la == 0 ? i0 + e : (g.la == 1 ? jj : kk);
      float sg[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) sg[c] = sig2[2 * li + g.sighalf[c]];
      const float ez = f4(Ez, e), ey = f4(Ey, e), ex = f4(Ex, e);
      const float hx = f4(Hx, e), hy = f4(Hy, e), hz = f4(Hz, e);
      const float ez_ip = e < 3 ? f4(Ez, e + 1) : Ez_n;
      const float ey_ip = e < 3 ? f4(Ey, e + 1) : Ey_n;
      const float hz_im = e > 0 ? f4(Hz, e - 1) : Hz_p;
      const float hy_im = e > 0 ? f4(Hy, e - 1) : Hy_p;
      const float cHx = (hz - f4(Hz_jm, e)) - (hy - f4(Hy_km, e));
      const float cHy = (hx - f4(Hx_km, e)) - (hz - hz_im);
      const float cHz = (hy - hy_im) - (hx - f4(Hx_jm, e));
      const float uEx = (f4(Ez_jp, e) - ez) - (f4(Ey_kp, e) - ey);
      const float uEy = (f4(Ex_kp, e) - ex) - (ez_ip - ez);
      const float uEz = (ey_ip - ey) - (f4(Ex_jp, e) - ex);
      float out[6];
      out[0] = sg[0] * hx + (TR ? -uEx : uEx);
      out[1] = sg[1] * hy + (TR ? -uEy : uEy);
      out[2] = sg[2] * hz + (TR ? -uEz : uEz);
      out[3] = TR ? sg[3] * ex + cHx : f4(ie0, e) * (sg[3] * ex - cHx);
      out[4] = TR ? sg[4] * ey + cHy : f4(ie1, e) * (sg[4] * ey - cHy);
      out[5] = TR ? sg[5] * ez + cHz : f4(ie2, e) * (sg[5] * ez - cHz);
      const unsigned me = e == 0 ? o0 : o1;
#pragma unroll
      for (int c = 0; c < 6; ++c) set4(o[c], e, (me >> c) & 1u ? 0.f : out[c] * tsj);
    }
    if (AUG) {
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const float4 q = ldw4(gsrc + c * (int64_t)nc, c0, o0, o1, c);
        o[c].x += gco * q.x;
        o[c].y += gco * q.y;
        o[c].z += gco * q.z;
        o[c].w += gco * q.w;
      }
    }
  }
};

// Items of one cell: any model and precision.
template <typename TT, int DIM, int AUG, int TR>
struct CellItem {
  using T = TT;
  using V = TT;
  static constexpr int NC = ncomp_of(DIM);
  static constexpr int BATCH = sizeof(T) == 4 || NC < 6 ? 8 : 4, MAXT = DIM == 3 ? 768 : 512;
  static __device__ __forceinline__ int64_t count(const Geo& g) { return g.ncell; }
  static __device__ __forceinline__ int64_t first(int64_t item) { return item; }
  static __device__ __forceinline__ V zero() { return T(0); }
  static __device__ __forceinline__ V load(const T* p) { return *p; }
  static __device__ __forceinline__ void store(T* p, const V& v) { *p = v; }
  static __device__ __forceinline__ T dot(const V& a, const V& b) { return a * b; }
  static __device__ __forceinline__ void sub(V& hi, V& lo, T c, const V& v) {
    if constexpr (sizeof(T) == 4) sub_fma(hi, lo, -c, v);
    else hi = fma(-c, v, hi);
  }
  static __device__ __forceinline__ V fold(const V& h, const V& l) { return sizeof(T) == 4 ? h + l : h; }
  static __device__ __forceinline__ void join(V& h, V& l, const V& a, const V& b) {
    if constexpr (sizeof(T) == 4) {
      add_two(h, l, a);
      l += b;
    } else {
      h += a;
    }
  }
  static __device__ __forceinline__ void apply(const Geo& g, const T* v, const T* __restrict__ ie,
                                               const T* __restrict__ sig2, const T* __restrict__ gsrc, T tsj, T gco,
                                               int64_t item, V* o) {
    const Cell q = make_cell(g, item);
    stencil<T, DIM, TR, TableMat<T>, true>(g, v, TableMat<T>{ie, sig2}, q, o);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      o[c] *= tsj;
      if (AUG) {
        if (!is_wall(g, c, q.i, q.j, q.k)) o[c] += gco * gsrc[(int64_t)c * g.ncell + item];
      }
    }
  }
};

// nti: items a block; the block's blockDim.x / nti groups of warps split the
// columns in chunks of eight.  Loads of a chunk carry no conditions (a column
// past the last reads the last again and is not used, an idle thread reads
// item 0), so that they are all in flight together.
template <typename P, int AUG>
__global__ void __launch_bounds__(P::MAXT, 1) k_coop(Geo g, SlotSet<typename P::T> ss, int m, int64_t ld,
                                                    const typename P::T* __restrict__ ie,
                                                    const typename P::T* __restrict__ sig2,
                                                    const typename P::T* __restrict__ gsrc, int ldh, double btol,
                                                    int nti, int kc, unsigned wait) {
  using T = typename P::T;
  using V = typename P::V;
  using SO = SumOf<T>;
  using S = typename SO::S;
  constexpr int NC = P::NC;
  extern __shared__ __align__(16) unsigned char co_dyn[];
  V* share = reinterpret_cast<V*>(co_dyn);            // groups x 2 NC x nti (more than one group)
  V* keep = share + ((int)blockDim.x > nti ? 2 * NC * blockDim.x : 0);   // columns 0 .. kc-1: kc x NC x nti
  __shared__ T acc[P::MAXT / 32][MMAX + 2];           // a warp's dots; column MMAX + 1: ||w||^2
  __shared__ S red[P::MAXT / 32];
  __shared__ double tot[MMAX + 8], scl[MMAX + 1], augs[2 * (MMAX + 1)];
  __shared__ T coef[MMAX + 8];
  __shared__ T sh_sj, sh_gco;                         // scale of v_j, factor of g
  __shared__ int halt, sh_bad;
  const Slot<T> s = slot_at(ss, blockIdx.y);
  SlotState* st = s.st;
  if (st->done || st->retired) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int grp = tid / nti, it = tid - grp * nti, ngrp = blockDim.x / nti, wpg = nti >> 5;
  const int b = blockIdx.x, G = gridDim.x;
  const bool rec = b == 0;
  unsigned* cnt = s.counter + 1;
  unsigned bars = 0;
  const int64_t item = (int64_t)b * nti + it;
  const bool act = item < P::count(g);
  const int64_t nc = g.ncell;
  T* Vc = s.V + (act ? P::first(item) : 0);           // this thread's part of column 0
  const bool augm = AUG && st->aug;
  // warp 0's own: double-precision work on few values, kept off the others
  const double omega = augm ? st->omega : 0.0, reta = augm ? 1.0 / st->eta : 0.0;
  double wmax2 = st->wmax * st->wmax, sj = s.scale[0], na = 0.0, nb = 0.0;
  if (tid == 0) {
    scl[0] = sj;
    augs[0] = s.aug[0];
    augs[1] = s.aug[1];
    sh_sj = (T)sj;
    sh_gco = augm ? (T)(-(sj * s.aug[0]) * reta) : T(0);
  }
  auto timeout = [&]() {
    if (tid == 0) {
      st->status = KX_ETIMEOUT;
      st->done = 1;
    }
  };
  if (grp == 0 && kc > 0) {
#pragma unroll
    for (int c = 0; c < NC; ++c) keep[c * nti + it] = act ? P::load(Vc + c * nc) : P::zero();
  }
  // this thread's part of columns col .. col + N - 1 (past j: column j)
  auto batch = [&](auto& v, int col, int j) {
    constexpr int N = sizeof(v) / sizeof(v[0]);
    if (min(col + N - 1, j) < kc) {
#pragma unroll
      for (int t = 0; t < N; ++t) {
        const V* vc = keep + min(col + t, j) * NC * nti + it;
#pragma unroll
        for (int c = 0; c < NC; ++c) v[t][c] = vc[c * nti];
      }
    } else {
#pragma unroll
      for (int t = 0; t < N; ++t) {
        const T* vc = Vc + (int64_t)min(col + t, j) * ld;
#pragma unroll
        for (int c = 0; c < NC; ++c) v[t][c] = P::load(vc + c * nc);
      }
    }
  };
  __syncthreads();
  for (int j = 0; j < m; ++j) {
    const int ncol = j + 1;
    // phase A
    V o[NC];
    if (act) {
      int64_t im = item;
      asm volatile("" : "+l"(im));   // the index work is redone each step: held over the loop it would spill
      P::apply(g, s.V + (int64_t)j * ld, ie, sig2, gsrc, sh_sj, sh_gco, im, o);
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c) o[c] = P::zero();
    }
    for (int c0 = 8 * grp; c0 < ncol; c0 += 8 * ngrp) {
      T p[8];
#pragma unroll
      for (int h = 0; h < 8; h += P::BATCH) {
        V v[P::BATCH][NC];
        batch(v, c0 + h, j);
#pragma unroll
        for (int t = 0; t < P::BATCH; ++t) {
          p[h + t] = T(0);
#pragma unroll
          for (int c = 0; c < NC; ++c) p[h + t] += P::dot(v[t][c], o[c]);
        }
      }
      const T x = warp_sum8(p, lane);
      const int col = c0 + column_of_lane8(lane);
      if ((lane & 3) == 0 && col < ncol) acc[warp][col] = x;
    }
    if (grp == 0) {
      T nrm = T(0);
#pragma unroll
      for (int c = 0; c < NC; ++c) nrm += P::dot(o[c], o[c]);
      nrm = warp_sum(nrm);
      if (lane == 0) acc[warp][MMAX + 1] = nrm;
    }
    __syncthreads();
    for (int col = tid; col <= ncol; col += blockDim.x) {
      const int w0 = col < ncol ? ((col >> 3) % ngrp) * wpg : 0, src = col < ncol ? col : MMAX + 1;
      S t = SO::of(acc[w0][src]);
      for (int w = 1; w < wpg; ++w) t = add(t, acc[w0 + w][src]);
      SO::put(s.part + (int64_t)col * s.ps + b, t);
    }
    bars += G;
    if (!grid_barrier(cnt, bars, wait)) return timeout();
    if constexpr (sizeof(T) == 4) {
      // the dots' totals in every block, eight columns a warp
      for (int c0 = 8 * warp; c0 <= ncol; c0 += 8 * nw) {
        S p[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) p[t] = SO::of(T(0));
#pragma unroll 2
        for (int q = lane; q < G; q += 32)
#pragma unroll
          for (int t = 0; t < 8; ++t) p[t] = add(p[t], SO::get(s.part + (int64_t)min(c0 + t, ncol) * s.ps + q));
        const S x = warp_total8(p, lane);
        if ((lane & 3) == 0 && c0 + column_of_lane8(lane) <= ncol) tot[c0 + column_of_lane8(lane)] = value(x);
      }
    } else {
      // one warp a column somewhere in the grid, and a barrier more: cheaper
      // than 65 columns of double-precision additions in every block
      for (int col = b + warp * G; col <= ncol; col += nw * G) {
        S x = SO::of(T(0));
        for (int q = lane; q < G; q += 32) x = add(x, SO::get(s.part + (int64_t)col * s.ps + q));
        x = warp_total(x);
        if (lane == 0) SO::put(s.part + (int64_t)TOT_COL * s.ps + col, x);
      }
      bars += G;
      if (!grid_barrier(cnt, bars, wait)) return timeout();
      for (int col = tid; col <= ncol; col += blockDim.x) tot[col] = SO::get(s.part + (int64_t)TOT_COL * s.ps + col);
    }
    __syncthreads();
    // h_ij and the phase entries' update (a lane a column)
    if (warp == 0) {
      const double wa = augm ? -omega * sj * augs[2 * j + 1] : 0.0, wb = augm ? omega * sj * augs[2 * j] : 0.0;
      double pa = 0.0, pb = 0.0;
      int bad = 0;
      for (int q = lane; q < ((ncol + 7) & ~7); q += 32) {
        double cc = 0.0;
        if (q < ncol) {
          double t = tot[q];
          if (AUG && augm) t += augs[2 * q] * wa + augs[2 * q + 1] * wb;
          const double h = scl[q] * t;
          cc = h * scl[q];
          if (rec) s.H[q + (int64_t)j * ldh] = h;
          bad |= !isfinite(h);
          if (AUG && augm) {
            pa += cc * augs[2 * q];
            pb += cc * augs[2 * q + 1];
          }
        }
        coef[q] = (T)cc;   // zero past the last column of the last chunk
      }
      if (AUG && augm) {
        na = wa - warp_sum(pa);
        nb = wb - warp_sum(pb);
      }
      const double wn2 = tot[ncol] + (wa * wa + wb * wb);
      bad |= !isfinite(wn2);
      if (wn2 > wmax2) wmax2 = wn2;
      bad = __any_sync(0xffffffffu, bad);
      if (lane == 0) sh_bad = bad;
    }
    __syncthreads();
    if (sh_bad) {
      if (rec && tid == 0) {
        st->status = KX_ENONFINITE;
        st->done = 1;
      }
      return;
    }
    // phase B: this group's columns, downwards
    V lo[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      lo[c] = P::zero();
      if (grp > 0) o[c] = P::zero();
    }
    {
      const int chunks = (ncol + 7) >> 3;
      for (int ch = grp + ((chunks - 1 - grp) / ngrp) * ngrp; ch >= 0 && ch < chunks; ch -= ngrp) {
        const int c0 = 8 * ch;
#pragma unroll
        for (int h = 8 - P::BATCH; h >= 0; h -= P::BATCH) {
          V v[P::BATCH][NC];
          batch(v, c0 + h, j);
#pragma unroll
          for (int t = P::BATCH - 1; t >= 0; --t)
#pragma unroll
            for (int c = 0; c < NC; ++c) P::sub(o[c], lo[c], coef[c0 + h + t], v[t][c]);
        }
      }
    }
    T* out = Vc + (int64_t)(j + 1) * ld;
    V* kout = keep + (j + 1) * NC * nti + it;
    const bool held = j + 1 < kc;
    // at most four squares (a quad's, or of three components of a cell) summed in
    // the working precision, as in pass B (plain method at 64^3, T = 400, twelve
    // media, field errors: 5.1e-7 with a thread's 24 squares in floats, 4.6e-7
    // so and by the per-step launches)
    constexpr int SQ = sizeof(V) > sizeof(T) ? 1 : 3;
    S t2 = SO::of(T(0));
    T sq = T(0);
    if (ngrp == 1) {
      if (act) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          o[c] = P::fold(o[c], lo[c]);
          P::store(out + c * nc, o[c]);
          sq += P::dot(o[c], o[c]);
          if (c % SQ == SQ - 1 || c == NC - 1) {
            t2 = add(t2, sq);
            sq = T(0);
          }
        }
      }
      if (held) {
#pragma unroll
        for (int c = 0; c < NC; ++c) kout[c * nti] = act ? o[c] : P::zero();
      }
    } else {
      // the groups' shares added, a component a group
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        share[((size_t)grp * 2 * NC + c) * nti + it] = o[c];
        share[((size_t)grp * 2 * NC + NC + c) * nti + it] = lo[c];
      }
      __syncthreads();
      if (held && !act)
        for (int c = grp; c < NC; c += ngrp) kout[c * nti] = P::zero();
      if (act)
        for (int c = grp; c < NC; c += ngrp) {
          V h = share[(size_t)c * nti + it], l = share[(size_t)(NC + c) * nti + it];
          for (int q = 1; q < ngrp; ++q)
            P::join(h, l, share[((size_t)q * 2 * NC + c) * nti + it], share[((size_t)q * 2 * NC + NC + c) * nti + it]);
          h = P::fold(h, l);
          P::store(out + c * nc, h);
          if (held) kout[c * nti] = h;
          sq += P::dot(h, h);   // cells: three components at most
          if (SQ == 1) {
            t2 = add(t2, sq);
            sq = T(0);
          }
        }
      if (SQ > 1) t2 = add(t2, sq);
    }
    const S n2 = warp_total(t2);
    if (lane == 0) red[warp] = n2;
    __syncthreads();
    if (tid == 0) {
      S t = red[0];
      for (int w = 1; w < nw; ++w) t = add(t, red[w]);
      SO::put(s.part + (int64_t)FINB_COL * s.ps + b, t);
      // the host's stop request, as block 0 sees it, for every block
      if (rec) s.counter[2] = abort_requested(st) ? 1u : 0u;
    }
    bars += G;
    if (!grid_barrier(cnt, bars, wait)) return timeout();
    if (warp == 0) {
      S xs = SO::of(T(0));
      for (int q = lane; q < G; q += 32) xs = add(xs, SO::get(s.part + (int64_t)FINB_COL * s.ps + q));
      const int abrt = __ldcg(s.counter + 2) != 0u;
      const double x = value(warp_total(xs)) + (na * na + nb * nb);   // h_{j+1,j}^2
      int stop = 0;
      double sc = 0.0;
      if (!isfinite(x)) stop = 2;
      else if (x <= btol * btol * wmax2) stop = 1;   // invariant subspace: the projection is exact
      else sc = rsqrt(x);
      sj = sc;
      if (lane == 0) {
        scl[j + 1] = sc;
        augs[2 * (j + 1)] = na;
        augs[2 * (j + 1) + 1] = nb;
        sh_sj = (T)sc;
        if (AUG) sh_gco = (T)(-(sc * na) * reta);
        halt = stop || abrt;
        if (rec) {
          s.scale[j + 1] = sc;
          if (AUG) {
            s.aug[2 * (j + 1)] = na;
            s.aug[2 * (j + 1) + 1] = nb;
          }
          st->m_done = j + 1;
          if (stop == 2) st->status = KX_ENONFINITE;
          if (stop || abrt) st->done = 1;
        }
      }
      if (rec && lane == 0) s.H[(j + 1) + (int64_t)j * ldh] = sqrt(x);
    }
    __syncthreads();
    if (halt) return;
  }
}

struct CoopPlan {
  int nti, groups, blocks, slots;   // slots: how many fit one launch
  int keep;                         // columns held in shared memory
  size_t smem;
};

// Blocks of nti items each; groups of warps that split the columns where that
// leaves CO_GROUPT threads half used or less.  slots: how many slots' blocks
// are resident at once.  The first columns are held in whole batches in `room`
// bytes a block, as far as none of `want` slots is put off for them.
CoopPlan coop_plan(const kx_ctx* c, const void* kernel, int64_t items, int nti, int want, int m, size_t vbytes, int ncomp,
                   int batch, size_t room) {
  CoopPlan p{nti, std::max(1, CO_GROUPT / nti), (int)((items + nti - 1) / nti), 0, 0, 0};
  const size_t part = (size_t)ncomp * p.nti * vbytes;   // a block's part of a column
  p.smem = p.groups > 1 ? p.groups * 2 * part : 0;
  auto slots = [&](size_t smem) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, p.nti * p.groups, smem) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return (int)((int64_t)occ * c->nsm / p.blocks);
  };
  p.slots = slots(p.smem);
  const int need = std::min(want, p.slots);
  int k = room > p.smem ? (int)std::min<size_t>(m, (room - p.smem) / part) : 0;
  if (k < m) k -= k % batch;
  for (; p.slots > 0 && k > 0; k = (k - 1) / batch * batch) {
    const int fit = slots(p.smem + k * part);
    if (fit < need) continue;
    p.keep = k;
    p.smem += k * part;
    p.slots = fit;
    break;
  }
  return p;
}

// Estimated microseconds of one step of `want` slots, on GB300: fixed cost of
// the barriers and sums, a value's products and update with m / 2 columns by
// the threads of an SM (its items, in as many blocks as share it), and the
// basis' two reads where that is more.  Measured (m = 64, items a block: us):
// 24^3 32: 12.9, 128: 15.3, 256: 20.4, 512: 32; double precision 24^3 96: 27.7,
// 256: 46.7; 2D 64^2 in double precision (m = 30) 32: 15.2, 256: 21.9.
double coop_us(const kx_ctx* c, const CoopPlan& p, int want, int m, int values) {
  const bool f64 = c->esize == 8;
  const int used = std::min(want, p.slots);
  const int share = (int)(((int64_t)used * p.blocks + c->nsm - 1) / c->nsm);
  const double work = (f64 ? 14.0 : 10.0) + (f64 ? 7e-4 : 5.6e-5) * share * p.nti * values * (0.5 * m);
  const double mem = (double)used * c->n * c->esize * m / 7.5e6;
  return std::max(work, mem) * ((want + p.slots - 1) / p.slots);
}
// The same with the per-step launches, which serve every slot: 24^3 1 slot 26,
// 32 slots 148; 36^3 31 and 466; 2D 128^2 in double precision 32 slots 233.
// Beside other contexts' launches the fixed cost is hidden by theirs.
double steps_us(const kx_ctx* c, int want, int m) {
  return 22.0 / c->sharers + (c->esize == 8 ? 5.5e-6 : 1.54e-6) * want * c->n * (0.5 * m);
}

template <typename P, int AUG>
kx_status coop_run(kx_ctx* c, int slot0, int ns, int want, int m, const void* g_aug, int64_t items, bool* ran) {
  using T = typename P::T;
  using V = typename P::V;
  const void* fn = (const void*)k_coop<P, AUG>;
  static SmemOptIn attr{};
  want *= c->sharers;
  // CO_SMEM less the kernel's own arrays (the largest: the warps' dots)
  constexpr size_t ROOM = CO_SMEM - (P::MAXT / 32 * (MMAX + 2) + MMAX) * sizeof(T) - 5 * 1024;
  static_assert(ROOM >= (size_t)2 * P::NC * CO_GROUPT * sizeof(V), "the groups' shares");
  const int64_t per = (items + c->nsm - 1) / c->nsm;
  if (per > P::MAXT) return KX_OK;
  const kx_status so = smem_opt_in(c, attr, fn, ROOM);
  if (so != KX_OK) return so;
  auto plan = [&](int nti) { return coop_plan(c, fn, items, nti, want, m, sizeof(V), P::NC, P::BATCH, ROOM); };
  // One block a SM, its threads an SM's share of the items (fewer, larger
  // blocks: half the partials and arrivals of two blocks a SM, 64^3 4.1 -> 3.8
  // ms): the shortest process.  A small grid's blocks then hold nearly every SM
  // and the slots of a lockstep batch would run one after the other, so where
  // they do not all fit at once, fuller blocks or the per-step launches, by the
  // estimates above.  They know the slots that may run (want, of every context
  // that the threaded driver runs beside this one), not those of one call: a
  // context's bits do not depend on how many still run.  plain, 32
  // frequencies, T = 60, one after the other / per-step launches / this rule:
  // 24^3 158 / 57 / 39 ms, 36^3 214 / 176 / 140, 30^3 in double precision 323 /
  // 284 / 274, 2D 64^2 in double precision 125 / 35 / 35.
  CoopPlan p = plan((int)((per + 31) / 32 * 32));
  if (p.slots > 0 && want > p.slots) {
    const int values = P::NC * (int)(sizeof(V) / sizeof(T));
    double best = coop_us(c, p, want, m, values);
    for (int nti = 64; nti <= std::min(CO_GROUPT, P::MAXT); nti += 64) {
      if (nti <= p.nti) continue;
      const CoopPlan f = plan(nti);
      const double us = f.slots > 0 ? coop_us(c, f, want, m, values) : best;
      if (us < best) {
        best = us;
        p = f;
      }
    }
    if (steps_us(c, want, m) < best) return KX_OK;
  }
  *ran = p.slots > 0;
  if (!*ran) return KX_OK;
  for (int q = 0; q < ns; q += p.slots) {
    const int nq = std::min(p.slots, ns - q);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.blocks, nq);
    cfg.blockDim = dim3(p.nti * p.groups);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = c->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const double vb = (double)c->n * c->esize;
    time_begin(c);
    const cudaError_t e =
        cudaLaunchKernelEx(&cfg, k_coop<P, AUG>, c->geo, make_slotset<T>(c, slot0 + q), m, c->ld,
                       (const T*)c->d_inv_eps, (const T*)c->d_sig2, (const T*)g_aug, c->m + 1,
                       sizeof(T) == 8 ? 1e-12 : 1e-6, p.nti, p.keep, c->wait_polls);
    // algorithmic bytes: per step v_j, V_0 .. V_{j-1} twice, v_{j+1}, 1/eps (and g)
    time_end(c, KX_K_PASS_A,
             nq * m * ((m + 2.0) * vb + (double)c->geo.ne * c->geo.ncell * c->esize + (g_aug ? vb : 0.0)));
    if (e == cudaErrorCooperativeLaunchTooLarge && q == 0) {
      // fewer multiprocessors than the device reports (a partition of it)
      cudaGetLastError();
      *ran = false;
      return KX_OK;
    }
    KX_CHECK_LAUNCH(c);
  }
  return KX_OK;
}

template <typename T, int AUG, int TR>
kx_status coop_model(kx_ctx* c, int slot0, int ns, int want, int m, const void* g_aug, bool* ran) {
  const Geo& g = c->geo;
  if (g.dim == 2 && g.pml) {
    if constexpr (TR) return KX_OK;   // the adjoint does not cover the PML model
    else return coop_run<CellItem<T, 4, AUG, 0>, AUG>(c, slot0, ns, want, m, g_aug, g.ncell, ran);
  }
  if (g.dim == 2) return coop_run<CellItem<T, 2, AUG, TR>, AUG>(c, slot0, ns, want, m, g_aug, g.ncell, ran);
  if constexpr (sizeof(T) == 4) {
    // the quads need 16-byte aligned rows of every array they read
    if (g.nx % 4 == 0 && (uintptr_t)g_aug % 16 == 0 && g.ncell < ((int64_t)1 << 31)) {
      // By the threads a block needs: up to 256 have 232 registers and four
      // columns in flight, up to 384 168 registers and still four (56^3, 64
      // steps: 2380 us, with two columns 2655; 60^3 2980 and 3132), above that
      // 128 registers and two (64^3: compiled for 448 threads 3655 us, for 512
      // 3748).
      const int64_t quads = g.ncell / 4, sm = c->nsm;
      if (quads <= sm * 256) return coop_run<QuadItem<AUG, TR, 256>, AUG>(c, slot0, ns, want, m, g_aug, quads, ran);
      if (quads <= sm * 384) return coop_run<QuadItem<AUG, TR, 384>, AUG>(c, slot0, ns, want, m, g_aug, quads, ran);
      if (quads <= sm * 448) return coop_run<QuadItem<AUG, TR, 448>, AUG>(c, slot0, ns, want, m, g_aug, quads, ran);
      return coop_run<QuadItem<AUG, TR, 512>, AUG>(c, slot0, ns, want, m, g_aug, quads, ran);
    }
  }
  return coop_run<CellItem<T, 3, AUG, TR>, AUG>(c, slot0, ns, want, m, g_aug, g.ncell, ran);
}

}  // namespace

kx_status coop_arnoldi(kx_ctx* c, int slot0, int ns, int want, int m, const void* g_aug, int transpose, bool* ran) {
  *ran = false;
  const bool f64 = c->d.precision == KX_FP64;
  if (transpose)
    return f64 ? coop_model<double, 0, 1>(c, slot0, ns, want, m, nullptr, ran)
               : coop_model<float, 0, 1>(c, slot0, ns, want, m, nullptr, ran);
  if (g_aug)
    return f64 ? coop_model<double, 1, 0>(c, slot0, ns, want, m, g_aug, ran)
               : coop_model<float, 1, 0>(c, slot0, ns, want, m, g_aug, ran);
  return f64 ? coop_model<double, 0, 0>(c, slot0, ns, want, m, nullptr, ran)
             : coop_model<float, 0, 0>(c, slot0, ns, want, m, nullptr, ran);
}

}  // namespace kx
