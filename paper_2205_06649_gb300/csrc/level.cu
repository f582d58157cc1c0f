// Level sweeps: the forward and adjoint sweeps of all subdomains advanced
// together, one launch per RK3 stage, with the states in HBM / L2.
//
// Design (GB300, sm_103a).  The cluster sweeps (sweep.cu) keep one box in one
// thread-block cluster for its whole window.  A box's stages are then a chain
// of cluster barriers with a few points per thread between them, clusters pack
// badly into GPCs, and neither the FP64 pipe (62-65 % of its rate over a sweep)
// nor HBM (7-12 %) is busy.  Where all boxes together have enough points per
// level, a stage of every box is one ordinary grid instead:
//   * FP64: 28-47 FP64 instructions per point take 16 SM cycles per warp each;
//     the 15-36 loads of a point are a tenth of that, so plain loads through L1
//     keep the FP64 pipe fed, and every SM works until the grid's end.  Bound:
//     the FP64 pipe, 83-88 % of its rate inside a launch of 2.9 million points
//     (profiles/level_sweeps_fp64.md), 57-58 % over the short launches of the medium
//     workload (14-28 us each, some 5 of them start, first loads and last tiles).
//   * FP32: a thread takes four neighbouring columns with 16-byte loads.  Bound:
//     latency of the loads (forward HBM at 55 % of its measured rate); groups of
//     boxes sized for L2, strips marching north with rows kept in registers, one
//     or two columns a thread at 1.7x the warps, and a whole step per launch with
//     rows in shared memory (11.9 / 17.9 ms for 9.6 / 17.6 of the batching
//     workload: 1.7x the instructions) all measured slower or equal.  The adjoint
//     of many tiles runs pipelined (lv_ring_adj_kernel).
// A tile is a run of points of one box (flat over rows, so that every lane has
// one); tiles are ordered longest window first, so the boxes still running at
// step l are a prefix and the grid shrinks with them.  CTAs of 128 threads: with
// 256 the last wave of a 175,000-point level leaves more of the SMs idle (FP64, 64
// boxes, forward / adjoint 1.93 / 2.43 ms, with 128 1.83 / 2.23; FP32, 645,000 points
// a level 1.75 / 3.32, with 128 1.73 / 3.20).  Launches overlap their set-up with the
// end of the launch before (programmatic dependent launch).
//
// Measured against the cluster sweeps with the launch shapes that the library
// chooses (forward / adjoint, ms):
//   batching workload (512 boxes, 3.9e8 points x steps), FP32: 15.8 / 30.7 ->
//     9.6 / 13.5; FP64: 102.8 / 156.7 -> 76.0 / 92.5 (a part of it from the FP64
//     adjoint's point function, without which the level sweeps took 77 / 112)
//   one 128-step window of the large workload (256 boxes), FP32: 15.4 / 29.6 -> 9.3 / 13.9
//   differentiation workload (FP32, 16-step checkpoints): 1.68 / 4.92 -> 1.73 / 3.20
//   medium workload (FP64, 64 boxes, 175,000 points): 1.86 / 2.32 -> 1.83 / 2.23
//
// The arithmetic per point is that of sweep.cu (point.cuh), so trajectories,
// stage states and gradients are the same bit for bit; J differs by the order
// of its partial sums.
#include "point.cuh"

#include <algorithm>
#include <cstdint>

namespace dd4dv {

namespace {

// The CTA's tile in shared memory: one coalesced load, and no registers held
// for the fields that only edges need.
#define LV_TILE(t)                                                                                    \
  __shared__ LvTile t;                                                                                \
  if (threadIdx.x < sizeof(LvTile) / 4)                                                               \
    reinterpret_cast<int*>(&t)[threadIdx.x] = reinterpret_cast<const int*>(a.tiles + blockIdx.x)[threadIdx.x]; \
  __syncthreads()
static_assert(sizeof(LvTile) % 4 == 0 && sizeof(LvTile) / 4 <= kLvThreads, "one word a thread");

// V consecutive values from / to global memory (aligned to V elements).
template <typename T, int V>
__device__ __forceinline__ void ldv(const T* p, T* x) {
  if constexpr (V == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    x[0] = q.x; x[1] = q.y; x[2] = q.z; x[3] = q.w;
  } else {
    x[0] = *p;
  }
}
template <typename T, int V>
__device__ __forceinline__ void stv(T* p, const T* x) {
  if constexpr (V == 4) *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
  else *p = x[0];
}

// A thread's V points (row r, columns k .. k + V - 1) of one buffer with the
// values around them: c[v][0] west of the first, c[v][V + 1] east of the last.
template <typename T, int V>
struct Patch {
  T c[3][V + 2], n[3][V], s[3][V];
};

template <typename T, int V>
__device__ __forceinline__ void point_of(const Patch<T, V>& z, int j, Pt5<T>& p) {
  p.h = z.c[0][j + 1]; p.u = z.c[1][j + 1]; p.v = z.c[2][j + 1];
  p.hE = z.c[0][j + 2]; p.uE = z.c[1][j + 2]; p.vE = z.c[2][j + 2];
  p.hW = z.c[0][j]; p.uW = z.c[1][j]; p.vW = z.c[2][j];
  p.hN = z.n[0][j]; p.uN = z.n[1][j]; p.vN = z.n[2][j];
  p.hS = z.s[0][j]; p.uS = z.s[1][j]; p.vS = z.s[2][j];
}

// Boundary-trajectory value at offset o of level B0, blended with half of
// level B1 where B1 is given (as bnd_val of sweep.cu).
template <typename T>
__device__ __forceinline__ T frozen(const T* B0, const T* B1, int o) {
  const T xa = B0[o];
  return B1 ? xfma((T)0.5, xa, xmul((T)0.5, B1[o])) : xa;
}

// The patch of a state buffer Y ([3][ny][nxp]) at element offset at = r nxp + k,
// ghosts by the box-edge rules: wall mirror (h, u, -v), periodic wrap, or the
// frozen boundary trajectory.  A box is wider than V, so a thread has at most
// one ghost column.
template <typename T, int V>
__device__ __forceinline__ void load_state_patch(const LvArgs<T>& a, const LvTile& t, const T* Y, int r, int k,
                                                 int at, const T* B0, const T* B1, Patch<T, V>& z) {
  const int pl = t.ny * t.nxp;
  const bool west = k == 0, east = k + V >= t.nx, north = r == t.ny - 1, south = r == 0;
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    const T* y = Y + (at + v * pl);
    ldv<T, V>(y, &z.c[v][1]);
    if (!west) z.c[v][0] = y[-1];
    if (!east) z.c[v][V + 1] = y[V];
    if (!north) ldv<T, V>(y + t.nxp, z.n[v]);
    if (!south) ldv<T, V>(y - t.nxp, z.s[v]);
  }
  if (west || east) {
    const bool per = t.flags & F_PERIODIC;
    const int pg = a.nlat * a.nlon;
    const int o = per ? r * t.nxp + (west ? t.nx - 1 : 0) : (t.j0 + r) * a.nlon + (west ? t.iw : t.ie);
    const T* src = (per ? Y : B0) + o;
    const int str = per ? pl : pg;
    T g[3];
#pragma unroll
    for (int v = 0; v < 3; ++v) g[v] = src[v * str];
    if (B1 && !per) {
#pragma unroll
      for (int v = 0; v < 3; ++v) g[v] = xfma((T)0.5, g[v], xmul((T)0.5, B1[o + v * pg]));
    }
    const int je = t.nx - k + 1;   // slot of column nx
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      if (west) z.c[v][0] = g[v];
#pragma unroll
      for (int j = 2; j < V + 2; ++j)
        if (east && j == je) z.c[v][j] = g[v];
    }
  }
  if (north || south) {
    const bool wall = t.flags & (north ? F_NWALL : F_SWALL);
    const int pg = a.nlat * a.nlon;
    const int row = (north ? t.j0 + t.ny : t.j0 - 1) * a.nlon;
#pragma unroll
    for (int j = 0; j < V; ++j) {
      int i = t.i0 + min(k + j, t.nx - 1);
      if (i >= a.nlon) i -= a.nlon;
      T g[3];
      if (wall) {
        g[0] = z.c[0][j + 1];
        g[1] = z.c[1][j + 1];
        g[2] = -z.c[2][j + 1];
      } else {
#pragma unroll
        for (int v = 0; v < 3; ++v) g[v] = frozen(B0, B1, row + v * pg + i);
      }
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        if (north) z.n[v][j] = g[v];
        else z.s[v][j] = g[v];
      }
    }
  }
}

// The patch of an adjoint buffer M: ghosts are zero but for the periodic wrap.
template <typename T, int V>
__device__ __forceinline__ void load_adjoint_patch(const LvTile& t, const T* M, int r, int k, int at,
                                                   Patch<T, V>& z) {
  const int pl = t.ny * t.nxp;
  const bool west = k == 0, east = k + V >= t.nx, north = r == t.ny - 1, south = r == 0;
  const bool per = t.flags & F_PERIODIC;
  const int je = t.nx - k + 1;
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    const T* y = M + (at + v * pl);
    ldv<T, V>(y, &z.c[v][1]);
    // periodic wrap: column -1 is nx - 1 of the row, column nx is 0
    z.c[v][0] = west ? (per ? y[t.nx - 1] : (T)0) : y[-1];
    const T e = east ? (per ? y[-k] : (T)0) : y[V];
    z.c[v][V + 1] = e;
#pragma unroll
    for (int j = 2; j < V + 1; ++j)
      if (east && j == je) z.c[v][j] = e;
#pragma unroll
    for (int j = 0; j < V; ++j) z.n[v][j] = z.s[v][j] = (T)0;
    if (!north) ldv<T, V>(y + t.nxp, z.n[v]);
    if (!south) ldv<T, V>(y - t.nxp, z.s[v]);
  }
}

template <typename T>
__device__ __forceinline__ size_t level_size(const LvTile& t) {
  return (size_t)3 * t.ny * t.nxp;
}
// Where the stage states of step l live: the stage buffer, the x1-only buffer
// of the subdomains that have one, or the one-level scratch.
template <typename T>
__device__ __forceinline__ T* x1_of(const LvArgs<T>& a, const LvTile& t, int l) {
  if (a.stg) return a.stg + t.stg_off + (size_t)2 * l * level_size<T>(t);
  if (a.stg1 && t.stg1_off >= 0) return a.stg1 + t.stg1_off + (size_t)l * level_size<T>(t);
  return a.x1s + t.lv_off;
}
template <typename T>
__device__ __forceinline__ T* x2_of(const LvArgs<T>& a, const LvTile& t, int l) {
  if (a.stg) return a.stg + t.stg_off + (size_t)(2 * l + 1) * level_size<T>(t);
  return a.x2s + t.lv_off;
}

__device__ __forceinline__ int lv_overlap_count(const LvTile& t, int l, int r, int k) {
  const int cx = 1 + (k < t.wL) + (k >= t.nx - t.wR);
  const int cy = 1 + (r < t.wS) + (r >= t.ny - t.wN);
  const int ct = 1 + (l < t.tA) + (l > t.L - t.tB);
  return cx * cy * ct - 1;
}
__device__ __forceinline__ bool lv_overlaps(const LvTile& t, int l) {
  return (l < t.tA) || (l > t.L - t.tB) || t.wL || t.wR || t.wS || t.wN;
}

// Sum of the block's values (fixed order), on thread 0.
__device__ __forceinline__ double lv_block_sum(double x, double* sh) {
  sh[threadIdx.x] = x;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
    for (int i = threadIdx.x; i < (int)blockDim.x; i += 32) s += sh[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  }
  return s;
}

// Observation misfits of one box at level l (one CTA): obs_force, and J_o
// added to the box's accumulator.
template <typename T>
__device__ void lv_obs(const LvArgs<T>& a, int s, int l, double* sh) {
  const SubDesc& d = a.subs[s];
  const int o0 = a.lvl_obs[d.obs_lvl + l], o1 = a.lvl_obs[d.obs_lvl + l + 1];
  if (o0 == o1) return;
  const int nxp = d.nxp;
  const size_t pl = (size_t)d.ny * nxp;
  const T* X = a.traj + d.traj_off + (size_t)l * 3 * pl;
  double Jo = 0.0;
  for (int o = o0 + threadIdx.x; o < o1; o += blockDim.x) {
    const ObsRec ob = a.obs[o];
    const T* x = X + ob.var * pl + (size_t)ob.r0 * nxp;
    const double x00 = (double)x[ob.k0];
    const double x01 = ob.di != 0.0 ? (double)x[ob.k1] : 0.0;
    const double x10 = ob.dj != 0.0 ? (double)x[nxp + ob.k0] : 0.0;
    const double x11 = (ob.dj != 0.0 && ob.di != 0.0) ? (double)x[nxp + ob.k1] : 0.0;
    a.obs_force[o] = obs_term(ob, x00, x01, x10, x11, a.lam_w, Jo);
  }
  Jo = lv_block_sum(Jo, sh);
  if (threadIdx.x == 0) a.acc_o[s] += Jo;
}

// Sum of FP32 terms without the rounding of its additions (TwoSum), so that
// the order of the points does not show in J; FP64 terms are added directly.
template <typename T>
struct Sum {
  T s = (T)0, e = (T)0;
  __device__ __forceinline__ void add(T x) {
    if constexpr (sizeof(T) == 4) {
      const float t = __fadd_rn(s, x), b = __fsub_rn(t, s);
      e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b)));
      s = t;
    } else {
      s += x;
    }
  }
  __device__ __forceinline__ double value() const { return sizeof(T) == 4 ? (double)s + (double)e : (double)s; }
};

// c sum_v (x_v - m_v)^2 / sigma_v^2 of one point (overlap_term of sweep.cu).
template <typename T>
__device__ __forceinline__ void overlap_add(Sum<T>& part, int c, T x0, T x1, T x2, T m0, T m1, T m2,
                                            const T (&isb2)[3]) {
  const T e0 = xsub(x0, m0), e1 = xsub(x1, m1), e2 = xsub(x2, m2);
  T sq = xmul(xmul(e0, e0), isb2[0]);
  sq = xfma(xmul(e1, e1), isb2[1], sq);
  sq = xfma(xmul(e2, e2), isb2[2], sq);
  if constexpr (sizeof(T) == 4) {
    const float p = xmul((float)c, sq);
    part.add(p);
    part.e = __fadd_rn(part.e, xfma((float)c, sq, -p));
  } else {
    part.s = xfma((T)c, sq, part.s);
  }
}

// Twice the overlap misfit of a thread's V points at level l (the terms of
// overlap_level of sweep.cu).
template <typename T, int V>
__device__ __forceinline__ void lv_overlap_part(const LvArgs<T>& a, const LvTile& t, const T* tg, int l, int r, int k,
                                                int at, const T (*o)[V], Sum<T>& part) {
  const int pl = t.ny * t.nxp;
  int c[V], any = 0;
#pragma unroll
  for (int j = 0; j < V; ++j) {
    c[j] = k + j < t.nx ? lv_overlap_count(t, l, r, k + j) : 0;
    any |= c[j];
  }
  if (!any) return;
  T m[3][V];
#pragma unroll
  for (int v = 0; v < 3; ++v) ldv<T, V>(tg + (at + v * pl), m[v]);
#pragma unroll
  for (int j = 0; j < V; ++j)
    if (c[j]) overlap_add(part, c[j], o[0][j], o[1][j], o[2][j], m[0][j], m[1][j], m[2][j], a.isb2);
}

// Terms of level 0 (the initial states): starts the accumulators of J.
template <typename T, int V>
__global__ void __launch_bounds__(kLvThreads) lv_start_kernel(const LvArgs<T> a) {
  LV_TILE(t);
  grid_wait();
  grid_release();
  if (a.active && a.active[t.s] != a.active_value) return;
  Sum<T> part;
  if (lv_overlaps(t, 0)) {
    const T* X = a.traj + t.traj_off;
    const int pl = t.ny * t.nxp;
    for (int p = t.p0 + threadIdx.x; p < t.p1; p += kLvThreads) {
      const int r = mdiv(p, t.mq), k = (p - r * t.nq) * V, at = r * t.nxp + k;
      T o[3][V];
#pragma unroll
      for (int v = 0; v < 3; ++v) ldv<T, V>(X + (at + v * pl), o[v]);
      lv_overlap_part<T, V>(a, t, a.tgt + t.traj_off, 0, r, k, at, o, part);
    }
  }
  a.acc_m[(size_t)blockIdx.x * kLvThreads + threadIdx.x] = part.value();
  if (t.p0 == 0 && threadIdx.x == 0) a.acc_o[t.s] = 0.0;
}

// RK3 stage ST of step l: out = cx X + cy (Y + dt F(Y)) of every tile.  The
// first stage's grid carries one more CTA per box of a.boxes for the
// observations of level l; with TERMS, the third stage adds level l + 1's
// overlap misfit.  skip1: leave the boxes out whose x1 is stored (first stage
// recomputed for the adjoint).
template <typename T, int V, int ST, bool TERMS>
__global__ void __launch_bounds__(kLvThreads, 6) lv_stage_kernel(const LvArgs<T> a) {
  constexpr bool DEV = sizeof(T) == 4;
  __shared__ double sh[ST == 1 ? kLvThreads : 1];
  const int l = a.l;
  if (ST == 1 && (int)blockIdx.x >= a.n_tile) {
    const int s = a.boxes[blockIdx.x - a.n_tile];
    grid_wait();
    grid_release();
    if (a.active && a.active[s] != a.active_value) return;
    lv_obs(a, s, l, sh);
    return;
  }
  LV_TILE(t);
  grid_wait();
  grid_release();
  if (a.active && a.active[t.s] != a.active_value) return;
  if (ST == 1 && a.skip1 && t.stg1_off >= 0) return;
  const size_t lvl = level_size<T>(t);
  const int pl = t.ny * t.nxp;
  const T* X = a.traj + t.traj_off + (size_t)l * lvl;
  const T* Y = ST == 1 ? X : ST == 2 ? x1_of(a, t, l) : x2_of(a, t, l);
  T* out = ST == 1 ? x1_of(a, t, l) : ST == 2 ? x2_of(a, t, l) : a.traj + t.traj_off + (size_t)(l + 1) * lvl;
  const size_t G = (size_t)3 * a.nlat * a.nlon;
  const int n = t.a + l;
  const T* B0 = a.bnd + (size_t)(ST == 2 ? n + 1 : n) * G;
  const T* B1 = ST == 3 ? B0 + G : nullptr;
  const T cx = ST == 1 ? (T)0 : ST == 2 ? (T)0.75 : (T)(1.0 / 3.0);
  const T cy = ST == 1 ? (T)1 : ST == 2 ? (T)0.25 : (T)(2.0 / 3.0);
  const bool ovl = TERMS && lv_overlaps(t, l + 1);
  const size_t slot = (size_t)blockIdx.x * kLvThreads + threadIdx.x;
  double acc = 0.0;
  if (ovl) acc = a.acc_m[slot];
  Sum<T> part;
  for (int p = t.p0 + threadIdx.x; p < t.p1; p += kLvThreads) {
    const int r = mdiv(p, t.mq), k = (p - r * t.nq) * V, at = r * t.nxp + k;
    Patch<T, V> z;
    load_state_patch<T, V>(a, t, Y, r, k, at, B0, B1, z);
    T x[3][V];
    if (ST != 1) {
#pragma unroll
      for (int v = 0; v < 3; ++v) ldv<T, V>(X + (at + v * pl), x[v]);
    }
    T rc[8];
    load_rec8(a.fw + 8 * (t.j0 + r), rc);
    T o[3][V];
#pragma unroll
    for (int j = 0; j < V; ++j) {
      Pt5<T> y;
      point_of(z, j, y);
      stage_math<T, DEV>(y, rc, a.dt, a.Bth, a.gBth, a.href, cx, cy, ST != 1 ? x[0][j] : (T)0,
                         ST != 1 ? x[1][j] : (T)0, ST != 1 ? x[2][j] : (T)0, o[0][j], o[1][j], o[2][j]);
    }
#pragma unroll
    for (int v = 0; v < 3; ++v) stv<T, V>(out + (at + v * pl), o[v]);
    if (ovl) lv_overlap_part<T, V>(a, t, a.tgt + t.traj_off + (size_t)(l + 1) * lvl, l + 1, r, k, at, o, part);
  }
  if (ovl) a.acc_m[slot] = acc + part.value();
}

// Overlap forcing of point j: mu c (x - m) / sigma^2, or for a Gauss-Newton
// product (m = dx) mu c dx / sigma^2 (the arithmetic of add_forcing and
// overlap_force in sweep.cu).
template <typename T, int V>
__device__ __forceinline__ void overlap_force_add(const LvArgs<T>& a, int c, int j, const T (*x)[V], const T (*m)[V],
                                                  T (*o)[V]) {
  const T cc = (T)c;
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    if (a.gn_dx) o[v][j] = o[v][j] + cc * a.musb2[v] * m[v][j];
    else o[v][j] = xfma(xmul(cc, a.musb2[v]), xsub(x[v][j], m[v][j]), o[v][j]);
  }
}

// The forcing of one thread's V points at level l that comes before the
// observations: external forcing, the Gauss-Newton overlap term or the overlap
// term.
template <typename T, int V>
__device__ __forceinline__ void lv_force(const LvArgs<T>& a, const LvTile& t, int l, int r, int k, const T (*x)[V],
                                         T (*o)[V]) {
  const size_t pl = (size_t)t.ny * t.nxp, lvl = level_size<T>(t);
  if (a.yforce) {
    const double* y = a.yforce + t.ptraj_off + (size_t)l * 3 * t.ny * t.nx;
#pragma unroll
    for (int j = 0; j < V; ++j)
      if (k + j < t.nx)
#pragma unroll
        for (int v = 0; v < 3; ++v) o[v][j] += (T)y[((size_t)v * t.ny + r) * t.nx + k + j];
    return;
  }
  if (!a.mu_on || !lv_overlaps(t, l)) return;
  int c[V], any = 0;
#pragma unroll
  for (int j = 0; j < V; ++j) {
    c[j] = k + j < t.nx ? lv_overlap_count(t, l, r, k + j) : 0;
    any |= c[j];
  }
  if (!any) return;
  const T* q = (a.gn_dx ? a.gn_dx : a.tgt) + t.traj_off + (size_t)l * lvl + (size_t)r * t.nxp + k;
  T m[3][V];
#pragma unroll
  for (int v = 0; v < 3; ++v) ldv<T, V>(q + v * pl, m[v]);
#pragma unroll
  for (int j = 0; j < V; ++j) {
    if (!c[j]) continue;
    overlap_force_add<T, V>(a, c[j], j, x, m, o);
  }
}

// Observation forcing H^T (lambda w d) of level l at the points for which
// mine(r, k) holds, added to the adjoint state (fixed order per target).
template <typename T, typename F>
__device__ __forceinline__ void lv_scatter_if(const LvArgs<T>& a, const LvTile& t, int l, T* lam, F&& mine) {
  if (a.yforce) return;
  const int t0 = a.lvl_sc[t.sc_lvl + l], t1 = a.lvl_sc[t.sc_lvl + l + 1];
  if (t0 == t1) return;
  __syncthreads();
  const int pl = t.ny * t.nxp;
  for (int i = t0 + threadIdx.x; i < t1; i += blockDim.x) {
    const int g = a.sc_tgt[i];
    const int vr = mdiv(g, t.mnx);   // v * ny + r
    const int v = mdiv(vr, t.mny);
    const int r = vr - v * t.ny, k = g - vr * t.nx;
    if (!mine(r, k)) continue;
    double acc = 0.0;
    for (int c = a.sc_off[i]; c < a.sc_off[i + 1]; ++c) acc += a.sc_w[c] * a.obs_force[a.sc_obs[c]];
    lam[v * pl + r * t.nxp + k] += (T)acc;
  }
}
template <typename T, int V>
__device__ __forceinline__ void lv_scatter(const LvArgs<T>& a, const LvTile& t, int l, T* lam) {
  lv_scatter_if(a, t, l, lam, [&](int r, int k) {
    const int p = r * t.nq + k / V;
    return p >= t.p0 && p < t.p1;
  });
}

// lambda(b) = forcing(b) of every tile, each box at its own last level.
template <typename T, int V>
__global__ void __launch_bounds__(kLvThreads) lv_lam_start_kernel(const LvArgs<T> a) {
  LV_TILE(t);
  grid_wait();
  grid_release();
  if (a.active && a.active[t.s] != a.active_value) return;
  const size_t lvl = level_size<T>(t);
  const int pl = t.ny * t.nxp;
  const T* X = a.traj + t.traj_off + (size_t)t.L * lvl;
  T* lam = a.lam + t.lv_off;
  for (int p = t.p0 + threadIdx.x; p < t.p1; p += kLvThreads) {
    const int r = mdiv(p, t.mq), k = (p - r * t.nq) * V, at = r * t.nxp + k;
    T x[3][V], o[3][V];
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      ldv<T, V>(X + v * pl + at, x[v]);
#pragma unroll
      for (int j = 0; j < V; ++j) o[v][j] = (T)0;
    }
    lv_force<T, V>(a, t, t.L, r, k, x, o);
#pragma unroll
    for (int v = 0; v < 3; ++v) stv<T, V>(lam + v * pl + at, o[v]);
  }
  lv_scatter<T, V>(a, t, t.L, lam);
}

// Phase K of the transposed RK3 step l (rescaled stage adjoints as in
// adj_kernel of sweep.cu):
//   K = 1: mu2 = lambda' + dt F'(x2)^T lambda'
//   K = 2: mu1 = mu2 + dt F'(x1)^T mu2
//   K = 3: lambda(n) = lambda'/3 + mu2/2 + (mu1 + dt F'(x)^T mu1)/6 + forcing(n)
template <typename T, int V, int K>
__global__ void __launch_bounds__(kLvThreads, 4) lv_adj_kernel(const LvArgs<T> a) {
  constexpr bool DEV = sizeof(T) == 4;
  LV_TILE(t);
  grid_wait();
  grid_release();
  if (a.active && a.active[t.s] != a.active_value) return;
  const int l = a.l;
  const size_t lvl = level_size<T>(t);
  const int pl = t.ny * t.nxp;
  const T* Z = K == 1 ? x2_of(a, t, l) : K == 2 ? x1_of(a, t, l) : a.traj + t.traj_off + (size_t)l * lvl;
  const T* M = (K == 1 ? a.lam : K == 2 ? a.mu2 : a.mu1) + t.lv_off;
  T* out = (K == 1 ? a.mu2 : K == 2 ? a.mu1 : a.lam) + t.lv_off;
  const size_t G = (size_t)3 * a.nlat * a.nlon;
  const int n = t.a + l;
  const T* B0 = a.bnd + (size_t)(K == 2 ? n + 1 : n) * G;
  const T* B1 = K == 1 ? B0 + G : nullptr;
  for (int p = t.p0 + threadIdx.x; p < t.p1; p += kLvThreads) {
    const int r = mdiv(p, t.mq), k = (p - r * t.nq) * V, at = r * t.nxp + k;
    Patch<T, V> z, m;
    load_state_patch<T, V>(a, t, Z, r, k, at, B0, B1, z);
    load_adjoint_patch<T, V>(t, M, r, k, at, m);
    T rc[8];
    load_rec8(a.bw + 8 * (t.j0 + r), rc);
    const int wall = (r == 0 && (t.flags & F_SWALL) ? 1 : 0) | (r == t.ny - 1 && (t.flags & F_NWALL) ? 2 : 0);
    T o[3][V], ll[3][V], l2[3][V];
    if (K == 3) {
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        ldv<T, V>(out + (at + v * pl), ll[v]);
        ldv<T, V>(a.mu2 + t.lv_off + (at + v * pl), l2[v]);
      }
    }
#pragma unroll
    for (int j = 0; j < V; ++j) {
      Pt5<T> zp, mp;
      point_of(z, j, zp);
      point_of(m, j, mp);
      if (K == 3)
        adj_lambda_math<T, DEV>(zp, mp, rc, a.dt, a.Bth_a, a.gBth_a, a.href, wall, ll[0][j], ll[1][j], ll[2][j],
                                l2[0][j], l2[1][j], l2[2][j], o[0][j], o[1][j], o[2][j]);
      else
        adj_stage_math<T, DEV>(zp, mp, rc, a.dt, a.Bth_a, a.gBth_a, a.href, wall, o[0][j], o[1][j], o[2][j]);
    }
    if (K == 3) {
      T x[3][V];
#pragma unroll
      for (int v = 0; v < 3; ++v)
#pragma unroll
        for (int j = 0; j < V; ++j) x[v][j] = z.c[v][j + 1];
      lv_force<T, V>(a, t, l, r, k, x, o);
    }
#pragma unroll
    for (int v = 0; v < 3; ++v) stv<T, V>(out + (at + v * pl), o[v]);
  }
  if (K == 3) lv_scatter<T, V>(a, t, l, out);
}

// ---- tangent-linear sweep of a Gauss-Newton product ----
// About the trajectory (and the stage states, where they are stored) of the
// last forward sweep: dx of every level to a.dx, the linear observations of
// every level to obs_force.  FP64 only: the FP32 sweep (tlm_kernel of sweep.cu)
// leaves the contraction of its arithmetic to the compiler, and its FP32
// roundings show in a product.  Bound: the FP64 pipe (some 55 instructions a
// point and stage).  Medium workload (64 boxes): 3.1 ms by clusters, 2.5 here (a
// product 7.55 -> 6.95 ms).
__device__ __forceinline__ void lv_obs_lin(const LvArgs<double>& a, int s, int l) {
  const SubDesc& d = a.subs[s];
  const int o0 = a.lvl_obs[d.obs_lvl + l], o1 = a.lvl_obs[d.obs_lvl + l + 1];
  const size_t pl = (size_t)d.ny * d.nxp;
  const double* X = a.dx + d.traj_off + (size_t)l * 3 * pl;
  for (int o = o0 + threadIdx.x; o < o1; o += blockDim.x) {
    const ObsRec ob = a.obs[o];
    const double* x = X + ob.var * pl + (size_t)ob.r0 * d.nxp;
    const double wj0 = 1.0 - ob.dj, wi0 = 1.0 - ob.di;
    double acc = (wj0 * wi0) * x[ob.k0];
    if (ob.di != 0.0) acc += (wj0 * ob.di) * x[ob.k1];
    if (ob.dj != 0.0) {
      acc += (ob.dj * wi0) * x[d.nxp + ob.k0];
      if (ob.di != 0.0) acc += (ob.dj * ob.di) * x[d.nxp + ob.k1];
    }
    a.obs_force[o] = a.lam_w * ob.w * acc;
  }
}
__global__ void __launch_bounds__(kLvThreads) lv_tl_start_kernel(const LvArgs<double> a) {
  LV_TILE(t);
  grid_wait();
  grid_release();
  if (a.active && a.active[t.s] != a.active_value) return;
  const int pl = t.ny * t.nxp;
  const double* src = a.dx0 + t.ctrl_off;
  double* D = a.dx + t.traj_off;
  for (int p = t.p0 + threadIdx.x; p < t.p1; p += kLvThreads) {
    const int r = mdiv(p, t.mq), k = p - r * t.nq, at = r * t.nxp + k;
#pragma unroll
    for (int v = 0; v < 3; ++v) D[at + v * pl] = src[((size_t)v * t.ny + r) * t.nx + k];
  }
}
// Stage ST of step l: out = cx dX + cy (dY + dt F'(Y) dY).  The first stage's
// grid carries the observations of level l as lv_stage_kernel does.
template <int ST>
__global__ void __launch_bounds__(kLvThreads, 4) lv_tl_kernel(const LvArgs<double> a) {
  const int l = a.l;
  if (ST == 1 && (int)blockIdx.x >= a.n_tile) {
    const int s = a.boxes[blockIdx.x - a.n_tile];
    grid_wait();
    grid_release();
    if (a.active && a.active[s] != a.active_value) return;
    lv_obs_lin(a, s, l);
    return;
  }
  LV_TILE(t);
  grid_wait();
  grid_release();
  if (a.active && a.active[t.s] != a.active_value) return;
  const size_t lvl = level_size<double>(t);
  const int pl = t.ny * t.nxp;
  const double* Y = ST == 1 ? a.traj + t.traj_off + (size_t)l * lvl : ST == 2 ? x1_of(a, t, l) : x2_of(a, t, l);
  const double* DX = a.dx + t.traj_off + (size_t)l * lvl;
  const double* DY = ST == 1 ? DX : (ST == 2 ? a.mu2 : a.mu1) + t.lv_off;
  double* out = ST == 3 ? a.dx + t.traj_off + (size_t)(l + 1) * lvl : (ST == 1 ? a.mu2 : a.mu1) + t.lv_off;
  const size_t G = (size_t)3 * a.nlat * a.nlon;
  const int n = t.a + l;
  const double* B0 = a.bnd + (size_t)(ST == 2 ? n + 1 : n) * G;
  const double* B1 = ST == 3 ? B0 + G : nullptr;
  const double cx = ST == 1 ? 0.0 : ST == 2 ? 0.75 : 1.0 / 3.0, cy = ST == 1 ? 1.0 : ST == 2 ? 0.25 : 2.0 / 3.0;
  for (int p = t.p0 + threadIdx.x; p < t.p1; p += kLvThreads) {
    const int r = mdiv(p, t.mq), k = p - r * t.nq, at = r * t.nxp + k;
    Patch<double, 1> z, d;
    load_state_patch<double, 1>(a, t, Y, r, k, at, B0, B1, z);
    load_adjoint_patch<double, 1>(t, DY, r, k, at, d);   // ghosts zero or periodic ...
    double rc[8];
    load_rec8(a.fw + 8 * (t.j0 + r), rc);
    double x[3];
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      x[v] = ST == 1 ? 0.0 : DX[at + v * pl];
      const double m = v == 2 ? -d.c[v][1] : d.c[v][1];   // ... but mirrored at walls
      if (r == 0 && (t.flags & F_SWALL)) d.s[v][0] = m;
      if (r == t.ny - 1 && (t.flags & F_NWALL)) d.n[v][0] = m;
    }
    Pt5<double> zp, dp;
    point_of(z, 0, zp);
    point_of(d, 0, dp);
    double Fh, Fu, Fv;
    rhs_tl_pt<double, false>(zp, dp, rc[0], rc[1], rc[2], rc[3], rc[4], rc[5], rc[6], a.Bth, a.gBth, a.href, Fh, Fu,
                             Fv);
    out[at] = cx * x[0] + cy * (dp.h + a.dt * Fh);
    out[at + pl] = cx * x[1] + cy * (dp.u + a.dt * Fu);
    out[at + 2 * pl] = cx * x[2] + cy * (dp.v + a.dt * Fv);
  }
}

// lambda(a) -> packed control layout (FP64); NaN where a pipelined phase of this
// sweep lost a copy, so that no caller takes the gradient for one.
template <typename T, int V>
__global__ void __launch_bounds__(kLvThreads) lv_export_kernel(const LvArgs<T> a) {
  LV_TILE(t);
  grid_wait();
  grid_release();
  if (a.active && a.active[t.s] != a.active_value) return;
  const bool lost = sizeof(T) == 4 && *a.err == kErrLostCopy;
  const size_t pl = (size_t)t.ny * t.nxp;
  const T* lam = a.lam + t.lv_off;
  double* out = a.lam_a + t.ctrl_off;
  for (int p = t.p0 + threadIdx.x; p < t.p1; p += kLvThreads) {
    const int r = mdiv(p, t.mq), k = (p - r * t.nq) * V;
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      T x[V];
      ldv<T, V>(lam + v * pl + (size_t)r * t.nxp + k, x);
#pragma unroll
      for (int j = 0; j < V; ++j)
        if (k + j < t.nx) out[((size_t)v * t.ny + r) * t.nx + k + j] = lost ? __longlong_as_double(-1LL) : (double)x[j];
    }
  }
}

// ---- pipelined adjoint phases (FP32) ----
// lv_adj_kernel holds its 30 loads in registers, a few at a time, and waits for
// each batch (120 registers, 16 warps an SM, 7.9 of 12.5 cycles an instruction
// spent waiting for memory, HBM at 30-39 % of its rate).  Here CTAs stay and
// take tile after tile of whole rows (one thread-point for each of 224
// threads), and a warp of its own copies the states of the tiles ahead into a
// ring of slots in shared memory: bulk copies for the rows and their constants,
// 4-byte copies for the ghosts, one barrier a slot, no barrier between the
// computing warps.  What is in flight no longer depends on the registers.
// Bound: instruction issue (44-48 % of the slots, 550 to 600 instructions for a warp's
// 128 points in phases 1 and 2) and the wait for a slot.  Phase 3 takes 128 registers
// a thread and spills 56 bytes.  Phases 1, 2, 3 of 2.9 million points: 40.6, 39.5,
// 63.8 -> 30.9, 27.8, 52.0 us; adjoint sweep of the batching
// workload 17.6 -> 13.5 ms, of a 128-step window of the large workload 17.7 ->
// 13.9 ms.  With the copies made by a computing warp and a CTA barrier a tile
// the same sweep took 16.7 ms; the row constants read through L1 (small beside
// the slots) cost another 3 %.  The forward stages, which hold half as much in
// registers, gained nothing from it (9.6 -> 12.3 ms) and stay plain.
constexpr int kRingWait = 1 << 20;   // polls before a copy counts as lost
constexpr int kDescs = 8;            // tile descriptors in shared memory
constexpr int kRingSlots = 4;        // at most

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ring_copy(void* dst, const void* src, int bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ void copy4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
template <int POLLS>
__device__ __forceinline__ bool ring_wait(uint64_t* bar, unsigned parity) {
  for (int i = 0; i < POLLS; ++i) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// A copy did not arrive in time: the result is not valid.  The export kernel then
// writes NaN for it, and the host reports it.
__device__ __noinline__ void ring_lost(int* err, int* late) {
  atomicExch(err, kErrLostCopy);
  *(volatile int*)late = kErrLostCopy;
  __threadfence_system();
}

// A slot: NF states with a ghost row on either side, NO states without, with
// BL (ghosts blended from two boundary levels) the second level's rows beyond
// the box, the rows' constants, and the ghost columns [level][side][v][row].
template <int NF, int NO, bool BL>
struct Slot {
  float* base;
  int R, nxp;
  __device__ __forceinline__ int full() const { return (R + 2) * nxp; }   // plane of a state with ghost rows
  __device__ __forceinline__ int own() const { return R * nxp; }
  __device__ __forceinline__ float* state(int i) const {
    return base + (i < NF ? 3 * i * full() : 3 * NF * full() + 3 * (i - NF) * own());
  }
  __device__ __forceinline__ float* rows2() const { return base + 3 * NF * full() + 3 * NO * own(); }
  __device__ __forceinline__ float* rec() const { return rows2() + (BL ? 6 * nxp : 0); }   // row constants
  __device__ __forceinline__ float* cols() const { return rec() + 8 * R; }
};
template <int NF, int NO, bool BL>
__device__ __forceinline__ Slot<NF, NO, BL> slot_of(const LvTile& t, float* base) {
  return Slot<NF, NO, BL>{base, mdiv(t.p1 - t.p0, t.mq), t.nxp};
}

// Starts the copies of tile t (one warp): src(i) is state i, B0 (B1 = B0 + G
// with BL) the boundary level of the first state's ghosts.
template <int NF, int NO, bool BL, typename S>
__device__ __forceinline__ void ring_issue(const LvArgs<float>& a, const LvTile& t, float* base, uint64_t* bar,
                                           bool skip, const float* rec, const float* B0, S&& src) {
  const int lane = threadIdx.x & 31;
  const Slot<NF, NO, BL> sl = slot_of<NF, NO, BL>(t, base);
  const int r0 = mdiv(t.p0, t.mq), r1 = r0 + sl.R, ra = max(r0 - 1, 0), rb = min(r1 + 1, t.ny);
  const int bf = (rb - ra) * t.nxp * 4, bo = sl.R * t.nxp * 4, pl = t.ny * t.nxp;
  if (lane == 0) {
    const int tx = skip ? 0 : 3 * (NF * bf + NO * bo) + 32 * sl.R;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(tx) : "memory");
  }
  __syncwarp();
  if (!skip) {
    if (lane < 3 * (NF + NO)) {
      const int i = lane / 3, v = lane - 3 * i;
      const float* s = src(i) + v * pl;
      if (i < NF) ring_copy(sl.state(i) + v * sl.full() + (ra - r0 + 1) * t.nxp, s + ra * t.nxp, bf, bar);
      else ring_copy(sl.state(i) + v * sl.own(), s + r0 * t.nxp, bo, bar);
    } else if (lane == 31) {
      ring_copy(sl.rec(), rec + 8 * (t.j0 + r0), 32 * sl.R, bar);
    }
    const int pg = a.nlat * a.nlon, G = 3 * pg;
    if (!(t.flags & F_PERIODIC)) {
      float* g = sl.cols();
      for (int r = lane; r < sl.R; r += 32) {
        const float* b = B0 + (t.j0 + r0 + r) * a.nlon;
#pragma unroll
        for (int v = 0; v < 3; ++v) {
          copy4(g + v * sl.R + r, b + v * pg + t.iw);
          copy4(g + (3 + v) * sl.R + r, b + v * pg + t.ie);
          if (BL) {
            copy4(g + (6 + v) * sl.R + r, b + G + v * pg + t.iw);
            copy4(g + (9 + v) * sl.R + r, b + G + v * pg + t.ie);
          }
        }
      }
    }
#pragma unroll
    for (int side = 0; side < 2; ++side) {   // rows beyond the box
      if (side ? r1 < t.ny : r0 > 0) continue;
      if (t.flags & (side ? F_NWALL : F_SWALL)) continue;
      const float* b = B0 + (t.j0 + (side ? t.ny : -1)) * a.nlon;
      float* d = sl.state(0) + (side ? sl.R + 1 : 0) * t.nxp;
      for (int k = lane; k < t.nx; k += 32) {
        int i = t.i0 + k;
        if (i >= a.nlon) i -= a.nlon;
#pragma unroll
        for (int v = 0; v < 3; ++v) {
          copy4(d + v * sl.full() + k, b + v * pg + i);
          if (BL) copy4(sl.rows2() + (3 * side + v) * t.nxp + k, b + G + v * pg + i);
        }
      }
    }
  }
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// The patch of the state in slot sl, ghosts as in load_state_patch.
template <int NF, int NO, bool BL>
__device__ __forceinline__ void ring_state(const LvTile& t, const Slot<NF, NO, BL>& sl, int rr, int r, int k,
                                           Patch<float, 4>& z) {
  const bool west = k == 0, east = k + 4 >= t.nx, north = r == t.ny - 1, south = r == 0;
  const bool per = t.flags & F_PERIODIC;
  const float* y = sl.state(0) + (rr + 1) * t.nxp + k;
  const float *w = y - 1, *e = y + 4;
  int sw = sl.full(), se = sw;
  if (west) {
    w = per ? y + t.nx - 1 : sl.cols() + rr;
    sw = per ? sw : sl.R;
  }
  if (east) {
    e = per ? y - k : sl.cols() + 3 * sl.R + rr;
    se = per ? se : sl.R;
  }
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    ldv<float, 4>(y + v * sl.full(), &z.c[v][1]);
    z.c[v][0] = w[v * sw];
    z.c[v][5] = e[v * se];
    ldv<float, 4>(y + v * sl.full() + t.nxp, z.n[v]);
    ldv<float, 4>(y + v * sl.full() - t.nxp, z.s[v]);
  }
  if (BL && !per && (west || east)) {
    const float* g = sl.cols() + (west ? 6 : 9) * sl.R + rr;
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      const float b = xfma(0.5f, west ? z.c[v][0] : z.c[v][5], xmul(0.5f, g[v * sl.R]));
      if (west) z.c[v][0] = b;
      else z.c[v][5] = b;
    }
  }
  if (east) {   // column nx inside the four columns
    const int je = t.nx - k + 1;
#pragma unroll
    for (int v = 0; v < 3; ++v)
#pragma unroll
      for (int j = 2; j < 5; ++j)
        if (j == je) z.c[v][j] = z.c[v][5];
  }
  if (north || south) {
    const bool wall = t.flags & (north ? F_NWALL : F_SWALL);
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      float g[4];
      if (BL && !wall) ldv<float, 4>(sl.rows2() + (north ? 3 + v : v) * t.nxp + k, g);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float x = north ? z.n[v][j] : z.s[v][j];
        if (wall) x = v == 2 ? -z.c[v][j + 1] : z.c[v][j + 1];
        else if (BL) x = xfma(0.5f, x, xmul(0.5f, g[j]));
        if (north) z.n[v][j] = x;
        else z.s[v][j] = x;
      }
    }
  }
}
// The patch of the adjoint state in slot sl, ghosts as in load_adjoint_patch.
template <int NF, int NO, bool BL>
__device__ __forceinline__ void ring_adjoint(const LvTile& t, const Slot<NF, NO, BL>& sl, int rr, int r, int k,
                                             Patch<float, 4>& z) {
  const bool west = k == 0, east = k + 4 >= t.nx, north = r == t.ny - 1, south = r == 0;
  const bool per = t.flags & F_PERIODIC;
  const float* y = sl.state(1) + (rr + 1) * t.nxp + k;
  const float* w = west ? y + t.nx - 1 : y - 1;
  const float* e = east ? y - k : y + 4;
  const int je = t.nx - k + 1;
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    const int o = v * sl.full();
    ldv<float, 4>(y + o, &z.c[v][1]);
    const float we = w[o], ee = e[o];
    z.c[v][0] = west && !per ? 0.f : we;
    const float x = east && !per ? 0.f : ee;
    z.c[v][5] = x;
#pragma unroll
    for (int j = 2; j < 5; ++j)
      if (east && j == je) z.c[v][j] = x;
    ldv<float, 4>(y + o + t.nxp, z.n[v]);
    ldv<float, 4>(y + o - t.nxp, z.s[v]);
  }
  if (north || south) {
#pragma unroll
    for (int v = 0; v < 3; ++v)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (north) z.n[v][j] = 0.f;
        if (south) z.s[v][j] = 0.f;
      }
  }
}

// The CTA's tiles b, b + n_cta, ...  The last warp copies: issue(t, slot base, barrier) starts a tile's copies.
// The others compute, each at its own pace: body(t, slot base, next, wait), which calls wait() before it
// reads the slot; next is the CTA's next tile or null.
// POLLS: kRingWait, or 0 in the kernels that a test of the waits runs.
template <int POLLS, typename I, typename B>
__device__ __forceinline__ void ring_run(const LvArgs<float>& a, float* smem, I&& issue, B&& body) {
  __shared__ __align__(16) LvTile desc[kDescs];
  __shared__ uint64_t full[kRingSlots], empty[kRingSlots];
  static_assert(sizeof(LvTile) % 16 == 0, "copied in 16-byte pieces");
  constexpr int kWords = sizeof(LvTile) / 4, kAhead = 3;   // descriptors ahead of the tile whose copies start
  static_assert(kDescs >= kRingSlots + kAhead + 1, "a descriptor stays until its tile is done");
  const int n = (a.n_tile - (int)blockIdx.x + a.n_cta - 1) / a.n_cta, S = a.slots;
  auto tile = [&](int j) { return (int)blockIdx.x + j * a.n_cta; };
  for (int i = threadIdx.x; i < min(kAhead, n) * kWords; i += kRingThreads)
    reinterpret_cast<int*>(desc)[i] = reinterpret_cast<const int*>(a.tiles + tile(i / kWords))[i % kWords];
  if (threadIdx.x < S) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 33;" ::"r"(smem_addr(full + threadIdx.x)) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(empty + threadIdx.x)),
                 "r"(kRingPoints / 32)
                 : "memory");
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async;" ::: "memory");
  __syncthreads();
  grid_wait();
  grid_release();
  if (threadIdx.x >= kRingPoints) {
    const int lane = threadIdx.x & 31;
    asm volatile("fence.proxy.async;" ::: "memory");   // earlier grids' stores, before the bulk copies read them
    int j = 0;
    for (; j < n; ++j) {
      const int slot = j % S;
      if (j >= S && !ring_wait<POLLS>(empty + slot, (unsigned)(j / S - 1) & 1u)) break;
      // one copy group a tile, with descriptor j + kAhead in it: all but the newest are
      // complete, so descriptors up to j + 1 are there before full[slot] can be
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncwarp();
      if (j + kAhead < n && lane < (int)sizeof(LvTile) / 16)
        copy16(reinterpret_cast<char*>(desc + (j + kAhead) % kDescs) + 16 * lane,
               reinterpret_cast<const char*>(a.tiles + tile(j + kAhead)) + 16 * lane);
      issue(desc[j % kDescs], smem + (size_t)slot * a.slot_floats, full + slot);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (j < n && lane == 0) ring_lost(a.err, a.late);   // a wait ran out
    // The copies of the last tiles end before this warp does, also where a
    // computing warp has given up on them: none may reach the shared memory of
    // the CTA that comes next.  (The copying warp has nothing else to do by then.)
    for (int q = max(j - S, 0); q < j; ++q) ring_wait<kRingWait>(full + q % S, (unsigned)(q / S) & 1u);
    return;
  }
  int slot = 0;
  unsigned parity = 0;
  for (int j = 0; j < n; ++j) {
    bool ok = true;
    body(desc[j % kDescs], smem + (size_t)slot * a.slot_floats, j + 1 < n ? desc + (j + 1) % kDescs : nullptr,
         [&]() { return ok = ring_wait<POLLS>(full + slot, parity); });
    if (!ok) {
      ring_lost(a.err, a.late);
      break;
    }
    __syncwarp();
    if ((threadIdx.x & 31) == 0)
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(empty + slot)) : "memory");
    if (++slot == S) {
      slot = 0;
      parity ^= 1u;
    }
  }
  // overlap values prefetched for a tile that was left out, or given up, may
  // still be on their way
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Whether one of the columns k .. k + 3 can be in an overlap.
__device__ __forceinline__ bool over_any(const LvTile& t, int l, int r, int k) {
  return l < t.tA || l > t.L - t.tB || r < t.wS || r >= t.ny - t.wN || k < t.wL || k + 4 > t.nx - t.wR;
}
// A thread's overlap counts and values (targets, or the tangent-linear run of a
// Gauss-Newton product).
struct Over {
  int c[4], any;
  float m[3][4];
};
// A thread's overlap values of the next tile, copied to 48 bytes of its own
// while it works on this one (see lv_force).
__device__ __forceinline__ void over_prefetch(const LvTile& t, const float* q, int l, float* own) {
  const int p = t.p0 + threadIdx.x;
  if (p < t.p1 && lv_overlaps(t, l)) {
    const int r = mdiv(p, t.mq), k = (p - r * t.nq) * 4, pl = t.ny * t.nxp;
    if (!over_any(t, l, r, k)) return;
    asm volatile("cp.async.wait_all;" ::: "memory");   // (values of a tile that was left out)
#pragma unroll
    for (int v = 0; v < 3; ++v) copy16(own + v * 4 * kRingPoints, q + (r * t.nxp + k + v * pl));
  }
}
__device__ __forceinline__ void over_take(const LvTile& t, int l, int r, int k, const float* own, Over& ov) {
  ov.any = 0;
  if (!over_any(t, l, r, k)) return;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    ov.c[j] = k + j < t.nx ? lv_overlap_count(t, l, r, k + j) : 0;
    ov.any |= ov.c[j];
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
  for (int v = 0; v < 3; ++v) ldv<float, 4>(own + v * 4 * kRingPoints, ov.m[v]);
}

// lv_adj_kernel, pipelined.
template <int K, int POLLS>
__global__ void __launch_bounds__(kRingThreads, 2) lv_ring_adj_kernel(const LvArgs<float> a) {
  constexpr int NO = K == 3 ? 2 : 0;
  constexpr bool BL = K == 1;
  const int l = a.l;
  const size_t G = (size_t)3 * a.nlat * a.nlon;
  auto skip = [&](const LvTile& t) { return a.active && a.active[t.s] != a.active_value; };
  float* const dst = K == 1 ? a.mu2 : K == 2 ? a.mu1 : a.lam;
  extern __shared__ __align__(16) float ring_smem[];
  float* own = ring_smem + threadIdx.x * 4;   // K = 3: the thread's overlap values, before the slots
  float* slots = ring_smem + (K == 3 ? 12 * kRingPoints : 0);
  const bool over = K == 3 && !a.yforce && a.mu_on;
  auto target = [&](const LvTile& t) {
    return (a.gn_dx ? a.gn_dx : a.tgt) + t.traj_off + (size_t)l * level_size<float>(t);
  };
  bool first = true;
  ring_run<POLLS>(
      a, slots,
      [&](const LvTile& t, float* base, uint64_t* bar) {
        const float* Z = K == 1   ? x2_of(a, t, l)
                         : K == 2 ? x1_of(a, t, l)
                                  : a.traj + t.traj_off + (size_t)l * level_size<float>(t);
        const float* M = (K == 1 ? a.lam : K == 2 ? a.mu2 : a.mu1) + t.lv_off;
        ring_issue<2, NO, BL>(a, t, base, bar, skip(t), a.bw, a.bnd + (size_t)(t.a + l + (K == 2)) * G, [&](int i) {
          return i == 0 ? Z : i == 1 ? M : i == 2 ? a.lam + t.lv_off : a.mu2 + t.lv_off;
        });
      },
      [&](const LvTile& t, float* base, const LvTile* next, auto&& wait) {
        const int pl = t.ny * t.nxp, p = t.p0 + threadIdx.x;
        const int r = mdiv(p, t.mq), k = (p - r * t.nq) * 4, at = r * t.nxp + k, rr = r - mdiv(t.p0, t.mq);
        const bool mine = p < t.p1 && !skip(t);
        if (over && first) over_prefetch(t, target(t), l, own);
        first = false;
        if (!wait()) return;
        if (mine) {
          const Slot<2, NO, BL> sl = slot_of<2, NO, BL>(t, base);
          float rc[8];
          load_rec8(sl.rec() + 8 * rr, rc);
          const int wall = (r == 0 && (t.flags & F_SWALL) ? 1 : 0) | (r == t.ny - 1 && (t.flags & F_NWALL) ? 2 : 0);
          Patch<float, 4> z, m;
          ring_state(t, sl, rr, r, k, z);
          ring_adjoint(t, sl, rr, r, k, m);
          float o[3][4], ll[3][4], l2[3][4];
          if (K == 3) {
#pragma unroll
            for (int v = 0; v < 3; ++v) {
              ldv<float, 4>(sl.state(2) + v * sl.own() + rr * t.nxp + k, ll[v]);
              ldv<float, 4>(sl.state(3) + v * sl.own() + rr * t.nxp + k, l2[v]);
            }
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            Pt5<float> zp, mp;
            point_of(z, j, zp);
            point_of(m, j, mp);
            if (K == 3)
              adj_lambda_math<float, true>(zp, mp, rc, a.dt, a.Bth_a, a.gBth_a, a.href, wall, ll[0][j], ll[1][j],
                                           ll[2][j], l2[0][j], l2[1][j], l2[2][j], o[0][j], o[1][j], o[2][j]);
            else
              adj_stage_math<float, true>(zp, mp, rc, a.dt, a.Bth_a, a.gBth_a, a.href, wall, o[0][j], o[1][j],
                                          o[2][j]);
          }
          if (K == 3 && (a.yforce || (over && lv_overlaps(t, l)))) {
            float x[3][4];
#pragma unroll
            for (int v = 0; v < 3; ++v)
#pragma unroll
              for (int j = 0; j < 4; ++j) x[v][j] = z.c[v][j + 1];
            if (over) {
              Over ov;
              over_take(t, l, r, k, own, ov);
              if (ov.any)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                  if (ov.c[j]) overlap_force_add<float, 4>(a, ov.c[j], j, x, ov.m, o);
            } else {
              lv_force<float, 4>(a, t, l, r, k, x, o);   // external forcing
            }
          }
          float* out = dst + t.lv_off + at;
#pragma unroll
          for (int v = 0; v < 3; ++v) stv<float, 4>(out + v * pl, o[v]);
        }
        if (over && next) over_prefetch(*next, target(*next), l, own);
      });
}

// Observation forcing of level l, a CTA per box that goes on beyond it (after
// the pipelined phase 3; lv_lam_start_kernel adds a box's last level).
__global__ void __launch_bounds__(kRingThreads) lv_scatter_kernel(const LvArgs<float> a) {
  const int s = a.boxes[blockIdx.x];
  grid_wait();
  grid_release();
  if (a.active && a.active[s] != a.active_value) return;
  const SubDesc& d = a.subs[s];
  const int t0 = a.lvl_sc[d.sc_lvl + a.l], t1 = a.lvl_sc[d.sc_lvl + a.l + 1];
  float* lam = a.lam + a.box_off[s];
  for (int i = t0 + threadIdx.x; i < t1; i += blockDim.x) {
    const int g = a.sc_tgt[i], vr = g / d.nx, k = g - vr * d.nx;   // vr = v ny + r
    double acc = 0.0;
    for (int c = a.sc_off[i]; c < a.sc_off[i + 1]; ++c) acc += a.sc_w[c] * a.obs_force[a.sc_obs[c]];
    lam[(size_t)vr * d.nxp + k] += (float)acc;
  }
}

template <typename T>
cudaError_t lv_launch(void (*kernel)(const LvArgs<T>), const LvArgs<T>& a, int blocks, cudaStream_t st) {
  if (blocks <= 0) return cudaSuccess;
  return launch_dependent(kernel, dim3((unsigned)blocks), kLvThreads, 0, st, a);
}

// Adjoint phase K: the plain kernel, or the pipelined one where the plan
// has rings.
template <typename T, int K>
cudaError_t lv_phase(const LvArgs<T>& base, const LvPlan& g, cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    const LvRing& rg = g.ring[K - 1];
    if (rg.slots) {
      auto ring = g.ring_expire ? lv_ring_adj_kernel<K, 0> : lv_ring_adj_kernel<K, kRingWait>;
      LvArgs<T> a = base;
      a.tiles = g.ring_tiles;
      a.n_tile = g.n_ring[a.l];
      a.n_cta = std::min(a.n_tile, rg.ctas);
      a.slots = rg.slots;
      a.slot_floats = rg.slot_floats;
      const size_t smem = ((size_t)rg.slots * rg.slot_floats + rg.own_floats) * sizeof(float);
      cudaError_t e = raise_smem_cap(ring);
      if (e != cudaSuccess) return e;
      return launch_dependent(ring, dim3((unsigned)a.n_cta), kRingThreads, smem, st, a);
    }
  }
  return lv_launch<T>(lv_adj_kernel<T, lv_width<T>(), K>, base, base.n_tile, st);
}

}  // namespace

#define LV_TRY(call)                    \
  do {                                  \
    cudaError_t e_ = (call);            \
    if (e_ != cudaSuccess) return e_;   \
    ++*launches;                        \
  } while (0)

// The list of a launch: the tiles that keep the order of J's sums, or those of one
// round where the plan has some.  Returns the number of all its tiles.
template <typename T>
int lv_list(LvArgs<T>& a, const LvArgs<T>& base, const LvPlan& g, int l, bool sums) {
  const bool fine = !sums && g.fine_tiles;
  const auto& n = fine ? g.n_fine : g.n_tile;
  a.l = l;
  a.tiles = fine ? g.fine_tiles : base.tiles;
  a.n_tile = l < (int)n.size() ? n[l] : 0;
  return fine ? g.fine : g.tiles;
}

template <typename T>
cudaError_t launch_level_forward(const LvArgs<T>& base, const LvPlan& g, cudaStream_t st, long long* launches) {
  constexpr int V = lv_width<T>();
  LvArgs<T> a = base;
  const int L = (int)g.n_tile.size();   // longest window
  if (a.terms) LV_TRY(lv_launch<T>(lv_start_kernel<T, V>, a, g.tiles, st));
  for (int l = 0; l <= L; ++l) {
    lv_list(a, base, g, l, false);
    const int nob = a.terms && g.obs[l] ? g.n_box[l] : 0;
    if (a.n_tile + nob) LV_TRY(lv_launch<T>(lv_stage_kernel<T, V, 1, false>, a, a.n_tile + nob, st));
    if (!a.n_tile) continue;
    LV_TRY(lv_launch<T>(lv_stage_kernel<T, V, 2, false>, a, a.n_tile, st));
    lv_list(a, base, g, l, a.terms);
    if (a.terms) LV_TRY(lv_launch<T>(lv_stage_kernel<T, V, 3, true>, a, a.n_tile, st));
    else LV_TRY(lv_launch<T>(lv_stage_kernel<T, V, 3, false>, a, a.n_tile, st));
  }
  return cudaSuccess;
}

template <typename T>
cudaError_t launch_level_adjoint(const LvArgs<T>& base, const LvPlan& g, cudaStream_t st, long long* launches) {
  constexpr int V = lv_width<T>();
  LvArgs<T> a = base;
  const int all = lv_list(a, base, g, 0, false);
  LV_TRY(lv_launch<T>(lv_lam_start_kernel<T, V>, a, all, st));
  for (int l = (int)g.n_tile.size() - 1; l >= 0; --l) {
    lv_list(a, base, g, l, false);
    if (!a.stg) {   // the stage states were not stored: recompute them
      a.skip1 = a.stg1 != nullptr;
      LV_TRY(lv_launch<T>(lv_stage_kernel<T, V, 1, false>, a, a.n_tile, st));
      LV_TRY(lv_launch<T>(lv_stage_kernel<T, V, 2, false>, a, a.n_tile, st));
    }
    LV_TRY((lv_phase<T, 1>(a, g, st)));
    LV_TRY((lv_phase<T, 2>(a, g, st)));
    LV_TRY((lv_phase<T, 3>(a, g, st)));
    if constexpr (sizeof(T) == 4)
      if (g.ring[2].slots && g.obs[l] && !a.yforce)
        LV_TRY(launch_dependent(lv_scatter_kernel, dim3((unsigned)g.n_box[l + 1]), kRingThreads, 0, st, a));
  }
  LV_TRY(lv_launch<T>(lv_export_kernel<T, V>, a, all, st));
  return cudaSuccess;
}

cudaError_t launch_level_tangent(const LvArgs<double>& base, const LvPlan& g, cudaStream_t st, long long* launches) {
  LvArgs<double> a = base;
  const int L = (int)g.n_tile.size();
  a.skip1 = a.stg1 != nullptr;
  const int all = lv_list(a, base, g, 0, false);
  LV_TRY(lv_launch<double>(lv_tl_start_kernel, a, all, st));
  for (int l = 0; l <= L; ++l) {
    lv_list(a, base, g, l, false);
    const int nob = g.obs[l] ? g.n_box[l] : 0;
    if (a.n_tile + nob) LV_TRY(lv_launch<double>(lv_tl_kernel<1>, a, a.n_tile + nob, st));
    if (!a.n_tile) continue;
    if (!a.stg) {   // the stage states were not stored: recompute them
      LV_TRY(lv_launch<double>(lv_stage_kernel<double, 1, 1, false>, a, a.n_tile, st));
      LV_TRY(lv_launch<double>(lv_stage_kernel<double, 1, 2, false>, a, a.n_tile, st));
    }
    LV_TRY(lv_launch<double>(lv_tl_kernel<2>, a, a.n_tile, st));
    LV_TRY(lv_launch<double>(lv_tl_kernel<3>, a, a.n_tile, st));
  }
  return cudaSuccess;
}

#define DD4DV_INST(T)                                                                                         \
  template cudaError_t launch_level_forward<T>(const LvArgs<T>&, const LvPlan&, cudaStream_t, long long*);   \
  template cudaError_t launch_level_adjoint<T>(const LvArgs<T>&, const LvPlan&, cudaStream_t, long long*);
DD4DV_INST(double)
DD4DV_INST(float)
#undef DD4DV_INST

}  // namespace dd4dv
