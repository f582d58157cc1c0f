// Per-point arithmetic of the shallow-water step, its adjoint and its
// linearisation, shared by every sweep (the shared-memory sweeps of sweep.cu and
// the level sweeps of level.cu), so that all of them round alike.
#pragma once

#include "common.cuh"

namespace dd4dv {

// Division by a constant d >= 1 of a CTA or tile through a precomputed multiplier
// m = ceil(2^32 / d) (m = 0 encodes d = 1): floor(a / d) = floor(a m / 2^32)
// exactly whenever a * d < 2^32.  (With m = (2^32 + e) / d, 0 <= e < d, the
// product is a / d + a e / (d 2^32); the extra term is below 1 / d, the gap
// from a / d up to the next integer, when a e < 2^32.)  In the cluster sweeps a
// dividend is an index into a CTA's shared-memory stripe, below 2^20, and a divisor
// a row length or a row count; the level sweeps divide indices of a whole box, up
// to three planes of it, and level_box_fits (tuning.h) holds their products below
// 2^32.
__host__ __device__ __forceinline__ unsigned magic_of(int d) {
  return d <= 1 ? 0u : (unsigned)(0xFFFFFFFFu / (unsigned)d + 1u);
}
__device__ __forceinline__ int mdiv(int a, unsigned m) {
  return m ? (int)__umulhi((unsigned)a, m) : a;
}

// Arithmetic with explicit rounding: the compiler neither contracts nor
// reorders these, so every inlined copy of the forward step (forward sweep,
// stage recomputation in the adjoint, checkpoint-segment recomputation,
// tangent-linear sweep) rounds identically and the copies agree bit for bit.
__device__ __forceinline__ double xmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float xmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double xsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float xsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double xfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float xfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }

template <typename T>
__device__ __forceinline__ void load_rec8(const T* p, T (&r)[8]) {
  if constexpr (sizeof(T) == 4) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    const float4 y = *reinterpret_cast<const float4*>(p + 4);
    r[0] = x.x; r[1] = x.y; r[2] = x.z; r[3] = x.w;
    r[4] = y.x; r[5] = y.y; r[6] = y.z; r[7] = y.w;
  } else {
    for (int q = 0; q < 4; ++q) {
      const double2 x = *reinterpret_cast<const double2*>(p + 2 * q);
      r[2 * q] = x.x;
      r[2 * q + 1] = x.y;
    }
  }
}

// The five stencil points: centre, east, west, north, south.
template <typename T>
struct Pt5 {
  T h, u, v, hE, uE, vE, hW, uW, vW, hN, uN, vN, hS, uS, vS;
};

// Tendencies F(Z) at one point (Sec. 7, centred differences):
//   F_u = -A u (uE-uW) - Bth v (uN-uS) + (f + tau u) v - gA (hE-hW)
//   F_v = -A u (vE-vW) - Bth v (vN-vS) - (f + tau u) u - gBth (hN-hS)
//   F_h = -A ((hu)_E - (hu)_W) - (Bth/c) ((h v c)_N - (h v c)_S)
// On the FP32 path h = h_ref + h' and the h_ref parts of the fluxes are
// formed from velocity differences.
template <typename T, bool DEV>
__device__ __forceinline__ void rhs_pt(const Pt5<T>& z, T A, T f, T tau, T BinvC, T gA, T cN, T cS, T Bth,
                                       T gBth, T href, T& Fh, T& Fu, T& Fv) {
  const T u = z.u, v = z.v;
  const T dUx = xsub(z.uE, z.uW), dUy = xsub(z.uN, z.uS);
  const T dVx = xsub(z.vE, z.vW), dVy = xsub(z.vN, z.vS);
  const T dHx = xsub(z.hE, z.hW), dHy = xsub(z.hN, z.hS);
  const T fu = xfma(tau, u, f);
  const T Au = xmul(A, u), Bv = xmul(Bth, v);
  Fu = xfma(fu, v, -xfma(Au, dUx, xfma(Bv, dUy, xmul(gA, dHx))));
  Fv = -xfma(Au, dVx, xfma(Bv, dVy, xfma(fu, u, xmul(gBth, dHy))));
  T flx = xfma(z.hE, z.uE, -xmul(z.hW, z.uW));
  T fly = xfma(xmul(z.hN, z.vN), cN, -xmul(xmul(z.hS, z.vS), cS));
  if (DEV) {
    flx = xfma(href, dUx, flx);
    fly = xfma(href, xfma(z.vN, cN, -xmul(z.vS, cS)), fly);
  }
  Fh = -xfma(A, flx, xmul(BinvC, fly));
}

// Adjoint of the tendencies: G = F'(Z)^T M at one point (derived by hand from
// rhs_pt; M holds zero at ghost points that carry no tendency).  Wall rows add
// the transposed ghost mirror (h, u, -v) of the edge row.
//   G_u = mu (tau v - A dU_x) - mv (A dV_x + f + 2 tau u) + A (muE uE - muW uW)
//         + A h (mhE - mhW) + Bth (muN vN - muS vS)
//   G_v = mu (f + tau u - Bth dU_y) - mv Bth dV_y + A (mvE uE - mvW uW)
//         + Bth (mvN vN - mvS vS) + (B c) h (mhN / cN - mhS / cS)
//   G_h = gA (muE - muW) + gBth (mvN - mvS) + A u (mhE - mhW)
//         + (B c) v (mhN / cN - mhS / cS)
// evaluated as 42 explicitly rounded operations, 21 of them fused
// multiply-adds.
template <typename T, bool DEV>
__device__ __forceinline__ void rhs_adj_pt(const Pt5<T>& z, const Pt5<T>& m, T A, T f, T tau, T gA, T BcC,
                                           T icN, T icS, T tau2, T Bth, T gBth, T href, int wall, T& Gh,
                                           T& Gu, T& Gv) {
  T h = z.h;
  if (DEV) h += href;
  const T u = z.u, v = z.v;
  const T mu = m.u, mv = m.v, mh = m.h;
  const T dUx = xsub(z.uE, z.uW), dVx = xsub(z.vE, z.vW);
  const T dUy = xsub(z.uN, z.uS), dVy = xsub(z.vN, z.vS);
  const T dmhEW = xsub(m.hE, m.hW);
  const T dmhNS = xfma(m.hN, icN, -xmul(m.hS, icS));
  Gh = xfma(xmul(BcC, v), dmhNS,
            xfma(xmul(A, u), dmhEW, xfma(gBth, xsub(m.vN, m.vS), xmul(gA, xsub(m.uE, m.uW)))));
  const T a1 = xfma(-A, dUx, xmul(tau, v));
  const T a2 = xfma(A, dVx, xfma(tau2, u, f));
  const T p1 = xfma(m.uE, z.uE, -xmul(m.uW, z.uW));
  const T p2 = xfma(m.uN, z.vN, -xmul(m.uS, z.vS));
  Gu = xfma(Bth, p2, xfma(xmul(A, h), dmhEW, xfma(A, p1, xfma(-mv, a2, xmul(mu, a1)))));
  const T b1 = xfma(-Bth, dUy, xfma(tau, u, f));
  const T q1 = xfma(m.vE, z.uE, -xmul(m.vW, z.uW));
  const T q2 = xfma(m.vN, z.vN, -xmul(m.vS, z.vS));
  Gv = xfma(xmul(BcC, h), dmhNS, xfma(Bth, q2, xfma(A, q1, xfma(-mv, xmul(Bth, dVy), xmul(mu, b1)))));
  if (wall == 1) {         // south wall: ghost row = (h, u, -v) of this row
    Gu = xfma(xmul(Bth, mu), v, Gu);
    Gv = xfma(-Bth, xfma(mv, v, xmul(h, mh)), Gv);
    Gh = xfma(gBth, mv, xfma(-Bth, xmul(v, mh), Gh));
  } else if (wall == 2) {  // north wall
    Gu = xfma(-xmul(Bth, mu), v, Gu);
    Gv = xfma(Bth, xfma(mv, v, xmul(h, mh)), Gv);
    Gh = xfma(Bth, xmul(v, mh), xfma(-gBth, mv, Gh));
  }
}

// Tangent-linear tendencies dF = F'(Z) dZ at one point.
template <typename T, bool DEV>
__device__ __forceinline__ void rhs_tl_pt(const Pt5<T>& z, const Pt5<T>& d, T A, T f, T tau, T BinvC, T gA,
                                          T cN, T cS, T Bth, T gBth, T href, T& dFh, T& dFu, T& dFv) {
  const T u = z.u, v = z.v;
  const T du = d.u, dv = d.v;
  const T uE = z.uE, uW = z.uW, uN = z.uN, uS = z.uS;
  const T vE = z.vE, vW = z.vW, vN = z.vN, vS = z.vS;
  T hE = z.hE, hW = z.hW, hN = z.hN, hS = z.hS;
  if (DEV) {
    hE += href; hW += href; hN += href; hS += href;
  }
  const T duE = d.uE, duW = d.uW, duN = d.uN, duS = d.uS;
  const T dvE = d.vE, dvW = d.vW, dvN = d.vN, dvS = d.vS;
  const T dhE = d.hE, dhW = d.hW, dhN = d.hN, dhS = d.hS;
  dFu = -A * (du * (uE - uW) + u * (duE - duW)) - Bth * (dv * (uN - uS) + v * (duN - duS)) +
        (f + tau * u) * dv + tau * du * v - gA * (dhE - dhW);
  dFv = -A * (du * (vE - vW) + u * (dvE - dvW)) - Bth * (dv * (vN - vS) + v * (dvN - dvS)) -
        (f + tau * u) * du - tau * du * u - gBth * (dhN - dhS);
  dFh = -A * ((dhE * uE + hE * duE) - (dhW * uW + hW * duW)) -
        BinvC * ((dhN * vN + hN * dvN) * cN - (dhS * vS + hS * dvS) * cS);
}

// Observation term of one record with explicit rounding, so that every
// sweep kernel that evaluates it rounds alike: the bilinear value of the
// corner values x00, x01 (i + 1), x10 (j + 1), x11 (only the corners with
// non-zero weight are used), d = H x - y, J_o += 1/2 w d^2; returns the
// forcing lambda w d.
__device__ __forceinline__ double obs_term(const ObsRec& ob, double x00, double x01, double x10, double x11,
                                           double lam, double& Jo) {
  const double wj0 = __dsub_rn(1.0, ob.dj), wi0 = __dsub_rn(1.0, ob.di);
  double acc = __dmul_rn(__dmul_rn(wj0, wi0), x00);
  if (ob.di != 0.0) acc = __fma_rn(__dmul_rn(wj0, ob.di), x01, acc);
  if (ob.dj != 0.0) {
    acc = __fma_rn(__dmul_rn(ob.dj, wi0), x10, acc);
    if (ob.di != 0.0) acc = __fma_rn(__dmul_rn(ob.dj, ob.di), x11, acc);
  }
  const double d = __dsub_rn(acc, ob.y);
  Jo = __fma_rn(__dmul_rn(__dmul_rn(0.5, ob.w), d), d, Jo);
  return __dmul_rn(__dmul_rn(lam, ob.w), d);
}

// Overlap misfit of one point with overlap count c, explicitly rounded:
// part + c ((x0 - t0)^2 i0 + (x1 - t1)^2 i1 + (x2 - t2)^2 i2).
template <typename T>
__device__ __forceinline__ T overlap_term(T part, int c, T x0, T x1, T x2, T t0, T t1, T t2, T i0, T i1,
                                          T i2) {
  const T e0 = xsub(x0, t0), e1 = xsub(x1, t1), e2 = xsub(x2, t2);
  T sq = xmul(xmul(e0, e0), i0);
  sq = xfma(xmul(e1, e1), i1, sq);
  sq = xfma(xmul(e2, e2), i2, sq);
  return xfma((T)c, sq, part);
}

// Row records of the sweeps (per row j, N = row j + 1, S = row j - 1, walls
// mirrored):
//   fw (both precisions): A, f, tau, Bth / c, g A, cN, cS, 0
//   bw FP32: A, f, tau, g A, Bth c, 1 / cN, 1 / cS, 2 tau
//   bw FP64: dt A, dt f, dt tau, dt g A, dt Bth c / cN, dt Bth c / cS, 2 dt tau, 0
template <typename T>
__host__ __device__ inline void fill_records(const RowConst& r, double cN, double cS, double dt, double Bth, T* fw,
                                             T* bw) {
  const double f[8] = {r.A, r.f, r.tau, r.BinvC, r.gA, cN, cS, 0.0};
  const double b32[8] = {r.A, r.f, r.tau, r.gA, Bth * r.c, 1.0 / cN, 1.0 / cS, 2.0 * r.tau};
  const double b64[8] = {dt * r.A, dt * r.f, dt * r.tau, dt * r.gA, dt * Bth * r.c / cN, dt * Bth * r.c / cS,
                         2.0 * dt * r.tau, 0.0};
  for (int q = 0; q < 8; ++q) {
    fw[q] = (T)f[q];
    bw[q] = (T)(sizeof(T) == 8 ? b64[q] : b32[q]);
  }
}

// One RK3 stage of the global model at one point, out = ca X + cb (Y + dt F(Y))
// from rec = A, f, tau, g A, Bth / c, cN, cS.  28 FP64 instructions (34 with X).
// Forecasts and model runs share it, so that a run from the background is the
// library's own background trajectory.  The tendencies are summed before they
// meet the state: h is some 4000 m, and with one fused operation a term into it
// (24 instructions) its roundings were 1.0-1.25x larger.
__host__ __device__ inline void fill_global_record(const RowConst& r, double cN, double cS, double* rec) {
  rec[0] = r.A;
  rec[1] = r.f;
  rec[2] = r.tau;
  rec[3] = r.gA;
  rec[4] = r.BinvC;
  rec[5] = cN;
  rec[6] = cS;
  rec[7] = 0.0;
}
__device__ __forceinline__ void global_pt(const Pt5<double>& y, const double (&rc)[8], double dt, double Bth,
                                          double gBth, double ca, double cb, double x0, double x1, double x2,
                                          double& oh, double& ou, double& ov) {
  const double fu = xfma(rc[2], y.u, rc[1]), Au = xmul(rc[0], y.u), Bv = xmul(Bth, y.v);
  double Fu = xfma(-Au, xsub(y.uE, y.uW), -xmul(Bv, xsub(y.uN, y.uS)));
  Fu = xfma(fu, y.v, Fu);
  Fu = xfma(-rc[3], xsub(y.hE, y.hW), Fu);
  double Fv = xfma(-Au, xsub(y.vE, y.vW), -xmul(Bv, xsub(y.vN, y.vS)));
  Fv = xfma(-fu, y.u, Fv);
  Fv = xfma(-gBth, xsub(y.hN, y.hS), Fv);
  const double fx = xfma(y.hE, y.uE, -xmul(y.hW, y.uW));
  const double fy = xfma(xmul(y.hN, y.vN), rc[5], -xmul(xmul(y.hS, y.vS), rc[6]));
  const double Fh = xfma(-rc[0], fx, -xmul(rc[4], fy));
  oh = xfma(dt, Fh, y.h);
  ou = xfma(dt, Fu, y.u);
  ov = xfma(dt, Fv, y.v);
  if (ca != 0.0) {
    oh = xfma(ca, x0, xmul(cb, oh));
    ou = xfma(ca, x1, xmul(cb, ou));
    ov = xfma(ca, x2, xmul(cb, ov));
  }
}

// The FP64 adjoint in its form of fewest FP64 instructions.  The FP64 pipe issues one warp
// instruction in 16 cycles per SM and bounds every FP64 sweep.  The records
// (and Bth, g Bth) hold dt times the constant, the cos ratios of the neighbour
// rows are folded into one constant each, and every term is one fused
// multiply-add into the value that it changes: a stage adjoint takes 38
// instructions instead of 45, lambda(n) 47 instead of 54 (medium workload, 64
// boxes of 72 x 36..40 points in clusters of 4 x 192 threads: adjoint 2.67 ->
// 2.32 ms).  The forward stages keep the order of rhs_pt and global_pt: their
// rounding of h, some 1e-13 of a misfit, is what an analysis amplifies, and a
// second order of roundings would show in it at 1e-10.
// M + dt F'(Z)^T M at one point (the terms of rhs_adj_pt).
__device__ __forceinline__ void adjoint_pt64(const Pt5<double>& z, const Pt5<double>& m, const double (&rc)[8],
                                             double Bth, double gBth, int wall, double& oh, double& ou, double& ov) {
  const double h = z.h, u = z.u, v = z.v, mu = m.u, mv = m.v;
  const double e1 = xmul(rc[0], xsub(m.hE, m.hW));
  const double e2 = xfma(rc[4], m.hN, -xmul(rc[5], m.hS));
  oh = xfma(rc[3], xsub(m.uE, m.uW), m.h);
  oh = xfma(gBth, xsub(m.vN, m.vS), oh);
  oh = xfma(u, e1, oh);
  oh = xfma(v, e2, oh);
  double s = xfma(m.uE, z.uE, -xmul(m.uW, z.uW));
  s = xfma(-mu, xsub(z.uE, z.uW), s);
  s = xfma(-mv, xsub(z.vE, z.vW), s);
  ou = xfma(rc[0], s, m.u);
  ou = xfma(h, e1, ou);
  ou = xfma(Bth, xfma(m.uN, z.vN, -xmul(m.uS, z.vS)), ou);
  ou = xfma(mu, xmul(rc[2], v), ou);
  ou = xfma(-mv, xfma(rc[6], u, rc[1]), ou);
  s = xfma(m.vN, z.vN, -xmul(m.vS, z.vS));
  s = xfma(-mu, xsub(z.uN, z.uS), s);
  s = xfma(-mv, xsub(z.vN, z.vS), s);
  ov = xfma(Bth, s, m.v);
  ov = xfma(h, e2, ov);
  ov = xfma(rc[0], xfma(m.vE, z.uE, -xmul(m.vW, z.uW)), ov);
  ov = xfma(mu, xfma(rc[2], u, rc[1]), ov);
  if (wall) {   // ghost row = (h, u, -v) of this row: south (1), north (2)
    const double B = wall == 1 ? Bth : -Bth, gB = wall == 1 ? gBth : -gBth;
    ou = xfma(xmul(B, mu), v, ou);
    ov = xfma(-B, xfma(mv, v, xmul(h, m.h)), ov);
    oh = xfma(gB, mv, xfma(-B, xmul(v, m.h), oh));
  }
}

// The arithmetic of one RK3 stage at one point, out = cx X + cy (Y + dt F(Y)),
// from the point's stencil y of Y, its row constants rc and its X values (read
// only when cx != 0).  Every sweep (forward, stage recomputation, checkpoint
// segments, tangent-linear, the deep-halo FP32 sweeps) calls this one
// function, so all of them round every stage identically.
template <typename T, bool DEV>
__device__ __forceinline__ void stage_math(const Pt5<T>& y, const T (&rc)[8], T dt, T Bth, T gBth, T href, T cx,
                                           T cy, T xh, T xu, T xv, T& o0, T& o1, T& o2) {
  T Fh, Fu, Fv;
  rhs_pt<T, DEV>(y, rc[0], rc[1], rc[2], rc[3], rc[4], rc[5], rc[6], Bth, gBth, href, Fh, Fu, Fv);
  o0 = xfma(dt, Fh, y.h);
  o1 = xfma(dt, Fu, y.u);
  o2 = xfma(dt, Fv, y.v);
  if (cy != (T)1) {
    o0 = xmul(cy, o0);
    o1 = xmul(cy, o1);
    o2 = xmul(cy, o2);
  }
  if (cx != (T)0) {
    o0 = xfma(cx, xh, o0);
    o1 = xfma(cx, xu, o1);
    o2 = xfma(cx, xv, o2);
  }
}


// The arithmetic of the transposed RK3 step at one point, shared by every
// adjoint sweep so that all of them round alike.  A stage adjoint
// mu_out = m + dt F'(z)^T m ...
template <typename T, bool DEV>
__device__ __forceinline__ void adj_stage_math(const Pt5<T>& z, const Pt5<T>& m, const T (&rc)[8], T dt, T Bth,
                                               T gBth, T href, int wall, T& v0, T& v1, T& v2) {
  if constexpr (sizeof(T) == 8) {
    adjoint_pt64(z, m, rc, Bth, gBth, wall, v0, v1, v2);
  } else {
    T Gh, Gu, Gv;
    rhs_adj_pt<T, DEV>(z, m, rc[0], rc[1], rc[2], rc[3], rc[4], rc[5], rc[6], rc[7], Bth, gBth, href, wall, Gh, Gu,
                       Gv);
    v0 = xfma(dt, Gh, m.h);
    v1 = xfma(dt, Gu, m.u);
    v2 = xfma(dt, Gv, m.v);
  }
}
// ... and lambda(n) = lambda'/3 + mu2/2 + (mu1 + dt F'(x)^T mu1)/6 from the
// stencil m of mu1, z of x, and lambda' = (ph, pu, pv), mu2 = (qh, qu, qv) at
// the point.
template <typename T, bool DEV>
__device__ __forceinline__ void adj_lambda_math(const Pt5<T>& z, const Pt5<T>& m, const T (&rc)[8], T dt, T Bth,
                                                T gBth, T href, int wall, T ph, T pu, T pv, T qh, T qu, T qv,
                                                T& v0, T& v1, T& v2) {
  const T c13 = (T)(1.0 / 3.0), c16 = (T)(1.0 / 6.0);
  T g0, g1, g2;
  adj_stage_math<T, DEV>(z, m, rc, dt, Bth, gBth, href, wall, g0, g1, g2);
  v0 = xfma(c16, g0, xfma((T)0.5, qh, xmul(c13, ph)));
  v1 = xfma(c16, g1, xfma((T)0.5, qu, xmul(c13, pu)));
  v2 = xfma(c16, g2, xfma((T)0.5, qv, xmul(c13, pv)));
}

}  // namespace dd4dv
