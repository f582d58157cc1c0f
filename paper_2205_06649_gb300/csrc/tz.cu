// The Turkel-Zwas scheme of Sec. 7 on the whole sphere: forward RK3 stages,
// tangent-linear stages and the transposed (adjoint) stages, FP64, one thread
// per grid point, global memory.
//
// Scheme (Sec. 7, the semi-discrete U_ij, V_ij, H_ij with longitude stride
// p, latitude stride q and averaging weight alpha; readings of the garbled
// print as in the oracle): advection with stride 1, pressure gradients over
// i +- p and j +- q, Coriolis terms of the u (v) equation averaged over
// i +- p (j +- q) with weight alpha, and the divergence of the continuity
// equation averaged over the diagonal points (i +- p, j +- q) with weight
// alpha.  Longitude is periodic; the walls mirror (h, u, -v) to depth q
// (ghost row -1 - s holds row s, row nlat + s holds row nlat - 1 - s, with
// the mirrored row's cos, f and tan).
//
// The tangent-linear stage is built from one list of partial derivatives per
// point (tz_jacobian: for each value of the state that F at the point reads,
// d F_out / d value_in).  The adjoint stage gathers the transposed list: a point
// collects, term by term, what the points that read it send back, without atomic
// additions.  (The observation forcing is still scattered by FP64 atomics, in
// tz_obs_scatter_kernel: where observations share a corner, the last bits of a
// gradient depend on their order.)
// Bound: launch latency on small grids (8 launches a step of about 3 us), the
// FP64 pipe on large ones.  Row constants hold every quotient (launch_tz_rows):
// the divisions were most of the FP64 work.  256 x 128 points, 128 steps,
// (p, q, alpha) = (2, 1, 1/2), J and gradient: 21.1 -> 7.6 ms.
//
// Roundings: h is some 4000 m and every operation on it rounds by up to 2e-13 m,
// in the combination (1/3) X + (2/3) Y to one side, so that a run drifts by its
// order of operations.  The order here (tendencies summed and multiplied by dt
// first, (1/3) X rounded by itself) is that of the plain stage: with dt in the row
// constants, one operation a term into the state and (2/3) Y rounded by itself,
// 2 % faster, gradients of 54- to 172-step runs were up to 2.3 times further from
// a plain 64-bit evaluation (236 x 98 points, 172 steps: 2.0e-12 against 8.6e-13).
#include "common.cuh"

namespace dd4dv {

namespace {

struct Loc {
  int j, i;
  double vs;   // -1 for v read through a wall mirror
};

__device__ __forceinline__ Loc tz_resolve(const TzArgs& t, int j, int i) {
  Loc L;
  L.i = ((i % t.nlon) + t.nlon) % t.nlon;
  L.vs = 1.0;
  if (j < 0) {
    L.j = -1 - j;
    L.vs = -1.0;
  } else if (j >= t.nlat) {
    L.j = 2 * t.nlat - 1 - j;
    L.vs = -1.0;
  } else {
    L.j = j;
  }
  return L;
}

__device__ __forceinline__ double tz_val(const TzArgs& t, const double* Y, int var, int j, int i) {
  const Loc L = tz_resolve(t, j, i);
  const double x = Y[((size_t)var * t.nlat + L.j) * t.nlon + L.i];
  return var == 2 ? L.vs * x : x;
}

// Semi-discrete Turkel-Zwas tendencies at (j, i):
//   F_u = -s_lon u/c (u[i+1] - u[i-1]) - s_lat v (u[j+1] - u[j-1]) - s_lon g/(p c) (h[i+p] - h[i-p])
//         + (1-alpha) C v + alpha/2 ((C v)[i+p] + (C v)[i-p])
//   F_v = -s_lon u/c (v[i+1] - v[i-1]) - s_lat v (v[j+1] - v[j-1]) - s_lat g/q (h[j+q] - h[j-q])
//         - (1-alpha) C u - alpha/2 ((C u)[j+q] + (C u)[j-q])
//   F_h = -{ s_lon u/c (h[i+1] - h[i-1]) + s_lat v (h[j+1] - h[j-1]) + s_lon h/(p c) Du + s_lat h/(q c) Dv }
//   Du = (1-alpha) (u[i+p] - u[i-p]) + alpha/2 (u[i+p,j+q] - u[i-p,j+q] + u[i+p,j-q] - u[i-p,j-q])
//   Dv = (1-alpha) ((v c)[j+q] - (v c)[j-q])
//        + alpha/2 ((v c)[i+p,j+q] - (v c)[i+p,j-q] + (v c)[i-p,j+q] - (v c)[i-p,j-q])
// with C = f + u tan(theta)/a at the point it multiplies (its own row's f, tan).

// Partial derivatives of (F_h, F_u, F_v) at (j, i) with respect to every
// state value they read: vis(out_var, in_var, row, col, coef) with the
// location resolved through the periodic wrap and the wall mirror (a v read
// through a mirror enters with the sign flipped).  Derived from F above term by
// term; a location read by several terms (p = 1 or q = 1) gets one entry
// per term.
template <typename Vis>
__device__ void tz_jacobian(const TzArgs& t, const double* Y, int j, int i, Vis&& vis) {
  const int p = t.p, q = t.q;
  const double al = t.alpha, sl = t.slon, st = t.slat, g = t.g;
  const RowConst rc = t.rows[j];
  const double c = rc.c, f = rc.f, tau = rc.tau;
  const RowConst rN = t.rows[tz_resolve(t, j + q, i).j], rS = t.rows[tz_resolve(t, j - q, i).j];
  auto emit = [&](int vo, int vi, int dj, int di, double coef) {
    const Loc L = tz_resolve(t, j + dj, i + di);
    vis(vo, vi, L.j, L.i, vi == 2 ? coef * L.vs : coef);
  };
  const double h = tz_val(t, Y, 0, j, i), u = tz_val(t, Y, 1, j, i), v = tz_val(t, Y, 2, j, i);
  const double C = f + u * tau;
  // F_u
  const double dux1 = tz_val(t, Y, 1, j, i + 1) - tz_val(t, Y, 1, j, i - 1);
  const double duy1 = tz_val(t, Y, 1, j + 1, i) - tz_val(t, Y, 1, j - 1, i);
  emit(1, 1, 0, 0, -sl / c * dux1 + (1.0 - al) * tau * v);
  emit(1, 1, 0, 1, -sl * u / c);
  emit(1, 1, 0, -1, sl * u / c);
  emit(1, 2, 0, 0, -st * duy1 + (1.0 - al) * C);
  emit(1, 1, 1, 0, -st * v);
  emit(1, 1, -1, 0, st * v);
  emit(1, 0, 0, p, -sl * g / (p * c));
  emit(1, 0, 0, -p, sl * g / (p * c));
  if (al != 0.0) {
    const double uEp = tz_val(t, Y, 1, j, i + p), vEp = tz_val(t, Y, 2, j, i + p);
    const double uWp = tz_val(t, Y, 1, j, i - p), vWp = tz_val(t, Y, 2, j, i - p);
    emit(1, 1, 0, p, 0.5 * al * tau * vEp);
    emit(1, 2, 0, p, 0.5 * al * (f + uEp * tau));
    emit(1, 1, 0, -p, 0.5 * al * tau * vWp);
    emit(1, 2, 0, -p, 0.5 * al * (f + uWp * tau));
  }
  // F_v
  const double dvx1 = tz_val(t, Y, 2, j, i + 1) - tz_val(t, Y, 2, j, i - 1);
  const double dvy1 = tz_val(t, Y, 2, j + 1, i) - tz_val(t, Y, 2, j - 1, i);
  emit(2, 1, 0, 0, -sl / c * dvx1 - (1.0 - al) * (f + 2.0 * u * tau));
  emit(2, 2, 0, 1, -sl * u / c);
  emit(2, 2, 0, -1, sl * u / c);
  emit(2, 2, 0, 0, -st * dvy1);
  emit(2, 2, 1, 0, -st * v);
  emit(2, 2, -1, 0, st * v);
  emit(2, 0, q, 0, -st * g / q);
  emit(2, 0, -q, 0, st * g / q);
  if (al != 0.0) {
    const double uNq = tz_val(t, Y, 1, j + q, i), uSq = tz_val(t, Y, 1, j - q, i);
    emit(2, 1, q, 0, -0.5 * al * (rN.f + 2.0 * uNq * rN.tau));
    emit(2, 1, -q, 0, -0.5 * al * (rS.f + 2.0 * uSq * rS.tau));
  }
  // F_h
  const double dhx1 = tz_val(t, Y, 0, j, i + 1) - tz_val(t, Y, 0, j, i - 1);
  const double dhy1 = tz_val(t, Y, 0, j + 1, i) - tz_val(t, Y, 0, j - 1, i);
  double du = (1.0 - al) * (tz_val(t, Y, 1, j, i + p) - tz_val(t, Y, 1, j, i - p));
  double dv = (1.0 - al) * (tz_val(t, Y, 2, j + q, i) * rN.c - tz_val(t, Y, 2, j - q, i) * rS.c);
  if (al != 0.0) {
    du += 0.5 * al * (tz_val(t, Y, 1, j + q, i + p) - tz_val(t, Y, 1, j + q, i - p) +
                      tz_val(t, Y, 1, j - q, i + p) - tz_val(t, Y, 1, j - q, i - p));
    dv += 0.5 * al * (tz_val(t, Y, 2, j + q, i + p) * rN.c - tz_val(t, Y, 2, j - q, i + p) * rS.c +
                      tz_val(t, Y, 2, j + q, i - p) * rN.c - tz_val(t, Y, 2, j - q, i - p) * rS.c);
  }
  const double ku = sl * h / (p * c), kv = st * h / (q * c);
  emit(0, 1, 0, 0, -sl / c * dhx1);
  emit(0, 0, 0, 1, -sl * u / c);
  emit(0, 0, 0, -1, sl * u / c);
  emit(0, 2, 0, 0, -st * dhy1);
  emit(0, 0, 1, 0, -st * v);
  emit(0, 0, -1, 0, st * v);
  emit(0, 0, 0, 0, -(sl / (p * c) * du + st / (q * c) * dv));
  emit(0, 1, 0, p, -ku * (1.0 - al));
  emit(0, 1, 0, -p, ku * (1.0 - al));
  emit(0, 2, q, 0, -kv * (1.0 - al) * rN.c);
  emit(0, 2, -q, 0, kv * (1.0 - al) * rS.c);
  if (al != 0.0) {
    const double a2 = 0.5 * al;
    emit(0, 1, q, p, -ku * a2);
    emit(0, 1, q, -p, ku * a2);
    emit(0, 1, -q, p, -ku * a2);
    emit(0, 1, -q, -p, ku * a2);
    emit(0, 2, q, p, -kv * a2 * rN.c);
    emit(0, 2, -q, p, kv * a2 * rS.c);
    emit(0, 2, q, -p, -kv * a2 * rN.c);
    emit(0, 2, -q, -p, kv * a2 * rS.c);
  }
}

constexpr int kTzThreads = 128;

// The point of a thread: flat over rows.
struct TzPt {
  int j, i;
  unsigned o;        // offset in a plane
  bool in;
  __device__ __forceinline__ explicit TzPt(const TzArgs& t) {
    o = blockIdx.x * kTzThreads + threadIdx.x;
    j = (int)(o / (unsigned)t.nlon);
    i = (int)(o - (unsigned)j * t.nlon);
    in = j < t.nlat;
  }
};
__device__ __forceinline__ int tz_wrap(int i, int n) { return i < 0 ? i + n : i >= n ? i - n : i; }
// Row s rows away (|s| < nlat), through the wall mirror; sg = -1 for a v read
// through it.
__device__ __forceinline__ int tz_row(int j, int s, int nlat, double& sg) {
  const int r = j + s;
  sg = r < 0 || r >= nlat ? -1.0 : 1.0;
  return r < 0 ? -1 - r : r >= nlat ? 2 * nlat - 1 - r : r;
}

// out = cx X + cy (Y + dt F(Y)), the tendencies F above with the row records
__global__ void __launch_bounds__(kTzThreads) tz_stage_kernel(TzArgs t, const double* X, const double* Y, double* out,
                                                              double cx, double cy) {
  const TzPt m(t);
  grid_wait();
  grid_release();
  if (!m.in) return;
  const size_t pl = (size_t)t.nlat * t.nlon, o = m.o;
  const double *H = Y, *U = Y + pl, *V = Y + 2 * pl;
  const size_t row = (size_t)m.j * t.nlon;
  const int iE = tz_wrap(m.i + 1, t.nlon), iW = tz_wrap(m.i - 1, t.nlon);
  const int pE = tz_wrap(m.i + t.p, t.nlon), pW = tz_wrap(m.i - t.p, t.nlon);
  double s1N, s1S, sN, sS;
  const size_t r1N = (size_t)tz_row(m.j, 1, t.nlat, s1N) * t.nlon, r1S = (size_t)tz_row(m.j, -1, t.nlat, s1S) * t.nlon;
  const int jN = tz_row(m.j, t.q, t.nlat, sN), jS = tz_row(m.j, -t.q, t.nlat, sS);
  const size_t rN = (size_t)jN * t.nlon, rS = (size_t)jS * t.nlon;
  const TzRow rc = t.rec[m.j];
  const double cN = sN * t.rec[jN].c, cS = sS * t.rec[jS].c;   // (v c) through the mirror
  const double h = H[o], u = U[o], v = V[o], al = t.alpha, a1 = 1.0 - al, a2 = 0.5 * al;
  const double Au = rc.a * u, Bv = t.slat * v, C = fma(rc.tau, u, rc.f);
  const double uEp = U[row + pE], uWp = U[row + pW], vN = V[rN + m.i], vS = V[rS + m.i];
  double cu = a1 * C * v, cv = a1 * C * u;
  double du = a1 * (uEp - uWp), dv = a1 * fma(vN, cN, -vS * cS);
  if (al != 0.0) {
    cu = fma(a2, fma(fma(rc.tau, uEp, rc.f), V[row + pE], fma(rc.tau, uWp, rc.f) * V[row + pW]), cu);
    const TzRow N = t.rec[jN], S = t.rec[jS];
    const double uN = U[rN + m.i], uS = U[rS + m.i];
    cv = fma(a2, fma(fma(N.tau, uN, N.f), uN, fma(S.tau, uS, S.f) * uS), cv);
    du = fma(a2, (U[rN + pE] - U[rN + pW]) + (U[rS + pE] - U[rS + pW]), du);
    dv = fma(a2, fma(V[rN + pE] + V[rN + pW], cN, -(V[rS + pE] + V[rS + pW]) * cS), dv);
  }
  double Fu = fma(Au, U[row + iE] - U[row + iW], Bv * (U[r1N + m.i] - U[r1S + m.i]));
  Fu = cu - fma(rc.kg, H[row + pE] - H[row + pW], Fu);
  double Fv = fma(Au, V[row + iE] - V[row + iW], Bv * (s1N * V[r1N + m.i] - s1S * V[r1S + m.i]));
  Fv = -cv - fma(t.gq, H[rN + m.i] - H[rS + m.i], Fv);
  double Fh = fma(Au, H[row + iE] - H[row + iW], Bv * (H[r1N + m.i] - H[r1S + m.i]));
  Fh = -fma(h, fma(rc.kp, du, rc.kq * dv), Fh);
  // One rounding of the size of h a stage, not one a term, and (1/3) X rounded by
  // itself: see the head of the file.
  double oh = fma(t.dt, Fh, h), ou = fma(t.dt, Fu, u), ov = fma(t.dt, Fv, v);
  if (cx != 0.0) {
    oh = fma(cy, oh, __dmul_rn(cx, X[o]));
    ou = fma(cy, ou, __dmul_rn(cx, X[o + pl]));
    ov = fma(cy, ov, __dmul_rn(cx, X[o + 2 * pl]));
  }
  out[o] = oh;
  out[o + pl] = ou;
  out[o + 2 * pl] = ov;
}

// G = M + dt F'(Y)^T M gathered at one point: per term of F, what the points
// that read this one send back.  A point s rows south (north) reads it with
// the sign of its northern (southern) neighbour; where the wall mirror folds
// that row back (row < s), the mirrored row reads it with its southern
// (northern) neighbour instead, and its v with the sign flipped, so that the
// terms odd in the row distance change sign (sg = -1) but for v.
__global__ void __launch_bounds__(kTzThreads) tz_adj_kernel(TzArgs t, const double* Y, const double* M,
                                                            const double* lam, const double* mu2, const double* force,
                                                            double* out) {
  const TzPt m(t);
  grid_wait();
  grid_release();
  if (!m.in) return;
  const size_t pl = (size_t)t.nlat * t.nlon, o = m.o;
  const double *H = Y, *U = Y + pl, *V = Y + 2 * pl;
  const double *mh = M, *mu = M + pl, *mv = M + 2 * pl;
  const size_t row = (size_t)m.j * t.nlon;
  const size_t E = row + tz_wrap(m.i + 1, t.nlon), W = row + tz_wrap(m.i - 1, t.nlon);
  const int pE = tz_wrap(m.i + t.p, t.nlon), pW = tz_wrap(m.i - t.p, t.nlon);
  // rows at distance 1 and q: the same as those this point reads, mirrors included
  double s1N, s1S, sN, sS;
  const int j1N = tz_row(m.j, 1, t.nlat, s1N), j1S = tz_row(m.j, -1, t.nlat, s1S);
  const int jN = tz_row(m.j, t.q, t.nlat, sN), jS = tz_row(m.j, -t.q, t.nlat, sS);
  const size_t N1 = (size_t)j1N * t.nlon + m.i, S1 = (size_t)j1S * t.nlon + m.i;
  const size_t rN = (size_t)jN * t.nlon, rS = (size_t)jS * t.nlon, Nq = rN + m.i, Sq = rS + m.i;
  const TzRow rc = t.rec[m.j], Rn = t.rec[jN], Rs = t.rec[jS];
  const double al = t.alpha, a1 = 1.0 - al, a2 = 0.5 * al;
  const double h = H[o], u = U[o], v = V[o], xh = mh[o], xu = mu[o], xv = mv[o];
  const double C = fma(rc.tau, u, rc.f);
  // products of the neighbours' velocities and adjoints
  const double uE = U[E], uW = U[W], vN = s1N * V[N1], vS = s1S * V[S1];
  const double muE = mu[E], muW = mu[W], mvE = mv[E], mvW = mv[W], mhE = mh[E], mhW = mh[W];
  // advection: what F of the four neighbours reads of (h, u, v) here.  The
  // northern neighbour reads this point as its south: + s_lat v m; a mirrored
  // one (sg = -1) with the other sign, and vN, vS carry that sign.
  double gh = rc.a * fma(uE, mhE, -uW * mhW);
  double gu = rc.a * fma(uE, muE, -uW * muW);
  double gv = rc.a * fma(uE, mvE, -uW * mvW);
  gh = fma(t.slat, fma(vN, mh[N1], -vS * mh[S1]), gh);
  gu = fma(t.slat, fma(vN, mu[N1], -vS * mu[S1]), gu);
  gv = fma(t.slat, fma(s1N * vN, mv[N1], -s1S * vS * mv[S1]), gv);
  // own coefficients: u and v multiply the centred differences of all three
  const double dhx = H[E] - H[W], dux = uE - uW, dvx = V[E] - V[W];
  const double dhy = H[N1] - H[S1], duy = U[N1] - U[S1], dvy = vN - vS;
  gu = fma(-rc.a, fma(xu, dux, fma(xv, dvx, xh * dhx)), gu);
  gv = fma(-t.slat, fma(xu, duy, fma(xv, dvy, xh * dhy)), gv);
  // Coriolis
  gu = fma(a1, fma(xu * rc.tau, v, -xv * fma(rc.tau, u, C)), gu);
  gv = fma(a1 * xu, C, gv);
  // pressure gradients
  const double muEp = mu[row + pE], muWp = mu[row + pW], mvN = mv[Nq], mvS = mv[Sq];
  gh = fma(rc.kg, muEp - muWp, gh);
  gh = fma(t.gq, sN * mvN - sS * mvS, gh);
  // divergence: h m_h of the points that read u, v here; h times the divergence
  const double kE = H[row + pE] * mh[row + pE], kW = H[row + pW] * mh[row + pW];
  const double kN = H[Nq] * mh[Nq], kS = H[Sq] * mh[Sq];
  gu = fma(a1 * rc.kp, kE - kW, gu);
  gv = fma(a1 * rc.c, fma(Rn.kq, kN, -Rs.kq * kS), gv);
  const double cN = sN * Rn.c, cS = sS * Rs.c;
  double du = a1 * (U[row + pE] - U[row + pW]), dv = a1 * fma(V[Nq], cN, -V[Sq] * cS);
  if (al != 0.0) {
    gu = fma(a2 * rc.tau * v, muEp + muWp, gu);
    gv = fma(a2 * C, muEp + muWp, gv);
    gu = fma(-a2 * fma(rc.tau, u, C), mvN + mvS, gu);
    const double kNE = H[rN + pE] * mh[rN + pE], kNW = H[rN + pW] * mh[rN + pW];
    const double kSE = H[rS + pE] * mh[rS + pE], kSW = H[rS + pW] * mh[rS + pW];
    gu = fma(a2, fma(Rn.kp, kNE - kNW, Rs.kp * (kSE - kSW)), gu);
    gv = fma(a2 * rc.c, fma(Rn.kq, kNE + kNW, -Rs.kq * (kSE + kSW)), gv);
    du = fma(a2, (U[rN + pE] - U[rN + pW]) + (U[rS + pE] - U[rS + pW]), du);
    dv = fma(a2, fma(V[rN + pE] + V[rN + pW], cN, -(V[rS + pE] + V[rS + pW]) * cS), dv);
  }
  gh = fma(-xh, fma(rc.kp, du, rc.kq * dv), gh);
  double g[3] = {fma(t.dt, gh, xh), fma(t.dt, gu, xu), fma(t.dt, gv, xv)};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const size_t q = o + c * pl;
    double r = g[c];
    if (lam) {
      r = fma(1.0 / 6.0, r, fma(0.5, mu2[q], (1.0 / 3.0) * lam[q]));
      if (force) r += force[q];
    }
    out[q] = r;
  }
}

// dout = cx dX + cy (dY + dt F'(Y) dY)
__global__ void tz_tl_stage_kernel(TzArgs t, const double* Y, const double* dX, const double* dY, double* dout,
                                   double cx, double cy) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i >= t.nlon) return;
  const size_t pl = (size_t)t.nlat * t.nlon, o = (size_t)j * t.nlon + i;
  double d[3] = {0.0, 0.0, 0.0};
  tz_jacobian(t, Y, j, i, [&](int vo, int vi, int jj, int ii, double coef) {
    d[vo] += coef * dY[vi * pl + (size_t)jj * t.nlon + ii];
  });
  for (int v = 0; v < 3; ++v) {
    double r = cy * (dY[v * pl + o] + t.dt * d[v]);
    if (cx != 0.0) r += cx * dX[v * pl + o];
    dout[v * pl + o] = r;
  }
}

// x0 = xb + sigma_v w (diagonal B) or grad = w + sigma_v lam
__global__ void tz_scale_add_kernel(double* out, const double* a, const double* b, const double* sigma, long long plane) {
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < 3 * plane;
       k += (long long)gridDim.x * blockDim.x)
    out[k] = a[k] + sigma[k / plane] * b[k];
}

// Sum of the block's values (fixed order), on thread 0.
__device__ double tz_block_sum(double x) {
  __shared__ double sh[8];
  for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh[w];
  return s;
}

// Observation misfits of the whole trajectory (obs sorted by level): forcing
// lam (H x - y) / sigma_o^2 per observation and lam/2 sum (H x - y)^2 /
// sigma_o^2, one partial sum per block in a fixed order.
__global__ void tz_obs_misfit_kernel(const double* traj, long long n, const int* level, const int* var,
                                     const double* fi, const double* fj, const double* y, const double* so,
                                     int nlon, int nlat, double lam, double* force, double* part) {
  double acc = 0.0;
  const size_t pl = (size_t)nlat * nlon;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
    const int i0 = (int)floor(fi[k]), j0 = (int)floor(fj[k]);
    const double di = fi[k] - i0, dj = fj[k] - j0;
    const int i1 = (i0 + 1) % nlon;
    const double* x = traj + ((size_t)level[k] * 3 + var[k]) * pl;
    double hx = (1.0 - dj) * (1.0 - di) * x[(size_t)j0 * nlon + i0];
    if (di != 0.0) hx += (1.0 - dj) * di * x[(size_t)j0 * nlon + i1];
    if (dj != 0.0) {
      hx += dj * (1.0 - di) * x[(size_t)(j0 + 1) * nlon + i0];
      if (di != 0.0) hx += dj * di * x[(size_t)(j0 + 1) * nlon + i1];
    }
    const double d = hx - y[k], w = 1.0 / (so[k] * so[k]);
    force[k] = lam * w * d;
    acc += 0.5 * lam * w * d * d;
  }
  const double s = tz_block_sum(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// lam += H^T force for the observations [k0, k1) (one level)
__global__ void tz_obs_scatter_kernel(long long k0, long long k1, const int* var, const double* fi,
                                      const double* fj, const double* force, int nlon, int nlat, double* lam) {
  const size_t pl = (size_t)nlat * nlon;
  for (long long k = k0 + (long long)blockIdx.x * blockDim.x + threadIdx.x; k < k1;
       k += (long long)gridDim.x * blockDim.x) {
    const int i0 = (int)floor(fi[k]), j0 = (int)floor(fj[k]);
    const double di = fi[k] - i0, dj = fj[k] - j0;
    const int i1 = (i0 + 1) % nlon;
    double* x = lam + (size_t)var[k] * pl;
    const double fk = force[k];
    atomicAdd(&x[(size_t)j0 * nlon + i0], (1.0 - dj) * (1.0 - di) * fk);
    if (di != 0.0) atomicAdd(&x[(size_t)j0 * nlon + i1], (1.0 - dj) * di * fk);
    if (dj != 0.0) {
      atomicAdd(&x[(size_t)(j0 + 1) * nlon + i0], dj * (1.0 - di) * fk);
      if (di != 0.0) atomicAdd(&x[(size_t)(j0 + 1) * nlon + i1], dj * di * fk);
    }
  }
}

// Partial sums of 1/2 w.w, then J = J_b + J_o in a fixed order.
__global__ void tz_background_kernel(const double* w, long long n, double* part) {
  double acc = 0.0;
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
    acc += w[k] * w[k];
  const double s = tz_block_sum(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = 0.5 * s;
}
__global__ void tz_finish_J_kernel(const double* part, int nobs, double* J) {
  double x = 0.0;
  if (threadIdx.x < kTzBlocks) x = part[kTzBlocks + threadIdx.x] + (nobs ? part[threadIdx.x] : 0.0);
  const double s = tz_block_sum(x);
  if (threadIdx.x == 0) *J = s;
}

__global__ void tz_rows_kernel(TzArgs t, TzRow* rec) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= t.nlat) return;
  const RowConst r = t.rows[j];
  TzRow q;
  q.a = t.slon / r.c;
  q.f = r.f;
  q.tau = r.tau;
  q.c = r.c;
  q.kg = t.slon * t.g / (t.p * r.c);
  q.kp = t.slon / (t.p * r.c);
  q.kq = t.slat / (t.q * r.c);
  q.pad = 0.0;
  rec[j] = q;
}

inline dim3 tz_flat(const TzArgs& t) {
  return dim3((unsigned)(((long long)t.nlon * t.nlat + kTzThreads - 1) / kTzThreads));
}
inline dim3 tz_grid(const TzArgs& t) { return dim3((t.nlon + 127) / 128, t.nlat); }
inline unsigned tz_blocks(long long n) {
  long long b = (n + 255) / 256;
  return (unsigned)(b < 1 ? 1 : (b > 152 * 16 ? 152 * 16 : b));
}

}  // namespace

cudaError_t launch_tz_rows(const TzArgs& t, TzRow* rec, cudaStream_t st) {
  tz_rows_kernel<<<(t.nlat + 127) / 128, 128, 0, st>>>(t, rec);
  return cudaGetLastError();
}
cudaError_t launch_tz_stage(const TzArgs& t, const double* X, const double* Y, double* out, double cx, double cy,
                            cudaStream_t st) {
  return launch_dependent(tz_stage_kernel, tz_flat(t), kTzThreads, 0, st, t, X, Y, out, cx, cy);
}
cudaError_t launch_tz_adj_stage(const TzArgs& t, const double* Y, const double* M, const double* lam,
                                const double* mu2, const double* force, double* out, cudaStream_t st) {
  return launch_dependent(tz_adj_kernel, tz_flat(t), kTzThreads, 0, st, t, Y, M, lam, mu2, force, out);
}
cudaError_t launch_tz_tl_stage(const TzArgs& t, const double* Y, const double* dX, const double* dY, double* dout,
                               double cx, double cy, cudaStream_t st) {
  tz_tl_stage_kernel<<<tz_grid(t), 128, 0, st>>>(t, Y, dX, dY, dout, cx, cy);
  return cudaGetLastError();
}
cudaError_t launch_tz_scale_add(double* out, const double* a, const double* b, const double* sigma, long long plane,
                                cudaStream_t st) {
  tz_scale_add_kernel<<<tz_blocks(3 * plane), 256, 0, st>>>(out, a, b, sigma, plane);
  return cudaGetLastError();
}
cudaError_t launch_tz_obs_misfit(const double* traj, long long n, const int* level, const int* var, const double* fi,
                                 const double* fj, const double* y, const double* so, int nlon, int nlat, double lam,
                                 double* force, double* part, cudaStream_t st) {
  tz_obs_misfit_kernel<<<kTzBlocks, 256, 0, st>>>(traj, n, level, var, fi, fj, y, so, nlon, nlat, lam, force, part);
  return cudaGetLastError();
}
cudaError_t launch_tz_obs_scatter(long long k0, long long k1, const int* var, const double* fi, const double* fj,
                                  const double* force, int nlon, int nlat, double* lam, cudaStream_t st) {
  if (k1 <= k0) return cudaSuccess;
  tz_obs_scatter_kernel<<<tz_blocks(k1 - k0), 256, 0, st>>>(k0, k1, var, fi, fj, force, nlon, nlat, lam);
  return cudaGetLastError();
}
cudaError_t launch_tz_finish_J(const double* w, long long n, int nobs, double* part, double* J, cudaStream_t st) {
  tz_background_kernel<<<kTzBlocks, 256, 0, st>>>(w, n, part + kTzBlocks);
  tz_finish_J_kernel<<<1, 128, 0, st>>>(part, nobs, J);
  return cudaGetLastError();
}

}  // namespace dd4dv
