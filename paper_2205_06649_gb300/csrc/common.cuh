// Internal declarations of the DD-4DVar GB300 library (not part of the C ABI).
//
// Device data layout (HBM):
//   * per-subdomain trajectories: traj[s] = [L+1 levels][3 vars][ny rows][nxp],
//     state type T (double, or float with h stored as h - h_ref), row pitch
//     nxp = nx rounded up to a multiple of 4 so every row starts on a 32-byte
//     boundary; subdomains are packed one after another (SubDesc::traj_off);
//   * overlap targets tgt[s]: same shape, the mean of the neighbours' values
//     at every point the subdomain shares with others (zero elsewhere);
//   * boundary trajectory bnd = [nsteps+1][3][nlat][nlon] (type T), the
//     partition-of-unity sum of the local trajectories (Eq. rest);
//   * stage states stg[s] = [L steps][2 stages][3 vars][ny][nxp]: the RK3
//     intermediate states x1, x2 of every step, stored by the forward sweep so
//     that the adjoint sweep loads them instead of recomputing them;
//   * controls, gradients, L-BFGS vectors: packed FP64 [3][ny][nx] per
//     subdomain (SubDesc::ctrl_off).
#pragma once

#include <cuda_runtime.h>
#include <cstdint>
#include <mutex>
#include <set>
#include <utility>
#include <vector>

namespace dd4dv {

enum { F_PERIODIC = 1, F_SWALL = 2, F_NWALL = 4 };

struct SubDesc {
  int i0, nx, j0, ny, a, b;   // box [i0, i0+nx) (lon, mod nlon) x [j0, j0+ny), levels [a, b]
  int nxp;                    // trajectory row pitch (elements)
  int flags;                  // F_PERIODIC | F_SWALL | F_NWALL
  int q, p2, p1;              // block coordinates
  int wL, wR, wS, wN;         // overlap band widths: lon west/east, lat south/north
  int tA, tB;                 // overlap level counts at window start / end
  int obs_lvl;                // first entry of this subdomain in lvl_obs (L+2 entries)
  int sc_lvl;                 // first entry in lvl_sc (L+2 entries)
  long long ctrl_off;         // packed control offset (doubles)
  long long traj_off;         // trajectory offset (elements of T)
  long long ptraj_off;        // packed public trajectory offset (doubles, pitch nx)
  long long stg_off;          // stage-state offset (elements of T): [L][2][3][ny][nxp]
  long long stg1_off;         // offset of x1 alone (elements of T): [L][3][ny][nxp]; -1: not stored
  long long seg_off;          // checkpoint-segment buffer offset (elements of T): [k+1][3][ny][nxp]
};

struct ObsRec {               // one observation as seen by one subdomain
  int var, r0, k0, k1;        // local lower corner row/col, east corner col (wrapped)
  double di, dj;              // fractional offsets (0 = corner not used)
  double y;                   // observed value (h: minus h_ref on the FP32 path)
  double w;                   // omega / sigma_o^2
};

struct RowConst {             // per global latitude row j
  double A;                   // 1 / (2 a cos(theta_j) dlambda)
  double f;                   // 2 Omega sin(theta_j)
  double tau;                 // tan(theta_j) / a
  double c;                   // cos(theta_j)
  double BinvC;               // Bth / cos(theta_j)
  double gA;                  // g A
};

// Arguments shared by the sweep kernels (forward, adjoint, tangent-linear).
template <typename T>
struct SweepArgs {
  const SubDesc* subs;
  const int* order;           // cluster -> subdomain (longest first)
  int n_sub;
  T* traj;
  T* stg;                     // RK3 stage states x1, x2 of every step, or nullptr (recompute)
  T* stg1;                    // with stg == nullptr: x1 of every step of the subdomains whose
                              // stg1_off >= 0 (x2 recomputed), or nullptr
  int ckpt;                   // 0: every level stored; k > 0: levels 0, k, 2k, ... stored and
                              // each k-step segment recomputed in the adjoint
  T* seg;                     // per-subdomain segment buffers for the recomputation
  const T* tgt;
  const T* bnd;
  const RowConst* rows;       // [nlat]
  double Bth, gBth, dt, h_ref;
  int nlon, nlat, nsteps;
  double isb2[3];             // 1 / sigma_b^2 per variable
  double lam, mu;
  // the same constants rounded once to the state precision on the host, so
  // that the FP32 sweeps run no FP64 conversion per stage or level
  T dt_s, Bth_s, gBth_s, href_s;
  T Bth_a, gBth_a;            // for the adjoint point functions (FP64: times dt)
  T isb2_s[3], musb2_s[3];    // 1 / sigma_b^2 and mu / sigma_b^2
  const ObsRec* obs;          // per-subdomain, per-level sorted
  const int* lvl_obs;         // obs ranges per (subdomain, level)
  double* obs_force;          // lambda * omega * d / sigma_o^2 per obs record
  const int* sc_tgt;          // adjoint scatter targets: var*ny*nx + r*nx + k
  const int* sc_off;          // contributions of each target
  const int* sc_obs;
  const double* sc_w;
  const int* lvl_sc;          // target ranges per (subdomain, level)
  double* part;               // [n_sub][cl_max][2] partial J_o, J_mu
  int cl_max;
  const int* active;          // per-subdomain mask (phase == active_value), or nullptr
  int active_value;
  double* lam_a;              // adjoint state at level a, packed control layout
  const double* yforce;       // external adjoint forcing (packed FP64 trajectories) or nullptr
  double* dx_out;             // tangent-linear output (packed FP64 trajectories)
  const double* dx0;          // tangent-linear initial perturbation (packed control layout)
  T* gn_dx;                   // Gauss-Newton products: the tangent-linear sweep stores dx here
                              // (trajectory layout) and sets obs_force = lambda w H dx; the
                              // adjoint sweep then takes its overlap forcing mu c dx / sb^2
                              // from it instead of mu c (x - m) / sb^2
  int R;                      // max rows per CTA
  int W;                      // shared-memory row pitch (>= max nx + 2)
  int* err;                   // device error word (0 = ok)
  int tgb_on;                 // set by the launcher: the FP32 sweep's shared memory holds a
                              // buffer of prefetched overlap targets (only if it still fits)
  int min_ny;                 // smallest box height of the decomposition
  int variant;                // 0: deep-halo FP32 sweeps where they apply, else the stripe
                              // sweeps; 1: stripe sweeps only; 2: the stripe adjoint with
                              // four state buffers (x(n) reloaded from HBM), the stripe
                              // forward with two (x(n) read from the stored level)
};

// Largest CTA of the stripe forward sweep: 384 threads on the FP32 path,
// whose forward kernel is compiled for up to 80 registers (2 CTAs of 384
// threads per SM), 1024 on the FP64 path (64 registers, one CTA of 1024 or two
// of 512 per SM).  The stripe adjoint takes up to 1024 threads (64 registers).
template <typename T> constexpr int max_threads_forward() { return sizeof(T) == 4 ? 384 : 1024; }
template <typename T> constexpr int min_blocks_forward() { return sizeof(T) == 4 ? 2 : 1; }
constexpr int kStripeAdjThreads = 1024;

// ---- programmatic dependent launch ----
// A chain of kernels on one stream whose set-up may overlap the end of the
// kernel before: every thread of every such kernel calls grid_wait before it
// reads what earlier kernels wrote, also where it then has nothing to do, so
// that a grid never ends before the ones it follows.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// Raises a kernel's dynamic shared-memory cap to the 227 KB opt-in maximum less
// its static part, once per (kernel, device) and never down again: the attribute
// belongs to the process, and another thread may be about to launch the kernel
// with more than this caller needs.  (It is set on the device current at the
// call, so a context on another device sets it again.)
template <typename K>
cudaError_t raise_smem_cap(K kernel) {
  static std::mutex mu;
  static std::set<std::pair<const void*, int>> done;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  const std::pair<const void*, int> key{reinterpret_cast<const void*>(kernel), dev};
  if (done.count(key)) return cudaSuccess;
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448 - (int)fa.sharedSizeBytes);
  if (e != cudaSuccess) return e;
  done.insert(key);
  return cudaSuccess;
}

// ---- launchers (sweep.cu) ----
// Which kernel a sweep launch with cl CTAs per subdomain and nthreads threads
// per CTA would run: 0 = none (shape not launchable), 1 = the stripe sweep
// (one halo row per stage), 2 = the deep-halo FP32 sweep (three halo rows, one
// exchange per step), 3 = the stripe adjoint with four state buffers, 4 =
// the stripe forward with two state buffers.
template <typename T> int forward_kind(const SweepArgs<T>& a, int cl, int nthreads);
template <typename T> int adjoint_kind(const SweepArgs<T>& a, int cl, int nthreads);
template <typename T> cudaError_t launch_forward(const SweepArgs<T>& a, int cl, int nthreads, cudaStream_t st);
template <typename T> cudaError_t launch_adjoint(const SweepArgs<T>& a, int cl, int nthreads, cudaStream_t st);
template <typename T> cudaError_t launch_tlm(const SweepArgs<T>& a, int cl, int nthreads, cudaStream_t st);
template <typename T> size_t smem_forward(int R, int W);
template <typename T> size_t smem_adjoint(int R, int W);
template <typename T> size_t smem_adjoint_rl(int R, int W);
template <typename T> size_t smem_tlm(int R, int W);
// resident clusters of the stripe adjoint sweep at cl CTAs per cluster
template <typename T> int active_clusters_adjoint(int R, int W, int cl, int nthreads);

// Device error words: 1 and 2, a cluster sweep rejected its launch (sweep.cu); 3, a
// wait of a pipelined level kernel ran out (level.cu).
constexpr int kErrLostCopy = 3;

// ---- level sweeps (level.cu) ----
// One tile: the thread-points [p0, p1) of one box (a thread-point is V
// neighbouring columns of a row), with everything of the box a kernel needs.
struct LvTile {
  int s, p0, p1;
  int nx, ny, nxp, nq;        // nq: thread-points per row
  unsigned mq, mnx, mny;      // multipliers for division by nq, nx, ny
  int i0, j0, a, L, flags;
  int iw, ie;                 // global columns of the west / east frozen ghosts
  int wL, wR, wS, wN, tA, tB;
  int sc_lvl;
  long long traj_off, ptraj_off, stg_off, stg1_off, ctrl_off;
  long long lv_off;           // one-level scratch offset (elements of T): [3][ny][nxp]
};
// A pipelined kernel's CTAs (at most), slots, floats per slot and before the
// slots; slots = 0: the plain kernel runs.
struct LvRing {
  int ctas = 0, slots = 0, slot_floats = 0, own_floats = 0;
};
// The tiles of every box, longest window first.
struct LvPlan {
  int tiles = 0;
  LvRing ring[3];                       // adjoint phases 1, 2, 3
  const LvTile* ring_tiles = nullptr;   // their tiles: whole rows
  bool ring_expire = false;             // their waits run out at once (a test of what follows)
  std::vector<int> n_ring;              // as n_tile
  // tiles of one round, for the kernels that add nothing up (null: the same tiles)
  const LvTile* fine_tiles = nullptr;
  int fine = 0;
  std::vector<int> n_fine;
  std::vector<int> n_tile;    // per step l: tiles of the boxes that take it (a prefix)
  std::vector<int> n_box;     // per level l: boxes that have it (a prefix of the box list)
  std::vector<char> obs;      // per level l: some box has observations there
};
template <typename T>
struct LvArgs {
  const LvTile* tiles;
  const int* boxes;           // longest window first
  const long long* box_off;   // lv_off of every box
  const SubDesc* subs;
  int n_tile;
  int n_cta, slots, slot_floats;   // pipelined kernels: CTAs, ring
  int* err;                   // device error word (0 = ok)
  int* late;                  // the same for lost copies in host memory: read without a synchronisation
  int l;                      // step / level
  int terms;                  // forward: accumulate the observation and overlap terms
  int skip1;                  // first stage recomputed only where x1 is not stored
  int mu_on;                  // mu != 0
  T *traj, *stg, *stg1;
  T *x1s, *x2s, *lam, *mu2, *mu1;   // one-level scratch states of every box
  const T *tgt, *bnd, *gn_dx;
  const T *fw, *bw;           // row constants [nlat][8] (the records of sweep.cu)
  T dt, Bth, gBth, href;
  T Bth_a, gBth_a;            // for the adjoint point functions (FP64: times dt)
  T isb2[3], musb2[3];
  int nlon, nlat;
  double lam_w;               // weight lambda of the observation term
  const ObsRec* obs;
  const int* lvl_obs;
  double* obs_force;
  const int *sc_tgt, *sc_off, *sc_obs, *lvl_sc;
  const double* sc_w;
  double *acc_m, *acc_o;      // per tile and thread: twice J_mu; per box: J_o
  const int* active;
  int active_value;
  double* lam_a;
  const double* yforce;
  T* dx;                      // tangent-linear sweep: dx (trajectory layout), and
  const double* dx0;          // dx(a), packed control layout
};
// Columns per thread: FP32 threads take four neighbouring points (16-byte
// accesses), FP64 threads one.
template <typename T> __host__ __device__ constexpr int lv_width() { return sizeof(T) == 4 ? 4 : 1; }
constexpr int kLvThreads = 128;
constexpr int kRingThreads = 256;   // pipelined kernels: a thread-point for each of the
constexpr int kRingPoints = 224;    // first 224 threads, the last warp copies
template <typename T>
cudaError_t launch_level_forward(const LvArgs<T>& a, const LvPlan& g, cudaStream_t st, long long* launches);
template <typename T>
cudaError_t launch_level_adjoint(const LvArgs<T>& a, const LvPlan& g, cudaStream_t st, long long* launches);

// tangent-linear sweep of a Gauss-Newton product (a.dx, obs_force from a.dx0)
cudaError_t launch_level_tangent(const LvArgs<double>& a, const LvPlan& g, cudaStream_t st, long long* launches);

// ---- auxiliary kernels (aux.cu) ----
struct RFArgs {
  const SubDesc* subs; int n_sub;
  double alpha, c; int npass;
  const int* active; int active_value;
};
// in place: lines along lon (rows) or lat (columns) of each [3][ny][nx] block
cudaError_t launch_rf_rows(double* x, const RFArgs& a, int max_ny, cudaStream_t st);
cudaError_t launch_rf_cols(double* x, const RFArgs& a, int max_nx, cudaStream_t st);

// fused V / V^T (one CTA per subdomain and variable, plane in shared memory)
template <typename T>
cudaError_t launch_vinit(const SubDesc* subs, int n_sub, const double* xb_a, const double* w,
                         const double* sigma, const RFArgs& rf, int use_rf, double h_ref, T* traj,
                         const int* active, int active_value, int max_plane, cudaStream_t st);
// R = precision of the recursive filter (the state precision)
template <typename R>
cudaError_t launch_vgrad(const SubDesc* subs, int n_sub, const double* w, const double* y, const double* sigma,
                         const RFArgs& rf, int use_rf, const double* scale, double* grad, const int* active,
                         int active_value, int max_plane, cudaStream_t st);
template <typename T>
cudaError_t launch_init_state(const SubDesc* subs, int n_sub, const double* xb_a, const double* vw,
                              const double* sigma, int scale_sigma, double h_ref, T* traj,
                              const int* active, int active_value, int max_pts, cudaStream_t st);
cudaError_t launch_scale_copy(const SubDesc* subs, int n_sub, const double* in, const double* sigma,
                              double* out, const int* active, int active_value, int max_pts,
                              cudaStream_t st);
cudaError_t launch_grad_finish(const SubDesc* subs, int n_sub, const double* w, const double* vty,
                               const double* scale, double* grad, const int* active,
                               int active_value, int max_pts, cudaStream_t st);
cudaError_t launch_finalize_J(const SubDesc* subs, int n_sub, const double* w, const double* part,
                              int cl_max, const double* vconst, double lam, double mu, double* J,
                              double* parts, const int* active, int active_value, cudaStream_t st);
// the same after a level forward sweep: J_o per box, twice J_mu in the box's
// tile_off[2 s + 1] slots from tile_off[2 s]
cudaError_t launch_finalize_J_tiles(const SubDesc* subs, int n_sub, const double* w, const double* acc_o,
                                    const double* acc_m, const int* tile_off, const double* vconst, double lam,
                                    double mu, double* J, double* parts, const int* active, int active_value,
                                    cudaStream_t st);

template <typename T>
struct ExchArgs {
  const SubDesc* subs; int n_sub;
  int P1, P2, Q;
  int nlon, nlat, nsteps;
  const T* traj; T* tgt; T* bnd;
  double isb2[3];
  double* vpart;              // [n_sub][blocks] partial sums of the overlap constant
  int vblocks;
  const int* lon_cov;         // [nlon][2][2] (p1, local col) or -1
  const int* lat_cov;         // [nlat][2][2]
  const int* t_cov;           // [nsteps+1][2][2]
};
template <typename T> cudaError_t launch_targets(const ExchArgs<T>& a, cudaStream_t st);
template <typename T> cudaError_t launch_assemble(const ExchArgs<T>& a, cudaStream_t st);
cudaError_t launch_sum_vconst(const double* vpart, int n_sub, int vblocks, double* vconst, cudaStream_t st);

template <typename T>
cudaError_t launch_restrict(const SubDesc* subs, int n_sub, int nlon, int nlat, const double* glob,
                            int g0, int g1, double h_ref, T* traj, int max_pts, cudaStream_t st);
template <typename T>
cudaError_t launch_export_traj(const SubDesc* subs, int n_sub, const T* traj, double h_ref,
                               double* out, int max_pts, int max_levels, cudaStream_t st);
template <typename T>
cudaError_t launch_bnd_from_global(const double* glob, long long n, double h_ref, int nlon, int nlat,
                                   T* bnd, cudaStream_t st);
template <typename T>
cudaError_t launch_bnd_to_global(const T* bnd, long long n, double h_ref, int nlon, int nlat,
                                 double* glob, cudaStream_t st);
cudaError_t launch_restrict_level(const SubDesc* subs, int n_sub, int nlon, int nlat, const double* glob,
                                  int g0, int g1, double* xb_a, int max_pts, cudaStream_t st);

// global model (whole sphere), FP64
// rec: records of every row (fill_global_record of point.cuh, 8 doubles a row)
struct GlobalStepPlan {
  int tx = 0, ty = 0;         // tile of the step kernel; 0: one launch per stage
};
GlobalStepPlan global_step_plan(int nlon, int nlat);
// one RK3 step x -> nx; s1, s2: scratch states of the stage kernels
cudaError_t launch_global_step(const GlobalStepPlan& plan, const double* x, double* s1, double* s2, double* nx,
                               const double* rec, double dt, double Bth, double gBth, int nlon, int nlat,
                               cudaStream_t st, long long* launches);
cudaError_t launch_observe(const double* traj, int g0, int g1, long long n, const int* level,
                           const int* var, const double* fi, const double* fj, int nlon, int nlat,
                           double* out, cudaStream_t st);

// L-BFGS (batched, one block per subdomain)
struct LbState {
  double J, Jt, gp, alpha, g0n, gn;
  int head, count, iter, trial, phase, status;
};
struct LbArgs {
  const SubDesc* subs; int n_sub;
  double* w; double* g; double* wt; double* gt; double* p;
  double* S; double* Y; double* rho;   // [m][total], [m][total], [n_sub][m]
  long long total;
  LbState* st;
  const double* J_eval;                // J of the last evaluation
  int m, max_iter, max_trials;
  double gtol, c1;
  int* counter;                        // [2]: # in line search, # needing a direction
  int* phase;                          // [n_sub] mirror of LbState::phase (sweep masks)
  const int* owned;                    // [n_sub] 1 = this context solves the subdomain, or nullptr
};
cudaError_t launch_lb_start(const LbArgs& a, cudaStream_t st);
cudaError_t launch_lb_direction(const LbArgs& a, cudaStream_t st);
cudaError_t launch_lb_linesearch(const LbArgs& a, cudaStream_t st);
// Batched conjugate gradients for the Gauss-Newton normal equations, one
// block per subdomain (fixed-order block reductions).
struct CgState {
  double rr, rr0, g0n;
  int k, status;   // status: 0 running, 1 converged, 2 iteration limit, 3 p.Ap <= 0, 4 skipped
};
struct CgArgs {
  const SubDesc* subs; int n_sub;
  const double* g;                     // gradient at the linearisation point (rhs = -g)
  double *r, *p, *Ap, *dw;             // packed control layout
  CgState* st;
  int* phase;                          // [n_sub] 1 = solving (sweep mask)
  int* counter;                        // # still solving
  int max_iter, first;                 // first: this is the first Gauss-Newton iteration
  double tol, gtol;
};
cudaError_t launch_cg_start(const CgArgs& a, cudaStream_t st);
cudaError_t launch_cg_step(const CgArgs& a, cudaStream_t st);
cudaError_t launch_axpy(double* y, const double* x, long long n, cudaStream_t st);   // y += x
cudaError_t launch_max_abs_diff(const double* a, const double* b, long long n, double* out,
                                cudaStream_t st);
cudaError_t launch_finite_check(const double* a, long long n, int* flag, cudaStream_t st);

// ---- Turkel-Zwas scheme on the whole sphere (tz.cu) ----
struct TzRow {                // per latitude row
  double a, f, tau, c;        // s_lon / c, f, tau, c
  double kg, kp, kq, pad;     // s_lon g / (p c), s_lon / (p c), s_lat / (q c)
};
struct TzArgs {
  const RowConst* rows;       // [nlat]
  const TzRow* rec;           // [nlat] (launch_tz_rows)
  int nlon, nlat, p, q;
  double alpha, slon, slat, g, dt;
  double gq;                  // s_lat g / q
};
cudaError_t launch_tz_rows(const TzArgs& t, TzRow* rec, cudaStream_t st);
cudaError_t launch_tz_stage(const TzArgs& t, const double* X, const double* Y, double* out, double cx, double cy,
                            cudaStream_t st);
cudaError_t launch_tz_tl_stage(const TzArgs& t, const double* Y, const double* dX, const double* dY, double* dout,
                               double cx, double cy, cudaStream_t st);
// out = M + dt F'(Y)^T M; with lam and mu2 given, the transposed step's last
// phase: out = lam / 3 + mu2 / 2 + (M + dt F'(Y)^T M) / 6 (+ force; out may be lam)
cudaError_t launch_tz_adj_stage(const TzArgs& t, const double* Y, const double* M, const double* lam,
                                const double* mu2, const double* force, double* out, cudaStream_t st);
cudaError_t launch_tz_scale_add(double* out, const double* a, const double* b, const double* sigma, long long plane,
                                cudaStream_t st);
// blocks of the observation misfit and of the background term (partial sums)
constexpr int kTzBlocks = 128;
cudaError_t launch_tz_obs_misfit(const double* traj, long long n, const int* level, const int* var, const double* fi,
                                 const double* fj, const double* y, const double* so, int nlon, int nlat, double lam,
                                 double* force, double* part, cudaStream_t st);
cudaError_t launch_tz_obs_scatter(long long k0, long long k1, const int* var, const double* fi, const double* fj,
                                  const double* force, int nlon, int nlat, double* lam, cudaStream_t st);
// J = 1/2 w.w + sum of the misfit's kTzBlocks partial sums in part[0 ..] (none: nobs = 0);
// part[kTzBlocks ..] is scratch
cudaError_t launch_tz_finish_J(const double* w, long long n, int nobs, double* part, double* J, cudaStream_t st);

}  // namespace dd4dv
