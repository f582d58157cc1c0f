// What the autotuner concludes from its timings, and which boxes the level sweeps'
// index arithmetic holds for.  Plain C++, no CUDA: the rules can be tested by
// themselves.
#pragma once

#include <vector>

namespace dd4dv {

constexpr double kNotTimed = 1e300;

// The fastest forward and adjoint sweep of each kind (ms) with one stage mode.
struct SweepTimes {
  double cluster_f = kNotTimed, cluster_a = kNotTimed, level_f = kNotTimed, level_a = kNotTimed;
};
struct SweepChoice {
  int stored = 0;                         // stage states stored (1) or recomputed (0)
  bool level_f = false, level_a = false;
  double ms = 2 * kNotTimed;
};

// The fastest pair of sweeps that can run together.  t[0]: stages recomputed,
// t[1]: stored (only where have_stored).  Under checkpoints the cluster forward
// stores some levels only, and the level adjoint, which reads every level, follows
// a level forward or does not run.
inline SweepChoice choose_sweeps(const SweepTimes (&t)[2], bool have_stored, bool checkpoints) {
  SweepChoice best;
  for (int u = 0; u <= (have_stored ? 1 : 0); ++u)
    for (int k = 0; k < 4; ++k) {
      const bool lf = k & 1, la = k & 2;
      if (checkpoints && la && !lf) continue;
      const double ms = (lf ? t[u].level_f : t[u].cluster_f) + (la ? t[u].level_a : t[u].cluster_a);
      if (ms < best.ms) best = {u, lf, la, ms};
    }
  return best;
}

// Checkpoint intervals worth timing for ckpt_k = -2.  Level sweeps store every
// level whatever the interval, and recompute the stage states alone: every
// interval would time the same kernels, and noise would choose one and keep its
// segment buffers.
constexpr int kTunedCkpt[3] = {8, 16, 32};
inline std::vector<int> checkpoint_candidates(bool level_f, bool level_a) {
  if (level_f && level_a) return {};
  return {kTunedCkpt, kTunedCkpt + 3};
}

// Whether the level sweeps' 32-bit index arithmetic is exact for a box of nx x ny
// points, rows padded to nxp, nq thread-points a row: a quotient a / d through
// magic_of(d) needs a d < 2^32 (thread-points by nq, scatter targets of three planes by
// nx, their rows by ny), an offset in a level 2^31.  Boxes that fit a cluster's
// shared memory, as every accepted box does, are far inside.
inline bool level_box_fits(long long nx, long long ny, long long nxp, long long nq) {
  const long long lim = 1LL << 32;
  return nq * ny * nq < lim && 3 * ny * nx * nx < lim && 3 * ny * ny < lim && 3 * ny * nxp < (lim >> 1);
}

}  // namespace dd4dv
