// Forward projector: plane tasks and launch shapes of a geometry, dispatch over the tap counts.
#include <algorithm>
#include <vector>

#include "forward.cuh"

namespace spdhg {

// Plane tasks of a geometry (host): every segment's planes in words of 32, at most four words a task.
void forward_layout(DevGeom& g, const SegDev* seg, std::vector<int4>& tasks) {
  tasks.clear();
  for (int k = 0; k < g.n_seg; ++k) {
    const int words = (seg[k].n + 31) / 32, n = (words + 3) / 4;
    for (int t = 0, w = 0; t < n; ++t) {
      const int take = (words - w + n - t - 1) / (n - t);
      tasks.push_back(make_int4(k, 32 * w, take, 0));
      w += take;
    }
  }
  g.n_tasks = (int)tasks.size();
  g.max_part_comps[0] = 1;
  for (int per = 1; per <= kFwdMaxWarps; ++per) {
    // most components spanned by the tasks of one block
    int mx = 1;
    for (int t0 = 0; t0 < g.n_tasks; t0 += per) {
      const SegDev& lo = seg[tasks[t0].x];
      const SegDev& hi = seg[tasks[std::min(g.n_tasks, t0 + per) - 1].x];
      mx = std::max(mx, hi.c0 + hi.nc - lo.c0);
    }
    g.max_part_comps[per] = mx;
  }
}

int forward_split(const DevGeom& g, int subset) {
  if (flat_geometry(g)) return 1;
  if (g.tune[SPDHG_TUNE_FWD_SPLIT]) return g.tune[SPDHG_TUNE_FWD_SPLIT];
  // enough blocks for every SM: one LOR line per block is too few for small subsets
  const int lines = subset_views(g, subset) * g.R * forward_parts(g);
  const int nrows = g.nx > g.ny ? g.nx : g.ny;
  int split = 1;
  while (split < 8 && lines * split < 152 && nrows / (split * 2) >= 32) split *= 2;
  return split;
}

// plane tasks per block: one per warp, parts of near-equal size
int forward_tasks_per_part(const DevGeom& g) {
  const int knob = g.tune[SPDHG_TUNE_FWD_WARPS], most = knob && knob < kFwdMaxWarps ? knob : kFwdMaxWarps;
  const int parts = (g.n_tasks + most - 1) / most;
  return (g.n_tasks + parts - 1) / parts;
}

int forward_parts(const DevGeom& g) {
  const int per = forward_tasks_per_part(g);
  return (g.n_tasks + per - 1) / per;
}

// entry groups per block: four warps per block where the tasks of a part need at most two (128 x 128 x
// 64, three components: 39 us with four warps, 47 with six, 50 with eight)
int forward_entry_groups(const DevGeom& g) {
  const int per = forward_tasks_per_part(g);
  int eg = g.tune[SPDHG_TUNE_FWD_GROUPS] ? g.tune[SPDHG_TUNE_FWD_GROUPS] : std::max(1, 4 / per);
  while (eg > 1 && per * eg > kFwdMaxWarps) --eg;
  return eg;
}

cudaError_t launch_forward(const DevGeom& g, int subset, int mode, const FwdArgs& a, cudaStream_t s) {
  if (flat_geometry(g)) return launch_forward_flat(g, subset, mode, a, s);
  switch (g.taps) {
    case 1: return launch_forward_nt<1>(g, subset, mode, a, s);
    case 2: return launch_forward_nt<2>(g, subset, mode, a, s);
    case 3: return launch_forward_nt<3>(g, subset, mode, a, s);
    case 4: return launch_forward_nt<4>(g, subset, mode, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace spdhg
