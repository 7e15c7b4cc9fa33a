// Backprojector: launch layout per geometry, tap-item table, dispatch over the tap counts.
#include <math.h>

#include <algorithm>
#include <vector>

#include "backward.cuh"

namespace spdhg {

// Tile, staged rows and component batches of a geometry (host; fills the bw_* fields of g and
// slot / len of comp).  slots receives per batch the copies (slot, plane), then the zero slots.
void backward_layout(DevGeom& g, const SegDev* seg, CompDev* comp, std::vector<int2>& slots, std::vector<BwdBatch>& batches) {
  const double inv = g.inv_drp;
  const int pad = g.taps - 1;
  // The ends of a footprint are FP32: with d the image's diagonal, |s| <= d / 2 pixels comes with at most five
  // roundings of it and four of half its size (products, directions, sum, half width, 1 / d_radial), the bin with one
  // of R / 2; a margin below that would drop bins that cut a corner (8192 pixels at nine bins a pixel: 0.0113).
  g.bw_margin = fmaxf(kBinMargin, (float)(ldexp(1.0, -24) * (4.0 * sqrt((double)g.nx * g.nx + (double)g.ny * g.ny) * inv + g.R)));
  auto rows = [&](int cpw) {
    // a tile of 2 cpw x 4 pixels projects onto 2 cpw |c| + 4 |s| pixels of s, at most the tile's
    // diagonal; the kernel widens the row range by twice its bin margin on both sides
    const double diag = sqrt(4.0 * cpw * cpw + 16.0);
    return (int)floor(diag * inv * (1.0 + 1e-5) + 4.0 * g.bw_margin) + 1;
  };
  // Runs of staged planes.  A component whose bins hold every plane of its range has its own run,
  // followed by a frame of taps - 1 zeros.  One that holds every second plane is staged without the
  // gaps; the lane masks keep its gather inside it, so the components of a segment share one run per
  // parity and no frame.  344 x 344 x 127 voxels, 121 components over 837 planes: 8200 slots with runs
  // and gaps per component, 837 shared.
  struct Run { int seg, step, lo, hi, slot; };
  g.bw_step2 = 0;
  std::vector<int> run_of(g.n_comp);
  std::vector<Run> runs;
  for (int c = 0; c < g.n_comp; ++c) {
    const int step = 1 + comp[c].smask;
    const int hi = comp[c].qlo + (comp[c].qhi - comp[c].qlo - 1) / step * step + 1;
    comp[c].len = hi - comp[c].qlo + (step == 2 ? 1 : pad);
    g.bw_step2 |= comp[c].smask;
    int k = (int)runs.size();
    if (step == 2) {
      for (k = 0; k < (int)runs.size(); ++k)
        if (runs[k].step == 2 && runs[k].seg == comp[c].seg && ((runs[k].lo ^ comp[c].qlo) & 1) == 0) break;
    }
    if (k == (int)runs.size()) runs.push_back(Run{comp[c].seg, step, comp[c].qlo, hi, -1});
    runs[k].lo = std::min(runs[k].lo, comp[c].qlo);
    runs[k].hi = std::max(runs[k].hi, hi);
    run_of[c] = k;
  }
  // slots a component's run takes at most (a plain run may need a frame on either side)
  auto run = [&](int c) {
    const Run& q = runs[run_of[c]];
    return (q.hi - q.lo + q.step - 1) / q.step + (q.step == 1 ? 2 * pad : 0);
  };
  int widest = 0;
  for (int c = 0; c < g.n_comp; ++c) widest = std::max(widest, run(c));
  // four columns per warp share a block's set-up and a warp's item records (171 x 171: 98 us against
  // 149 with one column, 128 x 128: 35 against 40); one column per warp where four would leave fewer
  // than two blocks per SM, or rows too long for shared memory
  const long long tiles4 = (long long)((g.nx + 7) / 8) * ((g.ny + 3) / 4);
  g.bw_cpw = tiles4 >= 2 * 152 && (size_t)rows(4) * widest * sizeof(float) <= 80 * 1024 ? 4 : 1;
  g.bw_rows = rows(g.bw_cpw);
  g.bw_cand = (int)floor(1.41422 * inv + 2.0 * g.bw_margin) + 1;
  // batches of components whose staged rows fit the buffer: 36 KB leave room for four blocks per SM
  // (171 x 171 x 92, three segments: 36 KB 97.7 us, 44 KB 108.7, 24 KB 115)
  const int room = 36 * 1024 / (int)sizeof(float) / g.bw_rows;
  batches.clear();
  slots.clear();
  g.bw_buf = 0;
  for (int c = 0; c < g.n_comp;) {
    BwdBatch b{c, c, (int)slots.size(), 0, 0, pad};
    std::vector<int2> zeros;
    bool framed = true;  // the slots before the next run are a frame
    auto frame = [&]() {
      for (int k = 0; k < pad; ++k) zeros.push_back(make_int2(b.slots++, -1));
      framed = true;
    };
    b.slots = 0;
    frame();
    for (Run& q : runs) q.slot = -1;
    while (c < g.n_comp) {
      Run& q = runs[run_of[c]];
      if (q.slot < 0) {
        if (c > b.c0 && b.slots + run(c) - (q.step == 1 && framed ? pad : 0) > room) break;
        if (q.step == 1 && !framed) frame();
        q.slot = b.slots;
        for (int p = q.lo; p < q.hi; p += q.step) slots.push_back(make_int2(b.slots++, seg[q.seg].p0 + p));
        if (q.step == 1) frame();
        else framed = false;
      }
      // a step-2 record counts from the component's first plane, the others from the frame below it
      comp[c].slot = q.step == 2 ? q.slot + (comp[c].qlo - q.lo) / 2 : q.slot - pad;
      ++c;
    }
    b.c1 = c;
    b.copies = (int)slots.size() - b.first;
    b.zeros = (int)zeros.size();
    slots.insert(slots.end(), zeros.begin(), zeros.end());
    batches.push_back(b);
    g.bw_buf = std::max(g.bw_buf, (g.bw_rows * b.slots + 3) & ~3);
  }
  g.bw_nb = (int)batches.size();
  // several views per stage where their rows are short (fewer barriers, fuller records) and their pair
  // lists fit: with many bins per pixel the lists, not the rows, take the room
  g.bw_views = 1;
  if (g.bw_nb == 1) {
    const int most = g.bins ? g.V : (g.V + g.m - 1) / g.m;
    const int lists = (int)(kPairBytes / ((size_t)kBwdWarps * g.bw_cpw * g.bw_cand * sizeof(PixItem)));
    const int fit = std::max(1, std::min(std::min(16, lists), room / batches[0].slots));
    const int stages = (most + fit - 1) / fit;
    g.bw_views = (most + stages - 1) / stages;
    g.bw_buf = (g.bw_views * g.bw_rows * batches[0].slots + 3) & ~3;
  }
}

// per stage: exclusive prefix sums of the warps' item counts, and the stage's total
__global__ void __launch_bounds__(1024) k_bwd_table_scan(const unsigned short* cnt, size_t recs_per_view,
                                                         unsigned* starts, unsigned* totals) {
  __shared__ int scratch[33];
  const size_t v = blockIdx.x;
  const unsigned short* c = cnt + v * recs_per_view;
  unsigned* st = starts + v * recs_per_view;
  const size_t per = (recs_per_view + blockDim.x - 1) / blockDim.x;
  const size_t lo = min(recs_per_view, threadIdx.x * per), hi = min(recs_per_view, lo + per);
  int sum = 0;
  for (size_t k = lo; k < hi; ++k) sum += c[k];
  int total;
  int run = block_exclusive_scan(sum, scratch, &total);
  for (size_t k = lo; k < hi; ++k) {
    st[k] = (unsigned)run;
    run += c[k];
  }
  if (threadIdx.x == 0) totals[v] = (unsigned)total;
}

// one batch of at most 128 components, three taps (the item's packing), view subsets; flat geometries
// compute their few bins
bool backward_table_possible(const DevGeom& g) {
  return !g.bins && !flat_geometry(g) && g.taps <= 3 && g.bw_nb == 1 && g.n_comp <= 128;
}

size_t backward_table_recs(const DevGeom& g) {
  const dim3 t = bwd_tiles(g);
  return (size_t)t.x * t.y * kBwdWarps;
}

int backward_table_stages(const DevGeom& g) { return g.m * bwd_groups(g, 0); }

static cudaError_t table_pass(const DevGeom& g, int pass, unsigned short* cnt, unsigned* bad, const unsigned* starts,
                              const unsigned* stage_base, float4* items, int2* hdr, cudaStream_t s) {
  if (!backward_table_possible(g)) return cudaErrorInvalidValue;
  switch (g.taps) {
    case 1: return backward_items_nt<1>(g, pass, cnt, bad, starts, stage_base, items, hdr, s);
    case 2: return backward_items_nt<2>(g, pass, cnt, bad, starts, stage_base, items, hdr, s);
    default: return backward_items_nt<3>(g, pass, cnt, bad, starts, stage_base, items, hdr, s);
  }
}

cudaError_t backward_table_count(const DevGeom& g, unsigned short* cnt, unsigned* bad, cudaStream_t s) {
  return table_pass(g, 0, cnt, bad, nullptr, nullptr, nullptr, nullptr, s);
}

cudaError_t backward_table_starts(const DevGeom& g, const unsigned short* cnt, unsigned* starts,
                                  unsigned* stage_totals, cudaStream_t s) {
  k_bwd_table_scan<<<backward_table_stages(g), 1024, 0, s>>>(cnt, backward_table_recs(g), starts, stage_totals);
  return cudaGetLastError();
}

cudaError_t backward_table_fill(const DevGeom& g, const unsigned* starts, const unsigned* stage_base,
                                float4* items, int2* hdr, cudaStream_t s) {
  return table_pass(g, 1, nullptr, nullptr, starts, stage_base, items, hdr, s);
}

cudaError_t launch_backward(const DevGeom& g, int subset, int mode, const BwdArgs& a, cudaStream_t s) {
  if (a.items && !backward_table_possible(g)) return cudaErrorInvalidValue;
  if (flat_geometry(g)) return launch_backward_flat(g, subset, mode, a, s);
  switch (g.taps) {
    case 1: return launch_backward_nt<1>(g, subset, mode, a, s);
    case 2: return launch_backward_nt<2>(g, subset, mode, a, s);
    case 3: return launch_backward_nt<3>(g, subset, mode, a, s);
    case 4: return launch_backward_nt<4>(g, subset, mode, a, s);
    default: return cudaErrorInvalidValue;
  }
}

__global__ void k_gather_subset(DevGeom g, int subset, const float* __restrict__ y,
                                const float* __restrict__ mult, float* __restrict__ w) {
  const int64_t per_view = (int64_t)g.R * g.P;
  const int64_t n = (int64_t)subset_views(g, subset) * per_view;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int l = (int)(i / per_view);
    const int64_t j = (int64_t)subset_view(g, subset, l) * per_view + (i - l * per_view);
    const float v = (y ? y[j] : 1.f) * (mult ? mult[j] : 1.f);
    w[i] = bin_in_subset(g, subset, (size_t)j) ? v : 0.f;
  }
}

cudaError_t launch_gather_subset(const DevGeom& g, int subset, const float* y, const float* mult,
                                 float* w_local, cudaStream_t s) {
  const int64_t n = (int64_t)subset_views(g, subset) * g.R * g.P;
  if (n == 0) return cudaSuccess;
  int blocks = (int)((n + 255) / 256);
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_gather_subset<<<blocks, 256, 0, s>>>(g, subset, y, mult, w_local);
  return cudaGetLastError();
}

}  // namespace spdhg
