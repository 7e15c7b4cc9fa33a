// Gather-based backprojector, fused with the dual-sum update and the next primal step of SPDHG.
// One translation unit per tap count NT instantiates launch_backward_nt / backward_items_nt.
#pragma once

#include <algorithm>

#include "lor.cuh"

namespace spdhg {

constexpr int kBwdWarps = 8;      // warps per block: 2 in x, 4 in y, CPW columns in x each
constexpr int kBwdFill = 32;      // item records a warp holds at a time (one per lane)
constexpr size_t kPairBytes = 48 * 1024;   // most of the warps' pair lists: what a kernel has by default
constexpr size_t kBwdMaxSmem = 220 * 1024;
constexpr int kSumItems = 12;     // records of several taps a column sums before the sum joins the others
constexpr float kBinMargin = 0.01f;   // radial bins: least margin of the footprint ends (backward_layout)

// A (bin, pixel interval) pair: the LOR lines of radial bin r of one view of the stage that cross
// a voxel column; row is the bin's row among the staged rows.
struct PixItem {
  int r, row;
  PixInt I;
};

// Radial rows [r_min, r_max] of view direction cs that the tile of TX x TY columns at (tx0, ty0)
// can touch: the span of its pixels' footprints, with a margin above the columns' own.
__device__ __forceinline__ int tile_rows(const DevGeom& g, const float4 cs, int tx0, int ty0, int TX, int TY, int* r_min) {
  const float Xm = (float)tx0 + 0.5f * (float)TX - 0.5f * (float)g.nx;
  const float Ym = (float)ty0 + 0.5f * (float)TY - 0.5f * (float)g.ny;
  const float mid = Xm * cs.x + Ym * cs.z;
  const float hw = 0.5f * ((float)TX * fabsf(cs.x) + (float)TY * fabsf(cs.z));
  *r_min = max(0, (int)ceilf((mid - hw) * g.inv_drp + g.half_R - 2.f * g.bw_margin));
  return min(g.R - 1, min(*r_min + g.bw_rows - 1, (int)floorf((mid + hw) * g.inv_drp + g.half_R + 2.f * g.bw_margin)));
}

// The stages of a subset: its views are cut into groups of near-equal size.
__device__ __forceinline__ int group_first(int group, int nviews, int groups) { return group * nviews / groups; }

// The warp's pairs for the nv views from l0 on, column-major: candidate bins of its CPW columns
// (lanes = column, view, candidate) are tested with pixel_interval and compacted into pix.
// counts: pairs per column.
template <int CPW>
__device__ __forceinline__ int warp_pairs(const DevGeom& g, int subset, int l0, int nv, int tx0, int ty0, int ix0, int iy,
                                          int lane, PixItem* pix, int counts[CPW]) {
  const int nc = g.bw_cand, per_col = nv * nc;
  const float Yc = (float)iy + 0.5f - 0.5f * (float)g.ny;
#pragma unroll
  for (int c = 0; c < CPW; ++c) counts[c] = 0;
  int np = 0;
  for (int i0 = 0; i0 < CPW * per_col; i0 += 32) {
    const int i = i0 + lane;
    const int col = i / per_col, rem = i - col * per_col, vi = rem / nc, cand = rem - vi * nc;
    const int ix = ix0 + col;
    bool ok = false;
    PixItem P;
    if (col < CPW && ix < g.nx && iy < g.ny) {
      const int v = subset_view(g, subset, l0 + vi);
      const float4 cs = g.view[v];
      int r_min;
      const int r_max = tile_rows(g, cs, tx0, ty0, 2 * CPW, 4, &r_min);
      const float hw = 0.5f * (fabsf(cs.x) + fabsf(cs.z));
      const float Xc = (float)ix + 0.5f - 0.5f * (float)g.nx;
      const float sc = Xc * cs.x + Yc * cs.z;
      const int r = (int)ceilf((sc - hw) * g.inv_drp + g.half_R - g.bw_margin) + cand;
      const int rhi = (int)floorf((sc + hw) * g.inv_drp + g.half_R + g.bw_margin);
      if (r >= r_min && r <= r_max && r <= rhi) {
        ok = pixel_interval(g, make_line(g, v, r), ix, iy, P.I);
        P.r = r;
        P.row = vi * g.bw_rows + r - r_min;
      }
    }
    const unsigned mask = __ballot_sync(0xffffffffu, ok);
    if (ok) pix[np + __popc(mask & ((1u << lane) - 1u))] = P;
#pragma unroll
    for (int c = 0; c < CPW; ++c) counts[c] += __popc(__ballot_sync(0xffffffffu, ok && col == c));
    np += __popc(mask);
  }
  return np;
}

// 32-bit mask of the lanes b with 0 <= b + off < len
__device__ __forceinline__ unsigned lane_range(int off, int len) {
  unsigned m;
  asm("bmsk.clamp.b32 %0, %1, %2;" : "=r"(m) : "r"(max(-off, 0)), "r"(max(min(len - off, len), 0)));
  return m;
}

// Item record word: 4 x (staged offset + kOffBias) | (taps - 1).  The words of step-2 components are marked
// kStep2; their low bits are a parity and kMoreTaps.
constexpr int kOffBias = 256;
constexpr unsigned kStep2 = 1u << 31, kMoreTaps = 2u;

// Word of an item whose tap 0 meets, in lane b, slot b + jp of a run of len lanes from row_slot on; `lanes`
// lanes (at most kOffBias) look at it, `taps` of its taps have a weight.  A component's planes may lie
// wholly above or below the image's slices: then no lane is in the run, the offset does not matter and may be
// too low for the bias, so that the word would carry the mark of a step-2 component.  Such an item becomes
// one without lanes at offset 0.  jp and len are what the masks are made of: lanes b with 0 <= b + jp < len,
// and with 0 <= b + jp + 2 < len for the taps above the second of a step-2 component.
__host__ __device__ inline unsigned item_word(int row_slot, int& jp, int& len, int taps, int lanes, int pad, bool step2) {
  if (step2) jp -= pad - 1;  // tap 1 of lane b meets plane b + jp of the component, if that is even
  const bool more = step2 && taps > 2;
  if (jp >= len || jp + (more ? 2 : 0) <= -lanes) {
    jp = len = 0;
    taps = 1;
  }
  if (!step2) return (unsigned)(4 * (row_slot + jp + kOffBias) | (taps - 1));
  return (unsigned)(4 * (row_slot + (jp >> 1) + kOffBias) | (jp & 1)) | (taps > 2 ? kMoreTaps : 0u) | kStep2;
}

// lane masks per record: one set, and one for the taps above the second of a step-2 component
template <int NT, bool MASHED>
__host__ __device__ constexpr int mask_sets() {
  return MASHED && NT > 2 ? 2 : 1;
}

// One tap of ZK slices: acc[k] += L * shared[addr + STRIDE k + OFF] in the lanes that m[k] holds.  The
// predicates are explicit because the compiler turns the equivalent branches into jumps.
template <int ZK, int OFF, int STRIDE = 128>
__device__ __forceinline__ void tap_fma(unsigned addr, float L, const unsigned* m, unsigned bit, float* acc) {
#pragma unroll
  for (int k = 0; k < ZK; ++k)
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t.reg .f32 f;\n\t"
        "and.b32 t, %1, %2;\n\t"
        "setp.ne.u32 p, t, 0;\n\t"
        "@p ld.shared.f32 f, [%3];\n\t"
        "@p fma.rn.f32 %0, %4, f, %0;\n\t}\n"
        : "+f"(acc[k])
        : "r"(m[k]), "r"(bit), "r"(addr + (OFF + STRIDE * k)), "f"(L));
}

// Accumulates one column's item records [i0, i1): voxel lane + 32 k adds sum_t L_t buf[off + lane +
// 32 k + t] where bit `lane` of the item's mask k is set.  `base` is the shared address of the
// buffer's slot lane - kOffBias.  A step-2 component holds planes of one parity, staged without
// gaps, so every second one of a lane's taps meets a plane: with u = lane + parity the lane reads slot
// u >> 1 in place of lane, at tap 0 where u is odd and tap 1 where it is even, and if the item has more
// than two taps also the slot after it, with masks of its own, at tap 2 or 3.  A tap of no weight
// reads nothing, so that no plane outside the LOR's slices is touched.
template <int NT, int ZK, bool MASHED>
__device__ __forceinline__ void gather_items(unsigned base, const float4* recA, const uint4* recM, const int* recO,
                                             int i0, int i1, unsigned bit, float* acc) {
  constexpr int MQ = (ZK + 3) / 4, MR = MQ * mask_sets<NT, MASHED>();
#pragma unroll 1
  for (int it = i0; it < i1; ++it) {
    const float4 A = recA[it];
    const unsigned word = NT > 3 ? (unsigned)recO[it] : __float_as_uint(A.w);
    const unsigned addr = base + (word & ~(kStep2 | 3u));
    unsigned m[4 * MQ];
#pragma unroll
    for (int q = 0; q < MQ; ++q) {
      const uint4 u = recM[it * MR + q];
      m[4 * q] = u.x;
      m[4 * q + 1] = u.y;
      m[4 * q + 2] = u.z;
      m[4 * q + 3] = u.w;
    }
    if constexpr (MASHED) {
      if (word & kStep2) {
        const int lane = threadIdx.x & 31, u = lane + (int)(word & 1u);
        const unsigned half = addr + 4 * ((u >> 1) - lane);
        const bool odd = u & 1;
        const float L = odd ? A.x : A.y;
        tap_fma<ZK, 0, 64>(half, L, m, L != 0.f ? bit : 0u, acc);
        if constexpr (NT > 2) {
          if (word & kMoreTaps) {
#pragma unroll
            for (int q = 0; q < MQ; ++q) {
              const uint4 v = recM[it * MR + MQ + q];
              m[4 * q] = v.x;
              m[4 * q + 1] = v.y;
              m[4 * q + 2] = v.z;
              m[4 * q + 3] = v.w;
            }
            const float L2 = odd ? A.z : (NT > 3 ? A.w : 0.f);
            tap_fma<ZK, 4, 64>(half, L2, m, L2 != 0.f ? bit : 0u, acc);
          }
        }
        continue;
      }
    }
    tap_fma<ZK, 0>(addr, A.x, m, bit, acc);
    if constexpr (NT > 1) {
      if (word & 3u) {
        tap_fma<ZK, 4>(addr, A.y, m, bit, acc);
        if constexpr (NT > 2) {
          if (word & 2u) {
            tap_fma<ZK, 8>(addr, A.z, m, bit, acc);
            if constexpr (NT > 3) {
              if ((word & 3u) == 3u) tap_fma<ZK, 12>(addr, A.w, m, bit, acc);
            }
          }
        }
      }
    }
  }
}

// Loads that must be issued where they stand (the compiler would sink them to their use).
__device__ __forceinline__ float ld_now(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

// Backprojection.  A block of 8 warps owns a tile of 2 CPW x 4 voxel columns, warp w the CPW
// columns at (w & 1, w >> 1).  Work is cut into stages (view group, component batch): the radial
// rows of the group's views that the tile's footprints touch are copied into shared memory
// (cp.async) as runs of planes (backward_layout), those of plain segments framed by NT - 1 zeros.  The
// (bin, interval, component) items of a warp's columns are read from the table spdhg_setup builds
// (TAB) or computed, one item per lane, and expanded to records in shared memory; a column's records are
// then accumulated with lanes along z, 32 slices per register; records of several taps kSumItems at a time.  A
// record carries, per 32 slices, the mask of the lanes whose planes lie in the run: one AND decides a lane,
// and words outside the run cost no shared-memory read.  In the last stage each column's x, z, T are
// requested before its gather and its epilogue follows at once, so the epilogue traffic of some
// warps overlaps the gathers of the others.  Between stages the sums rest in shared memory; with one
// stage in all (SINGLE) they never leave registers.
//
// Bound: instruction issue (76 % active at the mMR scale; the gather is half of the 82 M warp
// instructions, the rest is set-up, staging, records and the epilogue), so four columns share a
// warp's set-up and several views share a stage.  Measured on GB300: 344 x 344 x 127 voxels, one
// view of 344 x 837 bins, BWD_UPDATE 137 -> 100 us (302 MB algorithmic, 3.0 TB/s) against a block of
// 16 one-column warps whose epilogues ran in step; 171 x 171 x 92, 12-13 views x 250 planes,
// 128 -> 95 us; 128 x 128 x 64, 8-9 views, three mashed components, 51 -> 36 us; 64 x 64 x 1, 9 views,
// 19 -> 12 us; 344 x 344 x 127, one view, 121 components over 837 planes (BWD_OUT) 767 -> 747 us
// (870 when every component had its own gapped run).  Two buffers per block (the next stage's copies in flight) gave nothing over one:
// the other blocks of the SM cover the wait.  Frames of 31 zeros instead of lane masks (8-byte
// records, no masks) took the same time and room for fewer views.  Five blocks per SM spill.
// Error of the mMR backprojection against FP64, and its time with computed items: one running sum per
// column 9.10e-8, 96.5 us; sums of 8, 12, 16, 32 records 8.67, 8.83, 8.90, 8.99e-8 and 101.9, 99.6, 99.4, 98.3 us;
// each item's taps summed first 8.92e-8, 110 us.  Columns of more records gain more.  With one tap a record rounds
// once, so that one running sum is the closer one already (128 x 128 x 64, OSEM: 855 us, 875 in sums of twelve).
template <int NT, int ZK, int CPW, bool SINGLE, bool TAB, bool MASHED>
__global__ void __launch_bounds__(kBwdWarps * 32, ZK <= 4 ? 4 : 3)
    k_backward(const __grid_constant__ DevGeom g, int subset, int groups, int mode, const __grid_constant__ BwdArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int PAD = NT - 1;
  constexpr int MQ = (ZK + 3) / 4, MR = MQ * mask_sets<NT, MASHED>();
  constexpr int TX = 2 * CPW, TY = 4;
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const unsigned bit = 1u << lane;
  float4* recA = reinterpret_cast<float4*>(smem) + wi * kBwdFill;
  uint4* recM = reinterpret_cast<uint4*>(smem + kBwdWarps * kBwdFill * 16) + wi * kBwdFill * MR;
  unsigned char* rest = smem + kBwdWarps * kBwdFill * 16 * (1 + MR);
  int* recO = reinterpret_cast<int*>(rest) + wi * kBwdFill;
  if (NT > 3) rest += kBwdWarps * kBwdFill * 4;
  const int pix_cap = CPW * g.bw_views * g.bw_cand;
  PixItem* pix = reinterpret_cast<PixItem*>(rest) + wi * pix_cap;
  if (!TAB) rest += (kBwdWarps * pix_cap * (int)sizeof(PixItem) + 15) & ~15;
  const int nz = g.nz, nviews = subset_views(g, subset), nb = g.bw_nb;
  const int nst = SINGLE ? 1 : groups * nb;
  float* accs = reinterpret_cast<float*>(rest) + wi * CPW * ZK * 32 + lane;  // sums between stages
  if (!SINGLE) rest += kBwdWarps * CPW * ZK * 128;
  float* sw = reinterpret_cast<float*>(rest);
  const int tx0 = blockIdx.x * TX, ty0 = blockIdx.y * TY;
  const int ix0 = tx0 + (wi & 1) * CPW, iy = ty0 + (wi >> 1);

  // copies of stage st: rows r_min..r_max of its views, the planes of its components
  auto stage = [&](int st) {
    const int gr = SINGLE ? 0 : st / nb, b = SINGLE ? 0 : st - gr * nb;
    const BwdBatch bt = g.bw_batch[b];
    float* dst = sw;
    const int l1 = group_first(gr + 1, nviews, groups);
    for (int l = group_first(gr, nviews, groups); l < l1; ++l) {
      int r_min;
      const int r_max = tile_rows(g, g.view[subset_view(g, subset, l)], tx0, ty0, TX, TY, &r_min);
      const float* src = a.w + ((size_t)l * g.R + r_min) * g.P;
      const int nr = r_max - r_min + 1;
      for (int p = threadIdx.x; p < bt.copies; p += kBwdWarps * 32) {
        const int2 sp = __ldg(g.bw_slots + bt.first + p);  // slot, plane
        const float* s = src + sp.y;
        unsigned d = (unsigned)__cvta_generic_to_shared(dst + sp.x);
        for (int rr = 0; rr < nr; ++rr) {
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(s) : "memory");
          s += g.P;
          d += 4 * bt.slots;
        }
      }
      dst += g.bw_rows * bt.slots;
    }
  };
  // zeros of batch b: the frames; the copies never touch them
  auto zeros = [&](int b) {
    const BwdBatch bt = g.bw_batch[b];
    for (int p = threadIdx.x; p < bt.zeros; p += kBwdWarps * 32) {
      float* d = sw + __ldg(g.bw_slots + bt.first + bt.copies + p).x;
      for (int rr = 0; rr < g.bw_views * g.bw_rows; ++rr) d[rr * bt.slots] = 0.f;
    }
  };
  auto commit = [] { asm volatile("cp.async.commit_group;\n" ::: "memory"); };
  stage(0);
  commit();
  zeros(0);
  // the epilogue's lines of the tile go into L2 while the stages run
  if (mode == BWD_UPDATE || mode == BWD_EM) {
    const int ncol = min(TX, g.nx - tx0), row_lines = (ncol * nz + 31) / 32, nrow = min(TY, g.ny - ty0);
    for (int q = threadIdx.x; q < 3 * TY * row_lines; q += kBwdWarps * 32) {
      const int ar = q / row_lines, ln = q - ar * row_lines, arr = ar / TY, rr = ar - arr * TY;
      const float* base = arr == 0 ? (const float*)a.x : (arr == 1 ? (const float*)a.T : (const float*)a.z);
      if (rr < nrow && base)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(base + ((size_t)(ty0 + rr) * g.nx + tx0) * nz +
                                                      min(32 * ln, ncol * nz - 1)));
    }
  }

  // table: headers of 32 groups at a time (one per lane), items of the next fill one per lane
  int2 hd = make_int2(0, 0);
  float4 pre = make_float4(0.f, 0.f, 0.f, 0.f), pre_next = pre;
  unsigned start = 0, start_next = 0;
  int counts4 = 0, counts_next = 0, total = 0;
  auto items_of = [](int c4) { return (c4 & 255) + ((c4 >> 8) & 255) + ((c4 >> 16) & 255) + ((c4 >> 24) & 255); };
  // requests the first items of a view group (one group ahead of its use)
  auto request_group = [&](int gr) {
    if ((gr & 31) == 0) {
      hd = make_int2(0, 0);
      if (gr + lane < groups)
        hd = a.hdr[((((size_t)subset * groups + gr + lane) * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * kBwdWarps + wi];
    }
    start_next = (unsigned)__shfl_sync(0xffffffffu, hd.x, gr & 31);
    counts_next = __shfl_sync(0xffffffffu, hd.y, gr & 31);
    if (lane < items_of(counts_next)) pre_next = a.items[(size_t)start_next + lane];
  };
  if (TAB) request_group(0);

  int npairs = 0;
  int pcounts[CPW];
#pragma unroll
  for (int c = 0; c < CPW; ++c) pcounts[c] = 0;

  for (int st = 0; st < nst; ++st) {
    const int gr = SINGLE ? 0 : st / nb, b = SINGLE ? 0 : st - gr * nb;
    int cb = 0, cc = 0, slots = 0;
    if (TAB) {
      pre = pre_next;
      start = start_next;
      counts4 = counts_next;
      total = items_of(counts4);
      if (!SINGLE && gr + 1 < groups) request_group(gr + 1);
    } else {
      const BwdBatch bt = g.bw_batch[b];
      cb = bt.c0;
      cc = bt.c1 - bt.c0;
      slots = bt.slots;
      if (b == 0) {
        const int l0 = group_first(gr, nviews, groups);
        npairs = warp_pairs<CPW>(g, subset, l0, group_first(gr + 1, nviews, groups) - l0, tx0, ty0, ix0, iy, lane, pix, pcounts);
      }
      __syncwarp();
      total = npairs * cc;
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    const unsigned buf = (unsigned)__cvta_generic_to_shared(sw) + 4 * lane - 4 * kOffBias;
    const bool last = SINGLE || st == nst - 1;

    int it = 0, filled = 0, base = 0;
    // expands items [it, it + 32) of the warp to records, one per lane
    auto fill = [&]() {
      const int i = it + lane;
      __syncwarp();
      if (i < total) {
        float L[4] = {0.f, 0.f, 0.f, 0.f};
        int row_slot, jp, len, smask;
        if (TAB) {
          const unsigned pk = __float_as_uint(pre.w);
          L[0] = pre.x;
          L[1] = pre.y;
          L[2] = pre.z;
          row_slot = (int)(pk & 0xFFFFu);
          jp = (int)((pk >> 16) & 0x1FFu) - 256;
          len = g.comp[pk >> 25].len;
          smask = MASHED ? g.comp[pk >> 25].smask : 0;
        } else {
          const int pi = i / cc, ci = cb + (i - pi * cc);
          const PixItem Q = pix[pi];
          const CompDev cd = g.comp[ci];
          const int j0 = segment_taps<NT>(g, Q.r, ci, Q.I, L);
          row_slot = Q.row * slots + cd.slot;
          jp = j0 - cd.qlo + PAD;
          len = cd.len;
          smask = MASHED ? cd.smask : 0;
        }
        int nt = 1;
#pragma unroll
        for (int k = 1; k < NT; ++k)
          if (L[k] != 0.f) nt = k + 1;
        const bool step2 = MASHED && smask;
        // (without marks in the words an item of empty masks is harmless at any offset)
        const int word = MASHED ? (int)item_word(row_slot, jp, len, nt, 32 * ZK, PAD, step2) : 4 * (row_slot + jp + kOffBias) | (nt - 1);
        recA[lane] = make_float4(L[0], L[1], L[2], NT > 3 ? L[3] : __int_as_float(word));
        if (NT > 3) recO[lane] = word;
        auto masks = [&](uint4* to, int off) {
#pragma unroll
          for (int q = 0; q < MQ; ++q) {
            uint4 m;
            m.x = lane_range(off + 128 * q, len);
            m.y = ZK > 1 ? lane_range(off + 128 * q + 32, len) : 0u;
            m.z = ZK > 2 ? lane_range(off + 128 * q + 64, len) : 0u;
            m.w = ZK > 3 ? lane_range(off + 128 * q + 96, len) : 0u;
            to[q] = m;
          }
        };
        masks(recM + lane * MR, jp);
        if constexpr (mask_sets<NT, MASHED>() > 1) {
          if (word & (int)kStep2) masks(recM + lane * MR + MQ, jp + 2);
        }
      }
      base = it;
      filled = min(it + kBwdFill, total);
      if (TAB && filled + lane < total) pre = a.items[(size_t)start + filled + lane];
      __syncwarp();
    };
    // one column after the other: its records, then in the last stage its epilogue
#pragma unroll 1
    for (int c = 0; c < CPW; ++c) {
      const int ix = ix0 + c;
      const bool finish = last && ix < g.nx && iy < g.ny;
      const size_t col = ((size_t)iy * g.nx + ix) * nz;
      float ac[ZK], xr[ZK], zr[ZK], Tr[ZK];
      if (finish && mode != BWD_OUT) {
#pragma unroll
        for (int k = 0; k < ZK; ++k) {
          const int iz = lane + 32 * k;
          if (iz >= nz) continue;
          if (mode != BWD_SENS) xr[k] = ld_now(a.x + col + iz);
          if (mode == BWD_UPDATE) zr[k] = ld_now(a.z + col + iz);
          Tr[k] = ld_now(a.T + col + iz);
        }
      }
#pragma unroll
      for (int k = 0; k < ZK; ++k) ac[k] = !SINGLE && st > 0 ? accs[(c * ZK + k) * 32] : 0.f;
      int n = 0;
      if (TAB) n = (counts4 >> (8 * c)) & 255;
      else {
#pragma unroll
        for (int q = 0; q < CPW; ++q)
          if (q == c) n = pcounts[q] * cc;
      }
      const int end = it + n;
      while (it < end) {
        if (it == filled) fill();
        if constexpr (NT == 1) {
          // one rounding per record, where a product added to a sum has two
          const int e = min(end, filled);
          gather_items<NT, ZK, MASHED>(buf, recA, recM, recO, it - base, e - base, bit, ac);
          it = e;
        } else {
          // Sums of few records at a time: added tap by tap to one running sum, the roundings of a column
          // of many records grew with it (see above the kernel).
          const int e = min(min(end, filled), it + kSumItems);
          float part[ZK];
#pragma unroll
          for (int k = 0; k < ZK; ++k) part[k] = 0.f;
          gather_items<NT, ZK, MASHED>(buf, recA, recM, recO, it - base, e - base, bit, part);
#pragma unroll
          for (int k = 0; k < ZK; ++k) ac[k] += part[k];
          it = e;
        }
      }
      if (!last) {
#pragma unroll
        for (int k = 0; k < ZK; ++k) accs[(c * ZK + k) * 32] = ac[k];
      }
      if (!finish) continue;
#pragma unroll
      for (int k = 0; k < ZK; ++k) {
        const int iz = lane + 32 * k;
        if (iz >= nz) continue;
        const size_t idx = col + iz;
        if (mode == BWD_UPDATE) {
          // z = z + dz;  zbar = z + dz / p_i;  next primal step x = max(x - T zbar, 0)
          const float zn = zr[k] + ac[k];
          a.z[idx] = zn;
          a.x[idx] = prox_nonneg(xr[k] - Tr[k] * fmaf(ac[k], a.inv_p, zn));
        } else if (mode == BWD_OUT) {
          a.out[idx] = ac[k];
        } else if (mode == BWD_SENS) {
          // T_i = rho p_i / (gamma (P_i^T 1)); +inf (kept) where the subset does not see the voxel
          if (ac[k] > 0.f) a.T[idx] = fminf(Tr[k], a.sens_num / ac[k]);
        } else {
          // u <- u / (P_i^T 1) * P_i^T (b_i / (P_i u + r_i)), 0 where the subset does not see the voxel
          a.x[idx] = Tr[k] > 0.f ? xr[k] * ac[k] / Tr[k] : 0.f;
        }
      }
    }
    if (!SINGLE && st + 1 < nst) {
      __syncthreads();
      stage(st + 1);
      commit();
      if (nb > 1) {  // the next batch lays its runs out anew
        zeros((st + 1) % nb);
      }
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------------------
// tap-item table: the items of every stage, tile and warp in the kernel's order, computed once by
// the functions the kernel runs.  An item is (L0, L1, L2, row slot (16 bits) | jp + 256 (9) |
// component (7)); a header (one per stage and warp) is the first item and the columns' counts.
// Pass 0 counts the items per warp and flags an item that does not fit the packing; pass 1 fills.
// ---------------------------------------------------------------------------------------
template <int NT, int CPW, int PASS>
__global__ void __launch_bounds__(kBwdWarps * 32) k_bwd_items(const __grid_constant__ DevGeom g, int groups, unsigned short* cnt,
                                                              unsigned* bad, const unsigned* starts,
                                                              const unsigned* stage_base, float4* items, int2* hdr) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int PAD = NT - 1;
  constexpr int TX = 2 * CPW, TY = 4;
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  PixItem* pix = reinterpret_cast<PixItem*>(smem) + wi * CPW * g.bw_views * g.bw_cand;
  const int tx0 = blockIdx.x * TX, ty0 = blockIdx.y * TY;
  const int subset = blockIdx.z / groups, gr = blockIdx.z - subset * groups, nviews = subset_views(g, subset);
  const size_t rec = (((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * kBwdWarps + wi;
  int counts[CPW];
  const int l0 = group_first(gr, nviews, groups);
  const int np = warp_pairs<CPW>(g, subset, l0, group_first(gr + 1, nviews, groups) - l0, tx0, ty0, tx0 + (wi & 1) * CPW,
                                 ty0 + (wi >> 1), lane, pix, counts);
  __syncwarp();
  const int total = np * g.n_comp, slots = g.bw_batch[0].slots;
  bool misfit = false;
#pragma unroll
  for (int c = 0; c < CPW; ++c) misfit = misfit || counts[c] * g.n_comp > 255;
  unsigned base = 0;
  if (PASS == 1) base = stage_base[blockIdx.z] + starts[rec];
  for (int i = lane; i < total; i += 32) {
    const int pi = i / g.n_comp, ci = i - pi * g.n_comp;
    const PixItem Q = pix[pi];
    const CompDev cd = g.comp[ci];
    float L[4] = {0.f, 0.f, 0.f, 0.f};
    const int j0 = segment_taps<NT>(g, Q.r, ci, Q.I, L);
    const int row_slot = Q.row * slots + cd.slot, jp = j0 - cd.qlo + PAD + 256;
    if (PASS == 0) misfit = misfit || row_slot >= 65536 || jp < 0 || jp >= 512 || ci >= 128;
    else items[(size_t)base + i] = make_float4(L[0], L[1], L[2], __uint_as_float((unsigned)row_slot | ((unsigned)jp << 16) | ((unsigned)ci << 25)));
  }
  if (PASS == 0) {
    if (__any_sync(0xffffffffu, misfit) && lane == 0) atomicOr(bad, 1u);
    if (lane == 0) cnt[rec] = (unsigned short)min(total, 65535);
  } else if (lane == 0) {
    unsigned c4 = 0;
#pragma unroll
    for (int c = 0; c < CPW; ++c) c4 |= (unsigned)(counts[c] * g.n_comp) << (8 * c);
    hdr[rec] = make_int2((int)base, (int)c4);
  }
}

// ---------------------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------------------

// Bytes of the warps' pair lists.  backward_layout chooses the views per stage so that they stay within
// kPairBytes, with any geometry: neither kernel then needs more shared memory than it may ask for.
inline size_t bwd_pair_bytes(const DevGeom& g) {
  return ((size_t)kBwdWarps * g.bw_cpw * g.bw_views * g.bw_cand * sizeof(PixItem) + 15) & ~(size_t)15;
}

// Dynamic shared memory of k_backward (its carve-up in order): records, wide offsets, pairs, sums, staging.
inline size_t bwd_smem(const DevGeom& g, int nt, int zk, bool single, bool tab, bool mashed) {
  size_t smem = (size_t)kBwdWarps * kBwdFill * 16 * (1 + (zk + 3) / 4 * (mashed && nt > 2 ? 2 : 1));
  if (nt > 3) smem += (size_t)kBwdWarps * kBwdFill * 4;
  if (!tab) smem += bwd_pair_bytes(g);
  if (!single) smem += (size_t)kBwdWarps * g.bw_cpw * zk * 128;
  return smem + (size_t)g.bw_buf * sizeof(float);
}

inline dim3 bwd_tiles(const DevGeom& g) { return dim3((g.nx + 2 * g.bw_cpw - 1) / (2 * g.bw_cpw), (g.ny + 3) / 4); }

// view groups of a subset (the same for all subsets, whose view counts differ by at most one)
inline int bwd_groups(const DevGeom& g, int subset) {
  const int most = subset < 0 || g.bins ? g.V : (g.V + g.m - 1) / g.m;
  return (most + g.bw_views - 1) / g.bw_views;
}

template <int NT, int ZK, int CPW, bool SINGLE, bool TAB, bool MASHED>
cudaError_t bwd_run(const DevGeom& g, int subset, int mode, const BwdArgs& a, cudaStream_t s) {
  const int groups = bwd_groups(g, subset);
  const size_t smem = bwd_smem(g, NT, ZK, SINGLE, TAB, MASHED);
  if (smem > kBwdMaxSmem) return cudaErrorInvalidValue;
  auto kern = k_backward<NT, ZK, CPW, SINGLE, TAB, MASHED>;
  cudaError_t e = allow_dynamic_smem(kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<bwd_tiles(g), kBwdWarps * 32, smem, s>>>(g, subset, groups, mode, a);
  return cudaGetLastError();
}

template <int NT, int ZK, bool TAB, bool MASHED>
cudaError_t bwd_shape(const DevGeom& g, int subset, int mode, const BwdArgs& a, cudaStream_t s) {
  if (g.bw_cpw == 1) return bwd_run<NT, ZK, 1, false, TAB, MASHED>(g, subset, mode, a, s);
  if (bwd_groups(g, subset) * g.bw_nb == 1) return bwd_run<NT, ZK, 4, true, TAB, MASHED>(g, subset, mode, a, s);
  return bwd_run<NT, ZK, 4, false, TAB, MASHED>(g, subset, mode, a, s);
}

template <int NT, int ZK>
cudaError_t bwd_tab(const DevGeom& g, int subset, int mode, const BwdArgs& a, cudaStream_t s) {
  if constexpr (NT <= 3) {
    if (a.items)
      return g.bw_step2 ? bwd_shape<NT, ZK, true, true>(g, subset, mode, a, s) : bwd_shape<NT, ZK, true, false>(g, subset, mode, a, s);
  } else {
    if (a.items) return cudaErrorInvalidValue;
  }
  return g.bw_step2 ? bwd_shape<NT, ZK, false, true>(g, subset, mode, a, s) : bwd_shape<NT, ZK, false, false>(g, subset, mode, a, s);
}

// instantiated per tap count in backward_taps<NT>.cu
template <int NT>
cudaError_t launch_backward_nt(const DevGeom& g, int subset, int mode, const BwdArgs& a, cudaStream_t s) {
  const int zk = (g.nz + 31) / 32;
  if (zk <= 1) return bwd_tab<NT, 1>(g, subset, mode, a, s);
  if (zk <= 2) return bwd_tab<NT, 2>(g, subset, mode, a, s);
  if (zk <= 3) return bwd_tab<NT, 3>(g, subset, mode, a, s);
  if (zk <= 4) return bwd_tab<NT, 4>(g, subset, mode, a, s);
  if (zk <= 8) return bwd_tab<NT, 8>(g, subset, mode, a, s);
  return cudaErrorInvalidValue;
}

template <int NT>
cudaError_t backward_items_nt(const DevGeom& g, int pass, unsigned short* cnt, unsigned* bad, const unsigned* starts,
                              const unsigned* stage_base, float4* items, int2* hdr, cudaStream_t s) {
  const int groups = bwd_groups(g, 0);
  const dim3 t = bwd_tiles(g), grid(t.x, t.y, g.m * groups);
  const size_t smem = bwd_pair_bytes(g);
  auto go = [&](auto kern) {
    cudaError_t e = allow_dynamic_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, kBwdWarps * 32, smem, s>>>(g, groups, cnt, bad, starts, stage_base, items, hdr);
    return cudaGetLastError();
  };
  if (g.bw_cpw == 1) return pass == 0 ? go(k_bwd_items<NT, 1, 0>) : go(k_bwd_items<NT, 1, 1>);
  return pass == 0 ? go(k_bwd_items<NT, 4, 0>) : go(k_bwd_items<NT, 4, 1>);
}

extern template cudaError_t launch_backward_nt<1>(const DevGeom&, int, int, const BwdArgs&, cudaStream_t);
extern template cudaError_t launch_backward_nt<2>(const DevGeom&, int, int, const BwdArgs&, cudaStream_t);
extern template cudaError_t launch_backward_nt<3>(const DevGeom&, int, int, const BwdArgs&, cudaStream_t);
extern template cudaError_t launch_backward_nt<4>(const DevGeom&, int, int, const BwdArgs&, cudaStream_t);
extern template cudaError_t backward_items_nt<1>(const DevGeom&, int, unsigned short*, unsigned*, const unsigned*, const unsigned*, float4*, int2*, cudaStream_t);
extern template cudaError_t backward_items_nt<2>(const DevGeom&, int, unsigned short*, unsigned*, const unsigned*, const unsigned*, float4*, int2*, cudaStream_t);
extern template cudaError_t backward_items_nt<3>(const DevGeom&, int, unsigned short*, unsigned*, const unsigned*, const unsigned*, float4*, int2*, cudaStream_t);

}  // namespace spdhg
