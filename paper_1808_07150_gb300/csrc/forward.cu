// Ray-driven forward projector, fused with the KL dual prox of SPDHG.
#include <algorithm>
#include <type_traits>

#include "lor.cuh"

namespace spdhg {

// ---------------------------------------------------------------------------------------
// forward projection: one block per transaxial line (view, radial bin), threads over planes
// ---------------------------------------------------------------------------------------
struct Entry {
  int col;  // iy * nx + ix
  PixInt I;
};

constexpr int kCandPerRow = 4;

// Pixels of `row` (along the dominant axis of the line) that the line crosses.  Candidates come
// from approximate arithmetic (one pixel of margin on each side); pixel_interval decides exactly.
__device__ __forceinline__ int row_entries(const DevGeom& g, const Line& L, bool ydom, int row, Entry* e) {
  const float c = L.c_hi, s = L.s_hi, sp = L.sp_hi, h = L.h_hi;
  float t0, t1;
  if (ydom) {  // y in [Y0, Y0 + 1);  y(t) = sp s + t c
    const float Y0 = (float)row - 0.5f * (float)g.ny;
    t0 = (Y0 - sp * s) / c;
    t1 = (Y0 + 1.f - sp * s) / c;
  } else {     // x in [X0, X0 + 1);  x(t) = sp c - t s
    const float X0 = (float)row - 0.5f * (float)g.nx;
    t0 = (sp * c - X0) / s;
    t1 = (sp * c - X0 - 1.f) / s;
  }
  const float tlo = fmaxf(fminf(t0, t1), -h - 1e-2f), thi = fminf(fmaxf(t0, t1), h + 1e-2f);
  if (thi < tlo) return 0;
  const float ca = ydom ? sp * c - tlo * s : sp * s + tlo * c;
  const float cb = ydom ? sp * c - thi * s : sp * s + thi * c;
  const float half = 0.5f * (float)(ydom ? g.nx : g.ny);
  const int nc = ydom ? g.nx : g.ny;
  const int cmin = max((int)floorf(fminf(ca, cb) + half) - 1, 0);
  const int cmax = min((int)floorf(fmaxf(ca, cb) + half) + 1, nc - 1);
  int n = 0;
  for (int cc = cmin; cc <= cmax && n < kCandPerRow; ++cc) {
    const int ix = ydom ? cc : row, iy = ydom ? row : cc;
    PixInt I;
    if (pixel_interval(g, L, ix, iy, I)) {
      e[n].col = iy * g.nx + ix;
      e[n].I = I;
      ++n;
    }
  }
  return n;
}

constexpr int kFwdChunk = 32;  // pixel entries per double-buffered chunk
constexpr int kRunsPerWarp = 2;  // 32-plane runs per warp (lane = plane within a run)
// Entry groups: when a line has few plane runs (a shallow volume), several warps share each run,
// each taking every egroups-th pixel entry, and their partial sums are added in group order.
constexpr int kFwdMaxGroupWarps = 7;  // warps of groups 1.. (their sums are staged in shared)

// Axial taps of one (pixel entry, segment) pair as the gather reads them: lengths of taps
// 0..NT-1 and, in `off`, the offset of plane 0's tap 0 in the staged x column (low 28 bits) and
// the entry's own tap count (top bits; lengths past it are zero).
struct TapRec {
  float l0, l1, l2;
  int off;
};
struct TapRec4 {  // geometries whose LORs cross four slices inside a pixel
  float l0, l1, l2;
  int off;
  float l3, pad0, pad1, pad2;
};
template <int NT>
using TapRecT = typename std::conditional<(NT > 3), TapRec4, TapRec>::type;
constexpr int kOffBits = 28;
constexpr int kOffMask = (1 << kOffBits) - 1;

__device__ __forceinline__ float2 ffma2_bcast(float l, float xa, float xb, float2 acc) {
  return __ffma2_rn(make_float2(l, l), make_float2(xa, xb), acc);
}

// sum_t L_t x[-t] over the entry's taps (scalar; one plane)
template <int NT, class Rec>
__device__ __forceinline__ float taps_dot(const Rec& t, int nt, const float* xp, float acc) {
  acc = fmaf(t.l0, xp[0], acc);
  if (NT > 1 && nt > 1) {
    acc = fmaf(t.l1, xp[-1], acc);
    if (NT > 2 && nt > 2) {
      acc = fmaf(t.l2, xp[-2], acc);
      if constexpr (NT > 3) {
        if (nt > 3) acc = fmaf(t.l3, xp[-3], acc);
      }
    }
  }
  return acc;
}

// Forward projection.  Block (line, row part, plane part) owns the rows [row_lo, row_hi) of one
// transaxial LOR line (view, radial bin) and a contiguous range of the line's plane runs (32
// consecutive planes of one segment, segment-major); warp w owns two neighbouring runs and lane l
// plane q0 + l of each.  All threads first find the pixels the line crosses in those rows (exact
// intervals, compacted); the entries are then processed in chunks of kFwdChunk: the x columns of
// chunk c+1 are copied to shared memory (cp.async) inside zero frames wide enough for every tap
// of every plane of the segments (the axial bound of the geometry, so no plane needs a range
// test), and its axial taps computed while chunk c is accumulated.  When both runs of a warp lie
// in one segment, one tap record serves both and a packed FP32 FMA accumulates the two planes.
// When a line has few runs, egroups warps share each pair of runs, warp group k taking the
// entries k, k + egroups, ... of every chunk; group 0 adds the other groups' sums in group order.
// When several row parts share a line, each writes partial plane sums and the last one to finish
// reduces them in a fixed order.
template <int NT, int MODE, bool GROUPS>
__global__ void __launch_bounds__(512) k_forward(DevGeom g, int subset, int ecap, int rsplit, int xs_stride,
                                                 int runs_per_part, int ncomp_tab, int chunk, int egroups_arg,
                                                 FwdArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int scan_scratch[33];
  const int FL = g.fz_lo;
  float* xs = reinterpret_cast<float*>(smem);                                  // [2][chunk][xs_stride]
  using Rec = TapRecT<NT>;
  Rec* taps = reinterpret_cast<Rec*>(xs + 2 * chunk * xs_stride);              // [2][ncomp_tab][chunk]
  Entry* ent = reinterpret_cast<Entry*>(taps + 2 * ncomp_tab * chunk);         // [ecap]
  float* group_acc = reinterpret_cast<float*>(ent + ecap);  // [egroups - 1][nrw][2][32] partial sums
  const int nz = g.nz;

  const int line = blockIdx.x, rpart = blockIdx.y, ppart = blockIdx.z;
  const int l = line / g.R, r = line - l * g.R;
  const int v = subset_view(g, subset, l);
  const Line L = make_line(g, v, r);

  // this thread's planes: lane of runs rf + 2w and rf + 2w + 1 of the plane part, w = wi mod
  // nrw; warp wi takes every egroups-th pixel entry from entry wi / nrw on
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int egroups = GROUPS ? egroups_arg : 1;
  const int nrw = GROUPS ? nw / egroups : nw, rw = GROUPS ? wi % nrw : wi, eg = GROUPS ? wi / nrw : 0;
  const int rfirst = ppart * runs_per_part;
  const int rlast = min(g.n_runs, rfirst + runs_per_part) - 1;
  const int g_lo = g.runs[rfirst].x, g_hi = g.runs[rlast].x;
  // the LOR components of the block's segments, c_lo .. c_hi
  const int c_lo = g.seg[g_lo].c0, c_hi = g.seg[g_hi].c0 + g.seg[g_hi].nc - 1;
  int gs_[kRunsPerWarp], qv_[kRunsPerWarp], qr_[kRunsPerWarp];
  unsigned incl_[kRunsPerWarp];                  // mashed: components of the segment this plane sums
  bool valid_[kRunsPerWarp];
#pragma unroll
  for (int k = 0; k < kRunsPerWarp; ++k) {
    const int run = rfirst + kRunsPerWarp * rw + k;
    const int2 ru = g.runs[min(run, rlast)];
    const SegDev sd = g.seg[ru.x];
    gs_[k] = ru.x;
    qv_[k] = ru.y + lane;                        // the plane of this lane
    valid_[k] = run <= rlast && qv_[k] < sd.n;
    qr_[k] = min(qv_[k], sd.n - 1);              // the plane read (inside the segment's frames)
    incl_[k] = 0u;
    if (g.mashed)
      for (int c = 0; c < sd.nc; ++c) {
        const CompDev cd = g.comp[sd.c0 + c];
        const int dq = qv_[k] - cd.qlo;
        if (qv_[k] < cd.qhi && dq >= 0 && (dq & cd.smask) == 0) incl_[k] |= 1u << c;
      }
  }
  const bool same = gs_[0] == gs_[1];            // warp-uniform

  // zero frames of the staged columns (never overwritten); SIGMA stages ones: the projection of
  // the constant image is the chord of each LOR inside the image
  for (int i = threadIdx.x; i < 2 * chunk * xs_stride; i += blockDim.x) {
    const int k = i % xs_stride;
    if (MODE == FWD_SIGMA) xs[i] = (k >= FL && k < FL + nz) ? 1.f : 0.f;
    else if (k < FL || k >= FL + nz) xs[i] = 0.f;
  }
  const bool ydom = fabsf(L.c_hi) >= fabsf(L.s_hi);  // |dy| >= |dx|: walk the rows of y
  const int nrows_all = ydom ? g.ny : g.nx;
  const int rows_per_part = (nrows_all + rsplit - 1) / rsplit;
  const int row_lo = rpart * rows_per_part, row_hi = min(nrows_all, row_lo + rows_per_part);

  // A. this block's rows -> exact pixel intervals, compacted into ent[]
  int n_ent = 0;
  for (int row0 = row_lo; row0 < row_hi; row0 += blockDim.x) {
    Entry loc[kCandPerRow];
    const int row = row0 + threadIdx.x;
    const int cnt = row < row_hi ? row_entries(g, L, ydom, row, loc) : 0;
    int total;
    const int off = n_ent + block_exclusive_scan(cnt, scan_scratch, &total);
    for (int k = 0; k < cnt; ++k)
      if (off + k < ecap) ent[off + k] = loc[k];
    n_ent = min(n_ent + total, ecap);
  }
  __syncthreads();

  const int ncb = c_hi - c_lo + 1;
  auto stage = [&](int c) {  // x columns + taps of chunk c into buffer c & 1
    const int buf = c & 1;
    const int e0 = c * chunk, ne = min(chunk, n_ent - e0);
    float* xb = xs + buf * chunk * xs_stride;
    if (MODE != FWD_SIGMA) {
      // one warp per entry, lanes along z
      for (int e = wi; e < ne; e += nw) {
        const float* src = a.x + (size_t)ent[e0 + e].col * nz;
        float* dst = xb + e * xs_stride + FL;
        for (int iz = lane; iz < nz; iz += 32) cp_async4(dst + iz, src + iz);
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    Rec* tb = taps + buf * ncomp_tab * chunk;
    for (int it = threadIdx.x; it < ncb * ne; it += blockDim.x) {
      const int gs = it / ne, e = it - gs * ne;
      float Lk[4] = {0.f, 0.f, 0.f, 0.f};
      int j0 = segment_taps<NT>(g, r, c_lo + gs, ent[e0 + e].I, Lk);
      // the geometry's axial bound keeps every read inside the framed column; the clamp only
      // guards shared memory should a rounding case fall outside it
      const CompDev cd = g.comp[c_lo + gs];
      j0 = min(max(j0, cd.jlo), cd.jhi);
      int nt = NT;
      while (nt > 1 && Lk[nt - 1] == 0.f) --nt;
      Rec& rec = tb[gs * chunk + e];
      rec.l0 = Lk[0];
      rec.l1 = NT > 1 ? Lk[1] : 0.f;
      rec.l2 = NT > 2 ? Lk[2] : 0.f;
      rec.off = (e * xs_stride + FL - j0) | (nt << kOffBits);
      if constexpr (NT > 3) rec.l3 = Lk[3];
    }
  };

  float acc[kRunsPerWarp] = {0.f, 0.f};
  const int nchunks = (n_ent + chunk - 1) / chunk;
  if (nchunks > 0) stage(0);
  for (int c = 0; c < nchunks; ++c) {
    if (c + 1 < nchunks) {
      stage(c + 1);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
    const int buf = c & 1;
    const int ne = min(chunk, n_ent - c * chunk);
    const int nk = !GROUPS ? ne : (ne > eg ? (ne - eg + egroups - 1) / egroups : 0);  // entries eg + k egroups
    const float* xb = xs + buf * chunk * xs_stride;
    if (g.mashed) {
      // each plane sums the components of its segment it includes (exact mashing)
#pragma unroll
      for (int k = 0; k < kRunsPerWarp; ++k) {
        const SegDev sd = g.seg[gs_[k]];
        const Rec* trk = taps + buf * ncomp_tab * chunk + (sd.c0 - c_lo) * chunk;
        float sk = 0.f;
        for (int ci = 0; ci < sd.nc; ++ci) {
          const bool in = (incl_[k] >> ci) & 1u;
          const Rec* tc = trk + ci * chunk;
          float sc = 0.f;
          for (int kk = 0; kk < nk; ++kk) {
            const Rec t = tc[eg + kk * egroups];
            sc = taps_dot<NT>(t, NT > 1 ? (t.off >> kOffBits) : 1, xb + (t.off & kOffMask) + qr_[k], sc);
          }
          sk += in ? sc : 0.f;
        }
        acc[k] += sk;
      }
      __syncthreads();
      continue;
    }
    const Rec* tr0 = taps + buf * ncomp_tab * chunk + (gs_[0] - g_lo) * chunk;
    if (same) {
      float2 s2 = make_float2(0.f, 0.f);
#pragma unroll 1
      for (int k = 0; k < nk; ++k) {
        const Rec t = tr0[eg + k * egroups];
        const int off = t.off & kOffMask, nt = NT > 1 ? (t.off >> kOffBits) : 1;
        const float* xa = xb + off + qr_[0];
        // the warp's second run is the next 32 planes of the segment: a constant offset.  Lanes
        // past the segment's last plane read up to 31 slots beyond their column (the next
        // column, or the tap records after the last buffer) and are never written
        const float* xc = xa + 32;
        s2 = ffma2_bcast(t.l0, xa[0], xc[0], s2);
        if (NT > 1 && nt > 1) {
          s2 = ffma2_bcast(t.l1, xa[-1], xc[-1], s2);
          if (NT > 2 && nt > 2) {
            s2 = ffma2_bcast(t.l2, xa[-2], xc[-2], s2);
            if constexpr (NT > 3) {
              if (nt > 3) s2 = ffma2_bcast(t.l3, xa[-3], xc[-3], s2);
            }
          }
        }
      }
      acc[0] += s2.x;
      acc[1] += s2.y;
    } else {
      const Rec* tr1 = taps + buf * ncomp_tab * chunk + (gs_[1] - g_lo) * chunk;
      float s0 = 0.f, s1 = 0.f;
      for (int k = 0; k < nk; ++k) {
        const int e = eg + k * egroups;
        const Rec t0 = tr0[e], t1 = tr1[e];
        s0 = taps_dot<NT>(t0, NT > 1 ? (t0.off >> kOffBits) : 1, xb + (t0.off & kOffMask) + qr_[0], s0);
        s1 = taps_dot<NT>(t1, NT > 1 ? (t1.off >> kOffBits) : 1, xb + (t1.off & kOffMask) + qr_[1], s1);
      }
      acc[0] += s0;
      acc[1] += s1;
    }
    __syncthreads();
  }

  if (GROUPS) {
    // entry groups 1.. hand their partial sums to group 0, which adds them in group order
    if (eg > 0) {
#pragma unroll
      for (int k = 0; k < kRunsPerWarp; ++k) group_acc[(((eg - 1) * nrw + rw) * kRunsPerWarp + k) * 32 + lane] = acc[k];
    }
    __syncthreads();
    if (eg == 0) {
      for (int q = 1; q < egroups; ++q) {
#pragma unroll
        for (int k = 0; k < kRunsPerWarp; ++k) acc[k] += group_acc[(((q - 1) * nrw + rw) * kRunsPerWarp + k) * 32 + lane];
      }
    } else {
#pragma unroll
      for (int k = 0; k < kRunsPerWarp; ++k) valid_[k] = false;  // group 0 writes the planes
    }
  }

  if (rsplit > 1) {
    // publish this block's partial sums; the last row part of the (line, plane part) reduces them
    __shared__ unsigned last_sh;
    const size_t pbase = ((size_t)line * rsplit + rpart) * g.P;
#pragma unroll
    for (int k = 0; k < kRunsPerWarp; ++k)
      if (valid_[k]) a.part_acc[pbase + g.seg[gs_[k]].p0 + qv_[k]] = acc[k];
    __threadfence();
    __syncthreads();
    const size_t ticket = (size_t)line * gridDim.z + ppart;
    if (threadIdx.x == 0) last_sh = (atomicAdd(a.tickets + ticket, 1u) == (unsigned)rsplit - 1u) ? 1u : 0u;
    __syncthreads();
    if (!last_sh) return;
    __threadfence();
#pragma unroll
    for (int k = 0; k < kRunsPerWarp; ++k) {
      if (!valid_[k]) continue;
      float sa = 0.f;
      for (int q = 0; q < rsplit; ++q)  // fixed order: deterministic
        sa += __ldcg(a.part_acc + ((size_t)line * rsplit + q) * g.P + g.seg[gs_[k]].p0 + qv_[k]);
      acc[k] = sa;
    }
    if (threadIdx.x == 0) a.tickets[ticket] = 0u;  // ready for the next launch
  }

#pragma unroll
  for (int k = 0; k < kRunsPerWarp; ++k) {
    if (!valid_[k]) continue;
    const int p = g.seg[gs_[k]].p0 + qv_[k];
    const size_t j = ((size_t)v * g.R + r) * g.P + p;
    const size_t jl = ((size_t)l * g.R + r) * g.P + p;  // subset-local index (= j for bin subsets)
    if (!bin_in_subset(g, subset, j)) {  // a bin of another subset: not written; no dual change
      if (MODE == FWD_DATA || MODE == FWD_EM) a.wdy[jl] = 0.f;
      continue;
    }
    const float mu = a.mult ? a.mult[j] : 1.f;
    if (MODE == FWD_EM) {
      // EM ratio backprojected by P^T = L^T diag(mult): mult_j b_j / ((P x)_j + r_j)  (Eq. EQU:OSEM)
      const float bj = a.b[j];
      a.wdy[jl] = bj > 0.f ? mu * bj / fmaf(mu, acc[k], a.r[j]) : 0.f;
    } else if (MODE == FWD_PROJECT) {
      a.out[j] = mu * acc[k];
    } else if (MODE == FWD_SIGMA) {
      // sigma_j = gamma rho / (P_i 1)_j,  (P_i 1)_j = mult_j * chord_j  (Eq. EQU:STEPSIZE:PRECOND)
      const float a1 = mu * acc[k];
      a.out[j] = a1 > 0.f ? a.gamma_rho / a1 : 0.f;
    } else {
      // KL dual prox on this bin:  y+ = prox_{sigma varphi*}(y + sigma (P_i x)_j), evaluated as
      // 2 (w - sigma b) / (w + 1 + sqrt((w - 1)^2 + 4 sigma b)),  w = y + sigma ((P_i x)_j + r_j),
      // which equals 1/2 [w + 1 - sqrt((w - 1)^2 + 4 sigma b)] without its cancellation.
      const float sigma = a.sigma[j];
      const float yj = a.y[j];
      const float bj = a.b[j];
      const float w = fmaf(sigma, fmaf(mu, acc[k], a.r[j]), yj);
      const float sb = sigma * bj;
      const float wm = w - 1.f;
      const float root = sqrtf(fmaf(wm, wm, 4.f * sb));
      const float yn = 2.f * (w - sb) / (w + 1.f + root);
      a.y[j] = yn;
      a.wdy[jl] = mu * (yn - yj);
    }
  }
}

// ---------------------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------------------

int forward_split(const DevGeom& g, int subset) {
  if (g.tune[SPDHG_TUNE_FWD_SPLIT]) return g.tune[SPDHG_TUNE_FWD_SPLIT];
  // enough blocks for every SM: one LOR line per block is too few for small subsets
  const int lines = subset_views(g, subset) * g.R * forward_parts(g);
  const int nrows = g.nx > g.ny ? g.nx : g.ny;
  int split = 1;
  while (split < 8 && lines * split < 152 && nrows / (split * 2) >= 32) split *= 2;
  return split;
}

// plane runs per block: two per warp, at most 16 warps
static int forward_runs_per_part(const DevGeom& g) {
  const int w = g.tune[SPDHG_TUNE_FWD_WARPS] ? g.tune[SPDHG_TUNE_FWD_WARPS] : 16;
  return w * kRunsPerWarp;
}

int forward_parts(const DevGeom& g) {
  const int rpp = forward_runs_per_part(g);
  return (g.n_runs + rpp - 1) / rpp;
}

// entry groups per block: at least four warps per block when the runs of a part need fewer
int forward_entry_groups(const DevGeom& g) {
  const int rpp = forward_runs_per_part(g);
  const int nrw = (std::min(rpp, g.n_runs) + kRunsPerWarp - 1) / kRunsPerWarp;
  int eg = g.tune[SPDHG_TUNE_FWD_GROUPS] ? g.tune[SPDHG_TUNE_FWD_GROUPS] : std::max(1, 4 / nrw);
  while (eg > 1 && ((eg - 1) * nrw > kFwdMaxGroupWarps || nrw * eg > 16)) --eg;
  return eg;
}

template <int NT, int MODE>
static cudaError_t fwd_launch(const DevGeom& g, int subset, const FwdArgs& a, cudaStream_t s) {
  const int xs_stride = g.fz_stride;
  const int nrows = g.nx > g.ny ? g.nx : g.ny;
  const int ecap = 3 * nrows + 8;  // a line crosses at most two pixels per row of its dominant axis
  const int rpp = forward_runs_per_part(g);
  const int parts = (g.n_runs + rpp - 1) / rpp;
  const int nrw = (std::min(rpp, g.n_runs) + kRunsPerWarp - 1) / kRunsPerWarp;  // warps per entry group
  const int egroups = forward_entry_groups(g);
  if (egroups < 1 || (egroups - 1) * nrw > kFwdMaxGroupWarps || nrw * egroups > 16) return cudaErrorInvalidValue;
  const int threads = 32 * nrw * egroups;
  // a block computes the taps of the components of the segments its runs span
  const int ncomp_tab = g.max_part_comps[rpp / kRunsPerWarp];
  // entries per chunk: 32, fewer when a block holds the taps of many components (mashing)
  int chunk = kFwdChunk;
  while (chunk > 4 && (size_t)2 * ncomp_tab * chunk * sizeof(TapRecT<NT>) > 48 * 1024) chunk /= 2;
  const size_t smem = (size_t)2 * chunk * xs_stride * sizeof(float) +
                      (size_t)2 * ncomp_tab * chunk * sizeof(TapRecT<NT>) + (size_t)ecap * sizeof(Entry) +
                      (size_t)(egroups - 1) * nrw * kRunsPerWarp * 32 * sizeof(float);
  if (smem > 200 * 1024 || (size_t)chunk * xs_stride >= ((size_t)1 << kOffBits)) return cudaErrorInvalidValue;
  if (MODE == FWD_DATA && !a.sigma) return cudaErrorInvalidValue;
  if ((MODE == FWD_DATA || MODE == FWD_EM) && (!a.b || !a.r || !a.wdy)) return cudaErrorInvalidValue;
  auto kern = egroups > 1 ? k_forward<NT, MODE, true> : k_forward<NT, MODE, false>;
  {
    cudaError_t e = allow_dynamic_smem(kern, smem);
    if (e != cudaSuccess) return e;
  }
  const int lines = subset_views(g, subset) * g.R;
  if (lines == 0) return cudaSuccess;
  const int rsplit = forward_split(g, subset);
  if (rsplit > 1 && (!a.part_acc || !a.tickets || (size_t)lines * rsplit * g.P > a.part_cap ||
                     (size_t)lines * parts > a.ticket_cap))
    return cudaErrorInvalidValue;
  dim3 grid(lines, rsplit, parts);
  kern<<<grid, threads, smem, s>>>(g, subset, ecap, rsplit, xs_stride, rpp, ncomp_tab, chunk, egroups, a);
  return cudaGetLastError();
}

template <int MODE>
static cudaError_t fwd_nt(const DevGeom& g, int subset, const FwdArgs& a, cudaStream_t s) {
  switch (g.taps) {
    case 1: return fwd_launch<1, MODE>(g, subset, a, s);
    case 2: return fwd_launch<2, MODE>(g, subset, a, s);
    case 3: return fwd_launch<3, MODE>(g, subset, a, s);
    case 4: return fwd_launch<4, MODE>(g, subset, a, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_forward(const DevGeom& g, int subset, int mode, const FwdArgs& a, cudaStream_t s) {
  switch (mode) {
    case FWD_PROJECT: return fwd_nt<FWD_PROJECT>(g, subset, a, s);
    case FWD_SIGMA: return fwd_nt<FWD_SIGMA>(g, subset, a, s);
    case FWD_DATA: return fwd_nt<FWD_DATA>(g, subset, a, s);
    case FWD_EM: return fwd_nt<FWD_EM>(g, subset, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace spdhg
