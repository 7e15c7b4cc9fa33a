// Ray-driven forward projector, fused with the KL dual prox of SPDHG.  One translation unit per tap
// count NT instantiates launch_forward_nt.
#pragma once

#include <algorithm>

#include "lor.cuh"


namespace spdhg {

struct Entry {
  int col;  // iy * nx + ix
  PixInt I;
};

constexpr int kCandPerRow = 4;
constexpr float kPixMargin = 0.01f;  // pixels: covers the FP32 rounding of a row's crossing points

// Pixels of `row` (along the dominant axis of the line) that the line crosses.  Candidates come
// from approximate arithmetic with a margin; pixel_interval decides exactly.
__device__ __forceinline__ int row_entries(const DevGeom& g, const Line& L, bool ydom, int row, Entry* e) {
  const float c = L.c_hi, s = L.s_hi, sp = L.sp_hi, h = L.h_hi;
  float t0, t1;
  if (ydom) {  // y in [Y0, Y0 + 1);  y(t) = sp s + t c
    const float Y0 = (float)row - 0.5f * (float)g.ny;
    t0 = (Y0 - sp * s) * L.inv_dy;
    t1 = (Y0 + 1.f - sp * s) * L.inv_dy;
  } else {     // x in [X0, X0 + 1);  x(t) = sp c - t s
    const float X0 = (float)row - 0.5f * (float)g.nx;
    t0 = (X0 - sp * c) * L.inv_dx;
    t1 = (X0 + 1.f - sp * c) * L.inv_dx;
  }
  const float tlo = fmaxf(fminf(t0, t1), -h - kPixMargin), thi = fminf(fmaxf(t0, t1), h + kPixMargin);
  if (thi < tlo) return 0;
  const float ca = ydom ? sp * c - tlo * s : sp * s + tlo * c;
  const float cb = ydom ? sp * c - thi * s : sp * s + thi * c;
  const float half = 0.5f * (float)(ydom ? g.nx : g.ny);
  const int nc = ydom ? g.nx : g.ny;
  const int cmin = max((int)floorf(fminf(ca, cb) + half - kPixMargin), 0);
  const int cmax = min((int)floorf(fmaxf(ca, cb) + half + kPixMargin), nc - 1);
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

constexpr int kFwdChunk = 32;         // most pixel entries per double-buffered chunk
constexpr int kFwdMaxWarps = 12;      // warps per block

// Tap record of one (pixel entry, component): first tap's length and a word, 4 x the offset of plane
// 0's tap 0 in the chunk's staged x columns | taps - 1; the further taps' lengths apart.
template <int NT>
struct alignas(NT > 3 ? 16 : (NT > 2 ? 8 : 4)) MoreLengths {
  float l[NT > 3 ? 4 : (NT > 2 ? 2 : 1)];
};

__device__ __forceinline__ float2 ffma2_bcast(float l, float xa, float xb, float2 acc) {
  return __ffma2_rn(make_float2(l, l), make_float2(xa, xb), acc);
}

// s[w] += l p[32 w], w < W (two words per packed FMA)
template <int W>
__device__ __forceinline__ void words_fma(float l, const float* p, float2 s[2]) {
  if constexpr (W == 1) s[0].x = fmaf(l, p[0], s[0].x);
  if constexpr (W >= 2) s[0] = ffma2_bcast(l, p[0], p[32], s[0]);
  if constexpr (W == 3) s[1].x = fmaf(l, p[64], s[1].x);
  if constexpr (W == 4) s[1] = ffma2_bcast(l, p[64], p[96], s[1]);
}

// Sum of the entries e0, e0 + step, ... < ne of one chunk and component over W words of 32 planes;
// xl is the chunk's staged columns at this lane's first plane.
template <int NT, int W>
__device__ __forceinline__ void gather_entries(const float* xl, const float2* recA, const MoreLengths<NT>* recB, int e0,
                                               int ne, int step, float2 s[2]) {
#pragma unroll 2
  for (int e = e0; e < ne; e += step) {
    const float2 A = recA[e];
    const unsigned word = __float_as_uint(A.y);
    const float* p = reinterpret_cast<const float*>(reinterpret_cast<const char*>(xl) + (word & ~3u));
    words_fma<W>(A.x, p, s);
    if constexpr (NT > 1) {
      if (word & 3u) {
        const MoreLengths<NT> B = recB[e];
        words_fma<W>(B.l[0], p - 1, s);
        if constexpr (NT > 2) {
          if (word & 2u) {
            words_fma<W>(B.l[1], p - 2, s);
            if constexpr (NT > 3) {
              if ((word & 3u) == 3u) words_fma<W>(B.l[2], p - 3, s);
            }
          }
        }
      }
    }
  }
}

template <int NT>
__device__ __forceinline__ void gather_words(int words, const float* xl, const float2* recA, const MoreLengths<NT>* recB,
                                             int e0, int ne, int step, float2 s[2]) {
  switch (words) {  // warp-uniform
    case 4: gather_entries<NT, 4>(xl, recA, recB, e0, ne, step, s); break;
    case 3: gather_entries<NT, 3>(xl, recA, recB, e0, ne, step, s); break;
    case 2: gather_entries<NT, 2>(xl, recA, recB, e0, ne, step, s); break;
    case 1: gather_entries<NT, 1>(xl, recA, recB, e0, ne, step, s); break;
    default: break;
  }
}

__device__ __forceinline__ void cp_async4_if(unsigned d, const float* s, bool on) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p cp.async.ca.shared.global [%0], [%1], 4;\n\t}\n" ::"r"(d),
               "l"(s), "r"((int)on)
               : "memory");
}

// What a mode does with one bin's line integral `sum` (plane p of line (v, r); l: the view's place in
// the subset).
template <int MODE>
__device__ __forceinline__ void forward_epilogue(const DevGeom& g, const FwdArgs& a, int subset, int v, int l, int r, int p, float sum) {
  const size_t j = ((size_t)v * g.R + r) * g.P + p;
  const size_t jl = ((size_t)l * g.R + r) * g.P + p;  // subset-local index (= j for bin subsets)
  if (!bin_in_subset(g, subset, j)) {  // a bin of another subset: not written; no dual change
    if (MODE == FWD_DATA || MODE == FWD_EM) a.wdy[jl] = 0.f;
    return;
  }
  const float mu = a.mult ? a.mult[j] : 1.f;
  if (MODE == FWD_EM) {
    // EM ratio backprojected by P^T = L^T diag(mult): mult_j b_j / ((P x)_j + r_j)  (Eq. EQU:OSEM)
    const float bj = a.b[j];
    a.wdy[jl] = bj > 0.f ? mu * bj / fmaf(mu, sum, a.r[j]) : 0.f;
  } else if (MODE == FWD_PROJECT) {
    a.out[j] = mu * sum;
  } else if (MODE == FWD_SIGMA) {
    // sigma_j = gamma rho / (P_i 1)_j,  (P_i 1)_j = mult_j * chord_j  (Eq. EQU:STEPSIZE:PRECOND)
    const float a1 = mu * sum;
    a.out[j] = a1 > 0.f ? a.gamma_rho / a1 : 0.f;
  } else {
    // KL dual prox on this bin:  y+ = prox_{sigma varphi*}(y + sigma (P_i x)_j), evaluated as
    // 2 (u - sigma b) / (u + 1 + sqrt((u - 1)^2 + 4 sigma b)),  u = y + sigma ((P_i x)_j + r_j),
    // which equals 1/2 [u + 1 - sqrt((u - 1)^2 + 4 sigma b)] without its cancellation.
    const float sigma = a.sigma[j];
    const float yj = a.y[j];
    const float bj = a.b[j];
    const float u = fmaf(sigma, fmaf(mu, sum, a.r[j]), yj);
    const float sb = sigma * bj;
    const float um = u - 1.f;
    const float root = sqrtf(fmaf(um, um, 4.f * sb));
    const float yn = 2.f * (u - sb) / (u + 1.f + root);
    a.y[j] = yn;
    a.wdy[jl] = mu * (yn - yj);
  }
}

// Forward projection.  Block (line, row part, plane part) owns the rows [row_lo, row_hi) of one
// transaxial LOR line (view, radial bin) and a contiguous range of the geometry's plane tasks (up to
// four words of 32 consecutive planes of one segment); a warp owns one task, lane l plane q0 + l of
// each word.  All threads first find the pixels the line crosses in those rows (exact intervals,
// compacted); the entries are then processed in chunks: the x columns of chunk c+1 are copied to
// shared memory (cp.async, 16 bytes at a time where the columns are aligned) inside zero frames wide
// enough for every tap of every plane of the segments (the axial bound of the geometry, so no plane
// needs a range test; lanes past a segment's last plane read up to 31 floats beyond their frame, hence the
// 32 spare floats after the last column, and are not written), and its axial taps computed while chunk c is accumulated.  One tap record
// serves all words of a task, packed FP32 FMAs accumulate two words.  Mashed geometries sum the
// components of the segment one after the other, each kept by the planes that include it, and a chunk's
// component sums before they join the bin's (each joining by itself, a bin of nine components came to 2.7
// units (2^-24) from its FP64 value instead of 1.3, relative L2; 38.7 -> 39.1 us).  When a
// line has few tasks, egroups warps share each, warp group k taking the entries k, k + egroups, ...
// of every chunk; group 0 adds the other groups' sums in group order.  When several row parts share
// a line, each writes partial plane sums and the last one to finish reduces them in a fixed order.
//
// Bound: instruction issue (60 % active at the mMR scale, 36 M warp instructions, 58 M before with two
// words per warp), then latency with 344 lines on 152 SMs.  So a record's reads and address serve up
// to four words, and the copies of aligned columns are dealt out in 16-byte pieces.  Measured on
// GB300, per launch: 344 x 344 x 127 voxels, one view of 344 x 837 bins, 92 -> 63 us; 171 x 171 x 92,
// 12-13 views x 250 planes, 128 -> 77 us (115 with a warp per column of 4-byte copies); 128 x 128 x 64,
// 8-9 views, three mashed components, 58 -> 39 us.  Blocks with entry groups are bounded to 56
// registers (three blocks of 12 warps per SM; 39 against 43 us at 64), the others to 80 (63 against
// 65 us at the mMR scale).
template <int NT, int MODE, bool GROUPS, bool MASHED>
__global__ void __launch_bounds__(kFwdMaxWarps * 32, GROUPS ? 3 : 2)
    k_forward(const __grid_constant__ DevGeom g, int subset, int ecap, int rsplit, int tasks_per_part, int ncomp_tab,
              int chunk, int egroups_arg, const __grid_constant__ FwdArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int scan_scratch[33];
  const int FL = g.fz_lo, xs_stride = g.fz_stride;
  float* xs = reinterpret_cast<float*>(smem);                                        // [2][chunk][xs_stride] + 32 spare
  float2* recA = reinterpret_cast<float2*>(xs + 2 * chunk * xs_stride + 32);         // [2][ncomp_tab][chunk]
  MoreLengths<NT>* recB = reinterpret_cast<MoreLengths<NT>*>(recA + 2 * ncomp_tab * chunk);
  Entry* ent = reinterpret_cast<Entry*>(recB + (NT > 1 ? 2 * ncomp_tab * chunk : 0));  // [ecap]
  float* group_acc = reinterpret_cast<float*>(ent + ecap);                           // [egroups - 1][tasks][4][32]
  const int nz = g.nz;

  const int line = blockIdx.x, rpart = blockIdx.y, ppart = blockIdx.z;
  const int l = line / g.R, r = line - l * g.R;
  const int v = subset_view(g, subset, l);
  const Line L = make_line(g, v, r);

  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int egroups = GROUPS ? egroups_arg : 1;
  const int ntw = GROUPS ? nw / egroups : nw, tw = GROUPS ? wi % ntw : wi, eg = GROUPS ? wi / ntw : 0;
  const int tfirst = ppart * tasks_per_part, tlast = min(g.n_tasks, tfirst + tasks_per_part) - 1;
  const SegDev seg_lo = g.seg[g.tasks[tfirst].x], seg_hi = g.seg[g.tasks[tlast].x];
  const int c_lo = seg_lo.c0, ncb = seg_hi.c0 + seg_hi.nc - c_lo;  // the LOR components of the block's segments
  const int4 task = g.tasks[min(tfirst + tw, tlast)];              // segment, first plane, words
  const SegDev sd = g.seg[task.x];
  const int words = tfirst + tw <= tlast ? task.z : 0;
  const int q = task.y + lane;                                     // plane of word 0; word w: q + 32 w

  // zero frames of the staged columns (never overwritten); SIGMA stages ones: the projection of
  // the constant image is the chord of each LOR inside the image
  {
    const int per = xs_stride - nz;  // frame floats per column
    for (int i = threadIdx.x; i < 2 * chunk * per; i += blockDim.x) {
      const int col = i / per, k = i - col * per;
      xs[col * xs_stride + (k < FL ? k : k + nz)] = 0.f;
    }
  }
  if (MODE == FWD_SIGMA)
    for (int i = threadIdx.x; i < 2 * chunk * nz; i += blockDim.x) {
      const int col = i / nz;
      xs[col * xs_stride + FL + (i - col * nz)] = 1.f;
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

  const int csh = __ffs(chunk) - 1;  // chunk is a power of two
  const bool aligned = (nz & 3) == 0 && (reinterpret_cast<size_t>(a.x) & 15) == 0;
  const int nz4 = max(nz >> 2, 1), piece_e = threadIdx.x / nz4, piece_k = threadIdx.x - piece_e * nz4;
  const int step_e = blockDim.x / nz4, step_k = blockDim.x - step_e * nz4;
  auto stage = [&](int c) {  // x columns + taps of chunk c into buffer c & 1
    const int buf = c & 1;
    const int e0 = c << csh, ne = min(chunk, n_ent - e0);
    if (MODE != FWD_SIGMA) {
      const unsigned xb = (unsigned)__cvta_generic_to_shared(xs + (buf << csh) * xs_stride + FL);
      if (aligned) {
        // 16-byte pieces, dealt to the threads across the entries
        int e = piece_e, k = piece_k;
        while (e < ne) {
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(xb + 4 * e * xs_stride + 16 * k),
                       "l"(a.x + (size_t)ent[e0 + e].col * nz + 4 * k)
                       : "memory");
          e += step_e;
          k += step_k;
          if (k >= nz4) {
            k -= nz4;
            ++e;
          }
        }
      } else {
        // one warp per entry, lanes along z
        for (int e = wi; e < ne; e += nw) {
          const float* src = a.x + (size_t)ent[e0 + e].col * nz + lane;
          const unsigned dst = xb + 4 * e * xs_stride + 4 * lane;
          cp_async4_if(dst, src, lane < nz);
          if (nz > 32) cp_async4_if(dst + 128, src + 32, lane + 32 < nz);
          if (nz > 64) cp_async4_if(dst + 256, src + 64, lane + 64 < nz);
          if (nz > 96) cp_async4_if(dst + 384, src + 96, lane + 96 < nz);
          for (int k = 128; k + lane < nz; k += 32) cp_async4_if(dst + 4 * k, src + k, true);
        }
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    const int rb = (buf * ncomp_tab) << csh;
    for (int it = threadIdx.x; it < ncb << csh; it += blockDim.x) {
      const int gs = it >> csh, e = it & (chunk - 1);
      if (e >= ne) continue;
      float Lk[4] = {0.f, 0.f, 0.f, 0.f};
      int j0 = segment_taps<NT>(g, r, c_lo + gs, ent[e0 + e].I, Lk);
      // the geometry's axial bound keeps every read inside the framed column; the clamp only
      // guards shared memory should a rounding case fall outside it
      const CompDev cd = g.comp[c_lo + gs];
      j0 = min(max(j0, cd.jlo), cd.jhi);
      int nt = 1;
#pragma unroll
      for (int k = 1; k < NT; ++k)
        if (Lk[k] != 0.f) nt = k + 1;
      recA[rb + it] = make_float2(Lk[0], __uint_as_float((unsigned)(4 * (e * xs_stride + FL - j0)) | (unsigned)(nt - 1)));
      if constexpr (NT > 1) {
        MoreLengths<NT> B;
        B.l[0] = Lk[1];
        if constexpr (NT > 2) B.l[1] = Lk[2];
        if constexpr (NT > 3) B.l[2] = Lk[3];
        recB[rb + it] = B;
      }
    }
  };

  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  unsigned incl[4] = {0u, 0u, 0u, 0u};  // mashed: components of the segment each plane sums
  if (MASHED) {
#pragma unroll
    for (int w = 0; w < 4; ++w)
      for (int c = 0; c < sd.nc; ++c) {
        const CompDev cd = g.comp[sd.c0 + c];
        const int dq = q + 32 * w - cd.qlo;
        if (q + 32 * w < cd.qhi && dq >= 0 && (dq & cd.smask) == 0) incl[w] |= 1u << c;
      }
  }
  const int nchunks = (n_ent + chunk - 1) >> csh;
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
    const int ne = min(chunk, n_ent - (c << csh));
    const float* xl = xs + (buf << csh) * xs_stride + q;
    const int rb = (buf * ncomp_tab + sd.c0 - c_lo) << csh;
    if (!MASHED) {
      float2 s[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      gather_words<NT>(words, xl, recA + rb, recB + rb, eg, ne, egroups, s);
      acc[0] += s[0].x;
      acc[1] += s[0].y;
      acc[2] += s[1].x;
      acc[3] += s[1].y;
    } else {
      // the components' sums of the chunk are added first
      float sum[4] = {0.f, 0.f, 0.f, 0.f};
      for (int ci = 0; ci < sd.nc; ++ci) {
        float2 s[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        gather_words<NT>(words, xl, recA + rb + (ci << csh), recB + rb + (ci << csh), eg, ne, egroups, s);
        sum[0] += (incl[0] >> ci) & 1u ? s[0].x : 0.f;
        sum[1] += (incl[1] >> ci) & 1u ? s[0].y : 0.f;
        sum[2] += (incl[2] >> ci) & 1u ? s[1].x : 0.f;
        sum[3] += (incl[3] >> ci) & 1u ? s[1].y : 0.f;
      }
#pragma unroll
      for (int w = 0; w < 4; ++w) acc[w] += sum[w];
    }
    __syncthreads();
  }

  bool writes = true;
  if (GROUPS) {
    // entry groups 1.. hand their partial sums to group 0, which adds them in group order
    if (eg > 0) {
#pragma unroll
      for (int w = 0; w < 4; ++w) group_acc[(((eg - 1) * ntw + tw) * 4 + w) * 32 + lane] = acc[w];
    }
    __syncthreads();
    writes = eg == 0;  // group 0 writes the planes
    if (writes)
      for (int k = 1; k < egroups; ++k) {
#pragma unroll
        for (int w = 0; w < 4; ++w) acc[w] += group_acc[(((k - 1) * ntw + tw) * 4 + w) * 32 + lane];
      }
  }

  if (rsplit > 1) {
    // publish this block's partial sums; the last row part of the (line, plane part) reduces them
    __shared__ unsigned last_sh;
    const size_t pbase = ((size_t)line * rsplit + rpart) * g.P + sd.p0 + q;
#pragma unroll
    for (int w = 0; w < 4; ++w)
      if (writes && w < words && q + 32 * w < sd.n) a.part_acc[pbase + 32 * w] = acc[w];
    __threadfence();
    __syncthreads();
    const size_t ticket = (size_t)line * gridDim.z + ppart;
    if (threadIdx.x == 0) last_sh = (atomicAdd(a.tickets + ticket, 1u) == (unsigned)rsplit - 1u) ? 1u : 0u;
    __syncthreads();
    if (!last_sh) return;
    __threadfence();
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      if (!(writes && w < words && q + 32 * w < sd.n)) continue;
      float sa = 0.f;
      for (int k = 0; k < rsplit; ++k)  // fixed order: deterministic
        sa += __ldcg(a.part_acc + ((size_t)line * rsplit + k) * g.P + sd.p0 + q + 32 * w);
      acc[w] = sa;
    }
    if (threadIdx.x == 0) a.tickets[ticket] = 0u;  // ready for the next launch
  }

#pragma unroll
  for (int w = 0; w < 4; ++w) {
    if (!(writes && w < words && q + 32 * w < sd.n)) continue;
    forward_epilogue<MODE>(g, a, subset, v, l, r, sd.p0 + q + 32 * w, acc[w]);
  }
}

// instantiated per tap count in forward_taps<NT>.cu
template <int NT, int MODE>
cudaError_t fwd_launch(const DevGeom& g, int subset, const FwdArgs& a, cudaStream_t s) {
  const int nrows = g.nx > g.ny ? g.nx : g.ny;
  const int ecap = 3 * nrows + 8;  // at most two pixels per row of the dominant axis, and rounding slivers
  const int per_part = forward_tasks_per_part(g), parts = forward_parts(g), egroups = forward_entry_groups(g);
  const int threads = 32 * per_part * egroups;
  if (threads > 32 * kFwdMaxWarps) return cudaErrorInvalidValue;
  // a block computes the taps of the components of the segments its tasks span
  const int ncomp_tab = g.max_part_comps[per_part];
  const size_t rec = sizeof(float2) + (NT > 1 ? sizeof(MoreLengths<NT>) : 0);
  auto bytes = [&](int chunk) {
    return ((size_t)2 * chunk * g.fz_stride + 32) * sizeof(float) + (size_t)2 * ncomp_tab * chunk * rec +
           (size_t)ecap * sizeof(Entry) + (size_t)(egroups - 1) * per_part * 4 * 32 * sizeof(float);
  };
  // 72 KB leave room for three blocks per SM (the mMR scale: 71 KB, 63 us; 16 entries a chunk, 74 us)
  int chunk = kFwdChunk;
  while (chunk > 4 && bytes(chunk) > 72 * 1024) chunk /= 2;
  const size_t smem = bytes(chunk);
  if (smem > 200 * 1024) return cudaErrorInvalidValue;
  if (MODE == FWD_DATA && !a.sigma) return cudaErrorInvalidValue;
  if ((MODE == FWD_DATA || MODE == FWD_EM) && (!a.b || !a.r || !a.wdy)) return cudaErrorInvalidValue;
  auto kern = g.mashed ? (egroups > 1 ? k_forward<NT, MODE, true, true> : k_forward<NT, MODE, false, true>)
                       : (egroups > 1 ? k_forward<NT, MODE, true, false> : k_forward<NT, MODE, false, false>);
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
  kern<<<grid, threads, smem, s>>>(g, subset, ecap, rsplit, per_part, ncomp_tab, chunk, egroups, a);
  return cudaGetLastError();
}

template <int NT>
cudaError_t launch_forward_nt(const DevGeom& g, int subset, int mode, const FwdArgs& a, cudaStream_t s) {
  switch (mode) {
    case FWD_PROJECT: return fwd_launch<NT, FWD_PROJECT>(g, subset, a, s);
    case FWD_SIGMA: return fwd_launch<NT, FWD_SIGMA>(g, subset, a, s);
    case FWD_DATA: return fwd_launch<NT, FWD_DATA>(g, subset, a, s);
    case FWD_EM: return fwd_launch<NT, FWD_EM>(g, subset, a, s);
    default: return cudaErrorInvalidValue;
  }
}

extern template cudaError_t launch_forward_nt<1>(const DevGeom&, int, int, const FwdArgs&, cudaStream_t);
extern template cudaError_t launch_forward_nt<2>(const DevGeom&, int, int, const FwdArgs&, cudaStream_t);
extern template cudaError_t launch_forward_nt<3>(const DevGeom&, int, int, const FwdArgs&, cudaStream_t);
extern template cudaError_t launch_forward_nt<4>(const DevGeom&, int, int, const FwdArgs&, cudaStream_t);

}  // namespace spdhg
