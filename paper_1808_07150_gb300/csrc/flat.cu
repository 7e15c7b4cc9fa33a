// Projectors of flat geometries: one slice, one plane per line, no tilt (2-D scanners).  The general
// kernels put z along the lanes and leave 31 of 32 idle there; here the lanes hold the rows a line
// crosses (forward) or the pixels of an image row (backward).  Both evaluate pixel_interval and
// segment_taps on the general kernels' inputs, so lengths are the same bits.
#include "backward.cuh"
#include "forward.cuh"

namespace spdhg {

// A sum with the rounding errors of its products and additions kept beside it (two-product, two-sum):
// rounded once at the end, so the lanes' split costs no precision.
struct Comp {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float v, float err) {
    float t, e;
    two_sum(s, v, t, e);
    s = t;
    c = __fadd_rn(c, __fadd_rn(e, err));
  }
  __device__ __forceinline__ void fma(float a, float b) {
    float p, e;
    two_prod(a, b, p, e);
    add(p, e);
  }
  // s is the plain sum; where it has left the finite numbers the errors are NaN and s stands alone
  __device__ __forceinline__ float value() const {
    const float v = s + c;
    return v == v ? v : s;
  }
};

bool flat_geometry(const DevGeom& g) { return g.nz == 1 && g.P == 1 && g.n_comp == 1 && g.taps == 1; }

// Forward: `per_line` warps share a line, a lane takes every 32 per_line-th row of the dominant axis; the
// lanes' sums are added by a fixed tree, the warps' in order.  Bound: latency of one chain (table loads,
// a row's intervals, x, the bin's data).  64 x 64, 9 views x 95 bins: 14.9 -> 6.5 us.  One warp up to 32 rows, two up to
// 64 (64 x 64, 9 views x 96 bins: 10.1, 8.3, 9.9 us with 1, 2, 4), then four: 128 x 128 14.0, 12.2, 13.3 us, 256 x 256 24.5,
// 24.7, 25.4 us with 1, 2, 4, level within a tenth, and the shortest chain where an image is far longer.
template <int MODE>
__global__ void __launch_bounds__(128) k_forward_flat(const __grid_constant__ DevGeom g, int subset, int lines, int per_line,
                                                      const __grid_constant__ FwdArgs a) {
  __shared__ float2 sums[4];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, part = wi % per_line;
  const int line = blockIdx.x * (4 / per_line) + wi / per_line;
  Comp sum;
  int l = 0, r = 0, v = 0;
  if (line < lines) {
    l = line / g.R;
    r = line - l * g.R;
    v = subset_view(g, subset, l);
    const Line L = make_line(g, v, r);
    const bool ydom = fabsf(L.c_hi) >= fabsf(L.s_hi);
    const int nrows = ydom ? g.ny : g.nx;
    for (int row = 32 * part + lane; row < nrows; row += 32 * per_line) {
      Entry e[kCandPerRow];
      const int n = row_entries(g, L, ydom, row, e);
#pragma unroll
      for (int k = 0; k < kCandPerRow; ++k) {
        if (k >= n) break;
        float len[4];
        if (segment_taps<1>(g, r, 0, e[k].I, len) == 0) sum.fma(len[0], MODE == FWD_SIGMA ? 1.f : a.x[e[k].col]);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float so = __shfl_down_sync(0xffffffffu, sum.s, o), co = __shfl_down_sync(0xffffffffu, sum.c, o);
    sum.add(so, co);
  }
  if (per_line > 1) {
    if (lane == 0) sums[wi] = make_float2(sum.s, sum.c);
    __syncthreads();
    if (part == 0)
      for (int k = 1; k < per_line; ++k) sum.add(sums[wi + k].x, sums[wi + k].y);
  }
  if (lane == 0 && part == 0 && line < lines) forward_epilogue<MODE>(g, a, subset, v, l, r, 0, sum.value());
}

cudaError_t launch_forward_flat(const DevGeom& g, int subset, int mode, const FwdArgs& a, cudaStream_t s) {
  const int lines = subset_views(g, subset) * g.R, rows = g.nx > g.ny ? g.nx : g.ny;
  const int per_line = rows <= 32 ? 1 : (rows <= 64 ? 2 : 4), per_block = 4 / per_line;
  if (lines == 0) return cudaSuccess;
  if (mode == FWD_DATA && !a.sigma) return cudaErrorInvalidValue;
  if ((mode == FWD_DATA || mode == FWD_EM) && (!a.b || !a.r || !a.wdy)) return cudaErrorInvalidValue;
  const int grid = (lines + per_block - 1) / per_block;
  switch (mode) {
    case FWD_PROJECT: k_forward_flat<FWD_PROJECT><<<grid, 128, 0, s>>>(g, subset, lines, per_line, a); break;
    case FWD_SIGMA: k_forward_flat<FWD_SIGMA><<<grid, 128, 0, s>>>(g, subset, lines, per_line, a); break;
    case FWD_DATA: k_forward_flat<FWD_DATA><<<grid, 128, 0, s>>>(g, subset, lines, per_line, a); break;
    case FWD_EM: k_forward_flat<FWD_EM><<<grid, 128, 0, s>>>(g, subset, lines, per_line, a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Backward: a block owns 32 consecutive pixels of the image, warp w their views w, w + 8, ...; a lane adds
// up its pixel's bins, and warp 0 the warps' sums in order.  Bound: latency (table loads, a few candidate
// bins per view).  64 x 64, 9 views x 95 bins: 19.2 -> 7.0 us.
__global__ void __launch_bounds__(256) k_backward_flat(const __grid_constant__ DevGeom g, int subset, int mode,
                                                       const __grid_constant__ BwdArgs a) {
  __shared__ float2 sums[8][32];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, pix = blockIdx.x * 32 + lane, nviews = subset_views(g, subset);
  const bool live = pix < g.nx * g.ny;
  float xo = 0.f, zo = 0.f, To = 0.f;
  if (wi == 0 && live && mode != BWD_OUT) {  // requested before the sums
    To = a.T[pix];
    if (mode != BWD_SENS) xo = a.x[pix];
    if (mode == BWD_UPDATE) zo = a.z[pix];
  }
  Comp part;
  if (live) {
    const int iy = pix / g.nx, ix = pix - iy * g.nx;
    const float Xc = (float)ix + 0.5f - 0.5f * (float)g.nx, Yc = (float)iy + 0.5f - 0.5f * (float)g.ny;
    for (int l = wi; l < nviews; l += 8) {
      const int v = subset_view(g, subset, l);
      const float4 cs = g.view[v];
      const float hw = 0.5f * (fabsf(cs.x) + fabsf(cs.z)), sc = Xc * cs.x + Yc * cs.z;
      const int r1 = min(g.R - 1, (int)floorf((sc + hw) * g.inv_drp + g.half_R + g.bw_margin));
      for (int r = max(0, (int)ceilf((sc - hw) * g.inv_drp + g.half_R - g.bw_margin)); r <= r1; ++r) {
        PixInt I;
        float len[4];
        if (pixel_interval(g, make_line(g, v, r), ix, iy, I) && segment_taps<1>(g, r, 0, I, len) == 0)
          part.fma(len[0], a.w[(size_t)l * g.R + r]);
      }
    }
  }
  sums[wi][lane] = make_float2(part.s, part.c);
  __syncthreads();
  if (wi > 0 || !live) return;
#pragma unroll
  for (int k = 1; k < 8; ++k) part.add(sums[k][lane].x, sums[k][lane].y);
  const float sum = part.value();
  if (mode == BWD_UPDATE) {
    // z = z + dz;  zbar = z + dz / p_i;  next primal step x = max(x - T zbar, 0)
    const float zn = zo + sum;
    a.z[pix] = zn;
    a.x[pix] = prox_nonneg(xo - To * fmaf(sum, a.inv_p, zn));
  } else if (mode == BWD_OUT) {
    a.out[pix] = sum;
  } else if (mode == BWD_SENS) {
    if (sum > 0.f) a.T[pix] = fminf(To, a.sens_num / sum);
  } else {
    a.x[pix] = To > 0.f ? xo * sum / To : 0.f;
  }
}

cudaError_t launch_backward_flat(const DevGeom& g, int subset, int mode, const BwdArgs& a, cudaStream_t s) {
  if (mode != BWD_OUT && mode != BWD_SENS && mode != BWD_UPDATE && mode != BWD_EM) return cudaErrorInvalidValue;
  k_backward_flat<<<(g.nx * g.ny + 31) / 32, 256, 0, s>>>(g, subset, mode, a);
  return cudaGetLastError();
}

}  // namespace spdhg
