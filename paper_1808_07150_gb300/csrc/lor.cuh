// The line-integral model both projectors evaluate (device code):
//     (L x)_j = sum_k |LOR_j  intersect voxel_k| x_k
// through one factorisation:
//   * transaxially, a LOR (view v, radial bin r) is a 2-D line; its intersection with pixel
//     (ix, iy) is a parameter interval [ta, tb] (pixel_interval);
//   * axially, the LORs of one michelogram segment differ only by a shift of exactly one slice
//     per plane, so inside a pixel the LOR of plane q meets slab iz = q - j with a length that
//     depends only on j, the segment and [ta, tb] (segment_taps).
// Forward and back projection call these two functions with the same inputs, so each
// (LOR, voxel) length is bit-identical in both directions and the backprojector is the exact
// transpose of the projector (up to the order of the sums).  No float atomics are used.
#pragma once

#include "internal.cuh"

namespace spdhg {

// Error-free transformations (Knuth two-sum, FMA two-product): a + b = s + e, a * b = p + e.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
  p = __fmul_rn(a, b);
  e = __fmaf_rn(a, b, -p);
}

// Transaxial line of (view v, radial bin r) in pixel units: the points X n_perp with
// X . (c, s) = s_r, parameter t along (-s, c), t in [-h, h]  (all as double-float pairs).
struct Line {
  float c_hi, c_lo, s_hi, s_lo;
  float sp_hi, sp_lo, h_hi, h_lo;
  float inv_dx, inv_dy;  // 1 / (-s_hi), 1 / c_hi (0 for a zero component)
};

__device__ __forceinline__ Line make_line(const DevGeom& g, int v, int r) {
  const float4 a = g.view[v];
  const float4 b = g.rad[r];
  const float2 iv = g.view_inv[v];
  return Line{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, iv.x, iv.y};
}

// Intersection of a line with pixel (ix, iy), expressed relative to the foot point of the
// pixel centre on the line: t in tc + [ua, ub], tc = tch + tcl.  The offset of the line from
// the pixel centre and tc are evaluated with error-free transformations, so [ua, ub] is
// resolved to FP32 precision of quantities of order one pixel.  A line lying in a grid line
// belongs to the pixel whose lower edge holds it.
struct PixInt {
  float ua, ub, tch, tcl;
};

__device__ __forceinline__ bool pixel_interval(const DevGeom& g, const Line& L, int ix, int iy, PixInt& out) {
  const float Xc = (float)ix + 0.5f - 0.5f * (float)g.nx;  // pixel centre (exact)
  const float Yc = (float)iy + 0.5f - 0.5f * (float)g.ny;
  float p1, e1, p2, e2, S, eS, D, eD;
  // delta = Xc c + Yc s - s_r: signed distance of the pixel centre from the line
  two_prod(Xc, L.c_hi, p1, e1);
  two_prod(Yc, L.s_hi, p2, e2);
  two_sum(p1, p2, S, eS);
  two_sum(S, -L.sp_hi, D, eD);
  const float delta = __fadd_rn(D, __fadd_rn(__fadd_rn(__fadd_rn(e1, e2), __fadd_rn(eS, eD)),
                                              __fsub_rn(__fmaf_rn(Xc, L.c_lo, __fmul_rn(Yc, L.s_lo)), L.sp_lo)));
  // tc = Yc c - Xc s: line parameter of the foot point
  two_prod(Yc, L.c_hi, p1, e1);
  two_prod(-Xc, L.s_hi, p2, e2);
  two_sum(p1, p2, S, eS);
  two_sum(S, __fadd_rn(__fadd_rn(__fadd_rn(e1, e2), eS), __fsub_rn(__fmul_rn(Yc, L.c_lo), __fmul_rn(Xc, L.s_lo))),
          out.tch, out.tcl);
  // segment ends t = -h, h relative to tc
  float lo = __fadd_rn(__fsub_rn(-L.h_hi, out.tch), __fsub_rn(-L.h_lo, out.tcl));
  float hi = __fadd_rn(__fsub_rn(L.h_hi, out.tch), __fsub_rn(L.h_lo, out.tcl));
  const float ex = __fmul_rn(-delta, L.c_hi), ey = __fmul_rn(-delta, L.s_hi);  // foot point - centre
  const float dx = -L.s_hi, dy = L.c_hi;
  if (dx == 0.f) {
    if (!(ex >= -0.5f && ex < 0.5f)) return false;
  } else {
    const float u1 = __fmul_rn(__fsub_rn(-0.5f, ex), L.inv_dx), u2 = __fmul_rn(__fsub_rn(0.5f, ex), L.inv_dx);
    lo = fmaxf(lo, fminf(u1, u2));
    hi = fminf(hi, fmaxf(u1, u2));
  }
  if (dy == 0.f) {
    if (!(ey >= -0.5f && ey < 0.5f)) return false;
  } else {
    const float u1 = __fmul_rn(__fsub_rn(-0.5f, ey), L.inv_dy), u2 = __fmul_rn(__fsub_rn(0.5f, ey), L.inv_dy);
    lo = fmaxf(lo, fminf(u1, u2));
    hi = fminf(hi, fmaxf(u1, u2));
  }
  out.ua = lo;
  out.ub = hi;
  return hi > lo;
}

// Lengths (voxel units) of the plane-q LOR of component ci in slabs iz = q - (j0 + k), k < NT,
// inside the pixel interval I.  The LOR's slab coordinate at the foot point,
// zeta_c = f + kappa tc, is split exactly into an integer n0 and a fraction in [0, 1); the
// crossings are then solved in local quantities of order one.  Returns j0.
template <int NT>
__device__ __forceinline__ int segment_taps(const DevGeom& g, int r, int ci, const PixInt& I, float* Lk) {
  // ci: the LOR component (its axial tilt); the plane mid-points are those of its segment
  const float4 rs = g.rs[r * g.n_comp + ci];
  const SegDev sd = g.seg[g.comp[ci].seg];
  const float kh = rs.x, kl = rs.y, scale = rs.z;
  float p, e, s1, e1;
  two_prod(kh, I.tch, p, e);
  e = __fadd_rn(e, __fmaf_rn(kh, I.tcl, __fmul_rn(kl, I.tch)));
  two_sum(sd.f_hi, p, s1, e1);
  float n0 = floorf(s1);
  float frac = __fadd_rn(__fsub_rn(s1, n0), __fadd_rn(__fadd_rn(e1, e), sd.f_lo));
  if (frac >= 1.f) {
    frac -= 1.f;
    n0 += 1.f;
  } else if (frac < 0.f) {
    frac += 1.f;
    n0 -= 1.f;
  }
  const int in0 = (int)n0;
  if (kh == 0.f) {
    Lk[0] = __fmul_rn(__fsub_rn(I.ub, I.ua), scale);
#pragma unroll
    for (int k = 1; k < NT; ++k) Lk[k] = 0.f;
    return -in0;  // frac in [0, 1): the LOR stays in one slab
  }
  const float ka = __fmul_rn(kh, I.ua), kb = __fmul_rn(kh, I.ub);
  const float B = __fadd_rn(frac, fmaxf(ka, kb));
  const int j0l = (int)floorf(-B) + 1;  // smallest local j with frac + j + max(kappa u) > 0
  const float inv_k = __frcp_rn(kh);
#pragma unroll
  for (int k = 0; k < NT; ++k) {
    const float u0 = -__fadd_rn(frac, (float)(j0l + k));  // zeta = 0 at u = u0 / kappa
    const float u1 = __fadd_rn(u0, 1.f);                  // zeta = 1 at u = u1 / kappa
    const float t0 = __fmul_rn(u0, inv_k), t1 = __fmul_rn(u1, inv_k);
    const float lo = fmaxf(I.ua, fminf(t0, t1)), hi = fminf(I.ub, fmaxf(t0, t1));
    Lk[k] = hi > lo ? __fmul_rn(__fsub_rn(hi, lo), scale) : 0.f;
  }
  return j0l - in0;
}

// Block-wide exclusive prefix sum of one int per thread (blockDim <= 1024); returns the
// exclusive prefix and writes the total to *total.  Uses `scratch` (>= 33 ints of shared).
__device__ __forceinline__ int block_exclusive_scan(int v, int* scratch, int* total) {
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) scratch[wi] = incl;
  __syncthreads();
  if (wi == 0) {
    int t = lane < nw ? scratch[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    if (lane < nw) scratch[lane] = t;  // inclusive warp totals
    if (lane == 31) scratch[32] = t;
  }
  __syncthreads();
  const int excl = incl - v + (wi > 0 ? scratch[wi - 1] : 0);
  *total = scratch[32];
  __syncthreads();
  return excl;
}

}  // namespace spdhg
