// Prior block of SPDHG (block n of the generic problem, Eq. EQU:SETTING:TV):
//   q+ = prox_{sigma f_n*}(q + sigma A_n x),  dz = A_n^T (q+ - q),
// with A_n = grad (TV, aTV) or D grad (dTV), f_n = alpha||.||_{2,1} (TV, dTV) or alpha||.||_{1,1}
// (aTV), fused with the dual-sum update z += dz and the next primal step
// x = max(x - T (z + dz / p_n), 0).  grad is the forward difference with a zero last row
// (Neumann) at unit spacing.  The stencil reads x and q of the voxel and of its three lower
// neighbours, so x and q are ping-ponged (read *_in, write *_out) and tiles never race.
//
// All prior kernels march: a block owns `cols - 1` voxel columns in x (plus one halo column whose
// duals are recomputed, not written) and the whole z extent, lanes along z, one voxel per thread,
// and walks along y over `ychunk` rows (plus one warm-up row).  Every array is read straight into
// registers one row ahead; the stencil's x and z neighbours are loads that hit the lines the
// neighbouring threads requested a row before.  The dual change of the neighbour in y is carried in a
// register, the one in z comes by shuffle (shared memory between warps), the one in x through
// shared memory, double-buffered, with one barrier per row.
#include <algorithm>

#include "internal.cuh"

namespace spdhg {

// Dual update of one voxel: g = A_n x (forward differences; dTV: D g with
// D = I - gamma_d xi xi^T, xi = grad v / sqrt(|grad v|^2 + eta^2)), q+ = proj(q + sigma g),
// b = D^T (q+ - q).  The ball projection q+ = qa min(1, alpha / |qa|) uses one reciprocal
// square root.  Returns b and q+.
template <int KIND>
__device__ __forceinline__ void dual_update(const PriorArgs& a, const float gr_in[3], const float gv[3],
                                            const float qo[3], float b[3], float qn[3]) {
  float gr[3] = {gr_in[0], gr_in[1], gr_in[2]};
  float xi[3] = {0.f, 0.f, 0.f};
  if (KIND == SPDHG_PRIOR_DTV) {
    const float inv = rsqrtf(fmaf(gv[0], gv[0], fmaf(gv[1], gv[1], fmaf(gv[2], gv[2], a.eta2))));
#pragma unroll
    for (int k = 0; k < 3; ++k) xi[k] = gv[k] * inv;
    const float gd = a.gamma_d * (xi[0] * gr[0] + xi[1] * gr[1] + xi[2] * gr[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) gr[k] -= gd * xi[k];
  }
  float qa[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) qa[k] = fmaf(a.sigma, gr[k], qo[k]);
  if (KIND == SPDHG_PRIOR_ATV) {
#pragma unroll
    for (int k = 0; k < 3; ++k) qn[k] = fminf(fmaxf(qa[k], -a.alpha), a.alpha);
  } else {
    const float n2 = fmaf(qa[0], qa[0], fmaf(qa[1], qa[1], qa[2] * qa[2]));
    const float sc = fminf(1.f, a.alpha * rsqrtf(n2));  // n2 = 0 gives +inf -> 1
#pragma unroll
    for (int k = 0; k < 3; ++k) qn[k] = qa[k] * sc;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) b[k] = qn[k] - qo[k];
  if (KIND == SPDHG_PRIOR_DTV) {
    const float d = a.gamma_d * (xi[0] * b[0] + xi[1] * b[1] + xi[2] * b[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) b[k] -= d * xi[k];
  }
}

// The marching directions: z' along the lanes, x' across the columns, y' marched.  Flat images
// (nz = 1) march with x along the lanes, so that a warp holds 32 pixels instead of one: 256 x 256, TV 20.2 -> 6.6 us,
// TGV 45.6 -> 9.2 us a block.  At most eight warps of x, the width of the z columns; wider images still march
// with z along the lanes (257 x 257: TV 21.9 us where lanes along x would take 6.9).
struct March {
  int nx, ny, nz;    // extents along x', y', z'
  int sx, sy;        // voxel strides of x' and y' (z': 1)
  int kx, ky, kz;    // gradient component of each direction
  int cols, zw, ychunk;
};

static March march_of(const DevGeom& g) {
  if (g.nz == 1 && g.nx <= 256) return March{1, g.ny, g.nx, 0, g.nx, 2, 1, 0, 0, 0, 0};
  return March{g.nx, g.ny, g.nz, g.nz, g.nx * g.nz, 0, 1, 2, 0, 0, 0};
}

// Columns per block (at most `warps` warps) and rows per march: about one block per SM in all, so that
// few rows and columns are computed twice (344 x 344 x 127, dTV: 8 columns 141 us, 7 and 6 columns 169,
// blocks of 512 threads with 4 columns 191; 115 rows 141 us, 58 rows 143, 29 rows 145).
static bool march_shape(const DevGeom& g, March& m, int warps) {
  m.zw = (m.nz + 31) / 32;
  if (2 * m.zw > 32) return false;
  // cols columns of vz voxels a thread: what never fitted 32 warps stays refused, although a thread now
  // holds one voxel and the columns are bounded below
  const int knob = g.tune[SPDHG_TUNE_PRIOR_COLS], vz = std::max(1, g.tune[SPDHG_TUNE_PRIOR_VZ]);
  if (knob * ((g.nz + 32 * vz - 1) / (32 * vz)) > 32) return false;
  m.cols = std::max(2, std::min(warps / m.zw, knob ? knob : std::min(16, m.nx + 1)));
  const int gx = (m.nx + m.cols - 2) / (m.cols - 1);
  const int chunks = std::max(1, std::min(m.ny, 152 / gx));
  m.ychunk = g.tune[SPDHG_TUNE_PRIOR_YCHUNK] ? g.tune[SPDHG_TUNE_PRIOR_YCHUNK] : (m.ny + chunks - 1) / chunks;
  return true;
}

static dim3 march_grid(const March& m) {
  return dim3((m.nx + m.cols - 2) / (m.cols - 1), (m.ny + m.ychunk - 1) / m.ychunk);
}

constexpr int kPriorWarps = 32;  // one block per SM at 64 registers

// Bound: latency of one row's loads at 76 % of the measured copy bandwidth (dTV moves 48 bytes a voxel;
// 344 x 344 x 127: 147 -> 141 us, 87 M warp instructions, 115 M when x and v went through a shared-memory
// pipeline; 128 x 128 x 64, TV: 14.3 -> 12.5 us; 64 x 64 x 1, TV: 8.0 -> 6.3 us).  Copying q, z, T three
// rows ahead into shared memory took 302 us.
template <int KIND>
__global__ void __launch_bounds__(kPriorWarps * 32, 1) k_prior(March m, PriorArgs a, int N) {
  extern __shared__ float sh[];
  constexpr bool dtv = KIND == SPDHG_PRIOR_DTV;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c = w / m.zw, zi = w - c * m.zw, zc = m.zw * 32;
  const int iz = zi * 32 + lane, ix = blockIdx.x * (m.cols - 1) - 1 + c;  // column 0: the lower halo
  const int nx = m.nx, ny = m.ny, nz = m.nz, sx = m.sx, sy = m.sy;
  const bool live = ix >= 0 && ix < nx && iz < nz, owner = live && c >= 1;
  const bool hx = live && ix < nx - 1, hz = live && iz < nz - 1;
  const int y0 = blockIdx.y * m.ychunk, y1 = min(ny, y0 + m.ychunk);
  const int ys = y0 > 0 ? y0 - 1 : 0;               // first row computed (warm-up row for y0 > 0)
  float* sbx = sh;                                  // [2][cols][zc] b_x
  float* sbz = sh + 2 * m.cols * zc;                // [2][cols][zw] b_z of each warp's last lane
  const float *qx = a.q_in + (size_t)m.kx * N, *qy = a.q_in + (size_t)m.ky * N, *qz = a.q_in + (size_t)m.kz * N;
  float *ox = a.q_out + (size_t)m.kx * N, *oy = a.q_out + (size_t)m.ky * N, *oz = a.q_out + (size_t)m.kz * N;
  const float *X = a.x_in, *V = a.side;
  // Dead lanes read a live voxel (their duals are never used), and a neighbour past the end is the
  // voxel itself, so the loads need no tests.  The difference there is 0 also where the voxel is not finite.
  const int dx = hx ? sx : 0, dz1 = hz ? 1 : 0;
  int i = ys * sy + (live ? ix * sx + iz : 0);
  // this row: x and v of the voxel and of its neighbours in y, x, z; q, z, T
  float xc = X[i], xd = X[i + (ys < ny - 1 ? sy : 0)], xr = X[i + dx], xu = X[i + dz1];
  float vc = 0.f, vd = 0.f, vr = 0.f, vu = 0.f;
  if (dtv) {
    vc = V[i];
    vd = V[i + (ys < ny - 1 ? sy : 0)];
    vr = V[i + dx];
    vu = V[i + dz1];
  }
  float q0 = qx[i], q1 = qy[i], q2 = qz[i], zo = a.z[i], To = a.T[i], by = 0.f;
  float* bx = sbx + c * zc + iz;
  float* bz = sbz + c * m.zw + zi;
  int flip = m.cols * zc, flipz = m.cols * m.zw;
#pragma unroll 2
  for (int iy = ys; iy < y1; ++iy) {
    // the next row's operands (the last row asks for its own again)
    const int j = i + (iy + 1 < y1 ? sy : 0), jd = j + (iy + 2 < ny ? sy : 0);
    const float nxd = X[jd], nxr = X[j + dx], nxu = X[j + dz1];
    float nvd = 0.f, nvr = 0.f, nvu = 0.f;
    if (dtv) {
      nvd = V[jd];
      nvr = V[j + dx];
      nvu = V[j + dz1];
    }
    const float n0 = qx[j], n1 = qy[j], n2 = qz[j], nzo = a.z[j], nTo = a.T[j];
    float b[3], qn[3];
    const float gr[3] = {hx ? xr - xc : 0.f, iy < ny - 1 ? xd - xc : 0.f, hz ? xu - xc : 0.f}, gv[3] = {vr - vc, vd - vc, vu - vc}, qo[3] = {q0, q1, q2};
    dual_update<KIND>(a, gr, gv, qo, b, qn);
    *bx = b[0];
    if (lane == 31) *bz = b[2];
    const float below = __shfl_up_sync(0xffffffffu, b[2], 1);
    __syncthreads();  // the other buffer is rewritten only after the next row's barrier
    if (owner && iy >= y0) {
      ox[i] = qn[0];
      oy[i] = qn[1];
      oz[i] = qn[2];
      // dz = A_n^T dq = sum_a [k_a >= 1] b_a(k - e_a) - [k_a < n_a - 1] b_a(k)
      float dz = 0.f;
      if (ix > 0) dz += bx[-zc];
      if (iy > 0) dz += by;
      if (iz > 0) dz += lane > 0 ? below : bz[-1];
      if (hx) dz -= b[0];
      if (iy < ny - 1) dz -= b[1];
      if (hz) dz -= b[2];
      const float zn = zo + dz;
      a.z[i] = zn;
      a.x_out[i] = prox_nonneg(xc - To * fmaf(dz, a.inv_p, zn));
    }
    by = b[1];
    bx += flip;
    bz += flipz;
    flip = -flip;
    flipz = -flipz;
    i = j;
    xc = xd; xd = nxd; xr = nxr; xu = nxu;
    vc = vd; vd = nvd; vr = nvr; vu = nvu;
    q0 = n0; q1 = n1; q2 = n2; zo = nzo; To = nTo;
  }
}

bool prior_launch_ok(const DevGeom& g) {
  March m = march_of(g);
  return march_shape(g, m, kPriorWarps);
}

cudaError_t launch_prior(const DevGeom& g, const PriorArgs& a, cudaStream_t s) {
  March m = march_of(g);
  if (!march_shape(g, m, kPriorWarps)) return cudaErrorInvalidValue;
  const int threads = m.cols * m.zw * 32;
  const size_t smem = 2 * (size_t)m.cols * m.zw * 33 * sizeof(float);
  const int N = g.nx * g.ny * g.nz;
  switch (a.kind) {
    case SPDHG_PRIOR_TV: k_prior<SPDHG_PRIOR_TV><<<march_grid(m), threads, smem, s>>>(m, a, N); break;
    case SPDHG_PRIOR_DTV: k_prior<SPDHG_PRIOR_DTV><<<march_grid(m), threads, smem, s>>>(m, a, N); break;
    case SPDHG_PRIOR_ATV: k_prior<SPDHG_PRIOR_ATV><<<march_grid(m), threads, smem, s>>>(m, a, N); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// TGV (Sec. 4.3): x = (u, w); block n-1: A = (grad, -I), f = alpha0 ||.||_{2,1};
// block n: A = (0, E), f = alpha1 ||.||_{2,1} with E the symmetrised gradient built from the
// backward difference d-_a = -D_a^T (components xx, yy, zz, xy, xz, yz; off-diagonals count
// twice in the norm).  Each block is one march: the dual step of a row, then the z, w and u steps, so
// that the dual change b is never stored (171 x 171 x 92: blocks 0 and 1 on average 134 -> 65 us against
// a dual and a primal pass; 102 bytes a voxel, 4.2 TB/s; bound by the latency of one row's loads).
// ---------------------------------------------------------------------------------------

constexpr int kTgvWarps = 24;  // at 80 registers

// block 0: q+ = proj_{alpha0}(q + sigma (grad u - w)); b = q+ - q; dzu = grad^T b, dzw = -b
__global__ void __launch_bounds__(kTgvWarps * 32, 1) k_tgv0(March m, TgvArgs a, int N) {
  extern __shared__ float sh[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c = w / m.zw, zi = w - c * m.zw, zc = m.zw * 32;
  const int iz = zi * 32 + lane, ix = blockIdx.x * (m.cols - 1) - 1 + c;  // column 0: the lower halo
  const int nx = m.nx, ny = m.ny, nz = m.nz, sx = m.sx, sy = m.sy;
  const bool live = ix >= 0 && ix < nx && iz < nz, owner = live && c >= 1;
  const bool hx = live && ix < nx - 1, hz = live && iz < nz - 1;
  const int y0 = blockIdx.y * m.ychunk, y1 = min(ny, y0 + m.ychunk);
  const int ys = y0 > 0 ? y0 - 1 : 0;
  float* sbx = sh;                                  // [2][cols][zc] b_x
  float* sbz = sh + 2 * m.cols * zc;                // [2][cols][zw] b_z of each warp's last lane
  const int off[3] = {m.kx * N, m.ky * N, m.kz * N};
  const float* U = a.u_in;
  const int dx = hx ? sx : 0, dz1 = hz ? 1 : 0;     // as in k_prior: the loads need no tests
  int i = ys * sy + (live ? ix * sx + iz : 0);
  float uc = U[i], ud = U[i + (ys < ny - 1 ? sy : 0)], ur = U[i + dx], uu = U[i + dz1], zu = a.zu[i], Tu = a.Tu[i], by = 0.f;
  float wv[3], qo[3], zw[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    wv[k] = a.w_in[off[k] + i];
    qo[k] = a.q_in[off[k] + i];
    zw[k] = a.zw[off[k] + i];
  }
  float* bx = sbx + c * zc + iz;
  float* bz = sbz + c * m.zw + zi;
  int flip = m.cols * zc, flipz = m.cols * m.zw;
#pragma unroll 2
  for (int iy = ys; iy < y1; ++iy) {
    const int j = i + (iy + 1 < y1 ? sy : 0);
    const float nud = U[j + (iy + 2 < ny ? sy : 0)], nur = U[j + dx], nuu = U[j + dz1], nzu = a.zu[j], nTu = a.Tu[j];
    float nw[3], nq[3], nzw[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      nw[k] = a.w_in[off[k] + j];
      nq[k] = a.q_in[off[k] + j];
      nzw[k] = a.zw[off[k] + j];
    }
    float b[3], qn[3], qa[3];
    const float gr[3] = {hx ? ur - uc : 0.f, iy < ny - 1 ? ud - uc : 0.f, hz ? uu - uc : 0.f};
#pragma unroll
    for (int k = 0; k < 3; ++k) qa[k] = fmaf(a.sigma, gr[k] - wv[k], qo[k]);
    const float nrm = sqrtf(qa[0] * qa[0] + qa[1] * qa[1] + qa[2] * qa[2]);
    const float sc = fmaxf(1.f, nrm / a.alpha);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      qn[k] = qa[k] / sc;
      b[k] = qn[k] - qo[k];
    }
    *bx = b[0];
    if (lane == 31) *bz = b[2];
    const float below = __shfl_up_sync(0xffffffffu, b[2], 1);
    __syncthreads();
    if (owner && iy >= y0) {
      float dz = 0.f;
      if (hx) dz -= b[0];
      if (iy < ny - 1) dz -= b[1];
      if (hz) dz -= b[2];
      if (ix > 0) dz += bx[-zc];
      if (iy > 0) dz += by;
      if (iz > 0) dz += lane > 0 ? below : bz[-1];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        // w part: dzw = -dq;  zw += dzw;  w = w - Tw (zw + dzw / p)
        const float dzw = -b[k], zwn = zw[k] + dzw;
        a.q_out[off[k] + i] = qn[k];
        a.zw[off[k] + i] = zwn;
        a.w_out[off[k] + i] = wv[k] - a.Tw * fmaf(dzw, a.inv_p, zwn);
      }
      const float zn = zu + dz;
      a.zu[i] = zn;
      a.u_out[i] = prox_nonneg(uc - Tu * fmaf(dz, a.inv_p, zn));
    }
    by = b[1];
    bx += flip;
    bz += flipz;
    flip = -flip;
    flipz = -flipz;
    i = j;
    uc = ud; ud = nud; ur = nur; uu = nuu; zu = nzu; Tu = nTu;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      wv[k] = nw[k];
      qo[k] = nq[k];
      zw[k] = nzw[k];
    }
  }
}

// block 1: q+ = proj_{alpha1}(q + sigma E w) (Frobenius ball, off-diagonals counted twice); b = q+ - q;
// dzw = E^T b; z and primal step of w; u takes its primal step with zbar_u = z_u.  E^T reads b of the
// upper neighbours, so the march runs down in y and the halo column is the upper one.
__global__ void __launch_bounds__(kTgvWarps * 32, 1) k_tgv1(March m, TgvArgs a, int N) {
  extern __shared__ float sh[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c = w / m.zw, zi = w - c * m.zw, zc = m.zw * 32;
  const int iz = zi * 32 + lane, ix = blockIdx.x * (m.cols - 1) + c;  // column cols - 1: the upper halo
  const int nx = m.nx, ny = m.ny, nz = m.nz, sx = m.sx, sy = m.sy;
  const bool live = ix < nx && iz < nz, owner = live && c < m.cols - 1;
  const bool hx = live && ix < nx - 1, hz = live && iz < nz - 1, lx = live && ix > 0, lz = live && iz > 0;
  const int y0 = blockIdx.y * m.ychunk, y1 = min(ny, y0 + m.ychunk);
  const int ys = y1 < ny ? y1 : ny - 1;             // first row computed (warm-up row for y1 < ny)
  const int plane = m.cols * zc, edge = m.cols * m.zw;
  float* sbx = sh;                                  // [2][3][cols][zc] b of xx, xy, xz
  float* sbz = sh + 6 * plane;                      // [2][3][cols][zw] b of zz, xz, yz of each warp's first lane
  // w components along x', y', z' and the dual's components: xx, yy, zz, xy, xz, yz in those directions
  const int wo[3] = {m.kx * N, m.ky * N, m.kz * N};
  auto pair = [](int p, int r) { return 2 + p + r; };  // xy: 3, xz: 4, yz: 5
  const int qf[6] = {m.kx * N, m.ky * N, m.kz * N, pair(m.kx, m.ky) * N, pair(m.kx, m.kz) * N, pair(m.ky, m.kz) * N};
  // as in k_prior the loads need no tests; a difference's absent term is masked
  const int dx = lx ? sx : 0, dz1 = lz ? 1 : 0;
  int i = ys * sy + (live ? ix * sx + iz : 0);
  float wc[3], wl[3], zw[3], qo[6], u = a.u_in[i], zu = a.zu[i], Tu = a.Tu[i], by1 = 0.f, by3 = 0.f, by5 = 0.f;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    wc[k] = a.w_in[wo[k] + i];
    wl[k] = a.w_in[wo[k] + i - (ys > 0 ? sy : 0)];
    zw[k] = a.zw[wo[k] + i];
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) qo[k] = a.q_in[qf[k] + i];
  float* bx = sbx + c * zc + iz;
  float* bz = sbz + c * m.zw + zi;
  int flip = 3 * plane, flipz = 3 * edge;
  for (int iy = ys; iy >= y0; --iy) {
    // w of the lower neighbours in x and z (lines the neighbours requested a row ago)
    float wx[3], wz[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      wx[k] = a.w_in[wo[k] + i - dx];
      wz[k] = a.w_in[wo[k] + i - dz1];
    }
    const int j = i - (iy - 1 >= y0 ? sy : 0), jl = j - (iy - 1 > 0 ? sy : 0);
    float nwl[3], nzw[3], nq[6];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      nwl[k] = a.w_in[wo[k] + jl];
      nzw[k] = a.zw[wo[k] + j];
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) nq[k] = a.q_in[qf[k] + j];
    const float nu = a.u_in[j], nzu = a.zu[j], nTu = a.Tu[j];
    const bool hy = iy < ny - 1, ly = iy > 0;
    // d-_a w_c = [k_a < n_a - 1] w_c(k) - [k_a > 0] w_c(k - e_a)
    auto ddx = [&](int k) { return (hx ? wc[k] : 0.f) - (lx ? wx[k] : 0.f); };
    auto ddy = [&](int k) { return (hy ? wc[k] : 0.f) - (ly ? wl[k] : 0.f); };
    auto ddz = [&](int k) { return (hz ? wc[k] : 0.f) - (lz ? wz[k] : 0.f); };
    float e[6], qa[6], b[6], qn[6];
    e[0] = ddx(0);
    e[1] = ddy(1);
    e[2] = ddz(2);
    e[3] = 0.5f * (ddx(1) + ddy(0));
    e[4] = 0.5f * (ddx(2) + ddz(0));
    e[5] = 0.5f * (ddy(2) + ddz(1));
#pragma unroll
    for (int k = 0; k < 6; ++k) qa[k] = fmaf(a.sigma, e[k], qo[k]);
    const float n2 = qa[0] * qa[0] + qa[1] * qa[1] + qa[2] * qa[2] +
                     2.f * (qa[3] * qa[3] + qa[4] * qa[4] + qa[5] * qa[5]);
    const float sc = fmaxf(1.f, sqrtf(n2) / a.alpha);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      qn[k] = qa[k] / sc;
      b[k] = qn[k] - qo[k];
    }
    bx[0] = b[0];
    bx[plane] = b[3];
    bx[2 * plane] = b[4];
    if (lane == 0) {
      bz[0] = b[2];
      bz[edge] = b[4];
      bz[2 * edge] = b[5];
    }
    float up2 = __shfl_down_sync(0xffffffffu, b[2], 1), up4 = __shfl_down_sync(0xffffffffu, b[4], 1),
          up5 = __shfl_down_sync(0xffffffffu, b[5], 1);
    __syncthreads();
    if (owner && iy < y1) {
      if (lane == 31 && hz) {
        up2 = bz[1];
        up4 = bz[edge + 1];
        up5 = bz[2 * edge + 1];
      }
      // (d-_a)^T = -D_a: b(k) - b(k + e_a) for k_a < n_a - 1, else 0; off-diagonals: 2 in the inner
      // product times the 1/2 of the definition
      float dzw[3];
      dzw[0] = (hx ? b[0] - bx[zc] : 0.f) + (hy ? b[3] - by3 : 0.f) + (hz ? b[4] - up4 : 0.f);
      dzw[1] = (hy ? b[1] - by1 : 0.f) + (hx ? b[3] - bx[plane + zc] : 0.f) + (hz ? b[5] - up5 : 0.f);
      dzw[2] = (hz ? b[2] - up2 : 0.f) + (hx ? b[4] - bx[2 * plane + zc] : 0.f) + (hy ? b[5] - by5 : 0.f);
#pragma unroll
      for (int k = 0; k < 6; ++k) a.q_out[qf[k] + i] = qn[k];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float zwn = zw[k] + dzw[k];
        a.zw[wo[k] + i] = zwn;
        a.w_out[wo[k] + i] = wc[k] - a.Tw * fmaf(dzw[k], a.inv_p, zwn);
      }
      a.u_out[i] = prox_nonneg(u - Tu * zu);
    }
    by1 = b[1];
    by3 = b[3];
    by5 = b[5];
    bx += flip;
    bz += flipz;
    flip = -flip;
    flipz = -flipz;
    i = j;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      wc[k] = wl[k];
      wl[k] = nwl[k];
      zw[k] = nzw[k];
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) qo[k] = nq[k];
    u = nu; zu = nzu; Tu = nTu;
  }
}

__device__ __forceinline__ float4 step4(const float4 w, const float4 z, float T) {
  return make_float4(w.x - T * z.x, w.y - T * z.y, w.z - T * z.z, w.w - T * z.w);
}

// w -= Tw zw on 3N values (16-byte aligned buffers): 16 bytes and four independent pieces a thread
// (171 x 171 x 92: 20 -> 11 us).  As part of the backprojection's epilogue it cost 35 us.
__global__ void __launch_bounds__(256) k_w_step(int n4, int n, float* __restrict__ w, const float* __restrict__ zw, float Tw) {
  float4* w4 = reinterpret_cast<float4*>(w);
  const float4* z4 = reinterpret_cast<const float4*>(zw);
  const int i0 = blockIdx.x * 1024 + threadIdx.x;
  float4 a[4], b[4];
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (i0 + 256 * k < n4) {
      a[k] = w4[i0 + 256 * k];
      b[k] = z4[i0 + 256 * k];
    }
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (i0 + 256 * k < n4) w4[i0 + 256 * k] = step4(a[k], b[k], Tw);
  const int tail = 4 * n4 + threadIdx.x;
  if (blockIdx.x == 0 && tail < n) w[tail] = w[tail] - Tw * zw[tail];
}

cudaError_t launch_w_step(const DevGeom& g, float* w, const float* zw, float Tw, cudaStream_t s) {
  const int n = 3 * g.nx * g.ny * g.nz, n4 = n / 4;
  k_w_step<<<std::max(1, (n4 + 1023) / 1024), 256, 0, s>>>(n4, n, w, zw, Tw);
  return cudaGetLastError();
}

cudaError_t launch_tgv(const DevGeom& g0, const TgvArgs& a, cudaStream_t s) {
  DevGeom g = g0;
  g.tune[SPDHG_TUNE_PRIOR_COLS] = g.tune[SPDHG_TUNE_PRIOR_YCHUNK] = 0;  // knobs of the TV kernel
  March m = march_of(g);
  if (!march_shape(g, m, kTgvWarps)) return cudaErrorInvalidValue;
  const int threads = m.cols * m.zw * 32, N = g.nx * g.ny * g.nz;
  const size_t row = (size_t)m.cols * m.zw * 33 * sizeof(float);  // one value per voxel and one per warp
  if (a.block == 0) k_tgv0<<<march_grid(m), threads, 2 * row, s>>>(m, a, N);
  else k_tgv1<<<march_grid(m), threads, 6 * row, s>>>(m, a, N);
  return cudaGetLastError();
}

}  // namespace spdhg
