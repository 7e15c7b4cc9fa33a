// 3x3x3 convolutions of the learned warm start (forward, data gradient) on the tensor cores (tcgen05,
// BF16 x BF16 -> FP32 in TMEM) without an im2col gather.
//
// A tile is 16 consecutive x positions x 8 consecutive z slices at one y: 128 voxels, row r = 8 m + j
// <-> voxel (y, x0 + m, z0 + j).  Its input halo (3 y x 18 x x 10 z voxels, zero outside the volume) is
// staged by 8-channel groups, voxel (dy, xx, zz) of a group at ((dy * 18 + xx) * 10 + zz) * 16 bytes
// or, for the kernels that take whole dy planes, at (xx * 10 + zz) * 16 of plane (dy, group).  For tap
// (dy, dx, dz) the operand of the MMA is the same halo read from a shifted start: the z-run at x0 + m is
// one core matrix (8 voxels x 16 bytes), consecutive runs are 160 bytes apart.  So a tap costs no copies.
//
// Bound: the MMAs' reads of the 128 x 16 operand from shared memory (about 70 cycles a step at 16 output
// channels, where the step's products take 4), then the halo copies; so blocks are persistent, three
// halos are in flight, and the accumulator of one tile is read while the next tile's MMAs run.  Measured
// on GB300, 128 x 128 x 64 voxels: 32 -> 16 channels 202 -> 146 us, 16 -> 16 104 -> 58 us, 8 -> 16 101 -> 45 us
// (from the gather); 64 -> 32 at 64 x 64 x 32 165 -> 70 us, 128 -> 128 at 16 x 16 x 8 88 -> 23 us (gather).
// Inference 1411 -> 803 us, gradients of a mini-batch of four 22.0 -> 16.8 ms.  Inference with 128 threads:
// 897 us; with 512: 884 us.
// Included by igemm.cu, whose error flag and mode table it shares.
#pragma once

namespace spdhg {
namespace ig {

constexpr int HX = 18, HZ = 10, HPL = HX * HZ, HROWS = 3 * HPL;  // halo voxels: x, z, per dy plane, in all
constexpr int CTHREADS = 384;    // three warps per TMEM lane quarter: thread t reads lane t % 128
constexpr int CPARTS = CTHREADS / 128;
constexpr long long CWAIT = 4000000000ll;  // ~2 s at 2 GHz: a lost completion ends the kernel

struct Tile {
  int y, x0, z0;
};
__device__ __forceinline__ Tile tile_of(int t, const GemmArgs& g) {
  const int tz = (g.nz + 7) >> 3, tx = (g.nx + 15) >> 4;
  Tile r;
  const int q = t / tz;
  r.z0 = (t - q * tz) * 8;
  r.y = q / tx;
  r.x0 = (q - r.y * tx) * 16;
  return r;
}

// Byte offset of tap (dy, dx, dz)'s first core matrix in a halo of whole groups.
__host__ __device__ constexpr uint32_t tap_off(int tap) {
  return (uint32_t)(((tap / 9) * HX + (tap / 3) % 3) * HZ + tap % 3) * 16u;
}

__device__ __forceinline__ void drain_failed(int code) {
  set_error(code);
  // give MMAs that may still be in flight a bounded chance to finish before TMEM is released
  const long long t0 = clock64();
  while (clock64() - t0 < 2000000ll) {
  }
}

// Epilogue of one tile: thread t holds row t % 128 (TMEM lane) and every CPARTS-th group of eight of the
// Nt columns from n_first on; tmem is the accumulator.
__device__ __forceinline__ void conv_epilogue(const GemmArgs& g, const Tile& T, uint32_t tmem, int n_first, int Nt, const float* bias) {
  const int row = threadIdx.x & 127, x = T.x0 + (row >> 3), z = T.z0 + (row & 7);
  const uint32_t trow = tmem + ((uint32_t)(row & ~31) << 16);
  const bool ok = x < g.nx && z < g.nz;
  const size_t orow = ((size_t)T.y * g.nx + x) * g.nz + z;
  for (int n0 = 8 * (threadIdx.x >> 7); n0 < Nt; n0 += 8 * CPARTS) {
    float v[8];
    umma::tmem_ld8(trow + n0, v);
    if (!ok) continue;
    const int n = n_first + n0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      v[j] += bias[n0 + j];
      if (g.relu) v[j] = fmaxf(v[j], 0.f);
    }
    if (g.mask && n + 8 > g.mask_from) {
      const uint4 mk = *reinterpret_cast<const uint4*>(g.mask + orow * g.mask_stride + g.mask_off + n);
      const __nv_bfloat162* m2 = reinterpret_cast<const __nv_bfloat162*>(&mk);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 f = __bfloat1622float2(m2[j]);
        if (n + 2 * j >= g.mask_from && !(f.x > 0.f)) v[2 * j] = 0.f;
        if (n + 2 * j + 1 >= g.mask_from && !(f.y > 0.f)) v[2 * j + 1] = 0.f;
      }
    }
    __align__(16) __nv_bfloat162 h[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    *reinterpret_cast<uint4*>(g.out + orow * g.out_stride + g.out_off + n) = *reinterpret_cast<uint4*>(h);
  }
}

__device__ __forceinline__ void load_bias(const GemmArgs& g, int n_first, int Nt, float* sbias) {
  if ((int)threadIdx.x < Nt) sbias[threadIdx.x] = g.bias ? g.bias[n_first + threadIdx.x] : 0.f;
}

// ------------------------------------------------------------------------------------------
// up to 32 input channels: persistent blocks, all weights of an N slice resident, three halo buffers
// ------------------------------------------------------------------------------------------

constexpr int kHaloBufs = 3;
constexpr int kZeroBytes = (15 * HZ + 8) * 16;  // 16 core matrices at the halo's distance

template <int C>
__global__ void __launch_bounds__(CTHREADS) k_conv3_halo(const __grid_constant__ GemmArgs g, int tiles, int Nt) {
  constexpr int CG = C / 8;                            // channel groups
  constexpr uint32_t GP = HROWS * 16;                  // bytes of a group's halo
  constexpr int PIECES = (HROWS * CG + CTHREADS - 1) / CTHREADS;
  constexpr int TAPS = C == 8 ? 28 : 27;               // weight blocks (8 channels: a zero block at the end)
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint64_t mbar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ float sbias[32];
  const int tid = threadIdx.x, warp = tid >> 5, n_first = blockIdx.y * Nt;
  const uint32_t sh = umma::smem_u32(smem), halo = CG * GP, sb = sh + kHaloBufs * halo;
  const uint32_t tapb = (uint32_t)(Nt >> 3) * CG * 128;  // bytes of a tap's weights (this slice)
  uint32_t ncols = 32;
  while ((int)ncols < 2 * Nt) ncols <<= 1;
  if (warp == 0) umma::tmem_alloc(&tmem_slot, ncols);
  if (tid == 0) {
    umma::mbar_init(&mbar[0], 1);
    umma::mbar_init(&mbar[1], 1);
    umma::fence_mbar_init();
  }
  load_bias(g, n_first, Nt, sbias);
  if (C == 8)  // the zero operand after the weights
    for (int i = tid; i < kZeroBytes / 16; i += CTHREADS)
      *reinterpret_cast<uint4*>(smem + kHaloBufs * halo + TAPS * tapb + 16 * i) = make_uint4(0u, 0u, 0u, 0u);
  // weights: [tap][n / 8][c / 8] core matrices; the slice's rows of a tap are contiguous
  for (int i = tid; i < TAPS * (int)(tapb >> 4); i += CTHREADS) {
    const int tap = i / (int)(tapb >> 4), k = i - tap * (int)(tapb >> 4);
    umma::cp16(sb + 16 * i, g.b + ((size_t)tap * g.N + n_first) * C + 8 * k, 16u);
  }
  // this thread's pieces of a halo: (dy, xx, zz, group), groups fastest (32 contiguous bytes per voxel pair)
  auto stage = [&](int t, int buf) {
    const Tile T = tile_of(t, g);
    const __nv_bfloat16* base = g.a + g.a_off;
#pragma unroll 4
    for (int k = 0; k < PIECES; ++k) {
      const int idx = tid + CTHREADS * k;
      if (idx >= HROWS * CG) break;
      const int cg = idx % CG, h = idx / CG, dy = h / HPL, rem = h - dy * HPL, xx = rem / HZ, zz = rem - xx * HZ;
      const int yy = T.y + dy - 1, xg = T.x0 + xx - 1, zg = T.z0 + zz - 1;
      const bool ok = (unsigned)yy < (unsigned)g.ny && (unsigned)xg < (unsigned)g.nx && (unsigned)zg < (unsigned)g.nz;
      const __nv_bfloat16* src = ok ? base + ((size_t)(yy * g.nx + xg) * g.nz + zg) * g.a_stride + cg * 8 : g.a;
      umma::cp16(sh + buf * halo + cg * GP + h * 16, src, ok ? 16u : 0u);
    }
  };
  const int n = blockIdx.x < tiles ? (tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  auto tile_at = [&](int it) { return blockIdx.x + it * gridDim.x; };
  if (n > 0) stage(tile_at(0), 0);
  umma::cp_commit();  // the weights too
  if (n > 1) stage(tile_at(1), 1);
  umma::cp_commit();
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tmem = tmem_slot;
  const uint32_t idesc = umma::idesc_bf16(128, Nt, false, false);
  bool failed = false;
  for (int it = 0; it < n; ++it) {
    umma::cp_wait<1>();  // tile `it` has landed (this thread's copies)
    umma::fence_proxy_async_smem();
    umma::fence_before_sync();
    if (__syncthreads_or(failed)) break;
    if (tid == 0) {
      umma::fence_after_sync();
      const uint32_t a0 = sh + (it % kHaloBufs) * halo, d = tmem + (it & 1) * Nt;
      if (C == 8) {
        // a K step holds two taps; the distance of their starts is the leading-dimension offset.  The
        // last step pairs tap 26 with zeros (a voxel under a zero weight would spread infinities as NaN)
#pragma unroll
        for (int i = 0; i < 14; ++i) {
          const uint32_t t0 = a0 + tap_off(2 * i), t1 = i < 13 ? a0 + tap_off(2 * i + 1) : sb + TAPS * tapb;
          umma::mma_bf16(d, umma::smem_desc(t0, t1 - t0, HZ * 16), umma::smem_desc(sb + 2 * i * tapb, tapb, 128), idesc,
                         i > 0 ? 1u : 0u);
        }
      } else {
#pragma unroll
        for (int tap = 0; tap < 27; ++tap)
#pragma unroll
          for (int c16 = 0; c16 < C / 16; ++c16)
            umma::mma_bf16(d, umma::smem_desc(a0 + 2 * c16 * GP + tap_off(tap), GP, HZ * 16),
                           umma::smem_desc(sb + tap * tapb + 2 * c16 * 128, 128, CG * 128), idesc, tap + c16 > 0 ? 1u : 0u);
      }
      umma::commit(&mbar[it & 1]);
    }
    if (it > 0) {
      // the previous tile's accumulator, while this tile's MMAs run; its halo buffer is free then
      failed = __any_sync(0xffffffffu, !umma::mbar_wait(&mbar[(it - 1) & 1], ((it - 1) >> 1) & 1, CWAIT));
      umma::fence_after_sync();
      if (!failed) conv_epilogue(g, tile_of(tile_at(it - 1), g), tmem + ((it - 1) & 1) * Nt, n_first, Nt, sbias);
    }
    if (!failed && it + 2 < n) stage(tile_at(it + 2), (it + 2) % kHaloBufs);
    umma::cp_commit();
  }
  umma::cp_wait<0>();
  if (n > 0 && !failed) {
    failed = __any_sync(0xffffffffu, !umma::mbar_wait(&mbar[(n - 1) & 1], ((n - 1) >> 1) & 1, CWAIT));
    umma::fence_after_sync();
    if (!failed) conv_epilogue(g, tile_of(tile_at(n - 1), g), tmem + ((n - 1) & 1) * Nt, n_first, Nt, sbias);
  }
  if (__syncthreads_or(failed)) drain_failed(2);
  umma::fence_before_sync();
  __syncthreads();
  if (warp == 0) umma::tmem_dealloc(tmem, ncols);
}

// ------------------------------------------------------------------------------------------
// 64 and 128 input channels: one tile and N slice per block, the halo's dy planes resident, the
// weights streamed tap by tap (bulk copies, four in flight)
// ------------------------------------------------------------------------------------------

constexpr int kTapRing = 4;

template <int C>
__global__ void __launch_bounds__(CTHREADS) k_conv3_deep(const __grid_constant__ GemmArgs g, int Nt) {
  constexpr int CG = C / 8;
  constexpr uint32_t GP = HPL * 16, DY = CG * GP;      // bytes of a (dy, group) plane and of a dy plane
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint64_t full[kTapRing], empty[kTapRing], done;
  __shared__ uint32_t tmem_slot;
  __shared__ float sbias[32];
  const int tid = threadIdx.x, warp = tid >> 5, n_first = blockIdx.y * Nt;
  const uint32_t sh = umma::smem_u32(smem), sb = sh + 3 * DY;
  const uint32_t tapb = (uint32_t)Nt * C * 2;
  if (warp == 0) umma::tmem_alloc(&tmem_slot, 32);
  if (tid == 0) {
    for (int k = 0; k < kTapRing; ++k) {
      umma::mbar_init(&full[k], 1);
      umma::mbar_init(&empty[k], 1);
    }
    umma::mbar_init(&done, 1);
    umma::fence_mbar_init();
  }
  load_bias(g, n_first, Nt, sbias);
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  auto load_tap = [&](int tap) {
    const int s = tap % kTapRing;
    umma::bulk_load(sb + s * tapb, g.b + ((size_t)tap * g.N + n_first) * C, tapb, &full[s]);
  };
  if (tid == 0)
    for (int tap = 0; tap < kTapRing; ++tap) load_tap(tap);
  const Tile T = tile_of(blockIdx.x, g);
  for (int dy = 0; dy < 3; ++dy) {
    const int yy = T.y + dy - 1;
    for (int idx = tid; idx < HPL * CG; idx += CTHREADS) {
      const int cg = idx % CG, h = idx / CG, xx = h / HZ, zz = h - xx * HZ;
      const int xg = T.x0 + xx - 1, zg = T.z0 + zz - 1;
      const bool ok = (unsigned)yy < (unsigned)g.ny && (unsigned)xg < (unsigned)g.nx && (unsigned)zg < (unsigned)g.nz;
      const __nv_bfloat16* src = ok ? g.a + g.a_off + ((size_t)(yy * g.nx + xg) * g.nz + zg) * g.a_stride + cg * 8 : g.a;
      umma::cp16(sh + dy * DY + cg * GP + h * 16, src, ok ? 16u : 0u);
    }
    umma::cp_commit();
  }
  const uint32_t tmem = tmem_slot, idesc = umma::idesc_bf16(128, Nt, false, false);
  bool failed = false;
  for (int dy = 0; dy < 3; ++dy) {
    if (dy == 0) umma::cp_wait<2>();
    else if (dy == 1) umma::cp_wait<1>();
    else umma::cp_wait<0>();
    umma::fence_proxy_async_smem();
    __syncthreads();
    if (tid == 0) {
      for (int k = 0; k < 9 && !failed; ++k) {
        const int tap = 9 * dy + k, s = tap % kTapRing;
        failed = !umma::mbar_wait(&full[s], (tap / kTapRing) & 1, CWAIT);
        if (failed) break;
        umma::fence_after_sync();
        const uint32_t a0 = sh + dy * DY + (uint32_t)((k / 3) * HZ + k % 3) * 16, b0 = sb + s * tapb;
        for (int c16 = 0; c16 < C / 16; ++c16)
          umma::mma_bf16(tmem, umma::smem_desc(a0 + 2 * c16 * GP, GP, HZ * 16), umma::smem_desc(b0 + 2 * c16 * 128, 128, CG * 128),
                         idesc, tap + c16 > 0 ? 1u : 0u);
        umma::commit(&empty[s]);
        if (tap > 0 && tap - 1 + kTapRing < 27) {  // the slot of the previous tap, once its MMAs are done
          failed = !umma::mbar_wait(&empty[(tap - 1) % kTapRing], ((tap - 1) / kTapRing) & 1, CWAIT);
          if (!failed) load_tap(tap - 1 + kTapRing);
        }
      }
      if (dy == 2) umma::commit(&done);
    }
  }
  failed = !umma::mbar_wait(&done, 0, CWAIT) || failed;
  const bool any = __syncthreads_or(failed);
  if (any) drain_failed(3);
  umma::fence_after_sync();
  if (!any) conv_epilogue(g, T, tmem, n_first, Nt, sbias);
  umma::fence_before_sync();
  __syncthreads();
  if (warp == 0) umma::tmem_dealloc(tmem, 32);
}

cudaError_t launch_conv3(const GemmArgs& g, cudaStream_t s) {
  const int C = g.a_c, Nt = std::min(32, g.N);
  if ((C != 8 && C != 16 && C != 32 && C != 64 && C != 128) || (g.N != 16 && g.N % 32)) return cudaErrorNotSupported;
  const int tiles = ((g.nz + 7) / 8) * ((g.nx + 15) / 16) * g.ny;
  auto go = [&](auto kern, dim3 grid, size_t smem, auto... args) -> cudaError_t {
    cudaError_t e = allow_dynamic_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<grid, CTHREADS, smem, s>>>(g, args...);
    return cudaGetLastError();
  };
  if (C <= 32) {
    const size_t smem = (size_t)kHaloBufs * (C / 8) * HROWS * 16 +
                        (C == 8 ? (size_t)28 * Nt * 16 + kZeroBytes : (size_t)27 * Nt * C * 2);
    const int per_sm = std::max(1, std::min(4, (int)(220 * 1024 / (smem + 1024)))), slices = g.N / Nt;
    const dim3 grid(std::min(tiles, std::max(1, 152 * per_sm / slices)), slices);
    if (C == 8) return go(k_conv3_halo<8>, grid, smem, tiles, Nt);
    if (C == 16) return go(k_conv3_halo<16>, grid, smem, tiles, Nt);
    return go(k_conv3_halo<32>, grid, smem, tiles, Nt);
  }
  const size_t smem = (size_t)3 * (C / 8) * HPL * 16 + (size_t)kTapRing * Nt * C * 2;
  const dim3 grid(tiles, g.N / Nt);
  if (C == 64) return go(k_conv3_deep<64>, grid, smem, Nt);
  return go(k_conv3_deep<128>, grid, smem, Nt);
}

}  // namespace ig
}  // namespace spdhg
