// FP64 reductions of the objective Psi (Problem "PET Reconstruction with Subsets"):
//   D(P x) = sum_j  y_j + r_j - b_j + b_j log(b_j / (y_j + r_j))      (Eq. EQU:LOCALDISTANCE,
//            with 0 log 0 = 0 and +inf where y_j + r_j <= 0 < b_j)
//   alpha R(x) for TV / dTV / aTV, or the TGV value at the current (u, w).
// The per-term arithmetic and the sums run in double precision.  Reductions are deterministic:
// a fixed grid of blocks accumulates grid-strided terms, each block reduces in a fixed tree, and
// one block sums the partials in order.
#include "internal.cuh"

namespace spdhg {

__device__ __forceinline__ double block_sum(double v, double* sh) {
  const int t = threadIdx.x;
  sh[t] = v;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (t < s) sh[t] += sh[t + s];
    __syncthreads();
  }
  return sh[0];
}

__global__ void k_finish_sum(const double* partial, int n, double* out) {
  __shared__ double sh[256];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc += partial[i];
  const double s = block_sum(acc, sh);
  if (threadIdx.x == 0) *out = s;
}

__global__ void k_finish_max(const double* partial, int n, double* out) {
  __shared__ double sh[256];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc = fmax(acc, partial[i]);
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] = fmax(sh[threadIdx.x], sh[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

// The FP64 value of a positive normal float (conversions run at the FP64 rate, these at the integer's).
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x);
  return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
}

// log(1 + j / 256).  Computed by every block, the table cost a block as much as its share of a small
// sinogram.
__device__ const double kLogFrac[256] = {
    0.0, 0.003898640415657323, 0.007782140442054949, 0.011650617219975274, 0.015504186535965254, 0.019342962843130935,
    0.02316705928153438, 0.026976587698202076, 0.030771658666753687, 0.034552381506659735, 0.0383188643021366, 0.04207121392068706,
    0.0458095360312942, 0.04953393512227663, 0.053244514518812285, 0.056941376400138424, 0.06062462181643484, 0.06429435070539725,
    0.06795066190850775, 0.07159365318700882, 0.07522342123758753, 0.07884006170777602, 0.08244366921107459, 0.08603433734180316,
    0.08961215868968714, 0.0931772248541833, 0.09672962645855111, 0.10026945316367515, 0.10379679368164356, 0.10731173578908805,
    0.11081436634029011, 0.11430477128005863, 0.11778303565638346, 0.12124924363286968, 0.12470347850095724, 0.12814582269193003,
    0.13157635778871926, 0.13499516453750482, 0.13840232285911913, 0.14179791186025734, 0.1451820098444979, 0.14855469432313714,
    0.15191604202584197, 0.15526612891112396, 0.15860503017663857, 0.16193282026931324, 0.16524957289530717, 0.16855536102980667,
    0.17185025692665923, 0.17513433212784915, 0.1784076574728183, 0.18167030310763468, 0.184922338494012, 0.188163832418183,
    0.19139485299962947, 0.19461546769967167, 0.19782574332991987, 0.20102574606059073, 0.2042155414286909, 0.2073951943460706,
    0.21056476910734964, 0.21372432939771813, 0.21687393830061436, 0.2200136583052821, 0.22314355131420976, 0.22626367865045338,
    0.22937410106484582, 0.23247487874309405, 0.2355660713127669, 0.238647737850175, 0.24171993688714516, 0.24478272641769092,
    0.24783616390458127, 0.25088030628580943, 0.25391520998096345, 0.2569409308975004, 0.25995752443692605, 0.26296504550088134,
    0.26596354849713794, 0.26895308734550394, 0.27193371548364176, 0.2749054858727992, 0.2778684510034563, 0.2808226629008878,
    0.2837681731306446, 0.2867050328039543, 0.28963329258304266, 0.29255300268637746, 0.2954642128938359, 0.2983669725517973,
    0.3012613305781618, 0.3041473354672967, 0.3070250352949119, 0.3098944777228647, 0.3127557100038969, 0.31560877898630335,
    0.3184537311185346, 0.3212906124537343, 0.324119468654212, 0.32694034499585334, 0.329753286372468, 0.3325583373000766,
    0.3353555419211378, 0.3381449440087164, 0.3409265869705932, 0.34370051385331846, 0.34646676734620857, 0.34922538978528833,
    0.3519764231571782, 0.35471990910292905, 0.3574558889218038, 0.3601844035750078, 0.3629054936893685, 0.3656191995609647,
    0.3683255611587076, 0.3710246181278727, 0.37371640979358406, 0.3764009751642531, 0.37907835293496944, 0.38174858149084834,
    0.38441169891033206, 0.3870677429684483, 0.3897167511400252, 0.3923587606028639, 0.394993808240869, 0.39762193064713847,
    0.4002431641270127, 0.40285754470108354, 0.4054651081081644, 0.4080658898082217, 0.4106599249852684, 0.4132472485502193,
    0.415827895143711, 0.4184018991388838, 0.42096929464412963, 0.4235301155058033, 0.4260843953109001, 0.4286321673896988,
    0.4311734648183713, 0.4337083204215594, 0.43623676677491807, 0.43875883620762796, 0.4412745608048752, 0.443783972410301,
    0.44628710262841953, 0.4487839828270067, 0.45127464413945856, 0.4537591174671205, 0.4562374334815876, 0.4587096226269767,
    0.46117571512217015, 0.4636357409630325, 0.46608972992459924, 0.46853771156323926, 0.470979715218791, 0.4734157700166721,
    0.4758459048699639, 0.47827014848147026, 0.4806885293457519, 0.4831010757511358, 0.4855078157817008, 0.487908777319239,
    0.4903039880451938, 0.49269347544257525, 0.4950772667978515, 0.49745538920281895, 0.4998278695564493, 0.5021947345667155,
    0.5045560107523953, 0.5069117244448543, 0.5092619017898079, 0.5116065687490621, 0.5139457511022343, 0.5162794744484545,
    0.5186077642080457, 0.5209306456241853, 0.5232481437645479, 0.5255602835229274, 0.5278670896208424, 0.5301685866091216,
    0.5324647988694718, 0.5347557506160276, 0.5370414658968836, 0.5393219685956089, 0.5415972824327444, 0.5438674309672835,
    0.5461324375981357, 0.5483923255655732, 0.5506471179526623, 0.5528968376866777, 0.5551415075405016, 0.5573811501340064,
    0.5596157879354227, 0.5618454432626918, 0.564070138284803, 0.5662898950231159, 0.5685047353526688, 0.5707146810034716,
    0.5729197535617855, 0.575119974471388, 0.5773153650348236, 0.5795059464146423, 0.5816917396346225, 0.5838727655809827,
    0.5860490450035782, 0.5882205985170861, 0.5903874466021763, 0.5925496096066716, 0.5947071077466928, 0.5968599611077938,
    0.5990081896460834, 0.6011518131893349, 0.6032908514380843, 0.6054253239667169, 0.6075552502245418, 0.6096806495368553,
    0.6118015411059929, 0.6139179440123705, 0.616029877215514, 0.6181373595550788, 0.6202404097518576, 0.6223390464087788,
    0.6244332880118935, 0.6265231529313527, 0.6286086594223741, 0.6306898256261987, 0.6327666695710378, 0.6348392091730102,
    0.6369074622370692, 0.6389714464579207, 0.6410311794209312, 0.6430866786030273, 0.6451379613735847, 0.6471850449953096,
    0.6492279466251099, 0.6512666833149581, 0.6533012720127457, 0.6553317295631277, 0.65735807270836, 0.6593803180891278,
    0.661398482245365, 0.6634125816170663, 0.6654226325450905, 0.6674286512719562, 0.6694306539426292, 0.6714286566053024,
    0.6734226752121667, 0.6754127256201767, 0.6773988235918061, 0.6793809847957973, 0.6813592248079031, 0.6833335591116206,
    0.6853040030989194, 0.6872705720709603, 0.689233281238809, 0.691192145724142,
};

constexpr int kLogSpan = 100;  // ratios and counts within 2^+-100 take the table
struct LogTable {
  double frac[256];              // kLogFrac
  double pow2[2 * kLogSpan + 1];  // k log 2
};

// b log(b / e) + e - b for b, e > 0 in FP64.  The FP64 rate bounds the data term, so log(b / e) goes
// without a division and with about a third of the FP64 operations: c = 2^k (1 + j / 256) is the ratio
// rounded to eight bits (from FP32), r = (b - c e) / (c e) with |r| < 2^-8.9 by one Newton step from an
// FP32 reciprocal and one residual step, and log(b / e) = k log 2 + log(1 + j / 256) + log1p(r) with
// log1p by its series to r^6 (the table-driven scheme of Tang, ACM TOMS 16, 1990).  Its error is at most
// 2.7e-16 of max(1, |log|) (log(b / e): 1.9e-16), and 1e-22 where b and e agree to 1e-6 (1.1e-16).
// Values outside the span, and NaN, take log(b / e).  8.3 M bins: 753 -> 397 us.
__device__ __forceinline__ double kl_term(float bf, float ef, double e, const LogTable& tab) {
  const float y = bf * __frcp_rn(ef);
  if (!(y > 0x1p-99f && y < 0x1p99f && bf > 0x1p-99f && bf < 0x1p99f)) return e - (double)bf + (double)bf * log((double)bf / e);
  const unsigned bits = __float_as_uint(y) + 0x4000u;  // rounded to eight mantissa bits
  const int k = (int)(bits >> 23) - 127, j = (int)(bits >> 15) & 0xFF;
  const double b = widen(bf), c = __hiloint2double(((k + 1023) << 20) | (j << 12), 0);
  const double ce = c * e, num = fma(-c, e, b);
  const double x0 = widen(__frcp_rn(__uint_as_float(bits & 0xFFFF8000u) * ef));
  const double x1 = fma(x0, fma(-ce, x0, 1.0), x0);
  const double r0 = num * x1, r = fma(fma(-ce, r0, num), x1, r0);
  double p = fma(r, -1.0 / 6.0, 1.0 / 5.0);
  p = fma(r, p, -1.0 / 4.0);
  p = fma(r, p, 1.0 / 3.0);
  p = fma(r, p, -1.0 / 2.0);
  return fma(b, (tab.pow2[k + kLogSpan] + tab.frac[j]) + fma(r * r, p, r), e - b);
}

__global__ void k_data_term(const float* __restrict__ ax, const float* __restrict__ b,
                            const float* __restrict__ r, int64_t M, double* partial) {
  __shared__ double sh[256];
  __shared__ LogTable tab;
  tab.frac[threadIdx.x] = kLogFrac[threadIdx.x];
  if (threadIdx.x <= 2 * kLogSpan) tab.pow2[threadIdx.x] = ((int)threadIdx.x - kLogSpan) * 0.6931471805599453;
  __syncthreads();
  double acc = 0.0;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < M; j += (int64_t)gridDim.x * blockDim.x) {
    const float af = ax[j], rf = r[j], bj = b[j];
    const double e = (double)af + (double)rf;
    double phi;
    if (bj > 0.f) phi = (e > 0.0) ? kl_term(bj, af + rf, e, tab) : HUGE_VAL;
    else phi = e < 0.0 ? HUGE_VAL : e;
    acc += phi;
  }
  const double s = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// sum of squares (FP64) of v, for the power iteration of the operator norms
__global__ void k_sumsq(const float* __restrict__ v, int64_t n, double* partial) {
  __shared__ double sh[256];
  double acc = 0.0;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    const double a = v[j];
    acc += a * a;
  }
  const double s = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// v = y / sqrt(*ss)  (v = 0 if the norm is 0)
__global__ void k_normalize(const float* __restrict__ y, int64_t n, const double* __restrict__ ss, float* __restrict__ v) {
  const double q = *ss;
  const float inv = q > 0.0 ? (float)(1.0 / sqrt(q)) : 0.f;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
    v[j] = y[j] * inv;
}

cudaError_t launch_sumsq(const float* v, int64_t n, double* partial, int nblocks, double* out, cudaStream_t s) {
  k_sumsq<<<nblocks, 256, 0, s>>>(v, n, partial);
  k_finish_sum<<<1, 256, 0, s>>>(partial, nblocks, out);
  return cudaGetLastError();
}

cudaError_t launch_normalize(const float* y, int64_t n, const double* ss, float* v, cudaStream_t s) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 16) b = 152 * 16;
  k_normalize<<<(int)b, 256, 0, s>>>(y, n, ss, v);
  return cudaGetLastError();
}

cudaError_t launch_data_term(const float* ax, const float* b, const float* r, int64_t M,
                             double* partial, int nblocks, double* out, cudaStream_t s) {
  k_data_term<<<nblocks, 256, 0, s>>>(ax, b, r, M, partial);
  k_finish_sum<<<1, 256, 0, s>>>(partial, nblocks, out);
  return cudaGetLastError();
}

// forward differences (Neumann) of a float field at voxel (ix, iy, iz), in double
__device__ __forceinline__ void grad_d(const DevGeom& g, const float* u, int ix, int iy, int iz,
                                       int64_t j, double gr[3]) {
  const int sx = g.nz, sy = g.nx * g.nz;
  const double c = u[j];
  gr[0] = ix < g.nx - 1 ? (double)u[j + sx] - c : 0.0;
  gr[1] = iy < g.ny - 1 ? (double)u[j + sy] - c : 0.0;
  gr[2] = iz < g.nz - 1 ? (double)u[j + 1] - c : 0.0;
}

// d-_a w_c at j (backward difference, d- = -D^T)
__device__ __forceinline__ double dm_d(const DevGeom& g, const float* wc, int ax, int ix, int iy,
                                       int iz, int64_t j) {
  const int ja = ax == 0 ? ix : (ax == 1 ? iy : iz);
  const int na = ax == 0 ? g.nx : (ax == 1 ? g.ny : g.nz);
  const int st = ax == 0 ? g.nz : (ax == 1 ? g.nx * g.nz : 1);
  double r = 0.0;
  if (ja < na - 1) r += wc[j];
  if (ja > 0) r -= wc[j - st];
  return r;
}

__global__ void k_prior_term(DevGeom g, int kind, const float* __restrict__ x, const float* __restrict__ w,
                             const float* __restrict__ side, double gamma_d, double eta2, double* partial) {
  __shared__ double sh[256];
  const int64_t N = (int64_t)g.nx * g.ny * g.nz;
  double acc = 0.0;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < N; j += (int64_t)gridDim.x * blockDim.x) {
    const int iz = (int)(j % g.nz);
    const int64_t t = j / g.nz;
    const int ix = (int)(t % g.nx);
    const int iy = (int)(t / g.nx);
    double gr[3];
    grad_d(g, x, ix, iy, iz, j, gr);
    if (kind == SPDHG_PRIOR_ATV) {
      acc += fabs(gr[0]) + fabs(gr[1]) + fabs(gr[2]);
    } else if (kind == SPDHG_PRIOR_TGV) {
      const double a0 = gr[0] - w[j], a1 = gr[1] - w[N + j], a2 = gr[2] - w[2 * N + j];
      acc += sqrt(a0 * a0 + a1 * a1 + a2 * a2);  // weighted by alpha0 on the host
    } else {
      if (kind == SPDHG_PRIOR_DTV) {
        double gv[3];
        grad_d(g, side, ix, iy, iz, j, gv);
        const double inv = 1.0 / sqrt(gv[0] * gv[0] + gv[1] * gv[1] + gv[2] * gv[2] + eta2);
        const double xi0 = gv[0] * inv, xi1 = gv[1] * inv, xi2 = gv[2] * inv;
        const double d = gamma_d * (xi0 * gr[0] + xi1 * gr[1] + xi2 * gr[2]);
        gr[0] -= d * xi0;
        gr[1] -= d * xi1;
        gr[2] -= d * xi2;
      }
      acc += sqrt(gr[0] * gr[0] + gr[1] * gr[1] + gr[2] * gr[2]);
    }
  }
  const double s = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// sum_k |E w|_F (TGV second term; weighted by alpha1 on the host)
__global__ void k_tgv_sym_term(DevGeom g, const float* __restrict__ w, double* partial) {
  __shared__ double sh[256];
  const int64_t N = (int64_t)g.nx * g.ny * g.nz;
  double acc = 0.0;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < N; j += (int64_t)gridDim.x * blockDim.x) {
    const int iz = (int)(j % g.nz);
    const int64_t t = j / g.nz;
    const int ix = (int)(t % g.nx);
    const int iy = (int)(t / g.nx);
    const float* w0 = w;
    const float* w1 = w + N;
    const float* w2 = w + 2 * N;
    const double e0 = dm_d(g, w0, 0, ix, iy, iz, j);
    const double e1 = dm_d(g, w1, 1, ix, iy, iz, j);
    const double e2 = dm_d(g, w2, 2, ix, iy, iz, j);
    const double e3 = 0.5 * (dm_d(g, w1, 0, ix, iy, iz, j) + dm_d(g, w0, 1, ix, iy, iz, j));
    const double e4 = 0.5 * (dm_d(g, w2, 0, ix, iy, iz, j) + dm_d(g, w0, 2, ix, iy, iz, j));
    const double e5 = 0.5 * (dm_d(g, w2, 1, ix, iy, iz, j) + dm_d(g, w1, 2, ix, iy, iz, j));
    acc += sqrt(e0 * e0 + e1 * e1 + e2 * e2 + 2.0 * (e3 * e3 + e4 * e4 + e5 * e5));
  }
  const double s = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

cudaError_t launch_prior_term(const DevGeom& g, int kind, const float* x, const float* w,
                              const float* side, float gamma_d, float eta2, double* partial,
                              int nblocks, double* out, cudaStream_t s) {
  k_prior_term<<<nblocks, 256, 0, s>>>(g, kind, x, w, side, (double)gamma_d, (double)eta2, partial);
  k_finish_sum<<<1, 256, 0, s>>>(partial, nblocks, out);
  if (kind == SPDHG_PRIOR_TGV) {
    k_tgv_sym_term<<<nblocks, 256, 0, s>>>(g, w, partial);
    k_finish_sum<<<1, 256, 0, s>>>(partial, nblocks, out + 1);
  }
  return cudaGetLastError();
}

__global__ void k_side_max_grad(DevGeom g, const float* __restrict__ v, double* partial) {
  __shared__ double sh[256];
  const int64_t N = (int64_t)g.nx * g.ny * g.nz;
  double acc = 0.0;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < N; j += (int64_t)gridDim.x * blockDim.x) {
    const int iz = (int)(j % g.nz);
    const int64_t t = j / g.nz;
    const int ix = (int)(t % g.nx);
    const int iy = (int)(t / g.nx);
    double gv[3];
    grad_d(g, v, ix, iy, iz, j, gv);
    acc = fmax(acc, sqrt(gv[0] * gv[0] + gv[1] * gv[1] + gv[2] * gv[2]));
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sh[threadIdx.x] = fmax(sh[threadIdx.x], sh[threadIdx.x + s]);
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

cudaError_t launch_side_max_grad(const DevGeom& g, const float* side, double* partial, int nblocks,
                                 double* out, cudaStream_t s) {
  k_side_max_grad<<<nblocks, 256, 0, s>>>(g, side, partial);
  k_finish_max<<<1, 256, 0, s>>>(partial, nblocks, out);
  return cudaGetLastError();
}

// PSNR terms (Sec. 4): out[0] = sum_j (x_j - xs_j)^2, out[1] = max_j |xs_j|, both in FP64
__global__ void k_psnr_terms(const float* __restrict__ x, const float* __restrict__ xs, int64_t n,
                             double* partial_sq, double* partial_max) {
  __shared__ double sh[256];
  double acc = 0.0, mx = 0.0;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    const double d = (double)x[j] - (double)xs[j];
    acc += d * d;
    mx = fmax(mx, fabs((double)xs[j]));
  }
  const double s = block_sum(acc, sh);
  if (threadIdx.x == 0) partial_sq[blockIdx.x] = s;
  __syncthreads();
  sh[threadIdx.x] = mx;
  __syncthreads();
  for (int k = blockDim.x / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) sh[threadIdx.x] = fmax(sh[threadIdx.x], sh[threadIdx.x + k]);
    __syncthreads();
  }
  if (threadIdx.x == 0) partial_max[blockIdx.x] = sh[0];
}

cudaError_t launch_psnr_terms(const float* x, const float* xs, int64_t n, double* partial, int nblocks,
                              double* out, cudaStream_t s) {
  k_psnr_terms<<<nblocks, 256, 0, s>>>(x, xs, n, partial, partial + nblocks);
  k_finish_sum<<<1, 256, 0, s>>>(partial, nblocks, out);
  k_finish_max<<<1, 256, 0, s>>>(partial + nblocks, nblocks, out + 1);
  return cudaGetLastError();
}

}  // namespace spdhg
