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

// log(1 + j / 256) = kLogFrac[j] + kLogFracLo[j], the first a multiple of 2^-45 (rounded down).  Computed by every
// block, the tables cost a block as much as its share of a small sinogram.
__device__ const double kLogFrac[256] = {
    0.0, 0.0038986404156560184, 0.0077821404420319595, 0.011650617219970627, 0.015504186535963527, 0.019342962843126088,
    0.023167059281519187, 0.02697658769818645, 0.030771658666736812, 0.03455238150664286, 0.03831886430211284, 0.042071213920678474,
    0.045809536031271136, 0.04953393512226967, 0.05324451451880918, 0.056941376400118315, 0.060624621816430135, 0.06429435070538148,
    0.06795066190849752, 0.07159365318699429, 0.07522342123758108, 0.07884006170775137, 0.08244366921107371, 0.08603433734180044,
    0.08961215868967543, 0.09317722485417335, 0.09672962645854, 0.10026945316366209, 0.10379679368162442, 0.10731173578906805,
    0.11081436634026431, 0.11430477128004668, 0.11778303565637316, 0.12124924363286027, 0.12470347850094754, 0.12814582269191988,
    0.13157635778870258, 0.13499516453748583, 0.13840232285909337, 0.1417979118602375, 0.1451820098444898, 0.14855469432310997,
    0.15191604202581743, 0.15526612891110858, 0.15860503017663063, 0.16193282026929978, 0.16524957289530562, 0.16855536102980295,
    0.17185025692663203, 0.1751343321278398, 0.1784076574728033, 0.1816703031076088, 0.18492233849400463, 0.18816383241815515,
    0.1913948529996219, 0.19461546769966276, 0.19782574332990066, 0.20102574606056578, 0.20421554142868104, 0.20739519434604858,
    0.21056476910732158, 0.21372432939770647, 0.21687393830060842, 0.22001365830527675, 0.2231435513141946, 0.22626367865044017,
    0.22937410106482048, 0.23247487874309058, 0.23556607131274632, 0.23864773785015814, 0.24171993688713656, 0.24478272641766807,
    0.24783616390456586, 0.2508803062858078, 0.25391520998095984, 0.2569409308974855, 0.25995752443691345, 0.26296504550086297,
    0.2659635484971261, 0.26895308734549417, 0.271933715483641, 0.27490548587277885, 0.27786845100342816, 0.2808226629008743,
    0.28376817313062475, 0.2867050328039511, 0.2896332925830336, 0.2925530026863612, 0.29546421289381897, 0.2983669725517757,
    0.30126133057814286, 0.30414733546729167, 0.3070250352948847, 0.3098944777228496, 0.31275571000387004, 0.31560877898630224,
    0.3184537311185238, 0.3212906124537085, 0.32411946865420305, 0.32694034499584745, 0.3297532863724655, 0.3325583373000711,
    0.3353555419211318, 0.33814494400868966, 0.34092658697056777, 0.3437005138532925, 0.3464667673461861, 0.34922538978526063,
    0.3519764231571685, 0.3547199091029256, 0.35745588892177693, 0.3601844035750048, 0.3629054936893681, 0.365619199560939,
    0.3683255611586844, 0.3710246181278478, 0.373716409793559, 0.37640097516424476, 0.37907835293495395, 0.38174858149082525,
    0.384411698910327, 0.3870677429684406, 0.38971675114001414, 0.39235876060286046, 0.39499380824085506, 0.39762193064711937,
    0.400243164127005, 0.40285754470107804, 0.40546510810816017, 0.40806588980819924, 0.4106599249852536, 0.4132472485501921,
    0.4158278951437069, 0.41840189913887116, 0.4209692946441237, 0.4235301155057982, 0.4260843953108804, 0.42863216738967935,
    0.4311734648183574, 0.4337083204215446, 0.436236766774897, 0.4387588362076258, 0.4412745608048567, 0.443783972410273,
    0.44628710262841764, 0.4487839828269955, 0.4512746441394313, 0.45375911746711495, 0.45623743348156154, 0.45870962262696935,
    0.4611757151221525, 0.46363574096301363, 0.4660897299245903, 0.468537711563215, 0.4709797152187889, 0.4734157700166577,
    0.47584590486994216, 0.47827014848144245, 0.48068852934574124, 0.48310107575110806, 0.48550781578168767, 0.4879087773192339,
    0.49030398804518427, 0.4926934754425645, 0.4950772667978356, 0.4974553892027984, 0.4998278695564409, 0.5021947345667002,
    0.504556010752367, 0.5069117244448478, 0.5092619017897846, 0.5116065687490448, 0.5139457511022272, 0.5162794744484529,
    0.518607764208042, 0.520930645624162, 0.5232481437645333, 0.525560283522907, 0.5278670896208268, 0.5301685866091077,
    0.5324647988694551, 0.5347557506160001, 0.5370414658968627, 0.5393219685956012, 0.5415972824327184, 0.543867430967282,
    0.5461324375981178, 0.5483923255655725, 0.55064711795265, 0.5528968376866601, 0.5551415075404975, 0.557381150134006,
    0.5596157879353996, 0.5618454432626834, 0.5640701382847908, 0.5662898950230897, 0.5685047353526613, 0.5707146810034658,
    0.572919753561763, 0.5751199744713631, 0.5773153650348206, 0.5795059464146277, 0.5816917396346071, 0.5838727655809635,
    0.5860490450035627, 0.5882205985170685, 0.5903874466021648, 0.5925496096066638, 0.5947071077466717, 0.596859961107782,
    0.5990081896460708, 0.6011518131893183, 0.6032908514380608, 0.6054253239666991, 0.6075552502245216, 0.6096806495368412,
    0.61180154110599, 0.6139179440123428, 0.6160298772155102, 0.6181373595550781, 0.6202404097518297, 0.6223390464087686,
    0.6244332880118861, 0.6265231529313269, 0.6286086594223548, 0.6306898256261775, 0.6327666695710263, 0.6348392091730091,
    0.6369074622370476, 0.6389714464579015, 0.6410311794209065, 0.6430866786030265, 0.6451379613735639, 0.6471850449952967,
    0.6492279466251034, 0.6512666833149581, 0.653301272012726, 0.6553317295631018, 0.6573580727083481, 0.65938031808912,
    0.661398482245346, 0.6634125816170524, 0.6654226325450736, 0.6674286512719334, 0.6694306539426123, 0.6714286566052863,
    0.6734226752121515, 0.6754127256201627, 0.6773988235918011, 0.6793809847957846, 0.6813592248078919, 0.6833335591116168,
    0.6853040030989064, 0.6872705720709575, 0.6892332812387849, 0.6911921457241306,
};
__device__ const float kLogFracLo[256] = {
    0.f, 1.3046375e-15f, 2.298941e-14f, 4.647088e-15f, 1.7274568e-15f, 4.84659e-15f, 1.519153e-14f, 1.5626333e-14f, 1.6876434e-14f, 1.6873731e-14f,
    2.3756415e-14f, 8.580279e-15f, 2.3066786e-14f, 6.9631097e-15f, 3.10002e-15f, 2.0109399e-14f, 4.7072124e-15f, 1.5781652e-14f, 1.022665e-14f, 1.4529663e-14f,
    6.447241e-15f, 2.4650189e-14f, 8.8000106e-16f, 2.715811e-15f, 1.1707426e-14f, 9.943666e-15f, 1.1115548e-14f, 1.30570425e-14f, 1.9142946e-14f, 1.999834e-14f,
    2.5799992e-14f, 1.19538855e-14f, 1.0296122e-14f, 9.414425e-15f, 9.695922e-15f, 1.01631045e-14f, 1.6692224e-14f, 1.8996159e-14f, 2.5761623e-14f, 1.9858823e-14f,
    8.085115e-15f, 2.7172554e-14f, 2.4542412e-14f, 1.5370799e-14f, 7.949352e-15f, 1.3471228e-14f, 1.5442173e-15f, 3.714398e-15f, 2.7194442e-14f, 9.3500376e-15f,
    1.5003334e-14f, 2.5890065e-14f, 7.3582514e-15f, 2.7834345e-14f, 7.565143e-15f, 8.900253e-15f, 1.9219679e-14f, 2.496157e-14f, 9.8559636e-15f, 2.2003548e-14f,
    2.8056638e-14f, 1.16693264e-14f, 5.9442443e-15f, 5.3467464e-15f, 1.5145452e-14f, 1.3219558e-14f, 2.5350768e-14f, 3.4799447e-15f, 2.0592243e-14f, 1.687291e-14f,
    8.613129e-15f, 2.2843608e-14f, 1.5391912e-14f, 1.5973664e-15f, 3.6001767e-15f, 1.4938808e-14f, 1.26217294e-14f, 1.8381237e-14f, 1.1829215e-14f, 9.79053e-15f,
    7.779394e-16f, 2.0394995e-14f, 2.8143237e-14f, 1.3464382e-14f, 1.9852665e-14f, 3.2159677e-15f, 9.068854e-15f, 1.624344e-14f, 1.6909254e-14f, 2.1592694e-14f,
    1.8920255e-14f, 5.048551e-15f, 2.7188145e-14f, 1.5072841e-14f, 2.6852879e-14f, 1.0940915e-15f, 1.0796278e-14f, 2.580141e-14f, 8.9293375e-15f, 5.866691e-15f,
    2.5001238e-15f, 5.485152e-15f, 6.01355e-15f, 2.6734759e-14f, 2.5441575e-14f, 2.5967174e-14f, 2.2492303e-14f, 2.7672712e-14f, 9.701498e-15f, 3.4159676e-15f,
    2.684226e-14f, 2.988419e-15f, 3.670857e-16f, 2.5688034e-14f, 2.3230568e-14f, 2.4847772e-14f, 2.5057366e-14f, 8.310565e-15f, 1.5503491e-14f, 2.3094804e-14f,
    5.035393e-15f, 7.689993e-15f, 1.10740605e-14f, 3.4156229e-15f, 1.3918185e-14f, 1.9118699e-14f, 7.704701e-15f, 5.473839e-15f, 4.2159663e-15f, 2.2503704e-14f,
    1.4775504e-14f, 2.7205377e-14f, 4.08295e-15f, 1.2659154e-14f, 5.943423e-15f, 5.0742983e-15f, 1.9681466e-14f, 1.9407498e-14f, 1.395272e-14f, 1.4780381e-14f,
    2.10924e-14f, 2.1468971e-15f, 1.8510302e-14f, 2.797238e-14f, 1.8691965e-15f, 1.1212696e-14f, 2.7282753e-14f, 5.559214e-15f, 2.6055951e-14f, 7.315986e-15f,
    1.7669963e-14f, 1.8881393e-14f, 8.923179e-15f, 2.4272353e-14f, 2.1156558e-15f, 1.4442616e-14f, 2.175419e-14f, 2.7832864e-14f, 1.0663207e-14f, 2.7767182e-14f,
    1.3139525e-14f, 5.0959675e-15f, 9.56901e-15f, 1.0778788e-14f, 1.5923393e-14f, 2.052748e-14f, 8.456255e-15f, 1.5331515e-14f, 2.8285798e-14f, 6.576409e-15f,
    2.3358914e-14f, 1.7324079e-14f, 7.139403e-15f, 1.5942482e-15f, 3.6329984e-15f, 2.3287067e-14f, 1.4512088e-14f, 2.041445e-14f, 1.5539184e-14f, 1.3911888e-14f,
    1.6763453e-14f, 2.7561527e-14f, 2.090819e-14f, 7.654724e-15f, 2.594173e-14f, 1.5558788e-15f, 1.7846737e-14f, 6.7120675e-16f, 1.2301081e-14f, 1.7645577e-14f,
    4.0785873e-15f, 3.3666963e-16f, 2.3119493e-14f, 8.4429195e-15f, 1.2165318e-14f, 2.618819e-14f, 7.3842266e-15f, 5.7601836e-15f, 2.2563555e-14f, 2.4846951e-14f,
    2.9886986e-15f, 1.4508797e-14f, 1.5407971e-14f, 1.92193e-14f, 1.551254e-14f, 1.7504976e-14f, 1.1574217e-14f, 7.791316e-15f, 2.110799e-14f, 1.1781109e-14f,
    1.25672135e-14f, 1.6518083e-14f, 2.3435647e-14f, 1.7764571e-14f, 2.0180846e-14f, 1.40719295e-14f, 2.849182e-15f, 2.7705533e-14f, 3.8508943e-15f, 6.4192884e-16f,
    2.7826706e-14f, 1.016021e-14f, 7.36707e-15f, 2.588321e-14f, 1.936142e-14f, 2.122464e-14f, 1.14884e-14f, 1.1450252e-15f, 2.1592555e-14f, 1.9228403e-14f,
    2.480821e-14f, 8.306125e-16f, 2.0762106e-14f, 1.2829096e-14f, 6.4052106e-15f, 3.0881478e-17f, 1.960788e-14f, 2.5815201e-14f, 1.1912256e-14f, 7.816143e-15f,
    1.897721e-14f, 1.3840732e-14f, 1.6837695e-14f, 2.2785815e-14f, 1.7014649e-14f, 1.604518e-14f, 1.5231121e-14f, 1.3985026e-14f, 4.993906e-15f, 1.2779696e-14f,
    1.1163364e-14f, 3.9374945e-15f, 1.3038544e-14f, 2.725842e-15f, 2.4068633e-14f, 1.1390008e-14f,
};

constexpr int kLogSpan = 100;  // ratios and counts within 2^+-100 take the table
struct LogTable {
  double frac[256], pow2[2 * kLogSpan + 1];     // kLogFrac; k log 2, rounded down to a multiple of 2^-45
  float frac_lo[256], pow2_lo[2 * kLogSpan + 1];  // what is missing from them
};

// Entry t of the table.  k log 2 in units of 2^-45 is k (kLog2 + kLog2Lo 2^-24); integers keep it exact.
__device__ __forceinline__ void log_entry(LogTable& tab, int t) {
  constexpr long long kLog2 = 24387948313145ll, kLog2Lo = 15676793ll;
  tab.frac[t] = kLogFrac[t];
  tab.frac_lo[t] = kLogFracLo[t];
  if (t > 2 * kLogSpan) return;
  const long long k = t - kLogSpan, low = k * kLog2Lo;
  tab.pow2[t] = (double)(k * kLog2 + (low >> 24)) * 0x1p-45;
  tab.pow2_lo[t] = (float)(int)(low & 0xFFFFFF) * 0x1p-69f;
}

// b log(b / e) + e - b for b, e > 0 in FP64.  The FP64 rate bounds the data term, so log(b / e) goes
// without a division and with about a third of the FP64 operations: c = 2^k (1 + j / 256) is the ratio
// rounded to eight bits (from FP32), r = (b - c e) / (c e) with |r| < 2^-8.9 by one Newton step from an
// FP32 reciprocal and one residual step, and log(b / e) = k log 2 + log(1 + j / 256) + log1p(r) with
// log1p by its series to r^6 (the table-driven scheme of Tang, ACM TOMS 16, 1990).  The tables' upper parts
// add without rounding and their lower parts (FP32, not negative) join log1p(r), so the logarithm is rounded
// once: the term's error is at most 2.2e-16 of the largest of b |log|, b and e (library logarithm and
// division: 2.5e-16; tables of one double each: 4.0e-16), and 1e-20 where b and e agree to 1e-4 (1.1e-16).
// Values outside the span, and NaN, take log(b / e).  8.3 M bins: 753 -> 411 us.
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
  const unsigned lo = __float_as_uint(tab.pow2_lo[k + kLogSpan] + tab.frac_lo[j]);
  const double dlo = __hiloint2double(lo ? (int)((lo >> 3) + 0x38000000u) : 0, (int)(lo << 29));
  return fma(b, (tab.pow2[k + kLogSpan] + tab.frac[j]) + (fma(r * r, p, r) + dlo), e - b);
}

__global__ void k_data_term(const float* __restrict__ ax, const float* __restrict__ b,
                            const float* __restrict__ r, int64_t M, double* partial) {
  __shared__ double sh[256];
  __shared__ LogTable tab;
  log_entry(tab, threadIdx.x);
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
