// On-GPU TaylorF2 templates (the bank waveforms the search filters, Sec. II;
// non-spinning stationary-phase approximant with the 3.5PN phase of Buonanno,
// Iyer, Ochsner, Pan & Sathyaprakash 2009, Eq. 3.18, and Newtonian amplitude):
//   h~(f) = f^{-7/6} exp(-i Psi(f)),  f_low <= f <= min(f_ISCO, Nyquist), k < N/2,
//   Psi(f) = -pi/4 + 3 / (128 eta v^5) [1 + sum_k psi_k v^k (+ log terms)],  v = (pi M f)^{1/3},
// zero elsewhere.  Psi reaches ~1e5 rad at the lower frequencies, so it is
// evaluated in FP64 only at anchors K bins apart (K = 2^j with K df <= 0.25 Hz
// and K <= k_low / 4); each anchor keeps Psi mod 2 pi and the FP64 difference
// to the next anchor, both as FP32.  Between anchors the phase is the cubic
// Lagrange interpolant through the four nearest anchors, evaluated in FP32
// (differences of at most 3 K bins' worth of phase, so FP32 rounding stays
// near 1e-5 rad; the interpolation error is below 2e-4 rad, at the
// lightest templates' lowest frequencies), reduced to [-pi, pi] and turned into
// cos / sin.  The amplitude is exp2(-7/6 log2 f) (fast base-2 logarithm, ~1e-6 relative).
// The FP64 units bound the anchors (2 operations per clock and SM, and a whole warp's slots however few of its
// lanes are in use), so they have a kernel of their own that fills its warps and computes only the anchors that
// bins of the band interpolate between; as part of k_taylorf2 the 20 anchors of each 2,048 bins held up its CTAs
// (2.75 us per template at N = 2^20; now 0.65 us for the anchors and 0.9 us for the bins).
#include <cuda_runtime.h>

#include <cmath>
#include <string>
#include <vector>

#include "../../include/mf.h"
#include "mf_internal.h"

namespace mf {

namespace {

constexpr int kGenThreads = 256;
constexpr int kGenChunk = 2048;  // bins per CTA
constexpr double kMtsun = 4.925491025543576e-06;  // G M_sun / c^3, seconds
constexpr double kEulerGamma = 0.5772156649015329;
constexpr double kPi = 3.141592653589793;

struct TF2 {
  double p[8];        // psi_0 .. psi_7
  double log5, log6;  // coefficients of ln(v / v_lso) at v^5 and of ln v at v^6
  double piM;         // pi M (seconds)
  double pre;         // 3 / (128 eta)
  int64_t k_lo, k_hi; // band, inclusive
  int K_log2;         // anchors every 2^K_log2 bins
};

__device__ __forceinline__ double tf2_phase(const TF2& t, double f) {
  const double v = cbrt(t.piM * f);
  const double lv = log(v);
  const double v2 = v * v;
  const double s = t.p[0] + v2 * (t.p[2] + v * (t.p[3] + v * (t.p[4] + v * (t.p[5] + t.log5 * (lv + 0.8958797346140275) +
                                                                               v * (t.p[6] + t.log6 * lv + v * t.p[7])))));
  // 0.8958797346140275 = -ln(v_lso), v_lso = 6^{-1/2}
  const double v5 = v2 * v2 * v;
  return -0.25 * kPi + t.pre / v5 * s;
}

// Anchor a of a template is at bin (a - 1) K.  psi holds a row's anchors a0 .. a0 + n_anchor - 1, which are those that
// some template's band needs; the ones below half the lower band edge, or two intervals past the template's own upper one,
// are not needed and not written.
__global__ void __launch_bounds__(kGenThreads) k_tf2_anchors(const TF2* __restrict__ tmpl, double df, int n_anchor,
                                                             int64_t a0, double* __restrict__ psi) {
  const int i = blockIdx.x * kGenThreads + threadIdx.x;
  if (i >= n_anchor) return;
  const TF2& m = tmpl[blockIdx.y];
  const int K = 1 << m.K_log2;
  const int64_t k = (a0 + i - 1) * K;
  if (k < m.k_lo / 2 || k > m.k_hi + 2 * K) return;
  const TF2 t = m;
  psi[(int64_t)blockIdx.y * n_anchor + i] = tf2_phase(t, (double)k * df);
}

__global__ void __launch_bounds__(kGenThreads) k_taylorf2(const TF2* __restrict__ tmpl, const double* __restrict__ psi,
                                                          int n_anchor, int64_t a0, double df, float df32,
                                                          float2* __restrict__ out,
                                                          int64_t ld, int64_t nb) {
  __shared__ float mod2pi[kGenChunk + 4];  // anchor phase mod 2 pi
  __shared__ float dnext[kGenChunk + 4];   // Psi(anchor + 1) - Psi(anchor)
  const TF2 t = tmpl[blockIdx.y];
  float2* row = out + (int64_t)blockIdx.y * ld;
  const int64_t k0 = (int64_t)blockIdx.x * kGenChunk;
  const int64_t k1 = k0 + kGenChunk < nb ? k0 + kGenChunk : nb;
  if (k1 <= t.k_lo || k0 > t.k_hi) {  // chunk outside the band
    for (int64_t k = k0 + threadIdx.x; k < k1; k += kGenThreads) row[k] = make_float2(0.f, 0.f);
    return;
  }
  const int K = 1 << t.K_log2;
  // the band's bins of the chunk lie in intervals i0 .. i1; interval i has the anchors i .. i + 3
  const int i0 = (int)((k0 < t.k_lo ? t.k_lo - k0 : 0) >> t.K_log2);
  const int i1 = (int)(((k1 - 1 < t.k_hi ? k1 - 1 : t.k_hi) - k0) >> t.K_log2);
  const double* pa = psi + (int64_t)blockIdx.y * n_anchor + ((k0 >> t.K_log2) - a0);
  for (int a = i0 + threadIdx.x; a < i1 + 3; a += kGenThreads) {
    const double p = pa[a];
    const double two_pi = 2.0 * kPi;
    mod2pi[a] = (float)(p - two_pi * floor(p / two_pi));
    dnext[a] = (float)(pa[a + 1] - p);
  }
  __syncthreads();
  const float two_pi_f = 6.283185307179586f, inv_two_pi = 0.15915494309189535f;
  for (int64_t k = k0 + threadIdx.x; k < k1; k += kGenThreads) {
    if (k < t.k_lo || k > t.k_hi) {
      row[k] = make_float2(0.f, 0.f);
      continue;
    }
    const int64_t off = k - k0;
    const int i = (int)(off >> t.K_log2) + 1;  // anchor index of the interval's left end
    const float x = (float)(off & (K - 1)) * (1.0f / (float)K);
    // cubic Lagrange weights at nodes -1, 0, 1, 2 (node 0 contributes its own value, i.e. 0 here)
    const float wm = -x * (x - 1.f) * (x - 2.f) * (1.f / 6.f);
    const float w1 = -(x + 1.f) * x * (x - 2.f) * 0.5f;
    const float w2 = (x + 1.f) * x * (x - 1.f) * (1.f / 6.f);
    const float d0 = dnext[i], d1 = dnext[i + 1];
    float ph = mod2pi[i] - wm * dnext[i - 1] + w1 * d0 + w2 * (d0 + d1);
    ph -= two_pi_f * rintf(ph * inv_two_pi);
    float s, c;
    __sincosf(ph, &s, &c);
    const float f = df32 > 0.f ? (float)(int)k * df32 : (float)((double)k * df);
    const float amp = exp2f(-1.1666666666666667f * __log2f(f));
    row[k] = make_float2(amp * c, -amp * s);
  }
}

}  // namespace

// first bin of the band
static int64_t first_bin(double f_low, double df) {
  int64_t lo = (int64_t)std::ceil(f_low / df);
  while (lo > 0 && (double)(lo - 1) * df >= f_low) --lo;
  while ((double)lo * df < f_low) ++lo;
  return lo;
}

// anchors every 2^j bins (the same for every template of a call)
static int anchor_log2(int64_t lo, double df) {
  int lg = 0;
  while (2.0 * (1 << lg) * df <= 0.25 && 2 * (1 << lg) <= std::max<int64_t>(lo / 4, 1) && (1 << lg) < 1024) ++lg;
  return lg;
}

// host: per-template coefficients; the band uses the same float64 arithmetic as the host-side generators
static TF2 make_tf2(double m1, double m2, double fs, int64_t n, double f_low) {
  TF2 t{};
  const double M = (m1 + m2) * kMtsun;
  const double eta = m1 * m2 / ((m1 + m2) * (m1 + m2));
  const double pi = kPi;
  t.p[0] = 1.0;
  t.p[1] = 0.0;
  t.p[2] = 20.0 / 9.0 * (743.0 / 336.0 + 11.0 / 4.0 * eta);
  t.p[3] = -16.0 * pi;
  t.p[4] = 10.0 * (3058673.0 / 1016064.0 + 5429.0 / 1008.0 * eta + 617.0 / 144.0 * eta * eta);
  t.p[5] = pi * (38645.0 / 756.0 - 65.0 / 9.0 * eta);
  t.p[6] = 11583231236531.0 / 4694215680.0 - 640.0 / 3.0 * pi * pi - 6848.0 / 21.0 * kEulerGamma +
           eta * (-15737765635.0 / 3048192.0 + 2255.0 / 12.0 * pi * pi) + 76055.0 / 1728.0 * eta * eta -
           127825.0 / 1296.0 * eta * eta * eta - 6848.0 / 21.0 * std::log(4.0);
  t.p[7] = pi * (77096675.0 / 254016.0 + 378515.0 / 1512.0 * eta - 74045.0 / 756.0 * eta * eta);
  t.log5 = 3.0 * t.p[5];
  t.log6 = -6848.0 / 21.0;
  t.piM = pi * M;
  t.pre = 3.0 / (128.0 * eta);
  const double df = fs / (double)n;
  const double f_isco = 1.0 / (std::pow(6.0, 1.5) * pi * M);
  const double fhi = std::min(f_isco, fs / 2.0);
  const int64_t lo = first_bin(f_low, df);
  int64_t hi = (int64_t)std::floor(fhi / df);
  while ((double)(hi + 1) * df <= fhi) ++hi;
  while (hi >= 0 && (double)hi * df > fhi) --hi;
  hi = std::min<int64_t>(hi, n / 2 - 1);
  t.k_lo = lo;
  t.k_hi = hi;
  t.K_log2 = anchor_log2(lo, df);
  return t;
}

// the anchors that a call's rows need: from a0 on, to the second past the highest band edge k_hi
struct Anchors {
  int64_t a0;
  int count;
};
static Anchors anchors_of(int64_t n, double fs, double f_low, int64_t k_hi) {
  const double df = fs / (double)n;
  const int64_t lo = first_bin(f_low, df);
  const int lg = anchor_log2(lo, df);
  const int64_t a0 = ((lo / 2) >> lg) + 1, a1 = ((k_hi + 2 * (int64_t(1) << lg)) >> lg) + 2;
  return Anchors{a0, (int)std::max<int64_t>(a1 - a0, 0)};  // (k_hi < n / 2)
}

int64_t taylorf2_k_hi(const double* m1, const double* m2, int64_t n_tmpl, double fs, int64_t n, double f_low) {
  int64_t light = 0;
  for (int64_t i = 1; i < n_tmpl; ++i)
    if (m1[i] + m2[i] < m1[light] + m2[light]) light = i;
  return make_tf2(m1[light], m2[light], fs, n, f_low).k_hi;
}

size_t taylorf2_table_bytes(int64_t n_tmpl) { return ((size_t)n_tmpl * sizeof(TF2) + 255) / 256 * 256; }

size_t taylorf2_work_bytes(int64_t n_rows, double fs, int64_t n, double f_low, int64_t k_hi) {
  return ((size_t)n_rows * anchors_of(n, fs, f_low, k_hi).count * sizeof(double) + 255) / 256 * 256;
}

int64_t taylorf2_block(int64_t n_tmpl, double fs, int64_t n, double f_low, int64_t k_hi) {
  const int64_t row = std::max(anchors_of(n, fs, f_low, k_hi).count, 1) * (int64_t)sizeof(double);
  return std::max<int64_t>(1, std::min<int64_t>(n_tmpl, (int64_t(64) << 20) / row));
}

cudaError_t taylorf2_tables(const double* m1, const double* m2, int64_t n_tmpl, double fs, int64_t n, double f_low,
                            void* dev, cudaStream_t st) {
  std::vector<TF2> h((size_t)n_tmpl);
  for (int64_t i = 0; i < n_tmpl; ++i) h[(size_t)i] = make_tf2(m1[i], m2[i], fs, n, f_low);
  // pageable source: the copy has taken the host table by the time the call returns
  return cudaMemcpyAsync(dev, h.data(), (size_t)n_tmpl * sizeof(TF2), cudaMemcpyHostToDevice, st);
}

bool taylorf2_valid(const double* m1, const double* m2, int64_t n_tmpl, double fs, int64_t n, double f_low) {
  if (n_tmpl < 1 || n < 16 || !(fs > 0) || !(f_low > 0)) return false;
  for (int64_t i = 0; i < n_tmpl; ++i)
    if (!(m1[i] > 0) || !(m2[i] > 0)) return false;
  return true;
}

cudaError_t launch_taylorf2(const void* tables, int64_t t0, int64_t n_rows, double fs, int64_t n, double f_low,
                            int64_t k_hi, void* work, float2* out, int64_t ld, cudaStream_t st) {
  const double df = fs / (double)n;
  const int64_t nb = n / 2 + 1;
  // Only the anchors that a band needs.  Where an anchor per bin is called for (bins of 0.25 Hz) and the band is a small
  // part of the row, space and blocks for all of them took longer than the phases: 300 rows of 2^18 samples at
  // 65,536 Hz 649 us, 331 us so (425 us with the phases in the kernel of the bins).
  const Anchors an = anchors_of(n, fs, f_low, k_hi);
  const int na = an.count;
  // The frequency k df to FP32.  With a df that FP32 holds exactly (any whole sampling rate up to 2^24 Hz) the FP64
  // product is exact, so one FP32 multiplication rounds it alike; otherwise two conversions and a product in FP64, 2 of
  // which the chip does per clock and SM: 340 us of k_taylorf2 instead of 804 us for 384 rows at N = 2^20.
  const float df32 = (double)(float)df == df && nb <= 1 << 24 ? (float)df : 0.f;
  const TF2* d = static_cast<const TF2*>(tables) + t0;
  double* psi = static_cast<double*>(work);
  for (int64_t r = 0; r < n_rows; r += 65535) {
    const unsigned rows = (unsigned)std::min<int64_t>(65535, n_rows - r);
    if (na > 0) {
      k_tf2_anchors<<<dim3((unsigned)((na + kGenThreads - 1) / kGenThreads), rows), kGenThreads, 0, st>>>(
          d + r, df, na, an.a0, psi + r * na);
      add_launches(1);
    }
    k_taylorf2<<<dim3((unsigned)((nb + kGenChunk - 1) / kGenChunk), rows), kGenThreads, 0, st>>>(
        d + r, psi + r * na, na, an.a0, df, df32, out + r * ld, ld, nb);
    add_launches(1);
  }
  return cudaGetLastError();
}

}  // namespace mf

extern "C" mf_status mf_taylorf2(const double* m1, const double* m2, int64_t n_tmpl, double fs, int64_t n,
                                 double f_low, void* out, int64_t ld, void* cuda_stream) {
  if (!m1 || !m2 || !out) {
    mf::set_global_error("mf_taylorf2: null argument");
    return MF_EINVAL;
  }
  if (ld < n / 2 + 1 || !mf::taylorf2_valid(m1, m2, n_tmpl, fs, n, f_low)) {
    mf::set_global_error("mf_taylorf2: bad sizes, masses or band");
    return MF_EINVAL;
  }
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const int64_t k_hi = mf::taylorf2_k_hi(m1, m2, n_tmpl, fs, n, f_low);
  const int64_t block = mf::taylorf2_block(n_tmpl, fs, n, f_low, k_hi);
  const size_t table = mf::taylorf2_table_bytes(n_tmpl);
  char* dev = nullptr;
  cudaError_t e = cudaMalloc((void**)&dev, table + mf::taylorf2_work_bytes(block, fs, n, f_low, k_hi));
  if (e != cudaSuccess) cudaGetLastError();
  if (e == cudaSuccess) e = mf::taylorf2_tables(m1, m2, n_tmpl, fs, n, f_low, dev, st);
  for (int64_t r = 0; r < n_tmpl && e == cudaSuccess; r += block)
    e = mf::launch_taylorf2(dev, r, std::min(block, n_tmpl - r), fs, n, f_low, k_hi, dev + table,
                            static_cast<float2*>(out) + r * ld, ld, st);
  const cudaError_t e2 = cudaStreamSynchronize(st);
  if (dev) cudaFree(dev);
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) {
    mf::set_global_error(std::string("mf_taylorf2: ") + cudaGetErrorString(e));
    return MF_ECUDA;
  }
  return MF_OK;
}
