// PSD estimation upstream of the filter: Welch's method on the GPU.
//
// The weights of Eq. (2) need the one-sided PSD S_n of the data; the paper
// takes it from the data without describing the estimate.  Reading: Welch
// segments of seg_len samples every stride samples with a periodic Hann
// window and no detrending, averaged by the mean or by the median divided by
// its bias for exponential periodogram values (FINDCHIRP, Appendix B).
// The windowed segments go straight into the library's real-input transform (k_pass1 / k_pass2 with a windowing
// load), and k_welch_mean or k_welch_median reduces each bin's periodogram values, FP64, over the segments.
#include <cuda_runtime.h>

#include <cmath>
#include <string>

#include "../../include/mf.h"
#include "mf_common.cuh"

namespace mf {
namespace {

constexpr int kWT = 256;        // threads per reduction CTA
constexpr int kMaxSeg = 4096;   // segments held in shared memory by the median
constexpr int kMedianBytes = 48 << 10;

// psd[d][k] = average over segments s of norm |X_s[k]|^2, norm = c fs / sum w^2, with X the dt-normalised spectrum of
// the windowed segment (so |FFT|^2 = fs^2 |X|^2), sum w^2 = 3n/8 and c = 2 off DC and Nyquist (norm from the host).
struct Norm {
  double edge, inner;  // c = 1, c = 2
};

__device__ __forceinline__ double periodogram(float2 z, double norm) {
  return norm * abs2_f64(z);
}

// mean: a CTA takes 32 bins (256-byte reads), each of its W warps every W-th segment, the warps' sums in order.  Eight
// warps; beyond 4,096 segments their walk is longer than everything else in the call, and 32 share it (20,000 segments of
// 2^12 samples: 2,728 -> 2,140 us; a CTA per bin took 2,522).
template <int W>
__global__ void __launch_bounds__(32 * W) k_welch_mean(const float2* __restrict__ fd, int64_t ld_fd, int n_det,
                                                       int64_t n_seg, int64_t n, Norm nm, double* __restrict__ psd) {
  __shared__ double part[W][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, d = blockIdx.y;
  const int64_t k = (int64_t)blockIdx.x * 32 + lane;
  const double norm = k == 0 || k == n / 2 ? nm.edge : nm.inner;
  double s = 0.0;
  if (k <= n / 2)
    for (int64_t i = w; i < n_seg; i += W) s += periodogram(fd[(i * n_det + d) * ld_fd + k], norm);
  part[w][lane] = s;
  __syncthreads();
  if (w == 0 && k <= n / 2) {
    for (int i = 1; i < W; ++i) s += part[i][lane];
    psd[(int64_t)d * (n / 2 + 1) + k] = s / (double)n_seg;
  }
}

// The r-th smallest (from 0) of count >= r + 1 keys, 32 K >= count, by a warp: lane i holds keys i, i + 32, ... (absent
// ones all ones, which are above every key).  Quickselect over the range [lo, hi] that still holds it, the pivot a key
// of the range from another lane each time; *less = the number of keys below the result.
template <int K>
__device__ __forceinline__ unsigned long long select_key(const unsigned long long (&v)[K], int r, int* less) {
  unsigned long long lo = 0, hi = ~0ull - 1;
  for (int step = 0;; ++step) {
    unsigned long long mine = 0;
    bool have = false;
#pragma unroll
    for (int i = 0; i < K; ++i)
      if (v[i] >= lo && v[i] <= hi) {
        mine = v[i];
        have = true;
      }
    const unsigned m = __ballot_sync(0xffffffffu, have);
    if (!m) {  // (not reached by numbers: the range always holds the key)
      *less = 0;
      return ~0ull;
    }
    const int turn = (step * 11 + 16) & 31;
    const unsigned long long pivot =
        __shfl_sync(0xffffffffu, mine, ((__ffs(__funnelshift_r(m, m, turn)) - 1) + turn) & 31);
    int below = 0, equal = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      below += v[i] < pivot ? 1 : 0;
      equal += v[i] == pivot ? 1 : 0;
    }
    below = __reduce_add_sync(0xffffffffu, below);
    equal = __reduce_add_sync(0xffffffffu, equal);
    if (r < below) {
      hi = pivot - 1;
    } else if (r < below + equal) {
      *less = below;
      return pivot;
    } else {
      lo = pivot + 1;
    }
  }
}

// the median of n values >= 0 given by their bits in shared memory
template <int K>
__device__ __forceinline__ double median_of(const unsigned long long* s, int n) {
  const int lane = threadIdx.x & 31;
  unsigned long long v[K];
#pragma unroll
  for (int i = 0; i < K; ++i) v[i] = lane + 32 * i < n ? s[lane + 32 * i] : ~0ull;
  int less;
  const unsigned long long upper = select_key<K>(v, n / 2, &less);
  if (n & 1) return __longlong_as_double((long long)upper);
  unsigned long long lower = upper;  // the one before it: the largest key below it, or another equal to it
  if (less == n / 2) {
    lower = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) lower = v[i] < upper && v[i] > lower ? v[i] : lower;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long y = __shfl_xor_sync(0xffffffffu, lower, o);
      lower = y > lower ? y : lower;
    }
  }
  return 0.5 * (__longlong_as_double((long long)lower) + __longlong_as_double((long long)upper));
}

// median: a CTA takes `bins` bins (a power of two that fits shared memory) with all their values, then a warp per
// bin takes them into registers (K per lane, 32 K >= n_seg) and selects the middle ones.  The values are >= 0, so
// their bits are in their order: the comparisons are integer ones, not FP64 ones, of which the chip does 2 per clock
// and SM.  For 127 segments of two detectors and 8,193 bins: a CTA per bin that read one 8-byte value per row and
// sorted them 223 us, keys read from shared memory for each comparison 59 us, the
// same with keys in registers 44 us, and with abs2_f64 35 us.
// K goes in steps, for a lane compares all its K keys however few there are (segments of 2^14 samples, two detectors,
// the whole call: 1,000 segments 2,785 us with the sort, 3,211 with K = 128, 1,046 with K = 32; 2,000 of 2^12 samples 1,696,
// 1,753 and, K = 64, 943).  K = 128 needs more registers than there are (255, 480 bytes of spills): from 2,049 segments on
// it is what it is, 4,096 of 2^12 samples 3,293 us with the sort and 3,102 so.
template <int K>
__global__ void __launch_bounds__(kWT) k_welch_median(const float2* __restrict__ fd, int64_t ld_fd, int n_det,
                                                      int n_seg, int64_t n, Norm nm, double median_bias, int bins,
                                                      double* __restrict__ psd) {
  extern __shared__ unsigned long long keys[];  // [bins][n_seg | 1]
  const int pitch = n_seg | 1, d = blockIdx.y;
  const int64_t k0 = (int64_t)blockIdx.x * bins;
  const int b = threadIdx.x % bins;
  const double norm = k0 + b == 0 || k0 + b == n / 2 ? nm.edge : nm.inner;
  if (k0 + b <= n / 2)
    for (int i = threadIdx.x / bins; i < n_seg; i += kWT / bins)
      keys[b * pitch + i] = (unsigned long long)__double_as_longlong(
          periodogram(fd[((int64_t)i * n_det + d) * ld_fd + k0 + b], norm));
  __syncthreads();
  for (int c = threadIdx.x >> 5; c < bins && k0 + c <= n / 2; c += kWT / 32) {
    const unsigned long long* v = keys + c * pitch;
    const double med = median_of<K>(v, n_seg);
    if ((threadIdx.x & 31) == 0) psd[(int64_t)d * (n / 2 + 1) + k0 + c] = med / median_bias;
  }
}

}  // namespace
}  // namespace mf

extern "C" mf_status mf_psd_welch(double fs, int32_t n_det, int64_t n_samples, const float* strain, int64_t ld,
                                  int64_t seg_len, int64_t stride, int32_t average, double* psd, void* cuda_stream) {
  auto bad = [](const char* m) {
    mf::set_global_error(std::string("mf_psd_welch: ") + m);
    return MF_EINVAL;
  };
  if (!strain || !psd) return bad("null argument");
  if (!(fs > 0) || n_det < 1 || n_det > 8 || ld < n_samples) return bad("fs, n_det or ld");
  if (seg_len < 4096 || seg_len > mf::kMaxN || (seg_len & (seg_len - 1))) return bad("seg_len must be a power of two in [2^12, 2^20]");
  if (stride < 1 || n_samples < seg_len) return bad("stride < 1 or data shorter than one segment");
  if (average != 0 && average != 1) return bad("average must be 0 (mean) or 1 (median)");
  const int64_t n_seg = (n_samples - seg_len) / stride + 1;
  if (average == 1 && n_seg > mf::kMaxSeg) return bad("more than 4096 segments for the median");
  const int64_t rows = n_seg * n_det;
  const int64_t nb = seg_len / 2 + 1, ld_fd = (nb + 63) / 64 * 64;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  // one allocation for the call's work space (three, with their frees, were two thirds of a call's time; fewer bytes,
  // as intermediates of 8 MB of segments at a time, take as long to allocate and two more launches each: 302 -> 316 us)
  const size_t scratch_bytes = (size_t)rows * seg_len * sizeof(float2);
  char* work = nullptr;
  cudaError_t e = cudaMalloc((void**)&work, scratch_bytes + (size_t)rows * ld_fd * sizeof(float2));
  if (e != cudaSuccess) {
    cudaGetLastError();
    mf::set_global_error(std::string("mf_psd_welch: work space: ") + cudaGetErrorString(e));
    return MF_ENOMEM;
  }
  float2 *scratch = reinterpret_cast<float2*>(work), *fd = reinterpret_cast<float2*>(work + scratch_bytes);
  // median bias of n_seg exponential values: 1 - 1/2 + 1/3 - ... to 1/(2m+1), m = (n_seg - 1) / 2
  double bias = 1.0;
  for (int64_t i = 1; i <= (n_seg - 1) / 2; ++i) bias += 1.0 / (2.0 * i + 1.0) - 1.0 / (2.0 * i);
  const mf::Norm nm{1.0 * fs / (0.375 * (double)seg_len), 2.0 * fs / (0.375 * (double)seg_len)};
  e = mf::launch_welch_spectra(strain, ld, n_det, stride, (int)rows, seg_len, 1.0 / fs, scratch, fd, ld_fd, st);
  if (e == cudaSuccess) {
    if (average == 0) {
      const dim3 grid((unsigned)((nb + 31) / 32), (unsigned)n_det);
      if (n_seg <= 4096)
        mf::k_welch_mean<8><<<grid, 256, 0, st>>>(fd, ld_fd, n_det, n_seg, seg_len, nm, psd);
      else
        mf::k_welch_mean<32><<<grid, 1024, 0, st>>>(fd, ld_fd, n_det, n_seg, seg_len, nm, psd);
    } else {
      int bins = 32;
      while (bins > 1 && bins * (n_seg | 1) * 8 > mf::kMedianBytes) bins /= 2;
      auto k = n_seg <= 128    ? mf::k_welch_median<4>
               : n_seg <= 512  ? mf::k_welch_median<16>
               : n_seg <= 1024 ? mf::k_welch_median<32>
               : n_seg <= 2048 ? mf::k_welch_median<64>
                               : mf::k_welch_median<128>;
      k<<<dim3((unsigned)((nb + bins - 1) / bins), (unsigned)n_det), mf::kWT, (size_t)(bins * (n_seg | 1) * 8), st>>>(
          fd, ld_fd, n_det, (int)n_seg, seg_len, nm, bias, bins, psd);
    }
    mf::add_launches(1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(work);
  if (e != cudaSuccess) {
    mf::set_global_error(std::string("mf_psd_welch: ") + cudaGetErrorString(e));
    return MF_ECUDA;
  }
  return MF_OK;
}
