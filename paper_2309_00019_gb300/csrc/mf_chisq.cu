// Signal-based veto at trigger times: Allen's chi^2 over p bands of equal
// template power and the re-weighted SNR of Eq. (4).
//
// The filter output of a trigger, z = sum_k w s~ h~* e^{+2 pi i k j / N},
// is split by frequency band, z_l = the same sum over band l, and
//   chi^2 = p sum_l |z_l - z / p|^2 / sigma^2   (2p - 2 degrees of freedom),
//   rho~ = rho / [(1 + chi2_r^3) / 2]^{1/6} if chi2_r = chi^2 / (2p - 2) >= 1.
// Band l holds the bins k whose template power below k, C(k), satisfies
// floor(p C(k) / sigma^2) = l (clamped to p - 1): k_block_power and
// k_chisq_edges find the first bin of every band with FP64 block sums, once
// per bank and p; k_chisq then
// sums the triggers' terms in the bank's column layout (contiguous reads of
// the template and the weighted data), a CTA per run of up to eight triggers
// of one template and detector.
#include <algorithm>

#include "mf_common.cuh"

namespace mf {

namespace {

constexpr int kCT = 128;  // threads per CTA

template <int BT>
__device__ __forceinline__ float2 elem(const void* p, int64_t i) {
  return BankElem<BT>::get(p, i);
}

// Template power per block of PB = min(256, N2) consecutive bins in frequency
// order (block b = bins [b PB, (b + 1) PB), all in one row k1 of the column
// layout), FP64, from the column-layout bank: bpow[t][b] = sum w |h|^2.
// grid (N2 / PB, n_tmpl); each thread owns rows k1 and walks the PB columns of
// its block, so the reads of every column are contiguous and the sums have a
// fixed order.
template <int BT>
__global__ void __launch_bounds__(kCT) k_block_power(const void* __restrict__ bank, int64_t ld_bank, int n1, int n2,
                                                     int pb, const double* __restrict__ w, double* __restrict__ bpow) {
  const int64_t t = blockIdx.y;
  const int cb = blockIdx.x;
  const int R = n1 / 2;
  const int nbl_row = n2 / pb;
  const void* row = static_cast<const unsigned char*>(bank) + t * ld_bank * (BT == kBankF32 ? 8 : 4);
  for (int k1 = threadIdx.x; k1 < R; k1 += blockDim.x) {
    double acc = 0.0;
    for (int c = 0; c < pb; ++c) {
      const int k2 = cb * pb + c;
      const int64_t k = (int64_t)k1 * n2 + k2;
      const float2 h = BankElem<BT>::get(row, (int64_t)k2 * R + k1);
      if (h.x != 0.f || h.y != 0.f) {  // (FP64 bounds this kernel: exact zeros are skipped)
        const double wk = w[k];
        if (nonzero_f64(wk)) acc = fma(wk, abs2_f64(h), acc);
      }
    }
    bpow[t * ((int64_t)R * nbl_row) + (int64_t)k1 * nbl_row + cb] = acc;
  }
}

// edges[t][l] = first bin k of band l, i.e. the first k with w[k] != 0 and p C(k) / sigma^2 >= l, with C(k) the
// template power below k (l < p); edges[t][p] = nb.  One CTA per template: a prefix sum over the blocks, then a warp
// per edge finds its block by bisection and its bin by a prefix sum over the block.  (A warp per template whose lanes
// walked the blocks one by one, with an FP64 division each, took 0.7 ms for 150 templates at N = 2^18.)
constexpr int kEdgeThreads = 256;

template <int BT>
__global__ void __launch_bounds__(kEdgeThreads) k_chisq_edges(const void* __restrict__ bank, int64_t ld_bank, int n1,
                                                              int n2, int pb, const double* __restrict__ w, int64_t nb,
                                                              const double* __restrict__ bpow, int n_blocks, int p,
                                                              int32_t* __restrict__ edges) {
  extern __shared__ double below[];  // [n_blocks + 1] power below each block
  __shared__ double part[kEdgeThreads];
  const int64_t t = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31;
  const double* bp = bpow + t * n_blocks;
  const int per = (n_blocks + kEdgeThreads - 1) / kEdgeThreads, b0 = min(tid * per, n_blocks), b1 = min(b0 + per, n_blocks);
  double s = 0.0;
  for (int b = b0; b < b1; ++b) s += bp[b];
  part[tid] = s;
  __syncthreads();
  if (tid == 0) {
    double run = 0.0;
    for (int i = 0; i < kEdgeThreads; ++i) {
      const double v = part[i];
      part[i] = run;
      run += v;
    }
    below[n_blocks] = run;
  }
  __syncthreads();
  double run = part[tid];
  for (int b = b0; b < b1; ++b) {
    below[b] = run;
    run += bp[b];
  }
  __syncthreads();
  const double total = below[n_blocks];
  const int R = n1 / 2;
  const void* row = static_cast<const unsigned char*>(bank) + t * ld_bank * (BT == kBankF32 ? 8 : 4);
  for (int l = tid / 32; l <= p; l += kEdgeThreads / 32) {
    int64_t e = nb;
    if (l < p && total > 0.0) {
      const double target = (double)l * total / (double)p;
      int lo = 0, hi = n_blocks;  // the first block with power up to its end >= target
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (below[mid + 1] >= target) hi = mid; else lo = mid + 1;
      }
      for (int b = lo; b < n_blocks && e == nb; ++b) {
        double c = below[b];  // power below the bins at hand
        for (int k0 = b * pb; k0 < (b + 1) * pb && e == nb; k0 += 32) {
          const int64_t k = k0 + lane;
          const double wk = w[k];
          double v = 0.0;
          if (wk != 0.0) {
            const float2 h = BankElem<BT>::get(row, (k % n2) * R + k / n2);
            v = wk * abs2_f64(h);
          }
          double x = v;  // inclusive scan
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
          }
          const unsigned m = __ballot_sync(0xffffffffu, wk != 0.0 && c + (x - v) >= target);
          if (m) e = k0 + __ffs(m) - 1;
          c += __shfl_sync(0xffffffffu, x, 31);
        }
      }
    }
    if (lane == 0) edges[t * (p + 1) + l] = (int32_t)e;
  }
}

struct TrigRecC {
  int32_t det, tmpl;
  int64_t sample;
  float snr, phase;
};

// chi^2 of a run of up to G triggers of one template and detector at a time.
//
// With k = k1 N2 + k2 the phase splits, exp(2 pi i k j / N) = exp(2 pi i k1 j / N1) exp(2 pi i k2 j / N), so a
// thread takes one row k1 (or, below 256 rows, one of `parts` equal pieces of it, so that the CTA's pieces s are
// consecutive ranges of bins), walks its k2 with the phases of k2 from a table that the whole CTA shares, and
// turns the sum once.  Neighbouring threads read neighbouring k1, the bank's fastest index.  A band is a range
// of bins, so most pieces lie in one band: sums of whole pieces go to whole[s], of a piece's part behind a
// band's first bin to head[band], of its part in front of one to tail[band]; each has one writer, and a warp per
// band adds them in a fixed order (FP64).  The triggers of a run share the loads: reading the template and the data
// from L2 once per run is what bounds the kernel.  Before, a thread walked its own run of consecutive elements (no
// two lanes in one line) with a phase recurrence, and one thread added all partial sums: 4,105 us for the triggers of
// 150 templates of two detectors at N = 2^18, threshold 4.5 (2 MB of template and data each); now
// 377 us (469 us with runs of up to four).
constexpr int kChiThreads = 256;
constexpr int kChiRun = 8;  // triggers that share their loads, at most

// half of that where the tables of eight would leave one CTA per SM
constexpr int chisq_run_max(int n2) { return n2 <= 512 ? kChiRun : kChiRun / 2; }

template <int BT, int QT, int G>
__device__ __forceinline__ void chisq_run(const TrigRecC* __restrict__ trig, int64_t it, const void* __restrict__ bank,
                                          int64_t ld_bank, const void* __restrict__ q, int64_t ld_q, int n1, int n2,
                                          const int32_t* __restrict__ edges, int p, const float* __restrict__ ratio,
                                          const float* __restrict__ dscale, float* __restrict__ chi2,
                                          float* __restrict__ newsnr, int n_run, unsigned char* sm) {
  const int R = n1 / 2, tid = threadIdx.x;
  const int parts = R < kChiThreads ? kChiThreads / R : 1, len = n2 / parts, pieces = R * parts;
  float2* ph = reinterpret_cast<float2*>(sm);  // [n2][G] phases of k2
  float2* whole = ph + n2 * G;                 // [pieces][G]
  float2* head = whole + pieces * G;           // [p][G]
  float2* tail = head + p * G;                 // [p][G]
  double2* zl = reinterpret_cast<double2*>(tail + p * G);  // [p][G]
  int32_t* e = reinterpret_cast<int32_t*>(zl + p * G);     // [p + 1]
  const TrigRecC tr = trig[it];
  const uint32_t N = (uint32_t)n1 * (uint32_t)n2;
  const void* hrow = static_cast<const unsigned char*>(bank) + (int64_t)tr.tmpl * ld_bank * (BT == kBankF32 ? 8 : 4);
  const void* qrow = static_cast<const unsigned char*>(q) + (int64_t)tr.det * ld_q * (QT == kBankF32 ? 8 : 4);
  // a run shorter than G repeats its last trigger (products modulo powers of two: the low bits are all that counts)
  auto sample = [&](int g) { return (uint32_t)trig[it + min(g, n_run - 1)].sample; };
  for (int i = tid; i < n2 * G; i += kChiThreads) ph[i] = unit_root(((uint32_t)(i / G) * sample(i % G)) & (N - 1), N);
  for (int i = tid; i < (pieces + 2 * p) * G; i += kChiThreads) whole[i] = make_float2(0.f, 0.f);
  for (int i = tid; i <= p; i += kChiThreads) e[i] = edges[(int64_t)tr.tmpl * (p + 1) + i];
  __syncthreads();
  for (int s0 = tid; s0 < pieces; s0 += kChiThreads) {
    const int k1 = s0 % R, part = s0 / R, c0 = part * len, s = k1 * parts + part;
    const int first = k1 * n2 + c0;  // the piece's bins [first, first + len)
    int lo = -1, hi = p + 1;         // largest l with e[l] <= first (-1: below the bands)
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (e[mid] <= first) lo = mid; else hi = mid;
    }
    int band = lo, begin = 0;                                          // of the current stretch
    int next = band < p ? min(e[band + 1] - first, len) : len;         // its end
    float2 acc[G];
#pragma unroll
    for (int g = 0; g < G; ++g) acc[g] = make_float2(0.f, 0.f);
    auto flush = [&](int end) {  // the stretch [begin, end) of the piece is summed
      if (band >= 0 && band < p && end > begin) {
        float2* to = begin == 0 ? (end == len ? whole + s * G : tail + band * G) : head + band * G;
#pragma unroll
        for (int g = 0; g < G; ++g) {
          to[g] = cmul(acc[g], unit_root(((uint32_t)k1 * sample(g)) & (uint32_t)(n1 - 1), (uint32_t)n1));
        }
      }
#pragma unroll
      for (int g = 0; g < G; ++g) acc[g] = make_float2(0.f, 0.f);
    };
    auto add = [&](int c, float2 qv, float2 hv) {
      const float2 x = cmulc(qv, hv);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float2 w = ph[(c0 + c) * G + g];
        acc[g].x = fmaf(x.x, w.x, fmaf(-x.y, w.y, acc[g].x));
        acc[g].y = fmaf(x.x, w.y, fmaf(x.y, w.x, acc[g].y));
      }
    };
    constexpr int U = 8;  // loads in flight (len is a multiple of 8)
    for (int c = 0; c < len; c += U) {
      float2 qv[U], hv[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t i = (int64_t)(c0 + c + u) * R + k1;
        qv[u] = elem<QT>(qrow, i);
        hv[u] = elem<BT>(hrow, i);
      }
      if (c + U <= next) {
#pragma unroll
        for (int u = 0; u < U; ++u) add(c + u, qv[u], hv[u]);
      } else {
#pragma unroll 1
        for (int u = 0; u < U; ++u) {  // (loads again: their values stay in registers only in the unrolled path)
          while (c + u == next && next < len) {  // the next band (or an empty one) begins here
            flush(next);
            begin = next;
            ++band;
            next = band < p ? min(e[band + 1] - first, len) : len;
          }
          const int64_t i = (int64_t)(c0 + c + u) * R + k1;
          add(c + u, elem<QT>(qrow, i), elem<BT>(hrow, i));
        }
      }
    }
    flush(len);
  }
  __syncthreads();
  // z_l: the pieces of band l, by a warp
  const int lane = tid & 31;
  for (int i = tid / 32; i < p * G; i += kChiThreads / 32) {
    const int l = i / G, g = i % G;
    const int s_lo = e[l] / len, s_hi = (e[l + 1] < R * n2 ? e[l + 1] : R * n2) / len;  // whole pieces: (s_lo, s_hi)
    double a = 0.0, b = 0.0;
    if (e[l] < e[l + 1]) {
      for (int s = s_lo + lane; s < s_hi; s += 32) {
        if (s == s_lo && e[l] % len != 0) continue;  // its part in this band is head[l]
        a += whole[s * G + g].x;
        b += whole[s * G + g].y;
      }
      if (lane == 0) {
        a += head[i].x + (double)tail[i].x;
        b += head[i].y + (double)tail[i].y;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (lane == 0) zl[i] = make_double2(a, b);
  }
  __syncthreads();
  if (tid < n_run) {
    // z_l in stored units (data / sigma_ref, template / scale): |z_true| = |z| ratio / c_d
    float r = ratio[tr.tmpl];
    if (dscale) r /= dscale[tr.det];
    double zr = 0.0, zi = 0.0, c2 = 0.0;
    for (int l = 0; l < p; ++l) {
      zr += zl[l * G + tid].x;
      zi += zl[l * G + tid].y;
    }
    for (int l = 0; l < p; ++l) {
      const double dr = zl[l * G + tid].x - zr / p, di = zl[l * G + tid].y - zi / p;
      c2 += dr * dr + di * di;
    }
    c2 *= (double)p * (double)r * (double)r;
    chi2[it + tid] = (float)c2;
    const double cr = c2 / (2.0 * p - 2.0);
    const float snr = trig[it + tid].snr;
    newsnr[it + tid] = cr >= 1.0 ? (float)((double)snr / pow((1.0 + cr * cr * cr) / 2.0, 1.0 / 6.0)) : snr;
  }
  __syncthreads();
}

constexpr int chisq_smem(int n1, int n2, int p) {
  const int pieces = n1 / 2 < kChiThreads ? kChiThreads : n1 / 2, g = chisq_run_max(n2);
  return (n2 + pieces + 2 * p) * g * 8 + p * g * 16 + (p + 1) * 4;
}
constexpr int kChisqSmemMax =
    chisq_smem(1024, 512, 64) > chisq_smem(1024, 1024, 64) ? chisq_smem(1024, 512, 64) : chisq_smem(1024, 1024, 64);

// The list is ordered by detector and template.  Each stretch of triggers of one detector and template is cut into
// runs of G from its start on; a CTA takes the runs that begin in its block of `per` triggers.  G grows with the number
// of triggers up to chisq_run_max, so that few of them still spread over the grid.
template <int BT, int QT>
__global__ void __launch_bounds__(kChiThreads, 2) k_chisq(const TrigRecC* __restrict__ trig,
                                                       const int64_t* __restrict__ count, int64_t cap,
                                                       const void* __restrict__ bank, int64_t ld_bank,
                                                       const void* __restrict__ q, int64_t ld_q, int n1, int n2,
                                                       const int32_t* __restrict__ edges, int p,
                                                       const float* __restrict__ ratio,
                                                       const float* __restrict__ dscale, float* __restrict__ chi2,
                                                       float* __restrict__ newsnr) {
  extern __shared__ __align__(16) unsigned char smc[];
  const int64_t n_trig = *count < cap ? *count : cap;
  const int64_t per = (n_trig + gridDim.x - 1) / gridDim.x;
  const int G = (int)min((int64_t)chisq_run_max(n2), per), lane = threadIdx.x & 31;
  const int64_t b0 = blockIdx.x * per, b1 = min(b0 + per, n_trig);
  auto same = [&](int64_t a, int64_t b) { return trig[a].tmpl == trig[b].tmpl && trig[a].det == trig[b].det; };
  if (b0 >= b1) return;
  int64_t start = b0;  // of b0's stretch
  for (;;) {
    const int64_t i = start - 1 - lane;
    const unsigned other = __ballot_sync(0xffffffffu, i < 0 || !same(i, b0));
    start -= other ? __ffs(other) - 1 : 32;
    if (other) break;
  }
  for (int64_t it = b0; it < b1; ++it) {
    if (it > b0 && !same(it, it - 1)) start = it;
    if ((it - start) % G != 0) continue;
    int len = 1;
    while (len < G && it + len < n_trig && same(it, it + len)) ++len;
    if (len > 4)
      chisq_run<BT, QT, kChiRun>(trig, it, bank, ld_bank, q, ld_q, n1, n2, edges, p, ratio, dscale, chi2, newsnr, len, smc);
    else if (len > 2)
      chisq_run<BT, QT, 4>(trig, it, bank, ld_bank, q, ld_q, n1, n2, edges, p, ratio, dscale, chi2, newsnr, len, smc);
    else if (len == 2)
      chisq_run<BT, QT, 2>(trig, it, bank, ld_bank, q, ld_q, n1, n2, edges, p, ratio, dscale, chi2, newsnr, len, smc);
    else
      chisq_run<BT, QT, 1>(trig, it, bank, ld_bank, q, ld_q, n1, n2, edges, p, ratio, dscale, chi2, newsnr, len, smc);
  }
}

int sms_c() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

}  // namespace

// blocks of the template-power prefix: PB = min(256, N2) bins, N/2 / PB blocks
int chisq_pb(int n2) { return n2 < 256 ? n2 : 256; }
int64_t chisq_blocks(int n1, int n2) { return (int64_t)n1 / 2 * n2 / chisq_pb(n2); }

cudaError_t launch_chisq_edges(const void* bank, int bank_type, int64_t ld_bank, int64_t n_tmpl, int n1, int n2,
                               const double* w, int64_t nb, double* bpow, int p, int32_t* edges, cudaStream_t st) {
  if (p < 2 || p > 64 || n_tmpl <= 0) return cudaErrorInvalidValue;
  const int pb = chisq_pb(n2);
  const int64_t nbl = chisq_blocks(n1, n2);
  const size_t smem = (size_t)(nbl + 1) * sizeof(double);  // up to 2,048 blocks: 16 KB
  for (int64_t t0 = 0; t0 < n_tmpl; t0 += 65535) {
    const dim3 gp((unsigned)(n2 / pb), (unsigned)std::min<int64_t>(65535, n_tmpl - t0));
    const int64_t eb = bank_type == kBankF32 ? 8 : 4;
    const void* b0 = static_cast<const unsigned char*>(bank) + t0 * ld_bank * eb;
    double* o = bpow + t0 * nbl;
    switch (bank_type) {
      case kBankF32: k_block_power<kBankF32><<<gp, kCT, 0, st>>>(b0, ld_bank, n1, n2, pb, w, o); break;
      case kBankF16: k_block_power<kBankF16><<<gp, kCT, 0, st>>>(b0, ld_bank, n1, n2, pb, w, o); break;
      case kBankBF16: k_block_power<kBankBF16><<<gp, kCT, 0, st>>>(b0, ld_bank, n1, n2, pb, w, o); break;
      default: return cudaErrorInvalidValue;
    }
    add_launches(1);
  }
  switch (bank_type) {
    case kBankF32: k_chisq_edges<kBankF32><<<(unsigned)n_tmpl, kEdgeThreads, smem, st>>>(bank, ld_bank, n1, n2, pb, w, nb, bpow, (int)nbl, p, edges); break;
    case kBankF16: k_chisq_edges<kBankF16><<<(unsigned)n_tmpl, kEdgeThreads, smem, st>>>(bank, ld_bank, n1, n2, pb, w, nb, bpow, (int)nbl, p, edges); break;
    case kBankBF16: k_chisq_edges<kBankBF16><<<(unsigned)n_tmpl, kEdgeThreads, smem, st>>>(bank, ld_bank, n1, n2, pb, w, nb, bpow, (int)nbl, p, edges); break;
    default: return cudaErrorInvalidValue;
  }
  add_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_chisq(const void* trig, const int64_t* count, int64_t cap, const void* bank, int bank_type,
                         int64_t ld_bank, const void* q, int q_type, int64_t ld_q, int n1, int n2, const int32_t* edges,
                         int p, const float* ratio, const float* dscale, float* chi2, float* newsnr, cudaStream_t st) {
  if (p < 2 || p > 64) return cudaErrorInvalidValue;
  const int grid = sms_c() * 2;  // as many as are resident; twice as many have half the triggers each, and shorter runs: 417 us
  const int smem = chisq_smem(n1, n2, p);
  const TrigRecC* t = static_cast<const TrigRecC*>(trig);
#define MF_CHISQ(BT, QT)                                                                                        \
  do {                                                                                                          \
    auto k = k_chisq<BT, QT>;                                                                                   \
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kChisqSmemMax);  \
    if (e != cudaSuccess) return e;                                                                             \
    k<<<grid, kChiThreads, smem, st>>>(t, count, cap, bank, ld_bank, q, ld_q, n1, n2, edges, p, ratio, dscale, chi2, \
                                       newsnr);                                                                 \
  } while (0)
  if (q_type == kBankF32) {
    switch (bank_type) {
      case kBankF32: MF_CHISQ(kBankF32, kBankF32); break;
      case kBankF16: MF_CHISQ(kBankF16, kBankF32); break;
      case kBankBF16: MF_CHISQ(kBankBF16, kBankF32); break;
      default: return cudaErrorInvalidValue;
    }
  } else if (q_type == bank_type && q_type == kBankF16) {
    MF_CHISQ(kBankF16, kBankF16);
  } else if (q_type == bank_type && q_type == kBankBF16) {
    MF_CHISQ(kBankBF16, kBankBF16);
  } else {
    return cudaErrorInvalidValue;
  }
#undef MF_CHISQ
  add_launches(1);
  return cudaGetLastError();
}

namespace {

// One CTA per trigger: for a trigger of a template heavier than m_min and with rho~ >= snr_min, the SNR of
// every sine-Gaussian tile at the trigger sample.  Tile l of template t: f_l = f_final[t] + offsets[l]
// (skipped at or above f_high), g~[k] = exp(-(pi tau (f_k - f_l))^2), tau = qf / (sqrt(2) pi f_l); only the
// bins within 6 / (pi tau) of f_l enter (beyond, g~ < 3e-16).  rho_l^2 = |sum_k w s~ g~ e^{+2 pi i k j / N}|^2
// / sum_k w g~^2 with the weighted data read in the column layout and rescaled from its stored units.
// Bound by its few warps' latencies and FP64.  150 templates of two detectors at N = 2^18, those of 12 solar masses and
// more taken through it: the vetoes' call 11.8 ms with 64-bit divisions and an FP64 comparison per bin, 8.7 ms without.
template <int QT>
__global__ void __launch_bounds__(kCT) k_sgchisq(const TrigRecC* __restrict__ trig, const int64_t* __restrict__ count,
                                                 int64_t cap, const void* __restrict__ q, int64_t ld_q, int n1, int n2,
                                                 const double* __restrict__ w, double df, double f_high,
                                                 const float* __restrict__ f_final, const float* __restrict__ mtotal,
                                                 float m_min, float snr_min, SgTiles tiles, double q_to_true,
                                                 const float* __restrict__ dscale, const float* __restrict__ snr_in,
                                                 float* __restrict__ chi2_r, float* __restrict__ snr_hat) {
  __shared__ double red[3][kCT];
  const int64_t n_trig = *count < cap ? *count : cap;
  const int R = n1 / 2;
  const int64_t nb = (int64_t)R * n2 + 1;  // bins 0 .. N/2
  const uint32_t N = (uint32_t)n1 * (uint32_t)n2;  // (a power of two, as n1 and n2: masks, not 64-bit divisions, per bin)
  const int lg2 = __ffs(n2) - 1;
  for (int64_t it = blockIdx.x; it < n_trig; it += gridDim.x) {
    const TrigRecC tr = trig[it];
    const float rho = snr_in[it];
    if (!(mtotal[tr.tmpl] > m_min) || !(rho >= snr_min)) {
      if (threadIdx.x == 0) {
        chi2_r[it] = 0.f;
        snr_hat[it] = rho;
      }
      continue;
    }
    const void* qrow = static_cast<const unsigned char*>(q) + (int64_t)tr.det * ld_q * (QT == kBankF32 ? 8 : 4);
    const double scale = dscale ? q_to_true / (double)dscale[tr.det] : q_to_true;
    const uint32_t j = (uint32_t)tr.sample;
    double total = 0.0;
    int used = 0;
    for (int l = 0; l < tiles.n; ++l) {
      const double f0 = (double)f_final[tr.tmpl] + tiles.offset[l];
      if (!(f0 < f_high)) continue;
      const double tau = tiles.q / (1.4142135623730951 * 3.141592653589793 * f0);
      const double half = 6.0 / (3.141592653589793 * tau);
      // (a tile far below zero ends below bin 0, and with q < 8.5 begins above it: both ends are held to the bins before
      // they become 32-bit indices)
      const int klo = (int)min(nb, max((int64_t)1, (int64_t)ceil((f0 - half) / df)));
      const int khi = (int)max((int64_t)0, min(nb - 2, (int64_t)floor((f0 + half) / df)));
      float ar = 0.f, ai = 0.f;
      double s2 = 0.0;
      for (int k = klo + threadIdx.x; k <= khi; k += kCT) {
        const double wk = w[k];
        if (!nonzero_f64(wk)) continue;
        const float x = (float)(3.141592653589793 * tau * ((double)k * df - f0));
        const float g = expf(-x * x);
        const float2 qk = BankElem<QT>::get(qrow, (int64_t)(k & (n2 - 1)) * R + (k >> lg2));  // column layout
        float sn, cs;
        sincospif(2.0f * (float)(((uint32_t)k * j) & (N - 1)) / (float)N, &sn, &cs);
        ar += g * (qk.x * cs - qk.y * sn);
        ai += g * (qk.x * sn + qk.y * cs);
        s2 += wk * (double)g * (double)g;
      }
      red[0][threadIdx.x] = ar;
      red[1][threadIdx.x] = ai;
      red[2][threadIdx.x] = s2;
      __syncthreads();
      if (threadIdx.x == 0) {  // fixed-order sums
        double zr = 0.0, zi = 0.0, ss = 0.0;
        for (int i = 0; i < kCT; ++i) {
          zr += red[0][i];
          zi += red[1][i];
          ss += red[2][i];
        }
        if (ss > 0.0) {
          total += (zr * zr + zi * zi) * scale * scale / ss;
          ++used;
        }
      }
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      const float c = used ? (float)(total / (2.0 * used)) : 0.f;
      chi2_r[it] = c;
      // Eq. 3, inclusive at 6; decided on the stored single-precision value
      snr_hat[it] = c >= 6.f ? (float)((double)rho / sqrt((double)c)) : rho;
    }
  }
}

}  // namespace

cudaError_t launch_sgchisq(const void* trig, const int64_t* count, int64_t cap, const void* q, int q_type, int64_t ld_q,
                           int n1, int n2, const double* w, double df, double f_high, const float* f_final,
                           const float* mtotal, float m_min, float snr_min, const SgTiles& tiles, double q_to_true,
                           const float* dscale, const float* snr_in, float* chi2_r, float* snr_hat, cudaStream_t st) {
  if (tiles.n < 1 || tiles.n > kMaxSgTiles || !(tiles.q > 0)) return cudaErrorInvalidValue;
  const int grid = sms_c() * 4;
  const TrigRecC* t = static_cast<const TrigRecC*>(trig);
#define MF_SG(QT)                                                                                                  \
  k_sgchisq<QT><<<grid, kCT, 0, st>>>(t, count, cap, q, ld_q, n1, n2, w, df, f_high, f_final, mtotal, m_min, snr_min, \
                                      tiles, q_to_true, dscale, snr_in, chi2_r, snr_hat)
  switch (q_type) {
    case kBankF32: MF_SG(kBankF32); break;
    case kBankF16: MF_SG(kBankF16); break;
    case kBankBF16: MF_SG(kBankBF16); break;
    default: return cudaErrorInvalidValue;
  }
#undef MF_SG
  add_launches(1);
  return cudaGetLastError();
}

}  // namespace mf
