// Hierarchy glue kernels (Sec. III): decimation of the frequency-domain data to
// the stage-1 rate, two-detector coincidence with time shifts on the stage-1
// window maxima, and the union of the neighbourhoods of followed-up coarse
// templates that becomes the stage-2 template selection.
#include <algorithm>

#include "mf_internal.h"

namespace mf {

namespace {

int sms() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

__global__ void k_decimate(const float2* __restrict__ in, int64_t ld_in, float2* __restrict__ out, int64_t ld_out,
                           int64_t nb_out, int n_det) {
  const int64_t total = nb_out * n_det;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int d = (int)(i / nb_out);
    const int64_t k = i - (int64_t)d * nb_out;
    out[(int64_t)d * ld_out + k] = in[(int64_t)d * ld_in + k];
  }
}

// max rho^2 over the windows of detector 1, per selection position (a cheap
// bound that lets most detector-0 triggers skip the shift loop)
__global__ void k_max_rho2(const unsigned long long* __restrict__ slots, int64_t n_sel, int64_t n_win, float* out) {
  const int64_t p = blockIdx.x;
  const unsigned long long* row = slots + (n_sel + p) * n_win;  // detector 1
  unsigned int m = 0;
  for (int64_t w = threadIdx.x; w < n_win; w += blockDim.x) {
    const unsigned int hi = (unsigned int)(row[w] >> 32);
    m = hi > m ? hi : m;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned int y = __shfl_xor_sync(0xffffffffu, m, o);
    m = y > m ? y : m;
  }
  __shared__ unsigned int red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < (int)(blockDim.x >> 5); ++i) m = red[i] > m ? red[i] : m;
    m = red[0] > m ? red[0] : m;
    out[p] = __uint_as_float(m);
  }
}

struct CoincRec {
  int32_t tmpl, shift;
  int64_t sample0, sample1;
  float snr0, snr1, rho_c;
  int32_t pad;
};
static_assert(sizeof(CoincRec) == 40, "mf_coinc layout");

__device__ __forceinline__ int64_t key_sample(unsigned long long key) {
  const uint32_t lo = (uint32_t)(key & 0xffffffffull);
  return (int64_t)(((1u << kSampleBits) - 1u) - (lo >> kPhaseBits));
}
__device__ __forceinline__ float key_rho2(unsigned long long key) { return __uint_as_float((uint32_t)(key >> 32)); }

// The kernel for segments of more than kTmplWin windows and for rows with ranges of their own (see k_coinc_tmpl).
// One thread per detector-0 window maximum.  Sample positions are below 2^21, so the ring arithmetic is
// 32-bit, and the ring position of shift k follows from shift k - 1 by one subtraction.
__global__ void k_coinc(CoincArgs a) {
  const int64_t total = a.n_sel * a.n_win;
  const float need = fminf(a.rho_c_thr2, a.rho_c_store2);
  const int32_t R = (int32_t)(a.ring_end - a.ring_begin), rb = (int32_t)a.ring_begin;
  const int32_t win = (int32_t)a.window, cw = (int32_t)a.coinc_window;
  const int32_t step = (int32_t)(a.shift % (int64_t)R);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long kh = a.slots[i];  // detector 0, position p, window w
    if (kh == 0ull) continue;
    const int64_t p = i / a.n_win;
    const float r2h = key_rho2(kh);
    if (r2h + a.max_rho2_det1[p] < need) continue;
    const int64_t sh = key_sample(kh);
    const unsigned long long* row1 = a.slots + (a.n_sel + p) * a.n_win;
    const int32_t tmpl = a.sel[p];
    int32_t x = (int32_t)(sh - a.ring_begin);  // ring position of the detector-0 sample, in [0, R)
    for (int k = 0; k <= a.n_shifts; ++k) {
      // detector-1 triggers at ring position x +- window land on s_h after a shift of k * shift
      if (k > 0) {
        x -= step;
        if (x < 0) x += R;
      }
      int32_t lo[2], hi[2];
      int nint = 1;
      lo[0] = x - cw;
      hi[0] = x + cw;
      if (lo[0] < 0) {
        lo[1] = lo[0] + R; hi[1] = R - 1; lo[0] = 0; nint = 2;
      } else if (hi[0] >= R) {
        lo[1] = 0; hi[1] = hi[0] - R; hi[0] = R - 1; nint = 2;
      }
      for (int q = 0; q < nint; ++q) {
        const int32_t w0 = (lo[q] + rb) / win;
        const int32_t w1 = (hi[q] + rb) / win;
        for (int32_t w = w0; w <= w1; ++w) {
          const unsigned long long kl = row1[w];
          if (kl == 0ull) continue;
          const int32_t y = (int32_t)(key_sample(kl) - a.ring_begin);
          if (y < lo[q] || y > hi[q]) continue;
          const float r2l = key_rho2(kl);
          const float rc2 = r2h + r2l;
          if (rc2 >= a.rho_c_thr2) a.followed[tmpl] = 1;
          if (rc2 >= a.rho_c_store2) {
            const unsigned long long slot = atomicAdd(a.n_coinc, 1ull);
            if ((int64_t)slot < a.coinc_cap) {
              CoincRec* out = reinterpret_cast<CoincRec*>(a.coincs);
              out[slot] = CoincRec{tmpl, k, sh, (int64_t)y + a.ring_begin, sqrtf(r2h), sqrtf(r2l), sqrtf(rc2), 0};
            }
          }
        }
      }
    }
  }
}

// Coincidences of one template per CTA, or of a share of its detector-0 triggers where there are fewer templates than
// SMs.  Of the two triggers of a coincidence at least one has half of the least
// rho_c^2 that counts, and few triggers have: so the pairs (loud detector-0, any detector-1) and (other
// detector-0, loud detector-1) are all there is to look at, and for a pair the shifts follow from the difference
// of its times, k step in [D + m R - window, D + m R + window], without a walk over them.  What a CTA finds is
// collected in shared memory and written in one go.
// Where most triggers are loud the CTA walks over the shifts of every detector-0 trigger instead and looks into the
// windows of detector 1 that it falls on.
// What bounds both is the latency of short dependent steps.  In both a warp's lanes go from pair to pair, turn to turn or
// shift to shift together (a vote or a __syncwarp): a lane that finds something goes its own way, and left to themselves
// the lanes did not come together again but finished their loops one by one.
// Whole calls, us: one thread per detector-0 window over the shifts (k_coinc) / this kernel without that / now
//   2,000 templates, 2,048 windows, zero lag, rho_c 1.5 times the filter's threshold   77 / 90 / 60 (pairs alone 860)
//   300 templates, 64 windows, 501 shifts, 1.42 times                                 405 / 5,570 / 134
//   300 templates, 512 windows, 102 shifts, 1.8 times                                  70 / 18.4 / 18.6
constexpr int kTmplWin = 2048;   // windows whose triggers fit the CTA's shared memory
constexpr int kTmplRec = 512;    // records collected before they go out one by one
constexpr int kTmplSplit = 16;   // CTAs of one template, at most
constexpr int kWalkShifts = 64;  // shifts that a thread walks at a time, at most
constexpr size_t tmpl_smem(int64_t n_win) { return kTmplRec * sizeof(uint2) + (size_t)n_win * 18; }
constexpr uint16_t kNoTrigger = 0xffff;

template <int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS <= 256 ? 1280 / THREADS : 1) k_coinc_tmpl(CoincArgs a) {
  extern __shared__ __align__(16) unsigned char sm[];  // tmpl_smem(n_win)
  uint2* found = reinterpret_cast<uint2*>(sm);  // [kTmplRec] (detector-0 trigger | detector-1 trigger << 16, shift)
  // ring positions and rho^2 of the triggers of detector 0, 1: the loud ones from the front, the others from the end
  int32_t* pos0 = reinterpret_cast<int32_t*>(found + kTmplRec);
  int32_t* pos1 = pos0 + a.n_win;
  float* rho0 = reinterpret_cast<float*>(pos1 + a.n_win);
  float* rho1 = rho0 + a.n_win;
  __shared__ int n_loud[2], n_quiet[2];
  __shared__ unsigned n_found;  // collected, or found before it was seen that the collection is full
  __shared__ unsigned max1;     // the largest rho^2 of detector 1 (float bits)
  __shared__ unsigned long long base;
  const int64_t p = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, n_win = (int)a.n_win;
  if (tid < 2) n_loud[tid] = n_quiet[tid] = 0;
  if (tid == 2) n_found = max1 = 0;
  __syncthreads();
  const float need = fminf(a.rho_c_thr2, a.rho_c_store2), half = 0.5f * need;
  const int32_t rb = (int32_t)a.ring_begin;
  auto put = [&](int d, int w, unsigned long long key) {  // a warp's windows of detector d
    const float r = key_rho2(key);
    const bool listed = key != 0ull && (d == 1 || w % gridDim.y == blockIdx.y);  // detector 0: this CTA's share
    const unsigned big = __ballot_sync(0xffffffffu, listed && r >= half);
    const unsigned rest = __ballot_sync(0xffffffffu, listed) & ~big;
    if (!(big | rest)) return;
    int l0 = 0, q0 = 0;
    if (lane == 0) {
      if (big) l0 = atomicAdd(&n_loud[d], __popc(big));
      if (rest) q0 = atomicAdd(&n_quiet[d], __popc(rest));
    }
    l0 = __shfl_sync(0xffffffffu, l0, 0);
    q0 = __shfl_sync(0xffffffffu, q0, 0);
    const unsigned before = (1u << lane) - 1u;
    if (listed) {
      const int at = r >= half ? l0 + __popc(big & before) : n_win - 1 - q0 - __popc(rest & before);
      (d ? pos1 : pos0)[at] = (int32_t)key_sample(key) - rb;
      (d ? rho1 : rho0)[at] = r;
    }
  };
  const unsigned long long *s0 = a.slots + p * a.n_win, *s1 = a.slots + (a.n_sel + p) * a.n_win;
  constexpr int U = 2;  // windows per thread and detector in flight
  for (int i0 = tid - lane; i0 < n_win; i0 += U * THREADS) {
    unsigned long long k0[U], k1[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int w = i0 + u * THREADS + lane;
      k0[u] = w < n_win ? __ldg(s0 + w) : 0ull;
      k1[u] = w < n_win ? __ldg(s1 + w) : 0ull;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      put(0, i0 + u * THREADS + lane, k0[u]);
      put(1, i0 + u * THREADS + lane, k1[u]);
    }
  }
  __syncthreads();
  const int loud0 = n_loud[0], loud1 = n_loud[1], all0 = loud0 + n_quiet[0], all1 = loud1 + n_quiet[1];
  if (loud0 + loud1 == 0 || all0 == 0 || all1 == 0) return;
  auto trig0 = [&](int i) { return i < loud0 ? i : n_win - 1 - (i - loud0); };
  auto trig1 = [&](int i) { return i < loud1 ? i : n_win - 1 - (i - loud1); };
  const int32_t tmpl = a.sel[p];
  const int32_t R = (int32_t)(a.ring_end - a.ring_begin), step = (int32_t)(a.shift % R), cw = (int32_t)a.coinc_window;
  bool follow = false;
  auto record = [&](int h, int l, int32_t k) {
    return CoincRec{tmpl,
                    k,
                    (int64_t)pos0[h] + rb,
                    (int64_t)pos1[l] + rb,
                    sqrtf(rho0[h]),
                    sqrtf(rho1[l]),
                    sqrtf(rho0[h] + rho1[l]),
                    0};
  };
  // Straight to the list, counted in the 64 bits of n_coinc: a pair at the shifts k0 .. k1
  auto emit_run = [&](int h, int l, int32_t k0, int32_t k1) {
    unsigned long long slot = atomicAdd(a.n_coinc, (unsigned long long)(k1 - k0 + 1));
    for (; k0 <= k1 && slot < (unsigned long long)a.coinc_cap; ++k0)
      reinterpret_cast<CoincRec*>(a.coincs)[slot++] = record(h, l, k0);
  };
  // A template can have more records than 32 bits count (2,048 windows of each detector, millions of shifts): the
  // collection's counter stops when it is full (each thread that saw it free may add one more)
  auto emit = [&](int h, int l, int32_t k, float rc2) {
    follow |= rc2 >= a.rho_c_thr2;
    if (!(rc2 >= a.rho_c_store2)) return;
    unsigned at = kTmplRec;
    if (*(volatile unsigned*)&n_found < (unsigned)kTmplRec) at = atomicAdd(&n_found, 1u);
    if (at < (unsigned)kTmplRec)
      found[at] = make_uint2((uint32_t)h | (uint32_t)l << 16, (uint32_t)k);
    else
      emit_run(h, l, k, k);
  };
  const uint32_t inv = step > 0 ? 0xffffffffu / (uint32_t)step : 0u;
  // the triggers h = first(i / n), l = trig1(i % n) of the pairs i < m n
  auto pairs = [&](int m, int n, auto first) {
    if (m == 0 || n == 0) return;
    const int32_t last = a.n_shifts * step;
    const int ja = THREADS / n, jb = THREADS - ja * n;
    int ia = tid / n, ib = tid - ia * n;
    for (int i0 = tid - lane; i0 < m * n; i0 += THREADS) {
      const bool in = i0 + lane < m * n;
      const int h = first(min(ia, m - 1)), l = trig1(ib);
      ib += jb;
      ia += ja + (ib >= n ? 1 : 0);
      ib -= ib >= n ? n : 0;
      const float rc2 = rho0[h] + rho1[l];
      const bool live = in && rc2 >= need;
      if (!__any_sync(0xffffffffu, live)) continue;
      int32_t D = pos0[h] - pos1[l];
      if (D < 0) D += R;
      if (step == 0) {  // all shifts or none
        if (live && (D <= cw || R - D <= cw)) {
          follow |= rc2 >= a.rho_c_thr2;
          if (rc2 >= a.rho_c_store2) emit_run(h, l, 0, a.n_shifts);
        }
        __syncwarp();
        continue;
      }
      int32_t x = D + cw;  // the shifts k with x - 2 cw <= k step <= x, turn by turn (last + 4 R fits)
      x -= x >= R ? R : 0;
      bool more = live && x - 2 * cw <= last;
      while (__any_sync(0xffffffffu, more))
        if (more) {
          uint32_t k = __umulhi((uint32_t)x, inv);  // x / step, or one less
          k += (k + 1) * (uint32_t)step <= (uint32_t)x ? 1 : 0;
          for (int32_t j = (int32_t)k; j >= 0 && j * step >= x - 2 * cw; --j)
            if (j <= a.n_shifts) emit(h, l, j, rc2);
          x += R;
          more = x - 2 * cw <= last;
        }
    }
  };
  int len = kWalkShifts;  // shifts that a thread walks at a time: fewer where there are threads for them
  while (len > 8 && all0 * (a.n_shifts / len + 1) < THREADS) len >>= 1;
  const int items = all0 * (a.n_shifts / len + 1), steps = min(len, a.n_shifts + 1);
  // What the two ways cost a thread, fitted to 3,907 calls by both (12 lengths with their windows and thresholds, 1 to 2,000
  // templates, up to 1,501 shifts): 1 for a pair, 1 for each of its turns of the ring if its SNRs suffice (half of those
  // with one quiet trigger, say), 2 for a shift of the walk and 2 for each window that it looks into beyond the first.
  // The way so chosen takes 0.8% longer than the better one in the mean, 2.4 times as long at worst.
  auto rounds = [](int64_t n) { return (n + THREADS - 1) / THREADS; };
  const int64_t loud2 = (int64_t)loud0 * loud1;
  const int64_t mixed = (int64_t)loud0 * all1 + (int64_t)all0 * loud1 - 2 * loud2;
  if (rounds(loud2 + mixed) + a.turns * rounds(loud2 + mixed / 2) <= rounds(items) * steps * a.walk_step) {
    pairs(loud0, all1, trig0);
    pairs(all0 - loud0, loud1, [&](int i) { return trig0(loud0 + i); });
  } else {
    uint16_t* at = reinterpret_cast<uint16_t*>(rho1 + n_win);  // detector-1 trigger of each window
    for (int w = tid; w < n_win; w += THREADS) at[w] = kNoTrigger;
    __syncthreads();
    auto window_of = [&](int32_t x) { return (int)(((uint64_t)(x + rb) * a.win_recip) >> kRecipBits); };
    for (int i = tid; i < all1; i += THREADS) {
      const int l = trig1(i);
      at[window_of(pos1[l])] = (uint16_t)l;
      atomicMax(&max1, __float_as_uint(rho1[l]));
    }
    __syncthreads();
    for (int i0 = tid - lane; i0 < items; i0 += THREADS) {
      const int i = min(i0 + lane, items - 1), kb = i / all0 * len, h = trig0(i % all0);
      const float r0 = rho0[h];
      const bool live = i0 + lane < items && r0 + __uint_as_float(max1) >= need;
      if (!__any_sync(0xffffffffu, live)) continue;
      int32_t x = pos0[h] - kb * step % R;  // ring position at shift kb
      if (x < 0) x += R;
      for (int32_t k = kb; k < kb + steps; ++k) {
        // windows that meet [lo, hi] in the ring
        auto look = [&](int32_t lo, int32_t hi) {
          const int end = window_of(hi);
          for (int w = window_of(lo); w <= end; ++w) {
            const int l = at[w];
            if (l != kNoTrigger && pos1[l] >= lo && pos1[l] <= hi) emit(h, l, k, r0 + rho1[l]);
          }
        };
        if (live && k <= a.n_shifts) {
          look(max(x - cw, 0), min(x + cw, R - 1));
          if (x < cw) look(x - cw + R, R - 1);
          else if (x + cw >= R) look(0, x + cw - R);
        }
        __syncwarp();
        x -= step;
        if (x < 0) x += R;
      }
    }
  }
  if (follow) a.followed[tmpl] = 1;
  __syncthreads();
  const int count = (int)min(n_found, (unsigned)kTmplRec);
  if (tid == 0 && count > 0) base = atomicAdd(a.n_coinc, (unsigned long long)count);
  __syncthreads();
  for (int i = tid; i < count; i += THREADS)
    if ((int64_t)base + i < a.coinc_cap)
      reinterpret_cast<CoincRec*>(a.coincs)[base + i] =
          record((int)(found[i].x & 0xffffu), (int)(found[i].x >> 16), (int32_t)found[i].y);
}

// --- coincidence records in order (tmpl, shift, sample0, sample1) ------------------
// Counting sort over the (tmpl, shift) bins, then each record's rank in its bin: a bin holds at most a few records
// per window, so the ranks are counted directly.  That is quadratic in a bin's records, which a selection that names a
// template many times multiplies: 394,000 records in 21 bins take 4.4 ms here and 37 ms on the host, where bins of more
// than kCoincCrowd are left to.

constexpr int kScanSpan = 4096;  // bins per scan CTA (1024 threads x 4)

__global__ void k_co_hist(const CoincRec* __restrict__ rec, int64_t n, int n_shift, int32_t* bins) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(bins + (int64_t)rec[i].tmpl * n_shift + rec[i].shift, 1);
}

// exclusive scan of v over the CTA's 1024 threads; *total = the sum
__device__ __forceinline__ int32_t cta_scan(int32_t v, int32_t* total) {
  __shared__ int32_t ws[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  if (w == 0) {
    int32_t s = ws[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    ws[lane] = s;
  }
  __syncthreads();
  *total = ws[31];
  const int32_t r = x - v + (w > 0 ? ws[w - 1] : 0);
  __syncthreads();
  return r;
}

// bins[i] becomes the sum of the CTA's bins before it, sums[block] their total
__global__ void __launch_bounds__(1024) k_co_scan(int32_t* bins, int64_t n_bins, int32_t* sums) {
  const int64_t i0 = (int64_t)blockIdx.x * kScanSpan + threadIdx.x * 4;
  int32_t v[4], s = 0, total;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    v[u] = i0 + u < n_bins ? bins[i0 + u] : 0;
    s += v[u];
  }
  int32_t x = cta_scan(s, &total);
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    if (i0 + u < n_bins) bins[i0 + u] = x;
    x += v[u];
  }
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) k_co_scan_sums(int32_t* sums, int n) {  // one CTA
  int32_t carry = 0;
  for (int b = 0; b < n; b += 1024) {
    const int i = b + threadIdx.x;
    int32_t total;
    const int32_t x = cta_scan(i < n ? sums[i] : 0, &total);
    if (i < n) sums[i] = carry + x;
    carry += total;
  }
}

struct CoincKey {
  unsigned long long key;  // (sample0, sample1)
  int32_t rec, bin;
};

// records grouped by bin, in any order; afterwards bins[b] (with its CTA's sum) is the end of bin b
__global__ void k_co_group(const CoincRec* __restrict__ rec, int64_t n, int n_shift, int32_t* bins,
                           const int32_t* __restrict__ sums, CoincKey* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const CoincRec r = rec[i];
    const int32_t b = r.tmpl * n_shift + r.shift;
    out[atomicAdd(bins + b, 1) + sums[b / kScanSpan]] =
        CoincKey{((unsigned long long)r.sample0 << 32) | (uint32_t)r.sample1, (int32_t)i, b};
  }
}

__global__ void k_co_rank(const CoincRec* __restrict__ rec, const CoincKey* __restrict__ grouped, int64_t n,
                          const int32_t* __restrict__ bins, const int32_t* __restrict__ sums,
                          CoincRec* __restrict__ out, int32_t* __restrict__ crowded) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const CoincKey k = grouped[i];
    const int32_t begin = k.bin > 0 ? bins[k.bin - 1] + sums[(k.bin - 1) / kScanSpan] : 0;
    const int32_t end = bins[k.bin] + sums[k.bin / kScanSpan];
    if (end - begin > kCoincCrowd) {
      *crowded = 1;
      continue;
    }
    int32_t rank = begin;
    for (int32_t j = begin; j < end; ++j) {
      const unsigned long long o = grouped[j].key;
      rank += o < k.key || (o == k.key && j < i) ? 1 : 0;
    }
    out[rank] = rec[k.rec];
  }
}

__global__ void k_zero_i32(int32_t* p, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    p[i] = 0;
}

__global__ void k_mark(const int64_t* __restrict__ ptr, const int32_t* __restrict__ idx, int64_t n_coarse,
                       const int32_t* __restrict__ followed, int32_t* flags, int64_t n_fine) {
  for (int64_t c = blockIdx.x; c < n_coarse; c += gridDim.x) {
    if (!followed[c]) continue;
    for (int64_t e = ptr[c] + threadIdx.x; e < ptr[c + 1]; e += blockDim.x) {
      const int32_t f = idx[e];
      if (f >= 0 && f < n_fine) flags[f] = 1;
    }
  }
}

constexpr int kFB = 1024;  // threads per flag-compaction block, one flag each

__global__ void k_flag_count(const int32_t* __restrict__ flags, int64_t n, int64_t* bc) {
  const int64_t i = (int64_t)blockIdx.x * kFB + threadIdx.x;
  const int has = (i < n && flags[i]) ? 1 : 0;
  const int c = __syncthreads_count(has);
  if (threadIdx.x == 0) bc[blockIdx.x] = c;
}

__global__ void k_flag_scan(int64_t* bc, int64_t nblk, int64_t* total) {
  // nblk is small (n_fine / 1024): one thread walks it
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    int64_t run = 0;
    for (int64_t b = 0; b < nblk; ++b) {
      const int64_t v = bc[b];
      bc[b] = run;
      run += v;
    }
    *total = run;
  }
}

__global__ void k_flag_write(const int32_t* __restrict__ flags, int64_t n, const int64_t* __restrict__ bc,
                             int32_t* out) {
  __shared__ int wc[32];
  const int64_t i = (int64_t)blockIdx.x * kFB + threadIdx.x;
  const bool has = i < n && flags[i];
  const unsigned m = __ballot_sync(0xffffffffu, has);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) wc[wid] = __popc(m);
  __syncthreads();
  if (threadIdx.x == 0) {
    int run = 0;
    for (int w = 0; w < 32; ++w) {
      const int v = wc[w];
      wc[w] = run;
      run += v;
    }
  }
  __syncthreads();
  if (has) out[bc[blockIdx.x] + wc[wid] + __popc(m & ((1u << lane) - 1u))] = (int32_t)i;
}

}  // namespace

cudaError_t launch_decimate(const float2* in, int64_t ld_in, float2* out, int64_t ld_out, int64_t nb_out, int n_det,
                            cudaStream_t st) {
  k_decimate<<<sms() * 4, 256, 0, st>>>(in, ld_in, out, ld_out, nb_out, n_det);
  add_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_coinc(const CoincArgs& a, float* max_rho2_det1, cudaStream_t st) {
  if (a.n_sel <= 0) return cudaSuccess;
  if (a.n_sel > 0x7fffffff) return cudaErrorInvalidValue;
  // up to kTmplWin windows (16 KB of triggers per detector) k_coinc_tmpl; beyond, where rows have analysed
  // ranges of their own (times outside the ring), and where a shift's time overflows, the walk over windows and shifts
  const int64_t R = a.ring_end - a.ring_begin;
  if (a.n_win <= kTmplWin && !a.own_ranges &&
      (int64_t)a.n_shifts * (a.shift % R) + 4 * R + a.coinc_window < (int64_t(1) << 30) && a.n_shifts < (1 << 22)) {
    CoincArgs t = a;
    t.win_recip = window_recip(a.window);
    t.turns = ((int64_t)a.n_shifts * (a.shift % R) + a.coinc_window) / R + 2;
    t.walk_step = 2 + 4 * a.coinc_window / a.window;
    // Threads: a thread per window for short rows (2,000 templates of 64 windows with 128 threads 7% faster than with 256);
    // for long ones 256 where the CTAs wait for SMs (1,024 windows 5% faster than with 512, 2,048 as fast), else up to 1,024.
    // Where there are fewer templates than SMs, several CTAs share a template's detector-0 triggers: one template of 1,024
    // windows over 501 shifts 315 us with one CTA, 41 us with 16 (k_coinc 213 us).
    const size_t smem = tmpl_smem(a.n_win);
    const bool many = a.n_sel > 2 * sms();
    const dim3 g((unsigned)a.n_sel, (unsigned)(a.n_sel < sms() ? std::min<int64_t>(kTmplSplit, sms() / a.n_sel) : 1));
    if (a.n_win <= 128)
      k_coinc_tmpl<128><<<g, 128, smem, st>>>(t);
    else if (a.n_win <= 512 || many)
      k_coinc_tmpl<256><<<g, 256, smem, st>>>(t);
    else if (a.n_win <= 1024 || a.n_sel > sms())
      k_coinc_tmpl<512><<<g, 512, smem, st>>>(t);
    else
      k_coinc_tmpl<1024><<<g, 1024, smem, st>>>(t);
    add_launches(1);
    return cudaGetLastError();
  }
  k_max_rho2<<<(unsigned)a.n_sel, 256, 0, st>>>(a.slots, a.n_sel, a.n_win, max_rho2_det1);
  CoincArgs b = a;
  b.max_rho2_det1 = max_rho2_det1;
  k_coinc<<<sms() * 8, 256, 0, st>>>(b);
  add_launches(2);
  return cudaGetLastError();
}

size_t coinc_order_bytes(int64_t n, int64_t n_bins) {
  const int64_t sums = (n_bins + kScanSpan - 1) / kScanSpan;
  return (size_t)n * sizeof(CoincKey) + (size_t)(n_bins + sums + 1) * sizeof(int32_t);
}

cudaError_t launch_coinc_order(const void* rec, int64_t n, int64_t n_tmpl, int n_shift, void* work, void* out,
                               int32_t** crowded, cudaStream_t st) {
  const int64_t n_bins = n_tmpl * n_shift, n_sums = (n_bins + kScanSpan - 1) / kScanSpan;
  CoincKey* grouped = static_cast<CoincKey*>(work);
  int32_t* bins = reinterpret_cast<int32_t*>(grouped + n);
  int32_t* flag = bins + n_bins;  // cleared with the bins
  int32_t* sums = flag + 1;
  *crowded = flag;
  const CoincRec* r = static_cast<const CoincRec*>(rec);
  cudaError_t e = cudaMemsetAsync(bins, 0, (size_t)(n_bins + 1) * sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  const unsigned g = (unsigned)((n + 255) / 256 < sms() * 8 ? (n + 255) / 256 : sms() * 8);
  k_co_hist<<<g, 256, 0, st>>>(r, n, n_shift, bins);
  k_co_scan<<<(unsigned)n_sums, 1024, 0, st>>>(bins, n_bins, sums);
  k_co_scan_sums<<<1, 1024, 0, st>>>(sums, (int)n_sums);
  k_co_group<<<g, 256, 0, st>>>(r, n, n_shift, bins, sums, grouped);
  k_co_rank<<<g, 256, 0, st>>>(r, grouped, n, bins, sums, static_cast<CoincRec*>(out), flag);
  add_launches(5);
  return cudaGetLastError();
}

cudaError_t launch_union(const int64_t* ptr, const int32_t* idx, int64_t n_coarse, const int32_t* followed,
                         int32_t* flags, int64_t n_fine, int32_t* subset, int64_t* n_subset, int64_t* bc,
                         cudaStream_t st) {
  const int g = sms() * 4;
  k_zero_i32<<<g, 256, 0, st>>>(flags, n_fine);
  if (n_coarse > 0) k_mark<<<g, 128, 0, st>>>(ptr, idx, n_coarse, followed, flags, n_fine);
  const int64_t nblk = (n_fine + kFB - 1) / kFB;
  if (nblk == 0) return cudaMemsetAsync(n_subset, 0, sizeof(int64_t), st);
  k_flag_count<<<(unsigned)nblk, kFB, 0, st>>>(flags, n_fine, bc);
  k_flag_scan<<<1, 32, 0, st>>>(bc, nblk, n_subset);
  k_flag_write<<<(unsigned)nblk, kFB, 0, st>>>(flags, n_fine, bc, subset);
  add_launches(n_coarse > 0 ? 5 : 4);
  return cudaGetLastError();
}

}  // namespace mf
