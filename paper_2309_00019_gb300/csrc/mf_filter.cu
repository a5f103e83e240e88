// TMA-staged matched-filter kernels (the hot path of Eq. 1-2 / Sec. V.C).
//
// N = N1 N2 four-step transform on sm_103a: CTAs of 128 computing threads, as
// many per SM as fit (k_cols16: 16 independent warps per SM), each a persistent
// loop over work items whose inputs are brought into shared memory by the
// bulk-copy (TMA) engine while the previous item computes.
//   k_cols: item = C columns k2 of one (template, detector) series, the
//           detector fastest in the item order.  The
//           template bank and the weighted data are stored column-major over
//           the non-zero half (element k = k1 N2 + k2, k1 < N1/2, at
//           k2 N1/2 + k1), so an item's two tiles are two contiguous 1-D bulk
//           copies.  The product x = q conj(h) is formed on the shared-memory
//           read; N1-point column transforms, each column owned by one group
//           of T threads inside a warp (its exchange needs only a warp
//           barrier); the four-step twiddle exp(+2 pi i j1 k2 / N); stores to
//           the scratch in panels of P = max(T(N1) / 2, RW(N2)) rows:
//           element (j1, k2) of a series at (j1 / P) N2 P + k2 P + j1 % P,
//           so that a warp's store covers whole 128-byte lines.
//   k_cols16: k_cols for the FP16 and FP16-pair intermediates of N = 2^20: a warp per column,
//           stored in image order by one tensor-map copy per column.
//   k_rows: item = RW rows j1 of one panel, brought in by a 3-D tensor-map
//           copy (RW of the panel's P values at each k2; one 1-D bulk copy
//           when RW = P); N2-point row transforms; rho^2 = |z|^2 / sigma^2 of
//           z[j1 + N1 j2], threshold and window maxima in registers.
// Sub-FFT twiddles come from a per-CTA shared table.  All mbarrier waits are
// bounded (see mf_tma.cuh) and report through the plan's status word.
// Programmatic dependent launch: each kernel lets the next one launch only
// when a CTA has finished all its items, so the next kernel's CTAs (which wait
// for this one to complete before touching the scratch) take the slots of
// retiring CTAs instead of competing with this kernel's own CTAs for them.
#include <algorithm>

#include "mf_common.cuh"
#include "mf_tma.cuh"

namespace mf {

namespace {

constexpr int kT2 = 128;  // threads per CTA

constexpr int round128(int x) { return (x + 127) / 128 * 128; }

// generic-proxy writes of another grid -> async-proxy (TMA) reads of this one
__device__ __forceinline__ void fence_proxy_async_global_fwd() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

// Padded exchange buffer of the row transforms: RW rows of M values, row
// stride S >= PAD with S = K (mod 16) so that 64-bit accesses of a half-warp
// (K lanes per row) hit 16 distinct bank pairs.
template <int M, int K>
struct Xch {
  using G = SubFft<M>;
  static constexpr int S = stride_for(G::PAD, K);
  __device__ __forceinline__ static int idx(int c, int i) { return c * S + G::pidx(i); }
};

// Column regions of k_cols: column c of an item owns S float2 of a slot,
// first its template tile then its weighted-data tile (N1/2 values each) and,
// once its threads hold those in registers, its exchange buffer.  Thread
// (c = tid / T, t = tid % T) writes logical t RA + q of column c in pass a
// and reads j + r RA (j = t + T i) in pass b.  S is the even candidate in
// [base, base + 32), base = max(tiles, PAD), with the fewest repeated 8-byte
// bank pairs over every half-warp of both patterns (half-warps span two
// columns when T = 8); even keeps every region 16-byte aligned for TMA.
template <int M, int C, int BASE>
struct ColStride {
  using G = SubFft<M>;
  static constexpr int RA = G::RA, RB = G::RB, T = G::T, NB = G::NB;
  static constexpr int conflicts(int S) {
    int total = 0;
    for (int hw = 0; hw < kT2 / 16; ++hw) {
      for (int q = 0; q < RA; ++q) {
        int cnt[16] = {};
        for (int l = 0; l < 16; ++l) {
          const int tid = hw * 16 + l, c = tid / T, t = tid % T;
          ++cnt[(c * S + t * RA + q + t) & 15];
        }
        for (int b = 0; b < 16; ++b) total += cnt[b] > 1 ? cnt[b] - 1 : 0;
      }
      for (int i = 0; i < NB; ++i)
        for (int r = 0; r < RB; ++r) {
          int cnt[16] = {};
          for (int l = 0; l < 16; ++l) {
            const int tid = hw * 16 + l, c = tid / T, j = tid % T + T * i;
            ++cnt[(c * S + j + r * RA + r) & 15];
          }
          for (int b = 0; b < 16; ++b) total += cnt[b] > 1 ? cnt[b] - 1 : 0;
        }
    }
    return total;
  }
  static constexpr int pick() {
    const int b0 = (BASE + 1) / 2 * 2;
    int best = b0, bc = conflicts(b0);
    for (int s = b0 + 2; s < b0 + 32; s += 2) {
      const int c = conflicts(s);
      if (c < bc) {
        bc = c;
        best = s;
      }
    }
    return best;
  }
  static constexpr int S = pick();
};

constexpr int kColConsumers = kT2;             // compute threads of k_cols (4 warps)
constexpr int kColThreads = kColConsumers + 32;  // plus one producer warp

// Shared-memory plan of k_cols: two slots of C column regions (ColStride),
// then the sub-FFT twiddles and the barriers full[2], empty[2], twiddles.
template <int N1, int BT, int QT>
struct ColGeo {
  using G = SubFft<N1>;
  static constexpr int T = G::T;                          // threads per column
  static constexpr int C = kColConsumers / T;             // columns per item
  static constexpr int R = N1 / 2;                        // non-zero half of k1
  static constexpr int HB = BT == kBankF32 ? 8 : 4;       // bytes per template element
  static constexpr int QB = QT == kBankF32 ? 8 : 4;       // bytes per weighted-data element
  static constexpr int H_COL = R * HB;                    // one column's template tile, bytes
  static constexpr int Q_COL = R * QB;
  static constexpr int TILES = (H_COL + Q_COL) / 8;
  static constexpr int S = ColStride<N1, C, (TILES > G::PAD ? TILES : G::PAD)>::S;
  static constexpr int SLOT = C * S * 8;
  static constexpr int TW_BYTES = G::RB * G::RA * 8;
  static constexpr int TW_OFF = 2 * SLOT;
  static constexpr int BAR_OFF = TW_OFF + round128(TW_BYTES);
  static constexpr int SMEM = BAR_OFF + 64;
};

template <int N2>
struct RowGeo {
  using G = SubFft<N2>;
  static constexpr int RW = kT2 / G::T;                   // rows per item (the scratch panel height)
  static constexpr int ITEM = RW * N2;                    // complex values per item
  static constexpr int K = 16 / RW;                       // threads of one row in a half-warp
  using X = Xch<N2, K>;
  static constexpr int XCH_BYTES = RW * X::S * 8;
  static constexpr int SLOT = round128(ITEM * 8 > XCH_BYTES ? ITEM * 8 : XCH_BYTES);
  static constexpr int TW_BYTES = G::RB * G::RA * 8;
  static constexpr int TW_OFF = 2 * SLOT;
  static constexpr int BAR_OFF = TW_OFF + round128(TW_BYTES);
  static constexpr int SMEM = BAR_OFF + 32;
};

// Panel height P of the pass-1 -> pass-2 scratch.  A pass-1 warp stores, per
// instruction, T(N1) consecutive j1 of 32 / T(N1) consecutive columns k2; with
// P >= T/2 those are whole 128-byte lines of at most two panels.  P is also a
// multiple of the rows of one pass-2 item (RW(N2)), which are contiguous when
// P = RW.
template <int N1, int N2>
struct ScratchGeo {
  static constexpr int RW = RowGeo<N2>::RW;
  static constexpr int HT = SubFft<N1>::T / 2;
  static constexpr int P = HT > RW ? HT : RW;
  static constexpr int BOXY = N2 < 256 ? N2 : 256;  // k2 per tensor-map box (256 at most)
  static_assert(P % RW == 0 && N1 % P == 0 && N2 % BOXY == 0, "scratch panel geometry");
};

template <int BT>
__device__ __forceinline__ float2 smem_h(const unsigned char* base, int idx) {
  if constexpr (BT == kBankF32) {
    return reinterpret_cast<const float2*>(base)[idx];
  } else if constexpr (BT == kBankF16) {
    return __half22float2(reinterpret_cast<const __half2*>(base)[idx]);
  } else {
    return __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(base)[idx]);
  }
}

// w_M^{r j}, j < RA fastest, r < RB, written to global memory once per plan
template <int M>
__global__ void k_fill_twiddles(float2* tw) {
  using G = SubFft<M>;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < G::RB * G::RA; i += gridDim.x * blockDim.x) {
    const int r = i / G::RA, j = i % G::RA;
    tw[i] = unit_root((uint32_t)((r * j) % M), (uint32_t)M);
  }
}

// ---------------------------------------------------------------------------
// pass 1
// ---------------------------------------------------------------------------

// MP: the series of several plans' parts (FilterParts), each with its own bank, data rows and selection
template <int N1, int N2, int BT, int QT, bool MP>
__global__ void __launch_bounds__(kColThreads, 3) k_cols(FilterArgs a, const __grid_constant__ FilterParts ps) {
  static_assert(!MP || QT == kBankF32, "fused launches take FP32 weighted data");
  using G = SubFft<N1>;
  using P = ColGeo<N1, BT, QT>;
  constexpr int RA = G::RA, RB = G::RB, T = G::T, NB = G::NB, C = P::C, R = P::R, S = P::S;
  constexpr int NCB = N2 / C;
  constexpr uint32_t N = (uint32_t)N1 * (uint32_t)N2;
  constexpr int PH = ScratchGeo<N1, N2>::P;  // scratch panel height
  extern __shared__ __align__(128) unsigned char sm[];
  const float2* tw = reinterpret_cast<const float2*>(sm + P::TW_OFF);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + P::BAR_OFF);  // [0], [1]: tiles of the slot landed
  uint64_t* empty = full + 2;                                     // [0], [1]: every warp done with the slot
  uint64_t* twb = full + 4;                                       // the twiddle table landed
  const int tid = threadIdx.x;
  const int n_items = (MP ? ps.n_series : a.count * a.n_det) * NCB;
  if (tid == 0) {
    mbar_init(full + 0, 1);
    mbar_init(full + 1, 1);
    mbar_init(empty + 0, kColConsumers / 32);
    mbar_init(empty + 1, kColConsumers / 32);
    mbar_init(twb, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (tid >= kColConsumers) {
    // producer warp: one lane issues every item's tiles into the slot its consumers released
    if (tid == kColConsumers) {
      const unsigned char* qbase = static_cast<const unsigned char*>(QT == kBankF32 ? (const void*)a.q : a.q_lp);
      mbar_expect_tx(twb, (uint32_t)P::TW_BYTES);
      bulk_g2s(sm + P::TW_OFF, a.tw1, (uint32_t)P::TW_BYTES, twb);
      // the weighted data come from the kernel just before only for the first batch; otherwise
      // the first tiles (bank and data, both unchanged) load while the previous kernel drains
      if (a.first_batch) {
        pdl_wait();
        fence_proxy_async_global_fwd();
      }
      int k = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < n_items; item += gridDim.x, ++k) {
        const int slot = k & 1;
        if (k >= 2 && !(ok = mbar_wait_bounded(empty + slot, (uint32_t)(((k >> 1) + 1) & 1), a.status))) break;
        fence_proxy_async();
        int li = item, nd = a.n_det;
        const int32_t* sel = a.sel;
        int64_t pos0 = a.pos0, ld_bank = a.ld_bank, ld_q = a.ld_q;
        const unsigned char *hb = static_cast<const unsigned char*>(a.bank), *qb = qbase;
        if constexpr (MP) {
          const FilterPart& p = ps.p[part_of(ps, item, NCB)];
          li = item - p.series0 * NCB;
          nd = p.n_det;
          sel = p.sel;
          pos0 = p.pos0;
          hb = static_cast<const unsigned char*>(p.bank);
          ld_bank = p.ld_bank;
          qb = reinterpret_cast<const unsigned char*>(p.q);
          ld_q = p.ld_q;
        }
        // detector fastest: the n_det items of one bank tile are issued back to back, so the
        // tile is read from HBM once and from L2 for the other detectors
        const int d = li % nd, cb = (li / nd) % NCB, b = li / (nd * NCB);
        const int64_t tmpl = sel[pos0 + b];
        unsigned char* dst = sm + slot * P::SLOT;
        mbar_expect_tx(full + slot, (uint32_t)(C * (P::H_COL + P::Q_COL)));
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const int64_t col = (int64_t)cb * C + c;
          // default L2 priority: the n_det - 1 later items of this tile read it from L2
          bulk_g2s(dst + c * S * 8, hb + (tmpl * ld_bank + col * R) * P::HB, (uint32_t)P::H_COL, full + slot);
          bulk_g2s(dst + c * S * 8 + P::H_COL, qb + ((int64_t)d * ld_q + col * R) * P::QB, (uint32_t)P::Q_COL,
                   full + slot);
        }
      }
      // the consumers' last items are done: then let the next kernel launch
      for (int m = k - 2; ok && m < k; ++m)
        if (m >= 0) ok = mbar_wait_bounded(empty + (m & 1), (uint32_t)((m >> 1) & 1), a.status);
      if (!ok) {
        // a wait gave up: before the CTA exits, wait (bounded again) for the copies this lane issued
        // that no consumer may have waited for (the twiddles and the last two items' tiles); no later
        // copy went into those slots, so their phases cannot have wrapped
        mbar_wait_bounded(twb, 0, nullptr);
        for (int m = k - 2; m < k; ++m)
          if (m >= 0) mbar_wait_bounded(full + (m & 1), (uint32_t)((m >> 1) & 1), nullptr);
      }
      pdl_launch_dependents();
    }
    return;
  }
  // consumer warps: column ca of every item, T threads per column
  const int ca = tid / T, ta = tid % T;
  pdl_wait();  // the previous kernel (reader of the scratch we are about to write) has completed
  if (!mbar_wait_bounded(twb, 0, a.status)) return;
  int k = 0;
  for (int item = blockIdx.x; item < n_items; item += gridDim.x, ++k) {
    const int slot = k & 1;
    if (!mbar_wait_bounded(full + slot, (uint32_t)((k >> 1) & 1), a.status)) break;
    const unsigned char* col = sm + slot * P::SLOT + ca * S * 8;
    int li = item, nd = a.n_det, s0 = 0;
    if constexpr (MP) {
      const FilterPart& p = ps.p[part_of(ps, item, NCB)];
      li = item - p.series0 * NCB;
      nd = p.n_det;
      s0 = p.series0;
    }
    const int s = s0 + (li / (nd * NCB)) * nd + li % nd;
    float2 v[RA];
#pragma unroll
    for (int r = 0; r < RA; ++r) {
      if (r >= RA / 2) {
        v[r] = make_float2(0.f, 0.f);
      } else {
        const int idx = ta + r * RB;  // k1 < N1/2
        v[r] = cmulc(smem_h<QT>(col + P::H_COL, idx), smem_h<BT>(col, idx));
      }
    }
    __syncwarp();  // the column's tiles are read: its region becomes the exchange buffer
    dft<RA, true>(v);
    float2* xb = reinterpret_cast<float2*>(sm + slot * P::SLOT) + ca * S;
#pragma unroll
    for (int q = 0; q < RA; ++q) xb[ta * RA + q + ta] = v[q];
    __syncwarp();
    float2* out = a.scratch + (int64_t)s * N;
    const int k2 = ((li / nd) % NCB) * C + ca;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int j = ta + T * i;
      float2 u[RB];
      u[0] = xb[j];
#pragma unroll
      for (int r = 1; r < RB; ++r) u[r] = cmul(xb[j + r * RA + r], tw[r * RA + j]);
      dft<RB>(u);
      // four-step twiddle w_N^{(j + q RA) k2} = w_N^{j k2} (w_N^{RA k2})^q; the table row of
      // column k2 holds w_N^{j k2} for j <= RA, so a warp's loads are contiguous
      const float2* twr = a.tw4 + (int64_t)k2 * (RA + 1);
      float2 w = __ldg(twr + j);
      const float2 st = __ldg(twr + RA);
      if constexpr (RA % PH == 0) {  // j1 = j + q RA: q RA / PH whole panels past j's
        float2* ob = out + (int64_t)(j / PH) * (N2 * PH) + k2 * PH + (j % PH);
#pragma unroll
        for (int q = 0; q < RB; ++q) {
          ob[(int64_t)q * (RA / PH) * (N2 * PH)] = cmul(u[q], w);
          if (q + 1 < RB) w = cmul(w, st);
        }
      } else {
#pragma unroll
        for (int q = 0; q < RB; ++q) {
          const int j1 = j + q * RA;
          out[(int64_t)(j1 / PH) * (N2 * PH) + k2 * PH + (j1 % PH)] = cmul(u[q], w);
          if (q + 1 < RB) w = cmul(w, st);
        }
      }
    }
    // this warp is done with the slot: order its shared accesses before the next bulk copy into it
    fence_proxy_async();
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(empty + slot);
  }
  pdl_launch_dependents();  // our items are done: the next kernel may launch
}

// ---------------------------------------------------------------------------
// pass 1 into the FP16 intermediate (N = 2^20)
// ---------------------------------------------------------------------------

// Read-only loads that stay where they are written (a load in front of a wait is not moved behind it)
__device__ __forceinline__ float2 ldg_early(const float2* p) {
  float2 v;
  asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ float ldg_early(const float* p) {
  float v;
  asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ int32_t ldg_early(const int32_t* p) {
  int32_t v;
  asm volatile("ld.global.nc.s32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

constexpr int kImgWarps = 16;  // warps of k_cols16, one column each
constexpr int kImgThreads = kImgWarps * 32;

// Shared-memory plan of k_cols16: per warp a template tile and an exchange buffer, then the sub-FFT twiddles and the
// barriers: per warp "tile landed", then the twiddles'.
template <int BT>
struct ImgGeo {
  using G = SubFft<1024>;
  static constexpr int R = 512;                           // non-zero half of k1
  static constexpr int HB = BT == kBankF32 ? 8 : 4;       // bytes per template element
  static constexpr int TILE = R * HB;                     // a column's template tile, bytes
  static constexpr int XCH = round128(G::PAD * 8);
  static constexpr int WARP = TILE + XCH;
  static constexpr int TW_BYTES = G::RB * G::RA * 8;
  static constexpr int TW_OFF = kImgWarps * WARP;
  static constexpr int BAR_OFF = TW_OFF + TW_BYTES;
  static constexpr int SMEM = BAR_OFF + (kImgWarps + 1) * 8;
};

// The column pass of k_cols for the FP16 intermediate of the tensor-core row pass: each series is scaled by
// series_scale16 of its template and written in panels of kPanel16 rows that are the row pass's stage-1 operand
// image: with k2 = 32 p + q, part c (0 real, 1 imaginary) of element (j1, k2) is the half at panel j1 / 8,
// ((q 32 + p) 2 + c) 8 + j1 % 8 (an image of 2 N2 8 halves), i.e. the MN-major layout of rows m = 8 q + j1 % 8 and
// columns k = 2 p + c.  IM = 2: each panel holds the image of hi = the value rounded to FP16, then the image of
// lo = the remainder rounded to FP16.  MP: the series of several plans' parts (FilterParts).
//
// What bounds it is issue and the shared-memory / L1 data path together, with too few warps to hide one behind the
// other.  So:
//  - one CTA of 16 warps per SM, each with a column at a time and no barrier between them, instead of 12 in CTAs of
//    four with a producer each.  There is room for them because only the template tile is staged (4 KB, copied in
//    while the column before it is transformed); the weighted data, which all templates share and which L2 holds, go
//    straight into registers during the second transform of the column before.
//  - a column's values are staged over its exchange buffer in image order and scattered to the panels by one
//    tensor-map store.  From registers, a shuffle and a four-line store per value made up a quarter of the wavefronts.
//  - the transforms run in packed FP32 (dft_pairs).
// Per launch of 121 series (two detectors, FP32 bank) 0.229 -> 0.210 ms; issue slots used 72 -> 78%, the L1 data path
// 81 -> 74%.  Two series per thread, everything packed, issued a third less (34 instead of 50 instructions per
// point) and was slower (0.219 ms): a packed multiply-add of three register pairs takes three cycles, not two.  The
// FP32 column pass gains nothing from this form (it writes twice the bytes, near the memory's rate): k_cols stays.
template <int BT, int IM, bool MP>
__global__ void __launch_bounds__(kImgThreads, 1) k_cols16(const __grid_constant__ CUtensorMap tm, FilterArgs a,
                                                            const __grid_constant__ FilterParts ps) {
  constexpr int N1 = 1024, N2 = 1024, PH = kPanel16;
  constexpr int IMG = IM == 2 ? 2 : 1;  // FP16 images per panel
  using G = SubFft<N1>;
  using P = ImgGeo<BT>;
  constexpr int RA = G::RA, RB = G::RB, R = P::R;
  static_assert(RA == 32 && RB == 32 && RA % PH == 0, "one column per warp, whole panels");
  extern __shared__ __align__(128) unsigned char sm[];
  const float2* tw = reinterpret_cast<const float2*>(sm + P::TW_OFF);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* tile = sm + warp * P::WARP;
  float2* xb = reinterpret_cast<float2*>(tile + P::TILE);
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + P::BAR_OFF) + warp;       // the warp's tile landed
  uint64_t* twb = reinterpret_cast<uint64_t*>(sm + P::BAR_OFF) + kImgWarps;   // the twiddle table landed
  const int n_items = (MP ? ps.n_series : a.count * a.n_det) * N2;
  const int stride = gridDim.x * kImgWarps;
  struct Item {
    int s, k2;            // series, column
    int tmpl;
    const void* h;        // the column's template tile
    const float2* q;      // this thread's first weighted value
    const float* ratio;   // of all templates
  };
  auto item_of = [&](int item) {
    int li = item, nd = a.n_det, s0 = 0;
    const int32_t* sel = a.sel;
    const float* isg = a.inv_sigma;
    int64_t pos0 = a.pos0, ld_bank = a.ld_bank, ld_q = a.ld_q;
    const void* hb = a.bank;
    const float2* qb = a.q;
    if constexpr (MP) {
      const FilterPart& p = ps.p[part_of(ps, item, N2)];
      li = item - p.series0 * N2;
      nd = p.n_det;
      s0 = p.series0;
      sel = p.sel;
      isg = p.inv_sigma;
      pos0 = p.pos0;
      hb = p.bank;
      ld_bank = p.ld_bank;
      qb = p.q;
      ld_q = p.ld_q;
    }
    // detector fastest: the n_det items of one bank tile run at the same time, so the tile is read from HBM once
    // and from L2 for the other detectors; then columns 32 apart (the same q, consecutive p), whose parts of a
    // panel share lines
    Item it;
    const int d = li % nd, cb = (li / nd) % N2, b = li / (nd * N2);
    it.k2 = ((cb / 128) * 4 + cb % 4) * 32 + cb / 4 % 32;
    it.s = s0 + b * nd + d;
    it.tmpl = ldg_early(sel + pos0 + b);
    it.h = static_cast<const unsigned char*>(hb) + ((int64_t)it.tmpl * ld_bank + (int64_t)it.k2 * R) * P::HB;
    it.q = qb + (int64_t)d * ld_q + (int64_t)it.k2 * R + lane;
    it.ratio = isg;
    return it;
  };
  auto fetch = [&](const Item& it) {  // lane 0: the item's template tile
    mbar_expect_tx(full, (uint32_t)P::TILE);
    bulk_g2s(tile, it.h, (uint32_t)P::TILE, full);
  };
  float2 qv[RA / 2];  // the item's weighted data
  auto load_q = [&](const Item& it) {
#pragma unroll
    for (int r = 0; r < RA / 2; ++r) qv[r] = ldg_early(it.q + r * RB);
  };
  if (lane == 0) mbar_init(full, 1);
  if (tid == 0) mbar_init(twb, 1);
  if (lane == 0) fence_mbar_init();
  __syncthreads();
  if (tid == 0) {
    mbar_expect_tx(twb, (uint32_t)P::TW_BYTES);
    bulk_g2s(sm + P::TW_OFF, a.tw1, (uint32_t)P::TW_BYTES, twb);
  }
  int item = blockIdx.x * kImgWarps + warp;
  Item it{};
  // the weighted data come from the kernel just before only for the first batch; otherwise the first item's inputs
  // (bank and data, both unchanged) load while the previous kernel drains
  if (a.first_batch) pdl_wait();
  if (item < n_items) {
    it = item_of(item);
    if (lane == 0) fetch(it);
    load_q(it);
  }
  if (!a.first_batch) pdl_wait();  // the previous kernel (reader of the scratch we are about to write) has completed
  bool ok = mbar_wait_bounded(twb, 0, a.status);
  int k = 0;
  for (; item < n_items; ++k) {
    const int s = it.s, k2 = it.k2;
    // the column's table entries and scale: their latency passes under the first transform
    const float2* twr = a.tw4 + (int64_t)k2 * (RA + 1);
    float2 w = ldg_early(twr + lane);
    const float2 st = ldg_early(twr + RA);
    const float ratio = ldg_early(it.ratio + it.tmpl);
    ok = __all_sync(0xffffffffu, ok && mbar_wait_bounded(full, (uint32_t)(k & 1), a.status));
    if (!ok) break;
    float2 v[RA];
    float vx[RA], vy[RA];
#pragma unroll
    for (int r = 0; r < RA / 2; ++r) {  // k1 = lane + 32 r < N1/2
      const float2 x = cmulc(qv[r], smem_h<BT>(tile, lane + r * RB));
      vx[r] = x.x;
      vy[r] = x.y;
    }
    // the tile is in registers: order its reads before the next copy into it
    fence_proxy_async();
    __syncwarp();
    item += stride;
    if (item < n_items) {
      it = item_of(item);
      if (lane == 0) fetch(it);
    }
    dft_pairs<true>(vx, vy, v);
    if (k > 0) {  // the previous column's store has long read the exchange buffer
      if (lane == 0) bulk_wait_read();
      __syncwarp();
    }
#pragma unroll
    for (int q = 0; q < RA; ++q) xb[lane * RA + q + lane] = v[q];
    __syncwarp();
    const float sc = series_scale16(ratio);  // (before the loads below: late, it held up the stores)
    float2 u[RB];
    float ux[RB], uy[RB];
    ux[0] = xb[lane].x;
    uy[0] = xb[lane].y;
#pragma unroll
    for (int r = 1; r < RB; ++r) {
      const float2 z = cmul(xb[lane + r * RA + r], tw[r * RA + lane]);
      ux[r] = z.x;
      uy[r] = z.y;
    }
    if (item < n_items) load_q(it);
    dft_pairs<false>(ux, uy, u);
    // four-step twiddle w_N^{(j + q RA) k2} = w_N^{j k2} (w_N^{RA k2})^q, j = lane; the table row of column k2
    // holds w_N^{j k2} for j <= RA, so a warp's loads are contiguous
    w.x *= sc;
    w.y *= sc;
    // every value of the exchange buffer is in registers: it becomes the stage, [image][panel][part][row]
    constexpr int IMAGE = N1 / PH * 2 * PH;  // halves of a column in one image
    static_assert(IMG * IMAGE * 2 <= P::XCH && P::WARP % 128 == 0 && P::TILE % 128 == 0, "image stage");
    __syncwarp();
    __half* stage = reinterpret_cast<__half*>(xb) + (lane / PH) * (2 * PH) + (lane % PH);
#pragma unroll
    for (int q = 0; q < RB; ++q) {
      const float2 z = cmul(u[q], w);
      const __half2 h = __float22half2_rn(z);
      __half* dq = stage + q * (RA / PH) * (2 * PH);
      dq[0] = __low2half(h);
      dq[PH] = __high2half(h);
      if constexpr (IM == 2) {  // the remainder: z - hi is exact in FP32
        const float2 hf = __half22float2(h);
        const __half2 l = __float22half2_rn(make_float2(z.x - hf.x, z.y - hf.y));
        dq[IMAGE] = __low2half(l);
        dq[IMAGE + PH] = __high2half(l);
      }
      if (q + 1 < RB) w = cmul(w, st);
    }
    fence_proxy_async();  // the stage is written: the store reads it through the async proxy
    __syncwarp();
    if (lane == 0) {
      tma_store_4d(&tm, xb, 0, s * (N1 / PH), (k2 & 31) * 32 + (k2 >> 5), 0);
      bulk_commit();
    }
  }
  if (!ok && lane == 0) {
    // a wait gave up: before the CTA exits, wait (bounded again) for the copies that may still be in flight
    if (tid == 0) mbar_wait_bounded(twb, 0, nullptr);
    if (item < n_items) mbar_wait_bounded(full, (uint32_t)(k & 1), nullptr);
  }
  if (lane == 0) bulk_wait_all();  // the stores are in global memory before this grid counts as complete
  pdl_launch_dependents();         // our items are done: the next kernel may launch
}

// ---------------------------------------------------------------------------
// pass 2
// ---------------------------------------------------------------------------

// tm: the scratch as [series * N1 / PH panels][N2][PH] of 8-byte values, box
// {RW, BOXY, 1} (unused when RW = PH: an item is then one contiguous panel)
// MP: the series of several plans' parts (FilterParts), each with its own epilogue state
template <int N1, int N2, bool MP>
__global__ void __launch_bounds__(kT2, 3) k_rows(const __grid_constant__ CUtensorMap tm, FilterArgs a,
                                                 const __grid_constant__ FilterParts ps) {
  using G = SubFft<N2>;
  using P = RowGeo<N2>;
  using X = typename P::X;
  using SG = ScratchGeo<N1, N2>;
  constexpr int RA = G::RA, RB = G::RB, T = G::T, NB = G::NB, RW = P::RW, PH = SG::P;
  constexpr int NRB = N1 / RW;
  constexpr int64_t N = (int64_t)N1 * N2;
  extern __shared__ __align__(128) unsigned char sm[];
  const float2* tw = reinterpret_cast<const float2*>(sm + P::TW_OFF);
  uint64_t* bar = reinterpret_cast<uint64_t*>(sm + P::BAR_OFF);
  const int tid = threadIdx.x;
  const int row = tid % RW, t = tid / RW;  // rows fastest: the panel is [k2][row]
  // series in reverse order: the last ones pass 1 wrote are the likeliest to be still in L2
  const int n_series = MP ? ps.n_series : a.count * a.n_det;
  const int n_items = n_series * NRB;
  if (tid == 0) {
    mbar_init(bar + 0, 1);
    mbar_init(bar + 1, 1);
    mbar_init(bar + 2, 1);
    fence_mbar_init();
  }
  __syncthreads();
  const uint64_t pol_last_use = policy_evict_first();
  auto issue = [&](int item, int slot) {
    const int s = n_series - 1 - item / NRB, j10 = (item % NRB) * RW;
    mbar_expect_tx(bar + slot, (uint32_t)(P::ITEM * 8));
    if constexpr (RW == PH) {
      bulk_g2s_hint(sm + slot * P::SLOT, a.scratch + (int64_t)s * N + (int64_t)j10 * N2, (uint32_t)(P::ITEM * 8),
                    bar + slot, pol_last_use);
    } else {
      // rows j10 .. j10 + RW - 1 of panel j10 / PH: RW * 8 bytes at each k2, landing as [k2][row]
      const int z = s * (N1 / PH) + j10 / PH;
#pragma unroll
      for (int y = 0; y < N2; y += SG::BOXY)
        tma_load_3d_hint(sm + slot * P::SLOT + (size_t)y * RW * 8, &tm, j10 % PH, y, z, bar + slot, pol_last_use);
    }
  };
  if (tid == 0) {
    mbar_expect_tx(bar + 2, (uint32_t)P::TW_BYTES);
    bulk_g2s(sm + P::TW_OFF, a.tw2, (uint32_t)P::TW_BYTES, bar + 2);
    pdl_wait();  // the scratch is written by the kernel just before
    fence_proxy_async_global_fwd();
    if ((int)blockIdx.x < n_items) issue(blockIdx.x, 0);
  }
  if (__syncthreads_or(!mbar_wait_bounded(bar + 2, 0, a.status))) {
    if (tid == 0) {  // drain (bounded) the copies issued above before the CTA exits
      mbar_wait_bounded(bar + 2, 0, nullptr);
      if ((int)blockIdx.x < n_items) mbar_wait_bounded(bar + 0, 0, nullptr);
    }
    return;
  }
  RawEpi ep{a.sel, a.inv_sigma, a.thr_raw, a.q_type == kBankF32 ? nullptr : a.dscale, a.pos0, a.n_det, a.win_recip,
            a.valid_begin, a.valid_end, a.n_win, a.n_sel_total, a.slots, a.row_valid};
  int k = 0;
  for (int item = blockIdx.x; item < n_items; item += gridDim.x, ++k) {
    const int slot = k & 1;
    const bool fail = !mbar_wait_bounded(bar + slot, (uint32_t)((k >> 1) & 1), a.status);
    const float2* stage = reinterpret_cast<const float2*>(sm + slot * P::SLOT);
    const int s = n_series - 1 - item / NRB;
    const int j1 = (item % NRB) * RW + row;
    float2 v[RA];
#pragma unroll
    for (int r = 0; r < RA; ++r) v[r] = stage[(t + r * RB) * RW + row];
    if (__syncthreads_or(fail)) {
      // the copy into this slot may still be in flight: wait for it (bounded) before the CTA exits;
      // nothing was issued into the other slot since its last wait completed
      if (tid == 0) mbar_wait_bounded(bar + slot, (uint32_t)((k >> 1) & 1), nullptr);
      return;
    }
    if (tid == 0 && item + (int)gridDim.x < n_items) {
      fence_proxy_async();
      issue(item + gridDim.x, slot ^ 1);
    }
    dft<RA>(v);
    float2* xb = reinterpret_cast<float2*>(sm + slot * P::SLOT);
#pragma unroll
    for (int q = 0; q < RA; ++q) xb[X::idx(row, t * RA + q)] = v[q];
    __syncthreads();
    RawEpi::Ser se;
    if constexpr (MP) {
      const FilterPart& p = ps.p[part_of(ps, s, 1)];
      const RawEpi pe{p.sel,           p.inv_sigma, p.thr_raw,     nullptr, p.pos0,   p.n_det,      a.win_recip,
                      p.valid_begin,   p.valid_end, a.n_win,       p.n_sel_total,     p.slots,      p.row_valid};
      se = pe.series(s - p.series0);
    } else {
      se = ep.series(s);
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int j = t + T * i;
      float2 u[RB];
      u[0] = xb[X::idx(row, j)];
#pragma unroll
      for (int r = 1; r < RB; ++r) u[r] = cmul(xb[X::idx(row, j + r * RA)], tw[r * RA + j]);
      dft<RB>(u);
      // eight samples at a time against the threshold: with a compare and a branch per sample the warps waited for
      // branches a fifth of their time (N = 2^20, 640 series: k_rows 1,264 -> 1,040 us; 512 points a row, 4,000
      // series, threshold 3.5: 2,510 -> 2,270 us)
#pragma unroll
      for (int q0 = 0; q0 < RB; q0 += 8) {
        float mx = 0.f;
#pragma unroll
        for (int q = q0; q < q0 + 8; ++q) mx = fmaxf(mx, fmaf(u[q].x, u[q].x, u[q].y * u[q].y));
        if (mx >= se.thr) {  // rare: some sample is over it
#pragma unroll
          for (int q = q0; q < q0 + 8; ++q) ep(se, (int64_t)j1 + (int64_t)N1 * (j + q * RA), u[q]);
        }
      }
    }
  }
  pdl_launch_dependents();  // our items are done: the next kernel may launch
}

template <class K>
cudaError_t set_smem2(K kern, int bytes) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

// launch with programmatic stream serialization (overlaps our prologue with the previous kernel's tail)
template <class K, class... Args>
cudaError_t launch_pdl(K kern, int grid, int block, int smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// CTAs of a persistent launch: as many as fit the chip at once.  Three per SM at N1, N2 >= 512 (their shared memory);
// shorter transforms need less of it, and up to seven hide each other's waits.
template <class K>
int resident_ctas(K kern, int threads, int smem) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, (size_t)smem) != cudaSuccess || per_sm < 3)
    per_sm = 3;
  return sm_count() * per_sm;
}

template <int N1, int N2, int BT, int QT, bool MP = false>
cudaError_t run_cols(const FilterArgs& a, const FilterParts& ps, cudaStream_t st) {
  using P = ColGeo<N1, BT, QT>;
  static_assert(P::SMEM * 3 <= 230400, "k_cols: three CTAs per SM must fit in shared memory");
  auto k = k_cols<N1, N2, BT, QT, MP>;
  static int resident = 0;
  if (resident == 0) {
    cudaError_t e = set_smem2(k, P::SMEM);
    if (e != cudaSuccess) return e;
    resident = resident_ctas(k, kColThreads, P::SMEM);
  }
  const int items = (MP ? ps.n_series : a.count * a.n_det) * (N2 / P::C);
  cudaError_t e = launch_pdl(k, std::min(items, resident), kColThreads, P::SMEM, st, a, ps);
  add_launches(1);
  return e;
}

template <int BT, int IM, bool MP>
cudaError_t run_cols16(const FilterArgs& a, const FilterParts& ps, const ScratchMaps& tm, cudaStream_t st) {
  using P = ImgGeo<BT>;
  static_assert(P::SMEM <= 232448, "k_cols16: shared memory");
  auto k = k_cols16<BT, IM, MP>;
  static bool attr = false;
  if (!attr) {
    cudaError_t e = set_smem2(k, P::SMEM);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  const int ctas = (MP ? ps.n_series : a.count * a.n_det) * (1024 / kImgWarps), g = sm_count();
  cudaError_t e = launch_pdl(k, ctas < g ? ctas : g, kImgThreads, P::SMEM, st, IM == 2 ? tm.h16x2 : tm.h16, a, ps);
  add_launches(1);
  return e;
}

// FP16 intermediates for the tensor-core row pass: FP32 data, any bank (fused launches: an FP32 bank)
template <int IM>
cudaError_t run_cols16_bt(const FilterArgs& a, const FilterParts& ps, const ScratchMaps& tm, cudaStream_t st) {
  if (a.q_type != kBankF32) return cudaErrorInvalidValue;
  if (ps.n > 0) return a.bank_type == kBankF32 ? run_cols16<kBankF32, IM, true>(a, ps, tm, st) : cudaErrorInvalidValue;
  switch (a.bank_type) {
    case kBankF32: return run_cols16<kBankF32, IM, false>(a, ps, tm, st);
    case kBankF16: return run_cols16<kBankF16, IM, false>(a, ps, tm, st);
    case kBankBF16: return run_cols16<kBankBF16, IM, false>(a, ps, tm, st);
  }
  return cudaErrorInvalidValue;
}

// (bank, data) storage pairs: FP32 data with any bank; 16-bit data with a bank of the same type.
// Fused launches (ps.n > 0): FP32 data, an FP32 bank.
template <int N1, int N2>
cudaError_t run_cols_bt(const FilterArgs& a, const FilterParts& ps, const ScratchMaps& tm, cudaStream_t st) {
  if (a.inter != 0) {
    if constexpr (N1 == 1024 && N2 == 1024) {
      if (a.inter == 1) return run_cols16_bt<1>(a, ps, tm, st);
      if (a.inter == 2) return run_cols16_bt<2>(a, ps, tm, st);
    }
    return cudaErrorInvalidValue;
  }
  if (ps.n > 0) {
    if (a.q_type != kBankF32 || a.bank_type != kBankF32) return cudaErrorInvalidValue;
    return run_cols<N1, N2, kBankF32, kBankF32, true>(a, ps, st);
  }
  if (a.q_type == kBankF32) {
    switch (a.bank_type) {
      case kBankF32: return run_cols<N1, N2, kBankF32, kBankF32>(a, ps, st);
      case kBankF16: return run_cols<N1, N2, kBankF16, kBankF32>(a, ps, st);
      case kBankBF16: return run_cols<N1, N2, kBankBF16, kBankF32>(a, ps, st);
    }
  } else if (a.q_type == a.bank_type) {
    switch (a.bank_type) {
      case kBankF16: return run_cols<N1, N2, kBankF16, kBankF16>(a, ps, st);
      case kBankBF16: return run_cols<N1, N2, kBankBF16, kBankBF16>(a, ps, st);
    }
  }
  return cudaErrorInvalidValue;
}

template <int N1, int N2, bool MP>
cudaError_t run_rows_mp(const FilterArgs& a, const FilterParts& ps, const CUtensorMap& tm, cudaStream_t st) {
  using P = RowGeo<N2>;
  static_assert(P::SMEM * 3 <= 230400, "k_rows: three CTAs per SM must fit in shared memory");
  auto k = k_rows<N1, N2, MP>;
  static int resident = 0;
  if (resident == 0) {
    cudaError_t e = set_smem2(k, P::SMEM);
    if (e != cudaSuccess) return e;
    resident = resident_ctas(k, kT2, P::SMEM);
  }
  const int items = (MP ? ps.n_series : a.count * a.n_det) * (N1 / P::RW);
  cudaError_t e = launch_pdl(k, std::min(items, resident), kT2, P::SMEM, st, tm, a, ps);
  add_launches(1);
  return e;
}

template <int N1, int N2>
cudaError_t run_rows(const FilterArgs& a, const FilterParts& ps, const CUtensorMap& tm, cudaStream_t st) {
  if (ps.n > 0) {
    if (a.q_type != kBankF32) return cudaErrorInvalidValue;
    return run_rows_mp<N1, N2, true>(a, ps, tm, st);
  }
  return run_rows_mp<N1, N2, false>(a, ps, tm, st);
}

// signature of the driver's cuTensorMapEncodeTiled (CUDA 12.0 ABI), fetched at run time
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    cudaDriverEntryPointQueryResult q;
    void* p = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// The FP16 operand image of the scratch (FilterArgs::inter = images) by columns: position pos = 32 (k2 % 32) +
// k2 / 32 of a panel holds the 2 x 8 halves of column k2; (half, panel, pos, image), a box is one column of a series.
cudaError_t encode_image(const float2* scratch, int64_t series, int n1, int n2, int images, CUtensorMap* m) {
  auto fn = encode_fn();
  if (!fn || !scratch || series < 1) return cudaErrorInvalidValue;
  const cuuint64_t run = 2 * kPanel16, image = run * (cuuint64_t)n2 * 2;  // halves of a column in a panel; bytes
  cuuint64_t dims[4] = {run, (cuuint64_t)(series * (n1 / kPanel16)), (cuuint64_t)n2, (cuuint64_t)images};
  cuuint64_t strides[3] = {image * images, run * 2, image};
  cuuint32_t box[4] = {(cuuint32_t)run, (cuuint32_t)(n1 / kPanel16), 1u, (cuuint32_t)images};
  cuuint32_t es[4] = {1u, 1u, 1u, 1u};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT16, 4, const_cast<float2*>(scratch), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int N1, int N2>
cudaError_t encode_scratch_of(const float2* scratch, int64_t series, ScratchMaps* m) {
  using SG = ScratchGeo<N1, N2>;
  *m = ScratchMaps{};
  if constexpr (N1 == 1024 && N2 == 1024) {
    cudaError_t e = encode_image(scratch, series, N1, N2, 1, &m->h16);
    if (e == cudaSuccess) e = encode_image(scratch, series, N1, N2, 2, &m->h16x2);
    if (e != cudaSuccess) return e;
  }
  if (SG::RW == SG::P) return cudaSuccess;  // contiguous row-pass items: no tensor map
  auto fn = encode_fn();
  if (!fn || !scratch || series < 1) return cudaErrorInvalidValue;
  cuuint64_t dims[3] = {(cuuint64_t)SG::P, (cuuint64_t)N2, (cuuint64_t)(series * (N1 / SG::P))};
  cuuint64_t strides[2] = {(cuuint64_t)SG::P * 8, (cuuint64_t)N2 * SG::P * 8};
  cuuint32_t box[3] = {(cuuint32_t)SG::RW, (cuuint32_t)SG::BOXY, 1u};
  cuuint32_t es[3] = {1u, 1u, 1u};
  CUresult r = fn(&m->rows, CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, const_cast<float2*>(scratch), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

#define MF_DISPATCH2(n, FN, ARGS)            \
  switch (n) {                               \
    case 1 << 12: return FN<64, 64> ARGS;    \
    case 1 << 13: return FN<128, 64> ARGS;   \
    case 1 << 14: return FN<128, 128> ARGS;  \
    case 1 << 15: return FN<256, 128> ARGS;  \
    case 1 << 16: return FN<256, 256> ARGS;  \
    case 1 << 17: return FN<512, 256> ARGS;  \
    case 1 << 18: return FN<512, 512> ARGS;  \
    case 1 << 19: return FN<1024, 512> ARGS; \
    case 1 << 20: return FN<1024, 1024> ARGS;\
  }                                          \
  return cudaErrorInvalidValue;

template <int N1, int N2>
cudaError_t run_fill_tw(float2* tw1, float2* tw2, cudaStream_t st) {
  k_fill_twiddles<N1><<<4, 256, 0, st>>>(tw1);
  k_fill_twiddles<N2><<<4, 256, 0, st>>>(tw2);
  add_launches(2);
  return cudaGetLastError();
}

// four-step twiddles by column: tw4[k2 (ra + 1) + j] = w_N^{j k2}, j <= ra, k2 < n2
__global__ void k_fill_tw4(float2* tw4, int n2, int ra, uint32_t n) {
  const int64_t count = (int64_t)n2 * (ra + 1);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t k2 = (uint32_t)(i / (ra + 1)), j = (uint32_t)(i % (ra + 1));
    tw4[i] = unit_root((j * k2) % n, n);
  }
}

template <int N1, int N2>
cudaError_t run_fill_tw4(float2* tw4, cudaStream_t st) {
  k_fill_tw4<<<64, 256, 0, st>>>(tw4, N2, SubFft<N1>::RA, (uint32_t)N1 * (uint32_t)N2);
  add_launches(1);
  return cudaGetLastError();
}

template <int N1, int N2>
cudaError_t tw4_count_of(int64_t* c) {
  *c = (int64_t)N2 * (SubFft<N1>::RA + 1);
  return cudaSuccess;
}

}  // namespace

namespace {

const FilterParts kOnePlan{};  // n = 0: every per-series field from FilterArgs

cudaError_t pass1_parts(const FilterArgs& a, const FilterParts& ps, const ScratchMaps& tm, cudaStream_t st) {
  MF_DISPATCH2(a.n, run_cols_bt, (a, ps, tm, st))
}

cudaError_t pass2_parts(const FilterArgs& a, const FilterParts& ps, const ScratchMaps& tm, cudaStream_t st) {
  if (a.inter != 0) return launch_filter2_pass2_tc(a, st, ps.n > 0 ? &ps : nullptr);
  MF_DISPATCH2(a.n, run_rows, (a, ps, tm.rows, st))
}

}  // namespace

cudaError_t launch_filter2_pass1(const FilterArgs& a, const ScratchMaps& tm, cudaStream_t st) {
  return pass1_parts(a, kOnePlan, tm, st);
}

cudaError_t launch_filter2_pass2(const FilterArgs& a, const ScratchMaps& tm, cudaStream_t st) {
  return pass2_parts(a, kOnePlan, tm, st);
}

cudaError_t launch_filter2_fused(const FilterArgs& a, const FilterParts& ps, const ScratchMaps& tm, cudaStream_t st,
                                 cudaEvent_t between) {
  if (ps.n < 1 || ps.n > kMaxParts || ps.n_series < 1) return cudaErrorInvalidValue;
  cudaError_t e = pass1_parts(a, ps, tm, st);
  if (e == cudaSuccess && between) e = cudaEventRecord(between, st);
  if (e == cudaSuccess) e = pass2_parts(a, ps, tm, st);
  return e;
}

cudaError_t encode_scratch_maps(int64_t n, const float2* scratch, int64_t series, ScratchMaps* m) {
  MF_DISPATCH2(n, encode_scratch_of, (scratch, series, m))
}

cudaError_t launch_fill_tw4(int64_t n, float2* tw4, cudaStream_t st) { MF_DISPATCH2(n, run_fill_tw4, (tw4, st)) }

int64_t tw4_count(int64_t n) {
  int64_t c = 0;
  auto f = [&]() -> cudaError_t { MF_DISPATCH2(n, tw4_count_of, (&c)) };
  return f() == cudaSuccess ? c : 0;
}

cudaError_t launch_fill_twiddles(int64_t n, float2* tw1, float2* tw2, cudaStream_t st) {
  MF_DISPATCH2(n, run_fill_tw, (tw1, tw2, st))
}

}  // namespace mf
