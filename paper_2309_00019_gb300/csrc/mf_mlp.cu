// Learned proposal network: training and inference kernels.
//
// A small MLP scores the neighbourhood slots of a stage-1 candidate so that
// stage 2 (Sec. III) can filter only the best-ranked fine templates, with the
// full neighbourhood as the fallback.  Layers: x -> depth x (affine + GELU)
// -> affine -> masked softmax over the candidate's n_valid slots.  Weights are
// kept in FP32 (master copy for AdamW) and cast to BF16 for the products;
// every matrix product runs on the tensor cores (mma.sync m16n8k16, BF16
// inputs, FP32 accumulation).  Parameter layout (flat, FP32): W_1 [n_in][width],
// b_1, ..., W_depth, b_depth, W_out [width][n_out], b_out.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "../../include/mf.h"
#include "mf_internal.h"

typedef __nv_bfloat16 bf16;

namespace {

// ---------------------------------------------------------------------------
// GEMM: acc[M][N] = op(A)[M][K] op(B)[K][N], BF16 inputs, FP32 accumulation.
//   A(m,k) = TA ? A[k lda + m] : A[m lda + k];  B(k,n) = TB ? B[n ldb + k] : B[k ldb + n]
//
// The network is small (a training step is 4.4 GFLOP in 14 products): what bounds it is latency, the launches and
// the chain of K steps of each product.  64 x 32 tiles give 128 CTAs for a 1,024 x 256 product; K steps of 64 come
// in through a three-stage cp.async pipeline in 16-byte pieces (every operand is an internal copy whose rows are
// padded with zeros to 8 elements), and ldmatrix forms the fragments of both orientations.  The products of the
// backward pass that wait for the same operand share a launch, and the bias, GELU and GELU' are the epilogue's.
// K runs in steps of 16 in order whatever the tiles, so the sums are those of the plain loop.  64 x 64 tiles with
// 2-byte loads and no overlap took 65 us per product, 904 us of a training step's 1,259 us at batch 1,024, width 256
// and 2,000 slots; as ten launches 87 us of 159 (153 with z read ahead).
// ---------------------------------------------------------------------------

constexpr int kTM = 64, kTN = 32, kTK = 64, kStages = 3;
constexpr int kABytes = kTM * kTK * 2, kBBytes = kTN * kTK * 2, kStage = kABytes + kBBytes;

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <bool TRANS>
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
  if constexpr (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

// 16 bytes global -> shared, zeros when !ok
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}

// byte offset of 16-byte piece c of row r in a tile with rows of 128 bytes (8 pieces) or 64 bytes (4 pieces):
// the pieces of a row are permuted so that ldmatrix's 8 rows fall into different banks
__device__ __forceinline__ uint32_t swz128(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }
__device__ __forceinline__ uint32_t swz64(int r, int c) { return (uint32_t)(r * 64 + ((c ^ ((r >> 1) & 3)) << 4)); }

// what becomes of acc: kStore: C = acc (+ bias); kGelu: C = z = acc + bias, out = GELU(z);
// kGeluGrad: C = out = acc GELU'(z), with z what C holds (a thread reads and writes its own elements)
enum Epi { kStore = 0, kGelu = 1, kGeluGrad = 2 };

struct Gemm {
  int M, N, K;
  const bf16 *A, *B;  // rows 16-byte aligned (lda, ldb multiples of 8), zeros from the last element to the next 8
  int lda, ldb;
  float* C;
  int ldc;
  const float* bias;
  int epi;
  bf16* out;          // kGelu, kGeluGrad
  int ldo;
  int tiles_n, tiles;
};

__device__ __forceinline__ float gelu(float z);
__device__ __forceinline__ float gelu_grad(float z);

template <bool TA, bool TB>
__device__ __forceinline__ void gemm_tile(const Gemm& g, int tile, unsigned char* sm) {
  const int m0 = tile / g.tiles_n * kTM, n0 = tile % g.tiles_n * kTN;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 16;
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm);
  const int steps = (g.K + kTK - 1) / kTK;
  auto load = [&](int step) {
    if (step < steps) {
      const uint32_t sa = base + step % kStages * kStage, sb = sa + kABytes;
      const int k0 = step * kTK;
#pragma unroll
      for (int i = 0; i < kTM * kTK / 8 / 128; ++i) {  // 64 rows (m, or k when TA) of 8 pieces
        const int c = tid + 128 * i, r = c >> 3, p = c & 7;
        const int m = TA ? m0 + p * 8 : m0 + r, k = TA ? k0 + r : k0 + p * 8;
        const bool ok = m < g.M && k < g.K;
        cp_async16(sa + swz128(r, p), ok ? g.A + (TA ? (int64_t)k * g.lda + m : (int64_t)m * g.lda + k) : g.A, ok);
      }
#pragma unroll
      for (int i = 0; i < kTN * kTK / 8 / 128; ++i) {  // 32 rows n of 8 pieces (TB), or 64 rows k of 4
        const int c = tid + 128 * i, r = TB ? c >> 3 : c >> 2, p = TB ? c & 7 : c & 3;
        const int n = TB ? n0 + r : n0 + p * 8, k = TB ? k0 + p * 8 : k0 + r;
        const bool ok = n < g.N && k < g.K;
        cp_async16(sb + (TB ? swz128(r, p) : swz64(r, p)),
                   ok ? g.B + (TB ? (int64_t)n * g.ldb + k : (int64_t)k * g.ldb + n) : g.B, ok);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[2][2][4] = {};
  const int gr = lane >> 2, tq = lane & 3;
  auto row_of = [&](int mi, int e) { return m0 + wm + mi * 16 + gr + 8 * (e >> 1); };
  auto col_of = [&](int ni, int e) { return n0 + wn + ni * 8 + tq * 2 + (e & 1); };
  // read ahead: between the stores to C the reads would wait for one another (the training step 166 us, 153 us so)
  float z[2][2][4] = {};
  if (g.epi == kGeluGrad) {
#pragma unroll
    for (int mi = 0; mi < 2; ++mi)
#pragma unroll
      for (int ni = 0; ni < 2; ++ni)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (row_of(mi, e) < g.M && col_of(ni, e) < g.N) z[mi][ni][e] = g.C[(int64_t)row_of(mi, e) * g.ldc + col_of(ni, e)];
  }
#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) load(s);
  for (int step = 0; step < steps; ++step) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();  // the step's tiles are visible, and everyone is done with the stage that is loaded next
    load(step + kStages - 1);
    const uint32_t sa = base + step % kStages * kStage, sb = sa + kABytes;
    const int i8 = lane >> 3, r8 = lane & 7;
#pragma unroll
    for (int ks = 0; ks < kTK; ks += 16) {
      uint32_t a[2][4], b[4];
#pragma unroll
      for (int mi = 0; mi < 2; ++mi) {
        const int m = wm + mi * 16;
        if constexpr (TA)
          ldmatrix4<true>(a[mi], sa + swz128(ks + (i8 >> 1) * 8 + r8, (m >> 3) + (i8 & 1)));
        else
          ldmatrix4<false>(a[mi], sa + swz128(m + (i8 & 1) * 8 + r8, (ks >> 3) + (i8 >> 1)));
      }
      if constexpr (TB)
        ldmatrix4<false>(b, sb + swz128(wn + (i8 >> 1) * 8 + r8, (ks >> 3) + (i8 & 1)));
      else
        ldmatrix4<true>(b, sb + swz64(ks + (i8 & 1) * 8 + r8, (wn >> 3) + (i8 >> 1)));
#pragma unroll
      for (int mi = 0; mi < 2; ++mi) {
        mma_bf16(acc[mi][0], a[mi], b[0], b[1]);
        mma_bf16(acc[mi][1], a[mi], b[2], b[3]);
      }
    }
  }
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int ni = 0; ni < 2; ++ni)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int r = row_of(mi, e), c = col_of(ni, e);
        if (r >= g.M || c >= g.N) continue;
        float v = acc[mi][ni][e] + (g.bias ? g.bias[c] : 0.f);
        const int64_t at = (int64_t)r * g.ldc + c;
        if (g.epi == kGeluGrad) v = v * gelu_grad(z[mi][ni][e]);
        g.C[at] = v;
        if (g.epi == kGelu) g.out[(int64_t)r * g.ldo + c] = __float2bfloat16(gelu(v));
        if (g.epi == kGeluGrad) g.out[(int64_t)r * g.ldo + c] = __float2bfloat16(v);
      }
}

// a layer's forward product
__global__ void __launch_bounds__(128) k_gemm_fwd(const __grid_constant__ Gemm g) {
  __shared__ __align__(128) unsigned char sm[kStages * kStage];
  gemm_tile<false, false>(g, blockIdx.x, sm);
}

// a layer's backward products: dW = H^T dZ, and (from block dw.tiles on) dH = dZ W^T
__global__ void __launch_bounds__(128) k_gemm_bwd(const __grid_constant__ Gemm dw, const __grid_constant__ Gemm dh) {
  __shared__ __align__(128) unsigned char sm[kStages * kStage];
  if ((int)blockIdx.x < dw.tiles) gemm_tile<true, false>(dw, blockIdx.x, sm);
  else gemm_tile<false, true>(dh, blockIdx.x - dw.tiles, sm);
}

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
  return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

// rows x [B][n] -> BF16 rows y [B][ld], zeros from n to ld; also clears the loss
__global__ void k_rows_bf16(const float* __restrict__ x, int n, bf16* __restrict__ y, int ld, int64_t B, float* loss) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *loss = 0.f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < B * ld; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / ld;
    const int c = (int)(i - r * ld);
    y[i] = __float2bfloat16(c < n ? x[r * n + c] : 0.f);
  }
}

// Where the flat parameter vector's weights lie in their BF16 copy: layer l's matrix [din][dout] starts at w and
// its bias at b of the vector; in the copy its rows start at p and are ld elements apart.
struct Layers {
  int n;
  uint32_t w[17], b[17], p[17];
  int dout[17], ld[17];
};

// the weight i of the vector into the copy (biases are not in it)
__device__ __forceinline__ void put_weight(const Layers& L, uint32_t i, float t, bf16* __restrict__ wb) {
  int l = 0;
  while (l + 1 < L.n && i >= L.w[l + 1]) ++l;
  if (i >= L.b[l]) return;
  const uint32_t k = i - L.w[l], r = k / (uint32_t)L.dout[l], c = k - r * (uint32_t)L.dout[l];
  wb[L.p[l] + r * (uint32_t)L.ld[l] + c] = __float2bfloat16(t);
}

__global__ void k_pack(const float* __restrict__ theta, int64_t n, const __grid_constant__ Layers L,
                       bf16* __restrict__ wb) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    put_weight(L, (uint32_t)i, theta[i], wb);
}

// masked softmax cross-entropy, one CTA per row: loss += -log p[label] / B,
// grad = (p - onehot) / B on the valid slots, 0 elsewhere
__global__ void k_masked_ce(const float* __restrict__ logits, int n_out, const int32_t* __restrict__ n_valid,
                            const int32_t* __restrict__ label, int B, float* loss, float* __restrict__ g,
                            bf16* __restrict__ gb, int ldb) {
  const int row = blockIdx.x;
  const float* l = logits + (int64_t)row * n_out;
  const int nv = min(max(n_valid[row], 1), n_out);
  __shared__ float red[32];
  float m = -INFINITY;
  for (int j = threadIdx.x; j < nv; j += blockDim.x) m = fmaxf(m, l[j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : -INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (threadIdx.x == 0) red[0] = v;
  }
  __syncthreads();
  m = red[0];
  __syncthreads();
  float s = 0.f;
  for (int j = threadIdx.x; j < nv; j += blockDim.x) s += expf(l[j] - m);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) red[0] = v;
  }
  __syncthreads();
  s = red[0];
  const int lab = label[row];
  const float invB = 1.f / (float)B;
  for (int j = threadIdx.x; j < n_out; j += blockDim.x) {
    float gv = 0.f;
    if (j < nv) gv = (expf(l[j] - m) / s - (j == lab ? 1.f : 0.f)) * invB;
    g[(int64_t)row * n_out + j] = gv;
    gb[(int64_t)row * ldb + j] = __float2bfloat16(gv);
  }
  if (threadIdx.x == 0 && lab >= 0 && lab < nv) atomicAdd(loss, -(l[lab] - m - logf(s)) * invB);
}

// bias gradients of every layer, db[c] = sum_b G[b][c]: a CTA takes 32 columns, its 8 warps every eighth row each
// (32 running sums per warp in one line), then the warps' sums in order
struct ColSums {
  const float* G[17];
  float* db[17];
  int cols[17];
};
__global__ void __launch_bounds__(256) k_colsums(const __grid_constant__ ColSums s, int rows) {
  __shared__ float part[8][32];
  const int l = blockIdx.y, cols = s.cols[l], lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + lane;
  if (blockIdx.x * 32 >= cols) return;
  float v = 0.f;
  if (c < cols) {
    const float* G = s.G[l] + c;
#pragma unroll 8
    for (int b = w; b < rows; b += 8) v += G[(int64_t)b * cols];
  }
  part[w][lane] = v;
  __syncthreads();
  if (w == 0 && c < cols) {
#pragma unroll
    for (int i = 1; i < 8; ++i) v += part[i][lane];
    s.db[l][c] = v;
  }
}

__global__ void k_adamw(float* __restrict__ th, const float* __restrict__ g, float* __restrict__ m,
                        float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps, float wd, float c1,
                        float c2, const __grid_constant__ Layers L, bf16* __restrict__ wb) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float t = th[i] - lr * ((mi / c1) / (sqrtf(vi / c2) + eps) + wd * th[i]);
    th[i] = t;
    put_weight(L, (uint32_t)i, t, wb);
  }
}

// Best-scored valid slots per row (ties to the lower slot), in order, until
// their softmax probability (over the valid slots) reaches p_mass or k slots
// are taken; -1 padding; count[row] = slots taken.
__global__ void k_topk(const float* __restrict__ logits, int n_out, const int32_t* __restrict__ n_valid, int k,
                       float p_mass, int32_t* __restrict__ out, int32_t* __restrict__ count) {
  const int row = blockIdx.x;
  const float* l = logits + (int64_t)row * n_out;
  const int nv = min(max(n_valid[row], 0), n_out);
  __shared__ int s_slot;
  __shared__ float s_best;
  __shared__ float bv[32];
  __shared__ int bi[32];
  __shared__ float s_max, s_sum, s_cum;
  __shared__ int s_done;
  // softmax normaliser over the valid slots
  float m = -INFINITY;
  for (int j = threadIdx.x; j < nv; j += blockDim.x) m = fmaxf(m, l[j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) bv[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    float mm = -INFINITY;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mm = fmaxf(mm, bv[w]);
    s_max = mm;
  }
  __syncthreads();
  float sum = 0.f;
  for (int j = threadIdx.x; j < nv; j += blockDim.x) sum += expf(l[j] - s_max);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) bv[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    float ss = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) ss += bv[w];
    s_sum = ss;
    s_cum = 0.f;
    s_done = 0;
  }
  __syncthreads();
  // Each thread keeps the best of its slots that are not chosen yet; a round takes the best of those, and only its
  // owner looks through its slots again, for the best one that comes after it in the order (score, then slot).
  float best = -INFINITY;
  int besti = 0x7fffffff;
  auto rescan = [&](float v, int at) {  // the best of the slots behind (v, at)
    best = -INFINITY;
    besti = 0x7fffffff;
    for (int j = threadIdx.x; j < nv; j += blockDim.x) {
      const float x = l[j];
      const bool behind = x < v || (x == v && j > at);
      if (behind && (x > best || (x == best && j < besti))) {
        best = x;
        besti = j;
      }
    }
  };
  rescan(INFINITY, -1);
  int taken = 0;
  for (int r = 0; r < k; ++r) {
    float b = best;
    int bj = besti;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ob = __shfl_xor_sync(0xffffffffu, b, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bj, o);
      if (ob > b || (ob == b && oi < bj)) {
        b = ob;
        bj = oi;
      }
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
      bv[threadIdx.x >> 5] = b;
      bi[threadIdx.x >> 5] = bj;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      b = -INFINITY;
      int ii = 0x7fffffff;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
        if (bv[w] > b || (bv[w] == b && bi[w] < ii)) {
          b = bv[w];
          ii = bi[w];
        }
      const bool ok = !s_done && r < nv && ii != 0x7fffffff;
      s_slot = ok ? ii : -1;
      s_best = b;
      out[(int64_t)row * k + r] = s_slot;
      if (ok) {
        s_cum += expf(b - s_max) / s_sum;
        if (s_cum >= p_mass) s_done = 1;
      }
    }
    __syncthreads();
    if (s_slot < 0) {  // nothing is left to take: the rest is padding
      for (int q = r + 1 + threadIdx.x; q < k; q += blockDim.x) out[(int64_t)row * k + q] = -1;
      break;
    }
    ++taken;
    if (besti == s_slot) rescan(s_best, s_slot);
  }
  if (threadIdx.x == 0 && count) count[row] = taken;
}

int sms() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

}  // namespace

struct mf_mlp_s {
  int n_in = 0, width = 0, depth = 0, n_out = 0;
  int64_t max_batch = 0, n_params = 0, step = 0;
  cudaStream_t st = nullptr;
  std::string err;
  std::vector<int64_t> w_off, b_off;  // offsets of W_l, b_l in the flat parameter vector
  float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
  Layers layers{};
  int ldx = 0, ldh = 0, ldo = 0;       // padded rows of the BF16 operands: input, activations, logit gradients
  bf16* wb = nullptr;                  // BF16 copy of the weights, padded rows (the products' operand)
  bf16* xb = nullptr;                  // input [B][ldx]
  std::vector<float*> z;               // pre-activations [B][width], l = 1..depth; after the backward pass, gradients
  std::vector<bf16*> h;                // activations [B][ldh]
  float* logits = nullptr;             // [B][n_out]
  float* dlog = nullptr;               // [B][n_out]
  bf16* dlogb = nullptr;               // [B][ldo]
  bf16* dzb[2] = {nullptr, nullptr};   // [B][ldh], of the layer at hand and the one below
  float* loss = nullptr;
};

namespace {

mf_status mfail(mf_mlp_t p, mf_status s, const std::string& m) {
  if (p) p->err = m;
  mf::set_global_error(m);
  return s;
}

template <class T>
bool dal(T** ptr, size_t n) {
  return cudaMalloc((void**)ptr, std::max<size_t>(n, 1) * sizeof(T)) == cudaSuccess;
}

int pad8(int n) { return (n + 7) / 8 * 8; }

Gemm product(int M, int N, int K, const bf16* A, int lda, const bf16* B, int ldb, float* C, int ldc,
             const float* bias = nullptr) {
  Gemm g{};
  g.M = M;
  g.N = N;
  g.K = K;
  g.A = A;
  g.lda = lda;
  g.B = B;
  g.ldb = ldb;
  g.C = C;
  g.ldc = ldc;
  g.bias = bias;
  g.tiles_n = (N + kTN - 1) / kTN;
  g.tiles = g.tiles_n * ((M + kTM - 1) / kTM);
  return g;
}

// forward of a batch of B rows whose input (FP32, device) is x; leaves logits in `logits`, clears the loss
cudaError_t forward(mf_mlp_t p, const float* x, int B, float* logits) {
  const int64_t total = (int64_t)B * p->ldx;
  k_rows_bf16<<<(unsigned)std::min<int64_t>((total + 255) / 256, sms() * 4), 256, 0, p->st>>>(x, p->n_in, p->xb, p->ldx,
                                                                                              B, p->loss);
  const bf16* hin = p->xb;
  int kin = p->n_in, ld = p->ldx;
  for (int l = 0; l <= p->depth; ++l) {
    const bool last = l == p->depth;
    const int dout = last ? p->n_out : p->width;
    Gemm g = product(B, dout, kin, hin, ld, p->wb + p->layers.p[l], p->layers.ld[l], last ? logits : p->z[l], dout,
                     p->theta + p->b_off[l]);
    if (!last) {
      g.epi = kGelu;
      g.out = p->h[l];
      g.ldo = p->ldh;
    }
    k_gemm_fwd<<<g.tiles, 128, 0, p->st>>>(g);
    if (!last) {
      hin = p->h[l];
      kin = p->width;
      ld = p->ldh;
    }
  }
  mf::add_launches(p->depth + 2);
  return cudaGetLastError();
}

}  // namespace

extern "C" {

mf_status mf_mlp_create(mf_mlp_t* out, int32_t n_in, int32_t width, int32_t depth, int32_t n_out, int64_t max_batch,
                        void* cuda_stream) {
  if (!out) return mfail(nullptr, MF_EINVAL, "mf_mlp_create: null out");
  if (n_in < 1 || n_in > 4096 || width < 1 || width > 8192 || depth < 1 || depth > 16 || n_out < 1 ||
      n_out > 65536 || max_batch < 1 || max_batch > (1 << 20))
    return mfail(nullptr, MF_EINVAL, "mf_mlp_create: sizes out of range");
  mf_mlp_t p = new (std::nothrow) mf_mlp_s();
  if (!p) return mfail(nullptr, MF_ENOMEM, "mf_mlp_create: host allocation");
  p->n_in = n_in;
  p->width = width;
  p->depth = depth;
  p->n_out = n_out;
  p->max_batch = max_batch;
  p->st = (cudaStream_t)cuda_stream;
  int64_t o = 0, din = n_in;
  for (int l = 0; l <= depth; ++l) {
    const int64_t dout = l < depth ? width : n_out;
    p->w_off.push_back(o);
    o += din * dout;
    p->b_off.push_back(o);
    o += dout;
    din = width;
  }
  p->n_params = o;
  p->ldx = pad8(n_in);
  p->ldh = pad8(width);
  p->ldo = pad8(n_out);
  Layers& L = p->layers;
  L.n = depth + 1;
  int64_t wn = 0;  // elements of the padded BF16 copy
  for (int l = 0; l <= depth; ++l) {
    L.w[l] = (uint32_t)p->w_off[l];
    L.b[l] = (uint32_t)p->b_off[l];
    L.p[l] = (uint32_t)wn;
    L.dout[l] = l < depth ? width : n_out;
    L.ld[l] = pad8(L.dout[l]);
    wn += (int64_t)(l == 0 ? n_in : width) * L.ld[l];
  }
  const int64_t B = max_batch;
  bool ok = dal(&p->theta, o) && dal(&p->grad, o) && dal(&p->m, o) && dal(&p->v, o) && dal(&p->wb, wn) &&
            dal(&p->xb, B * p->ldx) && dal(&p->logits, B * n_out) && dal(&p->dlog, B * n_out) &&
            dal(&p->dlogb, B * p->ldo) && dal(&p->dzb[0], B * p->ldh) && dal(&p->dzb[1], B * p->ldh) &&
            dal(&p->loss, 1);
  for (int l = 0; ok && l < depth; ++l) {
    float* zz = nullptr;
    bf16* hh = nullptr;
    ok = dal(&zz, B * width) && dal(&hh, B * p->ldh);
    p->z.push_back(zz);
    p->h.push_back(hh);
    if (ok) cudaMemsetAsync(hh, 0, B * p->ldh * sizeof(bf16), p->st);
  }
  if (!ok) {
    cudaGetLastError();
    mf_mlp_destroy(p);
    return mfail(nullptr, MF_ENOMEM, "mf_mlp_create: device allocation");
  }
  cudaMemsetAsync(p->theta, 0, o * sizeof(float), p->st);
  // the rows' padding stays zero: the kernels write valid elements only
  cudaMemsetAsync(p->wb, 0, wn * sizeof(bf16), p->st);
  cudaMemsetAsync(p->dlogb, 0, B * p->ldo * sizeof(bf16), p->st);
  for (bf16* q : p->dzb) cudaMemsetAsync(q, 0, B * p->ldh * sizeof(bf16), p->st);
  cudaMemsetAsync(p->m, 0, o * sizeof(float), p->st);
  cudaMemsetAsync(p->v, 0, o * sizeof(float), p->st);
  *out = p;
  return MF_OK;
}

void mf_mlp_destroy(mf_mlp_t p) {
  if (!p) return;
  if (p->st) cudaStreamSynchronize(p->st); else cudaDeviceSynchronize();
  for (void* q : {(void*)p->theta, (void*)p->grad, (void*)p->m, (void*)p->v, (void*)p->wb, (void*)p->xb,
                  (void*)p->logits, (void*)p->dlog, (void*)p->dlogb, (void*)p->dzb[0], (void*)p->dzb[1],
                  (void*)p->loss})
    if (q) cudaFree(q);
  for (auto* q : p->z) if (q) cudaFree(q);
  for (auto* q : p->h) if (q) cudaFree(q);
  delete p;
}

int64_t mf_mlp_num_params(mf_mlp_t p) { return p ? p->n_params : -1; }

mf_status mf_mlp_set_params(mf_mlp_t p, const float* theta, int64_t n, int on_device) {
  if (!p || !theta) return mfail(p, MF_EINVAL, "mf_mlp_set_params: null argument");
  if (n != p->n_params) return mfail(p, MF_EINVAL, "mf_mlp_set_params: n must equal mf_mlp_num_params");
  cudaError_t e = cudaMemcpyAsync(p->theta, theta, n * sizeof(float),
                                  on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, p->st);
  if (e == cudaSuccess) {
    k_pack<<<sms() * 4, 256, 0, p->st>>>(p->theta, n, p->layers, p->wb);
    mf::add_launches(1);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(p->m, 0, n * sizeof(float), p->st);
  if (e == cudaSuccess) e = cudaMemsetAsync(p->v, 0, n * sizeof(float), p->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(p->st);
  if (e != cudaSuccess) return mfail(p, MF_ECUDA, std::string("mf_mlp_set_params: ") + cudaGetErrorString(e));
  p->step = 0;
  return MF_OK;
}

mf_status mf_mlp_get_params(mf_mlp_t p, float* theta, int64_t n) {
  if (!p || !theta || n != p->n_params) return mfail(p, MF_EINVAL, "mf_mlp_get_params: bad argument");
  cudaError_t e = cudaMemcpyAsync(theta, p->theta, n * sizeof(float), cudaMemcpyDeviceToHost, p->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(p->st);
  if (e != cudaSuccess) return mfail(p, MF_ECUDA, std::string("mf_mlp_get_params: ") + cudaGetErrorString(e));
  return MF_OK;
}

mf_status mf_mlp_forward(mf_mlp_t p, const float* x, int64_t B, float* logits) {
  if (!p || !x) return mfail(p, MF_EINVAL, "mf_mlp_forward: null argument");
  if (B < 1 || B > p->max_batch) return mfail(p, MF_EINVAL, "mf_mlp_forward: batch out of range");
  cudaError_t e = forward(p, x, (int)B, logits ? logits : p->logits);
  if (e != cudaSuccess) return mfail(p, MF_ECUDA, std::string("mf_mlp_forward: ") + cudaGetErrorString(e));
  return MF_OK;
}

mf_status mf_mlp_loss_grad(mf_mlp_t p, const float* x, const int32_t* n_valid, const int32_t* label, int64_t B,
                           float* loss, float* grad) {
  if (!p || !x || !n_valid || !label) return mfail(p, MF_EINVAL, "mf_mlp_loss_grad: null argument");
  if (B < 1 || B > p->max_batch) return mfail(p, MF_EINVAL, "mf_mlp_loss_grad: batch out of range");
  const int Bi = (int)B, W = p->width, D = p->depth;
  cudaError_t e = forward(p, x, Bi, p->logits);
  if (e != cudaSuccess) return mfail(p, MF_ECUDA, std::string("mf_mlp_loss_grad: ") + cudaGetErrorString(e));
  k_masked_ce<<<Bi, 256, 0, p->st>>>(p->logits, p->n_out, n_valid, label, Bi, p->loss, p->dlog, p->dlogb, p->ldo);
  // layer l: dW from its input's activations and its own gradient, and the gradient of the layer below, which
  // waits for the same operand: one launch
  const bf16* dz = p->dlogb;
  int ldz = p->ldo;
  for (int l = D; l >= 0; --l) {
    const int dout = p->layers.dout[l], din = l > 0 ? W : p->n_in;
    Gemm dw = product(din, dout, Bi, l > 0 ? p->h[l - 1] : p->xb, l > 0 ? p->ldh : p->ldx, dz, ldz,
                      p->grad + p->w_off[l], dout);
    Gemm dh{};
    if (l > 0) {
      dh = product(Bi, W, dout, dz, ldz, p->wb + p->layers.p[l], p->layers.ld[l], p->z[l - 1], W);
      dh.epi = kGeluGrad;
      dh.out = p->dzb[l & 1];
      dh.ldo = p->ldh;
    }
    k_gemm_bwd<<<dw.tiles + dh.tiles, 128, 0, p->st>>>(dw, dh);
    dz = dh.out;
    ldz = p->ldh;
  }
  ColSums cs{};
  int wide = 0;
  for (int l = 0; l <= D; ++l) {
    cs.G[l] = l < D ? p->z[l] : p->dlog;
    cs.db[l] = p->grad + p->b_off[l];
    cs.cols[l] = p->layers.dout[l];
    wide = std::max(wide, cs.cols[l]);
  }
  k_colsums<<<dim3((unsigned)((wide + 31) / 32), (unsigned)(D + 1)), 256, 0, p->st>>>(cs, Bi);
  mf::add_launches(D + 3);
  e = cudaGetLastError();
  if (e == cudaSuccess && loss) e = cudaMemcpyAsync(loss, p->loss, sizeof(float), cudaMemcpyDeviceToDevice, p->st);
  if (e == cudaSuccess && grad)
    e = cudaMemcpyAsync(grad, p->grad, p->n_params * sizeof(float), cudaMemcpyDeviceToDevice, p->st);
  if (e != cudaSuccess) return mfail(p, MF_ECUDA, std::string("mf_mlp_loss_grad: ") + cudaGetErrorString(e));
  return MF_OK;
}

mf_status mf_mlp_adamw_step(mf_mlp_t p, float lr, float beta1, float beta2, float eps, float weight_decay) {
  if (!p) return mfail(p, MF_EINVAL, "mf_mlp_adamw_step: null plan");
  p->step += 1;
  const float c1 = 1.f - std::pow(beta1, (float)p->step), c2 = 1.f - std::pow(beta2, (float)p->step);
  k_adamw<<<sms() * 4, 256, 0, p->st>>>(p->theta, p->grad, p->m, p->v, p->n_params, lr, beta1, beta2, eps,
                                         weight_decay, c1, c2, p->layers, p->wb);
  mf::add_launches(1);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return mfail(p, MF_ECUDA, std::string("mf_mlp_adamw_step: ") + cudaGetErrorString(e));
  return MF_OK;
}

mf_status mf_mlp_topk(mf_mlp_t p, const float* x, const int32_t* n_valid, int64_t B, int32_t k, float p_mass,
                      int32_t* out, int32_t* count) {
  if (!p || !x || !n_valid || !out) return mfail(p, MF_EINVAL, "mf_mlp_topk: null argument");
  if (B < 1 || B > p->max_batch || k < 1 || k > 64) return mfail(p, MF_EINVAL, "mf_mlp_topk: bad batch or k");
  cudaError_t e = forward(p, x, (int)B, p->logits);
  if (e == cudaSuccess) {
    k_topk<<<(unsigned)B, 128, 0, p->st>>>(p->logits, p->n_out, n_valid, k, p_mass, out, count);
    mf::add_launches(1);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return mfail(p, MF_ECUDA, std::string("mf_mlp_topk: ") + cudaGetErrorString(e));
  return MF_OK;
}

const char* mf_mlp_last_error(mf_mlp_t p) { return p ? p->err.c_str() : ""; }

}  // extern "C"
