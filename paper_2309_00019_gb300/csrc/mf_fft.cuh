// Register-resident small DFTs and Stockham pass helpers for the matched-filter
// kernels (sm_103a).  Everything here computes inverse-sign transforms,
// X[q] = sum_r v[r] exp(+2 pi i r q / R), unnormalised, which is the sign of the
// correlation over coalescence time in Eq. (1)-(2) (Sec. V.C: one inverse FFT
// per template and segment).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

namespace mf {

// ---------------------------------------------------------------------------
// compile-time loops and constants
// ---------------------------------------------------------------------------

template <int... Is, class F>
__device__ __forceinline__ void sfor_impl(std::integer_sequence<int, Is...>, F&& f) {
  (f(std::integral_constant<int, Is>{}), ...);
}
// Calls f(std::integral_constant<int, i>) for i = 0..N-1 with compile-time i.
template <int N, class F>
__device__ __forceinline__ void sfor(F&& f) {
  sfor_impl(std::make_integer_sequence<int, N>{}, f);
}

// cos / sin of 2 pi e / R evaluated at compile time: argument reduced to
// [-pi/4, pi/4] by octant symmetry, then Taylor series to 1e-19.
__host__ __device__ constexpr double kpow_term(double x, int n) {
  double t = 1.0;
  for (int i = 1; i <= n; ++i) t *= x / i;
  return t;
}
__host__ __device__ constexpr double ksin_small(double x) {
  double s = 0.0;
  for (int n = 1, sg = 1; n < 30; n += 2, sg = -sg) s += sg * kpow_term(x, n);
  return s;
}
__host__ __device__ constexpr double kcos_small(double x) {
  double s = 0.0;
  for (int n = 0, sg = 1; n < 30; n += 2, sg = -sg) s += sg * kpow_term(x, n);
  return s;
}
// returns cos(2 pi e / R) (which = 0) or sin (which = 1)
__host__ __device__ constexpr double kcossin(long e, long R, int which) {
  const double kPi = 3.14159265358979323846264338327950288;
  e %= R;
  if (e < 0) e += R;
  // angle = 2 pi e / R = (pi/4) * (8e/R); octant o = floor(8e/R), remainder in [0, pi/4)
  long num = 8 * e;
  long o = num / R;
  double rem = (double)(num - o * R) / (double)R * (kPi / 4.0);  // [0, pi/4)
  double c = 0, s = 0;
  switch (o & 7) {
    case 0: c = kcos_small(rem); s = ksin_small(rem); break;
    case 1: c = ksin_small(kPi / 4 - rem); s = kcos_small(kPi / 4 - rem); break;
    case 2: c = -ksin_small(rem); s = kcos_small(rem); break;
    case 3: c = -kcos_small(kPi / 4 - rem); s = ksin_small(kPi / 4 - rem); break;
    case 4: c = -kcos_small(rem); s = -ksin_small(rem); break;
    case 5: c = -ksin_small(kPi / 4 - rem); s = -kcos_small(kPi / 4 - rem); break;
    case 6: c = ksin_small(rem); s = -kcos_small(rem); break;
    default: c = kcos_small(kPi / 4 - rem); s = -ksin_small(kPi / 4 - rem); break;
  }
  return which == 0 ? c : s;
}

// ---------------------------------------------------------------------------
// complex helpers (float2 = re, im)
// ---------------------------------------------------------------------------

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a * conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
__device__ __forceinline__ float2 mul_i(float2 a) { return make_float2(-a.y, a.x); }
__device__ __forceinline__ float2 mul_mi(float2 a) { return make_float2(a.y, -a.x); }

// a * exp(+2 pi i E / R) with E, R compile-time; trivial factors cost nothing.
template <long E, long R>
__device__ __forceinline__ float2 twiddle(float2 a) {
  constexpr long e = ((E % R) + R) % R;
  if constexpr (e == 0) {
    return a;
  } else if constexpr (4 * e == R) {
    return mul_i(a);
  } else if constexpr (2 * e == R) {
    return make_float2(-a.x, -a.y);
  } else if constexpr (4 * e == 3 * R) {
    return mul_mi(a);
  } else if constexpr (8 * e == R) {
    constexpr float h = 0.707106781186547524f;
    return make_float2(h * (a.x - a.y), h * (a.x + a.y));
  } else if constexpr (8 * e == 3 * R) {
    constexpr float h = 0.707106781186547524f;
    return make_float2(-h * (a.x + a.y), h * (a.x - a.y));
  } else if constexpr (8 * e == 5 * R) {
    constexpr float h = 0.707106781186547524f;
    return make_float2(h * (a.y - a.x), -h * (a.x + a.y));
  } else if constexpr (8 * e == 7 * R) {
    constexpr float h = 0.707106781186547524f;
    return make_float2(h * (a.x + a.y), h * (a.y - a.x));
  } else {
    constexpr float c = (float)kcossin(e, R, 0);
    constexpr float s = (float)kcossin(e, R, 1);
    return make_float2(fmaf(a.x, c, -a.y * s), fmaf(a.x, s, a.y * c));
  }
}

// ---------------------------------------------------------------------------
// in-register DFT of size R (inverse sign, natural order in and out).
// ZH: the upper half of the inputs (v[R/2..R-1]) is known to be zero.
// ---------------------------------------------------------------------------

template <int R, bool ZH = false>
struct Dft;

template <bool ZH>
struct Dft<1, ZH> {
  template <class V>
  __device__ __forceinline__ static void run(V& v, int o, int s) {}
};

template <bool ZH>
struct Dft<2, ZH> {
  // v[o], v[o+s]
  template <class V>
  __device__ __forceinline__ static void run(V& v, int o, int s) {
    if constexpr (ZH) {
      v[o + s] = v[o];
    } else {
      float2 a = v[o], b = v[o + s];
      v[o] = cadd(a, b);
      v[o + s] = csub(a, b);
    }
  }
};

template <bool ZH>
struct Dft<4, ZH> {
  template <class V>
  __device__ __forceinline__ static void run(V& v, int o, int s) {
    float2 x0 = v[o], x1 = v[o + s];
    if constexpr (ZH) {
      float2 ix1 = mul_i(x1);
      v[o] = cadd(x0, x1);
      v[o + s] = cadd(x0, ix1);
      v[o + 2 * s] = csub(x0, x1);
      v[o + 3 * s] = csub(x0, ix1);
    } else {
      float2 x2 = v[o + 2 * s], x3 = v[o + 3 * s];
      float2 t0 = cadd(x0, x2), t1 = csub(x0, x2);
      float2 t2 = cadd(x1, x3), t3 = mul_i(csub(x1, x3));
      v[o] = cadd(t0, t2);
      v[o + 2 * s] = csub(t0, t2);
      v[o + s] = cadd(t1, t3);
      v[o + 3 * s] = csub(t1, t3);
    }
  }
};

// Generic R = A * B in registers:
//   r = B r1 + r2, q = q1 + A q2:
//   X[q1 + A q2] = sum_r2 w_B^{r2 q2} w_R^{r2 q1} sum_r1 v[B r1 + r2] w_A^{r1 q1}
template <int R>
struct Split {
  static constexpr int A = (R >= 16) ? 4 : 2;
  static constexpr int B = R / A;
};

template <int R, bool ZH>
struct Dft {
  static constexpr int A = Split<R>::A;
  static constexpr int B = Split<R>::B;
  // operates on v[o + s*i], i = 0..R-1, with a local copy (registers)
  template <class V>
  __device__ __forceinline__ static void run(V& v, int o, int s) {
    float2 u[R];
#pragma unroll
    for (int i = 0; i < R; ++i) u[i] = v[o + s * i];
    // step 1: A-point DFTs over r1 for each r2 (stride B); upper half of r1 zero if ZH
    sfor<B>([&](auto r2c) {
      constexpr int r2 = decltype(r2c)::value;
      Dft<A, ZH>::run(u, r2, B);
    });
    // after step 1: u[r2 + B q1] holds U[r2][q1]; twiddle by w_R^{r2 q1}
    sfor<B>([&](auto r2c) {
      constexpr int r2 = decltype(r2c)::value;
      sfor<A>([&](auto q1c) {
        constexpr int q1 = decltype(q1c)::value;
        u[r2 + B * q1] = twiddle<(long)r2 * q1, R>(u[r2 + B * q1]);
      });
    });
    // step 2: B-point DFT over r2 for each q1: elements u[B q1 + r2], stride 1
    sfor<A>([&](auto q1c) {
      constexpr int q1 = decltype(q1c)::value;
      Dft<B, false>::run(u, B * q1, 1);
    });
    // u[B q1 + q2] = X[q1 + A q2]
#pragma unroll
    for (int q1 = 0; q1 < A; ++q1)
#pragma unroll
      for (int q2 = 0; q2 < B; ++q2) v[o + s * (q1 + A * q2)] = u[B * q1 + q2];
  }
};

template <int R, bool ZH = false>
__device__ __forceinline__ void dft(float2 (&v)[R]) {
  Dft<R, ZH>::run(v, 0, 1);
}

// ---------------------------------------------------------------------------
// The 32-point transform on register pairs.  Packed FP32 instructions (add, multiply, fused multiply-add on two
// adjacent registers) take the FMA pipe as long as two scalar ones but one issue slot.  The early butterfly stages,
// which do the same to neighbouring inputs, run packed over the inputs (i, i + 1); the last stage, whose operands are
// the two halves of a pair, runs scalar (a pair's halves are ordinary registers, so nothing is moved).  Real and
// imaginary parts are separate arrays; multiplications by +-i are a choice of array and sign.
// Every operation and its rounding is that of Dft<32>, where the compiler joins the factor sqrt(1/2) of an eighth root
// to the addition that follows: the factor is kept pending and joined by hand (fma), of two such terms the first.
// ---------------------------------------------------------------------------

constexpr float kSqrtHalf = 0.707106781186547524f;

__device__ __forceinline__ float2 at2(const float* x, int i) { return make_float2(x[i], x[i + 1]); }
__device__ __forceinline__ void put2(float* x, int i, float2 v) {
  x[i] = v.x;
  x[i + 1] = v.y;
}
__device__ __forceinline__ float2 padd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 psub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// 4-point DFT of the inputs i + s {0, 1, 2, 3} and, in the other lane, of the next ones, in place
template <bool ZH>
__device__ __forceinline__ void dft4_lanes(float* x, float* y, int i, int s) {
  const float2 x0 = at2(x, i), y0 = at2(y, i), x1 = at2(x, i + s), y1 = at2(y, i + s);
  float2 ax, ay, bx, by, cx, cy, dx, dy;  // t0, t1, t2 and x1 - x3
  if constexpr (ZH) {
    ax = bx = x0;
    ay = by = y0;
    cx = dx = x1;
    cy = dy = y1;
  } else {
    const float2 x2 = at2(x, i + 2 * s), y2 = at2(y, i + 2 * s), x3 = at2(x, i + 3 * s), y3 = at2(y, i + 3 * s);
    ax = padd(x0, x2);
    ay = padd(y0, y2);
    bx = psub(x0, x2);
    by = psub(y0, y2);
    cx = padd(x1, x3);
    cy = padd(y1, y3);
    dx = psub(x1, x3);
    dy = psub(y1, y3);
  }
  put2(x, i, padd(ax, cx));
  put2(y, i, padd(ay, cy));
  put2(x, i + 2 * s, psub(ax, cx));
  put2(y, i + 2 * s, psub(ay, cy));
  put2(x, i + s, psub(bx, dy));
  put2(y, i + s, padd(by, dx));
  put2(x, i + 3 * s, padd(bx, dy));
  put2(y, i + 3 * s, psub(by, dx));
}

// (x, y) times exp(2 pi i E / R); an eighth root leaves its factor sqrt(1/2) pending
template <int E, int R>
__device__ __forceinline__ void rotate(float& x, float& y) {
  static_assert(E >= 0 && 8 * E < 8 * R && 8 * E != 5 * R && 8 * E != 7 * R, "rotations of the splits used here");
  const float a = x, b = y;
  if constexpr (E == 0) {
  } else if constexpr (4 * E == R) {
    x = -b;
    y = a;
  } else if constexpr (8 * E == R) {
    x = a - b;
    y = a + b;
  } else if constexpr (8 * E == 3 * R) {
    x = -(a + b);
    y = a - b;
  } else {
    constexpr float c = (float)kcossin(E, R, 0), s = (float)kcossin(E, R, 1);
    x = fmaf(a, c, -b * s);
    y = fmaf(a, s, b * c);
  }
}

// 4-point DFT whose first sums t0, t2 and differences t1, d are formed already: out[o + st {0, 1, 2, 3}]
__device__ __forceinline__ void dft4_last(float2* out, int o, int st, float t0x, float t0y, float t1x, float t1y,
                                          float t2x, float t2y, float dx, float dy) {
  out[o] = make_float2(t0x + t2x, t0y + t2y);
  out[o + st] = make_float2(t1x - dy, t1y + dx);
  out[o + 2 * st] = make_float2(t0x - t2x, t0y - t2y);
  out[o + 3 * st] = make_float2(t1x + dy, t1y - dx);
}

// 8-point DFT of x[i .. i + 7] into out[o + 4 q].  PEND: bit r set where input r has sqrt(1/2) pending (input 4, or
// 2 and 6).
template <int PEND>
__device__ __forceinline__ void dft8_last(const float* x, const float* y, int i, float2* out, int o) {
  static_assert(PEND == 0 || PEND == (1 << 4) || PEND == ((1 << 2) | (1 << 6)), "pending inputs");
  float sx[4], sy[4], dx[4], dy[4];  // sums and differences of inputs r, r + 4
#pragma unroll
  for (int h = 0; h < 4; h += 2) {
    const float2 ax = at2(x, i + h), ay = at2(y, i + h);
    float2 bx = at2(x, i + h + 4), by = at2(y, i + h + 4);
    const float2 f = make_float2(kSqrtHalf, 1.f), g = make_float2(-kSqrtHalf, -1.f);
    if (PEND == (1 << 4) && h == 0) {
      put2(sx, h, __ffma2_rn(bx, f, ax));
      put2(sy, h, __ffma2_rn(by, f, ay));
      put2(dx, h, __ffma2_rn(bx, g, ax));
      put2(dy, h, __ffma2_rn(by, g, ay));
    } else if (PEND == ((1 << 2) | (1 << 6)) && h == 2) {
      bx.x *= kSqrtHalf;
      by.x *= kSqrtHalf;
      put2(sx, h, __ffma2_rn(ax, f, bx));
      put2(sy, h, __ffma2_rn(ay, f, by));
      put2(dx, h, __ffma2_rn(ax, f, make_float2(-bx.x, -bx.y)));
      put2(dy, h, __ffma2_rn(ay, f, make_float2(-by.x, -by.y)));
    } else {
      put2(sx, h, padd(ax, bx));
      put2(sy, h, padd(ay, by));
      put2(dx, h, psub(ax, bx));
      put2(dy, h, psub(ay, by));
    }
  }
  {
    const float2 tx = padd(at2(sx, 0), at2(sx, 2)), ty = padd(at2(sy, 0), at2(sy, 2));
    const float2 ux = psub(at2(sx, 0), at2(sx, 2)), uy = psub(at2(sy, 0), at2(sy, 2));
    dft4_last(out, o, 8, tx.x, ty.x, ux.x, uy.x, tx.y, ty.y, ux.y, uy.y);
  }
  {
    const float e1x = dx[1] - dy[1], e1y = dx[1] + dy[1];
    const float nx = -kSqrtHalf * (dx[3] + dy[3]), ny = kSqrtHalf * (dx[3] - dy[3]);
    dft4_last(out, o + 4, 8, dx[0] - dy[2], dy[0] + dx[2], dx[0] + dy[2], dy[0] - dx[2], fmaf(kSqrtHalf, e1x, nx),
              fmaf(kSqrtHalf, e1y, ny), fmaf(kSqrtHalf, e1x, -nx), fmaf(kSqrtHalf, e1y, -ny));
  }
}

// out[q] = sum_r (x[r] + i y[r]) exp(2 pi i r q / 32).  x, y are overwritten.  ZH: the inputs r >= 16 are zero (not
// read).
template <bool ZH>
__device__ __forceinline__ void dft_pairs(float (&x)[32], float (&y)[32], float2 (&out)[32]) {
  // r = 8 r1 + r2, q = q1 + 4 q2
#pragma unroll
  for (int i = 0; i < 8; i += 2) dft4_lanes<ZH>(x, y, i, 8);
  sfor<4>([&](auto q1c) {
    constexpr int q1 = decltype(q1c)::value;
    sfor<8>([&](auto r2c) {
      constexpr int r2 = decltype(r2c)::value;
      rotate<r2 * q1, 32>(x[8 * q1 + r2], y[8 * q1 + r2]);
    });
    constexpr int pend = q1 == 0 ? 0 : q1 == 2 ? (1 << 2) | (1 << 6) : 1 << 4;
    dft8_last<pend>(x, y, 8 * q1, out, q1);
  });
}

// exp(+2 pi i p / q) for integers 0 <= p < q <= 2^24, q a power of two.
__device__ __forceinline__ float2 unit_root(uint32_t p, uint32_t q) {
  float s, c;
  sincospif(2.0f * (float)p / (float)q, &s, &c);
  return make_float2(c, s);
}

// ---------------------------------------------------------------------------
// two-pass Stockham geometry of an M-point sub-FFT: radices (RA, RB), M = RA*RB,
// RA >= RB, T = RB threads.  Pass a: thread t reads x[t + r RB] (r < RA),
// writes shared[t RA + a].  Pass b: thread t does RA/RB butterflies
// j = t + T i; reads shared[j + r RA] (r < RB), twiddles by w_M^{r j}, and
// produces X[j + a RA] (a < RB).
// ---------------------------------------------------------------------------

template <int M>
struct Geo;
template <>
struct Geo<64> { static constexpr int RA = 8, RB = 8; };
template <>
struct Geo<128> { static constexpr int RA = 16, RB = 8; };
template <>
struct Geo<256> { static constexpr int RA = 16, RB = 16; };
template <>
struct Geo<512> { static constexpr int RA = 32, RB = 16; };
template <>
struct Geo<1024> { static constexpr int RA = 32, RB = 32; };

template <int M>
struct SubFft {
  static constexpr int RA = Geo<M>::RA;
  static constexpr int RB = Geo<M>::RB;
  static constexpr int T = RB;           // threads per sub-FFT
  static constexpr int NB = RA / RB;     // pass-b butterflies per thread
  static constexpr int PAD = M + M / RA; // padded shared length (one pad per RA entries)
  // padded shared index of logical index i
  __device__ __forceinline__ static int pidx(int i) { return i + i / RA; }
};

}  // namespace mf
