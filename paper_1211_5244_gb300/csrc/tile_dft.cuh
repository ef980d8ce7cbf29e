// Compile-time DFTs of any length up to 32 held in registers, FP32 and FP64,
// for the tile kernels (tile_pass.cuh).
//
//   dft<R, DIR, MASK>(x)   x[k] <- sum_r x[r] exp(DIR 2 pi i r k / R), natural
//       order; inputs r whose bit is missing from MASK are zero and are not read
//       (the zero padding of §3), outputs the caller does not read are removed by
//       the compiler (the compaction of §3)
//   dft_pre<R, DIR>(x, tw, e, NR)   the same of x[r] W_N^{e r}, N = R NR (conjugated
//       for DIR = +1); tw[j] holds W_N^j as (cos, tan) (tan_pair)
//
// Powers of two run as radix-2 layers whose butterfly a +- w b takes six FMAs
// (u = (1 + i tan) b two, a +- cos u four; Linzer and Feig's form of the product) instead of
// four for the product and four adds: on GB300 the FP64 pipe (two lanes per
// clock and SM) bounds every FP64 pass, and FP32 passes are bound by issue, so
// the operation count is the time. Its rounding error is that of two roundings at
// the sums, less than the product's and the adds' three. (The other six-operation form,
// a - w b = 2 a - (a + w b), rounds half of the outputs once more: the error of a
// transform grows by a sixth.) A twiddle in front of the transform folds
// into the same layers: layer m applies W_N^{(R/m)(e + K NR)} = W^{e R/m} W_m^K,
// R - 1 table entries as for separate products. A 16-point transform behind
// twiddles takes 192 operations that way against 228 (168 + 15 products of 4).
// Coprime factors (6, 10, 12, 14, 15, ...) combine without twiddles
// (Good-Thomas index maps, resolved at compile time); odd primes use the
// symmetric pairs x_k +- x_{p-k}.
#pragma once

#include <utility>

#include "common.cuh"

namespace ps {
namespace tile {

// ------------------------------------------------------------ constants

// Values to twice the double's bits (hi + lo), so that the constants and the step tables
// (tan_twiddle_kernel) are the rounded true values: a Taylor sum in double is off by
// up to an ulp, and a quotient of two such values by two. `Op` gives the error of a product and
// operations that are not contracted into FMAs: Dekker's at compile time, the device's
// rounded intrinsics in a kernel.
struct ConstOp {
  static __host__ __device__ constexpr double add(double a, double b) { return a + b; }
  static __host__ __device__ constexpr double mul(double a, double b) { return a * b; }
  static __host__ __device__ constexpr double split(double a) { return 134217729.0 * a - (134217729.0 * a - a); }
  static __host__ __device__ constexpr double mul_err(double a, double b) {
    const double ah = split(a), al = a - ah, bh = split(b), bl = b - bh;
    return ((ah * bh - a * b) + ah * bl + al * bh) + al * bl;
  }
};
struct DeviceOp {
#ifdef __CUDA_ARCH__
  static __host__ __device__ double add(double a, double b) { return __dadd_rn(a, b); }
  static __host__ __device__ double mul(double a, double b) { return __dmul_rn(a, b); }
  static __host__ __device__ double mul_err(double a, double b) { return __fma_rn(a, b, -__dmul_rn(a, b)); }
#else
  static __host__ __device__ double add(double a, double b) { return a + b; }
  static __host__ __device__ double mul(double a, double b) { return a * b; }
  static __host__ __device__ double mul_err(double a, double b) { return ConstOp::mul_err(a, b); }
#endif
};
struct Wide { double hi, lo; };
template <class Op>
struct WideOps {
  static __host__ __device__ constexpr Wide sum(double a, double b) {  // |a| >= |b|
    const double s = Op::add(a, b);
    return {s, Op::add(b, -Op::add(s, -a))};
  }
  static __host__ __device__ constexpr Wide mul(Wide a, Wide b) {
    const double p = Op::mul(a.hi, b.hi);
    return sum(p, Op::add(Op::mul_err(a.hi, b.hi), Op::add(Op::mul(a.hi, b.lo), Op::mul(a.lo, b.hi))));
  }
  static __host__ __device__ constexpr Wide div(Wide a, double d) {
    const double q = a.hi / d;
    const double r = Op::add(Op::add(Op::add(a.hi, -Op::mul(q, d)), -Op::mul_err(q, d)), a.lo);
    return sum(q, r / d);
  }
  // 1 - y / (K (K + 1)) (1 - y / ((K + 2)(K + 3)) (1 - ...)), the Taylor sum of cos sqrt(y) (K = 1)
  // or sin sqrt(y) / sqrt(y) (K = 2) from its term J on: below 1e-24 past J = K + 20 for
  // y <= (pi/4)^2, and from J = K + 8 on, where a term's error counts for less than 1e-5 of
  // itself, in plain doubles
  template <int K, int J = K>
  static __host__ __device__ constexpr Wide series(Wide y) {
    if constexpr (J > K + 20) {
      return {1.0, 0.0};
    } else if constexpr (J >= K + 8) {
      return {Op::add(1.0, -Op::mul(Op::mul(y.hi, 1.0 / (J * (J + 1))), series<K, J + 2>(y).hi)), 0.0};
    } else {
      constexpr Wide r = WideOps<ConstOp>::div(Wide{1.0, 0.0}, (double)(J * (J + 1)));
      const Wide t = mul(mul(y, r), series<K, J + 2>(y)), s = sum(1.0, -t.hi);
      return sum(s.hi, Op::add(s.lo, -t.lo));
    }
  }
  // cos(2 pi m / N), reduced exactly in integers to an angle of at most pi/4
  static __host__ __device__ constexpr Wide cos_turn(long m, long N) {
    m = ((m % N) + N) % N;
    long p = 4 * m;            // angle = 2 pi p / (4 N)
    if (p > 2 * N) p = 4 * N - p;
    const bool neg = p > N;
    if (neg) p = 2 * N - p;    // 0 .. pi/2
    const bool sine = 2 * p > N;
    const Wide half_pi = {1.57079632679489655800, 6.12323399573676603587e-17};
    const Wide x = div(mul(half_pi, Wide{(double)(sine ? N - p : p), 0.0}), (double)N);
    const Wide y = mul(x, x);
    const Wide v = sine ? mul(x, series<2>(y)) : series<1>(y);
    return neg ? Wide{-v.hi, -v.lo} : v;
  }
  static __host__ __device__ constexpr Wide sin_turn(long m, long N) { return cos_turn(4 * m - N, 4 * N); }
};
constexpr double cos_turn(long m, long N) { return WideOps<ConstOp>::cos_turn(m, N).hi; }
constexpr double sin_turn(long m, long N) { return cos_turn(4 * m - N, 4 * N); }
// sin(2 pi m / N) / d
constexpr double sin_over(long m, long N, double d) { return WideOps<ConstOp>::div(WideOps<ConstOp>::sin_turn(m, N), d).hi; }
constexpr double cos_over(long m, long N, double d) { return sin_over(4 * m + N, 4 * N, d); }
// the error of a product a b in place of sin(2 pi m / N), and of cos
constexpr double sin_err(long m, long N, double a, double b) {
  const Wide v = WideOps<ConstOp>::sin_turn(m, N);
  return ((v.hi - a * b) - ConstOp::mul_err(a, b)) + v.lo;
}
constexpr double cos_err(long m, long N, double a, double b) { return sin_err(4 * m + N, 4 * N, a, b); }
constexpr double square(double v) { return v * v; }

// exp(-2 pi i j / N), each part rounded once
template <typename T>
__device__ inline cpx<T> turn(long j, long N) {
  if constexpr (sizeof(T) == 4) {
    double s, c;
    sincospi(2.0 * (double)j / (double)N, &s, &c);
    return mk((T)c, (T)(-s));
  } else {
    return mk(WideOps<DeviceOp>::cos_turn(j, N).hi, -WideOps<DeviceOp>::sin_turn(j, N).hi);
  }
}
// W_N^j = exp(-2 pi i j / N) as (c, t), W = c (1 + i t): the form of the tables behind dft_pre (see bfly_w,
// mul_t). t is of the rounded c, so that c t is the sine to one rounding; where the cosine
// is 0 a c far below the type's last bit of 1 stands for it (its product with t overflows for
// FP32 values from 2^100 on, FP64 from 2^964).
template <typename T>
__device__ inline cpx<T> tan_pair(int j, int N) {
  const bool zero = 4 * j == N || 4 * j == 3 * N;
  if constexpr (sizeof(T) == 4) {
    double s, co;
    sincospi(2.0 * j / N, &s, &co);
    const T c = zero ? T(1.0 / (1 << 28)) : (T)co;
    return mk(c, (T)(-s / (double)c));
  } else {
    const T c = zero ? T(1.0 / (1ll << 60)) : WideOps<DeviceOp>::cos_turn(j, N).hi;
    return mk(c, WideOps<DeviceOp>::div(WideOps<DeviceOp>::sin_turn(-j, N), c).hi);
  }
}

constexpr int gcd_(int a, int b) { return b == 0 ? a : gcd_(b, a % b); }
constexpr int inv_mod(int a, int m) {  // a^{-1} mod m for coprime a, m
  for (int x = 1; x < m; ++x)
    if ((a * x) % m == 1) return x;
  return 1;
}
constexpr int low_prime(int n) {
  for (int p = 2; p * p <= n; ++p)
    if (n % p == 0) return p;
  return n;
}
// the full power of n's lowest prime that divides n
constexpr int low_part(int n) {
  const int p = low_prime(n);
  int a = 1;
  while (n % p == 0) { n /= p; a *= p; }
  return a;
}
constexpr int bitrev(int i, int n) {
  int r = 0;
  for (int b = 1; b < n; b <<= 1, i >>= 1) r = 2 * r + (i & 1);
  return r;
}
using Mask = unsigned long long;
constexpr Mask full_mask(int n) { return n >= 64 ? ~0ull : (1ull << n) - 1; }
// the mask of y[i] = x[(start + step i) mod n], i < count
constexpr Mask pick_mask(Mask m, int n, int start, int step, int count) {
  Mask r = 0;
  for (int i = 0; i < count; ++i)
    if ((m >> ((start + step * i) % n)) & 1) r |= 1ull << i;
  return r;
}
// the columns y_c[i] = x[(scol c + step i) mod n], c < cols, that hold an input
constexpr Mask columns_mask(Mask m, int n, int scol, int step, int count, int cols) {
  Mask r = 0;
  for (int c = 0; c < cols; ++c)
    if (pick_mask(m, n, scol * c, step, count) != 0) r |= 1ull << c;
  return r;
}
// bit-reversed positions [start, start + len) of an n-point transform hold no input
constexpr bool empty_block(Mask m, int n, int start, int len) {
  for (int i = start; i < start + len; ++i)
    if ((m >> bitrev(i, n)) & 1) return false;
  return true;
}

// ------------------------------------------------------------ arithmetic

template <int... I, class F>
__device__ __forceinline__ void sfor_(std::integer_sequence<int, I...>, F&& f) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void sfor(F&& f) {
  sfor_(std::make_integer_sequence<int, N>{}, f);
}

__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }

// exp(2 pi i K / M) as c (1 + i tc) and as i s (1 - i ts)
template <class S, int M, int K>
struct TurnForms {
  static constexpr S c = (S)cos_turn(K, M), tc = (S)sin_over(K, M, (double)c);
  static constexpr S s = (S)sin_turn(K, M), ts = (S)cos_over(K, M, (double)s);
  static constexpr bool cos_out =
      square(cos_err(K, M, (double)c, 1.0)) + square(sin_err(K, M, (double)c, (double)tc)) <=
      square(cos_err(K, M, (double)s, (double)ts)) + square(sin_err(K, M, (double)s, 1.0));
};
// (a, b) <- (a + w b, a - w b), w = c (1 + i t)
template <class C, class S>
__device__ __forceinline__ void bfly_w(C& a, C& b, S c, S t) {
  const C u = mk(mad(-t, b.y, b.x), mad(t, b.x, b.y));
  b = mk(mad(-c, u.x, a.x), mad(-c, u.y, a.y));
  a = mk(mad(c, u.x, a.x), mad(c, u.y, a.y));
}
// constexpr |v|
constexpr double mag(double v) { return v < 0 ? -v : v; }
// the same for the constant w = exp(DIR 2 pi i K / M), 0 <= K < M / 2
template <int M, int K, int DIR, class C>
__device__ __forceinline__ void bfly_c(C& a, C& b) {
  using S = decltype(a.x);
  if constexpr (K == 0) {
    const C t = a;
    a = cadd(t, b);
    b = csub(t, b);
  } else if constexpr (4 * K == M) {
    const C t = a, u = cmul_i<DIR>(b);
    a = cadd(t, u);
    b = csub(t, u);
  } else {
    // cos or sin outside, whichever leaves the smaller error of the rounded constants (it adds up
    // over the steps, and over a transform and its inverse)
    using F = TurnForms<S, M, K>;
    if constexpr (F::cos_out) {
      bfly_w(a, b, F::c, DIR * F::tc);
    } else {
      constexpr S o = DIR * F::s, t = DIR * F::ts;  // w b = i o (1 - i t) b
      const C u = mk(mad(t, b.x, -b.y), mad(t, b.y, b.x));
      b = mk(mad(-o, u.x, a.x), mad(-o, u.y, a.y));
      a = mk(mad(o, u.x, a.x), mad(o, u.y, a.y));
    }
  }
}
// v exp(DIR 2 pi i K / M)
template <int M, int K, int DIR, class C>
__device__ __forceinline__ C mul_c(C v) {
  using S = decltype(v.x);
  if constexpr (K % M == 0) {
    return v;
  } else {
    constexpr S wr = (S)cos_turn(K, M), wi = (S)(DIR * sin_turn(K, M));
    return mk(mad(-wi, v.y, wr * v.x), mad(wi, v.x, wr * v.y));
  }
}
// v w, or v conj(w) for DIR = +1
template <int DIR, class C>
__device__ __forceinline__ C mul_w(C v, C w) {
  return DIR < 0 ? mk(mad(-w.y, v.y, w.x * v.x), mad(w.y, v.x, w.x * v.y))
                 : mk(mad(w.y, v.y, w.x * v.x), mad(-w.y, v.x, w.x * v.y));
}
// the same for w = (c, t) = c (1 + i t), the form of the step tables (tan_pair)
template <int DIR, class C>
__device__ __forceinline__ C mul_t(C v, C w) {
  return DIR < 0 ? mk(w.x * mad(-w.y, v.y, v.x), w.x * mad(w.y, v.x, v.y))
                 : mk(w.x * mad(w.y, v.y, v.x), w.x * mad(-w.y, v.x, v.y));
}

// ------------------------------------------------------------ transforms

// powers of two: radix-2 decimation in time, layer by layer on bit-reversed inputs
template <int R, int DIR, Mask MASK, int FROM, class C>
__device__ __forceinline__ void pow2_layers(C (&y)[R]) {  // layers of blocks of FROM .. R points
  auto layer = [&](auto mc) {
    constexpr int m = mc;
    sfor<R / m>([&](auto blk) {
      constexpr int base = blk * m;
      constexpr bool za = empty_block(MASK, R, base, m / 2), zb = empty_block(MASK, R, base + m / 2, m / 2);
      sfor<m / 2>([&](auto Kc) {
        constexpr int K = Kc, p = base + K, q = p + m / 2;
        if constexpr (zb) {
          if constexpr (!za) y[q] = y[p];
        } else if constexpr (za) {
          y[p] = mul_c<m, K, DIR>(y[q]);
          y[q] = mk(-y[p].x, -y[p].y);
        } else {
          bfly_c<m, K, DIR>(y[p], y[q]);
        }
      });
    });
  };
  if constexpr (FROM <= 2 && R >= 2) layer(std::integral_constant<int, 2>{});
  if constexpr (FROM <= 4 && R >= 4) layer(std::integral_constant<int, 4>{});
  if constexpr (R >= 8) layer(std::integral_constant<int, 8>{});
  if constexpr (R >= 16) layer(std::integral_constant<int, 16>{});
  if constexpr (R >= 32) layer(std::integral_constant<int, 32>{});
}
template <int R, int DIR, Mask MASK, class C>
__device__ __forceinline__ void dft_pow2(C (&x)[R]) {
  C y[R];
  sfor<R>([&](auto i) { y[bitrev(i, R)] = x[i]; });
  pow2_layers<R, DIR, MASK, 2>(y);
  sfor<R>([&](auto i) { x[i] = y[i]; });
}

// odd primes: y_m, y_{p-m} = t_m +- DIR i u_m with t_m = x_0 + sum_k cos(2 pi m k / p) a_k,
// u_m = sum_k sin(2 pi m k / p) b_k, a_k, b_k = x_k +- x_{p-k}, k = 1 .. (p-1)/2. One of the sines
// stays outside the sum: y_m, y_{p-m} = t_m +- DIR i s (u_m / s) as two FMAs per component, an
// operation less than adding u_m (5 points: 32 operations instead of 36).
// Which sine stays outside: sin(2 pi J / P) up to its sign, J the choice whose rounded constants come closest to
// the transform's. Measured on E, the error of the matrix S of the sines: its own norm, and that of
// S E + (S E)^T, what a transform and its inverse make of it.
template <class S, int P>
struct SineOut {
  static constexpr int H = (P - 1) / 2;
  // index 1 .. H and sign of sin(2 pi i / P)
  static constexpr int fold(int i) { return i % P > H ? P - i % P : i % P; }
  static constexpr double sign(int i) { return i % P > H ? -1.0 : 1.0; }
  static constexpr double error(const double (&e)[H + 1], const double (&s)[H + 1]) {  // e[i] of sine i
    double own = 0.0, both = 0.0;
    for (int i = 1; i <= H; ++i) own += e[i] * e[i] * H;
    for (int a = 1; a <= H; ++a)
      for (int b = 1; b <= H; ++b) {
        double v = 0.0;
        for (int m = 1; m <= H; ++m)
          v += sign(m * a) * s[fold(m * a)] * sign(m * b) * e[fold(m * b)] + sign(m * b) * s[fold(m * b)] * sign(m * a) * e[fold(m * a)];
        both += v * v;
      }
    return own / H + both / P;
  }
  static constexpr int choose() {
    double s[H + 1] = {}, e[H + 1] = {};
    for (int i = 1; i <= H; ++i) s[i] = sin_turn(i, P);
    int best = 1;
    double least = -1.0;
    for (int j = 1; j <= H; ++j) {
      const double o = (double)(S)s[j];
      for (int i = 1; i <= H; ++i) e[i] = sin_err(i, P, o, i == j ? 1.0 : (double)(S)sin_over(i, P, o));
      const double v = error(e, s);
      if (least < 0.0 || v < least) {
        least = v;
        best = j;
      }
    }
    return best;
  }
  static constexpr int choice = choose();
  // sine i (1 .. H) of a direction: rounded to nearest, but for 3 points (their only rounded
  // constant) inverse to the other side where that leaves less of both errors: a transform and
  // its inverse make a gain of them, and the gains of three axes add up. In FP64, -0.45 and
  // +0.55 of the last bit: 36^3 free, round trip of a solve, 3.2e-16 -> 2.2e-16
  static constexpr S value(int i, int dir) {
    const double v = (double)(S)sin_turn(i, P), e = -sin_err(i, P, v, 1.0);
    if (H > 1 || dir < 0 || e == 0.0) return (S)v;
    double ulp = sizeof(S) == 4 ? 1.0 / (1 << 24) : 1.0 / (1ll << 53);  // of [1/2, 1)
    for (double x = v; x < 0.5; x *= 2.0) ulp *= 0.5;
    const double f = e > 0.0 ? e - ulp : e + ulp;  // the neighbour's error
    return 4.0 * e * e + 0.5 * e * e > (e + f) * (e + f) + 0.5 * f * f ? (S)(v + (f - e)) : (S)v;
  }
  // the k of row m whose sine it is; another where that pair holds no input (0: none does)
  static constexpr int pick(int m, Mask mask) {
    int k0 = 0;
    for (int k = 1; k <= H; ++k)
      if ((((mask >> k) | (mask >> (P - k))) & 1) && (k0 == 0 || fold(m * k) == choice)) k0 = k;
    return k0;
  }
};
// the k of the i-th smallest cosine (or sine) of 2 pi m k / P, k = 1 .. (P-1)/2: sums take their small
// terms first, whose partial sums then round least
constexpr int by_size(int P, int m, int i, bool sine) {
  for (int k = 1; k <= (P - 1) / 2; ++k) {
    int smaller = 0;
    for (int l = 1; l <= (P - 1) / 2; ++l) {
      // the angles' distances from a zero, in turns / (4 P): 4 m k from the multiples of 2 P, or from the odd ones of P
      const int x = (4 * m * k + (sine ? 0 : P)) % (2 * P), y = (4 * m * l + (sine ? 0 : P)) % (2 * P);
      smaller += (y < 2 * P - y ? y : 2 * P - y) < (x < 2 * P - x ? x : 2 * P - x);
    }
    if (smaller == i) return k;
  }
  return 0;
}
template <int P, int DIR, Mask MASK, class C>
__device__ __forceinline__ void prime_pairs(C (&x)[P], C x0, const C (&a)[(P - 1) / 2], const C (&b)[(P - 1) / 2]) {
  using S = decltype(x0.x);
  constexpr int H = (P - 1) / 2;
  C sum = x0;
  sfor<H>([&](auto kc) {
    if constexpr (((MASK >> (kc + 1)) | (MASK >> (P - kc - 1))) & 1) sum = cadd(sum, a[kc]);
  });
  C y[P];
  y[0] = sum;
  sfor<H>([&](auto mc) {
    constexpr int m = mc + 1;
    C t = x0;
    sfor<H>([&](auto i) {
      constexpr int k = by_size(P, m, i, false);
      if constexpr (((MASK >> k) | (MASK >> (P - k))) & 1) {
        constexpr S c = (S)cos_turn(m * k, P);
        t = mk(mad(c, a[k - 1].x, t.x), mad(c, a[k - 1].y, t.y));
      }
    });
    constexpr int k0 = SineOut<S, P>::pick(m, MASK);
    C v = t, w = t;  // t +- DIR i s0 u
    if constexpr (k0 > 0) {
      constexpr S s0 = (S)(DIR * SineOut<S, P>::sign(m * k0)) * SineOut<S, P>::value(SineOut<S, P>::fold(m * k0), DIR);
      C u = b[k0 - 1];
      sfor<H>([&](auto i) {
        constexpr int k = by_size(P, m, i, true);
        if constexpr (k != k0 && (((MASK >> k) | (MASK >> (P - k))) & 1)) {
          constexpr S r = (S)(DIR * sin_over(m * k, P, (double)s0));
          u = mk(mad(r, b[k - 1].x, u.x), mad(r, b[k - 1].y, u.y));
        }
      });
      v = mk(mad(-s0, u.y, t.x), mad(s0, u.x, t.y));
      w = mk(mad(s0, u.y, t.x), mad(-s0, u.x, t.y));
    }
    y[m] = v;
    y[P - m] = w;
  });
  sfor<P>([&](auto i) { x[i] = y[i]; });
}

template <int P, int DIR, Mask MASK, class C>
__device__ __forceinline__ void dft_prime(C (&x)[P]) {
  using S = decltype(x[0].x);
  constexpr int H = (P - 1) / 2;
  C a[H], b[H];
  sfor<H>([&](auto kc) {
    constexpr int k = kc + 1;
    constexpr bool lo = (MASK >> k) & 1, hi = (MASK >> (P - k)) & 1;
    if constexpr (lo && hi) {
      a[k - 1] = cadd(x[k], x[P - k]);
      b[k - 1] = csub(x[k], x[P - k]);
    } else if constexpr (lo) {
      a[k - 1] = b[k - 1] = x[k];
    } else if constexpr (hi) {
      a[k - 1] = x[P - k];
      b[k - 1] = mk(-x[P - k].x, -x[P - k].y);
    }
  });
  prime_pairs<P, DIR, MASK>(x, (MASK & 1) ? x[0] : mk(S(0), S(0)), a, b);
}

// a_k, b_k = x_k W^k +- x_{P-k} W^{P-k}, W = exp(DIR 2 pi i K / R): the pairs of a P-point transform behind
// constant twiddles (R = P^2), two operations less each than twiddled apart
template <int P, int R, int K, int DIR, class C>
__device__ __forceinline__ void dft_prime_tw(C (&x)[P]) {
  constexpr int H = (P - 1) / 2;
  C a[H], b[H];
  sfor<H>([&](auto kc) {
    constexpr int k = kc + 1;
    a[kc] = mul_c<R, k * K, DIR>(x[k]);
    b[kc] = x[P - k];
    bfly_c<R, (P - k) * K, DIR>(a[kc], b[kc]);
  });
  prime_pairs<P, DIR, full_mask(P)>(x, x[0], a, b);
}

template <int R, int DIR, Mask MASK, class C>
__device__ __forceinline__ void dft(C (&x)[R]) {
  if constexpr (R == 1) {
  } else if constexpr ((R & (R - 1)) == 0) {
    dft_pow2<R, DIR, MASK>(x);
  } else if constexpr (low_prime(R) == R) {
    dft_prime<R, DIR, MASK>(x);
  } else {
    // R = A B: columns n2 of A-point transforms, then B-point ones over n2.
    // Coprime factors: n = B n1 + A n2, k = B (B^-1 mod A) k1 + A (A^-1 mod B) k2
    // (mod R), no twiddles; a prime power: n = n2 + B n1, k = k1 + A k2 with W_R^{n2 k1}
    constexpr bool coprime = low_part(R) < R;
    constexpr int A = coprime ? low_part(R) : R / low_prime(R), B = R / A;
    constexpr int sn1 = B, sn2 = coprime ? A : 1;
    constexpr int sk1 = coprime ? B * inv_mod(B % A, A) : 1, sk2 = coprime ? A * inv_mod(A % B, B) : A;
    constexpr Mask mb = columns_mask(MASK, R, sn2, sn1, A, B);
    constexpr bool twin = !coprime && A == B && B > 2 && mb == full_mask(B);  // 9, 25
    C z[B][A];
    sfor<B>([&](auto n2) {
      constexpr Mask mc = pick_mask(MASK, R, sn2 * n2, sn1, A);
      sfor<A>([&](auto n1) {
        if constexpr ((mc >> n1) & 1) z[n2][n1] = x[(sn1 * n1 + sn2 * n2) % R];
      });
      if constexpr (mc != 0) dft<A, DIR, mc>(z[n2]);
    });
    sfor<A>([&](auto k1) {
      C v[B];
      sfor<B>([&](auto n2) {
        if constexpr (pick_mask(MASK, R, sn2 * n2, sn1, A) != 0) {
          if constexpr (coprime || twin) v[n2] = z[n2][k1];
          else v[n2] = mul_c<R, n2 * k1, DIR>(z[n2][k1]);
        }
      });
      if constexpr (twin) dft_prime_tw<B, R, k1, DIR>(v);
      else dft<B, DIR, mb>(v);
      sfor<B>([&](auto k2) { x[(sk1 * k1 + sk2 * k2) % R] = v[k2]; });
    });
  }
}

// The transform of x[r] w(r) (conj(w(r)) for DIR = +1), A a power of two or a prime;
// w(0) = 1 unless W0. The first additions take pairs p +- w x of a twiddled p, five
// operations per component instead of six.
template <int A, int DIR, bool W0, class C, class W>
__device__ __forceinline__ void dft_tw(C (&x)[A], W&& w) {
  using S = decltype(x[0].x);
  auto first = [&](auto r) {
    if constexpr (r > 0 || W0) return mul_t<DIR>(x[r], w(r));
    else return x[r];
  };
  auto pair = [&](auto r, auto q, C& s, C& d) {  // w(r) x[r] +- w(q) x[q]
    s = first(r);
    d = x[q];
    const C f = w(q);
    bfly_w(s, d, f.x, DIR < 0 ? f.y : -f.y);
  };
  if constexpr ((A & (A - 1)) == 0) {
    C y[A];
    sfor<A / 2>([&](auto i) {
      constexpr int r = bitrev(2 * i, A);
      pair(std::integral_constant<int, r>{}, std::integral_constant<int, r + A / 2>{}, y[2 * i], y[2 * i + 1]);
    });
    pow2_layers<A, DIR, full_mask(A), 4>(y);
    sfor<A>([&](auto i) { x[i] = y[i]; });
  } else if constexpr (low_prime(A) == A) {
    constexpr int H = (A - 1) / 2;
    C a[H], b[H];
    sfor<H>([&](auto k) {
      pair(std::integral_constant<int, k + 1>{}, std::integral_constant<int, A - 1 - k>{}, a[k], b[k]);
    });
    const C x0 = first(std::integral_constant<int, 0>{});
    prime_pairs<A, DIR, full_mask(A)>(x, x0, a, b);
  } else {
    sfor<A>([&](auto r) { x[r] = first(r); });
    dft<A, DIR, full_mask(A)>(x);
  }
}

template <int R, int DIR, class C>
__device__ __forceinline__ void dft_pre(C (&x)[R], const C* tw, int e, int NR) {
  if constexpr (R == 1) {
  } else if constexpr ((R & (R - 1)) == 0) {
    C y[R];
    sfor<R>([&](auto i) { y[bitrev(i, R)] = x[i]; });
    auto layer = [&](auto mc) {
      constexpr int m = mc;
      sfor<m / 2>([&](auto Kc) {
        constexpr int K = Kc;
        const C w = tw[(R / m) * (e + K * NR)];
        sfor<R / m>([&](auto blk) {
          constexpr int p = blk * m + K;
          bfly_w(y[p], y[p + m / 2], w.x, DIR < 0 ? w.y : -w.y);
        });
      });
    };
    layer(std::integral_constant<int, 2>{});
    if constexpr (R >= 4) layer(std::integral_constant<int, 4>{});
    if constexpr (R >= 8) layer(std::integral_constant<int, 8>{});
    if constexpr (R >= 16) layer(std::integral_constant<int, 16>{});
    if constexpr (R >= 32) layer(std::integral_constant<int, 32>{});
    sfor<R>([&](auto i) { x[i] = y[i]; });
  } else if constexpr (low_prime(R) == R) {
    dft_tw<R, DIR, false>(x, [&](auto r) { return tw[e * r]; });
  } else {
    // as dft(), with the twiddles in the columns
    constexpr bool coprime = low_part(R) < R;
    constexpr int A = coprime ? low_part(R) : R / low_prime(R), B = R / A;
    constexpr int sn1 = B, sn2 = coprime ? A : 1;
    constexpr int sk1 = coprime ? B * inv_mod(B % A, A) : 1, sk2 = coprime ? A * inv_mod(A % B, B) : A;
    constexpr bool twin = !coprime && A == B && B > 2;
    C z[B][A];
    sfor<B>([&](auto n2) {
      sfor<A>([&](auto n1) { z[n2][n1] = x[(sn1 * n1 + sn2 * n2) % R]; });
      dft_tw<A, DIR, (n2 > 0)>(z[n2], [&](auto n1) { return tw[e * ((sn1 * n1 + sn2 * n2) % R)]; });
    });
    sfor<A>([&](auto k1) {
      C v[B];
      sfor<B>([&](auto n2) {
        if constexpr (coprime || twin) v[n2] = z[n2][k1];
        else v[n2] = mul_c<R, n2 * k1, DIR>(z[n2][k1]);
      });
      if constexpr (twin) dft_prime_tw<B, R, k1, DIR>(v);
      else dft<B, DIR, full_mask(B)>(v);
      sfor<B>([&](auto k2) { x[(sk1 * k1 + sk2 * k2) % R] = v[k2]; });
    });
  }
}

}  // namespace tile
}  // namespace ps
