// Compile-time DFTs of any length up to 32 held in registers, FP32 and FP64,
// for the tile kernels (tile_pass.cuh).
//
//   dft<R, DIR, MASK>(x)   x[k] <- sum_r x[r] exp(DIR 2 pi i r k / R), natural
//       order; inputs r whose bit is missing from MASK are zero and are not read
//       (the zero padding of §3), outputs the caller does not read are removed by
//       the compiler (the compaction of §3)
//   dft_pre<R, DIR>(x, tw, e, NR)   the same of x[r] W_N^{e r}, W_N^j = tw[j],
//       N = R NR (conjugated for DIR = +1)
//
// Powers of two run as radix-2 layers whose butterfly a +- w b takes six FMAs
// (a + w b as two per component, a - w b = 2 a - (a + w b) as one) instead of
// four for the product and four adds: on GB300 the FP64 pipe (two lanes per
// clock and SM) bounds every FP64 pass, and FP32 passes are bound by issue, so
// the operation count is the time. A twiddle in front of the transform folds
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

// cos and sin of |x| <= pi/4 by their Taylor series
constexpr double cos_small(double x) {
  const double y = x * x;
  return 1.0 + y * (-1.0 / 2 + y * (1.0 / 24 + y * (-1.0 / 720 + y * (1.0 / 40320 + y * (-1.0 / 3628800 +
         y * (1.0 / 479001600.0 + y * (-1.0 / 87178291200.0 + y * (1.0 / 20922789888000.0))))))));
}
constexpr double sin_small(double x) {
  const double y = x * x;
  return x * (1.0 + y * (-1.0 / 6 + y * (1.0 / 120 + y * (-1.0 / 5040 + y * (1.0 / 362880 + y * (-1.0 / 39916800.0 +
         y * (1.0 / 6227020800.0 + y * (-1.0 / 1307674368000.0 + y * (1.0 / 355687428096000.0)))))))));
}
// cos(2 pi m / N), reduced exactly in integers to an angle of at most pi/4
constexpr double cos_turn(long m, long N) {
  m = ((m % N) + N) % N;
  long p = 4 * m;            // angle = 2 pi p / (4 N)
  if (p > 2 * N) p = 4 * N - p;
  const bool neg = p > N;
  if (neg) p = 2 * N - p;    // 0 .. pi/2
  constexpr double half_pi = 1.57079632679489661923;
  const double v = 2 * p > N ? sin_small(half_pi * (double)(N - p) / (double)N) : cos_small(half_pi * (double)p / (double)N);
  return neg ? -v : v;
}
constexpr double sin_turn(long m, long N) { return cos_turn(4 * m - N, 4 * N); }

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

// (a, b) <- (a + w b, a - w b)
template <class C, class S>
__device__ __forceinline__ void bfly_w(C& a, C& b, S wr, S wi) {
  const C s = mk(mad(-wi, b.y, mad(wr, b.x, a.x)), mad(wi, b.x, mad(wr, b.y, a.y)));
  b = mk(mad(S(2), a.x, -s.x), mad(S(2), a.y, -s.y));
  a = s;
}
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
    constexpr S wr = (S)cos_turn(K, M), wi = (S)(DIR * sin_turn(K, M));
    bfly_w(a, b, wr, wi);
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
// u_m = sum_k sin(2 pi m k / p) b_k, a_k, b_k = x_k +- x_{p-k}, k = 1 .. (p-1)/2. From p = 5 on
// y_m is one chain of FMAs from t_m and y_{p-m} = 2 t_m - y_m, an operation less per
// component than forming u_m (5 points: 32 operations instead of 36).
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
    sfor<H>([&](auto kc) {
      constexpr int k = kc + 1;
      if constexpr (((MASK >> k) | (MASK >> (P - k))) & 1) {
        constexpr S c = (S)cos_turn(m * k, P);
        t = mk(mad(c, a[kc].x, t.x), mad(c, a[kc].y, t.y));
      }
    });
    C v = t, w = t;  // t +- DIR i u
    sfor<H>([&](auto kc) {
      constexpr int k = kc + 1;
      if constexpr (((MASK >> k) | (MASK >> (P - k))) & 1) {
        constexpr S s = (S)(DIR * sin_turn(m * k, P));
        v = mk(mad(-s, b[kc].y, v.x), mad(s, b[kc].x, v.y));
        if constexpr (H == 1) w = mk(mad(s, b[kc].y, w.x), mad(-s, b[kc].x, w.y));
      }
    });
    if constexpr (H > 1) w = mk(mad(S(2), t.x, -v.x), mad(S(2), t.y, -v.y));
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
          if constexpr (coprime) v[n2] = z[n2][k1];
          else v[n2] = mul_c<R, n2 * k1, DIR>(z[n2][k1]);
        }
      });
      constexpr Mask mb = columns_mask(MASK, R, sn2, sn1, A, B);
      dft<B, DIR, mb>(v);
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
    if constexpr (r > 0 || W0) return mul_w<DIR>(x[r], w(r));
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
    C z[B][A];
    sfor<B>([&](auto n2) {
      sfor<A>([&](auto n1) { z[n2][n1] = x[(sn1 * n1 + sn2 * n2) % R]; });
      dft_tw<A, DIR, (n2 > 0)>(z[n2], [&](auto n1) { return tw[e * ((sn1 * n1 + sn2 * n2) % R)]; });
    });
    sfor<A>([&](auto k1) {
      C v[B];
      sfor<B>([&](auto n2) {
        if constexpr (coprime) v[n2] = z[n2][k1];
        else v[n2] = mul_c<R, n2 * k1, DIR>(z[n2][k1]);
      });
      dft<B, DIR, full_mask(B)>(v);
      sfor<B>([&](auto k2) { x[(sk1 * k1 + sk2 * k2) % R] = v[k2]; });
    });
  }
}

}  // namespace tile
}  // namespace ps
