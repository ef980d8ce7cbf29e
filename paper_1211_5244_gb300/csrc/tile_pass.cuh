// Tile kernels: the passes of a solve for a line of any length that tile_radix
// (tile_launch.cu) factors, FP32 and FP64, along any axis, as two (or three) register
// DFT steps with one exchange through shared memory between them. It factors products of
// two or three radices up to 16, and a prime from 17 to 31 behind at most two of them;
// other lengths with a prime factor from 11 on run in Bluestein form (below). Smooth
// lengths that need a fourth radix (48 from 625 on: 625, 875, 1250, 2000, 2187, 4000, ...)
// and 2, 3, 5 and 7 stay on the Stockham kernels.
//
// A CTA owns a tile of tk lines; the butterflies of a step are spread over its threads
// (tasks). With
// N = Ra Rm Rl, n = n1 NRa + n2 Rl + n3 and k = k1 + Ra k2 + Ra Rm k3 the forward
// transform is
//   first  (n2, n3): Ra-point DFT over n1 -> k1, inputs straight from global memory
//   middle (k1, n3): inputs times W_N^{k1 Rl n2}, Rm-point DFT over n2 -> k2
//   last   (k1, k2): inputs times W_N^{(k1 + Ra k2) n3}, Rl-point DFT over n3 -> k3,
//                    outputs straight to global memory at k1 + Ra k2 + Ra Rm k3
// and the inverse the same steps backwards (twiddles before the middle and the
// final step). Every step replaces the tile elements it read, so one buffer
// serves all of them; the fused pass multiplies by K^F between the last forward
// and the first inverse step, which share their elements, in registers.
//
// What bounds them: in FP32 issue and latency (100 x 90 x 110 free, L = 200 x 180 x
// 220: 250 -> 63 us per solve against the Stockham and Bluestein kernels of
// passes.cu, which make a shared-memory round trip per stage and more for the load,
// the multiply and the store, and spend a third of their issue slots on integer
// instructions), in FP64 the two FP64 lanes per clock and SM (128^3 free: 1657
// -> 1161 us; the pipe was 84% busy before, so only fewer operations help).
#pragma once

#include "fft_fast.cuh"
#include "reduce.cuh"
#include "tile_dft.cuh"

namespace ps {
namespace tile {

// calls f(integral_constant<R>) for R in LO .. HI by a binary search of
// comparisons: a switch's jump table is a load and an indirect branch at every step
// of every tile, both waits at the 16 to 24 warps an SM holds (90 x 75 x 110 ppf:
// solve 28.5 -> 27.4 us; 32 uneven problems 872 -> 861 us)
template <int LO, int HI, class F>
__device__ __forceinline__ void pick_radix(int R, F&& f) {
  if constexpr (LO == HI) {
    f(std::integral_constant<int, LO>{});
  } else {
    constexpr int MID = (LO + HI) / 2;
    if (R <= MID) pick_radix<LO, MID>(R, f);
    else pick_radix<MID + 1, HI>(R, f);
  }
}

// calls f(integral_constant<R>) for the run-time radix R of a step. Class 0: radices
// up to 8, class 1: up to 16, class 2: a prime from 17 to 31 in the last forward
// (first inverse) step, LAST, and radices up to 16, or 1, in the others. The class
// bounds a kernel's registers, hence the separate instances.
template <int CLS, bool LAST, class F>
__device__ __forceinline__ void radix_switch(int R, F&& f) {
  if constexpr (CLS == 0) {
    pick_radix<2, 8>(R, f);
  } else if constexpr (CLS == 2 && LAST) {
    if (R <= 19) {
      if (R <= 17) f(std::integral_constant<int, 17>{});
      else f(std::integral_constant<int, 19>{});
    } else if (R <= 23) {
      f(std::integral_constant<int, 23>{});
    } else if (R <= 29) {
      f(std::integral_constant<int, 29>{});
    } else {
      f(std::integral_constant<int, 31>{});
    }
  } else {
    pick_radix<CLS == 2 ? 1 : 2, 16>(R, f);
  }
}

// The tile: lines [t * ls] of elements in shared memory, the table W_N^j after them.
template <class C>
struct Tile {
  C* sh;
  const C* tw;
};

// the tile's place, and the asynchronous copy of the twiddle table, which the
// first step does not read: steps_sync after it
template <class C>
__device__ __forceinline__ Tile<C> tile_setup(const TileArgs& a, unsigned char* raw) {
  Tile<C> s;
  s.sh = reinterpret_cast<C*>(raw);
  C* tw = s.sh + a.elems;
  const C* g = static_cast<const C*>(a.tw);
  for (int i = threadIdx.x; i < a.N; i += blockDim.x) {
    if constexpr (sizeof(C) == 8)
      cp_async8(tw + i, g + (long long)i * a.tws);
    else
      cp_async16(tw + i, g + (long long)i * a.tws);
  }
  cp_async_commit();
  s.tw = tw;
  return s;
}
__device__ __forceinline__ void steps_sync() {
  cp_async_wait_all();
  __syncthreads();
}

// calls f(t, b) for this thread's share of the nb butterflies of each of the
// tile's tk lines: consecutive threads along the lines' butterflies where the
// lines are the contiguous axis, else across the lines. No thread idles but in
// the last round, whatever nb is (an idle lane costs as much FP64 time as a busy one).
template <class F>
__device__ __forceinline__ void tasks(const TileArgs& a, int nb, unsigned mnb, F&& f) {
  const int n = nb << a.ltk;
  for (int w = threadIdx.x; w < n; w += blockDim.x) {
    int t, b;
    if (a.lc) {
      t = div_by(w, mnb);
      b = w - t * nb;
    } else {
      t = w & (a.tk - 1);
      b = w >> a.ltk;
    }
    f(t, b);
  }
}

// The tile's line t: its index along the tile axis and its plane; false beyond
// the last one. Tiles belong to one plane (blockIdx.y), or run over the lines of
// all planes in sequence (flat), so that only the last tile is ragged.
__device__ __forceinline__ bool line_of(const TileArgs& a, int t, int* line, int* pl) {
  const unsigned g = (blockIdx.x - a.shift) * (unsigned)a.tk + t;
  if (!a.flat) {
    *line = (int)g;
    *pl = blockIdx.y;
    return g < (unsigned)a.ntl;
  }
  const unsigned p = g / (unsigned)a.ntl;
  *line = (int)(g - p * (unsigned)a.ntl);
  *pl = (int)p;
  return p < (unsigned)a.npl;
}

// tile position and exponent (k1 + Ra k2) of butterfly bf of the last step
__device__ __forceinline__ void last_digits(const TileArgs& a, int bf, int* pos, int* e) {
  if (a.Rm == 1) {
    *pos = bf * a.s1;
    *e = bf;
  } else {
    const int k1 = div_by(bf, a.mRm), k2 = bf - k1 * a.Rm;
    *pos = k1 * a.s1 + k2 * a.s2;
    *e = k1 + a.Ra * k2;
  }
}
// tile position of output k after the last forward step
__device__ __forceinline__ int k_pos(const TileArgs& a, int k) {
  const int q = div_by(k, a.mRa), k1 = k - q * a.Ra;
  if (a.Rm == 1) return k1 * a.s1 + q * a.es;
  const int r = div_by(q, a.mRm), k2 = q - r * a.Rm;
  return k1 * a.s1 + k2 * a.s2 + r * a.es;
}

// first forward step: lines(t)(tile address, element) gives the inputs, half of them zero for HALF
template <int DIR, bool HALF, int CLS, class C, class Ln>
__device__ __forceinline__ void step_first(const TileArgs& a, const Tile<C>& s, Ln&& lines) {
  radix_switch<CLS, false>(a.Ra, [&](auto rc) {
    constexpr int R = rc;
    if constexpr (!HALF || R % 2 == 0) {
      constexpr int RN = HALF ? R / 2 : R;
      tasks(a, a.NRa, a.mNRa, [&](int t, int b) {
        const auto ld = lines(t);
        C* p = s.sh + t * a.ls + b * a.es;
        C x[R];
#pragma unroll
        for (int r = 0; r < RN; ++r) x[r] = ld(p + r * a.s1, b + r * a.NRa);
        dft<R, DIR, full_mask(RN)>(x);
#pragma unroll
        for (int r = 0; r < R; ++r) p[r * a.s1] = x[r];
      });
    }
  });
}
// final inverse step: lines(t)(tile address, element, value) takes the outputs, the lower half for HALF
template <bool HALF, int CLS, class C, class Ln>
__device__ __forceinline__ void step_final(const TileArgs& a, const Tile<C>& s, Ln&& lines) {
  radix_switch<CLS, false>(a.Ra, [&](auto rc) {
    constexpr int R = rc;
    if constexpr (!HALF || R % 2 == 0) {
      constexpr int RN = HALF ? R / 2 : R;
      tasks(a, a.NRa, a.mNRa, [&](int t, int b) {
        C x[R];
        C* p = s.sh + t * a.ls + b * a.es;
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = p[r * a.s1];
        dft_pre<R, 1>(x, s.tw, b, a.NRa);
        const auto st = lines(t);
#pragma unroll
        for (int r = 0; r < RN; ++r) st(p + r * a.s1, b + r * a.NRa, x[r]);
      });
    }
  });
}
// middle step of three, in place
template <int DIR, int CLS, class C>
__device__ __forceinline__ void step_middle(const TileArgs& a, const Tile<C>& s) {
  if (a.Rm == 1) return;
  const int NRm = a.Ra * a.Rl;
  radix_switch<CLS, false>(a.Rm, [&](auto rc) {
    constexpr int R = rc;
    tasks(a, NRm, a.mNRm, [&](int t, int b) {
      const int k1 = div_by(b, a.mRl), n3 = b - k1 * a.Rl;
      C* p = s.sh + t * a.ls + k1 * a.s1 + n3 * a.es;
      C x[R];
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = p[r * a.s2];
      dft_pre<R, DIR>(x, s.tw, DIR < 0 ? k1 * a.Rl : a.Ra * n3, NRm);
#pragma unroll
      for (int r = 0; r < R; ++r) p[r * a.s2] = x[r];
    });
  });
  __syncthreads();
}
// last forward step: lines(t)(tile address, k, value) takes the outputs
template <int CLS, class C, class Ln>
__device__ __forceinline__ void step_last(const TileArgs& a, const Tile<C>& s, Ln&& lines) {
  radix_switch<CLS, true>(a.Rl, [&](auto rc) {
    constexpr int R = rc;
    tasks(a, a.Kl, a.mKl, [&](int t, int b) {
      int pos, e;
      last_digits(a, b, &pos, &e);
      C* p = s.sh + t * a.ls + pos;
      C x[R];
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = p[r * a.es];
      dft_pre<R, -1>(x, s.tw, e, a.Kl);
      const auto st = lines(t);
#pragma unroll
      for (int r = 0; r < R; ++r) st(p + r * a.es, e + r * a.Kl, x[r]);
    });
  });
}
// first inverse step: lines(t)(tile address, k) gives the inputs
template <int CLS, class C, class Ln>
__device__ __forceinline__ void step_inv_first(const TileArgs& a, const Tile<C>& s, Ln&& lines) {
  radix_switch<CLS, true>(a.Rl, [&](auto rc) {
    constexpr int R = rc;
    tasks(a, a.Kl, a.mKl, [&](int t, int b) {
      const auto ld = lines(t);
      int pos, e;
      last_digits(a, b, &pos, &e);
      C* p = s.sh + t * a.ls + pos;
      C x[R];
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = ld(p + r * a.es, e + r * a.Kl);
      dft<R, 1, full_mask(R)>(x);
#pragma unroll
      for (int r = 0; r < R; ++r) p[r * a.es] = x[r];
    });
  });
}

// Resident CTAs (of 256 threads) per SM asked of the compiler. The FP32 passes are
// bound by latency, so more warps pay where the radices still fit their registers:
// the real passes and the Bluestein form take one CTA more (64 registers for class 1; 32
// uneven problems 860 -> 834 us). The fused pass spills there (128^3 ffp 59.3 -> 64.7 us),
// and the line pass loses by it (100 x 90 x 110 free 62.0 -> 63.0 us). The fused Bluestein
// pass spills 96 bytes and loses alone (the z pass of 74 x 79 x 83 free 40.9 -> 43.4 us, of 127 x 131 x
// 113 periodic 23.0 -> 25.2), but in a batch, where its CTAs share the SMs with other problems', the
// narrower one gains: 32 uneven problems 853 -> 837 us.
template <typename T, int CLS>
struct Bounds {
  static constexpr int per_sm = sizeof(T) == 4 ? (CLS == 0 ? 4 : CLS == 1 ? 3 : 2) : (CLS == 0 ? 3 : CLS == 1 ? 2 : 1);
  static constexpr int more = sizeof(T) == 4 && CLS < 2 ? per_sm + 1 : per_sm;
};

// ------------------------------------------------------------ complex lines

// DIR -1: nin inputs (the rest zero), N outputs; +1: N inputs, nout outputs
template <typename T, int DIR, bool HALF, int CLS>
__global__ void __launch_bounds__(256, Bounds<T, CLS>::per_sm) k_tile_line(const __grid_constant__ TileArgs a) {
  using C = cpx<T>;
  extern __shared__ __align__(16) unsigned char raw[];
  const Tile<C> s = tile_setup<C>(a, raw);
  // the lines of the tile at their source and destination
  auto in = [&](int t, bool* ok) {
    int line, pl;
    *ok = line_of(a, t, &line, &pl);
    return static_cast<const C*>(a.src) + (pl * a.sp_in + line * a.st_in);
  };
  auto out = [&](int t, bool* ok) {
    int line, pl;
    *ok = line_of(a, t, &line, &pl);
    return static_cast<C*>(a.dst) + (pl * a.sp_out + line * a.st_out);
  };
  pdl_wait();
  if constexpr (DIR < 0) {
    step_first<-1, HALF, CLS>(a, s, [&](int t) {
      bool ok;
      const C* src = in(t, &ok);
      return [&a, src, ok](C*, int e) { return ok && e < a.nin ? src[(long long)e * a.se_in] : mk(T(0), T(0)); };
    });
    steps_sync();
    step_middle<-1, CLS>(a, s);
    step_last<CLS>(a, s, [&](int t) {
      bool ok;
      C* dst = out(t, &ok);
      return [&a, dst, ok](C*, int k, C v) {
        if (ok) dst[(long long)k * a.se_out] = v;
      };
    });
  } else {
    step_inv_first<CLS>(a, s, [&](int t) {
      bool ok;
      const C* src = in(t, &ok);
      return [&a, src, ok](C*, int k) { return ok ? src[(long long)k * a.se_in] : mk(T(0), T(0)); };
    });
    steps_sync();
    step_middle<1, CLS>(a, s);
    step_final<HALF, CLS>(a, s, [&](int t) {
      bool ok;
      C* dst = out(t, &ok);
      return [&a, dst, ok](C*, int e, C v) {
        if (ok && e < a.nout) dst[(long long)e * a.se_out] = v;
      };
    });
  }
}

// ------------------------------------------------------------ forward, K^F, inverse

// The energy of a fused pass: a thread's value (its own lines' terms, in the plan's type)
// joins the others in 64 bits, across the warp here, across the warps after the next
// barrier, across the CTAs in the last pass (energy_total). FP32 values cross the warp as
// sums and their exact errors (Knuth's two-sum), 48 bits: as FP64 additions the five steps
// hold the two-lane pipe for 80 cycles a warp, with the CTA's barrier behind them (100 x 90 x
// 110 free, a solve: 32-bit sums 61.0 us, FP64 61.7, two-sums level with 32 bits;
// 128^3 ffp 62.6, 63.4 and +0.4 us).
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum(float v) {
  float hi = v, lo = 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float b = __shfl_xor_sync(0xffffffffu, hi, o), l = __shfl_xor_sync(0xffffffffu, lo, o);
    const float s = hi + b, t = s - hi;
    lo = (lo + l) + ((hi - (s - t)) + (b - t));
    hi = s;
  }
  // a sum beyond FP32's range, an infinity or a NaN (the same in every lane)
  if (!(fabsf(hi) <= 3.4028234e38f)) return warp_sum((double)v);
  return (double)hi + (double)lo;
}
template <typename T>
__device__ __forceinline__ void energy_lanes(T en, double* wsum) {
  const double v = warp_sum(en);
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
}
__device__ __forceinline__ void energy_cta_sum(const TileArgs& a, const double* wsum) {
  double sum = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += wsum[w];
  a.partials[blockIdx.y * gridDim.x + blockIdx.x] = sum;
}

template <typename T, bool HALF, int CLS>
__global__ void __launch_bounds__(256, Bounds<T, CLS>::per_sm) k_tile_conv(const __grid_constant__ TileArgs a) {
  using C = cpx<T>;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ double wsum[8];
  const Tile<C> s = tile_setup<C>(a, raw);
  auto at = [&](int t, int* line, int* pl) {
    const bool ok = line_of(a, t, line, pl);
    if (a.pair_pl && ok) *pl = paired_ky(*pl, a.npl);
    return ok;
  };
  auto ptr = [&](int t, bool* ok) {
    int line, pl;
    *ok = at(t, &line, &pl);
    return static_cast<C*>(a.dst) + (pl * a.sp_in + line * a.st_in);
  };
  pdl_wait();
  step_first<-1, HALF, CLS>(a, s, [&](int t) {
    bool ok;
    const C* src = ptr(t, &ok);
    return [&a, src, ok](C*, int e) { return ok && e < a.nin ? src[(long long)e * a.se_in] : mk(T(0), T(0)); };
  });
  steps_sync();
  step_middle<-1, CLS>(a, s);
  T en = T(0);
  radix_switch<CLS, true>(a.Rl, [&](auto rc) {
    constexpr int R = rc;
    tasks(a, a.Kl, a.mKl, [&](int t, int b) {
      int line, pl, pos, e;
      const bool ok = at(t, &line, &pl);
      const T* Kp = static_cast<const T*>(a.K) + (long long)min(pl, a.Lp - pl) * a.Ksp +
                    (long long)min(line, a.Lt - line) * a.Kst;
      last_digits(a, b, &pos, &e);
      T kk[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int k = e + r * a.Kl;
        kk[r] = ok ? __ldg(Kp + (long long)min(k, a.N - k) * a.Kse) : T(0);
      }
      C* p = s.sh + t * a.ls + pos;
      C x[R];
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = p[r * a.es];
      dft_pre<R, -1>(x, s.tw, e, a.Kl);
      if (a.E != nullptr) {  // a solve without the energy saves its products
        T el = T(0);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const C u = mk(kk[r] * x[r].x, kk[r] * x[r].y);
          el = mad(u.x, x[r].x, mad(u.y, x[r].y, el));  // K |rho^F|^2
          x[r] = u;
        }
        const int k0 = a.w_tile ? line : pl;
        en = mad(k0 == 0 || 2 * k0 == a.La0 ? T(1) : T(2), el, en);
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = mk(kk[r] * x[r].x, kk[r] * x[r].y);
      }
      dft<R, 1, full_mask(R)>(x);
#pragma unroll
      for (int r = 0; r < R; ++r) p[r * a.es] = x[r];
    });
  });
  if (a.E != nullptr) energy_lanes(en, wsum);
  __syncthreads();
  if (a.E != nullptr && threadIdx.x == 0) energy_cta_sum(a, wsum);
  step_middle<1, CLS>(a, s);
  step_final<HALF, CLS>(a, s, [&](int t) {
    bool ok;
    C* dst = ptr(t, &ok);
    return [&a, dst, ok](C*, int e, C v) {
      if (ok && e < a.nout) dst[(long long)e * a.se_out] = v;
    };
  });
}

// ------------------------------------------------------------ real passes

// PAIR: a line is two real sequences a + i b of length N (columns 2t and 2t + 1
// along y or z, or rows 2t and 2t + 1 of an odd x axis), separated by
//   A[k] = (Z[k] + conj Z[N-k]) / 2,  B[k] = (Z[k] - conj Z[N-k]) / 2i,  k <= N/2;
// else a row of length L = 2 N packed as z[m] = x[2m] + i x[2m+1], untangled by
//   X[k] = E[k] + W_L^k O[k],  E = (Z[k] + conj Z[N-k]) / 2,  O = -i (Z[k] - conj Z[N-k]) / 2.
// A line of a pair has its second sequence unless it is the last of an odd number.

// With the energy the last pass has one CTA more in x (shift = 1), which adds the
// partials of the fused pass and has no lines: its round trips to L2 would
// lengthen the pass by 1 to 3 us where they follow a CTA's own lines (128^3, 65 x 256
// lines: 15.9 against 12.5 us).
__device__ __forceinline__ bool energy_cta(const TileArgs& a) {
  if (a.shift == 0 || blockIdx.x != 0) return false;
  pdl_wait();
  if (blockIdx.y == 0) energy_total(a.partials, a.nparts, a.escale, a.E);
  return true;
}

// element e of line t of a real pass: the pair of reals at src, im_off apart
template <typename T, bool PAIR>
struct RealLine {
  T* p0;
  const T* add;  // the energy term's V at the line, and its factor
  T fac;
  bool ok, two;
  __device__ __forceinline__ RealLine(const TileArgs& a, const void* base, long long sp, long long st, int t) {
    int line, pl;
    ok = line_of(a, t, &line, &pl);
    p0 = const_cast<T*>(static_cast<const T*>(base)) + (pl * sp + line * st);
    two = PAIR && 2 * line + 1 < a.nreal;
    add = nullptr;
    if (a.addV != nullptr) {
      add = static_cast<const T*>(a.addV) + (pl * sp + line * st);
      fac = (T)(a.h3 * __ldg(a.gE));
    }
  }
  __device__ __forceinline__ cpx<T> load(const TileArgs& a, int e) const {
    cpx<T> v = mk(T(0), T(0));
    if (!ok || e >= a.nin) return v;
    const T* p = p0 + (long long)e * a.se_in;
    const bool im = PAIR ? two : 2 * e + 1 < a.nreal;
    if (a.vec && im) return *reinterpret_cast<const cpx<T>*>(p);
    v.x = p[0];
    if (im) v.y = p[a.im_off];
    return v;
  }
  __device__ __forceinline__ void store(const TileArgs& a, int e, cpx<T> v) const {
    if (!ok || e >= a.nout) return;
    T* p = p0 + (long long)e * a.se_out;
    const bool im = PAIR ? two : 2 * e + 1 < a.nreal;
    if (add != nullptr) {
      const T* q = add + (long long)e * a.se_out;
      v.x = mad(fac, q[0], v.x);
      if (im) v.y = mad(fac, q[a.im_off], v.y);
    }
    if (a.vec && im) {
      *reinterpret_cast<cpx<T>*>(p) = v;
    } else {
      p[0] = v.x;
      if (im) p[a.im_off] = v.y;
    }
  }
};

// the outputs of line t of a forward real pass at wavenumber k from Z[k], Z[N-k]
template <typename T, bool PAIR>
__device__ __forceinline__ void untangle(const TileArgs& a, int t, int k, int N, cpx<T> zk, cpx<T> zm) {
  using C = cpx<T>;
  int line, pl;
  if (!line_of(a, t, &line, &pl)) return;
  const C e = mk(T(0.5) * (zk.x + zm.x), T(0.5) * (zk.y - zm.y));
  const C o = mk(T(0.5) * (zk.y + zm.y), T(0.5) * (zm.x - zk.x));
  C* d = static_cast<C*>(a.dst) + (pl * a.sp_out + line * a.st_out);
  if constexpr (PAIR) {
    d[(long long)k * a.se_out] = e;
    if (2 * line + 1 < a.nreal) d[(long long)k * a.se_out + a.im_c] = o;
  } else {
    // outputs k and N - k from the same pair: X[N-k] = conj(E - W^k O)
    const C wo = mul_w<-1>(o, __ldg(static_cast<const C*>(a.twL) + k));
    d[k] = cadd(e, wo);
    if (2 * k != N) d[N - k] = mk(e.x - wo.x, wo.y - e.y);
  }
}

// Z[k] and Z[N-k] of line t of an inverse real pass
template <typename T, bool PAIR>
__device__ __forceinline__ void tangle(const TileArgs& a, int t, int k, int N, cpx<T>* zk, cpx<T>* zm) {
  using C = cpx<T>;
  int line, pl;
  *zk = *zm = mk(T(0), T(0));
  if (!line_of(a, t, &line, &pl)) return;
  const C* x = static_cast<const C*>(a.src) + (pl * a.sp_in + line * a.st_in);
  if constexpr (PAIR) {
    // Z[k] = A + i B, Z[N-k] = conj A + i conj B; A and B are real at k = 0 and
    // N/2, so their (rounding-level) imaginary parts there are dropped
    C A = x[(long long)k * a.se_in], B = mk(T(0), T(0));
    if (2 * line + 1 < a.nreal) B = x[(long long)k * a.se_in + a.im_c];
    if (k == 0 || 2 * k == N) A.y = B.y = T(0);
    *zk = mk(A.x - B.y, A.y + B.x);
    *zm = mk(A.x + B.y, B.x - A.y);
  } else {
    // Z[k] = E' + i O', E' = X[k] + conj X[N-k], O' = (X[k] - conj X[N-k]) conj W_L^k;
    // E'[N-k] = conj E'[k], O'[N-k] = conj O'[k]
    const C xk = x[k], xm = x[N - k];
    const C e = mk(xk.x + xm.x, xk.y - xm.y);
    const C o = mul_w<1>(mk(xk.x - xm.x, xk.y + xm.y), __ldg(static_cast<const C*>(a.twL) + k));
    *zk = mk(e.x - o.y, e.y + o.x);
    *zm = mk(e.x + o.y, o.x - e.y);
  }
}

template <typename T, bool PAIR, bool HALF, int CLS>
__global__ void __launch_bounds__(256, Bounds<T, CLS>::more) k_tile_r2c(const __grid_constant__ TileArgs a) {
  using C = cpx<T>;
  extern __shared__ __align__(16) unsigned char raw[];
  const Tile<C> s = tile_setup<C>(a, raw);
  pdl_wait();
  step_first<-1, HALF, CLS>(a, s, [&](int t) {
    const RealLine<T, PAIR> r(a, a.rsrc, a.sp_in, a.st_in, t);
    return [&a, r](C*, int e) { return r.load(a, e); };
  });
  steps_sync();
  step_middle<-1, CLS>(a, s);
  step_last<CLS>(a, s, [&](int) { return [](C* p, int, C v) { *p = v; }; });
  __syncthreads();
  tasks(a, a.N / 2 + 1, a.mout, [&](int t, int k) {
    const C* z = s.sh + t * a.ls;
    untangle<T, PAIR>(a, t, k, a.N, z[k_pos(a, k)], z[k_pos(a, k == 0 ? 0 : a.N - k)]);
  });
}

template <typename T, bool PAIR, bool HALF, int CLS>
__global__ void __launch_bounds__(256, Bounds<T, CLS>::more) k_tile_c2r(const __grid_constant__ TileArgs a) {
  using C = cpx<T>;
  extern __shared__ __align__(16) unsigned char raw[];
  if (energy_cta(a)) return;
  const Tile<C> s = tile_setup<C>(a, raw);
  const int N = a.N;
  pdl_wait();
  // Z[k] and Z[N-k] from the same pair of inputs
  tasks(a, N / 2 + 1, a.mout, [&](int t, int k) {
    C zk, zm;
    tangle<T, PAIR>(a, t, k, N, &zk, &zm);
    C* z = s.sh + t * a.ls;
    z[k_pos(a, k)] = zk;
    if (k != 0 && 2 * k != N) z[k_pos(a, N - k)] = zm;
  });
  __syncthreads();
  step_inv_first<CLS>(a, s, [&](int) { return [](C* p, int) { return *p; }; });
  steps_sync();
  step_middle<1, CLS>(a, s);
  step_final<HALF, CLS>(a, s, [&](int t) {
    const RealLine<T, PAIR> r(a, a.rdst, a.sp_out, a.st_out, t);
    return [&a, r](C*, int e, C v) { r.store(a, e, v); };
  });
}

// ------------------------------------------------------------ Bluestein form

// Lines whose length N has a prime factor from 11 on and no factorisation into steps (a
// prime above 31, two above 16, or 11 and 13 themselves): the chirp-z
// form X[k] = c[k] sum_m (x[m] c[m]) conj(c[k-m]), c[m] = exp(-i pi m^2 / N), as a
// cyclic convolution of length M >= 2 N on the steps above (a.N = M, a.Nt = N):
// the chirp product in the loads, the product with the transformed conjugate chirp Bf
// between the last forward and the first inverse step, the chirp again in the
// stores. DIR = +1 conjugates the chirp and Bf.

template <int DIR, int CLS, class C>
__device__ __forceinline__ void blue_multiply(const TileArgs& a, const Tile<C>& s) {
  radix_switch<CLS, true>(a.Rl, [&](auto rc) {
    constexpr int R = rc;
    tasks(a, a.Kl, a.mKl, [&](int t, int b) {
      int pos, e;
      last_digits(a, b, &pos, &e);
      C* p = s.sh + t * a.ls + pos;
      C x[R];
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = p[r * a.es];
      dft_pre<R, -1>(x, s.tw, e, a.Kl);
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = mul_w<DIR>(x[r], __ldg(static_cast<const C*>(a.Bf) + e + r * a.Kl));
      dft<R, 1, full_mask(R)>(x);
#pragma unroll
      for (int r = 0; r < R; ++r) p[r * a.es] = x[r];
    });
  });
  __syncthreads();
}
// the whole convolution: ld and st as of step_first and step_final, with chirps
template <int DIR, int CLS, class C, class Ld, class St>
__device__ __forceinline__ void blue_conv(const TileArgs& a, const Tile<C>& s, Ld&& ld, St&& st) {
  step_first<-1, true, CLS>(a, s, ld);
  steps_sync();
  step_middle<-1, CLS>(a, s);
  blue_multiply<DIR, CLS>(a, s);
  step_middle<1, CLS>(a, s);
  step_final<true, CLS>(a, s, st);
}
template <class C>
__device__ __forceinline__ C chirp(const TileArgs& a, int m) { return __ldg(static_cast<const C*>(a.chirp) + m); }
// tile position of element m before the first and after the final step
__device__ __forceinline__ int n_pos(const TileArgs& a, int m) {
  const int n1 = div_by(m, a.mNRa);
  return n1 * a.s1 + (m - n1 * a.NRa) * a.es;
}

template <typename T, int DIR, int CLS>
__global__ void __launch_bounds__(256, Bounds<T, CLS>::more) k_blue_line(const __grid_constant__ TileArgs a) {
  using C = cpx<T>;
  extern __shared__ __align__(16) unsigned char raw[];
  const Tile<C> s = tile_setup<C>(a, raw);
  pdl_wait();
  blue_conv<DIR, CLS>(
      a, s,
      [&](int t) {
        int line, pl;
        const bool ok = line_of(a, t, &line, &pl);
        const C* src = static_cast<const C*>(a.src) + (pl * a.sp_in + line * a.st_in);
        return [&a, src, ok](C*, int e) {
          return ok && e < a.nin ? mul_w<DIR>(src[(long long)e * a.se_in], chirp<C>(a, e)) : mk(T(0), T(0));
        };
      },
      [&](int t) {
        int line, pl;
        const bool ok = line_of(a, t, &line, &pl);
        C* dst = static_cast<C*>(a.dst) + (pl * a.sp_out + line * a.st_out);
        return [&a, dst, ok](C*, int e, C v) {
          if (ok && e < a.nout) dst[(long long)e * a.se_out] = mul_w<DIR>(v, chirp<C>(a, e));
        };
      });
}

// Forward, K^F, inverse: between the two convolutions the chirps cancel (|c| = 1), so
// u[k] = K[k] v[k] of the first one's values v is the second one's input, and
// |X|^2 = |v|^2 in the energy; the final step of the first and the first step of the
// second share their elements.
template <typename T, int CLS>
__global__ void __launch_bounds__(256, Bounds<T, CLS>::more) k_blue_conv(const __grid_constant__ TileArgs a) {
  using C = cpx<T>;
  extern __shared__ __align__(16) unsigned char raw[];
  __shared__ double wsum[8];
  const Tile<C> s = tile_setup<C>(a, raw);
  auto at = [&](int t, int* line, int* pl) {
    const bool ok = line_of(a, t, line, pl);
    if (a.pair_pl && ok) *pl = paired_ky(*pl, a.npl);
    return ok;
  };
  auto ptr = [&](int t, bool* ok) {
    int line, pl;
    *ok = at(t, &line, &pl);
    return static_cast<C*>(a.dst) + (pl * a.sp_in + line * a.st_in);
  };
  pdl_wait();
  step_first<-1, true, CLS>(a, s, [&](int t) {
    bool ok;
    const C* src = ptr(t, &ok);
    return [&a, src, ok](C*, int e) {
      return ok && e < a.nin ? mul_w<-1>(src[(long long)e * a.se_in], chirp<C>(a, e)) : mk(T(0), T(0));
    };
  });
  steps_sync();
  step_middle<-1, CLS>(a, s);
  blue_multiply<-1, CLS>(a, s);
  step_middle<1, CLS>(a, s);
  T en = T(0);
  radix_switch<CLS, false>(a.Ra, [&](auto rc) {
    constexpr int R = rc;
    if constexpr (R % 2 == 0) {
      tasks(a, a.NRa, a.mNRa, [&](int t, int b) {
        int line, pl;
        const bool ok = at(t, &line, &pl);
        const T* Kp = static_cast<const T*>(a.K) + (long long)min(pl, a.Lp - pl) * a.Ksp +
                      (long long)min(line, a.Lt - line) * a.Kst;
        C* p = s.sh + t * a.ls + b * a.es;
        C x[R];
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = p[r * a.s1];
        dft_pre<R, 1>(x, s.tw, b, a.NRa);
        T el = T(0);
#pragma unroll
        for (int r = 0; r < R / 2; ++r) {
          const int k = b + r * a.NRa;
          const T kk = ok && k < a.Nt ? __ldg(Kp + (long long)min(k, a.Nt - k) * a.Kse) : T(0);
          const C u = mk(kk * x[r].x, kk * x[r].y);
          el = mad(u.x, x[r].x, mad(u.y, x[r].y, el));
          x[r] = u;
        }
        const int k0 = a.w_tile ? line : pl;
        en = mad(k0 == 0 || 2 * k0 == a.La0 ? T(1) : T(2), el, en);
        dft<R, -1, full_mask(R / 2)>(x);
#pragma unroll
        for (int r = 0; r < R; ++r) p[r * a.s1] = x[r];
      });
    }
  });
  if (a.E != nullptr) energy_lanes(en, wsum);
  __syncthreads();
  if (a.E != nullptr && threadIdx.x == 0) energy_cta_sum(a, wsum);
  step_middle<-1, CLS>(a, s);
  blue_multiply<1, CLS>(a, s);
  step_middle<1, CLS>(a, s);
  step_final<true, CLS>(a, s, [&](int t) {
    bool ok;
    C* dst = ptr(t, &ok);
    return [&a, dst, ok](C*, int e, C v) {
      if (ok && e < a.nout) dst[(long long)e * a.se_out] = mul_w<1>(v, chirp<C>(a, e));
    };
  });
}

template <typename T, bool PAIR, int CLS>
__global__ void __launch_bounds__(256, Bounds<T, CLS>::more) k_blue_r2c(const __grid_constant__ TileArgs a) {
  using C = cpx<T>;
  extern __shared__ __align__(16) unsigned char raw[];
  const Tile<C> s = tile_setup<C>(a, raw);
  pdl_wait();
  blue_conv<-1, CLS>(
      a, s,
      [&](int t) {
        const RealLine<T, PAIR> r(a, a.rsrc, a.sp_in, a.st_in, t);
        return [&a, r](C*, int e) { return e < a.nin ? mul_w<-1>(r.load(a, e), chirp<C>(a, e)) : mk(T(0), T(0)); };
      },
      [&](int) {
        return [&a](C* p, int e, C v) {
          if (e < a.Nt) *p = mul_w<-1>(v, chirp<C>(a, e));
        };
      });
  __syncthreads();
  tasks(a, a.Nt / 2 + 1, a.mout, [&](int t, int k) {
    const C* z = s.sh + t * a.ls;
    untangle<T, PAIR>(a, t, k, a.Nt, z[n_pos(a, k)], z[n_pos(a, k == 0 ? 0 : a.Nt - k)]);
  });
}

template <typename T, bool PAIR, int CLS>
__global__ void __launch_bounds__(256, Bounds<T, CLS>::more) k_blue_c2r(const __grid_constant__ TileArgs a) {
  using C = cpx<T>;
  extern __shared__ __align__(16) unsigned char raw[];
  if (energy_cta(a)) return;
  const Tile<C> s = tile_setup<C>(a, raw);
  const int N = a.Nt;
  pdl_wait();
  tasks(a, N / 2 + 1, a.mout, [&](int t, int k) {
    C zk, zm;
    tangle<T, PAIR>(a, t, k, N, &zk, &zm);
    C* z = s.sh + t * a.ls;
    z[n_pos(a, k)] = mul_w<1>(zk, chirp<C>(a, k));
    if (k != 0 && 2 * k != N) z[n_pos(a, N - k)] = mul_w<1>(zm, chirp<C>(a, N - k));
  });
  __syncthreads();
  blue_conv<1, CLS>(
      a, s, [&](int) { return [&a](C* p, int e) { return e < a.Nt ? *p : mk(T(0), T(0)); }; },
      [&](int t) {
        const RealLine<T, PAIR> r(a, a.rdst, a.sp_out, a.st_out, t);
        return [&a, r](C*, int e, C v) {
          if (e < a.nout) r.store(a, e, mul_w<1>(v, chirp<C>(a, e)));
        };
      });
}

}  // namespace tile
}  // namespace ps
