// Specialised FP32 kernels for the y and z passes, power-of-two lengths and
// 96 = 24 x 4, 192 = 24 x 8 (radix-3 register DFTs).
//
// A CTA owns 16 lines adjacent in kx (the contiguous axis of A and B), so a
// warp reads or writes two runs of 16 consecutive complex numbers (2 x 128 B)
// per instruction; at L = 1024, 8 lines (64-byte runs), which keeps a CTA at
// 256 threads and 64 KB of shared memory. Each line of length L = P * Q is transformed by T = min(P, Q)
// threads with the four-step factorisation
//     X[k1 + P k2] = sum_b W_Q^{b k2} W_L^{b k1} sum_a x[b + Q a] W_P^{a k1},
// step 1 (P-point DFTs over a) and step 3 (Q-point DFTs over b) in registers,
// one exchange through shared memory between them. With zero padding (§3)
// the inputs x[b + Q a] with a >= P/2 are zero and are never loaded; on the
// inverse, outputs with a >= P/2 are never formed. The z pass runs the
// forward transform, the K^F multiplication (Eq. 3) and the inverse in one
// kernel: the inverse's first step needs exactly the k1 values the forward's
// last step left in each thread, so the spectrum never leaves registers.
#include "fft_fast.cuh"
#include "fft_regs.cuh"
#include "reduce.cuh"
#include "tile_dft.cuh"

namespace ps {

using regs::rdft;
using tile::dft;
using tile::dft_pre;
using tile::full_mask;

// The four transforms of a line: columns b forward (P points over a, then the twiddles
// W_L^{b k1}), rows k1 forward and inverse (Q points), columns inverse (the
// conjugate twiddles, then P points). FOLD (fft_fast.cuh: the z pass and the inverse y pass at
// L = 1024): the twiddles are folded into the radix-2 layers of the transform that follows
// them (480 operations for 32 points behind twiddles instead of about 570; the z pass at
// 512^3 2202 -> 2158 us, the inverse y pass 579 -> 564 us), on the table of (cos, tan) pairs, at a
// rounding error below that of separate products (32 x 16 x 1024 periodic, round trip of a
// solve: separate 2.45e-7, folded 2.04e-7). The forward y pass spills 28 bytes in that form
// (581 -> 620 us), and the shorter lengths gain no time by it.
template <int P, int Q, int KIND>
constexpr bool kFold = folded_twiddles(P * Q, KIND);

template <int P, int Q, bool HALF, bool FOLD>
__device__ __forceinline__ void col_fwd(float2 (&y)[P], const float2* tw, int b) {
  if constexpr (FOLD) {
    dft<P, -1, full_mask(HALF ? P / 2 : P)>(y);
  } else {
    rdft<P, -1, HALF>(y);
#pragma unroll
    for (int k1 = 1; k1 < P; ++k1) y[k1] = cmul(y[k1], tw[b * k1]);
  }
}
template <int P, int Q, bool FOLD>
__device__ __forceinline__ void row_fwd(float2 (&x)[Q], const float2* tw, int k1) {
  if constexpr (FOLD) dft_pre<Q, -1>(x, tw, k1, P);
  else rdft<Q, -1, false>(x);
}
template <int P, int Q, bool FOLD>
__device__ __forceinline__ void row_inv(float2 (&x)[Q], const float2* tw, int k1) {
  if constexpr (FOLD) {
    dft<Q, 1, full_mask(Q)>(x);
  } else {
    rdft<Q, 1, false>(x);
#pragma unroll
    for (int b = 1; b < Q; ++b) x[b] = cmulc(x[b], tw[b * k1]);
  }
}
template <int P, int Q, bool FOLD>
__device__ __forceinline__ void col_inv(float2 (&y)[P], const float2* tw, int b) {
  if constexpr (FOLD) dft_pre<P, 1>(y, tw, b, Q);
  else rdft<P, 1, false>(y);
}

constexpr int kTK = 16;  // lines per CTA

// z pass: rows ky and L2 - ky read the same row of the K^F octant; launch
// them from adjacent CTA rows (y = 0 -> ky = 0, y = 1 -> ky = L2/2, then
// pairs p, L2 - p) so the second read hits L2.
template <int P, int Q, int KIND, bool HALF, int TK>
__global__ void __launch_bounds__(TK*(P < Q ? P : Q),
                                  TK * (P < Q ? P : Q) <= 256 ? (KIND == 2 ? 2 : 3) : 1)
    k_strided(const void* src_v, void* dst_v, const float* __restrict__ K, const float2* __restrict__ tw,
              FastArgs a, double* partials, unsigned* counter, double escale, double* E) {
  pdl_wait();
  constexpr int L = P * Q;
  constexpr int T = P < Q ? P : Q;
  constexpr int NB = Q / T;            // step-1 transforms per thread
  constexpr int NK = P / T;            // step-3 transforms per thread
  constexpr int NA = HALF ? P / 2 : P; // a-range of the nonzero inputs / kept outputs
  extern __shared__ float2 sh[];       // [L][TK]: element e of line t at e * TK + t
  const float2* src = static_cast<const float2*>(src_v);
  float2* dst = static_cast<float2*>(dst_v);
  const int t = threadIdx.x % TK;
  const int j = threadIdx.x / TK;
  const int kx = blockIdx.x * TK + t;
  const bool valid = kx < a.c;
  const int yblk = KIND == 2 ? paired_ky(blockIdx.y, a.L2)
                             : (a.rev ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y);
  const float2* s = src + yblk * a.src_plane + kx;
  float2* d = dst + yblk * a.dst_plane + kx;
  float2 X[NK][Q];  // X[v][k2] = spectrum at k1 + P k2, k1 = j + T v

  if constexpr (KIND == 0 || KIND == 2) {
    float2 y[NB][P];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int b = j + T * u;
#pragma unroll
      for (int aa = 0; aa < P; ++aa) {
        y[u][aa] = make_float2(0.f, 0.f);
        if (aa < NA && valid && b + Q * aa < a.nl) y[u][aa] = s[(long long)(b + Q * aa) * a.src_elem];
      }
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int b = j + T * u;
      col_fwd<P, Q, HALF, kFold<P, Q, KIND>>(y[u], tw, b);
#pragma unroll
      for (int k1 = 0; k1 < P; ++k1) sh[(b * P + k1) * TK + t] = y[u][k1];
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < NK; ++v) {
      const int k1 = j + T * v;
#pragma unroll
      for (int b = 0; b < Q; ++b) X[v][b] = sh[(b * P + k1) * TK + t];
      row_fwd<P, Q, kFold<P, Q, KIND>>(X[v], tw, k1);
    }
  } else {
#pragma unroll
    for (int v = 0; v < NK; ++v) {
      const int k1 = j + T * v;
#pragma unroll
      for (int k2 = 0; k2 < Q; ++k2)
        X[v][k2] = valid ? s[(long long)(k1 + P * k2) * a.src_elem] : make_float2(0.f, 0.f);
    }
  }

  if constexpr (KIND == 0) {
    if (valid) {
#pragma unroll
      for (int v = 0; v < NK; ++v) {
        const int k1 = j + T * v;
#pragma unroll
        for (int k2 = 0; k2 < Q; ++k2) d[(long long)(k1 + P * k2) * a.dst_elem] = X[v][k2];
      }
    }
    return;
  } else {
    float eacc = 0.f;
    if constexpr (KIND == 2) {
      // V^F = K^F rho^F on the even octant of K^F; energy sum w(kx) K |rho^F|^2
      const int ky = yblk;
      const int kyo = min(ky, a.L2 - ky);
      const float* Kp = K + (long long)kyo * a.ldk + kx;
#pragma unroll
      for (int v = 0; v < NK; ++v) {
        const int k1 = j + T * v;
#pragma unroll
        for (int k2 = 0; k2 < Q; ++k2) {
          const int kz = k1 + P * k2;
          const int kzo = kz <= L / 2 ? kz : L - kz;
          const float kk = valid ? __ldg(&Kp[(long long)kzo * a.kz_stride]) : 0.f;
          const float2 x = X[v][k2];
          eacc = fmaf(kk, x.x * x.x + x.y * x.y, eacc);
          X[v][k2] = make_float2(kk * x.x, kk * x.y);
        }
      }
      eacc *= (kx == 0 || 2 * kx == a.L1) ? 1.f : 2.f;
    }
    // inverse: Q-point transforms over k2, exchange, conjugate twiddles and
    // P-point transforms over k1
#pragma unroll
    for (int v = 0; v < NK; ++v) row_inv<P, Q, kFold<P, Q, KIND>>(X[v], tw, j + T * v);
    // (KIND 2: back to the slots this thread read its rows from, no barrier before)
#pragma unroll
    for (int v = 0; v < NK; ++v) {
      const int k1 = j + T * v;
#pragma unroll
      for (int b = 0; b < Q; ++b) sh[(b * P + k1) * TK + t] = X[v][b];
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int b = j + T * u;
      float2 y[P];
#pragma unroll
      for (int k1 = 0; k1 < P; ++k1) y[k1] = sh[(b * P + k1) * TK + t];
      col_inv<P, Q, kFold<P, Q, KIND>>(y, tw, b);
      if (valid) {
#pragma unroll
        for (int aa = 0; aa < NA; ++aa)
          if (b + Q * aa < a.nl) d[(long long)(b + Q * aa) * a.dst_elem] = y[aa];
      }
    }
    if constexpr (KIND == 2) {
      if (E != nullptr) energy_partial_f32(eacc, partials);
    }
  }
}

template <int P, int Q, int TK = kTK>
static const void* pick_strided(int kind, bool half) {
  if (kind == 0) return half ? (const void*)k_strided<P, Q, 0, true, TK> : (const void*)k_strided<P, Q, 0, false, TK>;
  if (kind == 1) return half ? (const void*)k_strided<P, Q, 1, true, TK> : (const void*)k_strided<P, Q, 1, false, TK>;
  return half ? (const void*)k_strided<P, Q, 2, true, TK> : (const void*)k_strided<P, Q, 2, false, TK>;
}

// L = 1024 takes 8 lines per CTA (256 threads, 64 KB of shared memory); the
// shorter lengths 16
const void* strided_kernel(int L, int kind, bool half, int* threads, size_t* smem, int* tk) {
  const void* fn = nullptr;
  int T = 0, TK = kTK;
  switch (L) {
    case 64: fn = pick_strided<8, 8>(kind, half); T = 8; break;
    case 128: fn = pick_strided<16, 8>(kind, half); T = 8; break;
    case 256: fn = pick_strided<16, 16>(kind, half); T = 16; break;
    case 512: fn = pick_strided<16, 32>(kind, half); T = 16; break;
    case 1024: fn = pick_strided<32, 32, 8>(kind, half); T = 32; TK = 8; break;
    default: return nullptr;
  }
  *threads = TK * T;
  *smem = (size_t)L * TK * sizeof(float2);
  *tk = TK;
  return fn;
}

// ---------------------------------------------------------------- pipelined z

// Persistent z pass on unpacked lines (L3 = 256, and 1024, where a packed pair
// of 32-point transforms would not fit in registers): TK lines per tile, tiles
// = (kx tile, ky row in the paired order) with kx fastest. The tile's n3 input
// rows land in the exchange (cp.async), the K^F octant slice in a stage of its
// own; the next tile's K^F slice is copied once the current one has been
// used (after a CTA barrier), its input rows once the warp has read the exchange for the
// last time: a warp copies the rows that its own threads read, into slots that
// only they write.
// With 8 lines per tile (64-byte exchange rows) the exchange has one padding
// row after every 32: the four line positions j of a warp then write rows 33
// apart, on alternate halves of the banks, instead of 32 apart on the same
// 16 banks (a 4-way conflict in the forward write and the inverse read).
template <int P, int Q, bool HALF, int TK>
__global__ void __launch_bounds__(TK*(P < Q ? P : Q), P > Q ? 512 / (TK * Q) : (P * Q >= 1024 ? 2 : 3))
    k_zpipe_u(const void*, void* line_v, const float* __restrict__ K, const float2* __restrict__ tw, FastArgs a,
              double* partials, unsigned* counter, double escale, double* E) {
  constexpr int L = P * Q;
  constexpr int T = P < Q ? P : Q;
  constexpr int NB = Q / T;
  constexpr int NK = P / T;
  constexpr int NA = HALF ? P / 2 : P;
  constexpr int KROWS = L / 2 + 1;  // rows of the K^F octant
  constexpr int RG = TK * 8 < 128 ? P : 0;  // exchange rows per padded group (0: no padding)
  static_assert(RG == 0 || (P == RG && Q == RG), "padded exchange: P = Q = rows per group");
  constexpr int PP = RG ? P + 1 : P;         // row pitch of b in the exchange (rows b * PP + k1)
  constexpr int LP = RG ? L + L / RG : L;    // exchange rows including the padding
  extern __shared__ float2 sh[];    // exchange [LP][TK]; the K^F slice [KROWS][TK] floats; W_L^i, i < L
  float* const kstage = reinterpret_cast<float*>(sh + LP * TK);
  float2* const tws = reinterpret_cast<float2*>(kstage + ((KROWS * TK + 1) & ~1));
  for (int i = threadIdx.x; i < L; i += blockDim.x) tws[i] = __ldg(&tw[i]);  // before the first barrier
  float2* const base = static_cast<float2*>(line_v);
  const int t = threadIdx.x % TK;
  const int j = threadIdx.x / TK;
  const int ntk = a.ntk_loc;
  const int ntiles = ntk * a.L2;
  const long long es = a.src_elem;

  constexpr int NT = TK * T;
  constexpr int IPR = TK / 2;  // 16-byte pieces per input row
  // the rows b + Q aa of column b land in the exchange rows (b, aa), which only the
  // threads of column b (j = b) read and then write, copied by their own warp two aa at a time:
  // the inputs need no barrier of the CTA
  static_assert(NB == 1 && NA % 2 == 0 && 32 % TK == 0, "input copy shape");
  constexpr int GPW = 32 / TK;  // columns per warp
  const int lj = (threadIdx.x / 32) * GPW + (threadIdx.x % 32) / IPR % GPW, lh = (threadIdx.x % 32) / (IPR * GPW);
  const int irow0 = lj + Q * lh;
  const long long igoff = (long long)irow0 * es + 2 * (threadIdx.x % IPR);
  const long long igstep = (long long)(2 * Q) * es;
  float2* const is0 = sh + (lj * PP + lh) * TK + 2 * (threadIdx.x % IPR);
  const int ivalid = a.nl - irow0;
  constexpr int KPR = TK / 4;  // 16-byte pieces per K^F row
  constexpr int KSTEP = NT / KPR;
  constexpr int KIT = (KROWS + KSTEP - 1) / KSTEP;
  const int krow0 = threadIdx.x / KPR;
  const long long kgoff = (long long)krow0 * a.kz_stride + 4 * (threadIdx.x % KPR);
  const long long kgstep = (long long)KSTEP * a.kz_stride;
  float* const ks0 = kstage + krow0 * TK + 4 * (threadIdx.x % KPR);

  const int dkt = gridDim.x % ntk, dyi = gridDim.x / ntk;
  auto step_tile = [&](int& kt, int& yi) {
    kt += dkt;
    yi += dyi;
    if (kt >= ntk) {
      kt -= ntk;
      ++yi;
    }
  };
  auto issue_input = [&](int kt, int yi) {
    const float2* src0 = base + paired_ky(yi, a.L2) * a.src_plane + (a.kt0 + kt) * TK;
    const float2* src = src0 + igoff;
#pragma unroll
    for (int i = 0; i < NA / 2; ++i) {
      if (2 * Q * i < ivalid)
        cp_async16(is0 + i * 2 * TK, src);
      else  // beyond the physical z rows: zeros (nothing is read)
        cp_async16_zero(is0 + i * 2 * TK, src0);
      src += igstep;
    }
  };
  auto issue_k = [&](int kt, int yi) {
    const int ky = paired_ky(yi, a.L2);
    const int kyo = min(ky, a.L2 - ky);
    const float* src = K + (long long)kyo * a.ldk + (a.kt0 + kt) * TK + kgoff;
#pragma unroll
    for (int i = 0; i < KIT; ++i) {
      if ((i + 1) * KSTEP <= KROWS || krow0 + i * KSTEP < KROWS) cp_async16(ks0 + i * KSTEP * TK, src);
      src += kgstep;
    }
  };

  float eacc = 0.f;
  int tile = blockIdx.x;
  int kt = tile % ntk, yi = tile / ntk;
  int nkt = kt, nyi = yi;
  step_tile(nkt, nyi);
  if (tile < ntiles) issue_k(kt, yi);  // K^F is not written by any pass
  pdl_wait();
  if (tile < ntiles) issue_input(kt, yi);
  cp_async_commit();
  __syncthreads();  // the twiddle table
  for (; tile < ntiles; tile += gridDim.x) {
    const int next = tile + gridDim.x;
    const int kx = (a.kt0 + kt) * TK + t;
    const bool valid = kx < a.c;
    const int ky = paired_ky(yi, a.L2);
    float2* line = base + ky * a.src_plane + kx;
    cp_async_wait_all();
    __syncwarp();  // the warp's input rows have landed; the K^F slice is read after the next barrier

    float2 y[NB][P];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int b = j + T * u;
#pragma unroll
      for (int aa = 0; aa < P; ++aa) {
        y[u][aa] = make_float2(0.f, 0.f);
        if (aa < NA && valid) y[u][aa] = sh[(b * PP + aa) * TK + t];
      }
    }
    __syncwarp();  // inputs read: the warp's rows become the exchange
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int b = j + T * u;
      col_fwd<P, Q, HALF, kFold<P, Q, 2>>(y[u], tws, b);
#pragma unroll
      for (int k1 = 0; k1 < P; ++k1) sh[(b * PP + k1) * TK + t] = y[u][k1];
    }
    __syncthreads();
    float2 X[NK][Q];
    float e1 = 0.f;
#pragma unroll
    for (int v = 0; v < NK; ++v) {
      const int k1 = j + T * v;
#pragma unroll
      for (int b = 0; b < Q; ++b) X[v][b] = sh[(b * PP + k1) * TK + t];
      row_fwd<P, Q, kFold<P, Q, 2>>(X[v], tws, k1);
      // V^F = K^F rho^F on the even octant of K^F; energy sum K |rho^F|^2
#pragma unroll
      for (int k2 = 0; k2 < Q; ++k2) {
        const int kz = k1 + P * k2;
        const int kzo = kz <= L / 2 ? kz : L - kz;
        const float kk = valid ? kstage[kzo * TK + t] : 0.f;
        const float2 x = X[v][k2];
        e1 = fmaf(kk, x.x * x.x + x.y * x.y, e1);
        X[v][k2] = make_float2(kk * x.x, kk * x.y);
      }
      row_inv<P, Q, kFold<P, Q, 2>>(X[v], tws, k1);
    }
    eacc += e1 * ((kx == 0 || 2 * kx == a.L1) ? 1.f : 2.f);
    // back to the slots this thread read its rows from: no barrier before
#pragma unroll
    for (int v = 0; v < NK; ++v) {
      const int k1 = j + T * v;
#pragma unroll
      for (int b = 0; b < Q; ++b) sh[(b * PP + k1) * TK + t] = X[v][b];
    }
    __syncthreads();  // the K^F slice has been read too
    if (next < ntiles) issue_k(nkt, nyi);
    cp_async_commit();
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int b = j + T * u;
#pragma unroll
      for (int k1 = 0; k1 < P; ++k1) y[u][k1] = sh[(b * PP + k1) * TK + t];
    }
    __syncwarp();  // the warp has read its rows: the next tile's may land in them
    if (next < ntiles) issue_input(nkt, nyi);
    cp_async_commit();
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int b = j + T * u;
      col_inv<P, Q, kFold<P, Q, 2>>(y[u], tws, b);
      if (valid) {
#pragma unroll
        for (int aa = 0; aa < NA; ++aa)
          if (b + Q * aa < a.nl) line[(long long)(b + Q * aa) * es] = y[u][aa];
      }
    }
    kt = nkt;
    yi = nyi;
    step_tile(nkt, nyi);
  }
  cp_async_wait_all();
  if (E != nullptr) energy_partial_f32(eacc, partials);
}

const void* zpipe_u_kernel(int L, bool half, int* threads, size_t* smem, int* tk) {
  const void* fn = nullptr;
  int T = 0, TK = 8;
  switch (L) {
    case 96:  // 24 x 4 and 24 x 8 (radix-3 register DFTs), 16 lines per tile
      fn = half ? (const void*)k_zpipe_u<24, 4, true, 16> : (const void*)k_zpipe_u<24, 4, false, 16>;
      T = 4;
      TK = 16;
      break;
    case 192:
      fn = half ? (const void*)k_zpipe_u<24, 8, true, 16> : (const void*)k_zpipe_u<24, 8, false, 16>;
      T = 8;
      TK = 16;
      break;
    case 1024: fn = half ? (const void*)k_zpipe_u<32, 32, true, 8> : (const void*)k_zpipe_u<32, 32, false, 8>; T = 32;
      break;
    default: return nullptr;
  }
  *threads = TK * T;
  const int LP = TK * 8 < 128 ? L + L / T : L;  // exchange rows, with the kernel's padding rows
  *smem = (size_t)LP * TK * sizeof(float2) + (size_t)(((L / 2 + 1) * TK + 1) & ~1) * sizeof(float) +
          (size_t)L * sizeof(float2);
  *tk = TK;
  return fn;
}

// ---------------------------------------------------------------- pipelined y

// Persistent y pass (KIND 0 forward, 1 inverse), 16 lines per tile, tiles =
// (kx tile, z plane) with kx fastest. The shared-memory tile serves twice: as
// the landing area of the tile's input rows (copied with cp.async) and as the
// exchange of the four-step transform. Once a tile's exchange has been read,
// the next tile's rows are copied in while the last transform step and the
// stores of the current tile run. With 8 lines per tile (64-byte rows) the
// exchange has one padding row after every 32, as in the L = 1024 z kernel:
// the forward write and the inverse read of a warp then fall on alternate
// bank halves instead of 4-way on the same 16 banks. The input rows land in the
// exchange's own (padded) slots: forward, row b + Q aa in (b, aa), inverse, row k1 + P k2
// in (k2, k1). A warp copies exactly the rows that its threads read, and overwrites
// exactly their slots with its half of the exchange, so __syncwarp orders the copy, the
// reads and the writes; the exchange is then read across the warps, between two CTA
// barriers, the second before the next tile's copies.
template <int P, int Q, int KIND, bool HALF, int TK>
__global__ void __launch_bounds__(TK*(P < Q ? P : Q), P > Q ? 512 / (TK * Q) : (P * Q >= 512 ? 2 : 3))
    k_ypipe(const void* src_v, void* dst_v, const float*, const float2* __restrict__ tw, FastArgs a, double*,
            unsigned*, double, double*) {
  pdl_wait();
  constexpr int T = P < Q ? P : Q;
  constexpr int NB = Q / T;
  constexpr int NK = P / T;
  constexpr int NA = HALF ? P / 2 : P;
  constexpr int RG = TK * 8 < 128 ? P : 0;      // exchange rows per padded group (0: no padding)
  static_assert(RG == 0 || (P == RG && Q == RG), "padded exchange: P = Q = rows per group");
  constexpr int PP = RG ? P + 1 : P;             // row pitch of b in the exchange (rows b * PP + k1)
  extern __shared__ float2 sh[];               // the exchange [L + L / RG][TK]; the inputs land in its rows
  const float2* src = static_cast<const float2*>(src_v);
  float2* dst = static_cast<float2*>(dst_v);
  const int t = threadIdx.x % TK;
  const int j = threadIdx.x / TK;
  const int ntk = a.ntk_loc;  // kx tiles a.kt0 .. a.kt0 + ntk - 1
  const int ntiles = ntk * (int)a.nrows;  // nrows = number of z planes here

  // the input copy: rows of TK float2 in 16-byte pieces, per-thread offsets
  // computed once
  constexpr int NT = TK * T;
  constexpr int IPR = TK / 2;
  // the rows land where only the threads that read them write next, copied by their
  // own warp (no CTA barrier for the inputs): forward, row b + Q aa in the exchange row (b, aa), b = j + T u;
  // inverse, row k1 + P k2 in (k2, k1), k1 = j + T v
  static_assert(NA % 2 == 0 && Q % 2 == 0 && 32 % TK == 0 && NT % 32 == 0, "input copy shape");
  constexpr int GPW = 32 / TK;  // thread groups j per warp
  const int lj = (threadIdx.x / 32) * GPW + (threadIdx.x % 32) / IPR % GPW, lh = (threadIdx.x % 32) / (IPR * GPW);
  const int irow0 = lj + (KIND == 0 ? Q : P) * lh;
  const long long igoff = (long long)irow0 * a.src_elem + 2 * (threadIdx.x % IPR);
  float2* const is0 = sh + (KIND == 0 ? lj * PP + lh : lh * PP + lj) * TK + 2 * (threadIdx.x % IPR);
  const int ivalid = a.nl - irow0;  // forward: a copy is of a physical row iff 2 Q i + T u < ivalid
  auto plane = [&](int zi) { return a.rev ? (int)a.nrows - 1 - zi : zi; };
  auto prefetch = [&](int kt, int zi) {
    const float2* sp0 = src + (long long)plane(zi) * a.src_plane + (a.kt0 + kt) * TK;
    const float2* sp = sp0 + igoff;
    if constexpr (KIND == 0) {
      const long long ustep = (long long)T * a.src_elem, step = (long long)(2 * Q) * a.src_elem;
#pragma unroll
      for (int i = 0; i < NA / 2; ++i) {
#pragma unroll
        for (int u = 0; u < NB; ++u) {
          if (2 * Q * i + T * u < ivalid)
            cp_async16(is0 + (T * u * PP + i * 2) * TK, sp + u * ustep);
          else  // beyond the physical rows of the plane: zeros
            cp_async16_zero(is0 + (T * u * PP + i * 2) * TK, sp0);
        }
        sp += step;
      }
    } else {
      const long long vstep = (long long)T * a.src_elem, step = (long long)(2 * P) * a.src_elem;
#pragma unroll
      for (int i = 0; i < Q / 2; ++i) {
#pragma unroll
        for (int v = 0; v < NK; ++v) cp_async16(is0 + (i * 2 * PP + T * v) * TK, sp + v * vstep);
        sp += step;
      }
    }
  };
  // tile = kt + ntk * zi (kx tile fastest); the CTA steps by gridDim.x tiles
  const int dkt = gridDim.x % ntk, dzi = gridDim.x / ntk;
  auto step_tile = [&](int& kt, int& zi) {
    kt += dkt;
    zi += dzi;
    if (kt >= ntk) {
      kt -= ntk;
      ++zi;
    }
  };

  int tile = blockIdx.x;
  int kt = tile % ntk, zi = tile / ntk;
  int nkt = kt, nzi = zi;
  step_tile(nkt, nzi);
  if (tile < ntiles) prefetch(kt, zi);
  cp_async_commit();
  for (; tile < ntiles; tile += gridDim.x) {
    const int next = tile + gridDim.x;
    const int kx = (a.kt0 + kt) * TK + t;
    const bool valid = kx < a.c;
    float2* d = dst + (long long)plane(zi) * a.dst_plane + kx;
    cp_async_wait_all();
    __syncwarp();  // the warp's rows have landed
    float2 X[NK][Q];
    if constexpr (KIND == 0) {
      float2 y[NB][P];
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        const int b = j + T * u;
#pragma unroll
        for (int aa = 0; aa < P; ++aa) {
          y[u][aa] = make_float2(0.f, 0.f);
          if (aa < NA && valid) y[u][aa] = sh[(b * PP + aa) * TK + t];
        }
      }
      __syncwarp();  // inputs read: the warp's rows become the exchange
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        const int b = j + T * u;
        col_fwd<P, Q, HALF, kFold<P, Q, KIND>>(y[u], tw, b);
#pragma unroll
        for (int k1 = 0; k1 < P; ++k1) sh[(b * PP + k1) * TK + t] = y[u][k1];
      }
      __syncthreads();
#pragma unroll
      for (int v = 0; v < NK; ++v) {
        const int k1 = j + T * v;
#pragma unroll
        for (int b = 0; b < Q; ++b) X[v][b] = sh[(b * PP + k1) * TK + t];
      }
      __syncthreads();  // exchange read: the next tile's rows may land
      if (next < ntiles) prefetch(nkt, nzi);
      cp_async_commit();
#pragma unroll
      for (int v = 0; v < NK; ++v) {
        const int k1 = j + T * v;
        row_fwd<P, Q, kFold<P, Q, KIND>>(X[v], tw, k1);
        if (valid) {
#pragma unroll
          for (int k2 = 0; k2 < Q; ++k2) d[(long long)(k1 + P * k2) * a.dst_elem] = X[v][k2];
        }
      }
    } else {
#pragma unroll
      for (int v = 0; v < NK; ++v) {
        const int k1 = j + T * v;
#pragma unroll
        for (int k2 = 0; k2 < Q; ++k2)
          X[v][k2] = valid ? sh[(k2 * PP + k1) * TK + t] : make_float2(0.f, 0.f);
      }
      __syncwarp();  // inputs read: the warp's rows become the exchange
#pragma unroll
      for (int v = 0; v < NK; ++v) {
        const int k1 = j + T * v;
        row_inv<P, Q, kFold<P, Q, KIND>>(X[v], tw, k1);
#pragma unroll
        for (int b = 0; b < Q; ++b) sh[(b * PP + k1) * TK + t] = X[v][b];
      }
      __syncthreads();
      float2 y[NB][P];
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        const int b = j + T * u;
#pragma unroll
        for (int k1 = 0; k1 < P; ++k1) y[u][k1] = sh[(b * PP + k1) * TK + t];
      }
      __syncthreads();  // exchange read: the next tile's rows may land
      if (next < ntiles) prefetch(nkt, nzi);
      cp_async_commit();
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        const int b = j + T * u;
        col_inv<P, Q, kFold<P, Q, KIND>>(y[u], tw, b);
        if (valid) {
#pragma unroll
          for (int aa = 0; aa < NA; ++aa)
            if (b + Q * aa < a.nl) d[(long long)(b + Q * aa) * a.dst_elem] = y[u][aa];
        }
      }
    }
    kt = nkt;
    zi = nzi;
    step_tile(nkt, nzi);
  }
  cp_async_wait_all();
}

template <int P, int Q, int TK = kTK>
static const void* pick_ypipe(int kind, bool half) {
  if (kind == 0) return half ? (const void*)k_ypipe<P, Q, 0, true, TK> : (const void*)k_ypipe<P, Q, 0, false, TK>;
  return half ? (const void*)k_ypipe<P, Q, 1, true, TK> : (const void*)k_ypipe<P, Q, 1, false, TK>;
}

const void* ypipe_kernel(int L, int kind, bool half, int* threads, size_t* smem, int* tk) {
  const void* fn = nullptr;
  int T = 0, TK = kTK;
  switch (L) {
    case 96: fn = pick_ypipe<24, 4>(kind, half); T = 4; break;    // 24 x 4 (radix-3 register DFTs)
    case 192: fn = pick_ypipe<24, 8>(kind, half); T = 8; break;   // 24 x 8
    case 256: fn = pick_ypipe<16, 16>(kind, half); T = 16; break;
    case 512: fn = pick_ypipe<16, 32>(kind, half); T = 16; break;
    case 1024: fn = pick_ypipe<32, 32, 8>(kind, half); T = 32; TK = 8; break;
    default: return nullptr;
  }
  *threads = TK * T;
  const int LP = TK * 8 < 128 ? L + L / T : L;  // exchange rows, with the kernel's padding rows
  *smem = (size_t)LP * TK * sizeof(float2);
  *tk = TK;
  return fn;
}

}  // namespace ps
