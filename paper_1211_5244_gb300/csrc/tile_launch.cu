// Host side of the tile kernels (tile_pass.cuh): which passes run on them, the
// factorisation of a length into register steps, tile shapes and launches.
#include <algorithm>

#include "common.cuh"

namespace ps {
namespace {

// operations of an R-point register DFT (tile_dft.cuh), for comparing factorisations (9 points take
// eight less, which their pairs behind constant twiddles save)
double dft_ops(int R) {
  if (R == 1) return 0.0;
  if ((R & (R - 1)) == 0) {
    double f = 0.0;  // two trivial butterflies of 4 per layer, six operations for the others
    for (int m = 2; m <= R; m *= 2) f += (double)(R / m) * (m == 2 ? 4.0 : 8.0 + 6.0 * (m / 2 - 2));
    return f;
  }
  int p = 2;
  while (R % p) ++p;
  if (p == R) return p == 3 ? 12.0 : (double)(p - 1) * (p + 3);
  int A = p;
  while (R % (A * p) == 0) A *= p;
  if (A < R) return (R / A) * dft_ops(A) + A * dft_ops(R / A);
  return p * dft_ops(R / p) + (R / p) * dft_ops(p) + 4.0 * (p - 1) * (R / p - 1);
}

// ... behind twiddles: folded into the layers of a power of two, else four each
// less two per first pair
double dft_pre_ops(int R) {
  if ((R & (R - 1)) == 0) {
    double f = 0.0;
    for (int m = 2; m <= R; m *= 2) f += (double)(R / m) * 6.0 * (m / 2);
    return f;
  }
  return dft_ops(R) + 4.0 * (R - 1) - 2.0 * (R / 3);
}

}  // namespace

// The factorisation with the least operations per element; in FP32 a step
// counts two more (its shared-memory round trip, address arithmetic and barrier:
// measured over 21 lengths from 50 to 600, the rule is within 1.2% of the best
// factorisation of each). A radix of 2 spends a step on one butterfly layer,
// and larger radices take more registers (0.2 per point). In FP64 the pipe's
// operations are the time: 256 = 8 x 4 x 8 and 16 x 16 take 224 us each for 10368
// lines, 200 = 10 x 4 x 5 219 us where 10 x 2 x 10 takes 254.
// A length with one prime factor from 17 to 31 takes it as its last radix: about p + 3
// operations per element, where the Bluestein convolution of passes.cu runs two
// transforms of at least twice the length.
bool tile_radix(int N, bool even_first, bool f32, TileRadix* out, double* cost) {
  constexpr int kMax = 16;
  const double step = f32 ? 2.0 : 0.0;
  auto small = [](int R) { return R == 2 ? 4.0 : 0.0; };
  double best = -1.0;
  auto consider = [&](int Ra, int Rm, int Rl, int cls) {
    const int most = std::max(Ra, std::max(Rm, Rl));
    double c = dft_ops(Ra) / Ra + dft_pre_ops(Rl) / Rl + 2 * step + small(Ra) + small(Rl) + 0.2 * most;
    if (Rm > 1) c += dft_pre_ops(Rm) / Rm + step + small(Rm);
    if (best < 0.0 || c < best) {
      best = c;
      *out = TileRadix{Ra, Rm, Rl, cls};
      if (cost) *cost = c;
    }
  };
  for (int Ra = 2; Ra <= kMax; ++Ra) {
    if (N % Ra || (even_first && Ra % 2)) continue;
    const int q = N / Ra;
    for (int Rl = 2; Rl <= kMax; ++Rl)
      if (q % Rl == 0 && q / Rl <= kMax) consider(Ra, q / Rl, Rl, std::max(Ra, std::max(q / Rl, Rl)) > 8 ? 1 : 0);
  }
  if (best >= 0.0) return true;
  for (const int p : {17, 19, 23, 29, 31}) {
    if (N % p) continue;
    const int q = N / p;
    for (int Ra = q == 1 ? 1 : 2; Ra <= kMax; ++Ra)
      if (q % Ra == 0 && q / Ra <= kMax && !(even_first && Ra % 2)) consider(Ra, q / Ra, p, 2);
  }
  return best >= 0.0;
}

// The even M from 2 N (half of the convolution's input is zero) to 4 N with the
// least operations per line: its two transforms and the product with Bf.
int tile_blue_length(int N, bool f32, int max_M) {
  int best_M = 0;
  double best = 0.0;
  for (int M = 2 * N; M <= 4 * N && M <= max_M; M += 2) {
    TileRadix r;
    double c = 0.0;
    if (!tile_radix(M, true, f32, &r, &c) || r.cls == 2) continue;
    if (best_M == 0 || M * (2.0 * c + 6.0) < best) {
      best = M * (2.0 * c + 6.0);
      best_M = M;
    }
  }
  return best_M;
}

namespace {

// tile and plane axes of a pass along physical axis al
void tile_axes(int al, int* at, int* ap) {
  if (al == 0) {
    *at = 1;
    *ap = 2;
  } else {
    *at = 0;
    *ap = 3 - al;
  }
}

// Lines per tile (`want` where the plan's schedule sets it) and threads of a CTA.
//
// FP32 passes are bound by latency and issue: 8 threads per line (16 for N above
// 288, whose steps have more butterflies) on 16 lines, 8 lines for N above 160
// (L = 120 at 10368 lines: 12.1 us against 12.2 with 32 lines and 14.4 with one
// thread per butterfly; L = 240: 16.3 us against 18.3 with 32 lines; L = 320:
// 23.1 against 24.6).
//
// A fused z pass of few CTAs takes more threads per CTA: below 256 threads per SM
// the chip is idle for want of warps, and the steps of one tile are its time. The
// most threads whose last round of butterflies is not emptier by more than a tenth
// (90 x 75 x 110 ppf, L3 = 220, 450 CTAs: 64 -> 192 threads, solve 32.7 -> 28.5 us).
// With the line at 768 threads per SM a batch of 32 such problems, which fills the
// chip, goes from 865 to 894 us; the other passes gain nothing from more threads. (A plan
// does not know whether it runs alone: in a batch the other problems' CTAs fill the SMs, and
// the line lies between what that grid alone and that batch want.)
//
// In FP64 a warp instruction holds the pipe as long with one lane as with 32: the
// tile is the width with the fewest operations per SM, counting whole warps and
// whole tiles, and the threads those that split the steps' butterflies most evenly
// (L = 200, 8 lines: 160 threads 219 us, 128 threads 223 us). Tiles of 64-byte
// rows count 5% more.
// At most 72 KB, three CTAs per SM, else the widest tile that fits one.
struct TileShape { int tk, threads; };
TileShape pick_tile(const TileArgs& a, const TileRadix& r, int row, long long lines, int want, size_t esz, int sms,
                    bool conv) {
  const size_t csz = 2 * esz;
  const bool f32 = esz == 4;
  const int nb[3] = {a.NRa, a.Kl, r.Rm > 1 ? r.Ra * r.Rl : 0};
  const double ops[3] = {dft_ops(r.Ra), dft_pre_ops(r.Rl), dft_pre_ops(r.Rm)};
  auto bytes = [&](int tk) { return ((size_t)row * tk + a.N) * csz; };
  int tk = want;
  if (tk == 0 && f32) tk = a.Kl == 1 ? 32 : a.N <= 160 ? 16 : 8;
  if (tk == 0) {
    double best = -1.0;
    for (int v : {8, 16, 32, 4}) {
      if (bytes(v) > (size_t)72 * 1024) continue;
      double w = 0.0;
      for (int k = 0; k < 3; ++k) w += ((v * nb[k] + 31) / 32) * ops[k];
      double c = w * (double)((((lines + v - 1) / v) + sms - 1) / sms);
      if (v < 8) c *= 1.05;
      if (best < 0.0 || c < 0.97 * best) {
        best = c;
        tk = v;
      }
    }
    if (tk == 0) tk = 8;
  }
  while (tk > 1 && bytes(tk) > (size_t)72 * 1024) tk /= 2;
  if (bytes(tk) > (size_t)200 * 1024) return TileShape{0, 0};
  const int most = tk * std::max(nb[0], std::max(nb[1], nb[2]));
  const int cap = (std::min(most, 256) + 31) / 32 * 32;
  int threads = std::min(cap, std::max(64, (a.N <= 288 ? 8 : 16) * tk));
  auto rounds = [&](int th) {  // thread-operations of a CTA, idle threads of the last rounds counted
    double w = 0.0;
    for (int k = 0; k < 3; ++k) w += (double)((tk * nb[k] + th - 1) / th * th) * ops[k];
    return w;
  };
  const long long ctas = (lines + tk - 1) / tk;
  if (f32 && conv && ctas * threads < 256LL * sms) {
    const int base = threads;
    for (int th = base + 32; th <= cap; th += 32)
      if (rounds(th) <= 1.1 * rounds(base)) threads = th;
  }
  if (!f32) {
    double best = -1.0;
    for (int th = std::min(cap, 128); th <= cap; th += 32) {
      const double w = rounds(th);
      if (best < 0.0 || w < best) {
        best = w;
        threads = th;
      }
    }
  }
  return TileShape{tk, threads};
}

template <typename T>
cudaError_t configure_pass(ps_plan_s* p, int pass, int sms) {
  using C = cpx<T>;
  TileLaunch& tl = p->tile[pass];
  tl = TileLaunch{};
  const int al = pass_axis(p, pass);
  if (axis_radix(p, al) != 0) return cudaSuccess;  // the schedule asks for the Stockham stages
  const int N = xform_len(p, al), L = p->L[al], n = p->n[al];
  const bool real_pass = pass == P1 || pass == P5;
  const bool packed = real_pass && N != L;  // a real row of even length as N = L/2 complex points
  const bool half = 2 * n <= L;             // also for packed rows: (n + 1) / 2 <= N / 2 needs an even n or L > 2 n
  const int nin = packed ? (n + 1) / 2 : n;  // physical points of a line
  const bool zhalf = half && N % 2 == 0 && 2 * nin <= N;
  TileRadix r;
  const bool blue = !tile_radix(N, zhalf, sizeof(T) == 4, &r);
  const int M = blue ? p->blue[al].M : N;  // points of the steps
  if (blue && (M < 2 * N || !tile_radix(M, true, sizeof(T) == 4, &r) || r.cls == 2)) return cudaSuccess;
  tl.blue = blue;
  TileArgs& a = tl.a;
  a.N = M;
  a.Nt = N;
  a.Ra = r.Ra;
  a.Rm = r.Rm;
  a.Rl = r.Rl;
  a.NRa = M / r.Ra;
  a.Kl = r.Ra * r.Rm;
  a.mRa = div_magic((unsigned)a.Ra);
  a.mRm = div_magic((unsigned)a.Rm);
  a.mRl = div_magic((unsigned)a.Rl);
  a.mNRa = div_magic((unsigned)a.NRa);
  a.mNRm = div_magic((unsigned)(r.Ra * r.Rl));
  a.mKl = div_magic((unsigned)a.Kl);
  a.tws = blue ? 1 : L / N;
  a.lc = al == 0 ? 1 : 0;
  const int pad = (a.lc && a.NRa % 2 == 0) ? 1 : 0;  // odd stride of digit 1: rows of a step on different banks
  const int row = r.Ra * (a.NRa + pad);
  // arrays: rho and V, A (ext1, ld1), B (ext2, ld2), all x fastest
  const long long sr[3] = {1, p->n[0], (long long)p->n[0] * p->n[1]};
  const long long s1[3] = {1, (long long)p->ld1, (long long)p->ld1 * p->ext1[1]};
  const long long s2[3] = {1, (long long)p->ld2, (long long)p->ld2 * p->ext2[1]};
  int at, ap;
  tile_axes(al, &at, &ap);
  a.npl = 1;
  if (real_pass) {
    const bool fwd = pass == P1;
    const bool pair = !packed;
    long long rst, rsp, rse, cst, csp, cse;
    if (al == 0) {  // rows of rho and A, all z planes in one sequence
      const int rows = p->n[1] * p->n[2];
      const int m = pair ? 2 : 1;
      a.ntl = (rows + m - 1) / m;
      rst = (long long)m * p->n[0];
      cst = (long long)m * p->ld1;
      rsp = csp = 0;
      rse = packed ? 2 : 1;
      cse = 1;
      a.im_off = packed ? 1 : p->n[0];
      a.im_c = (long long)p->ld1;
      a.nreal = packed ? p->n[0] : rows;
    } else {        // columns x = 2 t, 2 t + 1 along y or z
      a.ntl = (p->n[0] + 1) / 2;
      rst = cst = 2;
      rsp = sr[ap];
      csp = s1[ap];
      rse = sr[al];
      cse = s1[al];
      a.im_off = a.im_c = 1;
      a.nreal = p->n[0];
      a.npl = p->n[ap];
    }
    a.nin = a.nout = nin;
    a.st_in = fwd ? rst : cst;
    a.sp_in = fwd ? rsp : csp;
    a.se_in = (int)(fwd ? rse : cse);
    a.st_out = fwd ? cst : rst;
    a.sp_out = fwd ? csp : rsp;
    a.se_out = (int)(fwd ? cse : rse);
    a.vec = a.im_off == 1 && p->n[0] % 2 == 0;  // and the pointer's alignment, at launch
    a.mout = div_magic((unsigned)(N / 2 + 1));
    tl.fn = fwd ? tile_r2c_kernel<T>(pair, zhalf, r.cls) : tile_c2r_kernel<T>(pair, zhalf, r.cls);
  } else {
    const long long* si = pass == P2 ? s1 : s2;
    const long long* so = pass == P4 ? s1 : s2;
    const int* ext = pass == P2 ? p->ext1 : p->ext2;
    a.ntl = ext[at];
    a.npl = ext[ap];
    a.st_in = si[at];
    a.sp_in = si[ap];
    a.se_in = (int)si[al];
    a.st_out = so[at];
    a.sp_out = so[ap];
    a.se_out = (int)so[al];
    if (si[al] > 0x7fffffffLL || so[al] > 0x7fffffffLL) return cudaSuccess;
    a.nin = pass == P4 ? N : n;
    a.nout = pass == P2 ? N : n;
    if (pass == P3) {
      const long long Ks[3] = {1, (long long)p->ldk, (long long)(p->H[1] + 1) * (long long)p->ldk};
      a.Lt = p->L[at];
      a.Lp = p->L[ap];
      a.Kst = (int)Ks[at];
      a.Ksp = (int)Ks[ap];
      a.Kse = (int)Ks[al];
      a.La0 = p->L[p->ord[0]];
      a.w_tile = p->ord[0] == at;
      a.pair_pl = ap == p->ord[1];
      tl.fn = tile_conv_kernel<T>(zhalf, r.cls);
    } else {
      tl.fn = tile_line_kernel<T>(pass == P2 ? -1 : 1, zhalf, r.cls);
    }
  }
  const long long lines = (long long)a.ntl * a.npl;
  const TileShape sh = pick_tile(a, r, row, lines, axis_tile(p, al), sizeof(T), sms, pass == P3);
  const int tk = sh.tk;
  if (tk == 0) return cudaSuccess;
  a.tk = tk;
  while ((1 << a.ltk) < tk) ++a.ltk;
  if (a.lc) {
    a.es = 1;
    a.ls = row;
    a.s1 = a.NRa + pad;
    a.s2 = a.Rl;
  } else {
    a.es = tk;
    a.ls = 1;
    a.s1 = a.NRa * tk;
    a.s2 = a.Rl * tk;
  }
  a.elems = row * tk;
  tl.threads = sh.threads;
  tl.smem = ((size_t)a.elems + M) * sizeof(C);
  if (blue) tl.fn = tile_blue_kernel<T>(pass, real_pass && !packed);
  // tiles of one plane keep their rows aligned; tiles across planes leave no
  // line slot empty, which pays where the arithmetic bounds the pass (FP64)
  const long long padded = (long long)((a.ntl + tk - 1) / tk) * tk;
  a.flat = sizeof(T) == 8 || (double)padded > 1.2 * a.ntl;
  tl.grid = a.flat ? dim3((unsigned)((lines + tk - 1) / tk))
                   : dim3((unsigned)((a.ntl + tk - 1) / tk), (unsigned)a.npl);
  cudaError_t e = cudaFuncSetAttribute(tl.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  if (e != cudaSuccess) return e;
  tl.on = 1;
  return cudaSuccess;
}

}  // namespace

template <typename T>
cudaError_t configure_tile(ps_plan_s* p) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  for (int k = 0; k < 5; ++k) {
    e = configure_pass<T>(p, k, sms);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
template cudaError_t configure_tile<float>(ps_plan_s*);
template cudaError_t configure_tile<double>(ps_plan_s*);

cudaError_t launch_tile(ps_plan_s* p, int pass, const void* src, void* dst, double* E, cudaStream_t s,
                        VjpTerm* add) {
  const TileLaunch& tl = p->tile[pass];
  TileArgs a = tl.a;
  const int al = pass_axis(p, pass);
  a.src = a.rsrc = src;
  a.dst = a.rdst = dst;
  a.K = p->K;
  a.twL = p->tw[al];
  a.tw = tl.blue ? p->blue[al].twMt : p->twt[al];
  a.chirp = p->blue[al].chirp;
  a.Bf = p->blue[al].Bf;
  a.partials = p->partials;
  a.nparts = z_pass_ctas(p);
  a.escale = 0.5 * p->h * p->h * p->h;
  a.E = E;
  if (pass == P5 && add != nullptr) {
    a.addV = add->V;
    a.gE = add->gE;
    a.h3 = p->h * p->h * p->h;
    add->fused = true;
  }
  if (a.vec) {
    const void* r = pass == P1 ? src : dst;
    a.vec = reinterpret_cast<uintptr_t>(r) % (2 * p->esz) == 0;
  }
  void* args[] = {(void*)&a};
  cudaLaunchConfig_t lc = {};
  lc.gridDim = tl.grid;
  if (pass == P5 && E != nullptr) {
    a.shift = 1;
    ++lc.gridDim.x;
  }
  lc.blockDim = dim3((unsigned)tl.threads);
  lc.dynamicSmemBytes = tl.smem;
  lc.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr;
  lc.numAttrs = pdl_launches() ? 1 : 0;
  return cudaLaunchKernelExC(&lc, tl.fn, args);
}

}  // namespace ps
