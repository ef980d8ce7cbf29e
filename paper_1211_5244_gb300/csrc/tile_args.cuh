// Arguments of the tile kernels (tile_pass.cuh) and their launcher's interface.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

struct ps_plan_s;

namespace ps {

struct VjpTerm;

// A line of length N = Ra Rm Rl (Rm = 1 for two steps): digits n = n1 NRa + n2 Rl
// + n3 of the input index, k = k1 + Ra k2 + Ra Rm k3 of the output index.
struct TileArgs {
  const void* src;
  void* dst;
  const void* K;    // K^F octant (conv)
  const void* tw;   // W_N^j at tw[j * tws], as (cos, tan) (tan_pair)
  const void* twL;  // x real passes of even length: W_L^k, L = 2 N
  int tws;
  int N, Ra, Rm, Rl;
  int NRa, Kl;         // N / Ra, Ra Rm
  int s1, s2, es;      // tile strides of digits 1 and 2 and of digit 3
  int ls;              // tile stride of the lines
  unsigned mRa, mRm, mRl, mNRa, mNRm, mKl;  // div_magic (NRm = Ra Rl)
  int tk, ltk;         // lines per CTA (a power of two)
  int lc;              // 1: threads run along the lines (the lines are the contiguous axis)
  int elems;           // complex elements of the tile (the twiddle table follows)
  // element e of line t0 + t of plane p at p * sp + (t0 + t) * st + e * se
  long long sp_in, st_in, sp_out, st_out;
  int se_in, se_out;
  int ntl, npl;        // lines along the tile axis, planes
  int flat;            // tiles run over the lines of all planes in sequence
  int nin, nout;       // elements loaded (the rest zero) and stored per line
  int pair_pl;         // planes in the paired order of paired_ky
  // conv: lengths of the tile and plane axes (K^F folds at L - k), octant
  // strides, and the energy weight: 1 where the wavenumber of the
  // real-to-complex axis (the tile axis when w_tile, else the plane axis) is 0 or
  // La0 / 2
  int Lt, Lp, La0, w_tile;
  int Kst, Ksp, Kse;
  // energy: partials of the fused pass, added by the last pass's first CTA
  double* partials;
  int nparts;
  // last pass of a vector-Jacobian product: outputs += h3 gE addV
  const void* addV;
  const double* gE;
  double h3;
  int shift;  // 1: the first CTA in x adds the partials and has no lines
  double escale;
  double* E;
  // real passes: line t holds two real sequences (or the even and odd elements
  // of one row); im_off is the offset of the second from the first in reals,
  // sr the stride of their elements, im_c / sc the same in the spectrum
  const void* rsrc;
  void* rdst;
  long long im_off, im_c;
  int nreal;   // reals of a row (even x passes), or real sequences in all (pairs)
  int vec;     // real pairs are adjacent and aligned: one access each
  unsigned mout;  // div_magic of the outputs per line in the untangling loop
  // Bluestein form: N is the convolution length, Nt the line's; the chirp and its transform
  int Nt;
  const void* chirp;
  const void* Bf;
};

struct TileLaunch {
  int on;           // the pass runs on the tile kernels
  int blue;         // in Bluestein form
  const void* fn;
  dim3 grid;
  int threads;
  size_t smem;
  TileArgs a;       // pointers filled at launch
};

// Factorisation of N into two (or three) register steps; false if there is none.
struct TileRadix { int Ra, Rm, Rl, cls; };
bool tile_radix(int N, bool even_first, bool f32, TileRadix* r, double* cost = nullptr);
// Convolution length of the Bluestein form of a length-N transform on the tile
// kernels, at most max_M (0: none).
int tile_blue_length(int N, bool f32, int max_M);

// kernels by kind (tile_*.cu): cls 0 radices up to 8, 1 up to 16; half: n <= N / 2
template <typename T> const void* tile_line_kernel(int dir, bool half, int cls);
template <typename T> const void* tile_conv_kernel(bool half, int cls);
template <typename T> const void* tile_r2c_kernel(bool pair, bool half, int cls);
template <typename T> const void* tile_c2r_kernel(bool pair, bool half, int cls);
// the same passes in Bluestein form: P1 .. P5
template <typename T> const void* tile_blue_kernel(int pass, bool pair);

// Fills p->tile[pass] for the passes that run here (before npart is taken).
template <typename T> cudaError_t configure_tile(ps_plan_s* p);
// Launches pass `pass`; src and dst as in launch_solve.
cudaError_t launch_tile(ps_plan_s* p, int pass, const void* src, void* dst, double* E, cudaStream_t s,
                        VjpTerm* add = nullptr);

}  // namespace ps
