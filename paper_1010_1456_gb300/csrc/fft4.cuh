// Four-step pencil FFTs with compile-time lengths L = L1 * L2.
//
// A length-L transform of one pencil is done as
//   step A (thread n2 < L2): v[n1] = x[L2 n1 + n2], DFT_L1 in registers,
//                            times w_L^(n2 k1), stored to shared memory;
//   step B (thread k1 < L1): the L2 values of row k1, DFT_L2 in registers,
//                            X[k1 + L1 k2] = result[k2].
// (X[k1 + L1 k2] = sum_n2 w_L2^(n2 k2) w_L^(n2 k1) sum_n1 x[L2 n1 + n2] w_L1^(n1 k1).)
// Compared with one shared-memory round trip per radix stage, a pencil makes
// one round trip (two for the fused forward-product-inverse x pass) and all
// index arithmetic inside the register DFTs is resolved at compile time.
// These kernels serve the padded lengths of AIM_FOURSTEP_LENGTHS; longer ones
// use the Stockham kernels of fft.cu.
//
// Twiddles: twL holds w_L^t for t < L (the Stockham kernels' table), then
// the same factors w_L^(k1 n2) laid out twice for the four-step kernels: as
// [k1][n2] at twL + L (step A: the lanes of a warp take consecutive n2) and
// as [n2][k1] at twL + 2L (the x pass's step B: consecutive k1), so each
// warp-wide twiddle load touches one or two cache lines instead of one line
// per lane.
//
// fft4_strided: the z and y passes (pencil along a strided axis, TX
// consecutive x columns per block, as in fft.cu).
// fft4_x: the fused x pass: forward transform of the nx zero-padded samples
// of RY rows (ky) x TG grids per block, product with the Ghat rows and the
// inverse transform, nx samples kept.
#pragma once

#include "fft_policy.h"

namespace aim {

struct StridedArgs4 {
  int n_in, n_out;  // samples read (rest zero) / samples written
  int X, A;         // contiguous extent, other-axis extent
  long long sG_in, sA_in, sP_in;
  long long sG_out, sA_out, sP_out;
  // optional [A][X] flags of the pencils that matter (z passes of a 3-D grid:
  // the (x, y) columns that hold a stencil node): the others read no input
  // (it is zero) and, in an inverse pass, write no output (nothing reads it)
  const uint8_t* cols = nullptr;
};

struct XArgs4 {
  int nx, px;      // samples per row, row length in memory
  int Ly, Lz, G;
  int RY, TG;      // rows and grids per block at a time
  int GB;          // grids per block in all (blockIdx.z picks them)
  long long sG;    // grid stride (elements)
  int hx, hy;      // octant extents of Ghat (x, y)
};

// Columns per block of the strided kernels for length L: the policy's
// preferred width, halved while one pencil set would need more than 48 KB of
// shared memory (so long pencils still leave several blocks per SM).
template <class P, int L> constexpr int strided_tx() {
  int tx = P::kTX;
  while (tx > 4 && (long long)L * tx * (long long)sizeof(typename P::S) > 48 * 1024) tx /= 2;
  return tx;
}

// Columns of TX values per row k1 of the tile: one more than L2 where a row of an even L2 would
// put the k1 of one access phase (128 bytes) on the same banks.
template <class P, int L1, int L2> constexpr int strided_row() {
  return L2 + (L2 % 2 == 0 && strided_tx<P, L1 * L2>() * sizeof(typename P::S) < 128 ? 1 : 0);
}

// Work units of a strided block.  The two steps have TX AY L2 and TX AY L1
// units; the block's threads are one round of the heavier step where the
// split is about even, else of the lighter one (whose units are the longer
// transforms), and the other takes several rounds: with one round of both, a
// 5 x 25 split kept four threads in five idle in step B (float-float y passes
// of 125^3 grids, 120 us).  About 256 threads, a tile of at most 48 KB.
// For complex64, which waits for memory rather than arithmetic, that pays from
// a ratio of 2.5 (243: y passes 338 -> 298 us; 512, ratio 2: 1.4 -> 1.7 ms).
template <class P> constexpr int strided_width(int L1, int L2) {
  const int lm = L1 > L2 ? L1 : L2, ls = L1 > L2 ? L2 : L1;
  return (sizeof(typename P::S) > 8 ? 8 * ls >= 5 * lm : 5 * ls >= 2 * lm) ? lm : ls;
}
template <class P, int L1, int L2> constexpr int strided_ay() {
  constexpr int TX = strided_tx<P, L1 * L2>();
  constexpr long long set = (long long)L1 * strided_row<P, L1, L2>() * TX * (long long)sizeof(typename P::S);
  int ay = 256 / (TX * strided_width<P>(L1, L2));
  const int fit = (int)(48 * 1024 / set);
  if (ay > fit) ay = fit;
  return ay < 1 ? 1 : ay;
}
template <class P, int L1, int L2> constexpr int strided_threads() {
  return (strided_ay<P, L1, L2>() * strided_tx<P, L1 * L2>() * strided_width<P>(L1, L2) + 31) / 32 * 32;
}

// Resident blocks per SM the complex64 kernels' registers must allow: their pencils' values (two
// registers each) and 18 more.  The passes are bound by the latency of memory (61 % of the DRAM
// rate on 288^3 grids), so resident warps count for more than a few spilled values.  The 16-byte
// policies are bound by arithmetic: 128 registers for DFTs of up to 24, twice the warps of the 255
// they would take (float-float y passes of 180^3 grids: 98 us, 131 with 255), and what they need above.
template <class P, int L1, int L2> constexpr int strided_min_blocks() {
  constexpr int LM = L1 > L2 ? L1 : L2;
  const int regs = sizeof(typename P::S) <= 8 ? 2 * LM + 18 : LM <= 24 ? 128 : 255;
  const int n = 65536 / (strided_threads<P, L1, L2>() * regs);
  return n < 1 ? 1 : n > 8 ? 8 : n;
}

// Shared-memory row length: odd, so lanes that walk a strided row hit
// distinct banks.
constexpr int odd_row(int n) { return n + (n % 2 == 0 ? 1 : 0); }

// Pencil tiles [L1][odd_row(L2)] of a block lie pencil_stride apart.  A phase of a warp's access
// (128 bytes: 16 or 8 elements) is free of bank conflicts within a pencil; one that spans two
// pencils is too when the stride continues the pattern: = L2 (mod a phase) for the accesses along
// n2 (steps A and C), = L1 odd_row(L2) for those down a column (step B).  Where L1 is a multiple
// of the phase step B never spans two, and the stride serves A and C; else B.
constexpr int pencil_stride(int L1, int L2, int phase) {
  int n = L1 * odd_row(L2);
  if (L1 % phase == 0)
    while (n % phase != L2 % phase) ++n;
  return n;
}

// Of the samples r, r + step, r + 2 step, ... of a padded axis of length L, the
// number that can lie below (L + 1) / 2, the largest unpadded extent (L >= 2 n - 1).
constexpr int half_terms(int L, int step) { return ((L + 1) / 2 + step - 1) / step; }

// A block transforms AY consecutive other-axis indices (ia) x TX columns, so
// short pencils still give every thread work.  Step A loads its L1 samples
// straight from global memory into registers (samples >= n_in are zero and
// never read); the only shared-memory round trip is the transpose between
// the two steps.  Step B writes the first n_out outputs.  (Copying the next
// grid's samples into shared memory, cp.async, while this one transforms was
// slower: y passes of 648^3 grids 13 to 15 ms against 10 to 11.)
// PRUNED: a padded axis, where at most (L + 1) / 2 samples are read (forward)
// or written (inverse) and the other side is whole; which samples that leaves
// out is known at compile time, so the register DFTs skip their arithmetic.
// Without it both sides are whole (the spectrum of Green's function).
template <class P, bool INV, int L1, int L2, bool PRUNED>
__global__ void __launch_bounds__(strided_threads<P, L1, L2>(), strided_min_blocks<P, L1, L2>())
    fft4_strided(const typename P::S* __restrict__ in, typename P::S* __restrict__ out, StridedArgs4 a,
                 const typename P::S* __restrict__ twL, int AY) {
  pdl_begin();
  using S = typename P::S;
  using T = typename P::T;
  constexpr int L = L1 * L2, TX = strided_tx<P, L>(), RP = strided_row<P, L1, L2>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  S* b = reinterpret_cast<S*>(smem_raw);  // [AY][L1][RP][TX]
  const int x0 = blockIdx.x * TX;
  const int ia0 = blockIdx.y * AY;
  const int nay = min(AY, a.A - ia0);
  const long long g = blockIdx.z;
  for (int u = threadIdx.x; u < nay * TX * L2; u += blockDim.x) {
    const int t = u / (TX * L2), rem = u - t * (TX * L2);
    const int c = rem % TX, n2 = rem / TX;
    const bool col = x0 + c < a.X && (!a.cols || a.cols[(long long)(ia0 + t) * a.X + x0 + c]);
    const S* src = in + g * a.sG_in + (long long)(ia0 + t) * a.sA_in + x0 + c;
    constexpr int H = PRUNED && !INV ? half_terms(L, L2) : L1;
    T v[L1];
    static_for<0, H>([&](auto n1) {
      const int p = L2 * decltype(n1)::value + n2;
      v[n1] = (col && p < a.n_in) ? P::ld(src[(long long)p * a.sP_in]) : P::zero();
    });
    RegDFT<P, L1, INV, all_mask(H)>::run(v);
    if (n2 > 0)
      static_for<1, L1>([&](auto k1) { v[k1] = P::mul(v[k1], P::conj_if(P::ld(twL[L + decltype(k1)::value * L2 + n2]), INV)); });
    S* y = b + t * L1 * RP * TX;
    static_for<0, L1>([&](auto k1) { y[(decltype(k1)::value * RP + n2) * TX + c] = P::st(v[k1]); });
  }
  __syncthreads();
  for (int u = threadIdx.x; u < nay * TX * L1; u += blockDim.x) {
    const int t = u / (TX * L1), rem = u - t * (TX * L1);
    const int c = rem % TX, k1 = rem / TX;
    const S* y = b + t * L1 * RP * TX;
    T w[L2];
    static_for<0, L2>([&](auto n2) { w[n2] = P::ld(y[(k1 * RP + decltype(n2)::value) * TX + c]); });
    RegDFT<P, L2, INV>::run(w);
    S* dst = out + g * a.sG_out + (long long)(ia0 + t) * a.sA_out + x0 + c;
    if (x0 + c < a.X && (!INV || !a.cols || a.cols[(long long)(ia0 + t) * a.X + x0 + c]))
      static_for<0, PRUNED && INV ? half_terms(L, L1) : L2>([&](auto k2) {
        const int p = k1 + L1 * decltype(k2)::value;
        if (!PRUNED || !INV || p < a.n_out) dst[(long long)p * a.sP_out] = P::st(w[k2]);
      });
  }
}

// The fused x pass.  With k = k1 + L1 k2 and n = n2 + L2 n1,
//   forward  X[k1 + L1 k2] = sum_n2 w_L2^(n2 k2) w_L^(n2 k1) sum_n1 x[L2 n1 + n2] w_L1^(n1 k1),
//   inverse  y[n2 + L2 n1] = sum_k1 w_L1^(-k1 n1) w_L^(-k1 n2) sum_k2 X[k1 + L1 k2] w_L2^(-k2 n2).
// The thread that finishes the forward transform for one k1 holds X[k1 + L1 k2]
// for every k2, which is exactly the input of the inverse's first step, so it
// multiplies by Ghat and starts the inverse in registers:
//   step A (unit n2, from global):   DFT_L1, twiddle, into row k1 column n2 of the tile;
//   step B (unit k1):                row k1: DFT_L2, x Ghat, inverse DFT_L2, twiddle,
//                                    written back over the same row;
//   step C (unit n2, to global):     column n2: inverse DFT_L1, samples < nx written.
// One [L1][odd L2] tile per pencil, two shared-memory round trips.  (Both
// twiddle products in step B, from one table, lengthen the longest step: 648^3
// 24.8 -> 30.9 ms.  Two pencils a thread with all operations packed halves the
// instructions and leaves too few warps: 27.7 ms.)  The block handles RY rows (ky)
// x TG grids at a time, in as many rounds of its threads as each step's units
// take (one where the split is even), and keeps the RY rows of Ghat in shared
// memory.  Complex64 is bound by the L1/shared-memory pipe and the latency of
// the rounds, so it runs in small blocks, whose barriers hold up fewer warps
// (648^3, 32 grids: 24.8 ms in 128-thread blocks, 26.5 in 256; 64 and 96 threads:
// 5 and 14 % slower); the 16-byte
// policies are bound by the FP32 or FP64 pipe.
template <class P> constexpr int x_threads() { return sizeof(typename P::S) <= 8 ? 128 : 256; }
// Resident blocks per SM the register allocation must allow.
template <class P, int L1, int L2> constexpr int x_min_blocks() {
  constexpr int LM = L1 > L2 ? L1 : L2;
  if (sizeof(typename P::S) <= 8) return LM <= 25 ? 8 : LM <= 27 ? 6 : 4;  // 64, 80, 128 registers
  return L1 * L2 > 648 ? 1 : 2;                                            // 255, 128 registers
}

template <class P, int L1, int L2>
__global__ void __launch_bounds__(x_threads<P>(), x_min_blocks<P, L1, L2>()) fft4_x(typename P::S* __restrict__ buf, XArgs4 a,
                                              const typename P::S* __restrict__ ghat,
                                              const typename P::S* __restrict__ twL) {
  pdl_begin();
  using S = typename P::S;
  using T = typename P::T;
  constexpr int L = L1 * L2;
  constexpr int RA = odd_row(L2);
  constexpr int PA = pencil_stride(L1, L2, 128 / (int)sizeof(S));  // per-pencil tile
  constexpr int H = half_terms(L, L2);  // the samples n2 + L2 n1 below nx have n1 < H
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int RY = a.RY, TG = a.TG;
  S* gr = reinterpret_cast<S*>(smem_raw);  // [RY][L]
  S* tile = gr + RY * L;                    // [RY * TG][L1][RA]
  const int ky0 = blockIdx.x * RY, kz = blockIdx.y;
  const int nry = min(RY, a.Ly - ky0);
  const int iz = min(kz, a.Lz - kz);
  for (int e = threadIdx.x; e < nry * L; e += blockDim.x) {
    const int r = e / L, p = e % L;
    const int ky = ky0 + r;
    const int iy = min(ky, a.Ly - ky);
    gr[e] = ghat[((long long)iz * a.hy + iy) * a.hx + min(p, L - p)];
  }
  const long long row0 = ((long long)kz * a.Ly + ky0) * a.px;
  const int gbeg = blockIdx.z * a.GB, gend = min(a.G, gbeg + a.GB);
  for (int g0 = gbeg; g0 < gend; g0 += TG) {
    const int ng = min(TG, gend - g0);
    const int np = nry * ng;  // pencil pc = r * ng + gl
    if (g0 > gbeg) __syncthreads();  // the previous group's step C has read its tiles
    // step A: forward DFT_L1 of the zero-padded row, straight from global memory
    for (int u = threadIdx.x; u < np * L2; u += blockDim.x) {
      const int n2 = u % L2, pc = u / L2;
      const int r = pc / ng, gl = pc - r * ng;
      const S* src = buf + (long long)(g0 + gl) * a.sG + row0 + (long long)r * a.px;
      T v[L1];
      static_for<0, H>([&](auto n1) {
        const int p = L2 * decltype(n1)::value + n2;
        v[n1] = p < a.nx ? P::ld(src[p]) : P::zero();
      });
      RegDFT<P, L1, false, all_mask(H)>::run(v);
      if (n2 > 0) static_for<1, L1>([&](auto k1) { v[k1] = P::mul(v[k1], P::ld(twL[L + decltype(k1)::value * L2 + n2])); });
      S* y = tile + pc * PA + n2;
      static_for<0, L1>([&](auto k1) { y[decltype(k1)::value * RA] = P::st(v[k1]); });
    }
    __syncthreads();  // also orders Ghat's staging before the first step B
    // step B: forward DFT_L2, product with Ghat, inverse DFT_L2, over one row
    for (int u = threadIdx.x; u < np * L1; u += blockDim.x) {
      const int k1 = u % L1, pc = u / L1;
      const int r = pc / ng;
      S* y = tile + pc * PA + k1 * RA;
      T w[L2];
      static_for<0, L2>([&](auto n2) { w[n2] = P::ld(y[decltype(n2)::value]); });
      RegDFT<P, L2, false>::run(w);
      const S* gg = gr + r * L + k1;
      static_for<0, L2>([&](auto k2) { w[k2] = P::mul(w[k2], P::ld(gg[L1 * decltype(k2)::value])); });
      RegDFT<P, L2, true>::run(w);
      if (k1 > 0)
        static_for<1, L2>([&](auto n2) { w[n2] = P::mul(w[n2], P::conj_if(P::ld(twL[2 * L + decltype(n2)::value * L1 + k1]), true)); });
      static_for<0, L2>([&](auto n2) { y[decltype(n2)::value] = P::st(w[n2]); });
    }
    __syncthreads();
    // step C: inverse DFT_L1 over one column, the first nx samples back to global memory
    for (int u = threadIdx.x; u < np * L2; u += blockDim.x) {
      const int n2 = u % L2, pc = u / L2;
      const int r = pc / ng, gl = pc - r * ng;
      const S* z = tile + pc * PA + n2;
      T v[L1];
      static_for<0, L1>([&](auto k1) { v[k1] = P::ld(z[decltype(k1)::value * RA]); });
      RegDFT<P, L1, true>::run(v);
      S* dst = buf + (long long)(g0 + gl) * a.sG + row0 + (long long)r * a.px;
      static_for<0, H>([&](auto n1) {
        const int p = n2 + L2 * decltype(n1)::value;
        if (p < a.nx) dst[p] = P::st(v[n1]);
      });
    }
  }
}

// Padded lengths with a four-step kernel, as (L, L1, L2): every 2,3,5-smooth
// length up to 900 that is the smallest one >= 2 n - 1 for some grid extent n
// (6, 10 and 16 never are: 5, 9 and 15 precede them), and 1296.  L1 * L2 is
// the most even split.  Six lists, one translation unit each per policy.
#define AIM_FOURSTEP_LENGTHS_0(X) \
  X(3, 1, 3) X(5, 5, 1) X(8, 2, 4) X(9, 3, 3) X(12, 3, 4) \
  X(15, 3, 5) X(18, 3, 6) X(20, 4, 5) X(24, 4, 6) X(25, 5, 5) \
  X(27, 3, 9) X(30, 5, 6) X(32, 4, 8) X(36, 6, 6) X(40, 5, 8) \
  X(45, 5, 9) X(48, 6, 8) X(50, 5, 10) X(54, 6, 9) X(60, 6, 10) \
  X(64, 8, 8) X(72, 8, 9) X(75, 5, 15) X(80, 8, 10) X(81, 9, 9) \
  X(90, 9, 10) X(96, 8, 12) X(100, 10, 10)
#define AIM_FOURSTEP_LENGTHS_1(X) \
  X(108, 9, 12) X(120, 10, 12) X(125, 5, 25) X(128, 8, 16) X(135, 9, 15) \
  X(144, 12, 12) X(150, 10, 15) X(160, 10, 16) X(162, 9, 18) X(180, 12, 15) \
  X(192, 12, 16) X(200, 10, 20)
#define AIM_FOURSTEP_LENGTHS_2(X) \
  X(216, 12, 18) X(225, 15, 15) X(240, 15, 16) X(243, 9, 27) X(250, 10, 25) \
  X(256, 16, 16) X(270, 15, 18) X(288, 16, 18) X(300, 15, 20) X(320, 16, 20)
#define AIM_FOURSTEP_LENGTHS_3(X) \
  X(324, 18, 18) X(360, 18, 20) X(375, 15, 25) X(384, 16, 24) X(400, 20, 20) \
  X(405, 15, 27) X(432, 18, 24) X(450, 18, 25) X(480, 20, 24) X(486, 18, 27) \
  X(500, 20, 25)
#define AIM_FOURSTEP_LENGTHS_4(X) \
  X(512, 16, 32) X(540, 20, 27) X(576, 24, 24) X(600, 24, 25) X(625, 25, 25) \
  X(640, 20, 32)
#define AIM_FOURSTEP_LENGTHS_5(X) \
  X(648, 24, 27) X(675, 25, 27) X(720, 24, 30) X(729, 27, 27) X(750, 25, 30) \
  X(768, 24, 32) X(800, 25, 32) X(810, 27, 30) X(864, 27, 32) X(900, 30, 30) \
  X(1296, 36, 36)
#define AIM_FOURSTEP_LENGTHS(X) \
  AIM_FOURSTEP_LENGTHS_0(X) AIM_FOURSTEP_LENGTHS_1(X) AIM_FOURSTEP_LENGTHS_2(X) \
  AIM_FOURSTEP_LENGTHS_3(X) AIM_FOURSTEP_LENGTHS_4(X) AIM_FOURSTEP_LENGTHS_5(X)
// The list (and translation unit) of length L.
constexpr int fourstep_part(int L) {
  return L <= 100 ? 0 : L <= 200 ? 1 : L <= 320 ? 2 : L <= 500 ? 3 : L <= 640 ? 4 : 5;
}
constexpr int kFourStepParts = 6;

}  // namespace aim
