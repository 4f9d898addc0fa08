// Launchers of the four-step FFT kernels for one arithmetic policy and one of
// the lists of lengths; each fft4_<policy>.cu includes this with
// AIM_FFT4_POLICY and AIM_FFT4_NAME set and is compiled once per list
// (AIM_FFT4_PART), so policies and lists compile in parallel.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "fft4.cuh"
#include "fft4_decl.h"

namespace aim {

namespace {
constexpr int kNotHandled = -1;
constexpr int kSMs = 152;
using Pol = AIM_FFT4_POLICY;
using S = Pol::S;

template <bool INV, int L1, int L2, bool PRUNED = true>
int launch_strided4(aim_ctx* c, const char* name, const S* in, S* out, const StridedArgs4& a, int G, const S* tw) {
  constexpr int TX = strided_tx<Pol, L1 * L2>();
  constexpr long long pencil_set = (long long)L1 * strided_row<Pol, L1, L2>() * TX * sizeof(S);
  int AY = std::min(strided_ay<Pol, L1, L2>(), a.A);
  // a small grid: fewer indices per block until there are four blocks per SM, down to two warps' worth of work
  const long long xt = (a.X + TX - 1) / TX;
  while (AY > 1 && xt * G * ((a.A + AY - 1) / AY) < 4 * kSMs && AY * TX * std::max(L1, L2) > 64) AY = (AY + 1) / 2;
  const int items = AY * TX * std::max(L1, L2);
  const int threads = std::min((items + 31) / 32 * 32, strided_threads<Pol, L1, L2>());
  const size_t sm = (size_t)AY * pencil_set;
  const auto kern = fft4_strided<Pol, INV, L1, L2, PRUNED>;
  static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  AIM_CUDA_TRY(attr);
  dim3 grid((unsigned)xt, (a.A + AY - 1) / AY, G);
  AIM_LAUNCH(c, name, (launch_pdl(!std::is_same<Pol, P64>::value, kern, grid, threads, sm, c->stream, in, out, a, tw, AY)));
  return launch_check(c, name);
}

// Rows (RY) and grids (TG) a block of T threads takes at a time.  A step's
// rounds each cost the length of its unit, a barrier and a memory latency;
// the last round over the grids is charged by a square root, since a thin one
// is a short one.  (225^3, 56 grids: 17 at a time 1.70 ms, 14 at a time 1.95;
// 125^3, 4 float-float grids: one round of the 5-point step per 25-point one
// 551 us.)
template <int L1, int L2> void x_shape(const XArgs4& a, int T, long long cap, int* RY, int* TG) {
  constexpr long long per_pencil = pencil_stride(L1, L2, 128 / (int)sizeof(S));
  const double unitA = L1 * std::log2(L1 + 1.0), unitB = 2 * L2 * std::log2(L2 + 1.0) + L2, fixed = 20.0;
  double best = 0.0;
  for (int np = 1; np <= 64; ++np) {
    const int its = (a.G + std::min(np, a.G) - 1) / std::min(np, a.G);
    const int tg = (a.G + its - 1) / its, ry = std::min(np / tg, a.Ly);
    const int n = tg * ry;
    if (ry < 1 || n * per_pencil + ry * (long long)L1 * L2 > cap) continue;
    const int rA = (n * L2 + T - 1) / T, rB = (n * L1 + T - 1) / T;
    const double cost = (2 * rA * (unitA + fixed) + rB * (unitB + fixed)) / n * std::sqrt((double)its * tg / a.G);
    if (best == 0.0 || cost < 0.97 * best) {
      best = cost;
      *RY = ry;
      *TG = tg;
    }
  }
}

template <int L1, int L2>
int launch_x4(aim_ctx* c, const char* name, S* buf, XArgs4 a, const S* ghat, const S* tw, int threads) {
  constexpr int L = L1 * L2;
  constexpr long long per_pencil = pencil_stride(L1, L2, 128 / (int)sizeof(S));
  constexpr int LM = std::max(L1, L2);
  const int T = std::min(threads, x_threads<Pol>());
  // shared memory of a block: an even share of an SM's among the resident blocks
  const long long cap = 220 * 1024 / (long long)sizeof(S) / (x_min_blocks<Pol, L1, L2>() * (x_threads<Pol>() / T));
  int TG = 0, RY = 0;
  x_shape<L1, L2>(a, T, cap, &RY, &TG);
  if (TG == 0) {  // a pencil larger than that share
    TG = RY = 1;
    if (L + per_pencil > 220 * 1024 / (long long)sizeof(S)) return kNotHandled;
  }
  int GB = a.G;
  // a small grid (a planar one, or few grids): blocks first split the rounds
  // over the grids among them, up to a dozen blocks per SM, then take fewer
  // rows and grids, until there are four per SM (whole blocks are shared out
  // evenly then) or a block is down to two warps, one warp where some SM would
  // stay idle.  A 120 x 108 plane of 4 float-float grids, 20 blocks of 5 rows:
  // 27 us; a 648 x 648 plane of 256 complex64 grids, 648 blocks of 64 rounds:
  // 416 us.
  const auto rows = [&] { return (long long)((a.Ly + RY - 1) / RY) * a.Lz; };
  const auto blocks = [&] { return rows() * ((a.G + GB - 1) / GB); };
  const auto more = [&] {
    const long long n = blocks();
    return n < kSMs ? RY * TG * LM > 32 : n < 4 * kSMs && RY * TG * LM > 64;
  };
  {
    const int rounds = (a.G + TG - 1) / TG;
    const int split = (int)std::min<long long>(rounds, (12LL * kSMs + rows() - 1) / rows());
    GB = (rounds + split - 1) / split * TG;
  }
  if (std::is_same<Pol, P64>::value) {
    // Bound by the FP64 pipe, where a warp costs the same with any number of its lanes in use: the smallest
    // blocks, as below, unless another of these shapes leaves the busiest SM a tenth less warp time (324 x
    // 324 plane, 4 grids: 648 blocks of 36 units, 105 us; 108 blocks of 216, 72; 400: 128 and 88)
    struct Shape {
      int ry, tg, gb;
      double t;
    };
    const auto shape = [&] {
      const int n = RY * TG;
      const double AC = 2.0 * ((n * L2 + 31) / 32) * L1 * std::log2(L1 + 1.0),
                   B = (double)((n * L1 + 31) / 32) * (2 * L2 * std::log2(L2 + 1.0) + L2);
      return Shape{RY, TG, GB, (AC + B) * ((GB + TG - 1) / TG) * (double)((blocks() + kSMs - 1) / kSMs)};
    };
    Shape best = shape(), last = best;
    while (more() && (RY > 1 || TG > 1)) {
      if (RY > 1) RY = (RY + 1) / 2;
      else GB = TG = (TG + 1) / 2;
      last = shape();
      if (last.t < best.t) best = last;
    }
    if (best.t >= 0.9 * last.t) best = last;
    RY = best.ry;
    TG = best.tg;
    GB = best.gb;
  } else {
    while (more() && RY > 1) RY = (RY + 1) / 2;
    while (more() && TG > 1) GB = TG = (TG + 1) / 2;
  }
  a.RY = RY;
  a.TG = TG;
  a.GB = GB;
  const size_t sm = (size_t)(RY * L + RY * TG * per_pencil) * sizeof(S);
  const int nthreads = std::min(T, (RY * TG * LM + 31) / 32 * 32);
  static const cudaError_t attr =
      cudaFuncSetAttribute(fft4_x<Pol, L1, L2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  AIM_CUDA_TRY(attr);
  dim3 grid((a.Ly + RY - 1) / RY, a.Lz, (a.G + GB - 1) / GB);
  AIM_LAUNCH(c, name, (launch_pdl(!std::is_same<Pol, P64>::value, fft4_x<Pol, L1, L2>, grid, nthreads, sm, c->stream, buf, a, ghat, tw)));
  return launch_check(c, name);
}
}  // namespace

#define AIM_CAT_(a, b) a##b
#define AIM_CAT(a, b) AIM_CAT_(a, b)
#define AIM_PART_LENGTHS AIM_CAT(AIM_FOURSTEP_LENGTHS_, AIM_FFT4_PART)

// 1: launched; 0: no four-step kernel for this length; < 0: -error code.
template <>
int AIM_FFT4_NAME(strided)<AIM_FFT4_PART>(aim_ctx* c, const char* name, bool inv, const S* in, S* out,
                                          const StridedArgs4& a, int G, int L, const S* tw) {
  int rc = AIM_OK;
  switch (L) {
#define AIM_CASE(LL, A1, A2)                                                                             \
  case LL:                                                                                               \
    if constexpr (std::is_same<Pol, P64>::value)                                                         \
      if (a.n_in == LL && a.n_out == LL) { /* whole on both sides: the spectrum of Green's function */  \
        rc = launch_strided4<false, A1, A2, false>(c, name, in, out, a, G, tw);                          \
        return rc == AIM_OK ? 1 : -rc;                                                                   \
      }                                                                                                  \
    rc = inv ? launch_strided4<true, A1, A2>(c, name, in, out, a, G, tw)                                 \
             : launch_strided4<false, A1, A2>(c, name, in, out, a, G, tw);                               \
    return rc == AIM_OK ? 1 : -rc;
    AIM_PART_LENGTHS(AIM_CASE)
#undef AIM_CASE
    default: return 0;
  }
}

template <>
int AIM_FFT4_NAME(x)<AIM_FFT4_PART>(aim_ctx* c, const char* name, S* buf, const XArgs4& a, int L, const S* ghat,
                                    const S* tw, int threads) {
  int rc = kNotHandled;
  switch (L) {
#define AIM_CASE(LL, A1, A2) \
  case LL: rc = launch_x4<A1, A2>(c, name, buf, a, ghat, tw, threads); break;
    AIM_PART_LENGTHS(AIM_CASE)
#undef AIM_CASE
    default: break;
  }
  return rc == kNotHandled ? 0 : rc == AIM_OK ? 1 : -rc;
}

}  // namespace aim
