// Plane-wave right-hand sides and bistatic RCS.
//
// Excitation (paper Section 2.1): E_inc = pol exp(-j k khat . r) and
// V_m = int f_m . E_inc dS (collapsed Gauss-Legendre 4x4 rule per triangle).
// Far field (paper eq. 1 ingredients): N(rhat) = sum_m x_m int f_m
// exp(+j k rhat . r) dS (3x3 rule), sigma = k^2 eta^2 / (4 pi) |e . N|^2.
// The far field is evaluated as a sum over triangle quadrature points that
// carry the point current J_p = sum over the basis functions on the
// triangle of x_m f_m(r_p) A w_p (FP64, then rounded to FP32).  Every
// (direction, point) pair needs one phase factor exp(j k rhat . r_p): the
// phase is formed in float-float arithmetic (k rhat and r_p as pairs of
// floats, about 48 bits), reduced modulo 2 pi with a three-part constant,
// and its cosine and sine are taken in FP32 at the reduced high part with a
// first-order correction by the low part; the products with J_p are FP32,
// summed in FP32 over runs of 64 points and in FP64 beyond.  Per pair the
// phase factor is good to about 1 FP32 ulp and the product to a few, all on
// the FP32 pipes: a 16 lambda sphere's 5.4 M points times 326 k directions
// take seconds instead of the minutes of FP64 phases.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.h"
#include "ff.h"
#include "geom.h"

namespace aim {

constexpr int kRhsRule = 4, kFarRule = 3;
__constant__ double c_rhs_rule[3][kMaxRule * kMaxRule];
__constant__ double c_far_rule[3][kMaxRule * kMaxRule];

static int upload_rules() {
  static const int rc = [] {
    TriRule a = make_tri_rule(kRhsRule), b = make_tri_rule(kFarRule);
    double ha[3][kMaxRule * kMaxRule], hb[3][kMaxRule * kMaxRule];
    for (int q = 0; q < a.q; ++q) {
      ha[0][q] = a.xi1[q];
      ha[1][q] = a.xi2[q];
      ha[2][q] = a.w[q];
    }
    for (int q = 0; q < b.q; ++q) {
      hb[0][q] = b.xi1[q];
      hb[1][q] = b.xi2[q];
      hb[2][q] = b.w[q];
    }
    if (cudaMemcpyToSymbol(c_rhs_rule, ha, sizeof(ha)) != cudaSuccess) return 1;
    if (cudaMemcpyToSymbol(c_far_rule, hb, sizeof(hb)) != cudaSuccess) return 1;
    return 0;
  }();
  if (rc) {
    set_error("failed to upload quadrature rules");
    return AIM_ECUDA;
  }
  return AIM_OK;
}

__device__ __forceinline__ V3 ldv(const double* v, int i) { return v3(v[3 * i], v[3 * i + 1], v[3 * i + 2]); }

__global__ void k_rhs(const double* __restrict__ verts, const int32_t* __restrict__ tris,
                      const int32_t* __restrict__ rtri, const int32_t* __restrict__ rfree,
                      const double* __restrict__ len, const double* __restrict__ area, const double* __restrict__ khat,
                      const double* __restrict__ pol, double2* __restrict__ V, int N, double k,
                      const double* __restrict__ nrm, double alpha) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  const int b = blockIdx.y;
  if (m >= N) return;
  const V3 kh = v3(khat[3 * b], khat[3 * b + 1], khat[3 * b + 2]);
  const V3 pe = v3(pol[3 * b], pol[3 * b + 1], pol[3 * b + 2]);
  double re = 0.0, im = 0.0;
  const int nq = kRhsRule * kRhsRule;
  for (int half = 0; half < 2; ++half) {
    const int t = rtri[2 * m + half];
    const V3 fv = ldv(verts, rfree[2 * m + half]);
    const V3 r0 = ldv(verts, tris[3 * t]), r1 = ldv(verts, tris[3 * t + 1]), r2 = ldv(verts, tris[3 * t + 2]);
    const double A = area[t];
    const double cf = (half ? -1.0 : 1.0) * len[m] / (2.0 * A);
    // CFIE: alpha E_inc + (1 - alpha) eta n x H_inc, both tangential-tested;
    // eta H_inc = khat x pol times the same phase, n constant on the triangle.
    V3 pt = pe;
    if (nrm) pt = alpha * pe + (1.0 - alpha) * cross(ldv(nrm, t), cross(kh, pe));
    for (int q = 0; q < nq; ++q) {
      const V3 r = tri_point(r0, r1, r2, c_rhs_rule[0][q], c_rhs_rule[1][q]);
      const double fp = cf * dot(r - fv, pt) * A * c_rhs_rule[2][q];
      double s, c;
      sincos(k * dot(kh, r), &s, &c);
      re += fp * c;
      im -= fp * s;
    }
  }
  V[(long long)b * N + m] = make_double2(re, im);
}

// point currents: J[b][p][3] for p = t * 9 + q, positions rp[p][3]
__global__ void k_point_currents(const double* __restrict__ verts, const int32_t* __restrict__ tris,
                                 const int32_t* __restrict__ rtri, const int32_t* __restrict__ rfree,
                                 const double* __restrict__ len, const double* __restrict__ area,
                                 const double2* __restrict__ X, double2* __restrict__ J, double* __restrict__ rp,
                                 int N, int nt, int nrhs) {
  // one thread per (basis, half, point); contributions added with atomics
  const int nq = kFarRule * kFarRule;
  const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (tid >= (long long)N * 2 * nq) return;
  const int q = (int)(tid % nq);
  const int half = (int)((tid / nq) % 2);
  const int m = (int)(tid / (2 * nq));
  const int t = rtri[2 * m + half];
  const V3 fv = ldv(verts, rfree[2 * m + half]);
  const V3 r0 = ldv(verts, tris[3 * t]), r1 = ldv(verts, tris[3 * t + 1]), r2 = ldv(verts, tris[3 * t + 2]);
  const double A = area[t];
  const V3 r = tri_point(r0, r1, r2, c_far_rule[0][q], c_far_rule[1][q]);
  const double cf = (half ? -1.0 : 1.0) * len[m] / (2.0 * A) * A * c_far_rule[2][q];
  const V3 f = cf * (r - fv);
  const long long p = (long long)t * nq + q;
  // every basis function on the triangle writes the same position
  rp[3 * p] = r.x;
  rp[3 * p + 1] = r.y;
  rp[3 * p + 2] = r.z;
  for (int b = 0; b < nrhs; ++b) {
    const double2 x = X[(long long)b * N + m];
    double2* Jp = J + ((long long)b * nt * nq + p) * 3;
    atomicAdd(&Jp[0].x, f.x * x.x);
    atomicAdd(&Jp[0].y, f.x * x.y);
    atomicAdd(&Jp[1].x, f.y * x.x);
    atomicAdd(&Jp[1].y, f.y * x.y);
    atomicAdd(&Jp[2].x, f.z * x.x);
    atomicAdd(&Jp[2].y, f.z * x.y);
  }
}

// Positions as float-float triples and currents in FP32 for the far-field
// kernel: rff [p][6] = (x.hi, x.lo, y.hi, y.lo, z.hi, z.lo), J32 [b][p][3].
__global__ void k_pack_points(const double* __restrict__ rp, const double2* __restrict__ J, float* __restrict__ rff,
                              float2* __restrict__ J32, long long npts, int nrhs) {
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < npts;
       p += (long long)gridDim.x * blockDim.x) {
    for (int d = 0; d < 3; ++d) {
      const ff v = ff_from_double(rp[3 * p + d]);
      rff[6 * p + 2 * d] = v.hi;
      rff[6 * p + 2 * d + 1] = v.lo;
    }
    for (int b = 0; b < nrhs; ++b)
      for (int d = 0; d < 3; ++d) {
        const double2 j = J[((long long)b * npts + p) * 3 + d];
        J32[((long long)b * npts + p) * 3 + d] = make_float2((float)j.x, (float)j.y);
      }
  }
}

// 2 pi = kC1 + kC2 + kC3 with 12-bit kC1 and kC2: n * kC1 and n * kC2 are
// exact for integers |n| < 2^12 (phases below 2.5e4 rad).
constexpr float kC1 = 6.283203125f, kC2 = -1.7814338207244873e-05f, kC3 = -3.482206523131026e-09f;
constexpr float kInv2Pi = 0.15915493667125702f;
constexpr int kFarChunk = 256;   // points staged per shared-memory chunk
constexpr int kFarRun = 64;      // points summed in FP32 before an FP64 add

// cos and sin of the phase k rhat . r for one direction (kr, float-float
// triple) and one point (r, float-float triple).
__device__ __forceinline__ void far_phase(const ff kr[3], const float* r, float& c, float& s) {
  ff p = ff_mul(kr[0], ff{r[0], r[1]});
  p = ff_mad(kr[1], ff{r[2], r[3]}, p);
  p = ff_mad(kr[2], ff{r[4], r[5]}, p);
  const float n = rintf(p.hi * kInv2Pi);
  const float a = __fmaf_rn(-n, kC1, p.hi);  // exact (Sterbenz; n kC1 has <= 24 bits)
  const ff b = ff_two_sum(a, -n * kC2);       // n kC2 exact
  const float lo = __fmaf_rn(-n, kC3, __fadd_rn(b.lo, p.lo));
  float sn, cs;
  sincosf(b.hi, &sn, &cs);
  s = __fmaf_rn(lo, cs, sn);
  c = __fmaf_rn(-lo, sn, cs);
}

// N[b][d][3] += sum over points [p_begin, p_end) of J_p exp(j k rhat_d . r_p)
// for NR right-hand sides b.  Block: 256 threads x D directions (d =
// blockIdx.x * 256 D + i * 256 + threadIdx.x); blockIdx.y picks the point
// range, a multiple of kFarRun.  N (FP64 complex [NR][ndir][3]) must be
// zeroed; partial sums of the point ranges are added atomically.
//
// Bound by FP32 issue: a phase factor takes about 75 instructions, its
// products with one right-hand side's current 12, so the phase is formed once
// for all NR (two right-hand sides of a 2 lambda sphere, 87 k points x 8192
// directions: 5.15 ms one at a time, 2.71 together).  NR D is at most 4, which
// keeps the FP64 accumulators in registers.
template <int NR, int D>
__global__ void __launch_bounds__(256) k_farfield(const float* __restrict__ rff, const float2* __restrict__ J32,
                                                  const double* __restrict__ theta, const double* __restrict__ phi,
                                                  double2* __restrict__ Nacc, long long npts, int ndir,
                                                  long long pts_per_block, double k) {
  __shared__ float sr[kFarChunk][6];
  __shared__ float2 sj[kFarChunk][NR][3];
  ff kr[D][3];
  double2 acc[D][NR][3];
  float2 part[D][NR][3];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const int d = min(blockIdx.x * (256 * D) + i * 256 + threadIdx.x, ndir - 1);
    const double st = sin(theta[d]), ct = cos(theta[d]), sp = sin(phi[d]), cp = cos(phi[d]);
    kr[i][0] = ff_from_double(k * st * cp);
    kr[i][1] = ff_from_double(k * st * sp);
    kr[i][2] = ff_from_double(k * ct);
#pragma unroll
    for (int b = 0; b < NR; ++b)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        acc[i][b][c] = make_double2(0.0, 0.0);
        part[i][b][c] = make_float2(0.f, 0.f);
      }
  }
  const long long p_begin = blockIdx.y * pts_per_block;
  const long long p_end = min(npts, p_begin + pts_per_block);
  for (long long p0 = p_begin; p0 < p_end; p0 += kFarChunk) {
    const int cnt = (int)(p_end - p0 < kFarChunk ? p_end - p0 : kFarChunk);
    __syncthreads();  // the previous chunk has been read
    if (threadIdx.x < cnt) {
      const long long p = p0 + threadIdx.x;
#pragma unroll
      for (int e = 0; e < 6; ++e) sr[threadIdx.x][e] = rff[6 * p + e];
#pragma unroll
      for (int b = 0; b < NR; ++b)
#pragma unroll
        for (int c = 0; c < 3; ++c) sj[threadIdx.x][b][c] = J32[3 * (b * npts + p) + c];
    }
    __syncthreads();
    for (int q = 0; q < cnt; ++q) {
#pragma unroll
      for (int i = 0; i < D; ++i) {
        float c, s;
        far_phase(kr[i], sr[q], c, s);
#pragma unroll
        for (int b = 0; b < NR; ++b)
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            const float2 j = sj[q][b][e];
            part[i][b][e].x = __fmaf_rn(j.x, c, __fmaf_rn(-j.y, s, part[i][b][e].x));
            part[i][b][e].y = __fmaf_rn(j.x, s, __fmaf_rn(j.y, c, part[i][b][e].y));
          }
      }
      if ((q & (kFarRun - 1)) == kFarRun - 1 || q == cnt - 1) {
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
          for (int b = 0; b < NR; ++b)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              acc[i][b][c].x += (double)part[i][b][c].x;
              acc[i][b][c].y += (double)part[i][b][c].y;
              part[i][b][c] = make_float2(0.f, 0.f);
            }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const int d = blockIdx.x * (256 * D) + i * 256 + threadIdx.x;
    if (d >= ndir) continue;
#pragma unroll
    for (int b = 0; b < NR; ++b)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        atomicAdd(&Nacc[3 * ((long long)b * ndir + d) + c].x, acc[i][b][c].x);
        atomicAdd(&Nacc[3 * ((long long)b * ndir + d) + c].y, acc[i][b][c].y);
      }
  }
}

// (N_theta, N_phi) [ndir] from the Cartesian far field N [ndir][3]; blockIdx.y: right-hand side
__global__ void k_far_project(const double2* __restrict__ Nacc, const double* __restrict__ theta,
                              const double* __restrict__ phi, double2* __restrict__ out, int ndir) {
  const int d = blockIdx.x * blockDim.x + threadIdx.x;
  if (d >= ndir) return;
  Nacc += 3LL * blockIdx.y * ndir;
  out += 2LL * blockIdx.y * ndir;
  const double st = sin(theta[d]), ct = cos(theta[d]), sp = sin(phi[d]), cp = cos(phi[d]);
  const double2 nx = Nacc[3 * (long long)d], ny = Nacc[3 * (long long)d + 1], nz = Nacc[3 * (long long)d + 2];
  out[2 * (long long)d] = make_double2(ct * cp * nx.x + ct * sp * ny.x - st * nz.x, ct * cp * nx.y + ct * sp * ny.y - st * nz.y);
  out[2 * (long long)d + 1] = make_double2(-sp * nx.x + cp * ny.x, -sp * nx.y + cp * ny.y);
}

int rhs_planewave(aim_ctx* c, int nrhs, const double* khat, const double* pol, double2* V) {
  AIM_TRY(upload_rules());
  double* dk = nullptr;
  AIM_CUDA_TRY(cudaMallocAsync(&dk, sizeof(double) * 6 * nrhs, c->stream));
  AIM_CUDA_TRY(cudaMemcpyAsync(dk, khat, sizeof(double) * 3 * nrhs, cudaMemcpyHostToDevice, c->stream));
  AIM_CUDA_TRY(cudaMemcpyAsync(dk + 3 * nrhs, pol, sizeof(double) * 3 * nrhs, cudaMemcpyHostToDevice, c->stream));
  dim3 grid((c->N + 127) / 128, nrhs);
  AIM_LAUNCH(c, "k_rhs", k_rhs<<<grid, 128, 0, c->stream>>>(c->d_verts, c->d_tris, c->rwg_tri, c->rwg_free, c->rwg_len, c->tri_area, dk,
                                     dk + 3 * nrhs, V, c->N, c->k, c->alpha < 1.0 ? c->tri_nrm : nullptr,
                                     c->alpha));
  AIM_TRY(launch_check(c, "k_rhs"));
  AIM_CUDA_TRY(cudaFreeAsync(dk, c->stream));
  AIM_CUDA_TRY(cudaStreamSynchronize(c->stream));
  return AIM_OK;
}

// Far fields of NR right-hand sides in one launch.  Point ranges of at least one FP32 run are
// split until every SM has about four blocks, each thread first giving up its extra directions
// (a plate of 1.5 k points and 1152 directions took 1.2 ms a right-hand side on two blocks).
template <int NR>
static int far_fields(aim_ctx* c, const float* rff, const float2* J32, const double* dang, double2* Nacc,
                      long long npts, int ndir) {
  constexpr int DMAX = 4 / NR;
  const long long runs = (npts + kFarRun - 1) / kFarRun;
  const auto launch = [&](auto dirs) -> int {
    constexpr int D = decltype(dirs)::value;
    const int bx = (ndir + 256 * D - 1) / (256 * D);
    const long long by = std::min(runs, std::max<long long>(1, (4LL * 152 + bx - 1) / bx));
    const long long ppb = (runs + by - 1) / by * kFarRun;
    AIM_LAUNCH(c, "k_farfield", (k_farfield<NR, D><<<dim3(bx, (unsigned)((npts + ppb - 1) / ppb)), 256, 0, c->stream>>>(
                                    rff, J32, dang, dang + ndir, Nacc, npts, ndir, ppb, c->k)));
    return launch_check(c, "k_farfield");
  };
  const bool wide = (ndir + 256 * DMAX - 1) / (256 * DMAX) * (runs / 4) >= 4 * 152;
  if constexpr (DMAX > 1)
    if (wide) return launch(std::integral_constant<int, DMAX>{});
  return launch(std::integral_constant<int, 1>{});
}

// Workspace kept with the context between calls up to this size (a call synchronises, so it is
// idle in between); larger ones, and those of a context with a memory budget, live for the call.
constexpr size_t kRcsKeep = 64ull << 20;

int rcs(aim_ctx* c, const double2* X, int nrhs, int ndir, const double* theta, const double* phi, double* sig_tt,
        double* sig_pp) {
  AIM_TRY(upload_rules());
  const int nq = kFarRule * kFarRule;
  const long long npts = (long long)c->nt * nq;
  // one block of memory: what must start as zero first
  size_t total = 0;
  const auto take = [&](size_t bytes) {
    const size_t at = total;
    total += (bytes + 255) / 256 * 256;
    return at;
  };
  const size_t oJ = take(sizeof(double2) * 3 * npts * nrhs), oN = take(sizeof(double2) * 3 * (size_t)ndir * nrhs),
               orp = take(sizeof(double) * 3 * npts), zeroed = total, orff = take(sizeof(float) * 6 * npts),
               oJ32 = take(sizeof(float2) * 3 * npts * nrhs), oang = take(sizeof(double) * 2 * ndir),
               oout = take(sizeof(double2) * 2 * (size_t)ndir * nrhs);
  struct Temp {  // freed on every way out
    void* p = nullptr;
    cudaStream_t st;
    ~Temp() {
      if (p) cudaFreeAsync(p, st);
    }
  } tmp;
  tmp.st = c->stream;
  char* base = nullptr;
  if (total <= kRcsKeep && c->opts.mem_budget == 0) {
    if (c->rcs_work_bytes < total) {
      cudaFree(c->rcs_work);
      c->rcs_work = nullptr;
      c->rcs_work_bytes = 0;
      AIM_CUDA_TRY(cudaMalloc(&c->rcs_work, total));
      c->rcs_work_bytes = total;
    }
    base = (char*)c->rcs_work;
  } else {
    AIM_CUDA_TRY(cudaMallocAsync(&tmp.p, total, c->stream));
    base = (char*)tmp.p;
  }
  double2 *J = (double2*)(base + oJ), *Nacc = (double2*)(base + oN), *out = (double2*)(base + oout);
  double *rp = (double*)(base + orp), *dang = (double*)(base + oang);
  float* rff = (float*)(base + orff);
  float2* J32 = (float2*)(base + oJ32);
  AIM_CUDA_TRY(cudaMemsetAsync(base, 0, zeroed, c->stream));
  AIM_CUDA_TRY(cudaMemcpyAsync(dang, theta, sizeof(double) * ndir, cudaMemcpyHostToDevice, c->stream));
  AIM_CUDA_TRY(cudaMemcpyAsync(dang + ndir, phi, sizeof(double) * ndir, cudaMemcpyHostToDevice, c->stream));
  const long long nthr = (long long)c->N * 2 * nq;
  AIM_LAUNCH(c, "k_point_currents", k_point_currents<<<(unsigned)((nthr + 255) / 256), 256, 0, c->stream>>>(
      c->d_verts, c->d_tris, c->rwg_tri, c->rwg_free, c->rwg_len, c->tri_area, X, J, rp, c->N, c->nt, nrhs));
  AIM_TRY(launch_check(c, "k_point_currents"));
  AIM_LAUNCH(c, "k_pack_points", k_pack_points<<<(unsigned)std::min<long long>((npts + 255) / 256, 152LL * 16), 256, 0,
                                                  c->stream>>>(rp, J, rff, J32, npts, nrhs));
  AIM_TRY(launch_check(c, "k_pack_points"));
  for (int b = 0; b < nrhs;) {
    const float2* Jb = J32 + (size_t)b * npts * 3;
    double2* Nb = Nacc + (size_t)b * ndir * 3;
    if (nrhs - b >= 4) {
      AIM_TRY(far_fields<4>(c, rff, Jb, dang, Nb, npts, ndir));
      b += 4;
    } else if (nrhs - b >= 2) {
      AIM_TRY(far_fields<2>(c, rff, Jb, dang, Nb, npts, ndir));
      b += 2;
    } else {
      AIM_TRY(far_fields<1>(c, rff, Jb, dang, Nb, npts, ndir));
      b += 1;
    }
  }
  for (int b = 0; b < nrhs; b += 32768) {
    AIM_LAUNCH(c, "k_far_project", (k_far_project<<<dim3((ndir + 255) / 256, std::min(32768, nrhs - b)), 256, 0, c->stream>>>(
                                       Nacc + (size_t)b * ndir * 3, dang, dang + ndir, out + (size_t)b * ndir * 2, ndir)));
    AIM_TRY(launch_check(c, "k_far_project"));
  }
  std::vector<double2> h((size_t)2 * ndir * nrhs);
  AIM_CUDA_TRY(cudaMemcpyAsync(h.data(), out, sizeof(double2) * h.size(), cudaMemcpyDeviceToHost, c->stream));
  AIM_CUDA_TRY(cudaStreamSynchronize(c->stream));
  const double fac = c->k * c->k * kEta0 * kEta0 / (4.0 * kPi);
  for (int b = 0; b < nrhs; ++b)
    for (int d = 0; d < ndir; ++d) {
      const double2 nt_ = h[((size_t)b * ndir + d) * 2], np_ = h[((size_t)b * ndir + d) * 2 + 1];
      sig_tt[(size_t)b * ndir + d] = fac * (nt_.x * nt_.x + nt_.y * nt_.y);
      if (sig_pp) sig_pp[(size_t)b * ndir + d] = fac * (np_.x * np_.x + np_.y * np_.y);
    }
  return AIM_OK;
}

}  // namespace aim
