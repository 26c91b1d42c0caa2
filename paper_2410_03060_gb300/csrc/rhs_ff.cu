// Right-hand sides (Eq. (4)) and far field / RCS (Sec. III-A, III-B), both in closed form.
//
// For a rooftop of half-width D centred at s_l on wire p (centre c, direction t):
//   int Lambda(s) exp(j beta s) ds = D exp(j beta s_l) sinc^2(beta D / 2),  sinc(z) = sin z / z.
// RHS:  b_{p,l} = (e.t) exp(-j k khat.c) D exp(-j k (khat.t) s_l) sinc^2(k (khat.t) D / 2)
// far:  F(r) = sum_p t_p D_p exp(j k r.c_p) sinc^2(k (r.t_p) D_p / 2) sum_l j_{p,l} exp(j k (r.t_p) s_l)
//       sigma_s = |e_s . F|^2 / (4 pi), e_s = theta_hat or phi_hat at r.
// The exp(j beta s_l) factors along a wire are a geometric progression in l.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "ctx.h"
#include "rhs_entry.cuh"
#include "sincos64.cuh"

namespace swm {

namespace {

// Right-hand sides, one thread per (wire, incidence; frames: per incidence khat[3], e[3]): the
// wire's incidence-dependent factors once (float64), then its m entries, each with its own phase
// ph0 + beta s_l formed in float64 (and, on the complex64 path, reduced mod 2 pi in float64 before
// the float32 sincos), as rhs_entry does per entry.
template <typename TV>
__global__ void k_rhs_wire(int64_t nw, RhsGeo g, const int64_t* __restrict__ off, double k,
                           const double* __restrict__ frames, int64_t N, cplx<TV>* __restrict__ B) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= nw) return;
  const int r = blockIdx.y;
  const double* f = frames + 6 * r;
  const double tx = g.tx[p], ty = g.ty[p], tz = g.tz[p];
  const double kt = f[0] * tx + f[1] * ty + f[2] * tz;
  const double et = f[3] * tx + f[4] * ty + f[5] * tz;
  const double ph0 = -k * (f[0] * g.cx[p] + f[1] * g.cy[p] + f[2] * g.cz[p]);
  const double Lp = g.L[p];
  const int ns = g.ns[p];
  const double D = Lp / ns;
  const double beta = -k * kt;
  const int64_t o = (int64_t)r * N + off[p];
  if constexpr (sizeof(TV) == 8) {
    const double sc = sinc_d(0.5 * beta * D);
    const double amp = et * D * sc * sc;
    for (int l = 0; l + 1 < ns; ++l) {
      double sa, ca;
      sincos(ph0 + beta * (-0.5 * Lp + (l + 1) * D), &sa, &ca);
      B[o + l] = mkc(amp * ca, amp * sa);
    }
  } else {
    const float sc = sinc_f((float)(0.5 * beta * D));
    const float amp = (float)(et * D) * sc * sc;
    for (int l = 0; l + 1 < ns; ++l) {
      float sa, ca;
      sincosf((float)reduce_2pi(ph0 + beta * (-0.5 * Lp + (l + 1) * D)), &sa, &ca);
      B[o + l] = mkc(amp * ca, amp * sa);
    }
  }
}

// Geometry access: structure-of-arrays (internal) or caller arrays (centres/dirs as nw x 3).
struct Geo {
  const double *cx, *cy, *cz, *tx, *ty, *tz;  // SoA when soa
  const double* c3;                           // AoS centres
  const double* t3;                           // AoS dirs
  const double* L;
  const int32_t* ns;
  const int64_t* off;
  int soa;
  __device__ __forceinline__ void get(int64_t p, double c[3], double t[3]) const {
    if (soa) {
      c[0] = cx[p];
      c[1] = cy[p];
      c[2] = cz[p];
      t[0] = tx[p];
      t[1] = ty[p];
      t[2] = tz[p];
    } else {
      c[0] = c3[3 * p];
      c[1] = c3[3 * p + 1];
      c[2] = c3[3 * p + 2];
      t[0] = t3[3 * p];
      t[1] = t3[3 * p + 1];
      t[2] = t3[3 * p + 2];
    }
  }
};

constexpr int kFFThreads = 128;

__device__ __forceinline__ void obs_frame(const double* obs, int stride, int o, double r[3], double th[3], double ph[3]) {
  double st, ct, sp, cp;
  sincos(obs[(int64_t)o * stride], &st, &ct);
  sincos(obs[(int64_t)o * stride + 1], &sp, &cp);
  r[0] = st * cp;
  r[1] = st * sp;
  r[2] = ct;
  th[0] = ct * cp;
  th[1] = ct * sp;
  th[2] = -st;
  ph[0] = -sp;
  ph[1] = cp;
  ph[2] = 0.0;
}

// sinc(z) and cos(z), sin(z) = z sinc(z): Taylor series to z^12 for z^2 <= kSmallZ2 (first neglected
// terms below 1.3e-19; segments of up to 0.086 wavelengths seen along their axis), else from the table.
constexpr double kSmallZ2 = 0.073;
__device__ __forceinline__ void sinc_cos(double z, double* sinc, double* c) {
  const double x = z * z;
  if (x <= kSmallZ2) {
    *sinc = fma(x, fma(x, fma(x, fma(x, fma(x, fma(x, 1.0 / 6227020800.0, -1.0 / 39916800.0), 1.0 / 362880.0),
                                     -1.0 / 5040.0), 1.0 / 120.0), -1.0 / 6.0), 1.0);
    *c = fma(x, fma(x, fma(x, fma(x, fma(x, fma(x, 1.0 / 479001600.0, -1.0 / 3628800.0), 1.0 / 40320.0),
                                  -1.0 / 720.0), 1.0 / 24.0), -0.5), 1.0);
  } else {
    double s;
    sincos_table(z, &s, c);
    *sinc = s / z;
  }
}

// Far field in float64: one thread per observation, RB incidences (monostatic: its own incidence) and
// chunk of wires, the threads numbered through all observations of the first RB incidences, then of the next.
// grid (ceil(threads / blockDim), nchunks); partial[chunk][r * n_obs + o][3] complex128 (monostatic: [r]).
// Bound by float64 issue, so the count of float64 instructions is what this layout reduces: a wire's
// phases serve all RB incidences; lengths are divided once per CTA, in the staged copy of the chunk's
// wires; one sincos (the wire's first rooftop) comes from the table, the ratio of consecutive
// rooftops e^{2jz} and sinc(z), z = k r.t D / 2, from one pair of short series; the rooftops are
// summed in Horner form, 4 instructions each.  About 45 + 26 per incidence against 180 per incidence
// and wire with CUDA's sincos and a running phase factor: 10,000 wires, 2 incidences, 361 angles
// 2.09 -> 0.71 ms.  Error against 112-bit arithmetic, 1,500 wires at 240 angles, 8.2e-15 (with CUDA's sincos
// 8.5e-15), 200 wires at 400 angles 3.75e-15 (3.72e-15); against a plain float64 evaluation 1.09e-14
// (9.6e-15): that evaluation rounds k r.c by itself, as the former kernel did and this one does not.
constexpr int kFFStage = 32;  // wires staged at a time
template <int RB>
__global__ void __launch_bounds__(kFFThreads) k_far_partial(Geo geo, int64_t nw, int64_t N, double k, int n_rhs,
                                                            const c128* __restrict__ cur, int n_obs,
                                                            const double* __restrict__ obs, int obs_stride, int mono,
                                                            int64_t chunk, c128* __restrict__ partial) {
  struct Wire {
    double c[3], t[3], s1, hd, D;  // hd = D / 2
    int64_t off;
    int n;
  };
  __shared__ Wire sw[kFFStage];
  const int64_t npairs = mono ? n_rhs : (int64_t)n_rhs * n_obs;
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int o = mono ? (int)g : (int)(g % n_obs);
  const int64_t r0 = mono ? g : g / n_obs * RB;
  const int nr = mono ? 1 : (int)min((int64_t)RB, n_rhs - r0);
  const int64_t p0 = blockIdx.y * chunk, p1 = min(nw, p0 + chunk);
  const bool on = r0 < n_rhs;
  double rh[3] = {0, 0, 0};
  if (on) {
    double th[3], ph[3];
    obs_frame(obs, obs_stride, o, rh, th, ph);
  }
  const c128* J = cur + r0 * N;
  double F[RB][6];
#pragma unroll
  for (int b = 0; b < RB; ++b)
#pragma unroll
    for (int i = 0; i < 6; ++i) F[b][i] = 0.0;
  for (int64_t q0 = p0; q0 < p1; q0 += kFFStage) {
    const int cnt = (int)min((int64_t)kFFStage, p1 - q0);
    __syncthreads();
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
      Wire w;
      geo.get(q0 + t, w.c, w.t);
      w.n = geo.ns[q0 + t];
      const double L = geo.L[q0 + t];
      w.D = L / w.n;
      w.s1 = -0.5 * L + w.D;
      w.hd = 0.5 * w.D;
      w.off = geo.off[q0 + t];
      sw[t] = w;
    }
    __syncthreads();
    if (!on) continue;
    for (int t = 0; t < cnt; ++t) {
      const Wire& w = sw[t];
      if (w.n < 2) continue;  // a wire without unknowns (the stateless entries take the counts unchecked)
      const double beta = k * (rh[0] * w.t[0] + rh[1] * w.t[1] + rh[2] * w.t[2]);
      const double x = rh[0] * w.c[0] + rh[1] * w.c[1] + rh[2] * w.c[2];
      double sa, ca, sc, cz;
      sincos_table(fma(k, x, beta * w.s1), &sa, &ca);  // the large product k r.c is not rounded by itself
      const double z = beta * w.hd;
      sinc_cos(z, &sc, &cz);
      const double sz = z * sc, s2 = sz + sz;
      const c128 rat = mkc(fma(-s2, sz, 1.0), s2 * cz);
      const double amp = w.D * sc * sc;
      const c128 z0 = mkc(amp * ca, amp * sa);
      const int n = w.n;
#pragma unroll
      for (int b = 0; b < RB; ++b) {
        if (b >= nr) break;
        const c128* Jp = J + (int64_t)b * N + w.off;
        c128 h = Jp[n - 2];
        for (int l = n - 3; l >= 0; --l) {
          const c128 Jl = Jp[l], hv = h;
          h.re = fma(hv.re, rat.re, fma(-hv.im, rat.im, Jl.re));
          h.im = fma(hv.re, rat.im, fma(hv.im, rat.re, Jl.im));
        }
        const double Sr = h.re * z0.re - h.im * z0.im, Si = h.re * z0.im + h.im * z0.re;
        F[b][0] = fma(w.t[0], Sr, F[b][0]);
        F[b][1] = fma(w.t[0], Si, F[b][1]);
        F[b][2] = fma(w.t[1], Sr, F[b][2]);
        F[b][3] = fma(w.t[1], Si, F[b][3]);
        F[b][4] = fma(w.t[2], Sr, F[b][4]);
        F[b][5] = fma(w.t[2], Si, F[b][5]);
      }
    }
  }
  if (!on) return;
#pragma unroll
  for (int b = 0; b < RB; ++b) {
    if (b >= nr) break;
    const int64_t e = mono ? r0 : (r0 + b) * n_obs + o;
    c128* out = partial + ((int64_t)blockIdx.y * npairs + e) * 3;
    out[0] = mkc(F[b][0], F[b][1]);
    out[1] = mkc(F[b][2], F[b][3]);
    out[2] = mkc(F[b][4], F[b][5]);
  }
}

// One warp per (incidence, observation) pair: sum the chunk partials, then sigma (or, with comp,
// the received components theta_hat . F and phi_hat . F as two complex numbers).  Partial (c, e)
// is at partial + (c * cstride + e * estride) * 3.
__global__ void k_far_reduce(int64_t npairs, int nchunks, const c128* __restrict__ partial, int64_t cstride,
                             int64_t estride, int n_obs, const double* __restrict__ obs, int obs_stride, int mono,
                             double* __restrict__ sigma, int comp = 0) {
  const int64_t e = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (e >= npairs) return;
  double F[6] = {0, 0, 0, 0, 0, 0};
  for (int c = lane; c < nchunks; c += 32) {
    const c128* in = partial + ((int64_t)c * cstride + e * estride) * 3;
    for (int d = 0; d < 3; ++d) {
      F[2 * d] += in[d].re;
      F[2 * d + 1] += in[d].im;
    }
  }
  for (int d = 0; d < 6; ++d) F[d] = warp_sum(F[d]);
  if (lane != 0) return;
  const int o = mono ? (int)e : (int)(e % n_obs);
  double rh[3], th[3], ph[3];
  obs_frame(obs, obs_stride, o, rh, th, ph);
  const double tr = th[0] * F[0] + th[1] * F[2] + th[2] * F[4], ti = th[0] * F[1] + th[1] * F[3] + th[2] * F[5];
  const double pr = ph[0] * F[0] + ph[1] * F[2] + ph[2] * F[4], pi = ph[0] * F[1] + ph[1] * F[3] + ph[2] * F[5];
  if (comp) {
    sigma[4 * e] = tr;
    sigma[4 * e + 1] = ti;
    sigma[4 * e + 2] = pr;
    sigma[4 * e + 3] = pi;
    return;
  }
  sigma[2 * e] = (tr * tr + ti * ti) / kFourPi;
  sigma[2 * e + 1] = (pr * pr + pi * pi) / kFourPi;
}

// Per-wire data of the float32 far field: the centre in cycles, c k / (2 pi), split into a float
// and its float remainder, the direction, the rooftop half-width D = L / n and the first rooftop
// centre s_1 = -L / 2 + D.
struct FFWire {
  float ch[3], cl[3], t[3], D, s1, pad;
};

__global__ void k_ff_wires(int64_t nw, const double* __restrict__ cx, const double* __restrict__ cy,
                           const double* __restrict__ cz, const double* __restrict__ tx, const double* __restrict__ ty,
                           const double* __restrict__ tz, const double* __restrict__ Ls,
                           const int32_t* __restrict__ ns, double k, FFWire* __restrict__ out) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= nw) return;
  const double s = k / (2.0 * kPi);
  const double c[3] = {cx[p] * s, cy[p] * s, cz[p] * s};
  FFWire w;
  for (int i = 0; i < 3; ++i) {
    w.ch[i] = (float)c[i];
    w.cl[i] = (float)(c[i] - (double)w.ch[i]);
  }
  w.t[0] = (float)tx[p];
  w.t[1] = (float)ty[p];
  w.t[2] = (float)tz[p];
  const double D = Ls[p] / ns[p];
  w.D = (float)D;
  w.s1 = (float)(-0.5 * Ls[p] + D);
  w.pad = 0.f;
  out[p] = w;
}

// Observation frame of the float32 far field, formed once per observation: the direction r, split
// into float hi/lo parts for the centre phase and in float64, and theta_hat, phi_hat in float64
// for the final projection.
struct FFObs {
  double r[3], th[3], ph[3];
  float rhi[3], rlo[3];
};

__global__ void k_ff_obs(int n, const double* __restrict__ obs, int obs_stride, FFObs* __restrict__ out) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= n) return;
  FFObs f;
  obs_frame(obs, obs_stride, o, f.r, f.th, f.ph);
  for (int i = 0; i < 3; ++i) {
    f.rhi[i] = (float)f.r[i];
    f.rlo[i] = (float)(f.r[i] - (double)f.rhi[i]);
  }
  out[o] = f;
}

// Sum of the chunk partials of each (incidence, observation) pair (one warp each, partial[c][e][3],
// complex64: the partials are float32 sums), four float accumulators per lane and component in a
// fixed order, then sigma in float64 with the frames of k_ff_obs.
__global__ void k_far_reduce_f32(int64_t npairs, int nchunks, const c64* __restrict__ partial, int n_obs, int mono,
                                 const FFObs* __restrict__ frames, double* __restrict__ sigma) {
  const int64_t e = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (e >= npairs) return;
  float A[4][6];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int d = 0; d < 6; ++d) A[a][d] = 0.f;
  // a lane's next eight chunks are loaded together (one round trip to L2 per 256 chunks)
  for (int c0 = 0; c0 < nchunks; c0 += 256) {
    c64 v[8][3];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int c = c0 + lane + 32 * u;
      const c64* in = partial + ((int64_t)c * npairs + e) * 3;
#pragma unroll
      for (int d = 0; d < 3; ++d) v[u][d] = c < nchunks ? in[d] : mkc(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        A[u & 3][2 * d] += v[u][d].re;
        A[u & 3][2 * d + 1] += v[u][d].im;
      }
  }
  double F[6];
#pragma unroll
  for (int d = 0; d < 6; ++d) F[d] = (double)warp_sum((A[0][d] + A[1][d]) + (A[2][d] + A[3][d]));
  if (lane != 0) return;
  const FFObs& f = frames[mono ? (int)e : (int)(e % n_obs)];
  const double tr = f.th[0] * F[0] + f.th[1] * F[2] + f.th[2] * F[4];
  const double ti = f.th[0] * F[1] + f.th[1] * F[3] + f.th[2] * F[5];
  const double pr = f.ph[0] * F[0] + f.ph[1] * F[2] + f.ph[2] * F[4];
  const double pi = f.ph[0] * F[1] + f.ph[1] * F[3] + f.ph[2] * F[5];
  sigma[2 * e] = (tr * tr + ti * ti) / kFourPi;
  sigma[2 * e + 1] = (pr * pr + pi * pi) / kFourPi;
}

// float32 far field.  The centre phase k r.c = 2 pi (r . c k / 2 pi) is formed modulo one cycle
// from the hi/lo splits of r and of the centre in cycles: each hi*hi product is split exactly
// into p + e with an FMA, and p - rint(p) is exact, so the phase keeps ~1e-7 cycles however far
// the wire is from the origin.  The currents' progression along a wire is summed in Horner form,
// sum_l J_l z0 q^l = z0 (J_0 + q (J_1 + q (...))).  One thread per (incidence, observation) pair
// and chunk of wires; the CTA stages the chunk's wire data (and, with one incidence, its currents)
// in shared memory.  Partials partial[chunk][e][3], complex64.
// One wire's factors for one observation: the centre phase (split in cycles) and the first
// rooftop's offset as z0 = e^{i(2 pi fr + beta s1)}, the ratio of consecutive rooftops
// e^{i beta D}, and the amplitude D sinc^2(beta D / 2), beta = k r.t.
struct FFTerm {
  c64 z0, rat;
  float amp;
};
__device__ __forceinline__ FFTerm ff_term(const FFWire& w, const float* rhi, const float* rlo, float k) {
  const float two_pi = 6.28318530717958647692f;
  float fr = 0.f;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float pr = rhi[i] * w.ch[i];
    const float er = fmaf(rhi[i], w.ch[i], -pr);
    fr += pr - rintf(pr);
    fr += er + rhi[i] * w.cl[i] + rlo[i] * w.ch[i];
  }
  fr -= rintf(fr);
  const float beta = k * (rhi[0] * w.t[0] + rhi[1] * w.t[1] + rhi[2] * w.t[2]);
  float sa, ca, sb, cb;
  __sincosf(fmaf(two_pi, fr, beta * w.s1), &sa, &ca);
  __sincosf(beta * w.D, &sb, &cb);
  const float sc = sinc_f(0.5f * beta * w.D);
  FFTerm t;
  t.z0 = mkc(ca, sa);
  t.rat = mkc(cb, sb);
  t.amp = w.D * sc * sc;
  return t;
}
// h = h * rat + J_l (one Horner step of sum_l J_l rat^l)
__device__ __forceinline__ void horner_step(c64& h, c64 rat, c64 Jl) {
  const c64 hv = h;
  h.re = fmaf(hv.re, rat.re, fmaf(-hv.im, rat.im, Jl.re));
  h.im = fmaf(hv.re, rat.im, fmaf(hv.im, rat.re, Jl.im));
}
// F += t_w amp z0 h
__device__ __forceinline__ void ff_accumulate(float* F, const FFWire& w, const FFTerm& t, c64 h) {
  const c64 acc = t.z0 * h;
  const float Sr = t.amp * acc.re, Si = t.amp * acc.im;
  F[0] = fmaf(w.t[0], Sr, F[0]);
  F[1] = fmaf(w.t[0], Si, F[1]);
  F[2] = fmaf(w.t[1], Sr, F[2]);
  F[3] = fmaf(w.t[1], Si, F[3]);
  F[4] = fmaf(w.t[2], Sr, F[4]);
  F[5] = fmaf(w.t[2], Si, F[5]);
}

constexpr int kFFChunkMax = 64;   // wires per chunk of the float32 far field
constexpr int kFFCurMax = 1024;   // staged currents per chunk
__global__ void __launch_bounds__(kFFThreads) k_far_partial_f32(const FFWire* __restrict__ wires,
                                                                const int32_t* __restrict__ ns,
                                                                const int64_t* __restrict__ off, int64_t nw, int64_t N,
                                                                float k, int n_rhs, const c64* __restrict__ cur,
                                                                int n_obs, const FFObs* __restrict__ frames, int mono,
                                                                int64_t chunk, c64* __restrict__ partial) {
  const int64_t npairs = mono ? n_rhs : (int64_t)n_rhs * n_obs;
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t p0 = blockIdx.y * chunk, p1 = min(nw, p0 + chunk);
  const int64_t ec = e < npairs ? e : npairs - 1;  // threads past the end help stage, then leave
  const int r = mono ? (int)ec : (int)(ec / n_obs);
  const int o = mono ? (int)ec : (int)(ec % n_obs);
  float rhi[3], rlo[3];
  for (int i = 0; i < 3; ++i) {
    rhi[i] = frames[o].rhi[i];
    rlo[i] = frames[o].rlo[i];
  }
  // the chunk's wires and their currents, staged once per CTA
  __shared__ FFWire sw[kFFChunkMax];
  __shared__ int sn[kFFChunkMax];
  __shared__ int soff[kFFChunkMax + 1];
  __shared__ c64 sJ[kFFCurMax];
  const int nwc = (int)(p1 - p0);
  const int64_t o0 = off[p0];
  const int ncur = (int)(off[p1] - o0);
  const bool stage_cur = mono == 0 && n_rhs == 1 && ncur <= kFFCurMax;
  for (int t = threadIdx.x; t < nwc; t += blockDim.x) {
    sw[t] = wires[p0 + t];
    sn[t] = ns[p0 + t];
    soff[t] = (int)(off[p0 + t] - o0);
  }
  if (stage_cur)
    for (int t = threadIdx.x; t < ncur; t += blockDim.x) sJ[t] = cur[o0 + t];
  __syncthreads();
  if (e >= npairs) return;
  const c64* J = cur + (int64_t)r * N + o0;
  float F[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  // two wires per pass: their phases, sincos and Horner sums are independent chains
  int q = 0;
  for (; q + 1 < nwc; q += 2) {
    FFTerm a = ff_term(sw[q], rhi, rlo, k), b = ff_term(sw[q + 1], rhi, rlo, k);
    const int na = sn[q], nb = sn[q + 1];
    const c64* Ja = stage_cur ? sJ + soff[q] : J + soff[q];
    const c64* Jb = stage_cur ? sJ + soff[q + 1] : J + soff[q + 1];
    c64 ha = Ja[na - 2], hb = Jb[nb - 2];
    for (int l = max(na, nb) - 3; l >= 0; --l) {
      if (l <= na - 3) horner_step(ha, a.rat, Ja[l]);
      if (l <= nb - 3) horner_step(hb, b.rat, Jb[l]);
    }
    ff_accumulate(F, sw[q], a, ha);
    ff_accumulate(F, sw[q + 1], b, hb);
  }
  if (q < nwc) {
    const FFTerm a = ff_term(sw[q], rhi, rlo, k);
    const int na = sn[q];
    const c64* Ja = stage_cur ? sJ + soff[q] : J + soff[q];
    c64 ha = Ja[na - 2];
    for (int l = na - 3; l >= 0; --l) horner_step(ha, a.rat, Ja[l]);
    ff_accumulate(F, sw[q], a, ha);
  }
  c64* out = partial + ((int64_t)blockIdx.y * npairs + e) * 3;
  out[0] = mkc(F[0], F[1]);
  out[1] = mkc(F[2], F[3]);
  out[2] = mkc(F[4], F[5]);
}

}  // namespace

// Launch shape shared by the scratch sizing and the launch itself.
static void ff_shape(int64_t nw, int64_t npairs, int64_t& nchunks, int64_t& chunk) {
  // about eight CTAs per SM (four or two where a thread takes two or four incidences), chunks of at
  // least 4 wires (200 wires at 360 angles: 150 CTAs; with 16 wires it was 39)
  const int64_t gx = ceil_div(npairs, kFFThreads);
  nchunks = std::max<int64_t>(1, std::min<int64_t>(ceil_div(nw, 4), ceil_div(8 * 152, gx)));
  nchunks = std::min<int64_t>(nchunks, 65535);
  chunk = ceil_div(nw, nchunks);
  nchunks = ceil_div(nw, chunk);
}

// Launch shape of the float32 far field: one wave of CTAs (`slots` = resident CTAs per SM x SMs,
// whose warps hide each other's sincos and Horner latencies), chunks of at least 8 wires and at
// most kFFChunkMax (the size of the CTA's staging arrays).
static void ff32_shape(int64_t nw, int64_t npairs, int64_t slots, int64_t& nchunks, int64_t& chunk) {
  const int64_t gx = ceil_div(npairs, kFFThreads);
  nchunks = std::max<int64_t>(1, std::min<int64_t>(ceil_div(nw, 8), ceil_div(std::max<int64_t>(slots, 1), gx)));
  nchunks = std::min<int64_t>(nchunks, 65535);
  chunk = std::min<int64_t>(ceil_div(nw, nchunks), kFFChunkMax);
  nchunks = ceil_div(nw, chunk);
}

// Resident CTAs of the float32 far-field kernel on the whole GPU.
static int64_t ff32_slots(const swm_ctx* ctx) {
  int occ = 0;
  if (occupancy_cached((const void*)k_far_partial_f32, kFFThreads, 0, &occ) != cudaSuccess || occ < 1) occ = 8;
  return (int64_t)occ * std::max(ctx->nsm, 1);
}


// The per-wire data of the float32 far field: allocated on the context's stream (before the build
// forks its second stream), filled on stream s.
int far_field_alloc(swm_ctx* ctx) {
  if (ctx->prec != SWM_C64) return SWM_OK;
  SWM_TRY(dalloc(ctx, ctx->build_bufs, &ctx->ffw, sizeof(FFWire) * ctx->nw));
  return SWM_OK;
}

int prepare_far_field(swm_ctx* ctx, cudaStream_t s) {
  if (ctx->prec != SWM_C64) return SWM_OK;
  k_ff_wires<<<(unsigned)ceil_div(ctx->nw, 256), 256, 0, s>>>(ctx->nw, ctx->cx, ctx->cy, ctx->cz, ctx->tx,
                                                                        ctx->ty, ctx->tz, ctx->L, ctx->ns, ctx->k,
                                                                        (FFWire*)ctx->ffw);
  SWM_LAUNCHED();
  return SWM_OK;
}

int far_field_f32_launch(swm_ctx* ctx, int n_obs, const double* obs, int obs_stride, bool mono, double* sigma,
                         void* scratch, size_t scratch_bytes) {
  const int R = ctx->n_rhs;
  const int64_t npairs = mono ? R : (int64_t)R * n_obs;
  int64_t nchunks, chunk;
  ff32_shape(ctx->nw, npairs, ff32_slots(ctx), nchunks, chunk);
  const size_t part_bytes = (size_t)nchunks * npairs * 3 * sizeof(c64);
  if (part_bytes + sizeof(FFObs) * (size_t)n_obs > scratch_bytes)
    return ctx->fail(SWM_EINVAL, "far field: scratch too small");
  c64* part = (c64*)scratch;
  FFObs* frames = reinterpret_cast<FFObs*>((char*)scratch + part_bytes);  // part_bytes is a multiple of 8
  k_ff_obs<<<(unsigned)ceil_div(n_obs, 128), 128, 0, ctx->stream>>>(n_obs, obs, obs_stride, frames);
  SWM_LAUNCHED();
  dim3 grid((unsigned)ceil_div(npairs, kFFThreads), (unsigned)nchunks);
  k_far_partial_f32<<<grid, kFFThreads, 0, ctx->stream>>>((const FFWire*)ctx->ffw, ctx->ns, ctx->off, ctx->nw, ctx->N,
                                                          (float)ctx->k, R, (const c64*)ctx->Xv, n_obs, frames, mono,
                                                          chunk, part);
  SWM_LAUNCHED();
  k_far_reduce_f32<<<(unsigned)ceil_div(npairs * 32, 256), 256, 0, ctx->stream>>>(npairs, (int)nchunks, part, n_obs,
                                                                                  mono, frames, sigma);
  SWM_LAUNCHED();
  return SWM_OK;
}

int compute_rhs(swm_ctx* ctx, int n_inc, const double* frames_dev) {
  SWM_TRY(ensure_rowinfo(ctx));
  const RhsGeo g{ctx->cx, ctx->cy, ctx->cz, ctx->tx, ctx->ty, ctx->tz, ctx->L, ctx->ns};
  const dim3 grid((unsigned)ceil_div(ctx->nw, 128), (unsigned)n_inc);
  ctx->prof_begin(SWM_K_RHS);
  if (ctx->prec == SWM_C128)
    k_rhs_wire<double><<<grid, 128, 0, ctx->stream>>>(ctx->nw, g, ctx->off, ctx->k, frames_dev, ctx->N,
                                                      (c128*)ctx->Bv);
  else
    k_rhs_wire<float><<<grid, 128, 0, ctx->stream>>>(ctx->nw, g, ctx->off, ctx->k, frames_dev, ctx->N,
                                                     (c64*)ctx->Bv);
  ctx->prof_end(SWM_K_RHS);
  SWM_LAUNCHED();
  return SWM_OK;
}

int compute_rhs_f64(swm_ctx* ctx, int n_inc, const double* frames_dev, c128* out) {
  SWM_TRY(ensure_rowinfo(ctx));
  const RhsGeo g{ctx->cx, ctx->cy, ctx->cz, ctx->tx, ctx->ty, ctx->tz, ctx->L, ctx->ns};
  const dim3 grid((unsigned)ceil_div(ctx->nw, 128), (unsigned)n_inc);
  k_rhs_wire<double><<<grid, 128, 0, ctx->stream>>>(ctx->nw, g, ctx->off, ctx->k, frames_dev, ctx->N, out);
  SWM_LAUNCHED();
  return SWM_OK;
}

size_t far_field_f32_scratch_bytes(const swm_ctx* ctx, int64_t npairs, int n_obs) {
  int64_t nchunks, chunk;
  ff32_shape(ctx->nw, npairs, ff32_slots(ctx), nchunks, chunk);
  return (size_t)nchunks * npairs * 3 * sizeof(c64) + sizeof(FFObs) * (size_t)n_obs;
}

size_t far_field_scratch_bytes(int64_t nw, int64_t npairs) {
  int64_t nchunks, chunk;
  ff_shape(nw, npairs, nchunks, chunk);
  return (size_t)nchunks * npairs * 3 * sizeof(c128);
}

// Far field + RCS.  Scratch must hold at least 3 * npairs complex128; with less than
// far_field_scratch_bytes() the wire range is cut into fewer chunks.
int far_field_launch(cudaStream_t st, int64_t* launches, const c128* cur, int64_t nw, int64_t N, const double* c3,
                     const double* t3, const double* cx, const double* cy, const double* cz, const double* tx,
                     const double* ty, const double* tz, const double* Ls, const int32_t* ns, const int64_t* off,
                     bool soa, double k, int n_rhs, int n_obs, const double* obs, int obs_stride, bool mono,
                     double* sigma, void* scratch, size_t scratch_bytes, std::string* err, bool components) {
  const int64_t npairs = mono ? n_rhs : (int64_t)n_rhs * n_obs;
  int64_t nchunks, chunk;
  ff_shape(nw, npairs, nchunks, chunk);
  const int64_t fit = (int64_t)(scratch_bytes / (3 * sizeof(c128) * (size_t)npairs));
  if (fit < 1) {
    *err = "far field: scratch too small for " + std::to_string(npairs) + " (incidence, observation) pairs";
    return SWM_EINVAL;
  }
  if (nchunks > fit) {
    nchunks = fit;
    chunk = ceil_div(nw, nchunks);
    nchunks = ceil_div(nw, chunk);
  }
  Geo g{cx, cy, cz, tx, ty, tz, c3, t3, Ls, ns, off, soa ? 1 : 0};
  c128* part = (c128*)scratch;
  // incidences per thread: the fewest float64 instructions over the warps of a wire (see k_far_partial).
  // 10,000 wires, one direction of 181 incidences: 91 threads of two 0.46 ms, against 4.40 ms with one busy
  // lane in each of 46 warps of four; 4 incidences x 1: 0.32 ms in four threads, 0.38 ms in one.
  auto threads_of = [&](int b) { return mono ? (int64_t)n_rhs : ceil_div(n_rhs, b) * n_obs; };
  auto cost = [&](int b) { return ceil_div(threads_of(b), 32) * (45 + 26 * std::min(b, n_rhs)); };
  int RB = 1;
  if (!mono)
    for (int b : {2, 4})
      if (cost(b) < cost(RB)) RB = b;
  const int64_t nt = threads_of(RB);
  const int threads = (int)std::min<int64_t>(kFFThreads, ceil_div(nt, 32) * 32);
  const int64_t gx = ceil_div(nt, threads);
  const dim3 grid((unsigned)gx, (unsigned)nchunks);
  auto kern = RB == 1 ? k_far_partial<1> : RB == 2 ? k_far_partial<2> : k_far_partial<4>;
  kern<<<grid, threads, 0, st>>>(g, nw, N, k, n_rhs, cur, n_obs, obs, obs_stride, mono ? 1 : 0, chunk, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    *err = std::string("far field launch: ") + cudaGetErrorString(e);
    return SWM_ECUDA;
  }
  k_far_reduce<<<(unsigned)ceil_div(npairs * 32, 256), 256, 0, st>>>(npairs, (int)nchunks, part, npairs, 1, n_obs,
                                                                     obs, obs_stride, mono, sigma,
                                                                     components ? 1 : 0);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    *err = std::string("far field reduce launch: ") + cudaGetErrorString(e);
    return SWM_ECUDA;
  }
  if (launches) *launches += 2;
  return SWM_OK;
}

}  // namespace swm
