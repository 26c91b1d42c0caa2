// The block-sparse product w = u + E u of the incidence-minor BiCGSTAB (complex64, several
// incidences) over a copy of E laid out for it (product form 76).
//
// Each wire of the cloud is one record in the product's order: its column map (K entries, padded to 16
// bytes), then its m x K entries of E column by column, mp = m rounded up to even entries per column.
// The order sorts the wires by (rows, columns) within windows of kPackWin wires of the cell order, so
// the wires that share a warp run the same unrolled row loop for about the same number of columns,
// while the concurrently running wires stay near one another in space (their gathers hit L2).
//
// A thread takes one wire and up to four incidences (two 16-byte gathers per column, of pairs q and
// q + RQ, each contiguous over the wire's RQ threads); floor(32 / RQ) wires share a warp.  Every warp
// stages its wires' records in its own part of shared memory by cp.async, as many columns at a time as
// fit, and multiplies with the rows unrolled: per entry of E one 8-byte shared load (the same address
// for a wire's threads, at a constant offset from the column's) and 16 multiply-adds, gathers two
// columns ahead.  No CTA barrier: a warp waits for its own copies only.
//
// Why this shape: the product is bound by the latency of its gathers and by issue, not by HBM.  Two
// incidences per thread in 80 registers (form 75) read each entry of E twice as often and spend most of
// their instructions on 64-bit addresses, predicates and packing operands for FFMA2 (which executes at
// half FFMA's rate, so plain FFMA loses nothing); here 384 M warp instructions per launch become 318 M
// and each warp has twice the gathers in flight.  250,000 wires at 37 incidences 0.696 -> 0.567 ms per
// launch, 1,000,000 wires 2.90 -> 2.36 ms; 120,000 at 13 incidences 0.37 (form 73) -> 0.20 ms; 60,000 at
// 91 incidences 0.64 (form 73) -> 0.44 ms.  Measured and not taken at 37 incidences: the gathers four
// columns ahead 0.74 ms, the first gathers beside the copies 0.65 ms (both spill), five and six CTAs per
// SM 0.84 and 1.14 ms (spills), CTAs of two warps 0.65 ms.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "ctx.h"
#include "krylov_common.cuh"

namespace swm {

namespace {

constexpr int kPackWin = 4096;
constexpr int kPackThreads = 128;
constexpr int kPackWarpBytes = 12288;  // staged records per warp; 16 warps per SM (128 registers)
constexpr int kPackSlack = 128;        // a row loop may read past its wire's last column, up to 8 entries

struct PackRec {
  int64_t at;         // first byte of the record
  int32_t row0, K, m, p;
};
static_assert(sizeof(PackRec) == 24, "record");

__device__ __forceinline__ int pack_mp(int m) { return (m + 1) & ~1; }
__device__ __forceinline__ int pack_k(int K) { return (K + 1) & ~1; }
__device__ __forceinline__ int pack_cb(int K) { return (4 * K + 15) & ~15; }

// One CTA per window: bitonic sort of (rows, columns, position); then the record sizes in order, or, with
// `order`, only the wires' numbers.
__global__ void __launch_bounds__(1024) k_pack_order(int64_t nw, Layout lay, const int64_t* __restrict__ off,
                                                     PackRec* __restrict__ rec, int64_t* __restrict__ bytes,
                                                     int32_t* __restrict__ order) {
  __shared__ unsigned long long key[kPackWin];
  const int64_t base = (int64_t)blockIdx.x * kPackWin;
  for (int t = threadIdx.x; t < kPackWin; t += blockDim.x) {
    const int64_t p = base + t;
    unsigned hi = 0xffffffffu;
    if (p < nw) hi = ((unsigned)(off[p + 1] - off[p]) << 24) | (unsigned)min(lay.K[p], (1 << 24) - 1);
    key[t] = ((unsigned long long)hi << 32) | (unsigned)t;
  }
  __syncthreads();
  for (int k = 2; k <= kPackWin; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < kPackWin; t += blockDim.x) {
        const int o = t ^ j;
        if (o > t) {
          const unsigned long long a = key[t], b = key[o];
          if ((a > b) == ((t & k) == 0)) {
            key[t] = b;
            key[o] = a;
          }
        }
      }
      __syncthreads();
    }
  for (int t = threadIdx.x; t < kPackWin; t += blockDim.x) {
    const int64_t i = base + t;
    if (i >= nw) continue;
    const int64_t p = base + (int64_t)(key[t] & 0xffffffffu);
    if (order) {
      order[i] = (int32_t)p;
      continue;
    }
    PackRec r;
    r.at = 0;
    r.row0 = (int32_t)off[p];
    r.K = pack_k(lay.K[p]);
    r.m = (int32_t)(off[p + 1] - off[p]);
    r.p = (int32_t)p;
    rec[i] = r;
    bytes[i] = pack_cb(r.K) + (int64_t)8 * pack_mp(r.m) * r.K;
  }
}

__global__ void k_pack_place(int64_t nw, const int64_t* __restrict__ at, PackRec* __restrict__ rec) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < nw) rec[i].at = at[i];
}

// The records: a warp per wire, 32 columns at a time (E read along its rows, written down the columns).
__global__ void __launch_bounds__(256) k_pack_fill(int64_t nw, const PackRec* __restrict__ rec, Layout lay,
                                                   const c64* __restrict__ E, unsigned char* __restrict__ pack) {
  const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= nw) return;
  const PackRec r = rec[i];
  const int mp = pack_mp(r.m);
  int32_t* cols = reinterpret_cast<int32_t*>(pack + r.at);
  c64* ent = reinterpret_cast<c64*>(pack + r.at + pack_cb(r.K));
  const int32_t* cm = lay.colmap + lay.cmbase[r.p];
  const c64* e = E + lay.rowbase[r.p];
  const int K = lay.K[r.p];  // r.K is K rounded up to even: a zero column at the wire's own first row
  for (int c = lane; c < pack_cb(r.K) / 4; c += 32) cols[c] = c < K ? cm[c] : r.row0;
  for (int c = lane; c < r.K; c += 32) {
    for (int q = 0; q < mp; q += 2) {
      const c64 z = mkc(0.f, 0.f);
      const c64 a = c < K ? e[(int64_t)q * K + c] : z;
      const c64 b = c < K && q + 1 < r.m ? e[(int64_t)(q + 1) * K + c] : z;
      *reinterpret_cast<float4*>(ent + (int64_t)c * mp + q) = make_float4(a.re, a.im, b.re, b.im);
    }
  }
}

__device__ __forceinline__ void pack_cp16(unsigned sdst, const void* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sdst), "l"(gsrc) : "memory");
}

// Accumulators of MW rows and four incidences over the staged columns [0, n) of the thread's wire.
template <int MW>
struct PackAcc {
  float4 a[MW], b[MW];  // pair q and pair q + RQ
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < MW; ++i) a[i] = b[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  static __device__ __forceinline__ void fma2(float4& s, float2 e, float4 x) {
    s.x = fmaf(e.x, x.x, s.x);
    s.y = fmaf(e.x, x.y, s.y);
    s.z = fmaf(e.x, x.z, s.z);
    s.w = fmaf(e.x, x.w, s.w);
    s.x = fmaf(-e.y, x.y, s.x);
    s.y = fmaf(e.y, x.x, s.y);
    s.z = fmaf(-e.y, x.w, s.z);
    s.w = fmaf(e.y, x.z, s.w);
  }
  struct X2 {
    float4 a0, b0, a1, b1;  // two columns of pairs q and q + RQ
  };
  static __device__ __forceinline__ X2 gather(const int32_t* cs, const c64* __restrict__ xa, const c64* __restrict__ xb,
                                              int xst) {
    const int2 c = *reinterpret_cast<const int2*>(cs);
    const int64_t o0 = (int64_t)c.x * xst, o1 = (int64_t)c.y * xst;
    X2 x;
    x.a0 = __ldg(reinterpret_cast<const float4*>(xa + o0));
    x.b0 = __ldg(reinterpret_cast<const float4*>(xb + o0));
    x.a1 = __ldg(reinterpret_cast<const float4*>(xa + o1));
    x.b1 = __ldg(reinterpret_cast<const float4*>(xb + o1));
    return x;
  }
  __device__ __forceinline__ void mul(const float2* es, int mp, const X2& x) {
#pragma unroll
    for (int i = 0; i < MW; ++i) {
      const float2 e = es[i];
      fma2(a[i], e, x.a0);
      fma2(b[i], e, x.b0);
    }
#pragma unroll
    for (int i = 0; i < MW; ++i) {
      const float2 e = es[mp + i];
      fma2(a[i], e, x.a1);
      fma2(b[i], e, x.b1);
    }
  }
  // n is even (an odd wire has a zero column), the gathers run two columns ahead
  __device__ __forceinline__ void run(int n, const int32_t* cs, const float2* es, int mp, const c64* __restrict__ xa,
                                      const c64* __restrict__ xb, int xst) {
    if (n <= 0) return;
    X2 p = gather(cs, xa, xb, xst);
#pragma unroll 1
    for (;;) {
      if (n > 2) {
        const X2 t = gather(cs + 2, xa, xb, xst);
        mul(es, mp, p);
        es += 2 * mp;
        if (n > 4) p = gather(cs + 4, xa, xb, xst);
        mul(es, mp, t);
        es += 2 * mp;
        cs += 4;
        n -= 4;
        if (n <= 0) break;
      } else {
        mul(es, mp, p);
        break;
      }
    }
  }
};

struct PackArgs {
  const PackRec* rec;
  const unsigned char* pack;
  int64_t nw;
  const c64 *U, *B;
  c64* W;
  int xst, RQ;  // entries per row of the vectors, threads per wire
};

// Rows i0 .. i0 + MW - 1 of the warp's wires (every lane; lanes without a wire have K = m = 0).
template <bool RES, int MW>
__device__ __forceinline__ void pack_rows(const PackArgs& A, int i0, int64_t at, int row0, int K, int m, int q, int g,
                                          int kmax, int kc, unsigned char* slot, int pa, int pb, bool wa, bool wb) {
  PackAcc<MW> acc;
  acc.clear();
  const int mp = pack_mp(m);
  const unsigned ss = (unsigned)__cvta_generic_to_shared(slot);
  const unsigned char* cols = A.pack + at;
  const unsigned char* ent = cols + pack_cb(K);
  const c64 *xa = A.U + 2 * pa, *xb = A.U + 2 * pb;
#pragma unroll 1
  for (int c0 = 0; c0 < kmax; c0 += kc) {
    const int n = min(kc, K - c0);
    if (c0 > 0) __syncwarp();  // every lane is done with the columns before
    if (n > 0) {
      const int cb = (4 * n + 15) & ~15, eb = 8 * mp * n;
      for (int x = 16 * q; x < cb; x += 16 * A.RQ) pack_cp16(ss + x, cols + 4 * (int64_t)c0 + x);
      const unsigned char* src = ent + (int64_t)8 * mp * c0;
      for (int x = 16 * q; x < eb; x += 16 * A.RQ) pack_cp16(ss + 4 * kc + x, src + x);
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    if (wa || wb)
      acc.run(n, reinterpret_cast<const int32_t*>(slot), reinterpret_cast<const float2*>(slot + 4 * kc) + i0, mp, xa,
              xb, A.xst);
  }
#pragma unroll
  for (int i = 0; i < MW; ++i) {
    if (i0 + i >= m) continue;
    const int64_t o = (int64_t)(row0 + i0 + i) * A.xst;
    auto put = [&](int pr, float4 s) {
      const float4 u = *reinterpret_cast<const float4*>(A.U + o + 2 * pr);
      float4 v = make_float4(u.x + s.x, u.y + s.y, u.z + s.z, u.w + s.w);
      if (RES) {
        const float4 b = *reinterpret_cast<const float4*>(A.B + o + 2 * pr);
        v = make_float4(b.x - v.x, b.y - v.y, b.z - v.z, b.w - v.w);
      }
      *reinterpret_cast<float4*>(A.W + o + 2 * pr) = v;
    };
    if (wa) put(pa, acc.a[i]);
    if (wb) put(pb, acc.b[i]);
  }
}

// w = u + E u for the pairs with an active incidence, or with RES w = b - (u + E u) for all.
template <bool RES>
__global__ void __launch_bounds__(kPackThreads, 4) k_spmv_pack(KPtr P, PackArgs A) {
  if (!RES && (P.st->cycle_done || P.st->j >= P.st->jmax)) return;
  extern __shared__ __align__(16) unsigned char sm_pk[];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int RQ = A.RQ, G = 32 / RQ;
  const int g = lane / RQ, q = lane - g * RQ;
  const int64_t pos = ((int64_t)blockIdx.x * (kPackThreads / 32) + wp) * G + g;
  const int np = A.xst >> 1;
  const int pa = blockIdx.y * 2 * RQ + q;
  int pb = pa + RQ;
  auto any = [&](int pr) {
    return pr < np && (RES || P.active[2 * pr] || (2 * pr + 1 < P.R && P.active[2 * pr + 1]));
  };
  const bool live = g < G && pos < A.nw;
  const bool wa = live && any(pa), wb = live && any(pb);
  if (!__any_sync(0xffffffffu, wa || wb)) return;
  int64_t at = 0;
  int row0 = 0, K = 0, m = 0;
  if (live) {
    const PackRec r = A.rec[pos];
    at = r.at;
    row0 = r.row0;
    K = r.K;
    m = r.m;
  }
  const int kmax = __reduce_max_sync(0xffffffffu, K), mmax = __reduce_max_sync(0xffffffffu, m);
  const int mpmax = pack_mp(mmax);
  // bytes per wire; not a multiple of 128, so that wires in step read different banks
  int sw = (kPackWarpBytes / G) & ~15;
  if (!(sw & 127)) sw -= 16;
  const int kc = max(4, (sw / (8 * max(mpmax, 1) + 4)) & ~3);  // columns staged at a time
  unsigned char* slot = sm_pk + wp * kPackWarpBytes + min(g, G - 1) * sw;
  const int sa = min(pa, np - 1), sb = min(pb, np - 1);  // pairs past the end gather the last one
  for (int i0 = 0; i0 < mmax; i0 += 8) {
    if (i0 > 0) __syncwarp();
    const int mw = min(8, mmax - i0);
#define SWM_PACK_CASE(W)                                                                                  \
  case W:                                                                                                 \
    pack_rows<RES, W>(A, i0, at, row0, K, m, q, g, kmax, kc, slot, sa, sb, wa, wb); \
    break;
    switch (mw) {
      SWM_PACK_CASE(1)
      SWM_PACK_CASE(2)
      SWM_PACK_CASE(3)
      SWM_PACK_CASE(4)
      SWM_PACK_CASE(5)
      SWM_PACK_CASE(6)
      SWM_PACK_CASE(7)
      default:
        pack_rows<RES, 8>(A, i0, at, row0, K, m, q, g, kmax, kc, slot, sa, sb, wa, wb);
    }
#undef SWM_PACK_CASE
  }
}

// Threads per wire: the RQ <= 32 with the most useful lanes (pairs of incidences over the slots of
// the ceil(pairs / 2 RQ) passes, times the warp lanes that hold a wire), less 6 % for every pass
// after the first, which reads E again.
int pack_rq(int np) {
  int best = 2;
  double be = 0.0;
  for (int q = 2; q <= 32; ++q) {  // at most 16 wires per warp: 768 bytes each hold four columns of 16 rows
    const int gy = (int)ceil_div(np, 2 * q);
    const double e = (double)np / (gy * 2 * q) * ((32 / q) * q / 32.0) - 0.06 * (gy - 1);
    if (e > be + 1e-9) {
      be = e;
      best = q;
    }
  }
  return best;
}

}  // namespace

// The copy's bytes at most: column maps rounded up to 16 bytes, one padding column and one padding row of
// entries per wire.
static size_t pack_most(const swm_ctx* ctx) {
  return std::max<size_t>((size_t)4 * ctx->offd.ncm + (size_t)(20 + 8 * (kMaxM + 1)) * ctx->nw +
                              (size_t)8 * (ctx->offd.nval + ctx->offd.ncm),
                          16);
}

// Only a second copy of an E that leaves the memory mostly free: up to a ninth of the card (a million
// wires take 5 GB).  Larger systems keep form 75, which reads E where it lies.
constexpr size_t kPackMost = (size_t)32 << 30;

static int make_pack(swm_ctx* ctx) {
  const int64_t nw = ctx->nw;
  SWM_CK(allow_max_dyn_smem((const void*)k_spmv_pack<true>, ctx->smem_optin));
  SWM_CK(allow_max_dyn_smem((const void*)k_spmv_pack<false>, ctx->smem_optin));
  if (!ctx->pkrec) {
    std::vector<Buf> tmp;
    int64_t *bytes = nullptr, *at = nullptr;
    int rc = dalloc(ctx, ctx->pattern_bufs, &ctx->pkrec, sizeof(PackRec) * nw);
    if (rc >= 0) rc = dalloc(ctx, tmp, (void**)&bytes, sizeof(int64_t) * nw);
    if (rc >= 0) rc = dalloc(ctx, tmp, (void**)&at, sizeof(int64_t) * (nw + 1));
    if (rc >= 0 && !ctx->pkrec) rc = SWM_ENOMEM;  // given back to make room
    if (rc >= 0) {
      PackRec* rec = reinterpret_cast<PackRec*>(ctx->pkrec);
      k_pack_order<<<(unsigned)ceil_div(nw, kPackWin), 1024, 0, ctx->stream>>>(nw, ctx->offd, ctx->off, rec, bytes, nullptr);
      SWM_LAUNCHED();
      const void* in[1] = {bytes};
      const int is64[1] = {1};
      int64_t* out[1] = {at};
      rc = exclusive_scan_multi(ctx, 1, in, is64, out, nw);
      if (rc >= 0 && !ctx->pkrec) rc = SWM_ENOMEM;
      if (rc >= 0) {
        k_pack_place<<<(unsigned)ceil_div(nw, 256), 256, 0, ctx->stream>>>(nw, at, rec);
        SWM_LAUNCHED();
      }
    }
    dfree_group(ctx, tmp);
    if (rc < 0) return rc;
  }
  if (!ctx->pack) {
    SWM_TRY(dalloc(ctx, ctx->build_bufs, &ctx->pack, pack_most(ctx)));
    if (!ctx->pkrec) return SWM_ENOMEM;  // given back to make room
    k_pack_fill<<<(unsigned)ceil_div(nw * 32, 256), 256, 0, ctx->stream>>>(
        nw, reinterpret_cast<const PackRec*>(ctx->pkrec), ctx->offd, (const c64*)ctx->Zp, (unsigned char*)ctx->pack);
    SWM_LAUNCHED();
  }
  return SWM_OK;
}

int ensure_pack(swm_ctx* ctx, bool* ok) {
  *ok = pack_most(ctx) <= kPackMost && !ctx->pack_refused;
  if (!*ok) return SWM_OK;
  const std::string err = ctx->err;
  const int rc = make_pack(ctx);
  if (rc >= 0) return rc;
  drop_pack(ctx);  // what there is of it is not complete
  *ok = false;
  if (rc != SWM_ENOMEM) return rc;
  ctx->err = err;  // the solve goes on without the copy
  release_spare(ctx);
  ctx->pack_refused = true;
  return SWM_OK;
}

// Sort (39 to 46 us), scan and placement (about 10 us) and fill (4 us and 0.4 ms per GB: 29 MB 16 us, 298 MB
// 121 us), measured from 300 to 300,000 wires.
double pack_ms(const swm_ctx* ctx) { return 0.06 + 0.4e-9 * (double)pack_most(ctx); }

int ensure_row_order(swm_ctx* ctx) {
  if (ctx->worder || ctx->nw <= 0 || ctx->nw > INT32_MAX) return SWM_OK;
  // under a caller's capture the order would not exist before the graph runs: the wires as they lie
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  SWM_CK(cudaStreamIsCapturing(ctx->stream, &cs));
  if (cs != cudaStreamCaptureStatusNone) return SWM_OK;
  int32_t* w = nullptr;
  const std::string err = ctx->err;
  const int rc = dalloc(ctx, ctx->pattern_bufs, (void**)&w, sizeof(int32_t) * ctx->nw);
  if (rc == SWM_ENOMEM) {  // the products run without it
    ctx->err = err;
    return SWM_OK;
  }
  if (rc < 0) return rc;
  k_pack_order<<<(unsigned)ceil_div(ctx->nw, kPackWin), 1024, 0, ctx->stream>>>(ctx->nw, ctx->offd, ctx->off, nullptr,
                                                                               nullptr, w);
  SWM_LAUNCHED();
  ctx->worder = w;
  return SWM_OK;
}

int launch_pack(swm_ctx* ctx, cudaStream_t s, const KPtr& P, const c64* src, c64* dst, const c64* Bv, int xst, bool res) {
  PackArgs A{};
  A.rec = reinterpret_cast<const PackRec*>(ctx->pkrec);
  A.pack = (const unsigned char*)ctx->pack;
  A.nw = ctx->nw;
  A.U = src;
  A.B = Bv;
  A.W = dst;
  A.xst = xst;
  A.RQ = pack_rq(xst / 2);
  const int wires = 32 / A.RQ * (kPackThreads / 32);
  const dim3 grid((unsigned)ceil_div(ctx->nw, wires), (unsigned)ceil_div(xst / 2, 2 * A.RQ));
  const size_t smem = (size_t)kPackWarpBytes * (kPackThreads / 32) + kPackSlack;
  if (res)
    k_spmv_pack<true><<<grid, kPackThreads, smem, s>>>(P, A);
  else
    k_spmv_pack<false><<<grid, kPackThreads, smem, s>>>(P, A);
  return SWM_OK;
}

}  // namespace swm
