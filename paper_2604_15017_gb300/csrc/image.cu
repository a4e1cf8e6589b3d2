// Image formation and its adjoint: delay-and-sum (Eq. das) and its transpose (Eq.
// das_adjoint), the Hilbert envelope along depth, log compression with the dynamic-range clip
// (Sec. 2.3.4), the l1/l2 loss (Eq. weighted_l1_l2_loss) and the envelope/log VJP.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>
#include <utility>

#include <cooperative_groups.h>

#include "image.cuh"

namespace cg = cooperative_groups;

namespace usrt {

// ------------------------------------------------------------------------------------------
// DAS delays (Eq. das), in samples, evaluated in float-float so that the interpolation
// position of a ~4000-sample delay is resolved to ~1e-6 samples:
//   u = (x sin(th) + z cos(th) + W/2 |sin(th)|) fs / c_bf + sqrt((x - x_e)^2 + z^2) fs / c_bf
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ ff ff_div_f(ff a, float b) {
  const float q = __fdiv_rn(a.hi, b);
  const float r = __fmaf_rn(-q, b, a.hi);
  return ff_fast(q, __fdiv_rn(__fadd_rn(r, a.lo), b));
}
// coordinate v0 + (v1 - v0) i / (n - 1)
__device__ __forceinline__ ff grid_coord(float v0, float v1, int i, int n) {
  if (n <= 1) return ff{v0, 0.0f};
  const ff span = ff_div_f(ff_two_sum(v1, -v0), (float)(n - 1));
  const ff off = ff_mulf(span, (float)i);
  return ff_addx(ff{v0, 0.0f}, off);
}
struct DasGeo {
  ff k;       // fs / c_bf
  ff half_w;  // (n_elem - 1) pitch / 2
};
__device__ __forceinline__ DasGeo das_geo(const Acq& q) {
  DasGeo g;
  g.k = ff_divf(q.fs, q.cbf);
  g.half_w = ff_mulf(ff{0.5f * (float)(q.ne - 1), 0.0f}, q.pitch);
  return g;
}
__device__ __forceinline__ ff das_utx(const Acq& q, const DasGeo& g, ff x, ff z, int t) {
  const float st = q.sin_tx[t];
  ff p = ff_mulf(x, st);
  p = ff_addx(p, ff_mul(z, ff{q.cos_tx[t], q.cos_lo[t]}));
  p = ff_addx(p, ff_mulf(g.half_w, fabsf(st)));
  return ff_mul(p, g.k);
}
// Receive side, in samples: the pixel's lateral position and squared depth and the element's
// position are scaled by fs / c_bf once, so that a (pixel, element) pair costs one difference, one
// square, one sum and a square root refined by its exact residual (relative error 2^-45): ~40
// instructions where the unscaled form, with an IEEE root and divide, took ~110.
struct DasRx {
  ff x;   // x fs / c_bf
  ff z2;  // (z fs / c_bf)^2
};
__device__ __forceinline__ DasRx das_rx(const DasGeo& g, ff x, ff z) {
  const ff zk = ff_mul(z, g.k);
  return DasRx{ff_mul(x, g.k), ff_mul(zk, zk)};
}
__device__ __forceinline__ ff das_elem(const Acq& q, const DasGeo& g, int e) {  // x_e fs / c_bf
  return ff_mul(ff_mulf(ff{(float)e - 0.5f * (float)(q.ne - 1), 0.0f}, q.pitch), g.k);
}
__device__ __forceinline__ ff das_urx(const DasRx& p, ff xe) {
  const ff dx = ff_addx(p.x, ff{-xe.hi, -xe.lo});
  const float h = __fmul_rn(dx.hi, dx.hi);
  const float l = __fmaf_rn(__fmul_rn(2.0f, dx.hi), dx.lo, __fmaf_rn(dx.hi, dx.hi, -h));
  const ff s = ff_two_sum(h, p.z2.hi);
  const float r2 = fmaxf(s.hi, 1e-30f);  // a pixel on the element: 1e-15 samples
  const float inv = rsqrtf(r2);
  const float r = __fmul_rn(r2, inv);
  const float res = __fadd_rn(__fmaf_rn(-r, r, r2), __fadd_rn(s.lo, __fadd_rn(l, p.z2.lo)));
  return ff{r, __fmul_rn(res, __fmul_rn(0.5f, inv))};
}
// the same for two elements at once (their negated positions side by side), operation by operation in
// packed FP32: the same bits, half the issue slots
struct DasRx2 {
  f32x2 xh, xl, zh, zl;
};
__device__ __forceinline__ DasRx2 das_rx2(const DasRx& p) {
  return DasRx2{pack2(p.x.hi, p.x.hi), pack2(p.x.lo, p.x.lo), pack2(p.z2.hi, p.z2.hi), pack2(p.z2.lo, p.z2.lo)};
}
__device__ __forceinline__ f32x2 two_sum2(f32x2 a, f32x2 b, f32x2& e) {
  const f32x2 s = add2(a, b), bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
  return s;
}
__device__ __forceinline__ void das_urx2(const DasRx2& p, f32x2 nxh, f32x2 nxl, ff& u0, ff& u1) {
  f32x2 e, e2;
  const f32x2 s = two_sum2(p.xh, nxh, e);
  const f32x2 t = add2(e, add2(p.xl, nxl));
  const f32x2 dh = add2(s, t), dl = sub2(t, sub2(dh, s));
  const f32x2 h = mul2(dh, dh);
  const f32x2 l = fma2(add2(dh, dh), dl, fma2(dh, dh, neg2(h)));
  const float2 sh = unpack2(two_sum2(h, p.zh, e2));
  const float ra = fmaxf(sh.x, 1e-30f), rb = fmaxf(sh.y, 1e-30f);
  const f32x2 r2 = pack2(ra, rb), inv = pack2(rsqrtf(ra), rsqrtf(rb));
  const f32x2 r = mul2(r2, inv);
  const f32x2 res = add2(fma2(neg2(r), r, r2), add2(e2, add2(l, p.zl)));
  const float2 hi = unpack2(r), lo = unpack2(mul2(res, mul2(pack2(0.5f, 0.5f), inv)));
  u0 = ff{hi.x, lo.x};
  u1 = ff{hi.y, lo.y};
}
__device__ __forceinline__ float hann_w(int e, int ne) {
  return 0.5f * (1.0f - cospif(2.0f * (float)(e + 1) / (float)(ne + 1)));
}
// Element weight w_e(x, z) of Eq. das: F-number <= 0, the Hann window over the array; F > 0,
// the dynamic receive aperture: cos^2(pi xi / 2) for |xi| < 1, xi = (x_e - x) / a, half-width
// a = max(z / 2F, pitch).  dw_dp (optional): its derivative in the pitch (x_e = p (e - (N_e -
// 1)/2), and a = p where clamped).
__device__ __forceinline__ float apod_w(const Acq& q, const Img& im, float x, float z, int e,
                                        float* dw_dp = nullptr) {
  if (dw_dp) *dw_dp = 0.0f;
  if (!(im.fnum > 0.0f)) return hann_w(e, q.ne);
  const float ce = (float)e - 0.5f * (float)(q.ne - 1);
  const float ad = z / (2.0f * im.fnum);
  const bool clamped = ad < q.pitch;
  const float a = clamped ? q.pitch : ad;
  const float xi = (ce * q.pitch - x) / a;
  if (fabsf(xi) >= 1.0f) return 0.0f;
  const float c = cospif(0.5f * xi);
  if (dw_dp) *dw_dp = -0.5f * PI_F * sinpif(xi) * (ce - (clamped ? xi : 0.0f)) / a;
  return c * c;
}
// The transmit and receive delays of a pixel are each split once into whole samples and a
// fraction in [0, 1) (exactly, from their float-float values); a tap then adds the two parts:
// the one float addition of the fractions rounds by at most 2^-24 samples.
__device__ __forceinline__ float2 das_split(ff u) {
  int i;
  float f;
  ff_floor(u, i, f);
  return make_float2(__int_as_float(i), f);
}
__device__ __forceinline__ void das_tap(float2 a, float2 b, int& i, float& f) {
  f = __fadd_rn(a.y, b.y);
  i = __float_as_int(a.x) + __float_as_int(b.x);
  if (f >= 1.0f) {
    f = __fsub_rn(f, 1.0f);  // exact on [1, 2)
    ++i;
  }
}
// One check for all taps of a pixel and two elements: the extremes of the transmit delays' whole
// samples (das_tx_range, once per pixel) and the two receive delays'.  Nothing passes where a
// transmit delay is past 2^22 samples, nor where a receive delay is past 2^24: records are
// shorter (make_acq), and no sum overflows.
__device__ __forceinline__ void das_tx_range(int& imin, int& imax) {
  if (imin < -(1 << 22) || imax > (1 << 22)) imin = -(1 << 28), imax = 0;
}
__device__ __forceinline__ bool das_inside(int ia, int ib, int imin, int imax, int ns) {
  const int lo = max(-(1 << 24), min(min(ia, ib), 1 << 24)), hi = max(-(1 << 24), min(max(ia, ib), 1 << 24));
  return lo + imin >= 0 && hi + imax + 2 < ns;  // every tap's two samples lie inside the record
}

// DAS.  A block owns a tile of DAS_TL lines x DAS_TD depths; a warp covers 8 lines x 4 depths.
// Bound by the L1's gathers: neighbouring depths are ~3 samples apart, neighbouring lines less than
// one on average, so a warp of 32 depths read 4 lines of 128 bytes per load and 12 bytes per tap
// from the L2, an 8 x 4 patch reads 1-2 lines and ~2.5 bytes per tap.  The transmit delays are
// staged per pixel in shared memory, their row offsets folded in; the receive delay serves all
// transmits of an element; taps are checked against the record once per (pixel, element), by
// the pixel's smallest and largest transmit delay.  The elements of a chunk are shared out over
// DAS_ES groups of threads, so that small images fill the GPU too; a pixel's sums over the
// transmits meet in shared memory and are weighted and added in element order by one thread.
// A thread takes two neighbouring elements at a time: their delays in packed FP32, one read of each
// transmit delay, four independent gathers in flight.  128 elements, 256 x 1024 pixels: 16
// transmits 921 us at first, 378 with an element at a time, 342 in pairs (5.4e8 taps); 1 transmit
// 239, 133, 109 us (there the delays, 3.4e7 of them, are most of it).  Elements split two ways
// instead of four, patches of 16 x 2 and 4 x 8, more blocks at fewer registers: equal or slower.
constexpr int DAS_THREADS = 256;
constexpr int DAS_ES = 4, DAS_TL = 8, DAS_TD = 8, DAS_PX = DAS_TL * DAS_TD;
constexpr int DAS_EC = 32;  // elements per chunk
static_assert(DAS_PX * DAS_ES == DAS_THREADS && DAS_TL == 8 && DAS_EC % (2 * DAS_ES) == 0,
              "a warp is 8 lines x 4 depths, its elements come in pairs");
__host__ __device__ constexpr size_t das_smem(int ne, int ntx, bool dynamic) {
  return sizeof(ulonglong2) * ((ne + 1) / 2) + sizeof(float2) * (size_t)ntx * DAS_PX +
         sizeof(float) * (ne + (dynamic ? 4 : 2) * DAS_EC * DAS_PX);
}
__global__ void __launch_bounds__(DAS_THREADS) k_das(Acq q, Img im, const float* __restrict__ rf,
                                                     float* __restrict__ irf) {
  extern __shared__ __align__(16) ulonglong2 das_sm[];
  ulonglong2* xe_s = das_sm;                                  // [(ne + 1) / 2] negated positions of element pairs
  float2* utx_s = reinterpret_cast<float2*>(xe_s + (q.ne + 1) / 2);  // [ntx][DAS_PX]: (first sample + row offset, fraction)
  float* w_s = reinterpret_cast<float*>(utx_s + q.ntx * DAS_PX);     // [ne] Hann weights
  float* s_s = w_s + q.ne;                                    // [2][DAS_EC][DAS_PX] sums over the transmits
  float* wd_s = s_s + 2 * DAS_EC * DAS_PX;                    // the same of the dynamic aperture's weights
  const DasGeo g = das_geo(q);
  const int tiles_d = (im.nd + DAS_TD - 1) / DAS_TD;
  const int tl = blockIdx.x / tiles_d;
  const int px = threadIdx.x % DAS_PX, es = threadIdx.x / DAS_PX;
  const int l = tl * DAS_TL + (px & 7), d = (blockIdx.x - tl * tiles_d) * DAS_TD + (px >> 3);
  const bool valid = l < im.nl && d < im.nd;
  const ff x = grid_coord(im.x0, im.x1, min(l, im.nl - 1), im.nl), z = grid_coord(im.z0, im.z1, min(d, im.nd - 1), im.nd);
  const int tstride = q.ne * q.ns;  // between one element's rows of two transmits
  for (int t = es; t < q.ntx; t += DAS_ES) {
    const float2 u = das_split(das_utx(q, g, x, z, t));
    utx_s[t * DAS_PX + px] = make_float2(__int_as_float(__float_as_int(u.x) + t * tstride), u.y);
  }
  for (int e = threadIdx.x; e < q.ne; e += DAS_THREADS) w_s[e] = hann_w(e, q.ne);
  for (int k = threadIdx.x; k < (q.ne + 1) / 2; k += DAS_THREADS) {
    const ff a = das_elem(q, g, 2 * k), b = das_elem(q, g, min(2 * k + 1, q.ne - 1));
    xe_s[k] = make_ulonglong2(pack2(-a.hi, -b.hi), pack2(-a.lo, -b.lo));
  }
  __syncthreads();
  int imin = 0x7FFFFFFF, imax = -0x7FFFFFFF;
  for (int t = 0; t < q.ntx; ++t) {
    const int i = __float_as_int(utx_s[t * DAS_PX + px].x) - t * tstride;
    imin = min(imin, i);
    imax = max(imax, i);
  }
  das_tx_range(imin, imax);
  const DasRx2 p = das_rx2(das_rx(g, x, z));
  const bool dynamic = im.fnum > 0.0f;
  float acc = 0.0f;
  for (int e0 = 0, buf = 0; e0 < q.ne; e0 += DAS_EC, buf ^= 1) {
    const int e1 = min(e0 + DAS_EC, q.ne);
    float* sb = s_s + buf * DAS_EC * DAS_PX + px;
    float* wb = wd_s + buf * DAS_EC * DAS_PX + px;
    for (int e = e0 + 2 * es; e < e1; e += 2 * DAS_ES) {  // elements e and e + 1 (e0 is even)
      const ulonglong2 xe = xe_s[e >> 1];
      ff ua, ub;
      das_urx2(p, xe.x, xe.y, ua, ub);
      const float2 ra = das_split(ua), rb = das_split(ub);
      const int ia = __float_as_int(ra.x), ib = __float_as_int(rb.x);
      const bool two = e + 1 < e1;
      float sa = 0.0f, sb2 = 0.0f;
      if (das_inside(ia, ib, imin, imax, q.ns)) {
        const float2 ba = make_float2(__int_as_float(ia + e * q.ns), ra.y);
        // past the last element of an odd array the pair's second is the last one again
        const float2 bb = make_float2(__int_as_float(ib + (two ? e + 1 : e) * q.ns), rb.y);
#pragma unroll 4
        for (int t = 0; t < q.ntx; ++t) {
          const float2 u = utx_s[t * DAS_PX + px];
          int i, j;
          float f, h;
          das_tap(u, ba, i, f);
          das_tap(u, bb, j, h);
          const float v0 = __ldg(&rf[i]), v1 = __ldg(&rf[i + 1]), w0 = __ldg(&rf[j]), w1 = __ldg(&rf[j + 1]);
          sa += fmaf(f, v1 - v0, v0);
          sb2 += fmaf(h, w1 - w0, w0);
        }
      } else {
        for (int k = 0; k < (two ? 2 : 1); ++k) {
          const float2 b = k ? rb : ra;
          float s = 0.0f;
          for (int t = 0; t < q.ntx; ++t) {
            float2 u = utx_s[t * DAS_PX + px];
            u.x = __int_as_float(__float_as_int(u.x) - t * tstride);
            int i;
            float f;
            das_tap(u, b, i, f);
            const float* row = rf + (size_t)t * tstride + (size_t)(e + k) * q.ns;
            const float v0 = (i >= 0 && i < q.ns) ? __ldg(&row[i]) : 0.0f;
            const float v1 = (i + 1 >= 0 && i + 1 < q.ns) ? __ldg(&row[i + 1]) : 0.0f;
            s += fmaf(f, v1 - v0, v0);
          }
          if (k) sb2 = s;
          else sa = s;
        }
      }
      sb[(e - e0) * DAS_PX] = sa;
      if (dynamic) wb[(e - e0) * DAS_PX] = apod_w(q, im, x.hi, z.hi, e);
      if (two) {
        sb[(e + 1 - e0) * DAS_PX] = sb2;
        if (dynamic) wb[(e + 1 - e0) * DAS_PX] = apod_w(q, im, x.hi, z.hi, e + 1);
      }
    }
    __syncthreads();  // the other buffer is written next; this one again only after the next barrier
    if (es == 0)
      for (int e = e0; e < e1; ++e)
        acc = fmaf(dynamic ? wb[(e - e0) * DAS_PX] : w_s[e], sb[(e - e0) * DAS_PX], acc);
  }
  if (es == 0 && valid) irf[(size_t)l * im.nd + d] = acc;
}

// ------------------------------------------------------------------------------------------
// DAS with the channel-data windows staged in shared memory by TMA bulk copies.
// A CTA owns a 4-line x 128-depth pixel tile (two pixels per thread).  For every (element,
// transmit) the samples the tile can touch form one contiguous window of the row (the delay
// grows monotonically with depth along each line).  One pipeline stage holds the windows of
// all transmits of one element: an elected thread issues them as cp.async.bulk copies that
// complete on the stage's mbarrier, the CTA interpolates from shared memory, and the stage is
// refilled with a later element once the CTA has moved on.  Every wait is bounded in time:
// on expiry the CTA records the timeout, stops using the staged buffers and reads the channel
// data directly (same result).
// ------------------------------------------------------------------------------------------
constexpr int DT_THREADS = 256, DT_DEPTHS = 128, DT_LINES = 4, DT_PX = 2;
constexpr int DT_SMEM_MAX = 200 * 1024;
constexpr int DT_STAGES = 3;
constexpr int DT_WIN = 512;            // floats per staged window
constexpr int DT_MAX_WINDOWS = 4096;   // (element, transmit) windows per tile
constexpr long long DT_WAIT_CYCLES = 2000000000ll;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
// bounded wait for phase `parity` of a stage's barrier; false on expiry
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > DT_WAIT_CYCLES) return false;
  return true;
}

// plain FP32 delay of pixel (l, d) for (element e, transmit t), in samples
__device__ __forceinline__ float das_delay_f32(const Acq& q, const Img& im, int l, int d, int e, int t) {
  const float k = q.fs / q.cbf;
  const float st = q.sin_tx[t], ct = q.cos_tx[t];
  const float hw = 0.5f * (q.ne - 1) * q.pitch * fabsf(st);
  const float xe = (e - 0.5f * (q.ne - 1)) * q.pitch;
  const float x = im.nl > 1 ? im.x0 + (im.x1 - im.x0) * (float)l / (float)(im.nl - 1) : im.x0;
  const float z = im.nd > 1 ? im.z0 + (im.z1 - im.z0) * (float)d / (float)(im.nd - 1) : im.z0;
  return (x * st + z * ct + hw) * k + sqrtf((x - xe) * (x - xe) + z * z) * k;
}
// sample window [start, start + len) covering delays in [lo, hi], padded by 2 samples and
// aligned to 4 (len 0: nothing in the record; -1: longer than max_len)
__device__ __forceinline__ int2 das_window_of(int ns, float lo, float hi, int max_len) {
  int a = (int)floorf(lo) - 2, b = (int)ceilf(hi) + 3;
  a = max(0, a) & ~3;
  b = min(ns, (b + 3) & ~3);
  if (b <= a) return make_int2(0, 0);
  if (b - a > max_len) return make_int2(a, -1);
  return make_int2(a, b - a);
}
// sample window of (element e, transmit t) for the tile: the delays at the tile's corners (the
// delay grows monotonically with depth along each line)
__device__ int2 das_window(const Acq& q, const Img& im, int l0, int l1, int d0, int d1, int e, int t) {
  float lo = 3.0e38f, hi = -3.0e38f;
  for (int l = l0; l <= l1; ++l)
    for (int r = 0; r < 2; ++r) {
      const float u = das_delay_f32(q, im, l, r ? d1 : d0, e, t);
      lo = fminf(lo, u);
      hi = fmaxf(hi, u);
    }
  return das_window_of(q.ns, lo, hi, DT_WIN);
}

__global__ void __launch_bounds__(DT_THREADS) k_das_tma(Acq q, Img im, const float* __restrict__ rf,
                                                        float* __restrict__ irf, int* status) {
  extern __shared__ __align__(128) unsigned char smraw[];
  const int ntx = q.ntx;
  float* win = reinterpret_cast<float*>(smraw);                                // [DT_STAGES][ntx][DT_WIN]
  uint64_t* bar = reinterpret_cast<uint64_t*>(win + (size_t)DT_STAGES * ntx * DT_WIN);  // [DT_STAGES]
  int2* table = reinterpret_cast<int2*>(bar + DT_STAGES);                     // [ne][ntx]
  float2* utx_s = reinterpret_cast<float2*>(table + q.ne * ntx);              // [ntx][DT_PX][DT_THREADS]
  __shared__ int use_tma;
  const int tiles_d = (im.nd + DT_DEPTHS - 1) / DT_DEPTHS;
  const int l0 = (blockIdx.x / tiles_d) * DT_LINES, d0 = (blockIdx.x % tiles_d) * DT_DEPTHS;
  const int l1 = min(l0 + DT_LINES - 1, im.nl - 1), d1 = min(d0 + DT_DEPTHS - 1, im.nd - 1);
  const int d = d0 + (threadIdx.x % DT_DEPTHS);
  int lp[DT_PX];
  bool valid[DT_PX];
  ff x[DT_PX], z[DT_PX];
  const DasGeo g = das_geo(q);
#pragma unroll
  for (int p = 0; p < DT_PX; ++p) {
    lp[p] = l0 + (threadIdx.x / DT_DEPTHS) + 2 * p;
    valid[p] = lp[p] < im.nl && d < im.nd;
    x[p] = grid_coord(im.x0, im.x1, valid[p] ? lp[p] : l0, im.nl);
    z[p] = grid_coord(im.z0, im.z1, valid[p] ? d : d0, im.nd);
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < DT_STAGES; ++s) mbar_init(&bar[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    use_tma = 1;
  }
  for (int w = threadIdx.x; w < q.ne * ntx; w += blockDim.x)
    table[w] = das_window(q, im, l0, l1, d0, d1, w / ntx, w % ntx);
  for (int t = 0; t < ntx; ++t)
#pragma unroll
    for (int p = 0; p < DT_PX; ++p)
      utx_s[(t * DT_PX + p) * DT_THREADS + threadIdx.x] = das_split(das_utx(q, g, x[p], z[p], t));
  __syncthreads();
  int issued[DT_STAGES];  // uses issued per stage (meaningful in thread 0, the only issuer)
  for (int k = 0; k < DT_STAGES; ++k) issued[k] = 0;
  auto issue = [&](int e) {  // all transmit windows of element e into stage e % DT_STAGES
    if (e >= q.ne) return;
    const int s = e % DT_STAGES;
    ++issued[s];
    uint32_t bytes = 0;
    for (int t = 0; t < ntx; ++t) {
      const int2 b = table[e * ntx + t];
      if (b.y > 0) bytes += (uint32_t)b.y * 4u;
    }
    mbar_arrive_tx(&bar[s], bytes);  // arrival + expected bytes; phase completes when all land
    for (int t = 0; t < ntx; ++t) {
      const int2 b = table[e * ntx + t];
      if (b.y > 0)
        bulk_g2s(win + ((size_t)s * ntx + t) * DT_WIN, rf + ((size_t)t * q.ne + e) * q.ns + b.x, (uint32_t)b.y * 4u,
                 &bar[s]);
    }
  };
  if (threadIdx.x == 0)
    for (int e = 0; e < DT_STAGES; ++e) issue(e);
  float acc[DT_PX];
#pragma unroll
  for (int p = 0; p < DT_PX; ++p) acc[p] = 0.0f;
  for (int e = 0; e < q.ne; ++e) {
    const int s = e % DT_STAGES;
    bool staged = use_tma;
    if (staged && !mbar_wait_bounded(&bar[s], (uint32_t)((e / DT_STAGES) & 1))) {
      use_tma = 0;  // benign race: every writer stores 0
      atomicOr(status, ST_TIMEOUT);
      staged = false;
    }
    float2 ur[DT_PX];
#pragma unroll
    for (int p = 0; p < DT_PX; ++p) ur[p] = das_split(das_urx(das_rx(g, x[p], z[p]), das_elem(q, g, e)));
    float se[DT_PX];
#pragma unroll
    for (int p = 0; p < DT_PX; ++p) se[p] = 0.0f;
    for (int t = 0; t < ntx; ++t) {
      const int2 b = table[e * ntx + t];
      const float* row = rf + ((size_t)t * q.ne + e) * q.ns;
      const float* sw = win + ((size_t)s * ntx + t) * DT_WIN;
#pragma unroll
      for (int p = 0; p < DT_PX; ++p) {
        int i;
        float f;
        das_tap(utx_s[(t * DT_PX + p) * DT_THREADS + threadIdx.x], ur[p], i, f);
        const int rel = i - b.x;
        float a0, a1;
        if (staged && b.y > 0 && rel >= 0 && rel + 1 < b.y) {
          a0 = sw[rel];
          a1 = sw[rel + 1];
        } else {
          a0 = (i >= 0 && i < q.ns) ? __ldg(&row[i]) : 0.0f;
          a1 = (i + 1 >= 0 && i + 1 < q.ns) ? __ldg(&row[i + 1]) : 0.0f;
        }
        se[p] += fmaf(f, a1 - a0, a0);
      }
    }
#pragma unroll
    for (int p = 0; p < DT_PX; ++p) acc[p] = fmaf(apod_w(q, im, x[p].hi, z[p].hi, e), se[p], acc[p]);
    __syncthreads();  // the CTA is done with stage s
    if (threadIdx.x == 0 && use_tma) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(e + DT_STAGES);
    }
  }
  // drain: every issued copy was waited on above unless a wait expired; then wait (bounded)
  // once more for the last use issued into each stage before the CTA's shared memory goes away
  if (threadIdx.x == 0 && !use_tma)
    for (int s = 0; s < DT_STAGES; ++s)
      if (issued[s] > 0) (void)mbar_wait_bounded(&bar[s], (uint32_t)((issued[s] - 1) & 1));
#pragma unroll
  for (int p = 0; p < DT_PX; ++p)
    if (valid[p]) irf[(size_t)lp[p] * im.nd + d] = acc[p];
}

size_t das_tma_smem(const Acq& q) {
  return sizeof(float) * DT_STAGES * (size_t)q.ntx * DT_WIN + sizeof(uint64_t) * DT_STAGES +
         sizeof(int2) * (size_t)q.ne * q.ntx + sizeof(float2) * (size_t)q.ntx * DT_PX * DT_THREADS;
}

// transposed DAS: every tap scatters w_e (1 - f) g and w_e f g to its two samples
// The transposed DAS accumulates in 64-bit fixed point so that its sums do not depend on the
// order of the atomics (integer addition is associative, and wraps harmlessly in between).  A
// pixel's weighted gradient w_e dL/dI becomes the integer W nearest w_e dL/dI 2^k, with 2^k the
// largest power of two for which max |dL/dI| 2^k < 2^40 and (pixel count) x max |dL/dI| 2^k
// < 2^62; a tap then splits W exactly into its two samples' shares, s1 = floor(W F / 2^23) and
// s0 = W - s1, F the interpolation fraction in units of 2^-23.  The second bound holds every
// entry's sum, since a pixel adds at most |W| to one row (w_e <= 1); the first keeps W F below
// 2^63 and lets the tiled kernel hold a tile's partial sums in two 32-bit words (below).  The
// quantum is 2^-40 of the largest pixel's contribution (2^-43 for 2^22 pixels), far below FP32
// rounding.  max |dL/dI| comes from an integer atomicMax on the float bits of |dL/dI|
// (order-independent too); a non-finite dL/dI makes every entry NaN.
__global__ void k_das_adj_max(const float* __restrict__ gi, int n, unsigned int* maxbits) {
  unsigned int m = 0u;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    m = max(m, __float_as_uint(fabsf(gi[i])));  // NaN's bits lie above +inf's
  // one atomic per block: with one per warp 8192 of them queued up at one address (7 -> 4 us)
  __shared__ unsigned int best;
  if (threadIdx.x == 0) best = 0u;
  __syncthreads();
  m = __reduce_max_sync(0xFFFFFFFFu, m);
  if ((threadIdx.x & 31) == 0 && m) atomicMax(&best, m);
  __syncthreads();
  if (threadIdx.x == 0 && best) atomicMax(maxbits, best);
}
constexpr unsigned int F32_INF_BITS = 0x7F800000u;
constexpr int DAS_ADJ_V_BITS = 40;  // |W| < 2^40 in fixed point
constexpr int DAS_ADJ_F_BITS = 23;  // interpolation fraction in units of 2^-23
static_assert(DAS_ADJ_V_BITS + DAS_ADJ_F_BITS <= 63, "W F fits a signed 64-bit integer");
// the exponent k: max |dL/dI| < 2^e and npx <= 2^c give npx max |dL/dI| < 2^(e + c)
__device__ __forceinline__ int das_adj_kexp(int npx, unsigned int maxbits) {
  if (maxbits == 0u) return 0;
  const int e = ilogbf(__uint_as_float(maxbits)) + 1;
  const int c = 32 - __clz(max(npx - 1, 1));
  return min(DAS_ADJ_V_BITS, 62 - c) - e;
}
// v (|v| < 2^43) rounded to the nearest integer (ties to even, as __float2ll_rn) and split as
// hi 2^22 + lo with lo in [0, 2^22), by FP32 additions only: a float -> 64-bit integer
// conversion runs on the FP64 pipe, a small fraction of the FP32 rate on this part.  Adding
// 2^23 (same sign as v) leaves an integer, exactly when |v| < 2^23 (larger v are integers
// already); 1.5 2^23 added with rounding toward -inf gives floor(v / 2^22) in the float's low
// mantissa bits; the remainder is an exact subtraction.
constexpr int DAS_ADJ_LO_BITS = 22;
__device__ __forceinline__ void das_adj_fixed(float v, int& hi, int& lo) {
  const float c = copysignf(8388608.0f, v);
  const float vr = fabsf(v) < 8388608.0f ? __fsub_rn(__fadd_rn(v, c), c) : v;
  const float h = __fadd_rd(vr * (1.0f / 4194304.0f), 12582912.0f);  // 1.5 2^23 + floor(vr / 2^22)
  hi = __float_as_int(h) - 0x4B400000;
  const float hf = __fsub_rn(h, 12582912.0f);
  const float lf = __fsub_rn(vr, hf * 4194304.0f);  // in [0, 2^22), exact
  lo = __float_as_int(__fadd_rn(lf, 8388608.0f)) - 0x4B000000;
}
// v 2^k (|v 2^k| < 2^43) without the range checks of ldexpf: two factors, each a normal float
__device__ __forceinline__ float das_adj_scaled(float v, int k) {
  const int a = k / 2, b = k - a;
  return v * __int_as_float((127 + a) << 23) * __int_as_float((127 + b) << 23);
}
// the two samples' shares of W = wh 2^22 + wl at interpolation fraction f in [0, 1): 1 + f
// rounded to the float grid of [1, 2) puts F = round(f 2^23) in the mantissa; the second
// sample's share is s1 = floor(W F / 2^23) = h1 2^22 + l1 with l1 in [0, 2^22), cut out of the
// 64-bit product; the first's is W - s1, word by word (its low word may be negative)
__device__ __forceinline__ void das_adj_second(long long W, float f, int& h1, int& l1) {
  const uint32_t F = (uint32_t)(__float_as_int(__fadd_rn(1.0f, f)) - 0x3F800000);
  const unsigned long long lo = (unsigned long long)(uint32_t)W * F;
  const int ph = (int)(W >> 32) * (int)F + (int)(lo >> 32);
  h1 = ph >> (DAS_ADJ_LO_BITS + DAS_ADJ_F_BITS - 32);
  l1 = (int)(__funnelshift_r((uint32_t)lo, (uint32_t)ph, DAS_ADJ_F_BITS) & ((1u << DAS_ADJ_LO_BITS) - 1u));
}
__device__ __forceinline__ long long das_adj_join(int hi, int lo) {
  return (long long)hi * (1ll << DAS_ADJ_LO_BITS) + (long long)lo;
}
__global__ void k_das_adj_finish(const unsigned long long* __restrict__ acc, long long n, int npx,
                                 const unsigned int* maxbits, float* grf) {
  const unsigned int mb = *maxbits;
  const int k = das_adj_kexp(npx, mb);
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n; j += (long long)gridDim.x * blockDim.x)
    grf[j] = mb >= F32_INF_BITS ? __int_as_float(0x7FC00000) : ldexpf(__ll2float_rn((long long)acc[j]), -k);
}

__global__ void __launch_bounds__(DAS_THREADS) k_das_adj(Acq q, Img im, const float* __restrict__ gi,
                                                         unsigned long long* acc, const unsigned int* maxbits) {
  extern __shared__ float2 utx_s[];
  const int npx = im.nl * im.nd;
  const DasGeo g = das_geo(q);
  const unsigned int mb = *maxbits;
  if (mb >= F32_INF_BITS) return;  // k_das_adj_finish writes NaN
  const int kexp = das_adj_kexp(npx, mb);
  for (int base = blockIdx.x * DAS_THREADS; base < npx; base += gridDim.x * DAS_THREADS) {
    const int p = base + threadIdx.x;
    const bool valid = p < npx;
    const int l = valid ? p / im.nd : 0, d = valid ? p - l * im.nd : 0;
    const ff x = grid_coord(im.x0, im.x1, l, im.nl), z = grid_coord(im.z0, im.z1, d, im.nd);
    for (int t = 0; t < q.ntx; ++t) utx_s[t * DAS_THREADS + threadIdx.x] = das_split(das_utx(q, g, x, z, t));
    const float gv = valid ? das_adj_scaled(gi[p], kexp) : 0.0f;
    if (gv != 0.0f) {
      for (int e = 0; e < q.ne; ++e) {
        const float2 ur = das_split(das_urx(das_rx(g, x, z), das_elem(q, g, e)));
        int wh, wl;
        das_adj_fixed(apod_w(q, im, x.hi, z.hi, e) * gv, wh, wl);
        const long long W = das_adj_join(wh, wl);
        for (int t = 0; t < q.ntx; ++t) {
          int i;
          float f;
          das_tap(utx_s[t * DAS_THREADS + threadIdx.x], ur, i, f);
          int h1, l1;
          das_adj_second(W, f, h1, l1);
          const long long s1 = das_adj_join(h1, l1);
          unsigned long long* row = acc + ((size_t)t * q.ne + e) * q.ns;
          if (i >= 0 && i < q.ns) atomicAdd(&row[i], (unsigned long long)(W - s1));
          if (i + 1 >= 0 && i + 1 < q.ns) atomicAdd(&row[i + 1], (unsigned long long)s1);
        }
      }
    }
  }
}

// Tiled transposed DAS.  A CTA owns a 16-line x 32-depth pixel tile (one pixel per thread; a
// warp holds 32 consecutive depths of one line, whose taps fall on different samples).  The
// elements go in batches of up to DJ_COLS (element, transmit) columns: the taps of a batch go
// into a sample window per column in shared memory, the samples the tile's delays can reach
// (FP32 delays at the tile's corners, padded); then every nonzero window entry goes to its row
// with one global atomic.  A window spans ~100-200 samples against the tile's 512 taps per
// column, so the global atomics drop several-fold.  A tap outside its window (an
// underestimated window, or one longer than `win`) goes to the row directly.
// A window entry is two 32-bit words with native shared atomics, hi 2^22 + lo: a share's high word
// is at most 2^18 in size, its low word below 2^22, and at most 512 pixels add to one entry, so
// neither sum can overflow (2^27 and 2^31) and the flush rebuilds the exact total.  The shares
// and their sums are those of k_das_adj, so the two kernels give the same bits.
// Bound by instruction issue (75 %) and shared memory (four atomics per tap, two wavefronts each).
// 128 elements, 256 x 1024 pixels: 16 transmits 1550 -> 1175 us, one transmit 410 -> 213 us (both
// shares used to be split from 64-bit values and every weight rescaled, 78 instructions per tap;
// every element had two barriers of its own; a tile was one block, 112 of them for 97 x 512 pixels).
constexpr int DJ_THREADS = 512, DJ_LINES = 16, DJ_DEPTHS = 32;
constexpr int DJ_COLS = 16;  // columns per batch (one element's transmits when those are more)
constexpr int DJ_BLOCKS = 2432;  // 1216: 16 transmits +6 %, 11 on 97 x 512 pixels -5 %
constexpr int DJ_SMEM_MAX = 226 * 1024;
constexpr int DJ_MAX_TX = 36;                    // beyond, the untiled kernel
constexpr int DJ_WIN_MIN = 128, DJ_WIN_MAX = 640;
static_assert(DJ_DEPTHS == 32 && DJ_LINES == 16 && DJ_THREADS / 32 == DJ_LINES, "a warp is one line's 32 depths");
static_assert(DAS_ADJ_V_BITS - DAS_ADJ_LO_BITS + 9 < 31 && DAS_ADJ_LO_BITS + 9 <= 31,
              "the tile's 512 contributions per entry fit both words");
__host__ __device__ constexpr int das_adj_batch(int ntx) { return ntx >= DJ_COLS ? 1 : DJ_COLS / ntx; }
__host__ __device__ constexpr size_t das_adj_tile_smem(int ne, int ntx, int win) {
  return (2 * sizeof(int) * win + 2 * sizeof(int2)) * (size_t)(das_adj_batch(ntx) * ntx) +
         sizeof(float2) * ((size_t)DJ_THREADS * ntx + ne) + sizeof(float) * ne;
}
static_assert(das_adj_tile_smem(MAX_ELEM, DJ_MAX_TX, 256) <= (size_t)DJ_SMEM_MAX, "the most transmits fit");
// window length for an image: the samples a tile's delays can span (a depth step moves a delay by
// at most its two-way time, a line step by 1 + |sin th| times its one-way time), as far as shared
// memory allows.  A fixed 192 sent every tap of a coarse depth grid (97 x 512 pixels over 58 mm)
// to the rows: 566 us against 224.
static int das_adj_win(const Acq& q, const Img& im) {
  double smax = 0.0;
  for (int t = 0; t < q.ntx; ++t) smax = std::max(smax, (double)std::fabs(q.sin_tx[t]));
  const double k = (double)q.fs / q.cbf;
  const double dz = im.nd > 1 ? std::fabs((double)im.z1 - im.z0) / (im.nd - 1) : 0.0;
  const double dx = im.nl > 1 ? std::fabs((double)im.x1 - im.x0) / (im.nl - 1) : 0.0;
  const double span = k * (2.0 * (DJ_DEPTHS - 1) * dz + (1.0 + smax) * (DJ_LINES - 1) * dx) + 12.0;
  int win = span < DJ_WIN_MAX ? std::max(DJ_WIN_MIN, ((int)span + 31) / 32 * 32) : DJ_WIN_MAX;
  while (win > DJ_WIN_MIN && das_adj_tile_smem(q.ne, q.ntx, win) > (size_t)DJ_SMEM_MAX) win -= 32;
  return win;
}
__global__ void __launch_bounds__(DJ_THREADS) k_das_adj_tile(Acq q, Img im, int win, const float* __restrict__ gi,
                                                             unsigned long long* acc, const unsigned int* maxbits) {
  extern __shared__ __align__(16) unsigned char dj_sm[];
  const int ntx = q.ntx, batch = das_adj_batch(ntx), ncol = batch * ntx;
  int* hi_s = reinterpret_cast<int*>(dj_sm);                                // [ncol][win]
  int* lo_s = hi_s + ncol * win;                                         // [ncol][win]
  float2* utx_s = reinterpret_cast<float2*>(lo_s + ncol * win);          // [ntx][DJ_THREADS]
  int2* win_s = reinterpret_cast<int2*>(utx_s + (size_t)ntx * DJ_THREADS);  // [2][ncol]
  float2* xe_s = reinterpret_cast<float2*>(win_s + 2 * ncol);               // [ne] element positions (float-float)
  float* w_s = reinterpret_cast<float*>(xe_s + q.ne);                       // [ne] Hann weights
  const unsigned int mb = *maxbits;
  if (mb >= F32_INF_BITS) return;  // k_das_adj_finish writes NaN
  // the tile's share of the elements: whole batches, split over gridDim.y blocks
  const int per = ((q.ne + batch - 1) / batch + gridDim.y - 1) / gridDim.y * batch;
  const int e_lo = blockIdx.y * per, e_hi = min(q.ne, e_lo + per);
  if (e_lo >= e_hi) return;
  const int tiles_d = (im.nd + DJ_DEPTHS - 1) / DJ_DEPTHS;
  const int l0 = (blockIdx.x / tiles_d) * DJ_LINES, d0 = (blockIdx.x % tiles_d) * DJ_DEPTHS;
  const int l1 = min(l0 + DJ_LINES - 1, im.nl - 1), d1 = min(d0 + DJ_DEPTHS - 1, im.nd - 1);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int l = l0 + warp, d = d0 + lane;
  const bool valid = l < im.nl && d < im.nd;
  const DasGeo g = das_geo(q);
  const ff x = grid_coord(im.x0, im.x1, valid ? l : l0, im.nl);
  const ff z = grid_coord(im.z0, im.z1, valid ? d : d0, im.nd);
  const float gv = valid ? das_adj_scaled(gi[(size_t)l * im.nd + d], das_adj_kexp(im.nl * im.nd, mb)) : 0.0f;
  for (int t = 0; t < ntx; ++t) utx_s[t * DJ_THREADS + threadIdx.x] = das_split(das_utx(q, g, x, z, t));
  for (int j = threadIdx.x; j < 2 * ncol * win; j += DJ_THREADS) hi_s[j] = 0;  // both words
  for (int e = e_lo + threadIdx.x; e < e_hi; e += DJ_THREADS) {
    const ff xe = das_elem(q, g, e);
    xe_s[e] = make_float2(xe.hi, xe.lo);
    w_s[e] = hann_w(e, q.ne);
  }
  const DasRx p = das_rx(g, x, z);
  const bool dynamic = im.fnum > 0.0f;
  // windows of a batch's columns: warp w takes columns w, w + 16, ...; its lanes hold the tile's 32
  // corner positions (16 lines x the two depth ends).  A window is (first sample, entries the
  // first share may go to): a tap is inside when its sample is less than that many past the
  // first; nothing is inside an empty or overlong one.
  const float cx = grid_coord(im.x0, im.x1, min(l0 + (lane & 15), l1), im.nl).hi;
  const float cz = grid_coord(im.z0, im.z1, (lane & 16) ? d1 : d0, im.nd).hi;
  const float kf = g.k.hi, hwf = g.half_w.hi;
  auto windows = [&](int e0, int2* out) {
    for (int c = warp; c < min(batch, e_hi - e0) * ntx; c += DJ_THREADS / 32) {  // warp-uniform
      const int eb = c / ntx, t = c - eb * ntx;
      const float dx = cx - (e0 + eb - 0.5f * (q.ne - 1)) * q.pitch;
      const float u = (fmaf(cx, q.sin_tx[t], fmaf(cz, q.cos_tx[t], hwf * fabsf(q.sin_tx[t]))) + sqrtf(fmaf(dx, dx, cz * cz))) * kf;
      const int lo = __reduce_min_sync(0xFFFFFFFFu, (int)floorf(u)), hi = __reduce_max_sync(0xFFFFFFFFu, (int)ceilf(u));
      if (lane == 0) {
        const int2 w = das_window_of(q.ns, lo, hi, win);
        out[c] = make_int2(w.x, max(0, w.y - 1));
      }
    }
  };
  windows(e_lo, win_s);
  __syncthreads();
  for (int e0 = e_lo, buf = 0; e0 < e_hi; e0 += batch, buf ^= 1) {
    const int nb = min(batch, e_hi - e0);
    const int2* wcur = win_s + buf * ncol;
    // the other buffer was last read by the previous batch's flush, before its barrier
    if (e0 + batch < e_hi) windows(e0 + batch, win_s + (buf ^ 1) * ncol);
    for (int eb = 0; eb < nb; ++eb) {
      const int e = e0 + eb;
      int wh, wl;
      das_adj_fixed((dynamic ? apod_w(q, im, x.hi, z.hi, e) : w_s[e]) * gv, wh, wl);
      if ((wh | wl) == 0) continue;
      const long long W = das_adj_join(wh, wl);
      const float2 xe = xe_s[e];
      const float2 ur = das_split(das_urx(p, ff{xe.x, xe.y}));
      int* hc = hi_s + eb * ntx * win;
      int* lc = lo_s + eb * ntx * win;
      const int2* wc = wcur + eb * ntx;
#pragma unroll 8
      for (int t = 0; t < ntx; ++t, hc += win, lc += win) {
        int i, h1, l1w;
        float f;
        das_tap(utx_s[t * DJ_THREADS + threadIdx.x], ur, i, f);
        das_adj_second(W, f, h1, l1w);
        const int2 w = wc[t];
        const unsigned rel = (unsigned)i - (unsigned)w.x;
        if (rel < (unsigned)w.y) {
          atomicAdd(&hc[rel], wh - h1);
          atomicAdd(&lc[rel], wl - l1w);
          atomicAdd(&hc[rel + 1], h1);
          atomicAdd(&lc[rel + 1], l1w);
        } else {
          const long long s1 = das_adj_join(h1, l1w);
          unsigned long long* row = acc + ((size_t)t * q.ne + e) * q.ns;
          if (i >= 0 && i < q.ns) atomicAdd(&row[i], (unsigned long long)(W - s1));
          if (i + 1 >= 0 && i + 1 < q.ns) atomicAdd(&row[i + 1], (unsigned long long)s1);
        }
      }
    }
    __syncthreads();
    for (int c = warp; c < nb * ntx; c += DJ_THREADS / 32) {  // a warp flushes a column
      const int eb = c / ntx, t = c - eb * ntx;
      const int2 w = wcur[c];
      unsigned long long* row = acc + ((size_t)t * q.ne + e0 + eb) * q.ns + w.x;
      for (int r = lane; r <= w.y; r += 32) {  // w.y + 1 entries; an empty window holds a zero
        const int j = c * win + r;
        const int h = hi_s[j], lo = lo_s[j];
        if (h | lo) {
          const long long v = das_adj_join(h, lo);
          if (v) atomicAdd(&row[r], (unsigned long long)v);
          hi_s[j] = 0;  // both words, also when they cancel (v = 0 with hi = -lo / 2^22)
          lo_s[j] = 0;
        }
      }
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------------
// shared-memory FFT of one line (N = n_depth, power of two): radix-2 butterflies, R consecutive
// stages at a time in the registers of one thread (the same butterflies with the same roundings
// as one stage at a time), so that a line of 1024 has 5 barriers per transform instead of 10.
// A line's transforms are bound by those barriers' latencies.
// ------------------------------------------------------------------------------------------
// slot of z[i]: one spare after every 16, so that strided groups spread over the banks
__host__ __device__ constexpr int fft_slot(int i) { return i + (i >> 4); }
__host__ __device__ constexpr size_t fft_line_bytes(int N) { return sizeof(float2) * (size_t)(fft_slot(N) + 1); }

template <int R, bool INVERSE>
__device__ __forceinline__ void fft_pass(float2* z, const float2* tw, int N, int s) {  // stages s .. s + R - 1 (from 1)
  constexpr int E = 1 << R;
  const int half = 1 << (s - 1);
  for (int g = threadIdx.x; g < (N >> R); g += blockDim.x) {
    const int kk = g & (half - 1), base = ((g >> (s - 1)) << (s - 1 + R)) + kk;
    float2 v[E];
#pragma unroll
    for (int j = 0; j < E; ++j) v[j] = z[fft_slot(base + j * half)];
#pragma unroll
    for (int r = 0; r < R; ++r) {
#pragma unroll
      for (int j = 0; j < E; ++j) {
        if (j & (1 << r)) continue;
        float2 w = tw[(kk + (j & ((1 << r) - 1)) * half) * (N >> (s + r))];
        if (INVERSE) w.y = -w.y;
        const float2 xi = v[j], xj = v[j + (1 << r)];
        const float2 t = make_float2(w.x * xj.x - w.y * xj.y, w.x * xj.y + w.y * xj.x);
        v[j + (1 << r)] = make_float2(xi.x - t.x, xi.y - t.y);
        v[j] = make_float2(xi.x + t.x, xi.y + t.y);
      }
    }
#pragma unroll
    for (int j = 0; j < E; ++j) z[fft_slot(base + j * half)] = v[j];
  }
  __syncthreads();
}
template <bool INVERSE>
__device__ void fft_smem(float2* z, const float2* tw, int N, int logN) {
  int s = 1;
  if (N >= 2048)  // as many groups of 8 as threads
    for (; s + 2 <= logN; s += 3) fft_pass<3, INVERSE>(z, tw, N, s);
  for (; s + 1 <= logN; s += 2) fft_pass<2, INVERSE>(z, tw, N, s);
  if (s <= logN) fft_pass<1, INVERSE>(z, tw, N, s);
}

__device__ void twiddles(float2* tw, int N) {
  for (int kk = threadIdx.x; kk < N / 2; kk += blockDim.x) {
    float s, c;
    sincospif(-2.0f * (float)kk / (float)N, &s, &c);
    tw[kk] = make_float2(c, s);
  }
}
__device__ __forceinline__ int bit_rev(int i, int logN) { return (int)(__brev((unsigned)i) >> (32 - logN)); }

// analytic signal of a real line (already bit-reversed into z): X = FFT(x); X *= h; IFFT / N
__device__ void analytic_smem(float2* z, const float2* tw, int N, int logN) {
  fft_smem<false>(z, tw, N, logN);
  // scale and bit-reverse in place for the inverse transform, a pair of slots per thread
  auto scale = [&](int kk) { return ((kk == 0 || 2 * kk == N) ? 1.0f : (2 * kk < N ? 2.0f : 0.0f)) / (float)N; };
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const int j = bit_rev(i, logN);
    if (i > j) continue;
    const float si = scale(i), sj = scale(j);
    const float2 a = z[fft_slot(i)], b = z[fft_slot(j)];
    z[fft_slot(i)] = make_float2(b.x * sj, b.y * sj);
    z[fft_slot(j)] = make_float2(a.x * si, a.y * si);
  }
  __syncthreads();
  fft_smem<true>(z, tw, N, logN);
}
// largest key of the block into *best (every thread calls; one shared atomic per warp)
__device__ __forceinline__ void block_max_key(unsigned long long key, unsigned long long* best) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long k = __shfl_xor_sync(0xFFFFFFFFu, key, o);
    key = k > key ? k : key;
  }
  if ((threadIdx.x & 31) == 0 && key) atomicMax(best, key);
}

// envelope of each line: E = |x + i H x|; per-image maximum (value, first index) into a
// packed 64-bit key (float bits << 32 | ~index) with atomicMax
__global__ void k_envelope(Img im, const float* __restrict__ irf, float* env, unsigned long long* emax_key) {
  extern __shared__ float2 sz[];
  const int N = im.nd;
  const int logN = 31 - __clz(N);
  float2* z = sz;
  float2* tw = sz + fft_slot(N) + 1;
  twiddles(tw, N);
  __shared__ unsigned long long best;
  if (threadIdx.x == 0) best = 0ull;
  unsigned long long own = 0ull;
  for (int l = blockIdx.x; l < im.nl; l += gridDim.x) {
    const float* x = irf + (size_t)l * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x) z[fft_slot(bit_rev(i, logN))] = make_float2(__ldg(&x[i]), 0.0f);
    __syncthreads();
    analytic_smem(z, tw, N, logN);
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      const float2 v = z[fft_slot(i)];
      const float e = sqrtf(v.x * v.x + v.y * v.y);
      env[(size_t)l * N + i] = e;
      const unsigned long long key =
          ((unsigned long long)__float_as_uint(e) << 32) | (0xFFFFFFFFu - (uint32_t)(l * N + i));
      own = key > own ? key : own;
    }
    __syncthreads();
  }
  block_max_key(own, &best);
  __syncthreads();
  if (threadIdx.x == 0) atomicMax(emax_key, best);
}

__device__ __forceinline__ float key_emax(unsigned long long k) { return __uint_as_float((uint32_t)(k >> 32)); }
__device__ __forceinline__ int key_argmax(unsigned long long k) { return (int)(0xFFFFFFFFu - (uint32_t)k); }

// ------------------------------------------------------------------------------------------
// Fused envelope + log compression: one cooperative launch whose blocks keep the envelope of
// their lines in shared memory, meet at one grid-wide barrier once every block has folded its
// maximum into the packed key, then write B = max(20 log10(E / E_max), -DR).  The barrier's
// wait is bounded in time (cooperative launches are co-resident, so it never expires in
// practice); should it expire, the block writes NaN instead of a wrong image and raises
// ST_TIMEOUT in the status word (when one is given).  `extra` arrivals beyond the grid are
// awaited as well: 0 in normal use; 1 injects the fault (an arrival no block makes) so that
// the timeout report can be tested, with the short limit `limit` (clock cycles).
// keyw[0] = packed maximum, keyw[1] = arrival counter (both zeroed before the launch).
// ------------------------------------------------------------------------------------------
constexpr long long BARRIER_CYCLES = 4000000000ll;     // ~2 s at the maximum SM clock
constexpr long long FAULT_BARRIER_CYCLES = 2000000ll;  // ~1 ms: the injected fault's wait

__global__ void k_envlog_fused(Img im, const float* __restrict__ irf, unsigned long long* keyw, float* b, int* status,
                               int extra, long long limit) {
  extern __shared__ float2 sz[];
  const int N = im.nd;
  const int logN = 31 - __clz(N);
  float2* z = sz;
  float2* tw = sz + fft_slot(N) + 1;
  float* ev = reinterpret_cast<float*>(tw + N / 2);  // envelopes of this block's lines
  twiddles(tw, N);
  __shared__ unsigned long long best;
  if (threadIdx.x == 0) best = 0ull;
  unsigned long long own = 0ull;
  int j = 0;
  for (int l = blockIdx.x; l < im.nl; l += gridDim.x, ++j) {
    const float* x = irf + (size_t)l * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x) z[fft_slot(bit_rev(i, logN))] = make_float2(__ldg(&x[i]), 0.0f);
    __syncthreads();
    analytic_smem(z, tw, N, logN);
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      const float2 v = z[fft_slot(i)];
      const float e = sqrtf(v.x * v.x + v.y * v.y);
      ev[j * N + i] = e;
      const unsigned long long key =
          ((unsigned long long)__float_as_uint(e) << 32) | (0xFFFFFFFFu - (uint32_t)(l * N + i));
      own = key > own ? key : own;
    }
    __syncthreads();
  }
  block_max_key(own, &best);
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) {
    atomicMax(&keyw[0], best);
    __threadfence();
    atomicAdd(&keyw[1], 1ull);
    const long long t0 = clock64();
    while (atomicAdd(&keyw[1], 0ull) < (unsigned long long)gridDim.x + (unsigned long long)extra) {
      if (clock64() - t0 > limit) {
        ok = false;
        break;
      }
      __nanosleep(64);
    }
    __threadfence();
    best = ok ? atomicAdd(&keyw[0], 0ull) : 0xFFFFFFFFFFFFFFFFull;
    if (!ok && status) atomicOr(status, ST_TIMEOUT);
  }
  __syncthreads();
  const unsigned long long kk = best;
  const float emax = __uint_as_float((uint32_t)(kk >> 32));
  const bool valid = kk != 0xFFFFFFFFFFFFFFFFull;
  j = 0;
  for (int l = blockIdx.x; l < im.nl; l += gridDim.x, ++j) {
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      const float e = ev[j * N + i];
      float v = -im.dr;
      if (!valid) v = __int_as_float(0x7FC00000);
      else if (emax > 0.0f && e > 0.0f) v = fmaxf(20.0f * log10f(e / emax), -im.dr);
      b[(size_t)l * N + i] = v;
    }
  }
}

// B = max(20 log10(E / E_max), -DR); E = 0 or E_max = 0 -> -DR
__global__ void k_logc(Img im, const float* __restrict__ env, const unsigned long long* emax_key, float* b) {
  const int n = im.nl * im.nd;
  const float emax = key_emax(*emax_key);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float e = env[i];
    float v = -im.dr;
    if (emax > 0.0f && e > 0.0f) v = fmaxf(20.0f * log10f(e / emax), -im.dr);
    b[i] = v;
  }
}

// ------------------------------------------------------------------------------------------
// loss: L = (l1 sum |r| + l2 sum r^2) / N, dL/dB = (l1 sign(r) + 2 l2 r) / N
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ float block_sum(float v) {
  __shared__ float ws[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  float s = 0.0f;
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? ws[threadIdx.x] : 0.0f;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  }
  __syncthreads();
  return s;  // valid in thread 0
}

__global__ void k_loss_partial(Img im, const float* __restrict__ b, const float* __restrict__ bref, float* gb,
                               float* part) {
  const int n = im.nl * im.nd;
  const float inv = 1.0f / (float)n;
  float s = 0.0f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float r = b[i] - bref[i];
    s += im.l1 * fabsf(r) + im.l2 * r * r;
    if (gb) gb[i] = (im.l1 * (r > 0.0f ? 1.0f : (r < 0.0f ? -1.0f : 0.0f)) + 2.0f * im.l2 * r) * inv;
  }
  s = block_sum(s);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// The loss in one launch for images of at most LOSS_ONE pixels: one cluster of LOSS_CTAS blocks,
// whose sums meet in the first one's shared memory.  A block's shared memory may be written from
// outside only once the block has started: every block arrives at a cluster barrier as it begins and
// waits for the others before its store, the pixels lying between the two.
// Bound by the reads of eight SMs.  In a graph, two kernels and one, in us: 128 x 512 pixels 3.3 and
// 3.2, 256 x 1024 3.9 and 5.4, 512 x 1024 4.5 and 8.7; but each launch costs the host 3 us as well, and
// envelope, loss and VJP called after one another take 37.2 and 32.3 us, 53.2 and 52.4, at 256 x 2048
// 70.9 and 72.8: one launch up to 2^18 pixels.
constexpr int LOSS_CTAS = 8, LOSS_THREADS = 1024, LOSS_ONE = 1 << 18;
__global__ void __cluster_dims__(LOSS_CTAS, 1, 1) __launch_bounds__(LOSS_THREADS)
    k_loss_cluster(Img im, const float* __restrict__ b, const float* __restrict__ bref, float* gb, float* loss) {
  __shared__ float sums[LOSS_CTAS];
  cg::cluster_group cl = cg::this_cluster();
  auto started = cl.barrier_arrive();
  const int n = im.nl * im.nd;
  const float inv = 1.0f / (float)n;
  float s = 0.0f;
#pragma unroll 8
  for (int i = blockIdx.x * LOSS_THREADS + threadIdx.x; i < n; i += LOSS_CTAS * LOSS_THREADS) {
    const float r = __ldg(&b[i]) - __ldg(&bref[i]);
    s += im.l1 * fabsf(r) + im.l2 * r * r;
    if (gb) gb[i] = (im.l1 * (r > 0.0f ? 1.0f : (r < 0.0f ? -1.0f : 0.0f)) + 2.0f * im.l2 * r) * inv;
  }
  s = block_sum(s);
  cl.barrier_wait(std::move(started));
  if (threadIdx.x == 0) cl.map_shared_rank(sums, 0)[cl.block_rank()] = s;
  cl.sync();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    float t = 0.0f;
    for (int k = 0; k < LOSS_CTAS; ++k) t += sums[k];
    loss[0] = t * inv;
  }
}

__global__ void k_sum_final(const float* part, int n, float scale, float* out) {
  float s = 0.0f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += part[i];
  s = block_sum(s);
  if (threadIdx.x == 0) out[0] = s * scale;
}

// sum over unclipped pixels of dL/dB (the E_max share of the log-compression derivative)
__global__ void k_live_sum(Img im, const float* __restrict__ env, const unsigned long long* emax_key,
                           const float* __restrict__ gb, float* part) {
  const int n = im.nl * im.nd;
  const float emax = key_emax(*emax_key);
  float s = 0.0f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float e = env[i];
    if (emax > 0.0f && e > 0.0f && 20.0f * log10f(e / emax) > -im.dr) s += gb[i];
  }
  s = block_sum(s);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// per line: g_E = dL/dB * (20/ln10) / E on unclipped pixels, minus (20/ln10) S / E_max at the
// argmax; then g_x = (x/E) g_E - H((y/E) g_E) (the Hilbert matrix is skew-symmetric)
__global__ void k_envlog_vjp(Img im, const float* __restrict__ irf, const float* __restrict__ gb,
                             const unsigned long long* emax_key, const float* live_sum, float* gi) {
  extern __shared__ float2 sz[];
  const int N = im.nd;
  const int logN = 31 - __clz(N);
  float2* z = sz;
  float2* v = sz + fft_slot(N) + 1;
  float2* tw = v + fft_slot(N) + 1;
  twiddles(tw, N);
  const float emax = key_emax(*emax_key);
  const int am = key_argmax(*emax_key);
  const float c = 8.685889638065036f;  // 20 / ln(10)
  const float S = *live_sum;
  for (int l = blockIdx.x; l < im.nl; l += gridDim.x) {
    const float* x = irf + (size_t)l * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x) z[fft_slot(bit_rev(i, logN))] = make_float2(__ldg(&x[i]), 0.0f);
    __syncthreads();
    analytic_smem(z, tw, N, logN);
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      const float xi = __ldg(&x[i]), yi = z[fft_slot(i)].y;
      const float e = sqrtf(xi * xi + yi * yi);
      const int p = l * N + i;
      float ge = 0.0f;
      if (emax > 0.0f && e > 0.0f && 20.0f * log10f(e / emax) > -im.dr) ge = gb[p] * c / e;
      if (p == am && emax > 0.0f) ge -= c * S / emax;
      const float vv = e > 0.0f ? yi / e * ge : 0.0f;
      z[fft_slot(i)] = make_float2(e > 0.0f ? xi / e * ge : 0.0f, 0.0f);  // keep (x/E) g_E in z.x
      v[fft_slot(bit_rev(i, logN))] = make_float2(vv, 0.0f);
    }
    __syncthreads();
    analytic_smem(v, tw, N, logN);
    for (int i = threadIdx.x; i < N; i += blockDim.x) gi[(size_t)l * N + i] = z[fft_slot(i)].x - v[fft_slot(i)].y;
    __syncthreads();
  }
}

// The same VJP in one cooperative launch: a block keeps its lines' analytic signals in shared
// memory, meets the others once for the maximum, and transforms back.  Only the line that holds
// the maximum needs the sum S over all unclipped pixels: its block alone waits for the others'
// partial sums (added in block order).  Both waits are bounded, as in k_envlog_fused; one that
// expires makes the block's lines NaN and raises ST_TIMEOUT, and a block that went on without the
// others' maximum gives NaN as its partial sum, so that the line with the maximum comes out NaN
// too.  `extra` arrivals more than there are blocks (a test's injected fault, else 0) are awaited by
// every block but block 0 in the first wait.  keyw: packed maximum, two arrival counters (zeroed
// before the launch).  256 lines of 1024: 47 us as four kernels, which computed the envelope's
// transform twice; 128 lines of 512: 30 us against 20.
__global__ void __launch_bounds__(256) k_envlog_vjp_fused(Img im, const float* __restrict__ irf,
                                                          const float* __restrict__ gb, unsigned long long* keyw,
                                                          float* part, float* gi, int* status, int extra,
                                                          long long limit) {
  extern __shared__ float2 sz[];
  const int N = im.nd, L = fft_slot(N) + 1;
  const int logN = 31 - __clz(N);
  float2* tw = sz;
  float2* v = tw + N / 2;
  float2* zl = v + L;  // the block's lines, L slots each
  __shared__ unsigned long long best;
  __shared__ float s_sum;
  __shared__ int s_ok;
  twiddles(tw, N);
  if (threadIdx.x == 0) {
    best = 0ull;
    s_ok = 1;
  }
  unsigned long long own = 0ull;
  int j = 0;
  for (int l = blockIdx.x; l < im.nl; l += gridDim.x, ++j) {
    const float* x = irf + (size_t)l * N;
    float2* z = zl + j * L;
    for (int i = threadIdx.x; i < N; i += blockDim.x) z[fft_slot(bit_rev(i, logN))] = make_float2(__ldg(&x[i]), 0.0f);
    __syncthreads();
    analytic_smem(z, tw, N, logN);
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      const float2 a = z[fft_slot(i)];
      const float e = sqrtf(a.x * a.x + a.y * a.y);
      const unsigned long long key =
          ((unsigned long long)__float_as_uint(e) << 32) | (0xFFFFFFFFu - (uint32_t)(l * N + i));
      own = key > own ? key : own;
    }
  }
  block_max_key(own, &best);
  __syncthreads();
  // thread 0: until so many blocks have arrived
  auto wait = [&](unsigned long long* counter, unsigned arrivals, long long cycles) {
    const long long t0 = clock64();
    while (atomicAdd(counter, 0ull) < (unsigned long long)arrivals) {
      if (clock64() - t0 > cycles) {
        if (status) atomicOr(status, ST_TIMEOUT);
        s_ok = 0;
        break;
      }
      __nanosleep(64);
    }
    __threadfence();
  };
  if (threadIdx.x == 0) {
    atomicMax(&keyw[0], best);
    __threadfence();
    atomicAdd(&keyw[1], 1ull);
    wait(&keyw[1], gridDim.x + (blockIdx.x ? (unsigned)extra : 0u), limit);
    best = atomicAdd(&keyw[0], 0ull);
  }
  __syncthreads();
  const float emax = key_emax(best);
  const int am = key_argmax(best);
  const float c = 8.685889638065036f;  // 20 / ln(10)
  float sum = 0.0f;
  j = 0;
  for (int l = blockIdx.x; l < im.nl; l += gridDim.x, ++j)
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      const float2 a = zl[j * L + fft_slot(i)];
      const float e = sqrtf(a.x * a.x + a.y * a.y);
      if (emax > 0.0f && e > 0.0f && 20.0f * log10f(e / emax) > -im.dr) sum += __ldg(&gb[(size_t)l * N + i]);
    }
  sum = block_sum(sum);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = s_ok ? sum : __int_as_float(0x7FC00000);
    __threadfence();
    atomicAdd(&keyw[2], 1ull);
  }
  const bool owner = emax > 0.0f && (am / N) % (int)gridDim.x == (int)blockIdx.x;
  float S = 0.0f;
  if (owner) {  // block-uniform
    if (threadIdx.x == 0) wait(&keyw[2], gridDim.x, 4 * limit);  // others may wait out the first before they arrive
    __syncthreads();
    float s = 0.0f;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) s += __ldcg(&part[b]);
    s = block_sum(s);
    if (threadIdx.x == 0) s_sum = s;
    __syncthreads();
    S = s_sum;
  }
  j = 0;
  for (int l = blockIdx.x; l < im.nl; l += gridDim.x, ++j) {
    const float* x = irf + (size_t)l * N;
    float2* z = zl + j * L;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      const float xi = __ldg(&x[i]), yi = z[fft_slot(i)].y;
      const float e = sqrtf(xi * xi + yi * yi);
      const int p = l * N + i;
      float ge = 0.0f;
      if (emax > 0.0f && e > 0.0f && 20.0f * log10f(e / emax) > -im.dr) ge = __ldg(&gb[p]) * c / e;
      if (p == am && emax > 0.0f) ge -= c * S / emax;
      const float vv = e > 0.0f ? yi / e * ge : 0.0f;
      z[fft_slot(i)].x = e > 0.0f ? xi / e * ge : 0.0f;  // keep (x/E) g_E in z.x
      v[fft_slot(bit_rev(i, logN))] = make_float2(vv, 0.0f);
    }
    __syncthreads();
    analytic_smem(v, tw, N, logN);
    for (int i = threadIdx.x; i < N; i += blockDim.x)
      gi[(size_t)l * N + i] = s_ok ? z[fft_slot(i)].x - v[fft_slot(i)].y : __int_as_float(0x7FC00000);
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------------
// DAS derivative in the acquisition parameters (Eq. das with the delays of Sec. 2.3.1),
// contracted with an image gradient gi, the RF held fixed:
//   out[0] = sum_p gi(p) dI(p)/dc_bf,  out[1] = .../dpitch,  out[2 + t] = .../dth_t.
// A tap at u = i + f has dI/du = w_e (rf[i + 1] - rf[i]) (the slope of its interpolation
// interval); du/dc_bf = -u / c_bf; du/dpitch = (W/2 |sin th| / p - (x - x_e) / r (e - (N_e -
// 1)/2)) fs / c_bf (transmit aperture and receive distance r); only the transmit delay holds
// th_t: du/dth = (x cos th - z sin th + W/2 sgn(sin th) cos th) fs / c_bf, sgn(0) = 0.  So a
// pixel needs, per transmit, S1 = sum_e w_e slope, and over all its taps sum w_e slope u and
// sum w_e slope du/dp.  One pixel per thread, a warp 8 lines x 4 depths as in k_das, elements outer
// (in pairs, their delays in packed FP32) and transmits inner, so the receive delay, its pitch
// derivative and the element weight are evaluated once per (pixel, element); the transmit delays
// and the per-transmit sums S1 sit in shared memory in thread-major rows; the other two sums are
// per-pixel scalars (their transmit weights are known before the sum).  Taps are checked against the
// record once per pair of elements and for the whole warp: a branch per pixel was slower even where
// every tap lies inside (253 us against 200 in the first size below).  Each block writes one row of
// 2 + ntx sums, reduced in a fixed order (deterministic).  Bound by issue and by the gathers'
// latency.  128 elements, 11 transmits, 96 x 512 pixels 377 -> 200 us; 95 elements, 5 transmits,
// F-number 1.5, 101 x 1024 pixels, 4 % of the taps past the record 188 -> 157 us (170 with a branch
// per pixel, 164 with a check per tap).
// ------------------------------------------------------------------------------------------
constexpr int DA_THREADS = 256;
constexpr int DA_TL = 8, DA_TD = 32;  // a block's lines x depths; a warp has 8 lines x 4 depths
static_assert(DA_TL * DA_TD == DA_THREADS, "a pixel per thread");
__host__ __device__ constexpr size_t das_acq_smem(int ne, int ntx) {
  return sizeof(ulonglong2) * ((ne + 1) / 2) + (sizeof(float2) + sizeof(float)) * DA_THREADS * ntx + sizeof(float) * ne;
}
__global__ void __launch_bounds__(DA_THREADS) k_das_acq(Acq q, Img im, const float* __restrict__ rf,
                                                        const float* __restrict__ gi, float* part) {
  extern __shared__ __align__(16) ulonglong2 da_sm[];
  ulonglong2* xe_s = da_sm;                                            // [(ne + 1) / 2] as in k_das
  float2* ut_s = reinterpret_cast<float2*>(xe_s + (q.ne + 1) / 2);     // [ntx][DA_THREADS]
  float* s1_s = reinterpret_cast<float*>(ut_s + q.ntx * DA_THREADS);   // [ntx][DA_THREADS]
  float* w_s = s1_s + q.ntx * DA_THREADS;                              // [ne] Hann weights
  const DasGeo g = das_geo(q);
  const int tiles_d = (im.nd + DA_TD - 1) / DA_TD;
  const int tl = blockIdx.x / tiles_d, td = blockIdx.x - tl * tiles_d;
  const int l = tl * DA_TL + (threadIdx.x & 7), d = td * DA_TD + (threadIdx.x >> 3);
  const bool valid = l < im.nl && d < im.nd;
  const ff x = grid_coord(im.x0, im.x1, valid ? l : 0, im.nl), z = grid_coord(im.z0, im.z1, valid ? d : 0, im.nd);
  const float gp = valid ? __ldg(&gi[(size_t)l * im.nd + d]) : 0.0f;
  const float kfs = q.fs / q.cbf, hn = 0.5f * (float)(q.ne - 1), hw = hn * q.pitch;
  for (int e = threadIdx.x; e < q.ne; e += DA_THREADS) w_s[e] = hann_w(e, q.ne);
  for (int k = threadIdx.x; k < (q.ne + 1) / 2; k += DA_THREADS) {
    const ff a = das_elem(q, g, 2 * k), b = das_elem(q, g, min(2 * k + 1, q.ne - 1));
    xe_s[k] = make_ulonglong2(pack2(-a.hi, -b.hi), pack2(-a.lo, -b.lo));
  }
  int imin = 0x7FFFFFFF, imax = -0x7FFFFFFF;
  for (int t = 0; t < q.ntx; ++t) {
    const float2 us = das_split(das_utx(q, g, x, z, t));
    const int ui = __float_as_int(us.x);
    imin = min(imin, ui);
    imax = max(imax, ui);
    ut_s[t * DA_THREADS + threadIdx.x] = us;
    s1_s[t * DA_THREADS + threadIdx.x] = 0.0f;
  }
  das_tx_range(imin, imax);
  __syncthreads();
  float c0 = 0.0f, cp = 0.0f;    // sum slope u; sum slope du/dp over the even elements
  float c0b = 0.0f, cpb = 0.0f;  // and over the odd ones
  const unsigned live = __ballot_sync(0xFFFFFFFFu, gp != 0.0f);
  if (gp != 0.0f) {
    const DasRx2 rx = das_rx2(das_rx(g, x, z));
    const bool dynamic = im.fnum > 0.0f;
    auto element = [&](int e, float& w, float& dwp, float& drp) {
      dwp = 0.0f;
      w = dynamic ? apod_w(q, im, x.hi, z.hi, e, &dwp) : w_s[e];
      const float ce = (float)e - hn;
      const float dx = x.hi - ce * q.pitch;
      drp = -dx * ce * kfs / sqrtf(fmaf(dx, dx, z.hi * z.hi));  // d(receive delay)/dp
    };
    auto tap = [&](auto inside, float2 u, float2 ur, const float* row, float w, float dwp, float drp, float dut,
                   float& c, float& cpp) {
      int i;
      float f;
      das_tap(u, ur, i, f);
      float a, b;
      if (inside) {
        a = __ldg(&row[i]);
        b = __ldg(&row[i + 1]);
      } else {
        a = (i >= 0 && i < q.ns) ? __ldg(&row[i]) : 0.0f;
        b = (i + 1 >= 0 && i + 1 < q.ns) ? __ldg(&row[i + 1]) : 0.0f;
      }
      const float sl = w * (b - a);
      c = fmaf(sl, (float)i + f, c);
      cpp = fmaf(sl, fmaf(dut, kfs, drp), cpp);
      if (dynamic) cpp = fmaf(dwp, fmaf(f, b - a, a), cpp);  // the weight's own pitch term
      return sl;
    };
    const size_t tstride = (size_t)q.ne * q.ns;
    for (int e = 0; e < q.ne; e += 2) {
      const ulonglong2 xe = xe_s[e >> 1];
      ff ua, ub;
      das_urx2(rx, xe.x, xe.y, ua, ub);
      const float2 ra = das_split(ua), rb = das_split(ub);
      float wa, wb, da, db, pa, pb;
      element(e, wa, da, pa);
      const float* row = rf + (size_t)e * q.ns;
      float2* u = ut_s + threadIdx.x;
      float* s1 = s1_s + threadIdx.x;
      auto pair = [&](auto inside) {
        element(e + 1, wb, db, pb);
#pragma unroll 2
        for (int t = 0; t < q.ntx; ++t, row += tstride, u += DA_THREADS, s1 += DA_THREADS) {
          const float2 ut = *u;
          const float dut = hn * fabsf(q.sin_tx[t]);
          const float sa = tap(inside, ut, ra, row, wa, da, pa, dut, c0, cp);
          const float sb = tap(inside, ut, rb, row + q.ns, wb, db, pb, dut, c0b, cpb);
          *s1 = (*s1 + sa) + sb;
        }
      };
      if (e + 1 < q.ne) {
        const bool in = das_inside(__float_as_int(ra.x), __float_as_int(rb.x), imin, imax, q.ns);
        if (__all_sync(live, in)) pair(std::true_type());  // warp-uniform
        else pair(std::false_type());
      } else {
        for (int t = 0; t < q.ntx; ++t, row += tstride, u += DA_THREADS, s1 += DA_THREADS)
          *s1 += tap(std::false_type(), *u, ra, row, wa, da, pa, hn * fabsf(q.sin_tx[t]), c0, cp);
      }
    }
    c0 += c0b;
    cp += cpb;
  }
  float* out = part + (size_t)blockIdx.x * (2 + q.ntx);
  for (int t = 0; t < q.ntx; ++t) {
    const float st = q.sin_tx[t], ct = q.cos_tx[t];
    const float sg = st > 0.0f ? 1.0f : (st < 0.0f ? -1.0f : 0.0f);
    const float du = (x.hi * ct - z.hi * st + hw * sg * ct) * kfs;
    const float v = block_sum(gp * du * s1_s[t * DA_THREADS + threadIdx.x]);
    if (threadIdx.x == 0) out[2 + t] = v;
  }
  const float v0 = block_sum(gp * c0);
  if (threadIdx.x == 0) out[0] = -v0 / q.cbf;
  const float v1 = block_sum(gp * cp);
  if (threadIdx.x == 0) out[1] = v1;
}

// ------------------------------------------------------------------------------------------
void launch_das(const Acq& q, const Img& im, const float* rf, float* irf, cudaStream_t st, int* status) {
  if (status && q.ne * q.ntx <= DT_MAX_WINDOWS && das_tma_smem(q) <= (size_t)DT_SMEM_MAX &&
      ((uintptr_t)rf & 15u) == 0) {
    const int tiles = ((im.nl + DT_LINES - 1) / DT_LINES) * ((im.nd + DT_DEPTHS - 1) / DT_DEPTHS);
    k_das_tma<<<tiles, DT_THREADS, das_tma_smem(q), st>>>(q, im, rf, irf, status);
    return;
  }
  const int tiles = ((im.nl + DAS_TL - 1) / DAS_TL) * ((im.nd + DAS_TD - 1) / DAS_TD);
  k_das<<<tiles, DAS_THREADS, das_smem(q.ne, q.ntx, im.fnum > 0.0f), st>>>(q, im, rf, irf);
}
int das_acq_blocks(const Img& im) {
  return ((im.nl + DA_TL - 1) / DA_TL) * ((im.nd + DA_TD - 1) / DA_TD);
}
void launch_das_acq(const Acq& q, const Img& im, const float* rf, const float* gi, float* part, cudaStream_t st) {
  k_das_acq<<<das_acq_blocks(im), DA_THREADS, das_acq_smem(q.ne, q.ntx), st>>>(q, im, rf, gi, part);
}
static std::atomic<int> g_das_adj_tiled{1};
void launch_das_adj(const Acq& q, const Img& im, const float* gi, float* grf, int grid, cudaStream_t st,
                    unsigned long long* acc, unsigned int* maxbits) {
  const long long n = (long long)q.ntx * q.ne * q.ns;
  const int npx = im.nl * im.nd;
  cudaMemsetAsync(acc, 0, sizeof(unsigned long long) * (size_t)n, st);
  cudaMemsetAsync(maxbits, 0, sizeof(unsigned int), st);
  k_das_adj_max<<<min(grid, (npx + 1023) / 1024), 256, 0, st>>>(gi, npx, maxbits);
  if (q.ntx <= DJ_MAX_TX && g_das_adj_tiled.load()) {
    const int tiles = ((im.nl + DJ_LINES - 1) / DJ_LINES) * ((im.nd + DJ_DEPTHS - 1) / DJ_DEPTHS);
    // a tile's elements over as many blocks as it takes to give the GPU DJ_BLOCKS of them
    const int batches = (q.ne + das_adj_batch(q.ntx) - 1) / das_adj_batch(q.ntx);
    const int split = max(1, min(batches, (DJ_BLOCKS + tiles - 1) / tiles));
    const int win = das_adj_win(q, im);
    k_das_adj_tile<<<dim3(tiles, split), DJ_THREADS, das_adj_tile_smem(q.ne, q.ntx, win), st>>>(q, im, win, gi, acc,
                                                                                               maxbits);
  } else {
    k_das_adj<<<grid, DAS_THREADS, sizeof(float2) * DAS_THREADS * q.ntx, st>>>(q, im, gi, acc, maxbits);
  }
  k_das_adj_finish<<<grid, 256, 0, st>>>(acc, n, npx, maxbits, grf);
}
// resident blocks on the current device (all SMs) of a kernel of 256 threads with `smem` bytes, asked
// of the runtime once per device, kernel and size: the answer never changes, and a query costs as
// much host time as a launch
static int resident_blocks(const void* kernel, size_t smem) {
  struct Entry {
    int dev;
    const void* kernel;
    size_t smem;
    int blocks;
  };
  constexpr int SLOTS = 32;
  static thread_local Entry seen[SLOTS];
  static thread_local int used = 0;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  for (int k = 0; k < std::min(used, SLOTS); ++k)
    if (seen[k].dev == dev && seen[k].kernel == kernel && seen[k].smem == smem) return seen[k].blocks;
  int per_sm = 0, sms = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, smem) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  seen[used++ % SLOTS] = Entry{dev, kernel, smem, per_sm * sms};
  return per_sm * sms;
}
constexpr int FUSED_SMEM_MAX = 202 * 1024;
// threads per line of the kernels that are not fused: a line of 64 has 16 pairs of butterflies per
// pass, and 256 threads at 48 registers leave room for five such blocks on an SM.  VJP of 4096 x 64
// pixels 61 us with 256 threads, 42 with 64; 3000 x 128 56 and 42; envelope of 8000 x 64 33 and 25
static int line_threads(int nd) { return std::min(256, std::max(64, nd)); }
static std::atomic<int> g_envlog_fused{1};

}  // namespace usrt

extern "C" void us_set_envlog_fused(int enable) { usrt::g_envlog_fused.store(enable ? 1 : 0); }
extern "C" void us_set_das_adj_tiled(int enable) { usrt::g_das_adj_tiled.store(enable ? 1 : 0); }

namespace usrt {

int launch_envlog(const Img& im, const float* irf, float* env, unsigned long long* key, float* bmode, int grid,
                  cudaStream_t st, int* status, int fault_barrier, cudaError_t* launch_err) {
  // every launch reports its own status: no cudaGetLastError, which would also take (and
  // clear) an error left by unrelated earlier work
  cudaError_t err = cudaMemsetAsync(key, 0, 2 * sizeof(unsigned long long), st);
  int launched = 0;
  if (bmode && g_envlog_fused.load() && err == cudaSuccess) {
    // fused path: every line's envelope stays in the shared memory of a co-resident block
    const size_t base = fft_line_bytes(im.nd) + sizeof(float2) * (size_t)(im.nd / 2);
    for (int lpb = 1; lpb <= 8; ++lpb) {
      const size_t smem = base + sizeof(float) * (size_t)lpb * im.nd;
      if (smem > (size_t)FUSED_SMEM_MAX) break;
      const int resident = resident_blocks((const void*)k_envlog_fused, smem);
      const int nb = (im.nl + lpb - 1) / lpb;
      if (resident > 0 && nb <= resident) {
        int extra = fault_barrier ? 1 : 0;
        long long limit = fault_barrier ? FAULT_BARRIER_CYCLES : BARRIER_CYCLES;
        void* args[] = {(void*)&im, (void*)&irf, (void*)&key, (void*)&bmode, (void*)&status, (void*)&extra,
                        (void*)&limit};
        if (cudaLaunchCooperativeKernel((const void*)k_envlog_fused, dim3(nb), dim3(256), args, smem, st) ==
            cudaSuccess) {
          if (launch_err) *launch_err = cudaSuccess;
          return 1;
        }
        cudaGetLastError();  // the refused cooperative launch: fall back to two kernels
        break;
      }
    }
  }
  const int nb = min(im.nl, grid);
  if (err == cudaSuccess) {
    void* args[] = {(void*)&im, (void*)&irf, (void*)&env, (void*)&key};
    err = cudaLaunchKernel((const void*)k_envelope, dim3(nb), dim3(line_threads(im.nd)), args,
                           fft_line_bytes(im.nd) + sizeof(float2) * (size_t)(im.nd / 2), st);
    launched += err == cudaSuccess;
  }
  if (bmode && err == cudaSuccess) {
    const unsigned long long* ckey = key;
    void* args[] = {(void*)&im, (void*)&env, (void*)&ckey, (void*)&bmode};
    err = cudaLaunchKernel((const void*)k_logc, dim3(grid), dim3(256), args, 0, st);
    launched += err == cudaSuccess;
  }
  if (launch_err) *launch_err = err;
  return launched;
}
int launch_loss(const Img& im, const float* b, const float* bref, float* gb, float* part, int nparts, float* loss,
                cudaStream_t st) {
  // in place (gb over b or bref) the single launch's reads through the read-only path may not run
  // beside its writes
  if (im.nl * (long long)im.nd <= LOSS_ONE && gb != b && gb != bref) {
    k_loss_cluster<<<LOSS_CTAS, LOSS_THREADS, 0, st>>>(im, b, bref, gb, loss);
    return 1;
  }
  k_loss_partial<<<nparts, 256, 0, st>>>(im, b, bref, gb, part);
  k_sum_final<<<1, 1024, 0, st>>>(part, nparts, 1.0f / (float)(im.nl * im.nd), loss);
  return 2;
}
int launch_envlog_vjp(const Img& im, const float* irf, const float* gb, float* env, unsigned long long* key,
                      float* part, int nparts, float* live_sum, float* gi, int grid, cudaStream_t st, int* status,
                      int fault_barrier) {
  if (g_envlog_fused.load() && gi != irf && gi != gb) {
    // lines per block: the fewest that keep the blocks co-resident, at most four (a block's lines follow
    // one another).  One, two, three, four lines, four kernels, in us: 256 x 4096 75, 105, 152, 200, 112;
    // 400 x 4096 -, -, 152, 200, 165; 600 x 4096 -, -, -, 201, 197; 608 x 2048 -, 68, 96, 102, 88;
    // 1000 x 1024 -, -, -, 80, 92
    for (int lpb = 1; lpb <= 4; ++lpb) {
      const size_t smem = (lpb + 1) * fft_line_bytes(im.nd) + sizeof(float2) * (size_t)(im.nd / 2);
      const int nb = (im.nl + lpb - 1) / lpb;
      if (smem > (size_t)FUSED_SMEM_MAX || nparts < nb) continue;
      if (nb > resident_blocks((const void*)k_envlog_vjp_fused, smem)) continue;
      if (cudaMemsetAsync(key, 0, 3 * sizeof(unsigned long long), st) != cudaSuccess) break;
      int extra = fault_barrier ? 1 : 0;
      long long limit = fault_barrier ? FAULT_BARRIER_CYCLES : BARRIER_CYCLES;
      void* args[] = {(void*)&im, (void*)&irf, (void*)&gb, (void*)&key, (void*)&part, (void*)&gi, (void*)&status,
                      (void*)&extra, (void*)&limit};
      if (cudaLaunchCooperativeKernel((const void*)k_envlog_vjp_fused, dim3(nb), dim3(256), args, smem, st) == cudaSuccess)
        return 1;
      cudaGetLastError();  // the refused cooperative launch: fall back to the four kernels
      break;
    }
  }
  launch_envlog(im, irf, env, key, nullptr, grid, st);
  k_live_sum<<<nparts, 256, 0, st>>>(im, env, key, gb, part);
  k_sum_final<<<1, 1024, 0, st>>>(part, nparts, 1.0f, live_sum);
  const int nb = min(im.nl, grid);
  k_envlog_vjp<<<nb, line_threads(im.nd), 2 * fft_line_bytes(im.nd) + sizeof(float2) * (size_t)(im.nd / 2), st>>>(
      im, irf, gb, key, live_sum, gi);
  return 4;
}
cudaError_t image_set_attrs(int nd) {
  cudaError_t ea = cudaFuncSetAttribute(k_das_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, DT_SMEM_MAX);
  if (ea != cudaSuccess) return ea;
  cudaError_t e0 = cudaFuncSetAttribute(k_envlog_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, FUSED_SMEM_MAX);
  if (e0 != cudaSuccess) return e0;
  e0 = cudaFuncSetAttribute(k_envlog_vjp_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, FUSED_SMEM_MAX);
  if (e0 != cudaSuccess) return e0;
  cudaError_t e = cudaFuncSetAttribute(k_das, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)das_smem(MAX_ELEM, MAX_TX, true));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_das_adj, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(sizeof(float2) * DAS_THREADS * MAX_TX));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_das_adj_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, DJ_SMEM_MAX);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_das_acq, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)das_acq_smem(MAX_ELEM, MAX_TX));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_envelope, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(fft_line_bytes(nd) + sizeof(float2) * (size_t)(nd / 2)));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_envlog_vjp, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(2 * fft_line_bytes(nd) + sizeof(float2) * (size_t)(nd / 2)));
}

}  // namespace usrt
