// Sort-based RF splat (Sec. 2.3.4, Eq. axial_sig): RF[row][n] = sum_i a_i s(n / fs - tau_i).
//
// No scatter of pulse taps with atomics.  Instead:
//   1. rows:   counting sort of the arrivals by row = tx * n_elem + e (histogram, scan, scatter);
//   2. per row (one CTA): counting sort by time bin b = floor(tau fs) into an L2-resident
//      scratch, then a segmented warp reduction of the Taylor moments
//        M_j(b) = sum_{i in b} a_i (-delta_i)^j,  delta_i = tau_i fs - (b + 1/2),  j < 8,
//      and finally the convolution RF[n] = sum_j sum_d G_j(d) M_j(n - d) with the table
//        G_j(d) = g^(j)(d - 1/2) / j!,  g(x) = s(x / fs)
//      (truncation after 8 moments: |delta| <= 1/2 sample gives < 1e-7 relative error).
#include "splat.cuh"

namespace usrt {

// ------------------------------------------------------------------------------------------
// pulse-derivative table: g(x) = Im h(x), h(x) = exp(-x^2 / S + i W x) with S = sigma fs^2 and
// W = 2 pi f0 / fs; with y = (x - i W S / 2) / sqrt(S),  h^(j)(x) = h(x) (-1/sqrt(S))^j H_j(y)
// (physicists' Hermite polynomials, H_{j+1} = 2 y H_j - 2 j H_{j-1}).
// ------------------------------------------------------------------------------------------
__global__ void k_pulse_table(SplatGeom g, float* G) {
  const int d = threadIdx.x;
  if (d >= g.ntaps) return;
  const float x = (float)(g.dlo + d) - 0.5f;
  const float S = g.Sig, W = g.Om;
  const float rs = rsqrtf(S);
  const float yr = x * rs, yi = -0.5f * W * S * rs;
  float e_s, e_c;
  const float mag = expf(-x * x / S);
  sincosf(W * x, &e_s, &e_c);
  const float hr = mag * e_c, hi = mag * e_s;  // h(x)
  float Hr0 = 1.0f, Hi0 = 0.0f, Hr1 = 2.0f * yr, Hi1 = 2.0f * yi;
  float fact = 1.0f, sc = 1.0f;
  for (int j = 0; j < K_MOM; ++j) {
    float Hr, Hi;
    if (j == 0) {
      Hr = Hr0;
      Hi = Hi0;
    } else if (j == 1) {
      Hr = Hr1;
      Hi = Hi1;
    } else {
      const float nr = 2.0f * (yr * Hr1 - yi * Hi1) - 2.0f * (j - 1) * Hr0;
      const float ni = 2.0f * (yr * Hi1 + yi * Hr1) - 2.0f * (j - 1) * Hi0;
      Hr0 = Hr1;
      Hi0 = Hi1;
      Hr1 = nr;
      Hi1 = ni;
      Hr = nr;
      Hi = ni;
    }
    if (j > 0) {
      fact *= (float)j;
      sc *= -rs;
    }
    // Im(h * H) * sc / j!
    G[j * g.ntaps + d] = (hr * Hi + hi * Hr) * sc / fact;
  }
}

// ------------------------------------------------------------------------------------------
// 1. bucket by row
// ------------------------------------------------------------------------------------------
// Where the arrivals come from: the transport's packed list (its count on the device), or the
// caller's four arrays, packed as they are read (a pass of its own that packed them, one atomic
// per warp on one counter, took 200 us for 7.9M arrivals).  get() gives (row, tq, bits(a)), false
// for an arrival outside the time range.  Up to 2^32 - 17 arrivals: the loops over them compare what is
// left with the next stride, as an index past the end of such a list would wrap (64-bit counters
// cost the bucketing of a small list 0.5 of 19 us).
struct PackedArrivals {
  const Arrival* arr;
  const uint32_t* n_arr;
  uint32_t cap;
  __device__ __forceinline__ uint32_t count() const { return min(*n_arr, cap); }
  __device__ __forceinline__ bool row(uint32_t i, uint32_t& r) const {
    r = arr[i].x;
    return true;
  }
  __device__ __forceinline__ bool get(uint32_t i, uint32_t& r, uint2& v) const {
    const Arrival A = arr[i];
    r = A.x;
    v = make_uint2(A.y, A.z);
    return true;
  }
};
struct ListedArrivals {
  const int32_t *tx, *e;
  const float *tau, *a;
  uint32_t n;
  int ne;
  float fs;
  __device__ __forceinline__ uint32_t count() const { return n; }
  __device__ __forceinline__ bool row(uint32_t i, uint32_t& r) const {
    r = (uint32_t)(__ldg(&tx[i]) * ne + __ldg(&e[i]));
    return time_to_tq(__ldg(&tau[i]), 0.0f, fs) != 0xFFFFFFFFu;
  }
  __device__ __forceinline__ bool get(uint32_t i, uint32_t& r, uint2& v) const {
    const uint32_t tq = time_to_tq(__ldg(&tau[i]), 0.0f, fs);
    r = (uint32_t)(__ldg(&tx[i]) * ne + __ldg(&e[i]));
    v = make_uint2(tq, __float_as_uint(__ldg(&a[i])));
    return tq != 0xFFFFFFFFu;
  }
};
template <class Src>
__global__ void k_row_hist(Src src, uint32_t* row_cnt, int nrows) {
  extern __shared__ uint32_t h[];
  const uint32_t n = src.count();
  if (blockIdx.x * blockDim.x >= n) return;
  for (int r = threadIdx.x; r < nrows; r += blockDim.x) h[r] = 0;
  __syncthreads();
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i = n - i > stride ? i + stride : n) {
    uint32_t r;
    if (src.row(i, r)) atomicAdd(&h[r], 1u);
  }
  __syncthreads();
  for (int r = threadIdx.x; r < nrows; r += blockDim.x)
    if (h[r]) atomicAdd(&row_cnt[r], h[r]);
}

// Exclusive scan of n counts by one block; off[n] = total, cursor zeroed.  Warp w owns 32 C
// consecutive counts, read once into C registers per lane with all reads in flight (one L2
// latency; reading each 32-count chunk twice, a latency each time, took 12 us for the ray
// sort's 17,408 buckets, now 6); the C chunk scans are independent shuffles, the 32 warp totals
// are scanned by every warp for itself.
constexpr int SCAN_THREADS = 1024;
template <int C>
__global__ void __launch_bounds__(SCAN_THREADS) k_row_scan(const uint32_t* __restrict__ cnt, uint32_t* off,
                                                           uint32_t* cursor, int n) {
  __shared__ uint32_t warp_total[SCAN_THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lo = warp * (32 * C) + lane;
  uint32_t v[C];
#pragma unroll
  for (int c = 0; c < C; ++c) v[c] = lo + 32 * c < n ? __ldg(&cnt[lo + 32 * c]) : 0u;
  uint32_t sum = 0u;
#pragma unroll
  for (int c = 0; c < C; ++c) sum += v[c];
  sum = __reduce_add_sync(0xFFFFFFFFu, sum);
  if (lane == 0) warp_total[warp] = sum;
  __syncthreads();
  const uint32_t wt = warp_total[lane];
  uint32_t run = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? wt : 0u);
  if (warp == 0) {
    const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, wt);
    if (lane == 0) off[n] = total;
  }
#pragma unroll
  for (int c = 0; c < C; ++c) {
    uint32_t x = v[c];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane >= o) x += u;
    }
    if (lo + 32 * c < n) {
      off[lo + 32 * c] = run + x - v[c];
      cursor[lo + 32 * c] = 0u;
    }
    run += __shfl_sync(0xFFFFFFFFu, x, 31);
  }
}
constexpr int SCAN_SMALL = 4, SCAN_LARGE = 17;  // up to 4096 counts (rows, job buckets), up to 17,408
static_assert(SCAN_THREADS * SCAN_LARGE == COUNT_SCAN_MAX, "one block holds every count");

// scatter into row buckets: each block takes chunks of CH arrivals, ranks them per row in
// shared memory and reserves one range per (chunk, row) with a single global atomic
constexpr int SC_THREADS = 512;
constexpr int SC_PER = 16;
constexpr int SC_CH = SC_THREADS * SC_PER;
template <class Src>
__global__ void __launch_bounds__(SC_THREADS) k_row_scatter(Src src, const uint32_t* off, uint32_t* cursor, uint2* out,
                                                            int nrows) {
  extern __shared__ uint32_t sm[];
  uint32_t* h = sm;           // per-row count in this chunk
  uint32_t* base = sm + nrows;
  const uint32_t n = src.count();
  const uint32_t stride = gridDim.x * SC_CH;
  for (uint32_t c0 = blockIdx.x * SC_CH; c0 < n; c0 = n - c0 > stride ? c0 + stride : n) {
    for (int r = threadIdx.x; r < nrows; r += blockDim.x) h[r] = 0;
    __syncthreads();
    uint32_t row[SC_PER], rank[SC_PER];
    uint2 val[SC_PER];
#pragma unroll
    for (int k = 0; k < SC_PER; ++k) {
      const uint32_t i = k * SC_THREADS + threadIdx.x;  // from c0
      row[k] = 0xFFFFFFFFu;
      uint32_t r;
      if (i < n - c0 && src.get(c0 + i, r, val[k])) {
        row[k] = r;
        rank[k] = atomicAdd(&h[r], 1u);
      }
    }
    __syncthreads();
    for (int r = threadIdx.x; r < nrows; r += blockDim.x)
      if (h[r]) base[r] = off[r] + atomicAdd(&cursor[r], h[r]);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < SC_PER; ++k)
      if (row[k] != 0xFFFFFFFFu) out[base[row[k]] + rank[k]] = val[k];
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------------
// 2. per row: sort by bin, then, segment by segment of the record, segmented moment reduction and
// convolution.  The moments of a whole 4096-sample row take 153 KB, one block per SM, whose
// barriers and dependent passes nothing hid; a segment's take 78 KB, so two blocks of 512 threads
// share an SM and overlap each other's phases.  A segment re-reduces its halo's arrivals (6 %).
// 2048 rows of 4096 samples, 7.9M arrivals: 459 -> 320 us (segments of 1024, three blocks: equal,
// and slower on a hundred rows); 64 nearly empty rows 18.7 -> 16.7 us.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(ROW_THREADS, 2) k_row_splat(SplatGeom g, const uint2* bucket, const uint32_t* off,
                                                              uint2* scratch, const float* Gtab, float* rf) {
  extern __shared__ float smf[];
  const int row = blockIdx.x;
  const int NB = g.nbins;         // bins -HALO .. ns + HALO - 1
  constexpr int MS = row_mom_stride(ROW_SEG);
  const int sh = row_mom_shift(g);  // bin x of a segment is stored at mom_slot(x + sh)
  float* M = smf;                 // [K_MOM][MS], padded: one spare slot after every 8
  float* G = M + K_MOM * MS;      // [K_MOM][MAX_TAPS], zero past ntaps
  uint32_t* hist = reinterpret_cast<uint32_t*>(G + K_MOM * MAX_TAPS);  // [NB]
  __shared__ uint32_t part[ROW_THREADS / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t a0 = off[row], a1 = off[row + 1];
  float* out_row = rf + (size_t)row * g.ns;
  if (a0 == a1) {  // nothing lands on this row
    for (int n = tid; n < g.ns; n += ROW_THREADS) out_row[n] = 0.0f;
    return;
  }
  for (int i = tid; i < NB; i += ROW_THREADS) hist[i] = 0;
  for (int i = tid; i < K_MOM * MAX_TAPS; i += ROW_THREADS) {
    const int j = i / MAX_TAPS, d = i - j * MAX_TAPS;
    G[i] = d < g.ntaps ? Gtab[j * g.ntaps + d] : 0.0f;
  }
  __syncthreads();
  const uint32_t mask = (1u << TQ_FRAC) - 1u;
  // pass 1: histogram of bins
  for (size_t i = (size_t)a0 + tid; i < a1; i += ROW_THREADS) {
    const int b = (int)(bucket[i].x >> TQ_FRAC) - TQ_OFFSET + HALO;
    if (b >= 0 && b < NB) atomicAdd(&hist[b], 1u);
  }
  __syncthreads();
  // exclusive scan of hist in place: a thread's own run of bins, then warps, then the block
  {
    const int per = (NB + ROW_THREADS - 1) / ROW_THREADS;
    const int lo = min(NB, tid * per), hi = min(NB, lo + per);
    uint32_t s = 0;
    for (int b = lo; b < hi; ++b) s += hist[b];
    uint32_t v = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, v, o);
      if (lane >= o) v += u;
    }
    if (lane == 31) part[warp] = v;
    __syncthreads();
    uint32_t run = v - s + __reduce_add_sync(0xFFFFFFFFu, lane < warp ? part[lane & (ROW_THREADS / 32 - 1)] : 0u);
    for (int b = lo; b < hi; ++b) {
      const uint32_t c = hist[b];
      hist[b] = run;
      run += c;
    }
  }
  __syncthreads();
  // pass 2: scatter into bin order (scratch shares the row's index range)
  for (size_t i = (size_t)a0 + tid; i < a1; i += ROW_THREADS) {
    const uint2 v = bucket[i];
    const int b = (int)(v.x >> TQ_FRAC) - TQ_OFFSET + HALO;
    if (b >= 0 && b < NB) scratch[a0 + atomicAdd(&hist[b], 1u)] = v;
  }
  __syncthreads();  // from here hist[b] = end of bin b
  for (int s0 = 0; s0 < g.ns; s0 += ROW_SEG) {  // samples s0 .. s0 + ROW_SEG - 1, bins s0 .. of the row's
    const int b1 = min(NB, s0 + ROW_SEG + 2 * HALO);
    const uint32_t r0 = s0 ? hist[s0 - 1] : 0u, r1 = hist[b1 - 1];
    const int n_seg = min(ROW_SEG, g.ns - s0);
    if (r0 == r1) {  // block-uniform
      for (int n = tid; n < n_seg; n += ROW_THREADS) out_row[s0 + n] = 0.0f;
      continue;
    }
    for (int i = tid; i < K_MOM * MS; i += ROW_THREADS) M[i] = 0.0f;
    __syncthreads();
    // segmented warp reduction of the moments over the bin-sorted arrivals
    for (size_t base = (size_t)r0 + (tid & ~31u); base < r1; base += ROW_THREADS) {
      const size_t i = base + lane;
      int b = -1;
      float m[K_MOM];
#pragma unroll
      for (int j = 0; j < K_MOM; ++j) m[j] = 0.0f;
      if (i < r1) {
        const uint2 v = scratch[a0 + i];
        b = (int)(v.x >> TQ_FRAC) - TQ_OFFSET + HALO - s0;
        const float delta = (float)(v.x & mask) * (1.0f / (float)(1u << TQ_FRAC)) - 0.5f;
        float p = __uint_as_float(v.y);
        m[0] = p;
#pragma unroll
        for (int j = 1; j < K_MOM; ++j) {
          p = p * (-delta);  // the 1/j! of the Taylor term lives in the pulse table
          m[j] = p;
        }
      }
      // inclusive segmented scan: lanes of one bin are contiguous (sorted)
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int bu = __shfl_up_sync(0xFFFFFFFFu, b, o);
#pragma unroll
        for (int j = 0; j < K_MOM; ++j) {
          const float mu = __shfl_up_sync(0xFFFFFFFFu, m[j], o);
          if (lane >= o && bu == b) m[j] += mu;
        }
      }
      const int bn = __shfl_down_sync(0xFFFFFFFFu, b, 1);
      const bool tail = (b >= 0) && (lane == 31 || bn != b);
      if (tail) {
#pragma unroll
        for (int j = 0; j < K_MOM; ++j) atomicAdd(&M[j * MS + mom_slot(b + sh)], m[j]);
      }
    }
    __syncthreads();
    // convolution: out[n] = sum_j sum_d G_j[d] M_j[bin n - dlo - d]; a thread produces 8 consecutive
    // samples (the half of the block that has none waits: the other block's warps fill the SM).
    // Taps go in blocks of 8: the 15 moments a block touches are read once into registers (a
    // sliding window) and feed 64 FMAs.  The shift sh puts every window start on a multiple of 8,
    // so the padded slots of the window are fixed offsets and the lanes of a warp read addresses
    // 9 apart: no bank conflicts.
    const int n0 = 8 * tid;
    if (n0 < n_seg) {
      float acc[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) acc[r] = 0.0f;
      const int xs0 = n0 - g.dlo + HALO + sh - 7;  // window start for taps 0..7, a multiple of 8
      const int ntp = (g.ntaps + 7) & ~7;
      for (int j = 0; j < K_MOM; ++j) {
        const float* Mj = M + j * MS;
        const float* Gj = G + j * MAX_TAPS;
        for (int d0 = 0; d0 < ntp; d0 += 8) {
          const float* W = Mj + 9 * ((xs0 - d0) >> 3);
          float w[15];
#pragma unroll
          for (int k = 0; k < 15; ++k) w[k] = W[k + (k >= 8 ? 1 : 0)];
#pragma unroll
          for (int dd = 0; dd < 8; ++dd) {
            const float gv = Gj[d0 + dd];
#pragma unroll
            for (int r = 0; r < 8; ++r) acc[r] = fmaf(gv, w[r - dd + 7], acc[r]);
          }
        }
      }
      float* out = out_row + s0 + n0;  // rows, segments and groups are whole float4s; rf is 16-byte aligned
      reinterpret_cast<float4*>(out)[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      if (n0 + 4 < n_seg) reinterpret_cast<float4*>(out)[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------------
size_t row_splat_smem(const SplatGeom& g) {
  return sizeof(float) * (size_t)K_MOM * row_mom_stride(ROW_SEG) + sizeof(uint32_t) * g.nbins +
         sizeof(float) * (size_t)K_MOM * MAX_TAPS;
}

void launch_pulse_table(const SplatGeom& g, float* G, cudaStream_t st) { k_pulse_table<<<1, 128, 0, st>>>(g, G); }

void launch_count_scan(const uint32_t* cnt, uint32_t* off, uint32_t* cursor, int n, cudaStream_t st) {
  if (n <= SCAN_THREADS * SCAN_SMALL)
    k_row_scan<SCAN_SMALL><<<1, SCAN_THREADS, 0, st>>>(cnt, off, cursor, n);
  else
    k_row_scan<SCAN_LARGE><<<1, SCAN_THREADS, 0, st>>>(cnt, off, cursor, n);
}

template <class Src>
static void splat_sort(const SplatGeom& g, const Src& src, SplatWork w, int grid, cudaStream_t st) {
  const int nrows = g.nrows;
  cudaMemsetAsync(w.row_cnt, 0, sizeof(uint32_t) * nrows, st);
  k_row_hist<<<grid, 256, sizeof(uint32_t) * nrows, st>>>(src, w.row_cnt, nrows);
  launch_count_scan(w.row_cnt, w.row_off, w.row_cursor, nrows, st);
  k_row_scatter<<<grid, SC_THREADS, 2 * sizeof(uint32_t) * nrows, st>>>(src, w.row_off, w.row_cursor, w.bucket, nrows);
}
void launch_splat_sort(const SplatGeom& g, const Arrival* arr, const uint32_t* n_arr, uint32_t cap, SplatWork w,
                       int grid, cudaStream_t st) {
  splat_sort(g, PackedArrivals{arr, n_arr, cap}, w, grid, st);
}
void launch_splat_sort_list(const SplatGeom& g, const int32_t* tx, const int32_t* e, const float* tau, const float* a,
                            uint32_t n, int ne, float fs, SplatWork w, int grid, cudaStream_t st) {
  splat_sort(g, ListedArrivals{tx, e, tau, a, n, ne, fs}, w, grid, st);
}
void launch_splat_rows(const SplatGeom& g, SplatWork w, const float* G, float* rf, cudaStream_t st) {
  k_row_splat<<<g.nrows, ROW_THREADS, row_splat_smem(g), st>>>(g, w.bucket, w.row_off, w.scratch, G, rf);
}

cudaError_t splat_set_attrs(const SplatGeom& g) {
  return cudaFuncSetAttribute(k_row_splat, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)row_splat_smem(g));
}
cudaError_t row_scatter_set_attrs(int nrows) {
  const int sm = (int)(2 * sizeof(uint32_t) * nrows);
  const cudaError_t e = cudaFuncSetAttribute(k_row_scatter<PackedArrivals>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_row_scatter<ListedArrivals>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
}
cudaError_t row_hist_set_attrs(int nrows) {
  const int sm = (int)(sizeof(uint32_t) * nrows);
  const cudaError_t e = cudaFuncSetAttribute(k_row_hist<PackedArrivals>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_row_hist<ListedArrivals>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
}

}  // namespace usrt
