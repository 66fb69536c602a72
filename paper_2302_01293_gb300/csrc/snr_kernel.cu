// Spectral S/N and best candidate (K3), one CTA per star, for sm_103a.
//
// Sec. 2.2 item 1 of arXiv:2302.01293, Eq. 1 with the paper's two changes:
//   trend(f)  the SR spectrum median-binned into N = round(1 + 3.322 log10 n)
//             equal-width frequency bins (Sturges), bin medians placed at the bin
//             centres and linearly interpolated (constant beyond the end centres);
//   sigma_SR  1.4826 x median |SR - median(SR)| (or of the detrended residual);
//   S/N(f)    (SR(f) - trend(f)) / sigma_SR;
// then the best candidate at the first maximum of S/N (Sec. 2.2 item 2 takes its
// BLS box as the initial P, T0, q and depth).
// Medians are exact order statistics of the FP32 spectrum, found by a radix select over
// order-preserving integer keys: 9-bit digits of the range that the spectrum uses, counted in
// shared memory for all selections at once, until every one is down to a short list, which a
// warp ranks (radix_select).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "qlp_internal.h"

namespace qlp {

// Spectrum keys cached in shared memory (longer spectra are formed again each pass): 24 KB, so
// that a single-sector batch keeps four CTAs per SM, or 96 KB where each CTA has an SM
constexpr int kSnrKeys = 6144, kSnrKeysFew = 24576;
constexpr int kDigitBits = 9, kDigits = 1 << kDigitBits;  // of the selection's digit counts
// Dynamic shared memory: digit counts of `targets` selections and the cached keys
constexpr size_t snr_smem(int targets, int keys) { return ((size_t)targets * kDigits + (size_t)keys) * sizeof(uint32_t); }

__device__ __forceinline__ uint32_t fkey(float v) {
  const uint32_t u = __float_as_uint(v);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float fdekey(uint32_t k) {
  const uint32_t u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
  return __uint_as_float(u);
}

// Sturges bin of spectrum entry k: min(N-1, floor((f_k - f_0) N / span)).
__device__ __forceinline__ int sturges_bin(double f, double f0, double span, int nbin) {
  if (!(span > 0.0)) return 0;
  const int i = (int)floor(__ddiv_rn(__dmul_rn(__dsub_rn(f, f0), (double)nbin), span));
  return min(nbin - 1, i);
}

// A trend segment as float pairs (hi + lo): node abscissa, node value, slope; and a bound on
// the magnitudes that meet in the segment's trend values.
struct TrendSeg {
  float xh, xl, yh, yl, sh, sl, bound;
};

struct SnrShared {
  int lo[kMaxSturges + 1];     // first spectrum index of each Sturges bin (lo[N] = n)
  double xc[kMaxSturges];      // the bins' centres
  int kc[kMaxSturges];         // first spectrum index at or above each
  double xs[kMaxSturges];      // centres of the non-empty bins
  double ys[kMaxSturges];      // their medians
  double sl[kMaxSturges];      // slope of the trend from node i to node i + 1
  int kx[kMaxSturges + 1];     // first spectrum index at or above node i (kx[nx] = n)
  TrendSeg seg[kMaxSturges + 1];  // [i + 1]: from node i; [0] below the first node
  int nx;
  float mh, ml, mlo, mhi;      // the median as a float pair, and the range of SR the pair serves
  int med_pair;
  // selection targets (a Sturges bin each, then the whole spectrum)
  uint32_t prefix[kMaxSturges + 1];  // the digits found so far, then the selected key
  int rank[kMaxSturges + 1];         // rank among the keys that share the prefix (-1: no target)
  int left[kMaxSturges + 1];         // keys that share it
  uint32_t next[kMaxSturges + 1];    // the next larger order statistic's key
  int even[kMaxSturges + 1];         // 1: that one is wanted
  int fill[kMaxSturges + 1];         // candidates gathered
  uint32_t kmin[32], kmax[32];
  int more;                          // some target still has more candidates than its list holds
  double med, sigma;
  float best_v[32];
  int best_i[32];
};

// Trend at spectrum entry k of frequency f, np.interp semantics, in FP64; i is the last node
// at or below f (-1 below the first). Each segment's slope is taken once.
__device__ __forceinline__ double trend_at(const SnrShared& sh, double f, int i) {
  if (i < 0) return sh.ys[0];
  if (i >= sh.nx - 1) return sh.ys[sh.nx - 1];
  return __dadd_rn(sh.ys[i], __dmul_rn(sh.sl[i], __dsub_rn(f, sh.xs[i])));
}
// That node for entry k: the caller's pointer, moved up as k grows.
__device__ __forceinline__ void move_node(const SnrShared& sh, int k, int& i) {
  while (i + 1 < sh.nx && k >= sh.kx[i + 1]) ++i;
}

// fl32(fl64(x / sigma)) from rs = fl64(1 / sigma): x rs lies within 3 ulps (FP64) of the
// rounded quotient, so both round to the same float unless x rs is within 16 ulps of the
// middle of two floats (its low 29 bits near 2^28), where, as for results outside the
// normal range, the quotient is taken exactly.
__device__ __forceinline__ float snr_of(double x, double sigma, double rs) {
  const double q = __dmul_rn(x, rs);
  const int mid = (__double2loint(q) & 0x1fffffff) - 0x10000000;
  const int e = (__double2hiint(q) >> 20) & 0x7ff;
  if (abs(mid) > 16 && e > 1023 - 100 && e < 1023 + 100) return __double2float_rn(q);
  return __double2float_rn(__ddiv_rn(x, sigma));
}

// Exact difference (s, e) = a - b (TwoSum).
__device__ __forceinline__ float two_diff(float a, float b, float& e) {
  const float s = __fsub_rn(a, b), bb = __fsub_rn(s, a);
  e = __fsub_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fadd_rn(b, bb));
  return s;
}

// fl32(fl64((v - trend(f)) / sigma)) without the FP64 pipe (1/64 of the FP32 rate here, and
// half of this kernel's time before): the same value in float pairs. Its roundings and
// the FP64 chain's own add up to less than 20 2^-48 of the magnitudes that meet (bound +
// |v|); err is 2^-43 of them. Where the pair's low part and err together stay inside the
// half spacing around its high part, every value within err rounds to the high part, the
// FP64 chain's too. False near the middle of two floats, at powers of two and for tiny
// results (a few entries in a thousand): the caller takes the FP64 chain.
__device__ __forceinline__ bool snr_pair(float v, double f, const TrendSeg& g, float rh, float rl, float c, float& out) {
  const uint32_t fhi = (uint32_t)__double2hiint(f), flo = (uint32_t)__double2loint(f);
  const float fh = __uint_as_float(((fhi - 0x38000000u) << 3) | (flo >> 29));  // f truncated to 24 bits
  const float fl = __fmul_rn(__uint2float_rn(flo & 0x1fffffffu), __uint_as_float(((fhi >> 20) - 948u) << 23));
  float e;
  const float s = two_diff(fh, g.xh, e);  // f - x
  const float t = __fadd_rn(e, __fsub_rn(fl, g.xl));
  const float dh = __fadd_rn(s, t), dl = __fsub_rn(t, __fsub_rn(dh, s));
  const float p = __fmul_rn(g.sh, dh);    // slope (f - x)
  const float pe = __fmaf_rn(g.sl, dh, __fmaf_rn(g.sh, dl, __fmaf_rn(g.sh, dh, -p)));
  const float a = two_diff(g.yh, -p, e);  // y + slope (f - x)
  const float al = __fadd_rn(e, __fadd_rn(g.yl, pe));
  const float d = two_diff(v, a, e);      // v - trend
  const float r = __fsub_rn(e, al);
  const float Dh = __fadd_rn(d, r), Dl = __fsub_rn(r, __fsub_rn(Dh, d));
  const float q = __fmul_rn(Dh, rh);      // over sigma
  const float qe = __fmaf_rn(Dl, rh, __fmaf_rn(Dh, rl, __fmaf_rn(Dh, rh, -q)));
  const float qh = __fadd_rn(q, qe), ql = __fsub_rn(qe, __fsub_rn(qh, q));
  const float err = __fmul_rn(__fadd_rn(g.bound, fabsf(v)), c);
  const uint32_t qb = __float_as_uint(qh);
  const uint32_t ex = qb & 0x7f800000u;
  out = qh;
  return (qb & 0x7fffffu) != 0u && ex > ((127u - 60u) << 23) && ex < ((127u + 60u) << 23) &&
         __fadd_rn(fabsf(ql), err) < __uint_as_float(ex - (24u << 23));
}

// fkey(fl32(fl64(|v - med|))): the median as a float pair of at most 31 bits and v within
// 2^20 of it (or 0), so that the difference fits 53 bits and its exact value, the sum of
// the two differences' parts, is rounded once; else, and where a part is not exact, in FP64.
__device__ __forceinline__ uint32_t mad_key(const SnrShared& sh, float v) {
  const float av = fabsf(v);
  if (sh.med_pair && (av == 0.f || (av >= sh.mlo && av <= sh.mhi))) {
    float e, e2;
    const float s = two_diff(v, sh.mh, e);
    const float t = two_diff(e, sh.ml, e2);
    if (e2 == 0.f) return fkey(fabsf(__fadd_rn(s, t)));
  }
  return fkey((float)fabs(__dsub_rn((double)v, sh.med)));
}
__device__ __forceinline__ void set_median(SnrShared& sh, double med) {
  sh.med = med;
  sh.mh = __double2float_rn(med);
  sh.ml = __double2float_rn(__dsub_rn(med, (double)sh.mh));
  const float a = fabsf(sh.mh);
  sh.mlo = a * 0x1p-19f;
  sh.mhi = a * 0x1p19f;
  sh.med_pair = (__double2loint(med) & 0x3fffff) == 0 && a > 1e-25f && a < 1e25f;
}

// First entry of the ascending grid at or above frequency x (positive, so that the bit
// patterns order as the values do), by one warp: 32 probes a step, three or four steps of one
// memory latency each where one thread's bisection takes a dozen.
__device__ __forceinline__ int first_at_or_above(const double2* fq, int n, double x) {
  const int lane = threadIdx.x & 31;
  const long long xb = __double_as_longlong(x);
  int a = 0, b = n;  // the answer lies in [a, b]
  while (a < b) {
    const int step = (b - a + 31) / 32, k = a + lane * step;
    const bool below = k < b && __double_as_longlong(fq[k].x) < xb;
    const int c = __popc(__ballot_sync(0xffffffffu, below));  // probes below x: the first c
    b = c < 32 ? min(b, a + c * step) : b;
    a = c > 0 ? a + (c - 1) * step + 1 : a;
  }
  return a;
}

// The trend's segment slopes and segments (the segments' boundaries kx are known).
__device__ __forceinline__ void trend_slopes(SnrShared& sh, double f_last) {
  for (int j = threadIdx.x; j <= sh.nx; j += blockDim.x) {
    const int i = max(j - 1, 0);
    double sl = 0.0, xe = f_last;
    if (j > 0 && j < sh.nx) {
      sl = __ddiv_rn(__dsub_rn(sh.ys[i + 1], sh.ys[i]), __dsub_rn(sh.xs[i + 1], sh.xs[i]));
      sh.sl[i] = sl;
      xe = sh.xs[i + 1];
    }
    TrendSeg g;
    g.xh = __double2float_rn(sh.xs[i]);
    g.xl = __double2float_rn(__dsub_rn(sh.xs[i], (double)g.xh));
    g.yh = __double2float_rn(sh.ys[i]);
    g.yl = __double2float_rn(__dsub_rn(sh.ys[i], (double)g.yh));
    g.sh = __double2float_rn(sl);
    g.sl = __double2float_rn(__dsub_rn(sl, (double)g.sh));
    g.bound = __double2float_ru(fabs(sh.ys[i]) + 2.0 * fabs(sl) * fmax(xe, sh.xs[i]));
    sh.seg[j] = g;
  }
}

// Selects, for each of the targets t with rank[t] >= 0, the rank[t]-th smallest key (into
// prefix[t]) and, where even[t], the next order statistic (into next[t]); target i <
// nbin takes the entries of Sturges bin i, target nbin all of them. Keys count from the
// spectrum's smallest, so that a digit of kDigitBits splits the range that is used (the
// top bits of the floats themselves are the same for nearly all entries, and their counts
// one contended word); a warp scans a target's digit counts. Once every target's digit
// holds at most kList keys, one more pass gathers them (and, for an upper middle value that
// may lie past them, the smallest key above), and a warp per target ranks its list: usually
// two or three passes over the spectrum rather than five. key_of(k) gives entry k's key;
// every thread visits the same entries each pass, so it caches them in keys (when not
// null) without a barrier.
constexpr int kList = 64;
template <typename KeyOf>
__device__ void radix_select(SnrShared& sh, uint32_t* hist, uint32_t* keys, int nbin, int n, KeyOf key_of) {
  const int nt = nbin + 1, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t lo = 0xffffffffu, hi = 0u;
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const uint32_t key = key_of(k);
    if (keys) keys[k] = key;
    lo = min(lo, key);
    hi = max(hi, key);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    sh.kmin[warp] = lo;
    sh.kmax[warp] = hi;
  }
  for (int t = threadIdx.x; t < nt; t += blockDim.x) {
    sh.prefix[t] = 0u;
    sh.next[t] = 0xffffffffu;
    sh.fill[t] = 0;
  }
  __syncthreads();
  lo = __reduce_min_sync(0xffffffffu, sh.kmin[min(lane, nw - 1)]);
  hi = __reduce_max_sync(0xffffffffu, sh.kmax[min(lane, nw - 1)]);
  int shift = max(0, 32 - __clz((int)(hi - lo)) - kDigitBits);
  uint32_t mask = 0u;  // digits found so far (of key - lo)
  for (;;) {           // at most four passes: 32 bits in digits of 9
    if (threadIdx.x == 0) sh.more = 0;
    for (int i = threadIdx.x; i < nt * (kDigits / 4); i += blockDim.x)
      reinterpret_cast<uint4*>(hist)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    int b = 0;
    const uint32_t pg = sh.prefix[nbin];
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const uint32_t key = (keys ? keys[k] : key_of(k)) - lo;
      const uint32_t dig = (key >> shift) & (kDigits - 1);
      if ((key & mask) == pg) atomicAdd(&hist[nbin * kDigits + dig], 1u);
      if (nbin > 0) {
        while (k >= sh.lo[b + 1]) ++b;
        if ((key & mask) == sh.prefix[b]) atomicAdd(&hist[b * kDigits + dig], 1u);
      }
    }
    __syncthreads();
    for (int t = warp; t < nt; t += nw) {
      const int r = sh.rank[t];
      if (r < 0) continue;
      constexpr int kPer = kDigits / 32;
      int c[kPer], own = 0;
#pragma unroll
      for (int i = 0; i < kPer; i += 4) {
        const uint4 v = reinterpret_cast<const uint4*>(hist + t * kDigits + kPer * lane)[i / 4];
        c[i] = (int)v.x; c[i + 1] = (int)v.y; c[i + 2] = (int)v.z; c[i + 3] = (int)v.w;
        own += c[i] + c[i + 1] + c[i + 2] + c[i + 3];
      }
      int incl = own;
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      const int before = incl - own;
      if (r >= before && r < incl) {  // one lane holds the digit
        int rest = r - before, d = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i)
          if (d == i && rest >= c[i]) {
            rest -= c[i];
            d = i + 1;
          }
        int cnt = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) cnt = i == d ? c[i] : cnt;
        sh.prefix[t] |= (uint32_t)(kPer * lane + d) << shift;
        sh.rank[t] = rest;
        sh.left[t] = cnt;
        if (cnt > kList && shift > 0) sh.more = 1;
      }
    }
    __syncthreads();
    mask |= (uint32_t)(kDigits - 1) << shift;
    if (!sh.more) break;  // block-uniform; shift = 0 always ends here
    mask = 0xffffffffu << shift;
    shift = max(0, shift - kDigitBits);
    __syncthreads();  // every thread has read more
  }
  // gather: the keys in each target's digit (where shift = 0 they are all equal), and the
  // smallest key above it
  mask = 0xffffffffu << shift;
  uint32_t* list = hist;  // kList keys per target, over the counts
  {
    int b = 0;
    const uint32_t pg = sh.prefix[nbin];
    const bool eg = sh.even[nbin] && sh.rank[nbin] + 1 >= sh.left[nbin];
    volatile uint32_t* next = sh.next;
    auto visit = [&](int t, uint32_t key, uint32_t p, bool above) {
      if ((key & mask) == p) {
        if (shift > 0) list[t * kList + atomicAdd(&sh.fill[t], 1)] = key;
      } else if (above && key > p && key < next[t]) {
        atomicMin(&sh.next[t], key);
      }
    };
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const uint32_t key = (keys ? keys[k] : key_of(k)) - lo;
      visit(nbin, key, pg, eg);
      if (nbin > 0) {
        while (k >= sh.lo[b + 1]) ++b;
        visit(b, key, sh.prefix[b], sh.even[b] && sh.rank[b] + 1 >= sh.left[b]);
      }
    }
  }
  __syncthreads();
  for (int t = warp; t < nt; t += nw) {
    const int r = sh.rank[t], m = sh.left[t];
    if (r < 0) continue;
    uint32_t v0 = sh.prefix[t], v1 = r + 1 < m ? v0 : sh.next[t];
    if (shift > 0) {  // rank the list's keys, two per lane (ties by place)
      const uint32_t ka = lane < m ? list[t * kList + lane] : 0xffffffffu;
      const uint32_t kb = lane + 32 < m ? list[t * kList + lane + 32] : 0xffffffffu;
      int ra = 0, rb = 0;
      for (int j = 0; j < m; ++j) {
        const uint32_t x = __shfl_sync(0xffffffffu, j < 32 ? ka : kb, j & 31);
        ra += x < ka || (x == ka && j < lane);
        rb += x < kb || (x == kb && j < lane + 32);
      }
      auto at = [&](int q) {  // the key of rank q
        const bool a = lane < m && ra == q, bb = lane + 32 < m && rb == q;
        return __reduce_min_sync(0xffffffffu, a ? ka : bb ? kb : 0xffffffffu);
      };
      v0 = at(r);
      if (r + 1 < m) v1 = at(r + 1);
    }
    if (lane == 0) {
      sh.prefix[t] = v0 + lo;
      sh.next[t] = v1 + lo;
    }
  }
  __syncthreads();
}

// rank and even of target t over c entries: the lower middle value, and whether the upper
// one is another entry
__device__ __forceinline__ void median_target(SnrShared& sh, int t, int c) {
  sh.rank[t] = c > 0 ? (c - 1) / 2 : -1;
  sh.even[t] = (c > 0 && (c & 1) == 0) ? 1 : 0;
}
__device__ __forceinline__ double median_of(const SnrShared& sh, int t, int c) {
  const double v0 = (double)fdekey(sh.prefix[t]);
  const double v1 = (c & 1) ? v0 : (double)fdekey(sh.next[t]);
  return __dmul_rn(0.5, __dadd_rn(v0, v1));
}

// THREADS 512, or 1,024 when the launch has fewer stars than the chip has SMs (a star's
// passes are then latency-bound). Time goes into the select's passes and barriers; before,
// into FP64 (two divisions and some twenty operations an entry at 1/64 of the FP32 rate),
// contended digit counts and 256 dependent loads per target and pass: 4,096 stars 2.30 ->
// 0.70 ms, 150 stars 249 -> 59 us, one star of 4,432 frequencies 120 -> 41 us.
template <int THREADS>
__global__ void __launch_bounds__(THREADS) snr_kernel(const SnrArgs a) {
  extern __shared__ __align__(16) uint32_t hist[];
  __shared__ SnrShared sh;
  const int s = blockIdx.x;
  const StarDev st = a.stars[s];
  const int n = st.n_f;
  qlp_bls_best* out = a.best + s;

  if (n <= 0 || st.status != 0) {
    if (threadIdx.x < kTrendDoubles && a.trend_out) a.trend_out[(size_t)s * kTrendDoubles + threadIdx.x] = 0.0;
    if (threadIdx.x == 0) {
      out->f_idx = -1;
      out->f = out->period = out->t0 = out->q = out->depth = out->sr = out->snr = 0.0;
      out->j = out->k = out->m = out->nbins = -1;
      out->status = st.status;
      out->pad = 0;
    }
    return;
  }
  const int nbin = st.sturges_nb;
  if (nbin < 1 || nbin > a.max_sturges) {
    if (threadIdx.x == 0) {
      atomicOr(a.err, kErrSturges);
      out->f_idx = -1;
      out->status = st.status;
    }
    return;
  }
  const float* sr = a.sr + st.f_off;
  const double2* fq = a.fq + st.f_off;
  float* snr = a.snr + st.f_off;
  uint32_t* keys = n <= a.key_cap ? hist + (a.max_sturges + 1) * kDigits : nullptr;

  if (a.trend_in) {
    // S/N from a given trend and sigma (the refined search of the learned proposal)
    const double* tr = a.trend_in + (size_t)s * kTrendDoubles;
    for (int i = threadIdx.x; i < kMaxSturges; i += blockDim.x) {
      sh.xs[i] = tr[4 + i];
      sh.ys[i] = tr[4 + kMaxSturges + i];
    }
    if (threadIdx.x == 0) {
      // a count that no record of this kernel holds is read as none: it bounds the nodes below
      sh.nx = tr[0] >= 1.0 && tr[0] <= (double)kMaxSturges ? (int)tr[0] : 0;
      sh.sigma = tr[1];
      sh.med = tr[2];
    }
    __syncthreads();
    if (sh.nx < 1) {
      if (threadIdx.x == 0) {
        out->f_idx = -1;
        out->status = st.status | QLP_STAR_ZERO_MAD;
        out->f = out->period = out->t0 = out->q = out->depth = out->sr = out->snr = 0.0;
        out->j = out->k = out->m = out->nbins = -1;
        out->pad = 0;
      }
      for (int k = threadIdx.x; k < n; k += blockDim.x) snr[k] = 0.f;
      return;
    }
    for (int i = threadIdx.x >> 5; i < sh.nx; i += THREADS / 32) {
      const int k = first_at_or_above(fq, n, sh.xs[i]);
      if ((threadIdx.x & 31) == 0) sh.kx[i] = k;
    }
    trend_slopes(sh, fq[n - 1].x);
    __syncthreads();
  } else {
  const double f0 = fq[0].x;
  const double span = __dsub_rn(fq[n - 1].x, f0);
  // bin boundaries: lo[i] = first k with bin(k) >= i (a warp each): found by the frequency
  // f0 + i span / N, then moved to where the bin's own expression says; and the bins'
  // centres with the first entry at or above each
  for (int i = threadIdx.x >> 5; i <= nbin; i += THREADS / 32) {
    int lo = i == 0 ? 0 : n, kx = 0;
    double xc = 0.0;
    if (i < nbin) {
      xc = __dadd_rn(f0, __ddiv_rn(__dmul_rn((double)i + 0.5, span), (double)nbin));
      kx = first_at_or_above(fq, n, xc);
      if (i > 0) {
        lo = first_at_or_above(fq, n, __dadd_rn(f0, __ddiv_rn(__dmul_rn((double)i, span), (double)nbin)));
        while (lo > 0 && sturges_bin(fq[lo - 1].x, f0, span, nbin) >= i) --lo;
        while (lo < n && sturges_bin(fq[lo].x, f0, span, nbin) < i) ++lo;
      }
    }
    if ((threadIdx.x & 31) == 0) {
      sh.lo[i] = lo;
      if (i < nbin) {
        sh.xc[i] = xc;
        sh.kc[i] = kx;
      }
    }
  }
  __syncthreads();

  // medians of every bin (targets 0 .. N - 1) and of the whole spectrum (N)
  for (int i = threadIdx.x; i <= nbin; i += blockDim.x)
    median_target(sh, i, (i < nbin) ? sh.lo[i + 1] - sh.lo[i] : n);
  __syncthreads();
  radix_select(sh, hist, keys, nbin, n, [&](int k) { return fkey(sr[k]); });
  if (threadIdx.x < 32) {  // nodes: the non-empty bins, in order
    const int lane = threadIdx.x;
    int nx = 0;
    for (int i0 = 0; i0 < nbin; i0 += 32) {
      const int i = i0 + lane;
      const int c = i < nbin ? sh.lo[i + 1] - sh.lo[i] : 0;
      const unsigned m = __ballot_sync(0xffffffffu, c > 0);
      if (c > 0) {
        const int x = nx + __popc(m & ((1u << lane) - 1u));
        sh.xs[x] = sh.xc[i];
        sh.kx[x] = sh.kc[i];
        sh.ys[x] = median_of(sh, i, c);
      }
      nx += __popc(m);
    }
    if (lane == 0) {
      sh.nx = nx;
      set_median(sh, median_of(sh, nbin, n));
    }
  }
  __syncthreads();
  trend_slopes(sh, fq[n - 1].x);
  if (threadIdx.x == 0) median_target(sh, 0, n);
  __syncthreads();

  if (a.mad_mode == QLP_MAD_RESID) {
    // of the residual SR - trend: its median, then the median of its distances from that
    int ti = -1, tk = 0;
    auto residual = [&](int k) {
      if (k < tk) ti = -1;  // a new pass starts again at the thread's first entry
      tk = k;
      move_node(sh, k, ti);
      const double f = fq[k].x;
      return __dsub_rn((double)sr[k], trend_at(sh, f, ti));
    };
    radix_select(sh, hist, keys, 0, n, [&](int k) { return fkey((float)residual(k)); });
    if (threadIdx.x == 0) {
      sh.med = median_of(sh, 0, n);
      median_target(sh, 0, n);
    }
    __syncthreads();
    radix_select(sh, hist, keys, 0, n, [&](int k) { return fkey((float)fabs(__dsub_rn(residual(k), sh.med))); });
  } else {
    radix_select(sh, hist, keys, 0, n, [&](int k) { return mad_key(sh, sr[k]); });
  }
  if (threadIdx.x == 0) sh.sigma = __dmul_rn(1.4826, median_of(sh, 0, n));
  __syncthreads();
  if (a.trend_out && threadIdx.x < kTrendDoubles) {
    const int i = threadIdx.x - 4, j = i - kMaxSturges;
    double v;
    if (i < 0) v = threadIdx.x == 0 ? (double)sh.nx : threadIdx.x == 1 ? sh.sigma : threadIdx.x == 2 ? sh.med : 0.0;
    else if (j < 0) v = i < sh.nx ? sh.xs[i] : 0.0;
    else v = j < sh.nx ? sh.ys[j] : 0.0;
    a.trend_out[(size_t)s * kTrendDoubles + threadIdx.x] = v;
  }
  }  // trend computed here
  const double sigma = sh.sigma;
  const double rs = __ddiv_rn(1.0, sigma);
  const bool pairs = sigma > 1e-18 && sigma < 1e18;
  const float rh = pairs ? __double2float_rn(rs) : 0.f;
  const float rl = pairs ? __double2float_rn(__dsub_rn(rs, (double)rh)) : 0.f, c = rh * 0x1p-43f;

  // S/N and its first maximum
  float bv = -3.0e38f;
  int bi = n, node = -1;
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    float v = 0.f;
    if (sigma > 0.0) {
      const float x = sr[k];
      const double f = fq[k].x;
      move_node(sh, k, node);
      if (!pairs || !snr_pair(x, f, sh.seg[node + 1], rh, rl, c, v))
        v = snr_of(__dsub_rn((double)x, trend_at(sh, f, node)), sigma, rs);
    }
    snr[k] = v;
    if (v > bv) { bv = v; bi = k; }   // k increases: first maximum per thread
  }
  for (int off = 16; off > 0; off >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, bv, off);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
    if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { sh.best_v[warp] = bv; sh.best_i[warp] = bi; }
  __syncthreads();
  if (warp > 0) return;
  bv = lane < THREADS / 32 ? sh.best_v[lane] : -3.0e38f;
  bi = lane < THREADS / 32 ? sh.best_i[lane] : n;
  for (int off = 16; off > 0; off >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, bv, off);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
    if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
  }
  if (lane == 0) {
    const int at = bi < n ? bi : 0;  // every value of the record's entry, loaded at once
    const int j = (bi < n) ? (int)a.qidx[st.f_off + at] : 255;
    const int kb = (int)a.kbin[st.f_off + at];
    const double r = (double)a.rbest[st.f_off + at];
    const double sv = (double)a.sbest[st.f_off + at];
    const double2 fb = fq[at];
    const float srb = sr[at];
    out->status = st.status;
    out->pad = 0;
    if (!(sigma > 0.0) || bi >= n || j >= a.nq) {
      if (!(sigma > 0.0)) out->status |= QLP_STAR_ZERO_MAD;
      out->f_idx = -1;
      out->f = out->period = out->t0 = out->q = out->depth = out->sr = out->snr = 0.0;
      out->j = out->k = out->m = out->nbins = -1;
    } else {
      const double f = fb.x;
      const double qmin = fb.y;
      // shared histogram: nbins(q_min) and the window m_j; per-duration histograms:
      // nbins(q_j) bins of q_j / noverlap and a window of noverlap bins
      const int nb = a.per_q ? (int)ceil(__ddiv_rn(a.noverlap, __dmul_rn(qmin, a.E[j])))
                             : (int)ceil(__ddiv_rn(a.noverlap, qmin));
      const int m = a.per_q ? a.m_perq
                            : max(1, (int)floor(__dadd_rn(__dmul_rn(__dmul_rn(qmin, a.E[j]), (double)nb), 0.5)));
      const double period = __ddiv_rn(1.0, f);
      const double mid = __ddiv_rn(__dadd_rn((double)kb, __dmul_rn(0.5, (double)m)), (double)nb);
      out->f_idx = bi;
      out->f = f;
      out->period = period;
      out->t0 = __dadd_rn(st.t_ref, __dmul_rn(period, __dsub_rn(mid, floor(mid))));
      out->q = __ddiv_rn((double)m, (double)nb);
      out->depth = -__ddiv_rn(sv, __dmul_rn(r, __dsub_rn(1.0, r)));
      out->sr = (double)srb;
      out->snr = (double)bv;
      out->j = j;
      out->k = kb;
      out->m = m;
      out->nbins = nb;
    }
  }
}

// Coarse spectrum of the learned proposal as the network input: out[s][k] =
// (asinh(S/N / 4), 1) for the star's searched coarse bins k (entry i of its
// spectrum is bin grid_k0 - i), (0, 0) elsewhere; BF16 [n_stars][n_bins][2]. The
// monotone asinh compression keeps the ordering of the S/N while bounding the
// range the network sees (S/N from -5 to 10^4 maps to about -1.1 to 8.5).
// The network input per coarse bin k: a(k) = asinh(S/N / 4) and 1 on searched bins,
// then a() at the harmonic bins k + d2, k - d2, k + d3, k - d3 (periods 2P, P/2, 3P,
// P/3), 0 off the grid or on bins not searched; with snr_rows, also the FP32 S/N
// itself per bin (0 elsewhere) in [star][bin] rows. Pass 1 writes channels 0 and 1;
// after the block barrier pass 2 copies channel 0 of the harmonic bins (the same
// BF16 values).
__global__ void coarse_tensor_kernel(const StarDev* stars, const float* snr, int n_bins, __nv_bfloat16* out,
                                     float* snr_rows, int d2, int d3) {
  constexpr int C = QLP_CNN_IN_CH;
  const int s = blockIdx.x;
  const StarDev st = stars[s];
  __nv_bfloat16* row = out + (size_t)s * n_bins * C;
  float* srow = snr_rows ? snr_rows + (size_t)s * n_bins : nullptr;
  const __nv_bfloat16 zero = __float2bfloat16_rn(0.f);
  for (int k = threadIdx.x; k < n_bins; k += blockDim.x) {
    row[C * k] = zero;
    row[C * k + 1] = zero;
    if (srow) srow[k] = 0.f;
  }
  __syncthreads();
  if (st.status == 0) {
    for (int i = threadIdx.x; i < st.n_f; i += blockDim.x) {
      const int k = st.grid_k0 - i;
      if (k < 0 || k >= n_bins) continue;
      const float v = snr[st.f_off + i];
      row[C * k] = __float2bfloat16_rn(asinhf(0.25f * v));
      row[C * k + 1] = __float2bfloat16_rn(1.f);
      if (srow) srow[k] = v;
    }
  }
  __syncthreads();
  const int dk[4] = {d2, -d2, d3, -d3};
  for (int k = threadIdx.x; k < n_bins; k += blockDim.x) {
    const bool here = __bfloat162float(row[C * k + 1]) > 0.f;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const int kh = k + dk[h];
      row[C * k + 2 + h] = (here && kh >= 0 && kh < n_bins) ? row[C * kh] : zero;
    }
  }
}

int launch_coarse_tensor(const StarDev* stars, int n_stars, const float* snr, int n_bins, void* out,
                         float* snr_rows, int d2, int d3, void* stream) {
  if (n_stars <= 0) return 0;
  coarse_tensor_kernel<<<n_stars, 256, 0, (cudaStream_t)stream>>>(stars, snr, n_bins,
                                                                   static_cast<__nv_bfloat16*>(out), snr_rows,
                                                                   d2, d3);
  return (int)cudaGetLastError();
}

// The k largest logits of each row among valid bins (x0 channel 1 > 0, rows of
// QLP_CNN_IN_CH channels), largest first, ties to the lower bin; -1 when fewer than k bins
// are valid. The row's logits sit in shared memory as order-preserving integer keys (0 where
// not valid or taken; below -3e38 and NaN are never taken) and every thread and warp keeps
// its best: a round compares the warps' bests, and only the warp that held the winner finds
// its next one, so a round costs a few warp-wide integer reductions and two barriers rather
// than a scan of the row (256 rows of 4,096, k = 32: 66 -> 16 us).
constexpr int kTopThreads = 256, kTopWarps = kTopThreads / 32;
constexpr int kTopMaxLen = 49088;
__global__ void __launch_bounds__(kTopThreads) topk_kernel(const float* logits, const __nv_bfloat16* x0, int len,
                                                           int k, int32_t* out) {
  extern __shared__ uint32_t s_z[];
  __shared__ uint32_t bv[kTopWarps];
  __shared__ int bi[kTopWarps];
  const int s = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* z = logits + (size_t)s * len;
  const __nv_bfloat16* m = x0 + (size_t)s * len * QLP_CNN_IN_CH;
  uint32_t v = 0u;  // the largest key of this thread's entries threadIdx.x + 256 j, the lowest index
  int idx = len;
#pragma unroll 4
  for (int i = threadIdx.x; i < len; i += kTopThreads) {
    const float x = z[i];
    const uint32_t key = __bfloat162float(m[QLP_CNN_IN_CH * i + 1]) > 0.f && x >= -3.0e38f ? fkey(x + 0.f) : 0u;
    s_z[i] = key;
    if (key > v) { v = key; idx = i; }
  }
  // the warp's best of (key, index): the largest key, then the lowest index that has it
  auto reduce = [](uint32_t key, int i, uint32_t& rk, int& ri) {
    rk = __reduce_max_sync(0xffffffffu, key);
    ri = (int)__reduce_min_sync(0xffffffffu, key == rk ? (unsigned)i : 0x7fffffffu);
  };
  auto warp_best = [&]() {
    uint32_t wk;
    int wi;
    reduce(v, idx, wk, wi);
    if (lane == 0) { bv[warp] = wk; bi[warp] = wi; }
  };
  warp_best();
  __syncthreads();
  for (int r = 0; r < k; ++r) {
    uint32_t tk;
    int ti;
    reduce(lane < kTopWarps ? bv[lane] : 0u, lane < kTopWarps ? bi[lane] : len, tk, ti);
    if (threadIdx.x == 0) out[(size_t)s * k + r] = tk > 0u ? ti : -1;
    if (tk == 0u) continue;  // block-uniform: none left
    __syncthreads();         // every thread has read the warps' bests
    const int col = ti & (kTopThreads - 1);  // the winner's thread: its warp finds its next best
    if (warp == (col >> 5)) {
      if (lane == 0) s_z[ti] = 0u;
      __syncwarp();
      uint32_t nk = 0u;
      int ni = len;
      for (int i = col + kTopThreads * lane; i < len; i += kTopThreads * 32)
        if (s_z[i] > nk) { nk = s_z[i]; ni = i; }
      reduce(nk, ni, nk, ni);
      if (threadIdx.x == (unsigned)col) { v = nk; idx = ni; }
      warp_best();
    }
    __syncthreads();
  }
}

int launch_topk(const float* logits, const void* x0, int batch, int len, int k, int32_t* out, void* stream) {
  if (batch <= 0) return 0;
  if (len > kTopMaxLen) return (int)cudaErrorInvalidValue;
  const int smem = len * (int)sizeof(float);
  // always the largest row's (one setting for every host thread; see launch_snr)
  const cudaError_t e = cudaFuncSetAttribute(topk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kTopMaxLen * (int)sizeof(float));
  if (e != cudaSuccess) return (int)e;
  topk_kernel<<<batch, kTopThreads, smem, (cudaStream_t)stream>>>(logits, static_cast<const __nv_bfloat16*>(x0), len,
                                                                   k, out);
  return (int)cudaGetLastError();
}

// The n strongest S/N peaks of each star: repeatedly the largest S/N (ties: the
// lowest index) among the frequencies not excluded yet, then every frequency
// with |f / f_pick - 1| < sep is excluded. The ratio is monotone along the
// ascending grid, so each exclusion is one index range, found by binary search.
constexpr int kMaxPeaks = 64;

__device__ __forceinline__ bool near_pick(double f, double fp, double sep) {
  return fabs(__dsub_rn(__ddiv_rn(f, fp), 1.0)) < sep;
}

__global__ void __launch_bounds__(256) peaks_kernel(const StarDev* stars, const double2* fq, const float* snr,
                                                    int n_peaks, double sep, int32_t* out) {
  __shared__ int s_lo[kMaxPeaks], s_hi[kMaxPeaks];
  __shared__ float bv[8];
  __shared__ int bi[8];
  __shared__ int s_pick;
  const int s = blockIdx.x;
  const StarDev st = stars[s];
  const int nf = st.n_f;
  const float* v = snr + st.f_off;
  const double2* f = fq + st.f_off;
  int32_t* o = out + (size_t)s * n_peaks;
  for (int r = threadIdx.x; r < n_peaks; r += blockDim.x) o[r] = -1;
  for (int r = 0; r < n_peaks; ++r) {
    float best = 0.f;
    int bidx = 0x7fffffff;
    for (int k = threadIdx.x; k < nf; k += blockDim.x) {
      bool ex = false;
      for (int i = 0; i < r; ++i) ex |= (k >= s_lo[i] && k <= s_hi[i]);
      if (ex) continue;
      const float x = v[k];
      if (bidx == 0x7fffffff || x > best || (x == best && k < bidx)) { best = x; bidx = k; }
    }
    for (int off = 16; off > 0; off >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, best, off);
      const int oi = __shfl_xor_sync(0xffffffffu, bidx, off);
      if (oi != 0x7fffffff && (bidx == 0x7fffffff || ov > best || (ov == best && oi < bidx))) {
        best = ov;
        bidx = oi;
      }
    }
    if ((threadIdx.x & 31) == 0) { bv[threadIdx.x >> 5] = best; bi[threadIdx.x >> 5] = bidx; }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; ++w)
        if (bi[w] != 0x7fffffff && (bidx == 0x7fffffff || bv[w] > best || (bv[w] == best && bi[w] < bidx))) {
          best = bv[w];
          bidx = bi[w];
        }
      s_pick = bidx;
      if (bidx != 0x7fffffff) {
        o[r] = bidx;
        const double fp = f[bidx].x;
        int a = 0, b = bidx;  // first index near the pick
        while (a < b) {
          const int m = (a + b) >> 1;
          if (near_pick(f[m].x, fp, sep)) b = m; else a = m + 1;
        }
        s_lo[r] = a;
        a = bidx;
        b = nf - 1;  // last index near the pick
        while (a < b) {
          const int m = (a + b + 1) >> 1;
          if (near_pick(f[m].x, fp, sep)) a = m; else b = m - 1;
        }
        s_hi[r] = a;
      }
    }
    __syncthreads();
    if (s_pick == 0x7fffffff) break;
  }
}

int launch_peaks(const StarDev* stars, int n_stars, const double2* fq, const float* snr, int n_peaks, double sep,
                 int32_t* out, void* stream) {
  if (n_stars <= 0) return 0;
  if (n_peaks < 1 || n_peaks > kMaxPeaks) return (int)cudaErrorInvalidValue;
  peaks_kernel<<<n_stars, 256, 0, (cudaStream_t)stream>>>(stars, fq, snr, n_peaks, sep, out);
  return (int)cudaGetLastError();
}

int launch_snr(const SnrArgs& in, void* stream) {
  if (in.n_stars <= 0) return 0;
  SnrArgs a = in;
  a.max_sturges = a.max_sturges < kMaxSturges ? (a.max_sturges > 1 ? a.max_sturges : 1) : kMaxSturges;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const bool few = a.n_stars < sms;
  const int cap = few ? kSnrKeysFew : kSnrKeys;
  a.key_cap = a.max_nf < cap ? a.max_nf : cap;
  // every bin and the whole spectrum
  const size_t smem = snr_smem(a.max_sturges + 1, a.key_cap);
  auto kern = few ? snr_kernel<1024> : snr_kernel<512>;
  // The attribute belongs to the kernel, not to the launch: it is set to the largest size
  // always, so that another host thread with a smaller plan cannot lower it in between.
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)snr_smem(kMaxSturges + 1, cap));
  if (e != cudaSuccess) return (int)e;
  kern<<<a.n_stars, few ? 1024 : 512, smem, (cudaStream_t)stream>>>(a);
  return (int)cudaGetLastError();
}

}  // namespace qlp
