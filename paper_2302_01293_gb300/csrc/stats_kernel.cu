// Post-BLS statistics of each star's best candidate (Sec. 2.2 items 2-5 of
// arXiv:2302.01293), one CTA per star, FP64:
//  * trapezoid model y = z - delta s(a), a = distance from the nearest
//    mid-transit time (period fixed to the BLS period), s = 1 on the flat
//    bottom a <= D/2 - q_in D, linear to 0 at a = D/2, 0 outside (D = q P);
//  * fit of (T0, delta, q, q_in, z) by Levenberg-Marquardt on the points within
//    two BLS durations of the transit centre (weights dy^-2), bounds
//    1e-6 <= q <= 1, 1e-3 <= q_in <= 0.5, start from the BLS box (q_in = 0.1,
//    z = weighted mean of the window outside the box): solve
//    (A + lam diag(max(A_ii, 1e-12 max A_jj))) h = J^T r (A = J^T J) by Gaussian
//    elimination with partial pivoting, clip to the bounds, accept when chi^2
//    falls (lam / 10) else lam x 10; stop after an accepted step with a relative
//    decrease below 1e-10 or lam > 1e10 (converged), or after 100 iterations;
//  * residuals of the fitted model over all points: sigma_w = RMS; sigma_r from
//    the residuals averaged in time bins of one fitted duration,
//    sigma_r^2 = max(0, mean square of the bin averages - sigma_w^2 / mean points
//    per occupied bin);
//  * S/N_pink = delta (1 - q_in) / sqrt(sigma_w^2 / n_in + sigma_r^2 / N_t)
//    (Eq. 2 with the depth replaced by the trapezoid's mean depth), n_in points
//    with a < D/2, N_t transits with a point at a <= D/2; points before
//    (-2D <= dt < -D/2) and after (D/2 < dt <= 2D) transit;
//  * detected = N_t >= 2 and S/N_pink > 9 and S/N > 9.
// The model's region decisions use explicitly rounded FP64 operations (no
// contraction), in the order the definition states them; the quotients they
// round down (the nearest transit index, the residual time bin) come from a
// reciprocal and fall back to the exact division wherever the two could round
// differently. Point sums are taken per thread over contiguous index ranges and
// combined in a fixed order, so the results do not depend on scheduling.
//
// GB300 executes FP64 at 1/64 of the FP32 rate, so the cost of this kernel is its
// count of FP64 operations per point: the fit's pass over a flat-bottom or
// outside point takes eight (the point's phase, residual and five sums; the
// weight 1/dy^2 and the (z, z) curvature, the sum of all weights, are taken once),
// and region tests compare FP64 bit patterns on the integer pipe. A warp issues an FP64
// instruction every 64 cycles at best, an SM one every 19, so a long fit left alone on an
// SM wants several warps: a star has four, or two in large batches (launch_stats). What is
// taken point by point (phases, weights, residuals, time bins) goes over the points 32 at a
// time, so that a warp's points share their nearest transit and equal errors their divisions;
// what is summed keeps 64 chains of contiguous points, each in order, whatever the warps do.
// The time is that of a batch's longest fits: 100 stars 14.9 -> 10.7 ms (another draw 10.3 ->
// 7.3), 1,000 stars 14.2 -> 10.1 (19.2 -> 12.2), 2,500 stars 24.5 -> 18.8 (26.7 -> 21.3),
// against two warps a star for all of it. With four warps three CTAs per SM (168 registers, 60
// bytes of them spilled) beat four, which spill far more: 12.3 against 14.2 ms on 1,000 stars.
#include <cuda_runtime.h>

#include <cstdint>

#include "qlp_internal.h"

namespace qlp {

namespace {

constexpr int kChains = 64;                // ordered partial sums of a star: contiguous ranges of its points
constexpr int kChainWarps = kChains / 32;  // warp g < kChainWarps owns chains 32 g .. 32 g + 31
constexpr int kEnt = 8;                    // addends of a chain per buffer between two warps
constexpr int kRampBuf = 64;  // queued ramp points per warp (a batch of 32 is taken at 32)
constexpr int kSums = 21;  // chi^2, g[5], A upper triangle [15]
constexpr double kQinMin = 1e-3, kQMin = 1e-6, kQinInit = 0.1;
constexpr double kLam0 = 1e-3, kRtol = 1e-10, kLamMax = 1e10;
constexpr int kMaxIt = 100;

// |v| of a double as its bit pattern: for non-negative doubles the order of the
// patterns (as integers) is the order of the values
__device__ __forceinline__ long long mag(double v) { return __double_as_longlong(v) & 0x7fffffffffffffffll; }

// floor(fl(fl(num / den) + add)), add = 0.5 (HALF) or 0, from rden = fl(1 / den).
// fl(num rden) lies within 3 2^-53 |num / den| of fl(num / den); below 2^20 in
// magnitude that is under 2^-31, and with the rounding of the sum the two floors
// agree unless the sum lies within 2^-30 of an integer. There, and for larger
// quotients, the quotient is taken exactly.
template <bool HALF>
__device__ __forceinline__ double floor_quot(double num, double den, double rden) {
  const double q = __dmul_rn(num, rden);
  const double b = HALF ? __dadd_rn(q, 0.5) : q;
  const double nn = floor(b);
  const double fr = __dsub_rn(b, nn);  // in [0, 1), accurate to 2^-53
  // the comparisons by bit patterns (fr >= 0, or NaN, whose pattern is the largest)
  const unsigned long long fb = (unsigned long long)__double_as_longlong(fr);
  if (fb > 0x3e10000000000000ull && fb < 0x3feffffff8000000ull && mag(b) < 0x4130000000000000ll) return nn;
  const double qe = __ddiv_rn(num, den);
  return floor(HALF ? __dadd_rn(qe, 0.5) : qe);
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the chains of n values per chain thread (n <= kSums) into tot[0 .. n-1] in shared
// memory (warp sums, then one thread per value adds the chain warps' partials in order).
// Called by every thread of the block.
__device__ __forceinline__ void block_sums(const double* v, int n, double (*red)[kSums], double* tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < kChainWarps)
    for (int i = 0; i < n; ++i) {
      const double w = warp_sum(v[i]);
      if (lane == 0) red[warp][i] = w;
    }
  __syncthreads();
  if (threadIdx.x < n) {
    double t = 0.0;
    for (int w = 0; w < kChainWarps; ++w) t += red[w][threadIdx.x];
    tot[threadIdx.x] = t;
  }
  __syncthreads();
}

// Named barriers between the two warps of a chain group (64 threads)
__device__ __forceinline__ void pair_sync(int id) { 
  __syncwarp();
  asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}
__device__ __forceinline__ void pair_arrive(int id) { 
  __syncwarp();
  asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory");
}

// The nearest transit of consecutive points: the last one's fl(P nn) serves while |u - fl(P
// nn)| < (1 - 2^-20) P / 2. With |nn| < 2^20 every rounding on the way to floor(fl(fl(u / P)
// + 0.5)) is below 2^-32, so that floor is nn there; else it is taken anew.
struct Nearest {
  double period, r_period;
  long long safe;
  double nn, pn;
  double last;  // fl(P nn) of the last call
  __device__ __forceinline__ Nearest(double p, double rp) {
    period = p;
    r_period = rp;
    safe = mag(__dmul_rn(__dmul_rn(0.5, p), 1.0 - 0x1p-20));
    nn = last = 0.0;
    pn = __longlong_as_double(0x7ff8000000000000ll);
  }
  // u - P nn for the nearest transit nn
  __device__ __forceinline__ double operator()(double u) {
    double d = __dsub_rn(u, pn);
    if (mag(d) >= safe) {  // also when pn is NaN (none yet, or |nn| too large to be kept)
      nn = floor_quot<true>(u, period, r_period);
      pn = __dmul_rn(period, nn);
      d = __dsub_rn(u, pn);
      last = pn;
      if (mag(nn) >= 0x4130000000000000ll) pn = __longlong_as_double(0x7ff8000000000000ll);
    } else {
      last = pn;
    }
    return d;
  }
};

__device__ __forceinline__ void clip(double* x) {
  x[2] = fmin(fmax(x[2], kQMin), 1.0);
  x[3] = fmin(fmax(x[3], kQinMin), 0.5);
}

__device__ __forceinline__ double shfl_d(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// Gaussian elimination with partial pivoting of the 5 x 5 system m h = b by one warp;
// false if singular. Lane 6 r + j holds entry (r, j) of the augmented matrix [m | b]
// (lanes 30 and 31 repeat lanes 24 and 25). Every entry goes through the same
// operations in the same order as in the serial elimination (pivot: the first row of
// the largest |m[r][c]|; m[r][j] -= (m[r][c] / m[c][c]) m[c][j]), and the back
// substitution runs in that order on every lane, so h is the serial result. The
// warp issues each step once for all entries: on GB300 a single thread's FP64
// instruction takes the pipe as long as a full warp's.
__device__ bool solve5_warp(double v, int r, int j, double* h) {
  for (int c = 0; c < 5; ++c) {
    int p = c;
    double best = shfl_d(v, 6 * c + c);
    for (int rr = c + 1; rr < 5; ++rr) {
      const double o = shfl_d(v, 6 * rr + c);
      if (fabs(o) > fabs(best)) {
        best = o;
        p = rr;
      }
    }
    if (best == 0.0) return false;
    const double vc = shfl_d(v, 6 * c + j), vp = shfl_d(v, 6 * p + j);
    if (r == c) v = vp;
    else if (r == p) v = vc;
    const double piv = shfl_d(v, 6 * c + c);
    const double rc = shfl_d(v, 6 * r + c);
    const double cj = shfl_d(v, 6 * c + j);
    if (r > c && j >= c) v = __dsub_rn(v, __dmul_rn(__ddiv_rn(rc, piv), cj));
  }
  double u[5][6];
#pragma unroll
  for (int rr = 0; rr < 5; ++rr)
#pragma unroll
    for (int jj = rr; jj < 6; ++jj) u[rr][jj] = shfl_d(v, 6 * rr + jj);
#pragma unroll
  for (int c = 4; c >= 0; --c) {
    double acc = u[c][5];
#pragma unroll
    for (int jj = c + 1; jj < 5; ++jj) acc = __dsub_rn(acc, __dmul_rn(u[c][jj], h[jj]));
    h[c] = __ddiv_rn(acc, u[c][c]);
  }
  return true;
}

}  // namespace

// Launch order of the statistics CTAs: stars by decreasing estimated fit cost (its
// window holds about 4 q n points), so that the longest fits start first rather
// than trail the launch. Half-octave buckets of q n; the order inside a bucket is
// free (each star's results do not depend on it). One CTA.
constexpr int kOrderBuckets = 64;
__global__ void __launch_bounds__(1024) stats_order_kernel(const StatsArgs a) {
  __shared__ int cnt[kOrderBuckets], pos[kOrderBuckets];
  if (threadIdx.x < kOrderBuckets) cnt[threadIdx.x] = 0;
  __syncthreads();
  auto bucket = [&](int s) {
    const double key = a.best[s].f_idx >= 0 ? a.best[s].q * (double)a.stars[s].n_pts : 0.0;
    const int e = key > 1.0 ? min((int)(2.0 * log2(key)), kOrderBuckets - 1) : 0;
    return kOrderBuckets - 1 - e;  // the largest first
  };
  for (int s = threadIdx.x; s < a.n_stars; s += blockDim.x) atomicAdd(&cnt[bucket(s)], 1);
  __syncthreads();
  if (threadIdx.x == 0) {
    int run = 0;
    for (int k = 0; k < kOrderBuckets; ++k) {
      pos[k] = run;
      run += cnt[k];
    }
  }
  __syncthreads();
  for (int s = threadIdx.x; s < a.n_stars; s += blockDim.x) a.order[atomicAdd(&pos[bucket(s)], 1)] = s;
}

// THREADS 128: two warps share a group of 32 chains; 64: one (launch_stats chooses).
template <int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 128 ? 3 : 6) stats_kernel(const StatsArgs a) {
  constexpr int kThreads = THREADS, kWarps = kThreads / 32;
  constexpr bool kPairs = kWarps > kChainWarps;
  __shared__ double red[kChainWarps][kSums];
  __shared__ double s_part[kChains][kSums + 1];  // per-chain sums of the fit's pass
  __shared__ double s_q[kChainWarps][kSums];
  __shared__ int s_ramp[kChainWarps][kRampBuf];
  // addends on their way to the summing warp (pairs), later the merged runs of the binned residuals
  __shared__ double s_ent[kPairs ? kChainWarps : 1][2][kPairs ? kEnt : 4][2][32];
  __shared__ int s_ne[kChainWarps][2];                   // how many; bit 8: the pass's last; bit 16 + j: the j-th are ramp points
  __shared__ double s_tot[kSums];  // block totals of the last reduction
  __shared__ double s_cur[kSums];  // chi^2, g, A at the accepted parameters (warp 0)
  __shared__ double s_x[5];
  __shared__ double s_fac[3];      // 1 / t_in, d(-delta s)/dq per unit a, delta / q_in
  __shared__ double s_lam;         // the damping (warp 0)
  __shared__ double s_wsum;        // sum of the window points' weights 1/dy^2
  __shared__ int s_go, s_ok;
  __shared__ int s_cnt[kChains + 1];  // window points before each chain's range
  __shared__ int s_wcnt[kWarps];
  // run partials for the binned residuals and the transit count (bins as the bit
  // patterns of their non-negative FP64 indices)
  __shared__ long long s_hbin[kChains], s_tbin[kChains], s_kf[kWarps], s_kl[kWarps];
  __shared__ double s_hsum[kChains], s_tsum[kChains];
  __shared__ int s_hcnt[kChains], s_tcnt[kChains], s_runs[kChains], s_kd[kWarps], s_n3[kWarps][3];

  const int s = a.order ? a.order[blockIdx.x] : (int)blockIdx.x;
  const int tid = threadIdx.x;
  const StarDev st = a.stars[s];
  const qlp_bls_best bb = a.best[s];
  qlp_bls_cand_stats* out = a.out + s;
  const int n = st.n_pts;
  if (bb.f_idx < 0 || n <= 0) {
    if (tid == 0) {
      *out = qlp_bls_cand_stats{};
      out->status = QLP_STATS_NO_CANDIDATE;
    }
    return;
  }
  const double* tp = a.tp + st.pt_off;
  const double* yv = a.y + st.pt_off;
  const double* dyv = a.dy + st.pt_off;
  WinRec* wrec = a.wrec + st.pt_off;
  const double period = bb.period;
  const double r_period = 1.0 / period;
  const double t0p = __dsub_rn(bb.t0, st.t_ref);
  const double q0 = bb.q;
  const long long lim_b = mag(__dmul_rn(2.0, __dmul_rn(q0, period)));
  const long long half0_b = mag(__dmul_rn(0.5, __dmul_rn(q0, period)));
  const int lane = tid & 31, warp = tid >> 5;
  const bool chain = tid < kChains;  // thread tid takes chain tid's sums
  const int seg = (n + kChains - 1) / kChains;
  const int i0 = min(n, tid * seg), i1 = chain ? min(n, i0 + seg) : i0;
  // what is taken point by point goes over the points in order, 32 at a time, each warp a
  // contiguous part
  const int per = ((n + kThreads - 1) / kThreads) * 32;
  const int p0 = min(n, warp * per), p1 = min(n, p0 + per);
  // 1. the fit window (ordered compaction): its points per warp and before each chain's range
  {
    Nearest near(period, r_period);
    int run = 0;
    for (int b = p0; b < p1; b += 32) {
      const int i = b + lane;
      bool in = false;
      if (i < p1) in = mag(near(__dsub_rn(tp[i], t0p))) <= lim_b;
      const unsigned mk = __ballot_sync(0xffffffffu, in);
      if (i < p1) {
        const unsigned c = (unsigned)i / (unsigned)seg;
        if (c * (unsigned)seg == (unsigned)i) s_cnt[c] = run + __popc(mk & ((1u << lane) - 1u));
      }
      run += __popc(mk);
    }
    if (lane == 0) s_wcnt[warp] = run;
  }
  __syncthreads();
  int nwin = 0, wbase = 0;
  for (int w = 0; w < kWarps; ++w) {
    if (w == warp) wbase = nwin;
    nwin += s_wcnt[w];
  }
  for (int ch = tid; ch <= kChains; ch += kThreads) {
    const long long at = (long long)ch * seg;  // the chain's first point
    int c = nwin;
    if (at < n) {
      c = s_cnt[ch];
      const int owner = (int)at / per;
      for (int w = 0; w < owner; ++w) c += s_wcnt[w];
    }
    s_cnt[ch] = c;
  }
  // the records: t', y, w and, until the level is known, 1 / (dy dy) in place of pn, its
  // sign set outside the box. Equal errors in a row share their divisions.
  {
    Nearest near(period, r_period);
    int run = wbase;
    double dy_c = __longlong_as_double(0x7ff8000000000000ll), w = 0.0, w2 = 0.0;
    for (int b = p0; b < p1; b += 32) {
      const int i = b + lane;
      long long db = lim_b + 1;
      double t = 0.0;
      if (i < p1) {
        t = tp[i];
        db = mag(near(__dsub_rn(t, t0p)));
      }
      const bool in = db <= lim_b;
      const unsigned mk = __ballot_sync(0xffffffffu, in);
      if (in) {
        const double dy = dyv[i];
        if (__double_as_longlong(dy) != __double_as_longlong(dy_c)) {
          const double inv = __ddiv_rn(1.0, dy);
          w = __dmul_rn(inv, inv);  // the (z, z) term of J^T J, as its product
          w2 = __ddiv_rn(1.0, __dmul_rn(dy, dy));
          dy_c = dy;
        }
        const long long out_bit = db > half0_b ? (long long)0x8000000000000000ull : 0ll;
        wrec[run + __popc(mk & ((1u << lane) - 1u))] =
            WinRec{t, __longlong_as_double(__double_as_longlong(w2) | out_bit), yv[i], w};
      }
      run += __popc(mk);
    }
  }
  __syncthreads();
  // the initial out-of-transit level (the whole window's when no point is out of transit)
  double v[2] = {0.0, 0.0}, ws = 0.0;
  const int c0 = chain ? s_cnt[tid] : 0, c1 = chain ? s_cnt[tid + 1] : 0;
#pragma unroll 4
  for (int k = c0; k < c1; ++k) {
    const WinRec pt = wrec[k];
    if (__double_as_longlong(pt.pn) < 0) {
      const double w2 = fabs(pt.pn);
      v[0] = __dadd_rn(v[0], __dmul_rn(w2, pt.y));
      v[1] = __dadd_rn(v[1], w2);
    }
    ws = __dadd_rn(ws, pt.w);
  }
  block_sums(&ws, 1, red, &s_wsum);
  block_sums(v, 2, red, s_tot);
  if (!(s_tot[1] > 0.0)) {  // block-uniform
    __syncthreads();
    v[0] = v[1] = 0.0;
    for (int k = c0; k < c1; ++k) {
      const WinRec pt = wrec[k];
      const double w2 = fabs(pt.pn);
      v[0] = __dadd_rn(v[0], __dmul_rn(w2, pt.y));
      v[1] = __dadd_rn(v[1], w2);
    }
    block_sums(v, 2, red, s_tot);
  }
  if (nwin < 6) {
    if (tid == 0) {
      *out = qlp_bls_cand_stats{};
      out->status = QLP_STATS_FEW_POINTS;
      out->n_fit = nwin;
    }
    return;
  }
  if (tid == 0) {
    s_x[0] = t0p;
    s_x[1] = bb.depth;
    s_x[2] = q0;
    s_x[3] = kQinInit;
    s_x[4] = s_tot[0] / s_tot[1];
    clip(s_x);
  }
  {  // each record's nearest transit
    Nearest near(period, r_period);
    const int wper = ((nwin + kThreads - 1) / kThreads) * 32;
    const int k1 = min(nwin, (warp + 1) * wper);
    for (int k = warp * wper + lane; k < k1; k += 32) {
      near(__dsub_rn(wrec[k].t, t0p));
      wrec[k].pn = near.last;
    }
  }
  __syncthreads();

  // 2. Levenberg-Marquardt (thread 0 keeps the state; every pass is block-wide)
  const int wseg = (nwin + kChains - 1) / kChains;
  const int grp = warp % kChainWarps;  // the warp's chains: 32 grp + lane
  const int ct = 32 * grp + lane;
  const int w0 = min(nwin, ct * wseg), w1 = min(nwin, w0 + wseg);
  // The model at s_x and its derivatives. Only points on a ramp have nonzero
  // derivatives in T0, q and q_in; flat-bottom points add to the (delta, z) block
  // and outside points to z alone, in place. Ramp points are queued per warp and
  // taken 32 at a time by all lanes, so that the long ramp branch runs once per 32
  // ramp points instead of whenever one lane meets one; its divisions are
  // multiplications by reciprocals taken once per evaluation. The region
  // decisions keep the FP64 expressions of the model's definition.
  //
  // On a ramp every derivative is 1/dy times a factor: phi = (c0 sg, -s, r_q a,
  // r_qin s, 1) with sg = sign(dt), c0 = -delta / t_in, r_q = -delta / (q_in q^2 P)
  // and r_qin = delta / q_in, so J^T J and J^T r over the ramp points follow from
  // nine weighted sums of 1, sg, s, a and their products and three of r / dy times
  // sg, s, a; the factors c0, r_q, r_qin multiply the block totals once.
  enum { kChi, kG4, kWeF, kWF, kGsg, kGs, kGa, kRw, kRsg, kRsgs, kRsga, kRss, kRsa, kRs, kRaa, kRa, kAcc };
  //
  // Pairs: two warps share a group of 32 chains: the first (a) takes the points' phases and the
  // ramps' own sums, the second (b) the other residuals, chi^2, g4 and the flat bottom's
  // sums, fed through shared memory, 8 points a chain at a time, in the order they come
  // (weight 0: nothing to add). A warp issues an FP64 instruction every 64
  // cycles at best, an SM one every 19, so one warp per 32 chains leaves a long fit alone on
  // an SM at half of its rate. Else one warp does both, each addend as it comes.
  int* rl = s_ramp[grp];
  const int bar = 1 + 4 * grp;  // named barriers: + buffer: filled, + 2 + buffer: emptied
  auto evaluate = [&]() {  // at s_x: chi^2, J^T r, J^T J into s_tot
    double x[5];
    for (int i = 0; i < 5; ++i) x[i] = s_x[i];
    const double d = __dmul_rn(x[2], period);
    const double t_in = __dmul_rn(x[3], d);
    if (warp == (kPairs ? kChainWarps : 0)) {  // the totals' factors: one division on three lanes
      const double den = lane == 1 ? __dmul_rn(__dmul_rn(__dmul_rn(x[3], x[2]), x[2]), period) : (lane == 0 ? t_in : x[3]);
      const double q = __ddiv_rn(lane == 1 ? -x[1] : (lane == 0 ? 1.0 : x[1]), den);
      if (lane < 3) s_fac[lane] = q;
    }
    const double m_flat = __dsub_rn(x[4], x[1]);  // the model on the flat bottom
    double chi = 0.0, g4 = 0.0, wef = 0.0, wfl = 0.0;
    const auto take = [&](double a, double w) {  // (y, +-w), w < 0 on the flat bottom
      const bool flat = __double_as_longlong(w) < 0;  // dm/ddelta = -s, dm/dz = 1
      const double wa = fabs(w);
      const double e = mag(w) == 0 ? 0.0 : __dsub_rn(a, flat ? m_flat : x[4]);
      const double we = __dmul_rn(wa, e);  // r / dy with r = e / dy
      chi = __fma_rn(we, e, chi);          // r^2
      g4 = __dadd_rn(g4, we);              // g4 = sum r / dy
      // -g1 over the flat bottom; A11 and -A14 there. No lane on it: only zeros to add
      if (__any_sync(0xffffffffu, flat)) {
        wef = __dadd_rn(wef, flat ? we : 0.0);
        wfl = __dadd_rn(wfl, flat ? wa : 0.0);
      }
    };
    const auto take_ramp = [&](double e, double w) {  // the residual is known, nothing flat
      const double ir = __dmul_rn(w, e);
      chi = __fma_rn(ir, e, chi);
      g4 = __dadd_rn(g4, ir);
    };
    if (warp < kChainWarps) {  // (a)
      double acc[kAcc];
      const double half = __dmul_rn(0.5, d);
      const double edge = __dsub_rn(half, t_in);
      const double hp = __dmul_rn(0.5, period);
      const double r_tin = 1.0 / t_in;
      for (int i = 0; i < kAcc; ++i) acc[i] = 0.0;
      const long long hp_b = mag(hp), edge_b = mag(edge), half_b = mag(half);
      auto dt_of = [&](const WinRec& pt) {
        const double u = __dsub_rn(pt.t, x[0]);
        double dt = __dsub_rn(u, pt.pn);
        if (mag(dt) > hp_b) {  // the epoch moved by half a period: the nearest transit changed
          const double nn = floor_quot<true>(u, period, r_period);
          dt = __dsub_rn(u, __dmul_rn(period, nn));
        }
        return dt;
      };
      int ne = 0, buf = 0, chunk = 0, rm = 0;  // rm: which of the buffer's addends are the ramps'
      auto flush = [&](int last) {
        if (lane == 0) s_ne[grp][buf] = ne | last | rm << 16;
        pair_arrive(bar + buf);
        ++chunk;
        buf ^= 1;
        ne = rm = 0;
        if (chunk >= 2) pair_sync(bar + 2 + buf);  // the chunk before the last has been read
      };
      auto emit = [&](double a, double w) {  // (y, +-w: - on the flat bottom), or a ramp point's (e, w)
        s_ent[grp][buf][ne][0][lane] = a;
        s_ent[grp][buf][ne][1][lane] = w;
        if (++ne == kEnt) flush(0);
      };
      auto ramp_batch = [&](int cnt) {  // lanes < cnt take the queued ramp points rl[lane]
        double e = 0.0, w = 0.0;
        if (lane < cnt) {
          const WinRec pt = wrec[rl[lane]];
          const double dt = dt_of(pt);
          const bool neg = __double_as_longlong(dt) < 0;  // sg = -1 (a ramp point has dt != 0)
          const double aa = fabs(dt);
          const double sv = __dmul_rn(__dsub_rn(half, aa), r_tin);
          e = __dsub_rn(pt.y, __dsub_rn(x[4], __dmul_rn(x[1], sv)));
          w = pt.w;
          const double ir = __dmul_rn(w, e);  // r / dy
          const double wsv = __dmul_rn(w, sv), wa = __dmul_rn(w, aa);
          acc[kGsg] = __dadd_rn(acc[kGsg], neg ? -ir : ir);
          acc[kGs] = __fma_rn(sv, ir, acc[kGs]);
          acc[kGa] = __fma_rn(aa, ir, acc[kGa]);
          acc[kRw] = __dadd_rn(acc[kRw], w);
          acc[kRsg] = __dadd_rn(acc[kRsg], neg ? -w : w);
          acc[kRsgs] = __dadd_rn(acc[kRsgs], neg ? -wsv : wsv);
          acc[kRsga] = __dadd_rn(acc[kRsga], neg ? -wa : wa);
          acc[kRss] = __fma_rn(wsv, sv, acc[kRss]);
          acc[kRsa] = __fma_rn(wsv, aa, acc[kRsa]);
          acc[kRs] = __dadd_rn(acc[kRs], wsv);
          acc[kRaa] = __fma_rn(wa, aa, acc[kRaa]);
          acc[kRa] = __dadd_rn(acc[kRa], wa);
        }
        if constexpr (kPairs) {
          rm |= 1 << ne;
          emit(e, w);
        } else {
          take_ramp(e, w);
        }
      };
      int nr = 0;  // queued ramp points of this warp (warp-uniform)
      // Four points of a chain at a time, so that their latencies overlap (one at a time a
      // pass was held by them: 900 cycles a point), the next four on their way.
      WinRec ahead[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) ahead[u] = wrec[min(w0 + u, nwin - 1)];
      for (int kb = 0; kb < wseg; kb += 4) {  // the same trip count on every lane
        double dt[4], y[4], w[4];
        bool far = false;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          dt[u] = __dsub_rn(__dsub_rn(ahead[u].t, x[0]), ahead[u].pn);
          far = far || mag(dt[u]) > hp_b;
          y[u] = ahead[u].y;
          w[u] = ahead[u].w;
        }
        if (far) {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (mag(dt[u]) > hp_b) dt[u] = dt_of(ahead[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) ahead[u] = wrec[min(w0 + kb + 4 + u, nwin - 1)];
        unsigned mk[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const long long ab = mag(dt[u]);
          const bool on = w0 + kb + u < w1;
          const bool ramp = on && ab > edge_b && ab < half_b;
          mk[u] = __ballot_sync(0xffffffffu, ramp);
          // flat bottom (s = 1) or outside (s = 0); weight 0 for a ramp point or past the chain's
          w[u] = on && !ramp ? (ab <= edge_b ? -w[u] : w[u]) : 0.0;
        }
        const unsigned below = (1u << lane) - 1u;
        const int steps = min(4, wseg - kb);
        if (steps == 4 && (!kPairs || ne <= kEnt - 4) &&
            nr + __popc(mk[0]) + __popc(mk[1]) + __popc(mk[2]) + __popc(mk[3]) < 32) {  // warp-uniform: no batch
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if constexpr (kPairs) {
              s_ent[grp][buf][ne + u][0][lane] = y[u];
              s_ent[grp][buf][ne + u][1][lane] = w[u];
            } else {
              take(y[u], w[u]);
            }
            if ((mk[u] >> lane) & 1u) rl[nr + __popc(mk[u] & below)] = w0 + kb + u;
            nr += __popc(mk[u]);
          }
          if constexpr (kPairs) {
            ne += 4;
            if (ne == kEnt) flush(0);
          }
          continue;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (u >= steps) break;
          if constexpr (kPairs) emit(y[u], w[u]);
          else take(y[u], w[u]);
          if ((mk[u] >> lane) & 1u) rl[nr + __popc(mk[u] & below)] = w0 + kb + u;
          nr += __popc(mk[u]);
          if (nr >= 32) {
            __syncwarp();
            ramp_batch(32);
            const int rest = nr - 32;
            const int moved = lane < rest ? rl[32 + lane] : 0;
            __syncwarp();
            if (lane < rest) rl[lane] = moved;
            __syncwarp();
            nr = rest;
          }
        }
      }
      __syncwarp();
      if (nr > 0) ramp_batch(nr);
      __syncwarp();
      if constexpr (kPairs) flush(0x100);
      for (int i = kGsg; i < kAcc; ++i) s_part[ct][i] = acc[i];
    } else if constexpr (kPairs) {  // (b)
      bool go = true;
      for (int buf = 0; go; buf ^= 1) {  // ends with the chunk marked as the last
        pair_sync(bar + buf);
        const int ne = s_ne[grp][buf];
        const auto& en = s_ent[grp][buf];
        if ((ne >> 16) == 0 && (ne & 0xff) == kEnt) {  // a full buffer without ramp points
          double a[kEnt], w[kEnt];
#pragma unroll
          for (int j = 0; j < kEnt; ++j) {
            a[j] = en[j][0][lane];
            w[j] = en[j][1][lane];
          }
#pragma unroll
          for (int j = 0; j < kEnt; ++j) take(a[j], w[j]);
        } else {
          for (int j = 0; j < (ne & 0xff); ++j) {
            if ((ne >> (16 + j)) & 1) take_ramp(en[j][0][lane], en[j][1][lane]);
            else take(en[j][0][lane], en[j][1][lane]);
          }
        }
        go = (ne & 0x100) == 0;
        if (go) pair_arrive(bar + 2 + buf);
      }
    }
    if (warp >= kWarps - kChainWarps) {  // (b), or the one warp
      s_part[ct][kChi] = chi;
      s_part[ct][kG4] = g4;
      s_part[ct][kWeF] = wef;
      s_part[ct][kWF] = wfl;
    }
    // sums over the chains through shared memory: each thread of the first kAcc x 2 sums one
    // value over 32 chains; then every entry of chi^2, g and A adds the halves of the sums
    // it takes, in order, and applies the factors
    __syncthreads();
    if (tid < kAcc * kChainWarps) {
      const int v = tid % kAcc, qq = tid / kAcc;
      double sum = 0.0;
      for (int r = 0; r < 32; ++r) sum += s_part[32 * qq + r][v];
      s_q[qq][v] = sum;
    }
    __syncthreads();
    if (tid < 32) {
      // entry tid: +- (T(a) + T(b)), or +- F1 F2 T(a), with the factors 0: 1, 1: c0, 2: r_q,
      // 3: r_qin; one instruction stream for all of them
      struct Entry {
        signed char a, b, f1, f2, neg;
      };
      constexpr Entry kEntry[32] = {
          {kChi, -1, 0, 0, 0},                                            // chi^2
          {kGsg, -1, 1, 0, 0}, {kWeF, kGs, 0, 0, 1}, {kGa, -1, 2, 0, 0},  // g0, g1, g2
          {kGs, -1, 3, 0, 0}, {kG4, -1, 0, 0, 0},                         // g3, g4
          {kRw, -1, 1, 1, 0}, {kRsgs, -1, 1, 0, 1}, {kRsga, -1, 1, 2, 0}, // A00, A01, A02
          {kRsgs, -1, 1, 3, 0}, {kRsg, -1, 1, 0, 0},                      // A03, A04
          {kRss, kWF, 0, 0, 0}, {kRsa, -1, 2, 0, 1}, {kRss, -1, 3, 0, 1}, // A11, A12, A13
          {kRs, kWF, 0, 0, 1},                                            // A14
          {kRaa, -1, 2, 2, 0}, {kRsa, -1, 2, 3, 0}, {kRa, -1, 2, 0, 0},   // A22, A23, A24
          {kRss, -1, 3, 3, 0}, {kRs, -1, 3, 0, 0}};                       // A33, A34; A44 is s_wsum
      unsigned ea = 0, eb = 0, ef = 0;  // this lane's entry, without a table in memory
#pragma unroll
      for (int i = 0; i < 20; ++i)
        if (lane == i) {
          ea = (unsigned)kEntry[i].a;
          eb = kEntry[i].b < 0 ? 31u : (unsigned)kEntry[i].b;
          ef = (unsigned)(kEntry[i].f1 | kEntry[i].f2 << 2 | kEntry[i].neg << 4);
        }
      auto T = [&](unsigned v) {
        double sum = 0.0;
        for (int qq = 0; qq < kChainWarps; ++qq) sum += s_q[qq][v];
        return sum;
      };
      const double cc0 = __dmul_rn(-x[1], s_fac[0]), r_q = s_fac[1], r_qin = s_fac[2];
      auto fac = [&](unsigned f) { return f == 0 ? 1.0 : (f == 1 ? cc0 : (f == 2 ? r_q : r_qin)); };
      const double ta = T(ea), tb = T(eb == 31u ? ea : eb);
      const double both = __dadd_rn(ta, tb);
      double v = __dmul_rn(__dmul_rn(fac(ef & 3u), fac((ef >> 2) & 3u)), ta);
      if (eb != 31u) v = both;
      if (ef >> 4) v = -v;
      if (lane == 20) v = s_wsum;  // every window point's weight
      if (lane < kSums) s_tot[lane] = v;
    }
    __syncthreads();
  };
  double xa[5];
  evaluate();
  if (tid < kSums) s_cur[tid] = s_tot[tid];
  if (tid == 0) s_lam = kLam0;
  for (int i = 0; i < 5; ++i) xa[i] = s_x[i];
  __syncthreads();  // warp 0 reads s_cur and s_lam
  int it = 0;
  bool conv = false;
  while (it < kMaxIt) {  // block-uniform: s_ok and s_go decide
    ++it;
    if (tid < 32) {  // warp 0: the damped normal equations and their solution
      // entry (r, j) of [A + lam diag(max(A_kk, 1e-12 max A_jj)) | g] on lane 6 r + j;
      // A's upper triangle is stored row by row after chi^2 and g
      const int r = min(lane / 6, 4), j = lane % 6;
      const int k = min(r, j), l = max(r, j);
      double v = j == 5 ? s_cur[1 + r] : s_cur[6 + 5 * k - k * (k - 1) / 2 + (l - k)];
      double dmax = 0.0;
      for (int kk = 0; kk < 5; ++kk) dmax = fmax(dmax, s_cur[6 + 5 * kk - kk * (kk - 1) / 2]);
      if (r == j) v = __dadd_rn(v, __dmul_rn(s_lam, fmax(v, __dmul_rn(1e-12, dmax))));
      double h[5];
      const bool ok = solve5_warp(v, r, j, h);
      if (tid == 0) {
        if (ok) {
          for (int kk = 0; kk < 5; ++kk) s_x[kk] = __dadd_rn(xa[kk], h[kk]);
          clip(s_x);
        }
        s_ok = ok ? 1 : 0;
      }
    }
    __syncthreads();
    const bool ok = s_ok != 0;
    if (ok) evaluate();
    if (tid < 32) {
      int act = 0;  // 0 continue, 1 stop
      const double cur = s_cur[0], tot = s_tot[0];
      double lam = s_lam;
      if (ok && tot < cur) {
        // the relative decrease and the next damping: one division on two lanes
        const double q = __ddiv_rn(lane == 0 ? __dsub_rn(cur, tot) : lam, lane == 0 ? cur : 10.0);
        const double rel = cur > 0.0 ? shfl_d(q, 0) : 0.0;
        lam = shfl_d(q, 1);
        for (int i = 0; i < 5; ++i) xa[i] = s_x[i];
        __syncwarp();
        if (lane < kSums) s_cur[lane] = s_tot[lane];
        if (rel < kRtol) { conv = true; act = 1; }
      } else {
        lam *= 10.0;
        if (lam > kLamMax) { conv = true; act = 1; }
      }
      __syncwarp();
      if (lane == 0) {
        s_lam = lam;
        for (int i = 0; i < 5; ++i) s_x[i] = xa[i];
        s_go = act;
      }
    }
    __syncthreads();
    if (s_go) break;
  }

  // 3. residuals over every point at the fitted parameters
  double x[5];
  for (int i = 0; i < 5; ++i) x[i] = s_x[i];
  const double D = __dmul_rn(x[2], period);
  const double r_D = 1.0 / D;
  const double hD = __dmul_rn(0.5, D), tD = __dmul_rn(2.0, D);
  const double t_in = __dmul_rn(x[3], D);
  const double edge = __dsub_rn(hD, t_in);
  const double m_flat = __dsub_rn(x[4], x[1]);
  const long long hD_b = mag(hD), tD_b = mag(tD), edge_b = mag(edge);
  // point by point: the residual and its time bin, left in the scratch (the fit's records
  // are no longer read), and the counts
  struct Res {
    double r;
    long long b;
  };
  auto res = [&](int i) { return reinterpret_cast<Res*>(wrec + i); };  // r, bin | closed run's sum, count
  {
    Nearest near(period, r_period);
    int n_in = 0, n_before = 0, n_after = 0, kd = 0;
    long long kf = 0, kl = 0;  // first and last transit index seen (valid when kd > 0)
    for (int b = p0; b < p1; b += 32) {
      const int i = b + lane;
      bool in_tr = false;
      long long k = 0;
      if (i < p1) {
        // the model (Sec. 2.2 item 2) at t'_i: nearest transit, distance, trapezoid
        const double t = tp[i];
        const double dt = near(__dsub_rn(t, x[0]));
        const long long ab = mag(dt);
        const bool neg = __double_as_longlong(dt) < 0;  // sign bit (ab > hD_b excludes -0)
        double m;
        if (ab <= edge_b) m = m_flat;
        else if (ab < hD_b) m = __dsub_rn(x[4], __dmul_rn(x[1], __ddiv_rn(__dsub_rn(hD, fabs(dt)), t_in)));
        else m = x[4];
        n_in += ab < hD_b;
        n_before += neg && ab > hD_b && ab <= tD_b;
        n_after += !neg && ab > hD_b && ab <= tD_b;
        in_tr = ab <= hD_b;
        if (in_tr) k = (long long)near.nn;
        // the residual's time bin floor(t' / D) (t' >= 0: the bit pattern orders and identifies it)
        *res(i) = Res{__dsub_rn(yv[i], m), __double_as_longlong(floor_quot<false>(t, D, r_D))};
      }
      const unsigned mk = __ballot_sync(0xffffffffu, in_tr);
      if (mk) {  // transit indices do not decrease along t: count where they change
        const unsigned below = mk & ((1u << lane) - 1u);
        const long long up = __shfl_sync(0xffffffffu, k, below ? 31 - __clz((int)below) : 0);
        const bool first = in_tr && (below ? k != up : (kd == 0 || k != kl));
        if (kd == 0) kf = __shfl_sync(0xffffffffu, k, __ffs((int)mk) - 1);
        kd += __popc(__ballot_sync(0xffffffffu, first));
        kl = __shfl_sync(0xffffffffu, k, 31 - __clz((int)mk));
      }
    }
    n_in = (int)__reduce_add_sync(0xffffffffu, (unsigned)n_in);
    n_before = (int)__reduce_add_sync(0xffffffffu, (unsigned)n_before);
    n_after = (int)__reduce_add_sync(0xffffffffu, (unsigned)n_after);
    if (lane == 0) {
      s_n3[warp][0] = n_in;
      s_n3[warp][1] = n_before;
      s_n3[warp][2] = n_after;
      s_kf[warp] = kf;
      s_kl[warp] = kl;
      s_kd[warp] = kd;
    }
  }
  __syncthreads();
  // chain by chain: the sum of squares and the runs of equal bin. A closed run's sum and
  // count wait in the chain's records, so that the chains' divisions run side by side.
  double r2 = 0.0, sb2 = 0.0;
  if (chain) {
    int runs = 0;
    long long cbin = -1, hbin = -1;
    double csum = 0.0, hsum = 0.0;
    int ccnt = 0, hcnt = 0;
    bool have_head = false;
    Res ahead[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) ahead[u] = *res(min(i0 + u, n - 1));
    for (int ib = i0; ib < i1; ib += 4)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = ib + u;
      if (i >= i1) break;
      const Res cu = ahead[u];
      ahead[u] = *res(min(i + 4, n - 1));
      r2 = __fma_rn(cu.r, cu.r, r2);
      if (ccnt > 0 && cu.b != cbin) {  // close the current run
        if (!have_head) { have_head = true; hbin = cbin; hsum = csum; hcnt = ccnt; }
        else { res(i0 + runs)[1] = Res{csum, ccnt}; ++runs; }
        ccnt = 0;
        csum = 0.0;
      }
      cbin = cu.b;
      csum = __dadd_rn(csum, cu.r);
      ++ccnt;
    }
    for (int k = 0; k < runs; ++k) {
      const Res cl = res(i0 + k)[1];
      const double mu = __ddiv_rn(cl.r, (double)(int)cl.b);
      sb2 = __fma_rn(mu, mu, sb2);
    }
    s_hbin[tid] = have_head ? hbin : cbin;
    s_hsum[tid] = have_head ? hsum : csum;
    s_hcnt[tid] = have_head ? hcnt : ccnt;
    s_tbin[tid] = have_head ? cbin : -1;  // the last run when it differs from the head
    s_tsum[tid] = have_head ? csum : 0.0;
    s_tcnt[tid] = have_head ? ccnt : 0;
    s_runs[tid] = runs;
  }
  const double part[2] = {r2, sb2};
  block_sums(part, 2, red, s_tot);
  // merge the run partials in thread order: thread 0 joins them, the block divides
  double* m_sum = &s_ent[0][0][0][0][0];  // at most two runs per chain
  double* m_cnt = m_sum + 2 * kChains;
  static_assert(sizeof(s_ent) >= 4 * kChains * sizeof(double), "the merged runs reuse the addends' buffers");
  if (tid == 0) {
    int nm = 0;
    long long carry_bin = -1;
    double carry_sum = 0.0;
    int carry_cnt = 0;
    auto flush = [&]() {
      if (carry_cnt > 0) {
        m_sum[nm] = carry_sum;
        m_cnt[nm++] = (double)carry_cnt;
      }
      carry_cnt = 0;
      carry_sum = 0.0;
    };
    for (int t = 0; t < kChains; ++t) {
      if (s_hcnt[t] == 0) continue;  // no points
      if (carry_cnt > 0 && s_hbin[t] == carry_bin) { carry_sum += s_hsum[t]; carry_cnt += s_hcnt[t]; }
      else { flush(); carry_bin = s_hbin[t]; carry_sum = s_hsum[t]; carry_cnt = s_hcnt[t]; }
      if (s_tcnt[t] > 0) { flush(); carry_bin = s_tbin[t]; carry_sum = s_tsum[t]; carry_cnt = s_tcnt[t]; }
    }
    flush();
    s_go = nm;
  }
  __syncthreads();
  for (int i = tid; i < s_go; i += kThreads) m_sum[i] = __ddiv_rn(m_sum[i], m_cnt[i]);  // at most 2 kChains
  __syncthreads();
  if (tid == 0) {
    int cn[3] = {0, 0, 0};
    for (int w = 0; w < kWarps; ++w)
      for (int i = 0; i < 3; ++i) cn[i] += s_n3[w][i];
    double sbm = s_tot[1];
    long long nb_occ = s_go;
    for (int t = 0; t < kChains; ++t) nb_occ += s_runs[t];
    for (int t = 0; t < s_go; ++t) sbm = __fma_rn(m_sum[t], m_sum[t], sbm);
    // transits: distinct indices over the warps' parts, adjacent duplicates removed
    int nt = 0;
    long long last = -1;
    bool have = false;
    for (int t = 0; t < kWarps; ++t) {
      if (s_kd[t] == 0) continue;
      nt += s_kd[t];
      if (have && s_kf[t] == last) --nt;
      last = s_kl[t];
      have = true;
    }
    const double sw = sqrt(s_tot[0] / n);
    const double nb_mean = (double)n / (double)nb_occ;
    const double sb2m = sbm / (double)nb_occ;
    const double sr = sqrt(fmax(0.0, sb2m - sw * sw / nb_mean));
    const int n_in_t = cn[0];
    const double depth_mean = x[1] * (1.0 - x[3]);
    const double den = (n_in_t ? sw * sw / n_in_t : 0.0) + (nt ? sr * sr / nt : 0.0);
    qlp_bls_cand_stats o{};
    o.t0 = x[0] + st.t_ref;
    o.depth = x[1];
    o.q = x[2];
    o.q_in = x[3];
    o.z = x[4];
    o.chi2 = s_cur[0];
    o.sigma_w = sw;
    o.sigma_r = sr;
    o.depth_mean = depth_mean;
    o.snr_pink = (n_in_t && nt && den > 0.0) ? depth_mean / sqrt(den) : 0.0;
    o.n_fit = nwin;
    o.n_in = n_in_t;
    o.n_before = cn[1];
    o.n_after = cn[2];
    o.n_transits = nt;
    o.iterations = it;
    o.status = conv ? QLP_STATS_OK : QLP_STATS_NOT_CONVERGED;
    o.detected = (nt >= 2 && o.snr_pink > 9.0 && bb.snr > 9.0) ? 1 : 0;
    *out = o;
  }
}

int launch_stats(const StatsArgs& a, void* stream) {
  if (a.n_stars <= 0) return 0;
  if (a.order) stats_order_kernel<<<1, 1024, 0, (cudaStream_t)stream>>>(a);
  // Pairs of warps while the end of the launch is that of its longest fits, which a pair takes at
  // up to twice the rate. With many stars the FP64 pipe sets the time, and 12 independent warps an
  // SM keep it busier than 6 pairs; short windows (a few points a chain) have little to share.
  // Pairs, one warp per 32 chains: stars of 10,400 points 10.2, 13.3 ms (912 stars), 16.8, 21.7
  // (2,048), 31.7, 29.5 (5,000), 50.5, 46.6 (8,192); of 2,200 points 4.0, 5.0 (2,000), 6.9, 5.8
  // (4,000); of 1,100 points 1.80, 1.84 (1,000), 3.1, 2.7 (2,000), 5.5, 4.5 (4,000).
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int per_sm = a.n_pts >= (int64_t)2000 * a.n_stars ? 26 : 8;
  if (a.n_stars < per_sm * sms) stats_kernel<128><<<a.n_stars, 128, 0, (cudaStream_t)stream>>>(a);
  else stats_kernel<64><<<a.n_stars, 64, 0, (cudaStream_t)stream>>>(a);
  return (int)cudaGetLastError();
}

}  // namespace qlp
