// Exact cell path of the BLS search (sm_103a): integer prefix sums at the bin
// edges, accumulated per phase bin in registers, and a streaming box sweep.
//
// Notation as in cells_kernels.cu: a trial frequency f with nbins bins has its
// phase-bin edges at tau_G = G D, D = 1/(f nbins), G = 0 .. g_end, and with the
// prefix sums C(tau) of (w, w d) over the points before tau every histogram bin
// of Sec. 2.1's BLS is a sum of differences C(tau_{G+1}) - C(tau_G) over the
// cycles. Here the weights are integers, w_int = round(w 2^kw) and
// y_int = round(w d 2^ky) (kw, ky per star), so every C is an exact 64-bit
// integer and the differences telescope: with
//     S[b] = sum over G = b (mod nbins), 0 <= G <= g_end, of C(tau_G)
// the cumulative histogram U[x] = sum_{b < x} H[b mod nbins] is
//     U[x] = S[x mod nbins] + ([b* < x mod nbins] + floor(x / nbins)) C_end
// up to a constant, where b* = g_end mod nbins and C_end = C(tau_{g_end}) is
// the star's total, and the box of m bins starting at bin k sums to
// U[k + m] - U[k]. So a lane owns one bin b, walks its edges b, b + nbins, ...
// (one per cycle) and adds C(tau_G) to a register: no histogram in shared
// memory, no atomics, no exchange between lanes, and the result does not depend
// on the order of the additions.
//
// K0x freq_rec_kernel (plan time): one FreqRec per trial frequency (bins, the
// edge step in 2^-40 cells, guard band, last edge, the box widths present and
// the lowest duration index of each).
// K1x prep_fixed_kernel (1 CTA per exact-path star): weights and the weighted
// mean in FP64 as the other prep kernels, the integer weights, their exact
// prefix sums and the per-cell tables (offset of the cell's point, prefix sums at
// the cell start as a 64-bit group base plus a 32-bit local part; the local part
// of w d carries a bias of 2^30, so that both local parts are non-negative and
// widen to 64 bits with a zero high word; the sums take the bias off once).
// K2x cells_fixed_kernel: persistent; work queue of (star, frequency chunk); the
// star's table in shared memory (three contiguous arrays, staged by bulk
// asynchronous copies on an mbarrier); warps take the item's frequencies one at a time.
// Per frequency the lanes' S values (lane = bin, 32 at a time) go to the warp's row in
// global memory; then, 64 bins at a time (two a lane), the exact differences H[x] = U[x +
// 1] - U[x] are scaled to FP32 (w, w d) pairs and written to a per-warp ring of 128 bins
// (bin x at x mod 128), and the boxes that start in the 64 bins before are swept.
// Stars whose table does not fit in shared memory take their edges window by window into a
// global workspace first (windowed_item), in a launch of their own.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "bls_device.cuh"
#include "qlp_internal.h"

namespace qlp {

constexpr int kRing = 128;  // float2 per warp: H of the last four blocks of 32 bins, at (bin mod 128)
constexpr long long kLocBias = 1ll << 30;  // added to the w d local parts of the cell table
constexpr uint32_t kHiBias = 1u << 15;  // added to the w d group sums of a window, in units of 2^31
constexpr long long kNarrowBias = 1ll << 31;  // added to the w d prefix sums of the 32-bit table
constexpr double kNarrowF = 4294836224.0;     // 2^32 - 2^17: the w scale of the 32-bit table
// prefix sums at a cell: the group base plus the local parts, widened from 32 bits with
// a zero high word (the w d part still carries kLocBias, taken off per sum of edges)
__device__ __forceinline__ void add_cell(long long& aw, long long& ay, const longlong2& bs, const int2& lc) {
  aw += bs.x + (long long)(uint32_t)lc.x;
  ay += bs.y + (long long)(uint32_t)lc.y;
}
// cells staged past the sentinel (copies of it): every edge G <= g_end lies before
// T + 2 D, at most 2 x 255 + 1 cells past the table, so the loop needs no clamp
constexpr int kPadCells = 544;

// Byte offsets of the table arrays in shared memory: dt (4 B per cell), loc (8 B
// per cell), base (16 B per 32 cells), then the rings.
__host__ __device__ __forceinline__ uint32_t fixed_loc_off(int ncs) { return ((uint32_t)ncs * 4u + 15u) & ~15u; }
__host__ __device__ __forceinline__ uint32_t fixed_base_off(int ncs) {
  return fixed_loc_off(ncs) + (((uint32_t)ncs * 8u + 15u) & ~15u);
}
__host__ __device__ __forceinline__ uint32_t fixed_ring_off(int ncs) {
  return fixed_base_off(ncs) + ((((uint32_t)ncs + 31u) / 32u * 16u + 15u) & ~15u);
}

// ------------------------------------------------------------------ K1x

__device__ __forceinline__ double warp_sum_down(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  return v;
}

// Scale exponent k with v 2^k < 2^25 for every |v| <= vmax (so that 32 such
// integers sum to less than 2^30 in magnitude).
__device__ __forceinline__ int fixed_exponent(double vmax) {
  if (!(vmax > 0.0)) return 0;
  int e = 0;
  frexp(vmax, &e);  // vmax < 2^e
  return max(-100, min(25 - e, 100));
}

// x + 1.5 2^52 rounds |x| < 2^51 to the nearest integer (ties to even), whose low 32 bits
// are the sum's low word: one FP64 addition instead of a conversion and its scaling.
constexpr double kMagic64 = 6755399441055744.0;

// cell_of from rh = fl(1 / h): t rh lies within 2^-29 of fl(t / h) for the planner's at
// most 2^22 cells, so further than 2^-28 from an integer both have the same floor q, and
// t - q h lies well inside [0, h): no correction. Nearer, the exact division decides.
__device__ __forceinline__ int cell_fast(double t, double h, double rh) {
  const double x = __dmul_rn(t, rh);
  const double m = __dadd_rn(x, kMagic64);
  const double d = __dsub_rn(x, __dsub_rn(m, kMagic64));  // in [-1/2, 1/2]
  const int dh = __double2hiint(d);
  if ((dh & 0x7fffffff) < ((1023 - 28) << 20)) return cell_of(t, h);
  return __double2loint(m) - (dh < 0 ? 1 : 0);
}

constexpr int kPrepThreads = 512;  // of a star, over the CTAs of its cluster
constexpr int kPrepWarps = kPrepThreads / 32;

// One cluster of 1, 2, 4 or 8 CTAs per star, 512 threads in all: thread v takes points v, v +
// 512, ... for the FP64 sums, whose order (each thread's points, the warp's shuffle tree,
// the 16 warps in turn) does not depend on the cluster's size, so neither do W and ybar.
// What bounds it is the FP64 pipe (1/64 of the FP32 rate): about 27 operations a point,
// down from about 70 with a division per cell index, and conversions and products repeated
// per pass. 1/dy^2 and then w wait in the star's part of the loc array (8 bytes a cell, at
// least one cell a point, written last), the point's integer record in its 16 bytes of
// scratch (both in L2), so any length is handled alike and shared memory stays free for
// more CTAs. The second half is integer: each warp scans a contiguous sixteenth of the
// records, 32 at a time in 32-bit words, and writes the cells that end at each point,
// coalesced, with no pass over the cells and no block barrier. Clusters spread a star
// where stars are few (launch_prep_fixed). 4,096 single-sector stars 4.83 -> 2.61 ms; 256
// stars of 1-4 sectors 2.46 -> 0.62 ms; one star of 1,267 points 43 -> 21 us.
__global__ void __launch_bounds__(kPrepThreads) prep_fixed_kernel(const PrepFixedArgs a) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  __shared__ double red[2][kPrepWarps];               // the 16 warps' partial sums (every CTA holds all)
  __shared__ unsigned long long redm[2][kPrepWarps];  // and maxima
  __shared__ longlong2 part_tot[kPrepWarps];          // and integer totals of their parts
  const int s = a.fixed_stars[blockIdx.x / C];
  const StarDev st = a.stars[s];
  const int n = st.n_pts;
  if (n <= 0) return;  // the same in every CTA of the cluster
  const double* tp = a.tp + st.pt_off;
  const double* y = a.y + st.pt_off;
  const double* dy = a.dy + st.pt_off;
  int4* rec = reinterpret_cast<int4*>(a.ipre + st.cpre_off);
  double* wv = reinterpret_cast<double*>(a.loc + st.cell_off);
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
  const int v0 = rank * T + tid;       // this thread of the star's 512
  const int vwarp = v0 >> 5;
  const int nc = st.n_cells;
  const double h = st.h, rh = 1.0 / st.h;
  auto share = [&](auto* r, auto v) {  // lane 0's value into every CTA's array
    if (lane == 0)
      for (int c = 0; c < C; ++c) *cl.map_shared_rank(r + vwarp, c) = v;
  };
  auto total = [&](const double* r) {
    double t = 0.0;
    for (int i = 0; i < kPrepWarps; ++i) t += r[i];
    return t;
  };
  if (C > 1) cl.sync();  // every CTA of the cluster runs: its shared memory may be written

  // weights w = dy^-2 / sum dy^-2 and the weighted mean (FP64)
  double acc = 0.0;
#pragma unroll 4
  for (int i = v0; i < n; i += kPrepThreads) {
    const double inv = 1.0 / (dy[i] * dy[i]);
    wv[i] = inv;
    acc += inv;
  }
  share(red[0], warp_sum_down(acc));
  cl.sync();
  const double rws = 1.0 / total(red[0]);
  acc = 0.0;
  unsigned long long mw = 0ull, md = 0ull;
#pragma unroll 4
  for (int i = v0; i < n; i += kPrepThreads) {
    const double w = __dmul_rn(wv[i], rws);
    wv[i] = w;
    // non-negative and finite (the planner keeps stars of larger spreads off this path):
    // the bit patterns order as the values
    mw = max(mw, (unsigned long long)__double_as_longlong(w));
    acc = __fma_rn(w, y[i], acc);
  }
  share(red[1], warp_sum_down(acc));
  cl.sync();
  const double ybar = total(red[1]);
#pragma unroll 4
  for (int i = v0; i < n; i += kPrepThreads)
    md = max(md, (unsigned long long)__double_as_longlong(__dmul_rn(wv[i], __dsub_rn(y[i], ybar))) &
                     0x7fffffffffffffffull);
  mw = warp_max_u64(mw);
  md = warp_max_u64(md);
  share(redm[0], mw);
  share(redm[1], md);
  cl.sync();
  for (int i = 0; i < kPrepWarps; ++i) {
    mw = max(mw, redm[0][i]);
    md = max(md, redm[1][i]);
  }
  const double dmw = __longlong_as_double((long long)mw), dmd = __longlong_as_double((long long)md);
  // 64-bit table: scales that keep 32 consecutive points below 2^30. 32-bit table:
  // w_int = round(w F) with F = 2^32 - 2^17, so that the N <= 2^16 roundings leave the
  // total below 2^32 (r is then the ratio of two integer sums), and the largest y scale
  // that keeps every point's |y_int| (this kernel's largest |w d|) and every prefix sum
  // of y_int (the planner's largest running sum; this kernel's lies within 2^-9 of it,
  // and the roundings add at most 2^15) below 2^30
  const bool narrow = st.narrow != 0;
  int kw = fixed_exponent(dmw), ky = fixed_exponent(dmd);
  if (narrow) {
    int e1 = 0, e2 = 0;
    frexp(st.y_exc * 1.00390625, &e1);  // y_exc (1 + 2^-8) < 2^e1
    frexp(dmd * 1.00390625, &e2);
    kw = 0;
    ky = max(-100, min(30 - max(e1, e2), 100));
  }
  const double pw = narrow ? kNarrowF : ldexp(1.0, kw), py = ldexp(1.0, ky);

  // each point's integers, its cell and its offset there as a 32-bit fraction: (t' - u h)
  // / h by a multiplication stays within (T/h + 3) 2^-53 cells of the exact offset, inside
  // the guard band's allowance of 2 (T/h) 2^-53 cells for the cell offsets. The scalings by
  // powers of two are exact, so they fold into the rounding addition (F rounds first); added
  // to 2^20 and rounded down, the offset's 32 bits are the sum's low word.
#pragma unroll 2
  for (int i = v0; i < n; i += kPrepThreads) {
    const double w = wv[i];
    const double wi = narrow ? __dadd_rn(__dmul_rn(w, pw), kMagic64) : __fma_rn(w, pw, kMagic64);
    const double yi = __fma_rn(__dmul_rn(w, __dsub_rn(y[i], ybar)), py, kMagic64);
    const double t = tp[i];
    const int u = cell_fast(t, h, rh);
    const double ud = __dsub_rn(__hiloint2double(0x43300000, u), 4503599627370496.0);  // u as FP64
    const double q = __dadd_rd(__dmul_rn(__dsub_rn(t, __dmul_rn(ud, h)), rh), 1048576.0);
    // an offset that rounds to the cell's width, or to the empty cell's mark, is the largest
    const uint32_t dq = __double2hiint(q) == 0x41300000 ? min((uint32_t)__double2loint(q), 0xfffffffeu) : 0xfffffffeu;
    rec[i] = make_int4(__double2loint(wi), __double2loint(yi), u, (int)dq);
  }
  cl.sync();  // every record is in place

  // this warp's part of the points, [p0, p1) (the last part ends with point n, the sentinel
  // past the last cell), and the exact integer sums before it
  const int per = ((n + kPrepWarps - 1) / kPrepWarps + 31) & ~31;
  const int p0 = min(n, vwarp * per), p1 = vwarp == kPrepWarps - 1 ? n + 1 : min(n, p0 + per);
  {
    long long sw = 0, sy = 0;
#pragma unroll 4
    for (int i = p0 + lane; i < min(p1, n); i += 32) {
      const int2 r = __ldcg(reinterpret_cast<const int2*>(rec + i));
      sw += (long long)(uint32_t)r.x;
      sy += r.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
      sw += __shfl_xor_sync(0xffffffffu, sw, o);
      sy += __shfl_xor_sync(0xffffffffu, sy, o);
    }
    share(part_tot, make_longlong2(sw, sy));
  }
  cl.sync();
  long long run_w = 0, run_y = 0;  // sums before the next point
  for (int c = 0; c < vwarp; ++c) {
    run_w += part_tot[c].x;
    run_y += part_tot[c].y;
  }
  // The 32 points before the next: the low words of their prefix sums, which of them open a
  // 32-cell group, and the last one's cell. Sums over 32 consecutive points fit 32 bits (w
  // unsigned, w d signed): on the 64-bit table each term is below 2^25, on the 32-bit one
  // every prefix sum of w is below 2^32 and of w d below 2^30 in magnitude.
  uint32_t pw32 = 0, py32 = 0, pflag = 0;
  int last = -1;
  if (p0 > 0) {
    const int i = p0 - 32 + lane;
    int4 r = make_int4(0, 0, 0, 0);
    int up = -1;
    if (i >= 0) r = __ldcg(rec + i);
    if (i > 0) up = __ldcg(rec + i - 1).z;
    uint32_t xw = (uint32_t)r.x, xy = (uint32_t)r.y;  // sums of this point and the later ones
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t aw = __shfl_down_sync(0xffffffffu, xw, o), ay = __shfl_down_sync(0xffffffffu, xy, o);
      if (lane + o < 32) {
        xw += aw;
        xy += ay;
      }
    }
    pw32 = (uint32_t)run_w - xw;
    py32 = (uint32_t)run_y - xy;
    pflag = __ballot_sync(0xffffffffu, i >= 0 && (up < 0 || (up >> 5) != (r.z >> 5)));
    last = __shfl_sync(0xffffffffu, r.z, 31);
  }
  // the 32-bit table keeps every prefix of w_int below 2^32 and of y_int below 2^30 in
  // magnitude by its scales; a sum past its word's range would wrap: raise the error bit
  // (the star's results are then void)
  bool out_of_range = false;
  for (int base = p0; base < p1; base += 32) {  // warp-uniform
    const int i = base + lane;
    const bool on = i < p1;
    int4 r = make_int4(0, 0, nc, -1);  // the sentinel's record
    if (i < min(p1, n)) r = __ldcg(rec + i);
    int up = __shfl_up_sync(0xffffffffu, r.z, 1);
    if (lane == 0) up = last;
    last = __shfl_sync(0xffffffffu, r.z, 31);
    uint32_t xw = (uint32_t)r.x, xy = (uint32_t)r.y;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t aw = __shfl_up_sync(0xffffffffu, xw, o), ay = __shfl_up_sync(0xffffffffu, xy, o);
      if (lane >= o) {
        xw += aw;
        xy += ay;
      }
    }
    const long long pre_w = run_w + (long long)(xw - (uint32_t)r.x), pre_y = run_y + (int)(xy - (uint32_t)r.y);
    run_w += (long long)__shfl_sync(0xffffffffu, xw, 31);
    run_y += (int)__shfl_sync(0xffffffffu, xy, 31);
    out_of_range =
        out_of_range || (narrow && (pre_w >= (1ll << 32) || pre_y >= kNarrowBias || pre_y <= -kNarrowBias));
    // cells (up, r.z] end at this point: the sums before it, the point's offset in the last
    // of them; on the 64-bit table relative to their 32-cell group's first point: the group
    // of cell up opened with one of the 32 points before (a group holds at most 32), a
    // group that starts after up opens here
    uint32_t gw = 0, gy = 0;
    if (!narrow) {  // warp-uniform
      const unsigned flag = __ballot_sync(0xffffffffu, on && (up < 0 || (up >> 5) != (r.z >> 5)));
      const unsigned long long m = ((unsigned long long)flag << 32 | pflag) & ((1ull << (32 + lane)) - 1ull);
      const int o = 63 - __clzll((long long)m);  // -1 for the star's first point, which needs none
      const uint32_t cw = __shfl_sync(0xffffffffu, (uint32_t)pre_w, o & 31), cy = __shfl_sync(0xffffffffu, (uint32_t)pre_y, o & 31);
      const uint32_t bw = __shfl_sync(0xffffffffu, pw32, o & 31), by = __shfl_sync(0xffffffffu, py32, o & 31);
      gw = o >= 32 ? cw : bw;
      gy = o >= 32 ? cy : by;
      pflag = flag;
      pw32 = (uint32_t)pre_w;
      py32 = (uint32_t)pre_y;
    }
    auto put = [&](int c, int iu, int ig, uint32_t q, long long p_w, long long p_y, uint32_t g_w, uint32_t g_y) {
      a.gidx[st.cell_off + c] = ig;
      a.dt[st.cell_off + c] = q;
      if (narrow) {  // the prefix sums themselves: w below 2^32, |y| below 2^30 + 2^15, biased by 2^31
        a.loc[st.cell_off + c] = make_int2((int)(uint32_t)p_w, (int)((uint32_t)p_y + (uint32_t)kNarrowBias));
        return;
      }
      // at most 31 points of weights below 2^25 lie between the group start and the
      // cell: both local parts are below 2^30 in magnitude
      const bool old = iu >= 0 && (c >> 5) == (iu >> 5);
      a.loc[st.cell_off + c] = make_int2(old ? (int)((uint32_t)p_w - g_w) : 0,
                                         (int)((old ? (uint32_t)p_y - g_y : 0u) + (uint32_t)kLocBias));
      if ((c & 31) == 0) a.base[st.base_off + (c >> 5)] = make_longlong2(p_w, p_y);
    };
    if (on && r.z > up) put(r.z, up, i, (uint32_t)r.w, pre_w, pre_y, gw, gy);
    unsigned gaps = __ballot_sync(0xffffffffu, on && r.z - up > 1);  // empty cells before the point: the warp fills them
    while (gaps) {
      const int src = __ffs((int)gaps) - 1;
      gaps &= gaps - 1u;
      const int gu = __shfl_sync(0xffffffffu, up, src), gz = __shfl_sync(0xffffffffu, r.z, src);
      const long long p_w = __shfl_sync(0xffffffffu, pre_w, src), p_y = __shfl_sync(0xffffffffu, pre_y, src);
      const uint32_t g_w = __shfl_sync(0xffffffffu, gw, src), g_y = __shfl_sync(0xffffffffu, gy, src);
      for (int c = gu + 1 + lane; c < gz; c += 32) put(c, gu, base + src, 0xffffffffu, p_w, p_y, g_w, g_y);
    }
    if (on && i == n) {
      FixedStar f;
      f.w_tot = pre_w;
      f.y_tot = pre_y;
      f.kw = kw;
      f.ky = ky;
      f.scw = narrow ? (float)(1.0 / (double)pre_w) : __int_as_float((127 - kw) << 23);  // 1 / w_tot or 2^-kw
      f.narrow = narrow ? 1 : 0;
      a.fx[s] = f;
    }
  }
  if (out_of_range) atomicOr(a.err, kErrRange);
}

// K0x freq_rec_kernel (1 CTA per exact-path star, at plan time): one FreqRec per
// trial frequency. It depends on the grid and the star's cell width only, not on
// the fluxes, so a plan computes it once for all its searches.
__global__ void __launch_bounds__(256) freq_rec_kernel(const PrepFixedArgs a) {
  const int s = a.fixed_stars[blockIdx.x];
  const StarDev st = a.stars[s];
  const double h = st.h;
  const int tid = threadIdx.x;
  // per trial frequency: the same FP64 operations as the other search kernels
  for (int k = tid; k < st.n_f; k += blockDim.x) {
    const int64_t fidx = st.f_off + k;
    const double2 fq = a.fq[fidx];
    FreqRec r;
    r.K = 0ull;
    r.jlow = 0ull;
    r.nb = 0;
    r.band_q = 0u;
    r.gq_bstar = 0u;
    r.wmask = 0u;
    const int nb = (int)ceil(__ddiv_rn(a.noverlap, fq.y));
    if (nb >= 32 && nb <= min(a.nb_cap, 8192)) {
      const double F = __dmul_rn(fq.x, (double)nb);
      const double D = __ddiv_rn(1.0, F);  // bin duration (days)
      const double yT = __dmul_rn(st.baseline, F);
      const int g_end = (int)floor(yT) + 2;  // edges 0 .. g_end; tau_{g_end} > T
      r.gq_bstar = ((uint32_t)(g_end / nb) << 13) | (uint32_t)(g_end % nb);
      r.K = __double2ull_rn(__dmul_rn(__ddiv_rn(D, h), 1099511627776.0));  // D/h < 2^8 in 2^-40 units
      // guard band in 2^-32 cell units, twice the sum of the bounds on: the FP64 fold's
      // error, (T F + nbins) 2^-53 bins = (T F + nbins) (D/h) 2^-21 units; the edge step's
      // rounding, 2^-41 cells per edge (g_end 2^-9 units); the FP64 cell offsets of the
      // points and of D/h, (T/h) 2^-20 units; and the two 32-bit truncations
      r.band_q = (uint32_t)fmin(
          __dmul_rn(__dmul_rn(__dadd_rn(yT, (double)nb), __ddiv_rn(D, h)), 9.5367431640625e-07) +
              (double)(g_end >> 8) + __dmul_rn(__ddiv_rn(st.baseline, h), 3.814697265625e-06) + 16.0,
          1073741824.0);
      // box widths m_j and, per width, its lowest j (m_j is non-decreasing in j)
      unsigned long long jl = 0ull;
      uint32_t wm = 0u;
      for (int j = a.nq - 1; j >= 0; --j) {
        const int m = min(15, max(1, (int)floor(__dadd_rn(__dmul_rn(__dmul_rn(fq.y, a.E[j]), (double)nb), 0.5))));
        wm |= 1u << (m - 1);
        jl = (jl & ~(0xfull << (4 * (m - 1)))) | ((unsigned long long)j << (4 * (m - 1)));
      }
      r.jlow = jl;
      r.wmask = wm;
      r.nb = nb;
    }
    a.frec[fidx] = r;
  }
}

int launch_freq_recs(const PrepFixedArgs& a, void* stream) {
  if (a.n <= 0) return 0;
  freq_rec_kernel<<<a.n, 256, 0, (cudaStream_t)stream>>>(a);
  return (int)cudaGetLastError();
}

// CTAs per star: one where the stars alone fill the chip's SMs several times over, more
// where they are few, so that the longest stars do not run on one SM each while the others
// idle (FP64-bound: a 4-sector star takes 0.35 ms of one SM).
static int prep_cluster(int stars, int sms) {
  int c = 1;
  while (c < 8 && stars * c < 8 * sms) c *= 2;
  return c;
}

int launch_prep_fixed(const PrepFixedArgs& a, void* stream) {
  if (a.n <= 0) return 0;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int c = prep_cluster(a.n, sms);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(a.n * c));
  cfg.blockDim = dim3((unsigned)(kPrepThreads / c));
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)c;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, prep_fixed_kernel, a);
  return e != cudaSuccess ? (int)e : (int)cudaGetLastError();
}

// ------------------------------------------------------------------ K2x

// Box sweep of the two start bins ka (even) and ka + 1 over the ring (H[x] at ring[x mod
// 128]): the lane's running sums of both starts are (w, w d) pairs, added as packed FP32
// pairs; a start at or past the last bin begins with s = NaN, so that it never scores. Every width w = o + 1 present is scored
// s^2 / (r (1 - r)) for 0 < r < 1 and compared division-free with the lane's best so far.
// An exact FP32 tie keeps the lane's earlier candidate: within a pair of blocks the
// narrower width, then the lower start; across the lane's pairs (disjoint boxes, tied
// only by a coincidence of their FP32 sums) the earlier pair. Ties between lanes go to
// the lower duration index, then the lower start (the warp argmax).
template <bool ALL>
__device__ __forceinline__ void sweep_pair(const float2* ring, int ka, bool ain, bool bin, int mmax, uint32_t wmask,
                                           float& bs2, float& bd, int& bkey) {
  constexpr int NO = ALL ? 11 : 15;
  auto ld = [&](int t) { return *reinterpret_cast<const float4*>(ring + ((ka + 2 * t) & 127)); };
  int code = -1;  // 2 o + (start - ka) of the lane's best in this pair
  auto score = [&](const float2 acc, int c) {
    const float dd = __fmaf_rn(-acc.x, acc.x, acc.x);  // r (1 - r)
    const float s2 = __fmul_rn(acc.y, acc.y);
    const float lhs = __fmul_rn(s2, bd), rhs = __fmul_rn(bs2, dd);
    const bool better = dd > 0.f && lhs > rhs;
    bs2 = better ? s2 : bs2;
    bd = better ? dd : bd;
    code = better ? c : code;
  };
  const float none = __int_as_float(0x7fffffff);
  float2 A = make_float2(0.f, ain ? 0.f : none), B = make_float2(0.f, bin ? 0.f : none);
  float4 cur = ld(0);
#pragma unroll
  for (int o = 0; o < NO; ++o) {
    if (ALL || o < mmax) {
      if ((o & 1) == 0) {  // A += H[ka + o], B += H[ka + o + 1]
        A = __fadd2_rn(A, make_float2(cur.x, cur.y));
        B = __fadd2_rn(B, make_float2(cur.z, cur.w));
      } else {
        const float4 nxt = ld((o + 1) >> 1);
        A = __fadd2_rn(A, make_float2(cur.z, cur.w));
        B = __fadd2_rn(B, make_float2(nxt.x, nxt.y));
        cur = nxt;
      }
      if (ALL ? o >= 2 : ((wmask >> o) & 1u) != 0u) {
        score(A, 2 * o);
        score(B, 2 * o + 1);
      }
    }
  }
  if (code >= 0) bkey = ((code >> 1) << 16) | (ka + (code & 1));
}

// This warp's row of exact bin sums in the block's workspace: ws_block / kFixedWarps
// entries, at least the bins of every whole-table star of the plan, then the warp's
// kFixedPendRows entries of pending boxes (pend_rows).
__device__ __forceinline__ longlong2* warp_row(const FixedArgs& a) {
  return a.ws + (size_t)blockIdx.x * (size_t)a.ws_block +
         (size_t)(threadIdx.x >> 5) * (size_t)(a.ws_block / kFixedWarps);
}
__device__ __forceinline__ longlong2* pend_rows(const FixedArgs& a) {
  return warp_row(a) + (a.ws_block / kFixedWarps - kFixedPendRows);
}

// A whole-table frequency's chosen box, left by lane 0 for rescoring: its exact
// integer sums (w, w d) and, in the second half, (frequency in the item, the packed
// (j, width, k) word, s^2, r (1 - r)) of the FP32 sweep; s^2 < 0 when no box counts.
__device__ __forceinline__ void put_pending(longlong2* rows, int p, long long dw, long long dy, int fl,
                                            uint32_t key, float s2, float d) {
  int4* r = reinterpret_cast<int4*>(rows) + 2 * p;
  r[0] = make_int4((int)(uint32_t)dw, (int)(dw >> 32), (int)(uint32_t)dy, (int)(dy >> 32));
  r[1] = make_int4(fl, (int)key, __float_as_int(s2), __float_as_int(d));
}

// Lane t scores the t-th pending box again from its exact sums in double-float
// arithmetic (r and 1 - r over the star's total on the 32-bit table, scaled by 2^-kw
// on the 64-bit one; s scaled by 2^-ky) and stores it: the rescoring of up to 32
// frequencies takes one instruction stream (lane 0 alone, one frequency at a time,
// took 2.7 % of the launch). f0 is the item's first frequency.
__device__ __forceinline__ void flush_pending(const FixedArgs& a, const FixedStar& fx, int64_t f0,
                                              const longlong2* rows, int n, int lane) {
  __syncwarp();  // lane 0's records are visible to the warp
  if (lane < n) {
    const int4 r0 = reinterpret_cast<const int4*>(rows)[2 * lane];
    const int4 r1 = reinterpret_cast<const int4*>(rows)[2 * lane + 1];
    const long long dw = (long long)(((unsigned long long)(uint32_t)r0.y << 32) | (uint32_t)r0.x);
    const long long dy = (long long)(((unsigned long long)(uint32_t)r0.w << 32) | (uint32_t)r0.z);
    const uint32_t key = (uint32_t)r1.y;
    BoxBest bb;
    bb.s2 = __int_as_float(r1.z);
    bb.d = __int_as_float(r1.w);
    bb.s = 0.f;
    bb.r = 0.f;
    const bool nobox = bb.s2 < 0.f;
    bb.j = nobox ? 255 : (int)(key >> 20);
    bb.k = nobox ? -1 : (int)(key & 0xffffu);
    bb.xv = false;
    if (!nobox) {
      if (fx.narrow) {  // r = dw / w_tot and 1 - r = (w_tot - dw) / w_tot, both sums below 2^32
        const DF wt = df_from_ll_scaled(fx.w_tot, 0);
        bb.xr = df_div(df_from_ll_scaled(dw, 0), wt);
        bb.xq = df_div(df_from_ll_scaled(fx.w_tot - dw, 0), wt);
      } else {
        // kw lies in [24, 46] on this path: the largest weight is at most 1 and at least
        // 1/N with N <= 2^21 points, and w_max 2^kw lies in [2^24, 2^25)
        const int kw = min(max(fx.kw, 0), 62);
        bb.xr = df_from_ll_scaled(dw, kw);
        bb.xq = df_from_ll_scaled((1ll << kw) - dw, kw);  // 1 - r
      }
      bb.xs = df_from_ll_scaled(dy, fx.ky);
      bb.xv = true;
    }
    store_box(bb, 0, f0 + r1.x, a.sr, a.qidx, a.kbin, a.sbest, a.rbest);
  }
  __syncwarp();  // the records are read before the warp writes new ones
}

// One trial frequency on a warp: the exact bin sums S into the row srow (from the staged
// table's edges, 32 bins at a time), or already there from the window passes (WS); then
// per 64 bins their FP32 histogram records into the ring and the sweep, the warp argmax
// and the store. The box the FP32 sweep chose is scored once more from its exact integer
// sums in the row: at once when WS, else from the pending record put at prow[pend] (fl:
// the frequency within the item) and rescored in the caller's next flush_pending.
//
// Bound by shared memory and issue, each about 70-75 % busy: an edge takes two dependent
// gathers (7.2 wavefronts with the conflicts of cells D/h apart) and 16 instructions, and
// half of all instructions are the blocks' own. With the edges, the histogram and the sweep
// in one loop over 32 bins, U and its wrapped-around copies were carried from block to block
// by eight shuffles and the loop's registers spilled; reading the sums back from the row
// (L2, a pair of blocks ahead) gives each lane its two bins' neighbours by address: 2.664e9
// -> 2.443e9 instructions and 2.74 -> 2.66 ms on 150 stars, 6.48 -> 6.12 ms for the windowed
// search of 256 coarse spectra.
template <bool WS, bool NARROW>
__device__ __forceinline__ void run_frequency(const FixedArgs& a, int64_t fidx, const FreqRec& R,
                                              const FixedStar& fx, const unsigned char* smem,
                                              uint32_t loc_off, uint32_t base_off, int nc, float2* ring,
                                              int lane, float scw, float scy, const double* tp,
                                              const int32_t* gidx, uint32_t st4, uint32_t st8, uint32_t st16,
                                              longlong2* srow, longlong2* prow, int& pend, int fl) {
  const int nb = R.nb;
  const double f = a.fq[fidx].x;  // for the exact decision near ties
  const uint32_t wmask = R.wmask;
  const int mmax = 32 - __clz(wmask);
  const bool all_widths = wmask == 0x7fcu;  // exactly 3 .. 11 bins
  const int gq = (int)(R.gq_bstar >> 13), bstar = (int)(R.gq_bstar & 8191u);
  const int g_end = gq * nb + bstar;
  // edge step in 32.32 fixed point, so that the cell and the position in it are the
  // two halves of G K with no shift. Rounding the 24.40 step to it adds at most
  // 2^-33 cells per step, G / 2 units of 2^-32 cells at edge G: the guard band
  // grows by twice that at the last edge (g_end < 2^27: at most 16384 cycles of
  // 8192 bins; so the band stays below 2^31)
  const unsigned long long K32 = (R.K + 128ull) >> 8;
  const uint32_t k_lo = (uint32_t)K32, k_hi = (uint32_t)(K32 >> 32);
  const uint32_t band_q = R.band_q + (uint32_t)g_end;
  const int nblk = (nb + 31) >> 5;

  float bs2 = 0.f, bd = 1.f;   // best box of this lane: s^2, r (1 - r) and its key
  int bkey = 0x7fffffff;
  if constexpr (!WS) {
    for (int i = 0; i < nblk; ++i) {  // the bin sums S, 32 bins at a time: lanes x < nb own bin x
      const int x = (i << 5) + lane;
      // edges G = G0, G0 + nb, ... <= g_end (one per cycle). The edge at t' = 0
      // (G = 0) is skipped: no point lies before it. A block of r <= 16 bins spreads
      // each bin's cycles over P = 32 / r lanes (phase ph: cycles ph, ph + P, ...),
      // summed by shuffles afterwards. Idle lanes walk a real bin's edges
      // (discarded), so that every edge stays inside the staged table.
      const int r = nb - (i << 5);
      const bool split = r <= 16;
      int P = 1, ph = 0, xb = x;
      if (split) {
        P = 32 / r;
        ph = lane / r;
        xb = (i << 5) + (lane - ph * r);
      }
      const bool idle = split ? ph >= P : x >= nb;
      const int G0 = idle ? (i << 5) : (xb == 0 ? nb : xb + ph * nb);
      const int gstep = P * nb;
      // the w sums of the 32-bit table in wrapping 32-bit words: every bin and box sum
      // of w lies in [0, 2^32), so sums modulo 2^32 give them exactly
      using WAcc = std::conditional_t<NARROW, uint32_t, long long>;
      WAcc aw = 0;
      long long ay = 0;
      // the smallest (dq - fr + band) mod 2^32 over the lane's edges: some edge lies
      // within the guard band of its cell's point exactly when it is <= 2 band
      uint32_t nmin = 0xffffffffu;
      // every lane takes cnt edges; only in the last one may a lane be past g_end
      const int cnt0 = gq + ((i << 5) > bstar ? 0 : 1);
      const int cnt = split ? (cnt0 + P - 1) / P : cnt0;  // no division in full blocks
      // tau_G / h in 32.32 fixed point, X = G K (below 2^54: the cell index u < 2^22),
      // stepped by gstep K from edge to edge (the same bits as the product)
      auto xpos = [&](int G) {
        return (unsigned long long)(uint32_t)G * k_lo + ((unsigned long long)((uint32_t)G * k_hi) << 32);
      };
      const unsigned long long XS = xpos(gstep);
      unsigned long long X = xpos(G0);
      auto edge = [&](unsigned long long X, bool valid, bool clamp) {
        // cell u and position fr (2^-32 of a cell)
        int u = (int)(uint32_t)(X >> 32);
        if (clamp) u = min(u, nc);
        const uint32_t fr = (uint32_t)X;
        const uint32_t dq = *reinterpret_cast<const uint32_t*>(smem + (uint32_t)u * st4);
        nmin = min(nmin, dq - fr + band_q);
        const int v = u + (dq < fr ? 1 : 0);  // past the cell's point if it lies before tau_G
        const int2 lc = *reinterpret_cast<const int2*>(smem + loc_off + (uint32_t)v * st8);
        if constexpr (NARROW) {  // the 32-bit prefix sums themselves
          if (valid) {
            aw += (uint32_t)lc.x;
            ay += (long long)(uint32_t)lc.y;
          }
        } else {
          const longlong2 bs = *reinterpret_cast<const longlong2*>(smem + base_off + (uint32_t)(v >> 5) * st16);
          if (valid) add_cell(aw, ay, bs, lc);
        }
      };
      int c = 0;
      for (; c + 4 < cnt; c += 4) {
        const unsigned long long X1 = X + XS, X2 = X1 + XS, X3 = X2 + XS;
        edge(X, true, false);
        edge(X1, true, false);
        edge(X2, true, false);
        edge(X3, true, false);
        X = X3 + XS;
      }
      for (; c + 1 < cnt; ++c) {
        edge(X, true, false);
        X += XS;
      }
      const bool last = G0 + (cnt - 1) * gstep <= g_end;
      edge(X, last, true);
      ay -= (long long)(cnt - (last ? 0 : 1)) * (NARROW ? kNarrowBias : kLocBias);  // the bias of the edges taken
      bool near = nmin <= 2u * band_q;  // an edge within the guard band of its cell's point
      if (split) {  // warp-uniform: add the other phases of each bin into lanes 0 .. r-1
        for (int q = 1; q < P; ++q) {
          const WAcc ow = __shfl_down_sync(0xffffffffu, aw, q * r);
          const long long oy = __shfl_down_sync(0xffffffffu, ay, q * r);
          const bool on = __shfl_down_sync(0xffffffffu, near ? 1 : 0, q * r) != 0;
          if (lane < r) {
            aw += ow;
            ay += oy;
            near = near || on;
          }
        }
      }
      near = near && x < nb;  // lanes past the last bin accumulated nothing meaningful
      if (__any_sync(0xffffffffu, near)) {  // rare: redo the bin, near-ties by the exact FP64 fold
        if (near) {
          aw = 0;
          ay = 0;
          for (int g = x == 0 ? nb : x; g <= g_end; g += nb) {
            const unsigned long long X =
                (unsigned long long)(uint32_t)g * k_lo + ((unsigned long long)((uint32_t)g * k_hi) << 32);
            const int u = min((int)(uint32_t)(X >> 32), nc);
            const uint32_t fr = (uint32_t)X;
            const uint32_t dq = reinterpret_cast<const uint32_t*>(smem)[u];
            int sel = dq < fr ? 1 : 0;
            if (dq != 0xffffffffu && (uint32_t)(dq - fr + band_q) <= 2u * band_q)
              sel = exact_before(tp, gidx[u], f, nb, g);
            const int v = u + sel;
            const int2 lc = reinterpret_cast<const int2*>(smem + loc_off)[v];
            if constexpr (NARROW) {
              aw += (uint32_t)lc.x;
              ay += (long long)(uint32_t)lc.y - kNarrowBias;
            } else {
              const longlong2 bs = reinterpret_cast<const longlong2*>(smem + base_off)[v >> 5];
              add_cell(aw, ay, bs, lc);
              ay -= kLocBias;
            }
          }
        }
      }
      if (x < nb) srow[x] = make_longlong2((long long)aw, ay);
    }
    __syncwarp();  // the row is written before its bins are read
  }
  // 64 bins at a time, two a lane: H[x] = U[x + 1] - U[x] = S[x + 1] - S[x] (+ C_end at x =
  // b*), indices mod nb, exact, then FP32 in the ring; then the sweep of the 64 before
  // (boxes of up to 15 bins starting in them), whose last boxes reach into these. The sums
  // come from the row (L2) a pair of blocks ahead.
  const int npair = (nb + 63) >> 6;
  longlong2 s0, s1, s2;
  auto fetch = [&](int p) {
    const int x = (p << 6) + 2 * lane;
    if ((p << 6) + 65 < nb) {  // warp-uniform: no bin past the last
      s0 = srow[x];
      s1 = srow[x + 1];
      s2 = srow[x + 2];
    } else {  // bins past the last are the first ones; further than that they are not used
      auto wrap = [&](int b) { return min(b < nb ? b : b - nb, nb - 1); };
      s0 = srow[wrap(x)];
      s1 = srow[wrap(x + 1)];
      s2 = srow[wrap(x + 2)];
    }
  };
  fetch(0);
  for (int p = 0; p <= npair; ++p) {
    const int ka = (p << 6) + 2 * lane;
    const int b0 = ka < nb ? ka : ka - nb, b1 = ka + 1 < nb ? ka + 1 : ka + 1 - nb;
    const long long y0 = s1.y - s0.y + (b0 == bstar ? fx.y_tot : 0), y1 = s2.y - s1.y + (b1 == bstar ? fx.y_tot : 0);
    float4 hv;
    if constexpr (NARROW) {
      // the 32-bit table's bin sums: the w sum lies in [0, 2^32) (a part of the star's
      // total below 2^32), so the difference of the low words is exact; the w d sum goes
      // through 32 bits when every lane's fits (the same rounding either way)
      const uint32_t w0 = (uint32_t)s1.x - (uint32_t)s0.x + (b0 == bstar ? (uint32_t)fx.w_tot : 0u);
      const uint32_t w1 = (uint32_t)s2.x - (uint32_t)s1.x + (b1 == bstar ? (uint32_t)fx.w_tot : 0u);
      hv.x = __uint2float_rn(w0);
      hv.z = __uint2float_rn(w1);
      if (__all_sync(0xffffffffu, y0 == (long long)(int)y0 && y1 == (long long)(int)y1)) {
        hv.y = __int2float_rn((int)y0);
        hv.w = __int2float_rn((int)y1);
      } else {
        hv.y = __ll2float_rn(y0);
        hv.w = __ll2float_rn(y1);
      }
    } else {
      hv.x = __ll2float_rn(s1.x - s0.x + (b0 == bstar ? fx.w_tot : 0));
      hv.y = __ll2float_rn(y0);
      hv.z = __ll2float_rn(s2.x - s1.x + (b1 == bstar ? fx.w_tot : 0));
      hv.w = __ll2float_rn(y1);
    }
    hv.x = __fmul_rn(hv.x, scw);
    hv.y = __fmul_rn(hv.y, scy);
    hv.z = __fmul_rn(hv.z, scw);
    hv.w = __fmul_rn(hv.w, scy);
    *reinterpret_cast<float4*>(ring + (ka & 127)) = hv;
    __syncwarp();
    if (p < npair) fetch(p + 1);
    if (p > 0) {
      const int kp = ka - 64;
      if (all_widths) sweep_pair<true>(ring, kp, kp < nb, kp + 1 < nb, mmax, wmask, bs2, bd, bkey);
      else sweep_pair<false>(ring, kp, kp < nb, kp + 1 < nb, mmax, wmask, bs2, bd, bkey);
    }
    __syncwarp();  // the sweep is done before its blocks' records are overwritten
  }
  const bool none = bkey == 0x7fffffff;
  bs2 = none ? -1.f : bs2;
  const int bo = bkey >> 16;
  // the lowest duration index of each width, read again here rather than kept live
  const unsigned long long jlow = a.frec[fidx].jlow;
  // (j, width, k) in one word: j in bits 20-23, the width index in 16-19, k in 0-15;
  // one j has one width, so the word orders as (j, k) does
  uint32_t key = none ? 0xffffffffu
                      : ((uint32_t)((jlow >> (4 * bo)) & 15ull) << 20) | ((uint32_t)bo << 16) | (uint32_t)(bkey & 0xffff);
  for (int off = 16; off > 0; off >>= 1) {
    const float o_s2 = __shfl_xor_sync(0xffffffffu, bs2, off);
    const float o_d = __shfl_xor_sync(0xffffffffu, bd, off);
    const uint32_t o_key = __shfl_xor_sync(0xffffffffu, key, off);
    // strict: larger s^2 / d, then the lower (j, k); s^2 < 0 is no box
    bool take;
    if (o_s2 < 0.f) take = false;
    else if (bs2 < 0.f) take = true;
    else {
      const float lhs = o_s2 * bd, rhs = bs2 * o_d;
      take = lhs != rhs ? lhs > rhs : o_key < key;
    }
    if (take) {
      bs2 = o_s2; bd = o_d; key = o_key;
    }
  }
  const bool nobox = bs2 < 0.f;
  const int bj = nobox ? 255 : (int)(key >> 20);
  const int bk = nobox ? -1 : (int)(key & 0xffffu);
  const int bm = nobox ? 0 : (int)((key >> 16) & 15u) + 1;  // bins of the box
  if constexpr (!WS) {  // whole tables: the box's exact sums wait for a batch rescoring
    if (lane == 0) {
      long long dw = 0, dy = 0;
      if (bk >= 0) {  // U[bk + bm] - U[bk] as below
        const int k2 = bk + bm;
        const int k2m = k2 >= nb ? k2 - nb : k2;
        const longlong2* row = srow;
        const longlong2 a0 = row[bk], a1 = row[k2m];
        const long long nwrap = (bstar < k2m ? 1 : 0) + (k2 >= nb ? 1 : 0) - (bstar < bk ? 1 : 0);
        dw = a1.x - a0.x + nwrap * fx.w_tot;
        dy = a1.y - a0.y + nwrap * fx.y_tot;
        if (NARROW) dw = (long long)(uint32_t)dw;  // the rows hold the w sums modulo 2^32
      }
      put_pending(prow, pend, dw, dy, fl, key, bs2, bd);
    }
    ++pend;
    return;
  }
  BoxBest bb;
  bb.s2 = bs2; bb.d = bd; bb.s = 0.f; bb.r = 0.f; bb.j = bj; bb.k = bk;
  bb.xv = false;
  if (lane == 0 && bk >= 0) {
    // the chosen box [bk, bk + bm) from the exact integer sums: U[bk + bm] - U[bk],
    // U[x] = S[x mod nb] + ([b* < x mod nb] + floor(x / nb)) C_end; the difference is
    // a box sum (below 2^46), so it and 2^kw - it split into exact float pairs
    const int k2 = bk + bm;
    const int k2m = k2 >= nb ? k2 - nb : k2;
    const longlong2* row = srow;
    const longlong2 a0 = row[bk], a1 = row[k2m];
    const long long nwrap = (bstar < k2m ? 1 : 0) + (k2 >= nb ? 1 : 0) - (bstar < bk ? 1 : 0);
    long long dw = a1.x - a0.x + nwrap * fx.w_tot;
    const long long dy = a1.y - a0.y + nwrap * fx.y_tot;
    if (NARROW) {  // r = dw / w_tot and 1 - r = (w_tot - dw) / w_tot, both sums below 2^32
      dw = (long long)(uint32_t)dw;  // the rows hold the w sums modulo 2^32
      const DF wt = df_from_ll_scaled(fx.w_tot, 0);
      bb.xr = df_div(df_from_ll_scaled(dw, 0), wt);
      bb.xq = df_div(df_from_ll_scaled(fx.w_tot - dw, 0), wt);
    } else {
      // kw lies in [24, 46] on this path: the largest weight is at most 1 and at least
      // 1/N with N <= 2^21 points, and w_max 2^kw lies in [2^24, 2^25)
      const int kw = min(max(fx.kw, 0), 62);
      bb.xr = df_from_ll_scaled(dw, kw);
      bb.xq = df_from_ll_scaled((1ll << kw) - dw, kw);  // 1 - r
    }
    bb.xs = df_from_ll_scaled(dy, fx.ky);
    bb.xv = true;
  }
  store_box(bb, lane, fidx, a.sr, a.qidx, a.kbin, a.sbest, a.rbest);
}

// One work item of a star whose table is longer than shared memory. Pass A, window
// by window (the window's cells staged once for all the item's frequencies): every
// warp adds, for each of its frequencies and bins, the prefix sums C(tau_G) of the
// window's edges G (the edges of a window are those in [ceil(w C h F),
// ceil((w+1) C h F)), the same FP64 expression on both sides of each boundary, so
// the windows partition them) to the bin's row of this block's workspace. Pass B:
// each frequency runs the block pipeline from its row.
//
// Bound by shared-memory wavefronts and issue together: an edge takes three dependent
// gathers at cells D/h apart (about 2.5 + 5.2 + 1 wavefronts with the conflicts such strides
// have) and 22 instructions, a block of bins in a window about 100 more. So the 64-bit
// group bases (16 bytes a lane) are folded into the local parts when a window is staged,
// all but 16 + 16 bits of each; edges that every bin of the block has run unrolled with no
// test; the row's old sums are fetched a block ahead. 40 stars of 1-13 sectors 60.1 ->
// 48.9 ms, 256 coarse spectra of 1-4 sectors 6.18 -> 5.3 ms.
template <int NW>
__device__ void windowed_item(const FixedArgs& a, const WorkItem& wi, const StarDev& st, const FixedStar& fx,
                              unsigned char* smem, int warp, int lane, uint32_t st4, uint32_t st8, uint32_t st16) {
  const int nc = st.n_cells;
  const int cap = st.win_cap + 1;  // staged cells of a window, plus one past its end
  const uint32_t loc_off = fixed_loc_off(cap), base_off = fixed_base_off(cap);
  // pass B reads the workspace rows only: its rings overlay the window's table
  float2* ring = reinterpret_cast<float2*>(smem) + warp * kRing;
  const int stride = wi.pad0;      // workspace row length (bins)
  longlong2* ws = a.ws + (size_t)blockIdx.x * (size_t)a.ws_block;
  const double h = st.h;
  const double* tp = a.tp + st.pt_off;
  const int32_t* gidx = a.gidx + st.cell_off;
  const uint32_t* s_dt = reinterpret_cast<const uint32_t*>(smem);
  for (int w = 0; w < st.n_win; ++w) {
    const int cstart = w * st.win_cells;
    const int lo = (w == 0) ? 0 : ((cstart - 1) >> 5) << 5;
    const int hi = (w == st.n_win - 1) ? nc : min(nc, (w + 1) * st.win_cells + st.win_ovl);
    const int n_loc = hi - lo + 1;
    __syncthreads();  // the previous window's passes are done
    {
      uint32_t* d_dt = reinterpret_cast<uint32_t*>(smem);
      int2* d_loc = reinterpret_cast<int2*>(smem + loc_off);
      uint32_t* d_hi = reinterpret_cast<uint32_t*>(smem + base_off);
      const int2 lnc = a.loc[st.cell_off + nc];
      // a warp stages the 32 cells of a group (lo is a multiple of 32): the low 31 bits of
      // the group's bases go into the local parts (below 2^31 + 2^30 then), the rest (below
      // 2^15 in magnitude: the sums are below 2^46) stays the group's
      for (int i = threadIdx.x; i <= n_loc; i += NW * 32) {  // n_loc + 1 cells
        const int c = lo + i, g = c >> 5;
        const longlong2 bs = g <= (nc >> 5) ? a.base[st.base_off + g] : make_longlong2(fx.w_tot, fx.y_tot);
        const int2 lc = c <= nc ? a.loc[st.cell_off + c] : (g == (nc >> 5) ? lnc : make_int2(0, (int)kLocBias));
        d_dt[i] = c <= nc ? a.dt[st.cell_off + c] : 0xffffffffu;
        d_loc[i] = make_int2((int)((uint32_t)lc.x + ((uint32_t)bs.x & 0x7fffffffu)),
                             (int)((uint32_t)lc.y + ((uint32_t)bs.y & 0x7fffffffu)));
        if (lane == 0) d_hi[i >> 5] = (uint32_t)(bs.x >> 31) | (((uint32_t)(bs.y >> 31) + kHiBias) << 16);
      }
    }
    __syncthreads();
    for (int fl = warp; fl < wi.f_count; fl += NW) {
      const int64_t fidx = st.f_off + wi.f_begin + fl;
      const FreqRec R = a.frec[fidx];
      const int nb = R.nb;
      if (nb == 0) continue;  // reported by pass B
      const double f = a.fq[fidx].x;
      const double Fq = __dmul_rn(f, (double)nb);
      const int gq = (int)(R.gq_bstar >> 13), bstar = (int)(R.gq_bstar & 8191u);
      const int g_end = gq * nb + bstar;
      const int gs = (w == 0) ? 0 : (int)ceil(__dmul_rn(__dmul_rn((double)cstart, h), Fq));
      const int ge = (w == st.n_win - 1) ? g_end + 1
                                          : (int)ceil(__dmul_rn(__dmul_rn((double)((w + 1) * st.win_cells), h), Fq));
      // a bin's edges from the first in the window: tau_G / h in 32.32 fixed point relative to
      // the staged cells, stepped by nb K. The first is the 24.40 product truncated, the step
      // rounded, so edge k lies within (k + 2) / 2 units of 2^-32 cells of its product
      const unsigned long long XS = ((unsigned long long)(uint32_t)nb * R.K + 128ull) >> 8;
      const unsigned long long XL = (unsigned long long)(uint32_t)lo << 40;
      const uint32_t u_last = (uint32_t)(n_loc - 1);
      longlong2* row = ws + (size_t)fl * (size_t)stride;
      // this bin's edges in [gs, ge): cycles c0 = max(0, ceil((gs - x) / nb)) .. c1 =
      // floor((ge - 1 - x) / nb) for x = 32 i + lane. With A = gs + nb - 1 - 32 i = qa nb + ra
      // and B = ge - 1 - 32 i = qb nb + rb (0 <= ra, rb < nb) and lane < 32 <= nb, they are
      // qa - [lane > ra] (at least 0) and qb - [lane > rb] (below 0: no edge); (q, r) step
      // down by 32 bins per block with at most one borrow, so the divisions are once per
      // window and frequency
      int qa = (gs + nb - 1) / nb, ra = (gs + nb - 1) - qa * nb;
      int qb, rb;
      if (ge - 1 >= 0) {
        qb = (ge - 1) / nb;
        rb = (ge - 1) - qb * nb;
      } else {
        qb = -1;
        rb = ge - 1 + nb;
      }
      // the bins' sums of the windows before, fetched a block ahead
      longlong2 next = make_longlong2(0, 0);
      if (w > 0) next = row[lane];  // lane < 32 <= nb
      for (int i = 0; (i << 5) < nb; ++i) {
        const int x = (i << 5) + lane;
        const bool inb = x < nb;
        // the edge at t' = 0 is skipped
        int c0 = max(0, qa - (lane > ra ? 1 : 0));
        if (x == 0 && c0 == 0) c0 = 1;
        const int c1 = qb - (lane > rb ? 1 : 0);
        ra -= 32;
        if (ra < 0) {
          ra += nb;
          --qa;
        }
        rb -= 32;
        if (rb < 0) {
          rb += nb;
          --qb;
        }
        const int cntl = inb ? max(0, c1 - c0 + 1) : 0;
        const int cmax = (int)__reduce_max_sync(0xffffffffu, (unsigned)cntl);
        const longlong2 prev = next;
        if (w > 0 && x + 32 < nb) next = row[x + 32];
        if (cmax == 0 && w > 0) continue;  // no edge of these bins in this window
        // edges that every bin of the block has, then (two at most, three at the start) those
        // that only some have; lanes past the last bin walk along, discarded
        const int call = min(cmax, (int)__reduce_min_sync(0xffffffffu, inb ? (unsigned)cntl : 0x7fffffffu));
        const uint32_t band = R.band_q + (uint32_t)cmax + 2u;
        unsigned long long X = ((unsigned long long)(uint32_t)(x + c0 * nb) * R.K - XL) >> 8;
        long long aw = 0, ay = 0;     // sums of the local parts
        uint32_t hw = 0, hy = 0;      // and of the groups', in units of 2^31 (at most 2^14 edges of at most 2^16)
        uint32_t nmin = 0xffffffffu;  // the smallest (dq - fr + band) mod 2^32, as on whole tables
        auto edge = [&](unsigned long long X, bool valid) {
          const uint32_t ul = min((uint32_t)(X >> 32), u_last);  // staged cell
          const uint32_t fr = (uint32_t)X;
          const uint32_t dq = *reinterpret_cast<const uint32_t*>(smem + ul * st4);
          const uint32_t d = dq - fr + band;
          const uint32_t v = ul + (dq < fr ? 1u : 0u);
          const int2 lc = *reinterpret_cast<const int2*>(smem + loc_off + v * st8);
          const uint32_t hi = *reinterpret_cast<const uint32_t*>(smem + base_off + (v >> 5) * st4);
          if (valid) {
            nmin = min(nmin, d);
            aw += (long long)(uint32_t)lc.x;
            ay += (long long)(uint32_t)lc.y;
            hw = __dp2a_lo(hi, 0x0001u, hw);  // + the low half, + the high half
            hy = __dp2a_lo(hi, 0x0100u, hy);
          }
        };
        int k = 0;
        for (; k + 4 <= call; k += 4) {
          const unsigned long long X1 = X + XS, X2 = X1 + XS, X3 = X2 + XS;
          edge(X, true);
          edge(X1, true);
          edge(X2, true);
          edge(X3, true);
          X = X3 + XS;
        }
        if (k + 2 <= call) {
          const unsigned long long X1 = X + XS;
          edge(X, true);
          edge(X1, true);
          X = X1 + XS;
          k += 2;
        }
        if (k < call) {
          edge(X, true);
          X += XS;
          ++k;
        }
        for (; k < cmax; ++k, X += XS) edge(X, k < cntl);
        ay -= (long long)cntl * kLocBias;
        const bool near = inb && nmin <= 2u * band;
        if (__any_sync(0xffffffffu, near)) {  // rare: redo, near-ties by the exact FP64 fold
          if (near) {
            aw = 0;
            ay = 0;
            hw = 0;
            hy = 0;
            for (int c = c0; c <= c1; ++c) {
              const int G = x + c * nb;
              const unsigned long long X = ((unsigned long long)(uint32_t)G * R.K - XL) >> 8;
              const uint32_t ul = min((uint32_t)(X >> 32), u_last);
              const uint32_t fr = (uint32_t)X;
              const uint32_t dq = s_dt[ul];
              int sel = dq < fr ? 1 : 0;
              if (dq != 0xffffffffu && dq - fr + band <= 2u * band)
                sel = exact_before(tp, gidx[lo + (int)ul], f, nb, G);
              const uint32_t v = ul + (uint32_t)sel;
              const int2 lc = reinterpret_cast<const int2*>(smem + loc_off)[v];
              const uint32_t hi = reinterpret_cast<const uint32_t*>(smem + base_off)[v >> 5];
              aw += (long long)(uint32_t)lc.x;
              ay += (long long)(uint32_t)lc.y - kLocBias;
              hw += hi & 0xffffu;
              hy += hi >> 16;
            }
          }
        }
        aw += (long long)hw << 31;
        ay += (long long)((int)hy - cntl * (int)kHiBias) << 31;
        if (inb) row[x] = make_longlong2(prev.x + aw, prev.y + ay);
      }
    }
  }
  __syncthreads();  // every window's sums are in the workspace
  const float scw = fx.scw;
  const float scy = __int_as_float((127 - fx.ky) << 23);
  for (int fl = warp; fl < wi.f_count; fl += NW) {
    const int64_t fidx = st.f_off + wi.f_begin + fl;
    const FreqRec R = a.frec[fidx];
    if (R.nb == 0) {
      if (lane == 0) {
        atomicOr(a.err, kErrNbins);
        a.sr[fidx] = 0.f;
        if (a.qidx) a.qidx[fidx] = 255;
        if (a.kbin) a.kbin[fidx] = 0xffffffffu;
        if (a.sbest) a.sbest[fidx] = 0.f;
        if (a.rbest) a.rbest[fidx] = 0.f;
      }
      continue;
    }
    int no_pend = 0;
    run_frequency<true, false>(a, fidx, R, fx, smem, loc_off, base_off, nc, ring, lane, scw, scy, tp, gidx, st4, st8,
                               st16, ws + (size_t)fl * (size_t)stride, nullptr, no_pend, fl);
  }
}

// Bulk asynchronous copy global -> shared of `bytes` (a multiple of 16; both addresses
// 16-byte aligned), completing on the mbarrier.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          (uint32_t)__cvta_generic_to_shared(dst)),
      "l"(src), "r"(bytes), "r"((uint32_t)__cvta_generic_to_shared(bar))
      : "memory");
}
constexpr uint32_t kCopyWaitLimit = 1u << 24;  // polls of a table copy (each ends after ~1 us at most)

// WIN: the launch of the time-windowed tables' items, else that of the whole tables'. Each is
// compiled for its own kind (the plan keeps their items apart): with both in one kernel the
// whole-table path spilled.
template <int NW, bool WIN>
__global__ void __launch_bounds__(NW * 32, 1) cells_fixed_kernel(const FixedArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  __shared__ int s_item, s_star, s_next;
  __shared__ __align__(8) uint64_t s_tbar;  // completion of a table's bulk copies
  uint32_t tphase = 0;                       // its phase (thread 0)
  if (threadIdx.x == 0) {
    s_star = -1;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"((uint32_t)__cvta_generic_to_shared(&s_tbar))
                 : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // element strides as run-time values, so that the table addresses are formed by
  // integer multiply-adds rather than by the (busier) integer logic pipe
  const uint32_t st4 = a.stride4, st8 = 2u * a.stride4, st16 = 4u * a.stride4;

  bool done = false;
  const int iter_lim = a.loop_bound > 0 ? min(a.loop_bound, a.n_items) : a.n_items;
  for (int iter = 0; iter <= iter_lim; ++iter) {
    __syncthreads();
    if (threadIdx.x == 0) {
      s_item = atomicAdd(a.cursor, 1);
      s_next = 0;
    }
    __syncthreads();
    const int it = s_item;
    if (it >= a.n_items) { done = true; break; }
    const WorkItem wi = a.items[it];
    const StarDev st = a.stars[wi.star];
    const FixedStar fx = a.fx[wi.star];
    if (WIN != (st.n_win > 1)) {  // block-uniform; the plan hands each launch its own kind of table
      if (threadIdx.x == 0) atomicOr(a.err, kErrNbins);
      continue;
    }
    if constexpr (WIN) {
      windowed_item<NW>(a, wi, st, fx, smem, warp, lane, st4, st8, st16);
    } else {
    const int nc = st.n_cells;  // sentinel cell index
    const int ncp = nc + 1 + kPadCells;
    const uint32_t loc_off = fixed_loc_off(ncp), base_off = fixed_base_off(ncp);
    float2* ring = reinterpret_cast<float2*>(smem + fixed_ring_off(ncp)) + warp * kRing;
    if (s_star != wi.star) {  // block-uniform: stage the star's table and its padding
      uint32_t* d_dt = reinterpret_cast<uint32_t*>(smem);
      int2* d_loc = reinterpret_cast<int2*>(smem + loc_off);
      longlong2* d_base = reinterpret_cast<longlong2*>(smem + base_off);
      // cells [0, nb4) and groups [0, ng) by bulk copies (the table starts at a 16-byte
      // boundary: cell_off is a multiple of 4), the rest of the table and the padding by
      // the threads; the two parts do not overlap
      // (the 32-bit table has no group bases: its padding cells repeat the sentinel's sums)
      const bool narrow = fx.narrow != 0;
      const int nb4 = (nc + 1) & ~3, ng = narrow ? 0 : (nc >> 5) + 1;
      if (threadIdx.x == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // after the last item's reads
        const uint32_t bytes = (uint32_t)nb4 * 12u + (uint32_t)ng * 16u;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(&s_tbar)), "r"(bytes)
                     : "memory");
        if (nb4 > 0) {
          bulk_g2s(d_dt, a.dt + st.cell_off, (uint32_t)nb4 * 4u, &s_tbar);
          bulk_g2s(d_loc, a.loc + st.cell_off, (uint32_t)nb4 * 8u, &s_tbar);
        }
        if (ng > 0) bulk_g2s(d_base, a.base + st.base_off, (uint32_t)ng * 16u, &s_tbar);
      }
      const int2 lnc = a.loc[st.cell_off + nc];
      for (int i = nb4 + (int)threadIdx.x; i < ncp; i += NW * 32) {
        const bool in = i <= nc;
        d_dt[i] = in ? a.dt[st.cell_off + i] : 0xffffffffu;
        d_loc[i] = in ? a.loc[st.cell_off + i]
                      : ((narrow || (i >> 5) == (nc >> 5)) ? lnc : make_int2(0, (int)kLocBias));
      }
      if (!narrow)
        for (int i = ng + (int)threadIdx.x; i < (ncp + 31) / 32; i += NW * 32)
          d_base[i] = make_longlong2(fx.w_tot, fx.y_tot);
      if (threadIdx.x == 0) {  // bounded wait for the copies
        bool ok = false;
        for (uint32_t k = 0; k < kCopyWaitLimit && !ok; ++k) {
          uint32_t done;
          asm volatile(
              "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
              "selp.u32 %0, 1, 0, p;\n\t}"
              : "=r"(done)
              : "r"((uint32_t)__cvta_generic_to_shared(&s_tbar)), "r"(tphase)
              : "memory");
          ok = done != 0;
        }
        if (!ok) atomicOr(a.err, kErrCopyWait);
        tphase ^= 1u;
        s_star = ok ? wi.star : -1;
      }
      __syncthreads();
    }
    const float scw = fx.scw;  // 2^-kw, or 1 / w_tot on the 32-bit table
    const float scy = __int_as_float((127 - fx.ky) << 23);  // 2^-ky (|ky| <= 100)
    const double* tp = a.tp + st.pt_off;
    const int32_t* gidx = a.gidx + st.cell_off;

    longlong2* const srow = warp_row(a);
    longlong2* const prow = pend_rows(a);
    const int64_t f0 = st.f_off + wi.f_begin;
    int pend = 0;  // boxes waiting in prow for their rescoring (warp-uniform)
    for (int fi = 0; fi <= wi.f_count; ++fi) {  // bounded: each pass takes one frequency
      int fl = 0;
      if (lane == 0) fl = atomicAdd(&s_next, 1);
      fl = __shfl_sync(0xffffffffu, fl, 0);
      if (fl >= wi.f_count) break;
      const int64_t fidx = st.f_off + wi.f_begin + fl;
      const FreqRec R = a.frec[fidx];
      const int nb = R.nb;
      if (nb == 0) {
        if (lane == 0) {
          atomicOr(a.err, kErrNbins);
          a.sr[fidx] = 0.f;
          if (a.qidx) a.qidx[fidx] = 255;
          if (a.kbin) a.kbin[fidx] = 0xffffffffu;
          if (a.sbest) a.sbest[fidx] = 0.f;
          if (a.rbest) a.rbest[fidx] = 0.f;
        }
        continue;
      }
      if (fx.narrow)  // block-uniform
        run_frequency<false, true>(a, fidx, R, fx, smem, loc_off, base_off, nc, ring, lane, scw, scy, tp, gidx, st4,
                                   st8, st16, srow, prow, pend, fl);
      else
        run_frequency<false, false>(a, fidx, R, fx, smem, loc_off, base_off, nc, ring, lane, scw, scy, tp, gidx, st4,
                                    st8, st16, srow, prow, pend, fl);
      if (pend == 32) {
        flush_pending(a, fx, f0, prow, pend, lane);
        pend = 0;
      }
    }
    if (pend > 0) flush_pending(a, fx, f0, prow, pend, lane);
    }
  }
  if (!done && threadIdx.x == 0) atomicOr(a.err, kErrQueueBound);
}

uint32_t fixed_smem_bytes(int ncs) { return fixed_ring_off(ncs + kPadCells) + (uint32_t)kFixedWarps * kRing * 8u; }
uint32_t fixed_window_smem_bytes(int ncs) {
  return fixed_ring_off(ncs) > (uint32_t)kFixedWarps * kRing * 8u ? fixed_ring_off(ncs) : (uint32_t)kFixedWarps * kRing * 8u;
}

int launch_cells_fixed(const FixedArgs& a, bool windowed, int blocks, size_t smem, void* stream) {
  auto kern = windowed ? cells_fixed_kernel<kFixedWarps, true> : cells_fixed_kernel<kFixedWarps, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, search_smem_limit());
  if (e != cudaSuccess) return (int)e;
  kern<<<blocks, kFixedWarps * 32, smem, (cudaStream_t)stream>>>(a);
  return (int)cudaGetLastError();
}

int fixed_blocks_per_sm(size_t smem) {  // the fewer of the two instantiations'
  int nmin = 0;
  for (int k = 0; k < 2; ++k) {
    auto kern = k ? cells_fixed_kernel<kFixedWarps, true> : cells_fixed_kernel<kFixedWarps, false>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, search_smem_limit()) != cudaSuccess)
      return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kFixedWarps * 32, smem) != cudaSuccess) return 0;
    nmin = (k == 0 || nb < nmin) ? nb : nmin;
  }
  return nmin;
}

}  // namespace qlp
