// 1-D CNN of the learned period proposal (sm_103a): the 64 -> 64 channel
// convolutions (kernel 9, "same" padding) as implicit GEMMs on the 5th-generation
// tensor cores, BF16 operands, FP32 accumulation in tensor memory.
//
// Layouts. Activations are channels-last BF16 [B][L][64] (one 128-byte row per
// position). A tile is 128 positions x 64 output channels:
//   Y[l, co] = sum_{kk=0..8} sum_{ci} W[kk][co][ci] X[l + kk - 4, ci]
// Its 136 input rows l0-4 .. l0+131 sit in shared memory as they are in memory,
// one 128-byte row per position, in the 128-byte-swizzled K-major layout (chunk c
// of row r at chunk c ^ (r & 7)), so tap kk is the same tile shifted by kk rows:
// its A descriptor starts kk * 128 bytes later (the swizzle follows the address
// bits, so a shifted start reads the shifted rows). The weights (9 taps x 64 x 64)
// stay resident in the same layout, 64 rows of 128 bytes per tap. Each tile takes
// 9 taps x 4 K-steps of tcgen05.mma (M = 128, N = 64, K = 16, the K step 32 bytes
// along the row) into a TMEM accumulator of 64 FP32 columns.
//
// Pipeline (one persistent CTA per SM, warp roles): warp 0 copies the weights in
// one bulk asynchronous copy (on their own barrier, which the MMA issuer waits for)
// and loads tiles with TMA into a ring of kStages buffers (one box of 64 channels x 136 rows per tile, of a
// 3-D tensor map over [B][L][64] with the 128-byte swizzle, so rows outside
// [0, L) of the tile's own sample come back as zeros); warp 1 issues the MMAs of
// each tile into one of kAcc accumulators and commits them to the buffer's
// "empty" barrier and the accumulator's "full" barrier; warps 2-9 (two per TMEM
// lane quarter, 32 output channels each) read an accumulator back (one tcgen05.ld
// of 32 columns), apply bias and ReLU or the backward ReLU mask, store BF16 and
// release the accumulator. Every barrier wait
// is bounded; a wait that runs out raises QLP error bit 16, and the CTA still
// waits (bounded) for its copies and MMAs in flight before it frees TMEM.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "qlp_internal.h"
#include "tc_common.cuh"

namespace qlp {

constexpr int kC = 64;             // channels of the middle layers
constexpr int kTaps = 9;           // kernel size
constexpr int kTileM = 128;        // positions per tile
constexpr int kRows = kTileM + kTaps - 1;  // staged rows per tile
constexpr int kABytes = kRows * kC * 2;     // 17,408 = 17 swizzle atoms of 1,024 bytes
constexpr int kWBytes = kTaps * kC * kC * 2;  // 73,728 = 72 atoms
constexpr int kStages = 6;         // tile buffers in flight
constexpr int kAcc = 4;            // TMEM accumulators (64 columns each)
constexpr int kEpiWarps = 8;       // two per TMEM lane quarter, 32 columns each
constexpr int kConvThreads = 64 + 32 * kEpiWarps;  // producer, MMA, epilogue warps
constexpr int kOutBytes = kTileM * kC * 2;  // one BF16 output tile (16 KB), staged for a TMA store
constexpr int kOutBufs = 2;
constexpr uint32_t kWaitLimit = 1u << 26;

struct ConvTcArgs {
  const uint4* wpack;          // packed weights, kWBytes
  const float* bias;           // [64] or null
  const __nv_bfloat16* mask;   // [B][L][64]: multiply by (mask > 0) (backward), or null
  int32_t* err;
  int32_t batch;
  int32_t len;                 // multiple of 128
  int32_t relu;
};

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// One TMA box of the 3-D map (channel x, row y, sample z) into shared memory,
// completing `bytes` on the barrier. x must be a multiple of 8 (16 bytes).
__device__ __forceinline__ void tma_load3(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

// A shared-memory box to the 3-D map (channel x, row y, sample z) as one bulk group
// of this thread. x = 0 and y >= 0: the store starts at a 16-byte boundary.
__device__ __forceinline__ void tma_store3(const CUtensorMap* map, const void* src, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];\n\t"
      "cp.async.bulk.commit_group;" ::"l"(reinterpret_cast<uint64_t>(map)),
      "r"(x), "r"(y), "r"(z), "r"(smem_u32(src))
      : "memory");
}
// This thread's bulk groups have finished reading shared memory / have completed.
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// Barrier of the epilogue warps (id 1) that also ANDs a predicate over them.
__device__ __forceinline__ bool epi_barrier_and(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.and.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v), "n"(32 * kEpiWarps)
      : "memory");
  return r != 0;
}

// Epilogue of one tile: accumulator columns [col + c0, col + c0 + 32) (output
// channels c0 .. c0+31) for the lane quarter q of this warp, row r = 32 q + lane;
// one TMEM load and wait, the accumulator released, then bias, ReLU or the backward
// mask, BF16, into the staging tile `out` (128 rows of 128 bytes, 1024-byte aligned)
// with the 128-byte swizzle of the store's tensor map: 16-byte chunk j of row r at
// chunk j ^ (r & 7), so that eight lanes fill the 32 banks once. `keep` has the backward
// mask's bit for each of the row's 32 channels (MASK).
template <bool MASK>
__device__ __forceinline__ void conv_epilogue(const ConvTcArgs& a, const float* s_bias, uint32_t tmem,
                                              uint32_t col, int c0, int q, uint64_t* acc_empty,
                                              unsigned char* out, uint32_t keep) {
  const int lane = threadIdx.x & 31;
  const int r = 32 * q + lane;
  float v[32];
  tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + col + (uint32_t)c0, v);
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive(acc_empty);  // the values are in registers: the MMA may reuse the columns
#pragma unroll
  for (int h = 0; h < 32; h += 8) {
    const int j = (c0 + h) >> 3;  // the 16-byte chunk of the 128-byte row
    uint4* chunk = reinterpret_cast<uint4*>(out + r * 128 + ((j ^ (r & 7)) << 4));
    uint32_t ow[4];
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      float z0 = v[h + i] + s_bias[c0 + h + i], z1 = v[h + i + 1] + s_bias[c0 + h + i + 1];
      if (a.relu) { z0 = fmaxf(z0, 0.f); z1 = fmaxf(z1, 0.f); }
      if (MASK) {  // the forward activation (BF16) was not positive
        if (!((keep >> (h + i)) & 1u)) z0 = 0.f;
        if (!((keep >> (h + i + 1)) & 1u)) z1 = 0.f;
      }
      ow[i >> 1] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(z0)) |
                   ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(z1)) << 16);
    }
    *chunk = make_uint4(ow[0], ow[1], ow[2], ow[3]);
  }
}

// Tile i of this CTA is tile blockIdx.x + i gridDim.x (all roles walk the same list).
template <bool MASK>
__global__ void __launch_bounds__(kConvThreads, 1)
    conv64_tc_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap ymap,
                     const ConvTcArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  // everything from the next 1024-byte boundary (the 128-byte swizzle's period): the
  // weights, kStages tile buffers of kABytes and kOutBufs output staging tiles, each a
  // whole number of 1,024-byte atoms
  unsigned char* wsm = smem + ((1024u - (smem_u32(smem) & 1023u)) & 1023u);
  unsigned char* ring = wsm + kWBytes;
  unsigned char* obuf = ring + kStages * kABytes;
  __shared__ __align__(8) uint64_t full[kStages], empty[kStages], accf[kAcc], acce[kAcc], fin;
  __shared__ uint32_t tmem_base;
  __shared__ float s_bias[kC];
  __shared__ __align__(16) unsigned char s_mask[MASK ? 2 : 1][MASK ? kTileM * 8 : 16];  // a bit per value of the backward mask
  __shared__ int s_fail;

  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int tiles_per_sample = a.len / kTileM;
  const int n_tiles = a.batch * tiles_per_sample;
  const int n_my = (int)blockIdx.x < n_tiles ? (n_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  // resident weights (one bulk asynchronous copy, issued below with the first tiles) and
  // bias; barriers; TMEM
  __shared__ __align__(8) uint64_t wbar;
  if (tid < kC) s_bias[tid] = a.bias ? a.bias[tid] : 0.f;
  if (tid == 0) {
    for (int k = 0; k < kStages; ++k) {
      mbar_init(&full[k], 1);
      mbar_init(&empty[k], 1);
    }
    for (int k = 0; k < kAcc; ++k) {
      mbar_init(&accf[k], 1);
      mbar_init(&acce[k], kEpiWarps);  // one arrival per epilogue warp
    }
    mbar_init(&fin, 1);
    mbar_init(&wbar, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(&tmem_base, kAcc * kC);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  bool ok = true;

  if (warp == 0 && lane == 0) {  // TMA producer
    mbar_arrive_expect_tx(&wbar, (uint32_t)kWBytes);
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(wsm)),
                 "l"(a.wpack), "r"((uint32_t)kWBytes), "r"(smem_u32(&wbar))
                 : "memory");
    int issued = 0;
    for (int i = 0; i < n_my && ok; ++i) {
      const int s = i % kStages;
      if (i >= kStages) ok = mbar_wait(&empty[s], (uint32_t)((i / kStages - 1) & 1), kWaitLimit);
      if (!ok) break;
      const int t = (int)blockIdx.x + i * (int)gridDim.x;
      const int b = t / tiles_per_sample, l0 = (t % tiles_per_sample) * kTileM;
      unsigned char* buf = ring + s * kABytes;
      mbar_arrive_expect_tx(&full[s], (uint32_t)kABytes);
      tma_load3(buf, &xmap, 0, l0 - kTaps / 2, b, &full[s]);
      issued = i + 1;
    }
    // every copy issued has landed before the CTA goes on (bounded)
    for (int i = issued > kStages ? issued - kStages : 0; i < issued; ++i)
      if (!mbar_wait(&full[i % kStages], (uint32_t)((i / kStages) & 1), kWaitLimit)) ok = false;
    if (!mbar_wait(&wbar, 0u, kWaitLimit)) ok = false;
  } else if (warp == 1 && lane == 0) {  // MMA issuer
    const uint32_t idesc = idesc_bf16_f32(kTileM, kC);
    // descriptors as a base plus a compile-time offset: every offset is a multiple of
    // 16 bytes and every address stays below 2^18, so (addr + off) >> 4 = (addr >> 4)
    // + (off >> 4) within the 14-bit start-address field
    const uint64_t bdesc0 = smem_desc_sw128(smem_u32(wsm));
    if (n_my > 0) ok = mbar_wait(&wbar, 0u, kWaitLimit);  // the weights have landed
    for (int i = 0; i < n_my && ok; ++i) {
      const int s = i % kStages, ac = i % kAcc;
      ok = mbar_wait(&full[s], (uint32_t)((i / kStages) & 1), kWaitLimit);
      if (ok && i >= kAcc) ok = mbar_wait(&acce[ac], (uint32_t)((i / kAcc - 1) & 1), kWaitLimit);
      if (!ok) break;
      tc_fence_after();
      const uint64_t adesc0 = smem_desc_sw128(smem_u32(ring + s * kABytes));
      const uint32_t dst = tmem + (uint32_t)(ac * kC);
#pragma unroll
      for (int kk = 0; kk < kTaps; ++kk) {
#pragma unroll
        for (int ks = 0; ks < kC / 16; ++ks) {  // tap kk: kk rows on; K step ks: 32 bytes along the row
          const uint64_t ad = adesc0 + (uint64_t)((kk * 128 + ks * 32) >> 4);
          const uint64_t bd = bdesc0 + (uint64_t)((kk * kC * 128 + ks * 32) >> 4);
          mma_bf16(dst, ad, bd, idesc, kk > 0 || ks > 0);
        }
      }
      mma_commit(&empty[s]);  // the buffer is free once these MMAs have read it
      mma_commit(&accf[ac]);  // the accumulator is ready
    }
    // every MMA issued has completed before TMEM is freed (bounded)
    mma_commit(&fin);
    if (!mbar_wait(&fin, 0u, kWaitLimit)) ok = false;
  } else if (warp >= 2) {  // epilogue: TMEM lane quarter warp % 4, channels c0 .. c0+31
    const int q = warp & 3, c0 = 32 * ((warp - 2) / 4);
    const bool issuer = warp == 2 && lane == 0;  // issues the tile's TMA store
    // The backward mask of a tile as one bit per value: each of the eight warps reads 16 rows,
    // four whole rows a load (a thread reading its own row's 64 bytes touched 32 lines a
    // load: 66 -> 53 us of 128 x 4,096), and leaves a byte per 8 channels, one tile ahead
    // so that the loads overlap this tile's MMAs and the tile's barrier hands the bytes over.
    const int mrow = 16 * (warp - 2) + (lane >> 3), mchunk = lane & 7;
    uint4 mk[4];
    auto mask_load = [&](int t) {
      const uint4* src = reinterpret_cast<const uint4*>(
          a.mask + ((size_t)(t / tiles_per_sample) * a.len + (t % tiles_per_sample) * kTileM + mrow) * kC) + mchunk;
#pragma unroll
      for (int j = 0; j < 4; ++j) mk[j] = __ldg(src + 4 * j * (kC / 8));
    };
    auto mask_put = [&](int buf) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t w[4] = {mk[j].x, mk[j].y, mk[j].z, mk[j].w};
        uint32_t bits = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          bits |= (__uint_as_float(w[e] << 16) > 0.f ? 1u : 0u) << (2 * e);
          bits |= (__uint_as_float(w[e] & 0xffff0000u) > 0.f ? 1u : 0u) << (2 * e + 1);
        }
        s_mask[buf][(mrow + 4 * j) * 8 + mchunk] = (unsigned char)bits;
      }
    };
    if (MASK && n_my > 0) {
      mask_load(blockIdx.x);
      mask_put(0);
      ok = epi_barrier_and(true);
    }
    for (int i = 0; i < n_my; ++i) {
      const int ac = i % kAcc;
      const int t = (int)blockIdx.x + i * (int)gridDim.x;
      // staging tile i % 2: its store (tile i - 2) finished reading before the last barrier
      unsigned char* out = obuf + (i % kOutBufs) * kOutBytes;
      const bool ahead = MASK && i + 1 < n_my;
      if (ahead) mask_load(t + (int)gridDim.x);
      bool mine = mbar_wait(&accf[ac], (uint32_t)((i / kAcc) & 1), kWaitLimit);
      mine = __all_sync(0xffffffffu, mine) != 0;
      if (mine) {
        tc_fence_after();
        const uint32_t keep =
            MASK ? *reinterpret_cast<const uint32_t*>(&s_mask[i & 1][(32 * q + lane) * 8 + (c0 >> 3)]) : 0u;
        conv_epilogue<MASK>(a, s_bias, tmem, (uint32_t)(ac * kC), c0, q, &acce[ac], out, keep);
        fence_proxy_async_smem();  // the staged tile becomes visible to the TMA store
      }
      if (ahead) mask_put((i + 1) & 1);  // its readers, two tiles ago, passed the last barrier
      if (issuer) bulk_wait_read_all();  // tile i - 1's store has read the other staging tile
      ok = epi_barrier_and(mine);  // every epilogue warp takes the same branch
      if (!ok) break;
      if (issuer) tma_store3(&ymap, out, 0, (t % tiles_per_sample) * kTileM, t / tiles_per_sample);
    }
    if (issuer) bulk_wait_all();  // the stores are complete before the CTA ends
  }
  if (!ok) atomicExch(&s_fail, 1);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid == 0 && s_fail) atomicOr(a.err, kErrMmaWait);
  if (warp == 1) tmem_dealloc(tmem, kAcc * kC);
}

// W[kk][co][ci] (FP32) -> BF16 planes for the tensor-core kernel. transpose=1
// packs the weights of the input-gradient convolution: W'[kk][ci][co] = W[8-kk][co][ci].
// Per tap kk, 64 rows n (the output channel) of 128 bytes (the 64 reduction channels),
// 16-byte chunk j of row n at chunk j ^ (n & 7): the MMA's 128-byte-swizzled layout.
__device__ __forceinline__ void pack_chunk(const float* w, uint4* out, int transpose, int i) {
  const int kk = i / (kC * 8);  // (kk, row n, chunk j)
  const int n = (i / 8) % kC;
  const int j = i % 8;
  __align__(16) __nv_bfloat16 v[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int k = 8 * j + e;  // reduction channel
    const float x = transpose ? w[((kTaps - 1 - kk) * kC + k) * kC + n] : w[(kk * kC + n) * kC + k];
    v[e] = __float2bfloat16_rn(x);
  }
  out[(kk * kC + n) * 8 + (j ^ (n & 7))] = *reinterpret_cast<const uint4*>(v);
}
__global__ void pack_w64_kernel(const float* w, uint4* out, int transpose) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < kTaps * kC * 8) pack_chunk(w, out, transpose, i);
}
// All of a network's 64 -> 64 layers, both forms, in one launch (blockIdx.y: layer and
// form): eight launches of 3 us before.
struct PackArgs {
  const float* w[4];
  uint4 *fwd[4], *bwd[4];
};
__global__ void pack_all_kernel(const PackArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y >> 1;
  if (i >= kTaps * kC * 8) return;
  if (blockIdx.y & 1) pack_chunk(a.w[k], a.bwd[k], 1, i);
  else pack_chunk(a.w[k], a.fwd[k], 0, i);
}

// Shared memory of the conv kernel: resident weights, the row tiles and the output
// staging tiles (with up to 1 KB to align them).
int conv64_smem_bytes() { return kWBytes + kStages * kABytes + 1024 + kOutBufs * kOutBytes; }

// cuTensorMapEncodeTiled from the driver, found once through the runtime (a static's
// initialiser: a second host thread waits for the first to have found it)
static PFN_cuTensorMapEncodeTiled_v12000 encode_tiled() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    const bool ok = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                        cudaSuccess &&
                    q == cudaDriverEntryPointSuccess;
    return ok ? reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p) : nullptr;
  }();
  return fn;
}

// The tensor [B][L][64] (BF16) in boxes of 64 channels x `rows` positions of one sample,
// 128-byte swizzle, zeros outside the sample's [0, len). The driver's encoder wants the
// thread's context current, which a runtime call of this thread has to have made: every
// launcher sets its kernel's attribute first.
static cudaError_t map_rows64(CUtensorMap* map, const void* base, int batch, int len, int rows) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {(cuuint64_t)kC, (cuuint64_t)len, (cuuint64_t)batch};
  const cuuint64_t strides[2] = {(cuuint64_t)kC * 2, (cuuint64_t)len * kC * 2};
  const cuuint32_t box[3] = {(cuuint32_t)kC, (cuuint32_t)rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? cudaSuccess
             : cudaErrorInvalidValue;
}

int launch_conv64(const void* xv, const void* wv, const float* bias, const void* mv, void* yv,
                  int32_t* err, int batch, int len, int relu, void* stream) {
  const uint4* wpack = static_cast<const uint4*>(wv);
  const __nv_bfloat16* mask = static_cast<const __nv_bfloat16*>(mv);
  if (batch <= 0) return 0;
  const int smem = conv64_smem_bytes();
  auto kern = mask ? conv64_tc_kernel<true> : conv64_tc_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  // the input in boxes of a whole tile with its halo rows (136), the output in boxes of a
  // whole tile (128 rows)
  alignas(64) CUtensorMap map, ymap;
  if (e == cudaSuccess) e = map_rows64(&map, xv, batch, len, kRows);
  if (e == cudaSuccess) e = map_rows64(&ymap, yv, batch, len, kTileM);
  if (e != cudaSuccess) return (int)e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int tiles = batch * (len / kTileM);
  const int grid = tiles < sms ? tiles : sms;
  ConvTcArgs a{wpack, bias, mask, err, batch, len, relu};
  kern<<<grid, kConvThreads, smem, (cudaStream_t)stream>>>(map, ymap, a);
  return (int)cudaGetLastError();
}

int launch_pack_all(const float* const* w, void* const* fwd, void* const* bwd, void* stream) {
  PackArgs a{};
  for (int k = 0; k < 4; ++k) {
    a.w[k] = w[k];
    a.fwd[k] = static_cast<uint4*>(fwd[k]);
    a.bwd[k] = static_cast<uint4*>(bwd[k]);
  }
  pack_all_kernel<<<dim3((kTaps * kC * 8 + 127) / 128, 8), 128, 0, (cudaStream_t)stream>>>(a);
  return (int)cudaGetLastError();
}

int launch_pack_w64(const float* w, void* out, int transpose, void* stream) {
  const int n = kTaps * kC * 8;
  pack_w64_kernel<<<(n + 127) / 128, 128, 0, (cudaStream_t)stream>>>(w, static_cast<uint4*>(out), transpose);
  return (int)cudaGetLastError();
}


// ------------------------------------------------------------------ other layers
// First layer QLP_CNN_IN_CH -> 64 channels and last layer 64 -> 1 channel (kernel 9, same
// padding) on the CUDA cores, the first layer's weight gradient on the tensor cores; weight
// and bias gradients as two-stage reductions (per-CTA partial sums, then a sum over CTAs);
// BCE with logits; Adam with FP32 master weights.

constexpr int kSmTile = 128;  // a sample's length is a multiple of this many positions

// x0 [B][L][CI] BF16 -> a1 [B][L][64] BF16 = relu(b1 + conv(x0, W1)), W1 [9][64][CI], FP32
// weights: lane = two output channels (one packed FP32 pair), warp = 16 positions of a
// 64-position tile. A lane walks the 24 staged rows its positions see and adds each row's CI
// values to the positions it reaches, so that a position's sum runs over the taps and then
// the channels as written (the BF16 results depend on that order); per row it issues up
// to 96 packed FMAs on 16 independent sums for three broadcast loads (the values staged
// twice, as pairs). Bound by the FP32 pipes (54 FMAs per output: 45 us of 524,288 positions);
// one thread per channel with a window of rows in registers reached half of that (128 x
// 4,096: 89 -> 74 us). The next tile's values are fetched while this one is summed.
constexpr int kInTile = 64, kInRows = kInTile + kTaps - 1, kInPos = 16, kInThreads = 32 * kInTile / kInPos;
__global__ void __launch_bounds__(kInThreads, 3) conv_in_kernel(const __nv_bfloat16* x0, const float* w1,
                                                                const float* b1, __nv_bfloat16* a1, int batch,
                                                                int len) {
  constexpr int CI = QLP_CNN_IN_CH, kVals = kInRows * CI, kFetch = (kVals + kInThreads - 1) / kInThreads;
  static_assert(CI == 6, "a row is three 16-byte loads of value pairs");
  __shared__ __align__(16) float2 s_x[2][kVals];
  const int lane = threadIdx.x & 31, q0 = kInPos * (threadIdx.x >> 5);
  float2 w[kTaps][CI];
#pragma unroll
  for (int kk = 0; kk < kTaps; ++kk)
#pragma unroll
    for (int ci = 0; ci < CI; ++ci)
      w[kk][ci] = make_float2(w1[(kk * kC + 2 * lane) * CI + ci], w1[(kk * kC + 2 * lane + 1) * CI + ci]);
  const float2 bias = make_float2(b1[2 * lane], b1[2 * lane + 1]);
  const int tps = len / kInTile, n_tiles = batch * tps;
  unsigned short nxt[kFetch];  // as loaded: converting here would wait for the loads
  auto fetch = [&](int t) {  // the tile's staged rows l0 - 4 .. l0 + 67 are consecutive values
    const int b = t / tps, l0 = (t - b * tps) * kInTile;
    const unsigned short* src =
        reinterpret_cast<const unsigned short*>(x0) + ((long long)b * len + l0 - kTaps / 2) * CI;
#pragma unroll
    for (int j = 0; j < kFetch; ++j) {
      const int e = threadIdx.x + kInThreads * j, l = l0 - kTaps / 2 + e / CI;
      nxt[j] = 0;
      if (e < kVals && l >= 0 && l < len) nxt[j] = src[e];
    }
  };
  int buf = 0;
  if ((int)blockIdx.x < n_tiles) fetch(blockIdx.x);
  for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, buf ^= 1) {
#pragma unroll
    for (int j = 0; j < kFetch; ++j) {
      const int e = threadIdx.x + kInThreads * j;
      const float v = __uint_as_float((uint32_t)nxt[j] << 16);
      if (e < kVals) s_x[buf][e] = make_float2(v, v);
    }
    __syncthreads();  // the other buffer's readers passed the last barrier before this tile's stores
    if (t + (int)gridDim.x < n_tiles) fetch(t + gridDim.x);
    float2 acc[kInPos];
#pragma unroll
    for (int q = 0; q < kInPos; ++q) acc[q] = bias;
    const float4* row = reinterpret_cast<const float4*>(s_x[buf] + q0 * CI);
#pragma unroll
    for (int r = 0; r < kInPos + kTaps - 1; ++r) {
      float2 x[CI];
#pragma unroll
      for (int c = 0; c < CI / 2; ++c) {
        const float4 v = row[r * (CI / 2) + c];
        x[2 * c] = make_float2(v.x, v.y);
        x[2 * c + 1] = make_float2(v.z, v.w);
      }
#pragma unroll
      for (int ci = 0; ci < CI; ++ci)
#pragma unroll
        for (int q = 0; q < kInPos; ++q)
          if (r - q >= 0 && r - q < kTaps) acc[q] = __ffma2_rn(w[r - q][ci], x[ci], acc[q]);
    }
    const int b = t / tps, l0 = (t - b * tps) * kInTile;
    __nv_bfloat162* out = reinterpret_cast<__nv_bfloat162*>(a1 + ((size_t)b * len + l0 + q0) * kC) + lane;
#pragma unroll
    for (int q = 0; q < kInPos; ++q)
      out[(size_t)q * (kC / 2)] = __floats2bfloat162_rn(fmaxf(acc[q].x, 0.f), fmaxf(acc[q].y, 0.f));
  }
}

// a5 [B][L][64] BF16 -> logit [B][L] FP32 = b6 + conv(a5, W6), W6 [9][64]. A tile is 512 rows
// of one sample, staged by two TMA boxes (128-byte swizzle, zeros outside the sample); a
// thread takes four of them (128 apart) and forms P[kk] = sum_ci W6[kk][ci] a5[ci] for every
// tap, the taps in packed FP32 pairs (the channels four by four from the last, the order
// the kept logits were defined with), then logit[q] = b6 + sum_kk P[q + kk][kk] for the
// tile's 504 inner rows. The weights' broadcast loads (36 bytes a channel into every lane)
// are what bounds it: four rows share each, where one row per thread spent 31 us on them
// and staging 136 rows with three barriers as long (128 x 4,096: 43 -> 24.5 us; reading
// a5 takes 10).
constexpr int kOutThreads = 128, kOutSlots = 4, kOutRows = kOutThreads * kOutSlots;
constexpr int kOutTile = kOutRows - (kTaps - 1), kOutW = 12;
constexpr int kOutABytes = kOutRows * kC * 2;
constexpr int kOutSmem = kOutABytes + 1024;  // with up to 1 KB to align it
__global__ void __launch_bounds__(kOutThreads, 2) conv_out_kernel(const __grid_constant__ CUtensorMap amap,
                                                                  const float* w6, const float* b6, float* logit,
                                                                  int32_t* err, int batch, int len) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* tile = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  __shared__ __align__(16) float s_w[kC * kOutW];  // [channel][tap], 48 bytes a channel
  __shared__ float s_p[kTaps][kOutRows];
  __shared__ __align__(8) uint64_t full;
  const int tid = threadIdx.x;
  for (int i = tid; i < kTaps * kC; i += kOutThreads) s_w[(i % kC) * kOutW + i / kC] = w6[i];
  if (tid == 0) {
    mbar_init(&full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const float bias = b6[0];
  const int tps = (len + kOutTile - 1) / kOutTile, n_tiles = batch * tps;
  auto load = [&](int t) {  // thread 0
    const int b = t / tps, l0 = (t - b * tps) * kOutTile;
    mbar_arrive_expect_tx(&full, (uint32_t)kOutABytes);
    tma_load3(tile, &amap, 0, l0 - kTaps / 2, b, &full);
    tma_load3(tile + kOutABytes / 2, &amap, 0, l0 - kTaps / 2 + kOutRows / 2, b, &full);
  };
  if (tid == 0 && (int)blockIdx.x < n_tiles) load(blockIdx.x);
  uint32_t phase = 0;
  for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, phase ^= 1u) {
    const int b = t / tps, l0 = (t - b * tps) * kOutTile;
    const bool ok = __syncthreads_and(mbar_wait(&full, phase, kWaitLimit)) != 0;
    if (!ok) {  // the copy did not land in its bound
      if (tid == 0) atomicOr(err, kErrMmaWait);
      return;
    }
    const int slots = min(kOutSlots, (len - l0 + kTaps - 1 + kOutThreads - 1) / kOutThreads);  // with rows to sum
    float2 acc[kOutSlots][kTaps / 2];
    float acc8[kOutSlots];
#pragma unroll
    for (int s = 0; s < kOutSlots; ++s) {
      acc8[s] = 0.f;
#pragma unroll
      for (int i = 0; i < kTaps / 2; ++i) acc[s][i] = make_float2(0.f, 0.f);
    }
    auto sums = [&](auto n_slots) {
      constexpr int NS = decltype(n_slots)::value;
#pragma unroll 2
      for (int c = 0; c < kC / 8; ++c) {
        uint4 v[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s)  // rows tid + 128 s: the same place in their swizzle atoms
          v[s] = *reinterpret_cast<const uint4*>(tile + (tid + kOutThreads * s) * 128 + ((c ^ (tid & 7)) << 4));
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int e = (i & 4) | (3 - (i & 3));  // 3 2 1 0 7 6 5 4
          const float* w = s_w + (8 * c + e) * kOutW;
          const float4 wa = *reinterpret_cast<const float4*>(w), wb = *reinterpret_cast<const float4*>(w + 4);
          const float w8 = w[8];
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            const uint32_t u = e < 2 ? v[s].x : e < 4 ? v[s].y : e < 6 ? v[s].z : v[s].w;
            const float f = __uint_as_float((e & 1) ? (u & 0xffff0000u) : (u << 16));
            const float2 x = make_float2(f, f);
            acc[s][0] = __ffma2_rn(make_float2(wa.x, wa.y), x, acc[s][0]);
            acc[s][1] = __ffma2_rn(make_float2(wa.z, wa.w), x, acc[s][1]);
            acc[s][2] = __ffma2_rn(make_float2(wb.x, wb.y), x, acc[s][2]);
            acc[s][3] = __ffma2_rn(make_float2(wb.z, wb.w), x, acc[s][3]);
            acc8[s] = fmaf(w8, f, acc8[s]);
          }
        }
      }
    };
    if (slots > 1) sums(std::integral_constant<int, kOutSlots>{});
    else sums(std::integral_constant<int, 1>{});  // a sample's short last tile
#pragma unroll
    for (int s = 0; s < kOutSlots; ++s) {
      const int r = tid + kOutThreads * s;
#pragma unroll
      for (int i = 0; i < kTaps / 2; ++i) {
        s_p[2 * i][r] = acc[s][i].x;
        s_p[2 * i + 1][r] = acc[s][i].y;
      }
      s_p[kTaps - 1][r] = acc8[s];
    }
    __syncthreads();  // the rows are read and the sums in place
    if (tid == 0 && t + (int)gridDim.x < n_tiles) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // after the tile's reads
      load(t + gridDim.x);
    }
#pragma unroll
    for (int s = 0; s < kOutSlots; ++s) {
      const int q = tid + kOutThreads * s;
      if (q < kOutTile && l0 + q < len) {
        float z = bias;
#pragma unroll
        for (int kk = 0; kk < kTaps; ++kk) z += s_p[kk][q + kk];
        logit[(size_t)b * len + l0 + q] = z;
      }
    }
  }
}

// Weighted BCE with logits, mean over B L: loss_i = pw y softplus(-z) + (1-y) softplus(z);
// dlogit_i = (pw y (sigmoid(z) - 1) + (1 - y) sigmoid(z)) / (B L).
__global__ void __launch_bounds__(256) bce_kernel(const float* logit, const float* label, float* dlogit,
                                                  float* loss, int n, float pos_weight) {
  __shared__ float red[8];
  float acc = 0.f;
  const float inv = 1.f / (float)n;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float z = logit[i], y = label[i];
    const float sp_pos = fmaxf(z, 0.f) + log1pf(expf(-fabsf(z)));  // softplus(z)
    const float sp_neg = sp_pos - z;                                // softplus(-z)
    acc += pos_weight * y * sp_neg + (1.f - y) * sp_pos;
    const float sg = 1.f / (1.f + expf(-z));
    dlogit[i] = (pos_weight * y * (sg - 1.f) + (1.f - y) * sg) * inv;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    atomicAdd(loss, s * inv);
  }
}

// Backward of the last layer in one pass over a5 (two kernels read it twice before: 128 x
// 4,096, 52 + 46 -> 35 us): its input gradient
//   da5[b][l][ci] = (a5 > 0) * sum_kk W6[kk][ci] dlogit[b][l - kk + 4]
// and this CTA's part of its weight and bias gradients
//   dW6[kk][ci] = sum_p a5[p][ci] dlogit[p - kk + 4], db6 = sum_p dlogit[p],
// which need the same nine logit gradients around a row. Thread = (4-channel chunk, run of 8
// consecutive positions of one sample): its 9 x 4 weights and 9 x 4 sums as packed FP32
// pairs, the 16 logit gradients around the run in registers, the run's eight 8-byte chunks
// of a5 fetched at once; 16 threads cover a position's row. The runs' sums are added in a
// fixed order at the end.
constexpr int kBwdRun = 8, kBwdThreads = 128, kBwdRuns = kBwdThreads / 16;
constexpr int kDwOutN = kTaps * kC + 1;  // dW6 then db6
__global__ void __launch_bounds__(kBwdThreads, 3) conv_out_bwd_kernel(const float* dlogit, const float* w6,
                                                                      const __nv_bfloat16* a5, __nv_bfloat16* da5,
                                                                      float* partial, int batch, int len) {
  __shared__ float s_red[kBwdThreads / 32][16][kTaps * 4 + 1];
  const int c4 = threadIdx.x & 15;
  float2 w[kTaps][2], g[kTaps][2];
#pragma unroll
  for (int kk = 0; kk < kTaps; ++kk) {
    const float4 v = *reinterpret_cast<const float4*>(w6 + kk * kC + 4 * c4);
    w[kk][0] = make_float2(v.x, v.y);
    w[kk][1] = make_float2(v.z, v.w);
    g[kk][0] = g[kk][1] = make_float2(0.f, 0.f);
  }
  float db = 0.f;
  const long long total = (long long)batch * len;  // a multiple of 128: a run stays in one sample
  for (long long p0 = ((long long)blockIdx.x * kBwdRuns + (threadIdx.x >> 4)) * kBwdRun; p0 < total;
       p0 += (long long)gridDim.x * kBwdRuns * kBwdRun) {
    const int l0 = (int)(p0 % len);
    uint2 av[kBwdRun];
#pragma unroll
    for (int j = 0; j < kBwdRun; ++j) av[j] = reinterpret_cast<const uint2*>(a5 + (p0 + j) * kC)[c4];
    float d[kBwdRun + kTaps - 1];  // d[j] = dlogit[l0 - 4 + j], zero outside the sample
#pragma unroll
    for (int j = 0; j < kBwdRun + kTaps - 1; j += 4) {
      const int ll = l0 - kTaps / 2 + j;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (ll >= 0 && ll < len) v = *reinterpret_cast<const float4*>(dlogit + p0 - kTaps / 2 + j);
      d[j] = v.x; d[j + 1] = v.y; d[j + 2] = v.z; d[j + 3] = v.w;
    }
#pragma unroll
    for (int j = 0; j < kBwdRun; ++j) {
      const float2 x0 = make_float2(__uint_as_float(av[j].x << 16), __uint_as_float(av[j].x & 0xffff0000u));
      const float2 x1 = make_float2(__uint_as_float(av[j].y << 16), __uint_as_float(av[j].y & 0xffff0000u));
      float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll
      for (int kk = 0; kk < kTaps; ++kk) {  // dlogit[l - kk + 4] with l = l0 + j
        const float2 dd = make_float2(d[j + kTaps - 1 - kk], d[j + kTaps - 1 - kk]);
        s0 = __ffma2_rn(w[kk][0], dd, s0);
        s1 = __ffma2_rn(w[kk][1], dd, s1);
        g[kk][0] = __ffma2_rn(x0, dd, g[kk][0]);
        g[kk][1] = __ffma2_rn(x1, dd, g[kk][1]);
      }
      __nv_bfloat162 o[2];
      o[0] = __floats2bfloat162_rn(x0.x > 0.f ? s0.x : 0.f, x0.y > 0.f ? s0.y : 0.f);
      o[1] = __floats2bfloat162_rn(x1.x > 0.f ? s1.x : 0.f, x1.y > 0.f ? s1.y : 0.f);
      reinterpret_cast<uint2*>(da5 + (p0 + j) * kC)[c4] = *reinterpret_cast<const uint2*>(o);
      db += d[j + kTaps / 2];
    }
  }
  // the warp's two runs, then the warps in order
#pragma unroll
  for (int kk = 0; kk < kTaps; ++kk) {
    const float v[4] = {g[kk][0].x, g[kk][0].y, g[kk][1].x, g[kk][1].y};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float o = v[e] + __shfl_down_sync(0xffffffffu, v[e], 16);
      if ((threadIdx.x & 16) == 0) s_red[threadIdx.x >> 5][c4][kk * 4 + e] = o;
    }
  }
  const float dbo = db + __shfl_down_sync(0xffffffffu, db, 16);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5][0][kTaps * 4] = dbo;
  __syncthreads();
  float* out = partial + (size_t)blockIdx.x * kDwOutN;
  for (int i = threadIdx.x; i < kDwOutN; i += kBwdThreads) {
    const int kk = i / kC, ci = i % kC;  // i = 576: the bias gradient
    float v = 0.f;
    for (int q = 0; q < kBwdThreads / 32; ++q)
      v += i < kTaps * kC ? s_red[q][ci >> 2][kk * 4 + (ci & 3)] : s_red[q][0][kTaps * 4];
    out[i] = v;
  }
}

// Gradient outputs of a 64 -> 64 layer: dW [9][64][64] then db [64].
constexpr int kDwOut = kTaps * kC * kC + kC;

// Weight and bias gradients of a 64 -> 64 layer on the tensor cores:
//   dW[kk][co][ci] = sum_p dY[p][co] X[p + kk - 4][ci] = sum_q dY[q - kk + 4][co] X[q][ci],
// a GEMM over positions q (K) with M = output channel and N = input channel. A
// CTA walks 128-position tiles (K = 128 each) and accumulates all nine taps in
// TMEM across its tiles. Both operands are read "MN-major" from the channels-last rows as
// TMA lays them out with the 128-byte swizzle: a 128-byte row holds 64 M (or N) elements
// of one k, eight rows an atom, so a shift along positions is a descriptor that starts
// that many rows later (the swizzle follows the address bits). Taps are paired in M =
// 128: the descriptor's second block of 64 M elements starts one row (128 bytes) after the
// first, which is the same dY rows one tap earlier, so rows 0..63 hold tap kk + 1 and rows
// 64..127 tap kk from one copy of dY. Pairs (1,0), (3,2), (5,4), (7,6), (8,7): 5 x 64 TMEM
// columns; the second tap 7 is discarded.
// Warp roles: warp 0 loads each tile with two TMA boxes (dY: 136 rows from the tile's row
// - 4; X: its 128 rows; zeros outside the sample) into a ring of 6 buffers; one thread of
// warp 1 issues the tile's 40 MMAs and commits them to the buffer's empty barrier; warps
// 2-3 add the tile's own dY rows into the bias gradient (thread = 8 output channels of every
// eighth row) and arrive on the same barrier. After the last tile all four warps read the accumulators
// (lane quarter = warp) into the CTA's partial sums.
// Bound by the MMAs' shared-memory reads (6 KB each, 48 cycles at 128 bytes a cycle: 25 us
// of 128 x 4,096); with 16-byte planes per 8 channels a tile took 24 boxes of 16-byte rows
// and 52 KB, and the copies held it: 58 -> 43 us.
constexpr int kWgTile = 128;                     // positions per tile (K)
constexpr int kWgRows = kWgTile + kTaps - 1;     // 136 staged dY rows
constexpr int kWgABytes = kWgRows * kC * 2;      // 17,408 B = 17 swizzle atoms
constexpr int kWgBBytes = kWgTile * kC * 2;      // 16,384 B = 16 atoms
constexpr int kWgStage = kWgABytes + kWgBBytes;  // 33,792 B per stage
constexpr int kWgStages = 6;
constexpr int kWgPairs = 5;
constexpr int kWgThreads = 128;
constexpr int kWgSmem = kWgStages * kWgStage + 1024;  // with up to 1 KB to align it: one CTA per SM (512 TMEM columns)

// Bias gradient of a tile by two warps: thread v of 64 takes the 8 channels of chunk v & 7
// in rows r0 + (v >> 3) + 8 j of the swizzled tile of 128-byte rows (16-byte loads: 128
// wavefronts a tile, half of what one channel per thread took).
__device__ __forceinline__ void add_rows_sw128(const unsigned char* tile, int r0, int v, float2 (&sum)[4]) {
#pragma unroll 4
  for (int j = 0; j < kWgTile / 8; ++j) {
    const int r = r0 + (v >> 3) + 8 * j;
    const uint4 u = *reinterpret_cast<const uint4*>(tile + r * 128 + ((((v ^ r) & 7)) << 4));
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      sum[e] = __fadd2_rn(sum[e], make_float2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u)));
  }
}
// The 64 threads' sums to the 64 channels' totals, the row groups in order (thread v: channel v).
__device__ __forceinline__ float bias_total(float (&s_db)[8][kC], int v) {
  float t = 0.f;
#pragma unroll
  for (int g = 0; g < 8; ++g) t += s_db[g][v];
  return t;
}
__device__ __forceinline__ void bias_store(float (&s_db)[8][kC], int v, const float2 (&sum)[4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    s_db[v >> 3][8 * (v & 7) + 2 * e] = sum[e].x;
    s_db[v >> 3][8 * (v & 7) + 2 * e + 1] = sum[e].y;
  }
}

__global__ void __launch_bounds__(kWgThreads, 1)
    wgrad64_tc_kernel(const __grid_constant__ CUtensorMap dymap, const __grid_constant__ CUtensorMap xmap,
                      float* partial, int32_t* err, int batch, int len) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);  // the swizzle's period
  __shared__ __align__(8) uint64_t full[kWgStages], empty[kWgStages], fin;
  __shared__ uint32_t tmem_base;
  __shared__ int s_fail;
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int tiles_per_sample = len / kWgTile;
  const int n_tiles = batch * tiles_per_sample;
  const int n_my = (int)blockIdx.x < n_tiles ? (n_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  if (tid == 0) {
    for (int k = 0; k < kWgStages; ++k) {
      mbar_init(&full[k], 1);
      mbar_init(&empty[k], 3);  // the MMAs' commit and the two bias warps
    }
    mbar_init(&fin, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(&tmem_base, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  bool ok = true;
  float2 db[4] = {};
  __shared__ float s_db[8][kC];

  if (warp == 0 && lane == 0) {  // TMA producer
    int issued = 0;
    for (int i = 0; i < n_my && ok; ++i) {
      const int s = i % kWgStages;
      if (i >= kWgStages) ok = mbar_wait(&empty[s], (uint32_t)((i / kWgStages - 1) & 1), kWaitLimit);
      if (!ok) break;
      const int t = (int)blockIdx.x + i * (int)gridDim.x;
      const int b = t / tiles_per_sample, q0 = (t % tiles_per_sample) * kWgTile;
      unsigned char* buf = smem + s * kWgStage;
      mbar_arrive_expect_tx(&full[s], (uint32_t)kWgStage);
      tma_load3(buf, &dymap, 0, q0 - kTaps / 2, b, &full[s]);
      tma_load3(buf + kWgABytes, &xmap, 0, q0, b, &full[s]);
      issued = i + 1;
    }
    for (int i = issued > kWgStages ? issued - kWgStages : 0; i < issued; ++i)  // every copy has landed
      if (!mbar_wait(&full[i % kWgStages], (uint32_t)((i / kWgStages) & 1), kWaitLimit)) ok = false;
  } else if (warp == 1 && lane == 0) {  // MMA issuer: M = 128, N = 64, A and B MN-major
    const uint32_t idesc = idesc_bf16_f32(128, kC) | (1u << 15) | (1u << 16);
    for (int i = 0; i < n_my && ok; ++i) {
      const int s = i % kWgStages;
      ok = mbar_wait(&full[s], (uint32_t)((i / kWgStages) & 1), kWaitLimit);
      if (!ok) break;
      tc_fence_after();
      const uint64_t ad0 = smem_desc_mn_sw128(smem_u32(smem + s * kWgStage), 128u);
      const uint64_t bd0 = smem_desc_mn_sw128(smem_u32(smem + s * kWgStage + kWgABytes), 128u);
#pragma unroll
      for (int ks = 0; ks < kWgTile / 16; ++ks) {
#pragma unroll
        for (int g = 0; g < kWgPairs; ++g) {  // consecutive MMAs into different accumulators
          // staged dY row of position i under tap kk: i - kk + 8; the first block's tap is
          // 2 g + 1 (8 in the last pair), the second's one less
          const int row = g < kWgPairs - 1 ? kTaps - 2 - 2 * g : 0;
          mma_bf16(tmem + (uint32_t)(g * kC), ad0 + (uint64_t)(((row + 16 * ks) * 128) >> 4),
                   bd0 + (uint64_t)((16 * ks * 128) >> 4), idesc, i > 0 || ks > 0);
        }
      }
      mma_commit(&empty[s]);  // the buffer is free once these MMAs have read it
    }
    mma_commit(&fin);  // every MMA issued has completed before TMEM is read or freed (bounded)
    if (!mbar_wait(&fin, 0u, kWaitLimit)) ok = false;
  } else if (warp >= 2) {  // bias gradient: the tile's own dY rows (staged rows 4 .. 131)
    for (int i = 0; i < n_my && ok; ++i) {
      const int s = i % kWgStages;
      ok = mbar_wait(&full[s], (uint32_t)((i / kWgStages) & 1), kWaitLimit);
      ok = __all_sync(0xffffffffu, ok) != 0;
      if (!ok) break;
      add_rows_sw128(smem + s * kWgStage, kTaps / 2, tid - 64, db);
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[s]);
    }
  }
  if (warp == 2 || warp == 3) bias_store(s_db, tid - 64, db);
  if (!ok) atomicExch(&s_fail, 1);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  float* out = partial + (size_t)blockIdx.x * kDwOut;
  if (!s_fail && n_my > 0) {
    // TMEM lane m = 32 warp + lane: output channel m % 64 of tap 2g + 1 (m < 64) or 2g, in
    // the last pair 8 or (discarded) 7; column = input channel
    const int m = 32 * warp + lane;
    const int co = m & (kC - 1);
#pragma unroll 1
    for (int g = 0; g < kWgPairs; ++g) {
      const int kk = g < kWgPairs - 1 ? 2 * g + (m < kC ? 1 : 0) : (m < kC ? kTaps - 1 : kTaps);
#pragma unroll
      for (int c0 = 0; c0 < kC; c0 += 16) {
        float v[16];
        tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(g * kC + c0), v);
        if (kk < kTaps) {
          float4* dst = reinterpret_cast<float4*>(out + (kk * kC + co) * kC + c0);
          dst[0] = make_float4(v[0], v[1], v[2], v[3]);
          dst[1] = make_float4(v[4], v[5], v[6], v[7]);
          dst[2] = make_float4(v[8], v[9], v[10], v[11]);
          dst[3] = make_float4(v[12], v[13], v[14], v[15]);
        }
      }
    }
    if (warp >= 2) out[kTaps * kC * kC + (tid - 64)] = bias_total(s_db, tid - 64);
  } else if (!s_fail) {  // no tiles: zero partial sums
    for (int i = tid; i < kDwOut; i += kWgThreads) out[i] = 0.f;
  } else if (tid == 0) {
    atomicOr(err, kErrMmaWait);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// Weight and bias gradients of the first layer on the tensor cores:
//   dW1[kk][co][ci] = sum_q dY[q][co] X[q + kk - 4][ci], db1[co] = sum_q dY[q][co],
// a GEMM over positions with M = (tap, input channel) and N = output channel. X's rows
// (CI channels, 12 bytes: no TMA) are staged by pairs of warps as one 16-byte core-matrix row
// of 8 channels (the last two zero) per position, MN-major without swizzle: the core
// matrices of the next 8 M elements start 16 bytes on, which is the next position, that
// is the next tap, so one MMA of M = 128 covers all nine taps (the rows of taps 9 .. 15 are
// computed and discarded) and a tile takes 8 MMAs. dY comes as in the 64 -> 64 layers'
// kernel. Eight TMEM accumulators take the tiles in turn and are added in FP32 at the end,
// so that each one's running sum is an eighth as long. Bound by reading dY (67 MB of 128 x
// 4,096); 54 FP32 FMAs per value on the CUDA cores took 92 -> 22 us.
constexpr int kWiRows = kWgTile + 16;                    // staged X rows: taps 0 .. 15 of the last position
constexpr int kWiABytes = 3072;                          // 144 x 16 B, to a multiple of 1,024
constexpr int kWiStage = kWgBBytes + kWiABytes;          // dY (128 rows), X
constexpr int kWiStages = 8, kWiAcc = 8;
constexpr int kWiStagers = 4;                            // pairs of warps that stage X, tiles in turn
constexpr int kWiThreads = 128 + 64 * kWiStagers;
constexpr int kWiSmem = kWiStages * kWiStage + 1024;
constexpr int kDwIn = kTaps * kC * QLP_CNN_IN_CH + kC;   // dW1 then db1

__global__ void __launch_bounds__(kWiThreads, 1)
    wgrad_in_tc_kernel(const __grid_constant__ CUtensorMap dymap, const __nv_bfloat16* x, float* partial, int32_t* err,
                       int batch, int len) {
  constexpr int CI = QLP_CNN_IN_CH;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  __shared__ __align__(8) uint64_t full[kWiStages], empty[kWiStages], fin;
  __shared__ uint32_t tmem_base;
  __shared__ int s_fail;
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int tiles_per_sample = len / kWgTile;
  const int n_tiles = batch * tiles_per_sample;
  const int n_my = (int)blockIdx.x < n_tiles ? (n_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  if (tid == 0) {
    for (int k = 0; k < kWiStages; ++k) {
      mbar_init(&full[k], 3);   // the TMA producer and the two staging warps
      mbar_init(&empty[k], 3);  // the MMAs' commit and the two bias warps
    }
    mbar_init(&fin, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(&tmem_base, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  bool ok = true;
  float2 db[4] = {};
  __shared__ float s_db[8][kC];

  if (warp == 0 && lane == 0) {  // TMA producer
    int issued = 0;
    for (int i = 0; i < n_my && ok; ++i) {
      const int s = i % kWiStages;
      if (i >= kWiStages) ok = mbar_wait(&empty[s], (uint32_t)((i / kWiStages - 1) & 1), kWaitLimit);
      if (!ok) break;
      const int t = (int)blockIdx.x + i * (int)gridDim.x;
      mbar_arrive_expect_tx(&full[s], (uint32_t)kWgBBytes);
      tma_load3(smem + s * kWiStage, &dymap, 0, (t % tiles_per_sample) * kWgTile, t / tiles_per_sample, &full[s]);
      issued = i + 1;
    }
    // every copy has landed: the staging warps' arrivals come too unless they gave up, and
    // they give up only with an error already raised
    for (int i = issued > kWiStages ? issued - kWiStages : 0; i < issued; ++i)
      if (!mbar_wait(&full[i % kWiStages], (uint32_t)((i / kWiStages) & 1), kWaitLimit)) ok = false;
  } else if (warp == 1 && lane == 0) {  // MMA issuer: M = 128, N = 64, A and B MN-major
    const uint32_t idesc = idesc_bf16_f32(128, kC) | (1u << 15) | (1u << 16);
    for (int i = 0; i < n_my && ok; ++i) {
      const int s = i % kWiStages;
      ok = mbar_wait(&full[s], (uint32_t)((i / kWiStages) & 1), kWaitLimit);
      if (!ok) break;
      tc_fence_after();
      const uint64_t ad0 = smem_desc(smem_u32(smem + s * kWiStage + kWgBBytes), 128u, 16u);
      const uint64_t bd0 = smem_desc_mn_sw128(smem_u32(smem + s * kWiStage), 128u);
      const uint32_t dst = tmem + (uint32_t)((i % kWiAcc) * kC);
#pragma unroll
      for (int ks = 0; ks < kWgTile / 16; ++ks)
        mma_bf16(dst, ad0 + (uint64_t)((16 * ks * 16) >> 4), bd0 + (uint64_t)((16 * ks * 128) >> 4), idesc,
                 i >= kWiAcc || ks > 0);
      mma_commit(&empty[s]);
    }
    mma_commit(&fin);
    if (!mbar_wait(&fin, 0u, kWaitLimit)) ok = false;
  } else if (warp == 2 || warp == 3) {  // bias gradient
    for (int i = 0; i < n_my && ok; ++i) {
      const int s = i % kWiStages;
      ok = mbar_wait(&full[s], (uint32_t)((i / kWiStages) & 1), kWaitLimit);
      ok = __all_sync(0xffffffffu, ok) != 0;
      if (!ok) break;
      add_rows_sw128(smem + s * kWiStage, 0, tid - 64, db);
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[s]);
    }
  } else if (warp >= 4) {  // X rows l0 - 4 .. l0 + 139 as 16-byte records, zeros outside the sample
    const int v0 = (tid - 128) & 63;
    for (int i = (warp - 4) >> 1; i < n_my && ok; i += kWiStagers) {
      const int s = i % kWiStages;
      const int t = (int)blockIdx.x + i * (int)gridDim.x;
      const int b = t / tiles_per_sample, q0 = (t % tiles_per_sample) * kWgTile;
      uint4 v[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) {  // fetched before the wait for the buffer
        const int r = v0 + 64 * j, l = q0 - kTaps / 2 + r;
        uint32_t h[CI] = {};
        if (r < kWiRows && l >= 0 && l < len) {
          const unsigned short* src = reinterpret_cast<const unsigned short*>(x) + ((size_t)b * len + l) * CI;
#pragma unroll
          for (int c = 0; c < CI; ++c) h[c] = __ldg(src + c);
        }
        v[j] = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, 0u);
      }
      if (i >= kWiStages) ok = mbar_wait(&empty[s], (uint32_t)((i / kWiStages - 1) & 1), kWaitLimit);
      ok = __all_sync(0xffffffffu, ok) != 0;
      if (!ok) break;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int r = v0 + 64 * j;
        if (r < kWiRows) *reinterpret_cast<uint4*>(smem + s * kWiStage + kWgBBytes + r * 16) = v[j];
      }
      fence_proxy_async_smem();  // the records become visible to the tensor core
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[s]);
    }
  }
  if (warp == 2 || warp == 3) bias_store(s_db, tid - 64, db);
  if (!ok) atomicExch(&s_fail, 1);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  float* out = partial + (size_t)blockIdx.x * kDwIn;
  if (!s_fail && n_my > 0) {
    // TMEM lane m = 8 tap + input channel, column = output channel; the accumulators in order
    const int m = 32 * warp + lane, kk = m >> 3, ci = m & 7;
    if (warp < 3) {  // taps 0 .. 11
      const int n_acc = n_my < kWiAcc ? n_my : kWiAcc;
#pragma unroll 1
      for (int c0 = 0; c0 < kC; c0 += 16) {
        float sum[16];
#pragma unroll 1
        for (int g = 0; g < n_acc; ++g) {
          float v[16];
          tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(g * kC + c0), v);
#pragma unroll
          for (int e = 0; e < 16; ++e) sum[e] = g == 0 ? v[e] : sum[e] + v[e];
        }
        if (kk < kTaps && ci < CI)
#pragma unroll
          for (int e = 0; e < 16; ++e) out[(kk * kC + c0 + e) * CI + ci] = sum[e];
      }
    }
    if (warp == 2 || warp == 3) out[kTaps * kC * CI + (tid - 64)] = bias_total(s_db, tid - 64);
  } else if (!s_fail) {
    for (int i = tid; i < kDwIn; i += kWiThreads) out[i] = 0.f;
  } else if (tid == 0) {
    atomicOr(err, kErrMmaWait);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// out[o] = sum over the CTA partials g of partial[g][o]: a CTA takes 32 outputs, its 8
// warps the partials g = w, w + 8, ... (in that order), then warp 0 adds the 8 sums in
// warp order (a fixed order: deterministic).
constexpr int kRedSlices = 8;
__global__ void __launch_bounds__(32 * kRedSlices) reduce_partials_kernel(const float* partial, int n_parts,
                                                                         int n_out, float* out) {
  __shared__ float red[kRedSlices][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int o = blockIdx.x * 32 + lane;
  float s = 0.f;
  if (o < n_out)
#pragma unroll 8
    for (int g = w; g < n_parts; g += kRedSlices) s += partial[(size_t)g * n_out + o];
  red[w][lane] = s;
  __syncthreads();
  if (w == 0 && o < n_out) {
    float t = 0.f;
    for (int k = 0; k < kRedSlices; ++k) t += red[k][lane];
    out[o] = t;
  }
}
static void launch_reduce_partials(const float* partial, int n_parts, int n_out, float* out, cudaStream_t s) {
  reduce_partials_kernel<<<(n_out + 31) / 32, 32 * kRedSlices, 0, s>>>(partial, n_parts, n_out, out);
}

// Adam with the decay rates and their complements given separately (each the
// FP32 rounding of its exact decimal value: 1 - 0.999f is 1.3e-5 away from 0.001)
// and the bias corrections c1 = 1 - b1^t, c2 = 1 - b2^t computed in FP64 by the host.
__global__ void adam_kernel(float* p, const float* g, float* m, float* v, int n, float lr, float b1, float b2,
                            float omb1, float omb2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + omb1 * gi;
  const float vi = b2 * v[i] + omb2 * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// ------------------------------------------------------------------ launchers

// CTAs of a small-layer kernel: a few per SM, each walking its share of the tiles
static int tile_grid(long long tiles, int per_sm) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return (int)(tiles < (long long)per_sm * sms ? tiles : (long long)per_sm * sms);
}

int launch_conv_in(const void* x0, const float* w1, const float* b1, void* a1, int batch, int len, void* s) {
  if (batch <= 0 || len % kSmTile != 0) return batch <= 0 ? 0 : (int)cudaErrorInvalidValue;
  conv_in_kernel<<<tile_grid((long long)batch * (len / kInTile), 3), kInThreads, 0, (cudaStream_t)s>>>(
      static_cast<const __nv_bfloat16*>(x0), w1, b1, static_cast<__nv_bfloat16*>(a1), batch, len);
  return (int)cudaGetLastError();
}

int launch_conv_out(const void* a5, const float* w6, const float* b6, float* logit, int32_t* err, int batch, int len,
                    void* s) {
  if (batch <= 0 || len % kSmTile != 0) return batch <= 0 ? 0 : (int)cudaErrorInvalidValue;
  alignas(64) CUtensorMap amap;
  cudaError_t e = cudaFuncSetAttribute(conv_out_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kOutSmem);
  if (e == cudaSuccess) e = map_rows64(&amap, a5, batch, len, kOutRows / 2);
  if (e != cudaSuccess) return (int)e;
  conv_out_kernel<<<tile_grid((long long)batch * ((len + kOutTile - 1) / kOutTile), 2), kOutThreads, kOutSmem,
                    (cudaStream_t)s>>>(amap, w6, b6, logit, err, batch, len);
  return (int)cudaGetLastError();
}

int launch_bce(const float* logit, const float* label, float* dlogit, float* loss, int n, float pw, void* s) {
  const int blocks = (n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024;
  bce_kernel<<<blocks, 256, 0, (cudaStream_t)s>>>(logit, label, dlogit, loss, n, pw);
  return (int)cudaGetLastError();
}

// Input gradient of the last layer (BF16 da5) and its weight and bias gradients (out: dW6
// [9][64], db6), the CTAs' parts summed in order. `partial` holds at least one 64 -> 64
// layer's part per 128 positions (or per SM), 64 times what 64 positions need here.
int launch_conv_out_bwd(const float* dlogit, const float* w6, const void* a5, void* da5, float* partial, float* out,
                        int batch, int len, void* s) {
  if (batch <= 0) return 0;
  if (len % kSmTile != 0) return (int)cudaErrorInvalidValue;
  const int parts = tile_grid((long long)batch * len / (kBwdRuns * kBwdRun), 3);
  conv_out_bwd_kernel<<<parts, kBwdThreads, 0, (cudaStream_t)s>>>(dlogit, w6, static_cast<const __nv_bfloat16*>(a5),
                                                                  static_cast<__nv_bfloat16*>(da5), partial, batch,
                                                                  len);
  launch_reduce_partials(partial, parts, kDwOutN, out, (cudaStream_t)s);
  return (int)cudaGetLastError();
}

int wgrad64_parts(int batch, int len) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int tiles = batch * (len / kWgTile);
  return tiles < sms ? tiles : sms;
}

// CTAs of a weight-gradient launch, at most wgrad64_parts: the fewest that leave the longest
// one as few tiles as one per SM would, since every CTA writes its partial gradients (148 KB
// for a 64 -> 64 layer) and the reduction reads them all. 180 tiles: 90 CTAs of two tiles
// instead of 152 of one or two.
static int wgrad_grid(int batch, int len) {
  const int tiles = batch * (len / kWgTile), most = wgrad64_parts(batch, len);
  const int each = (tiles + most - 1) / most;
  return (tiles + each - 1) / each;
}

// dW and db of a 64 -> 64 layer on the tensor cores (len a multiple of 128):
// per-CTA partial sums, then their sum into out[kDwOut]
int launch_wgrad64(const void* dy, const void* x, float* partial, float* out, int32_t* err, int batch, int len,
                   void* s) {
  if (batch <= 0) return 0;
  const int parts = wgrad_grid(batch, len);
  alignas(64) CUtensorMap dymap, xmap;
  cudaError_t e = cudaFuncSetAttribute(wgrad64_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmem);
  if (e == cudaSuccess) e = map_rows64(&dymap, dy, batch, len, kWgRows);
  if (e == cudaSuccess) e = map_rows64(&xmap, x, batch, len, kWgTile);
  if (e != cudaSuccess) return (int)e;
  wgrad64_tc_kernel<<<parts, kWgThreads, kWgSmem, (cudaStream_t)s>>>(dymap, xmap, partial, err, batch, len);
  launch_reduce_partials(partial, parts, kDwOut, out, (cudaStream_t)s);
  return (int)cudaGetLastError();
}

// dW1 [9][64][QLP_CNN_IN_CH] and db1 of the first layer (dy BF16 [B][L][64], x BF16
// [B][L][QLP_CNN_IN_CH]) into out
int launch_wgrad_in(const void* dy, const void* x, float* partial, float* out, int32_t* err, int batch, int len,
                    void* s) {
  if (batch <= 0) return 0;
  if (len % kWgTile != 0) return (int)cudaErrorInvalidValue;
  const int parts = wgrad_grid(batch, len);
  alignas(64) CUtensorMap dymap;
  cudaError_t e = cudaFuncSetAttribute(wgrad_in_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWiSmem);
  if (e == cudaSuccess) e = map_rows64(&dymap, dy, batch, len, kWgTile);
  if (e != cudaSuccess) return (int)e;
  wgrad_in_tc_kernel<<<parts, kWiThreads, kWiSmem, (cudaStream_t)s>>>(dymap, static_cast<const __nv_bfloat16*>(x),
                                                                      partial, err, batch, len);
  launch_reduce_partials(partial, parts, kDwIn, out, (cudaStream_t)s);
  return (int)cudaGetLastError();
}

int launch_adam(float* p, const float* g, float* m, float* v, int n, float lr, float b1, float b2, float omb1,
                float omb2, float eps, float c1, float c2, void* s) {
  adam_kernel<<<(n + 255) / 256, 256, 0, (cudaStream_t)s>>>(p, g, m, v, n, lr, b1, b2, omb1, omb2, eps, c1, c2);
  return (int)cudaGetLastError();
}

}  // namespace qlp
