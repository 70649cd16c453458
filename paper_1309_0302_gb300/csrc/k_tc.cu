// Streaming product on the 5th-generation tensor cores (tcgen05, sm_103a).
//
//   part/out = Zsrc (rows x K, float32, row-major) * B (K x RP)   to float32 accuracy
//
// Two-term float16 split ("2xFP16"): with a power-of-two scale s_Z, each element is
// written x s_Z = h1 + 2^-11 h2, h1 = x s_Z cut to 11 significant bits (exact in
// float16), h2 = fp16((x s_Z - h1) 2^11) rounded to nearest; the
// skinny operand likewise, b s_B = c1 + 2^-11 c2, arrives already split and transposed
// as [c1^T; c2^T] (2 RP x K float16) from the step that produced it.  Then
//   x b s_Z s_B = h1 c1 + 2^-11 (h1 c2 + h2 c1) + O(2^-22),
// the dropped h2 c2 term being the only truncation.  Per 16-wide K step:
//   D[:, 0:2RP] += h1 [c1; c2]^T   and   D[:, RP:RP+RPl] += h2 (rows 0..RPl-1 of [c1; c2])^T,
// RPl = RP rounded up to 16 (the MMA's N granularity): columns RP..2RP-1 receive h2 c1,
// columns beyond 2RP collect a product nobody reads.  The result is
// (D[:, :RP] + 2^-11 D[:, RP:2RP]) / (s_Z s_B).  float16 MMAs run at twice the TF32
// rate with twice the K per instruction.
//
// This kernel serves products with a caller's float32 matrix (k_prod.cu serves the library's
// own split copies).  A copier thread moves each landed 128 x 64 float32 tile of Zsrc from
// shared memory into tensor memory (tcgen05.cp) and frees the shared-memory slot when the
// copy completes; converter warps then scale the tile (s_Z from its exact maximum) and turn
// it into the two packed float16 blocks (h1, h2) in place with TMEM loads and stores.  The
// working warps thus leave the shared-memory load path to the TMA stream.
//
// Work split: the (128-row tile, 64-wide K stage) iteration space is cut into equal
// contiguous ranges, one per persistent CTA ("stream-K"), so every SM streams the same
// number of bytes whatever the tile count.  The tensor core accumulates a chunk of
// kChunk stages in TMEM (double-buffered); the 4 epilogue warps drain each chunk into
// float32 registers, so the tensor core's own accumulation never runs over more than
// kChunk * 64 terms (its additions are not round-to-nearest, and over thousands of
// terms of one sign the bias would show).  At a tile boundary the running sum goes to
// a partial slot.  The last segment of a tile to arrive adds the slots in order
// (deterministic), unscales and writes the rows.
//
// Warps: 0 TMA producer of Zsrc tiles, 1 MMA issuer (and TMEM owner), 2-9 converters
// (two per TMEM lane quarter, one per 32-column half of the tile), 10-13 epilogue,
// 14 TMA producer of the skinny operand, 15 copier.
// TMEM (512 columns): 0-255 two accumulators of 128 columns, 256-447 three stage slots of
// 64 columns (the float32 tile, then per 32-column half 16 columns of packed h1 and 16
// of packed h2).
// Synchronisation per stage: TMA -> afull -> copier (after sfree) -> aempty (slot
// refilled) and cpdone -> converters -> tfull (after the skinny tile's bfull too) -> MMA
// -> sfree -> the stage slot and the skinny TMA slot.  The MMA issuer waits once and
// commits once per stage.
// Every wait is bounded; a CTA that gives up drains, makes the output rows of the tiles it had
// a share of NaN (the calls do not synchronise and have no status to give) and exits.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include "godec_internal.cuh"
#include "tc_util.cuh"

namespace godec {

namespace {

using namespace tc;

constexpr int BM = 128, BK = 64;   // rows per tile, K per stage (4 MMA steps of 16)
constexpr int NA = 5;              // shared-memory slots for Zsrc tiles (TMA ring)
constexpr int NS = 4;              // stage slots: skinny-operand tile in shared memory + converted
                                   // Zsrc tile in TMEM, freed together by one MMA commit
constexpr int kThreads = 512;
constexpr int kConvWarps = 8;
constexpr uint32_t kTmemCols = 512, kTA0 = 256, kTASlot = 64;
constexpr size_t kBoxA = (size_t)BM * 32 * 4;               // one 32-column float32 box, 16 KB
constexpr size_t kStageA = 2 * kBoxA;                       // 32 KB
constexpr size_t kStageB = (size_t)2 * kMaxRP * BK * 2;     // 16 KB (room for 2 x 64 rows of 64 halves)
constexpr size_t kOffA = 0;
constexpr size_t kOffB = kOffA + NA * kStageA;
constexpr size_t kTcSmem = kOffB + NS * kStageB + 1024;     // + alignment slack
constexpr uint32_t kWaitLimit = 1u << 20;
constexpr float kLoScale = 2048.f, kLoInv = 1.f / 2048.f;
#ifndef GODEC_TC_CHUNK
#define GODEC_TC_CHUNK 2
#endif
constexpr int kChunk = GODEC_TC_CHUNK;   // K stages accumulated in TMEM before a drain
static_assert(kTcSmem <= 232448 - 1024, "shared memory of the tensor-core product");

struct TcArgs {
  int64_t rows, K;
  int RP;                   // columns kept (multiple of 8)
  int64_t ks, S;            // K stages per tile, total stages
  int G;                    // CTAs
  int maxseg;
  float* part;              // tiles x maxseg x BM x RP
  unsigned* counters;       // tiles
  float* out;               // rows x oc, oc <= RP
  int oc;
  const float* cscale;      // per-column output factor 1 / s_B (nullable: 1)
  const float* zscale;      // {s_Z, 1 / s_Z} (nullable: 1)
  int* pend;                // G x maxpend: tiles each CTA completes, deferred to its end
  int maxpend;
  uint32_t limit;           // polls after which a wait of the pipeline gives up
  int withhold;             // self-test: the CTA whose matrix loads are not issued (-1: none)
};

__device__ __forceinline__ int64_t cta_of(int64_t g, int64_t S, int G) { return ((g + 1) * (int64_t)G - 1) / S; }

// cvt.rn.f16x2: first source goes to the upper half, so element k sits in bits 0-15.
__device__ __forceinline__ uint32_t pack_h2(float even, float odd) {
  uint32_t d;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(odd), "f"(even));
  return d;
}

// Completion of tile t by its last segment, run by the whole block (u = 0 .. nthr-1): the
// partial slots are added in slot order (deterministic whoever finishes), unscaled and
// written; csc = per-column output factors 1 / s_B, zi = 1 / s_Z.  Consecutive threads take
// consecutive float4s (coalesced), four items each and up to four slots of each in flight.
__device__ void tile_finish(const TcArgs& a, int64_t t, int nseg, int u, int nthr, const float* csc, float zi) {
  const int RP = a.RP, RP4 = RP / 4;
  const int64_t o0 = t * BM;
  const int nrow = (int)(a.rows - o0 < BM ? a.rows - o0 : BM);
  __threadfence();   // the other segments' slots: written before their counter increments
  if (u == 0) a.counters[t] = 0u;
  const float4* part = reinterpret_cast<const float4*>(a.part + t * a.maxseg * (int64_t)BM * RP);
  const int64_t slot4 = (int64_t)BM * RP4;
  const int nitem = nrow * RP4;
  for (int it0 = u; it0 < nitem; it0 += 4 * nthr) {
    float4 acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < nseg; s0 += 4) {
      float4 v[4][4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int it = it0 + q * nthr;
          v[q][k] = (s0 + k < nseg && it < nitem) ? __ldcg(part + (s0 + k) * slot4 + it) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          acc[q].x += v[q][k].x;
          acc[q].y += v[q][k].y;
          acc[q].z += v[q][k].z;
          acc[q].w += v[q][k].w;
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int it = it0 + q * nthr;
      if (it < nitem) {
        const int c = (it % RP4) * 4;
        const float w[4] = {acc[q].x * (csc[c] * zi), acc[q].y * (csc[c + 1] * zi), acc[q].z * (csc[c + 2] * zi),
                            acc[q].w * (csc[c + 3] * zi)};
        float* o = a.out + (o0 + it / RP4) * a.oc + c;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (c + k < a.oc) o[k] = w[k];
      }
    }
  }
}

// One TMA producer loop over this CTA's stages [g0, g1).  Zsrc stages are two
// 32-column float32 boxes (the second is skipped when it starts at or beyond K);
// skinny-operand stages are one 64-column float16 box.
template <bool IS_A>
__device__ void produce(const CUtensorMap* map, unsigned char* ring, int nslot, size_t slot_bytes, uint32_t box_bytes,
                        uint64_t* fullb, uint64_t* emptyb, int64_t g0, int64_t g1, int64_t ks, uint32_t limit,
                        volatile int* s_err) {
  int64_t t = g0 / ks, kst = g0 % ks, issued = 0;
  int s = 0;
  uint32_t ph = 0;
  // Zsrc is streamed once per product and is larger than L2: its lines go first, which
  // leaves L2 to the skinny operand (read by every CTA) and the partial slots
  const uint64_t pol = policy_evict_first();
  for (int64_t g = g0; g < g1 && !*s_err; ++g) {
    if (!mbar_wait(&emptyb[s], ph ^ 1u, limit)) { *s_err = 1; break; }
    unsigned char* dst = ring + (size_t)s * slot_bytes;
    if (IS_A) {
      // both boxes always: columns at and past K are zero-filled
      mbar_expect_tx(&fullb[s], 2 * box_bytes);
      tma_load_2d_hint(dst, map, &fullb[s], (int)(kst * BK), (int)(t * BM), pol);
      tma_load_2d_hint(dst + box_bytes, map, &fullb[s], (int)(kst * BK + 32), (int)(t * BM), pol);
    } else {
      mbar_expect_tx(&fullb[s], box_bytes);
      tma_load_2d(dst, map, &fullb[s], (int)(kst * BK), 0);
    }
    ++issued;
    if (++kst == ks) { kst = 0; ++t; }
    if (++s == nslot) { s = 0; ph ^= 1u; }
  }
  // Every copy issued has landed before the CTA may exit (immediate in the normal case).
  for (int64_t j = (issued > nslot ? issued - nslot : 0); j < issued; ++j)
    if (!mbar_wait(&fullb[(int)(j % nslot)], (uint32_t)((j / nslot) & 1), kWaitLimit)) *s_err = 1;
}

// Warp-uniform bounded wait: lane 0 polls, the warp follows (__syncwarp orders the
// other lanes' later accesses after lane 0's acquire).
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, int lane, uint32_t limit) {
  int ok = 1;
  if (lane == 0) ok = mbar_wait(bar, parity, limit) ? 1 : 0;
  ok = __shfl_sync(0xffffffffu, ok, 0);
  __syncwarp();
  return ok != 0;
}

template <int RPp>
__global__ void __launch_bounds__(kThreads, 1)
k_prod_tc(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, TcArgs a) {
  const uint32_t limit = a.limit;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* sA = sm + kOffA;
  unsigned char* sB = sm + kOffB;
  __shared__ uint64_t afull[NA], aempty[NA], bfull[NS], tfull[NS], sfree[NS], cpdone[NS];
  __shared__ uint64_t accfull[2], accempty[2], mma_done;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int s_err;   // set by any role that gives up; every loop polls it
  __shared__ int s_stop, s_last;   // epilogue-wide decisions, written between two named barriers
  __shared__ int s_npend;   // tiles this CTA completes (listed in a.pend), done at its end
  __shared__ float s_csc[kMaxRP];
  __shared__ float s_zi;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int c = blockIdx.x;
  const int64_t S = a.S, ks = a.ks;
  const int G = a.G;
  const int64_t g0 = (int64_t)c * S / G, g1 = (int64_t)(c + 1) * S / G;
  if (tid == 0) {
    for (int s = 0; s < NA; ++s) {
      mbar_init(&afull[s], 1);
      mbar_init(&aempty[s], 1);   // the copier's commit
    }
    for (int s = 0; s < NS; ++s) {
      mbar_init(&bfull[s], 1);
      mbar_init(&tfull[s], kConvWarps);
      mbar_init(&sfree[s], 1);
      mbar_init(&cpdone[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accfull[b], 1);
      mbar_init(&accempty[b], 4);
    }
    mbar_init(&mma_done, 1);
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base, kTmemCols);
  if (tid == 0) {
    s_err = 0;
    s_npend = 0;
    s_zi = a.zscale ? a.zscale[1] : 1.f;
  }
  if (tid < kMaxRP) s_csc[tid] = (tid < a.RP && a.cscale) ? a.cscale[tid] : 1.f;
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = tmem_base;

  if (warp == 0) {
    // ---------------- TMA producer: Zsrc tiles ----------------
    if (lane == 0 && c != a.withhold)
      produce<true>(&mapA, sA, NA, kStageA, (uint32_t)kBoxA, afull, aempty, g0, g1, ks, limit, &s_err);
  } else if (warp == 14) {
    // ---------------- TMA producer: skinny-operand tiles ----------------
    if (lane == 0)
      produce<false>(&mapB, sB, NS, kStageB, (uint32_t)(2 * a.RP * BK * 2), bfull, sfree, g0, g1, ks, limit,
                     &s_err);
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      const int RP = a.RP;
      const uint32_t id_hi = idesc_f16(BM, 2 * RP), id_lo = idesc_f16(BM, RPp);   // RPp: RP rounded up to 16
      int ch = 0;   // chunks issued by this CTA
      int st = 0;
      uint32_t ph = 0;
      int64_t kst = g0 % ks;
      int64_t g = g0;
      while (g < g1 && !s_err) {
        // this chunk: up to kChunk stages, not past the end of the tile or of the range
        int64_t n = ks - kst;
        if (n > kChunk) n = kChunk;
        if (n > g1 - g) n = g1 - g;
        const int b = ch & 1;
        if (!mbar_wait(&accempty[b], (uint32_t)(((ch >> 1) & 1) ^ 1), limit)) { s_err = 1; break; }
        tc_fence_after();
        const uint32_t dcol = tbase + (uint32_t)(b * 128);
        uint32_t acc = 0;
        for (int64_t e = 0; e < n; ++e) {
          if (!mbar_wait(&tfull[st], ph, limit)) { s_err = 1; break; }
          tc_fence_after();
          const uint64_t db = sdesc_k128(sB + (size_t)st * kStageB);
          // slot columns: [h of K 0..31 | l of K 0..31 | h of K 32..63 | l of K 32..63], 16 each
          const uint32_t aslot = tbase + kTA0 + (uint32_t)st * kTASlot;
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            const uint64_t off = (uint64_t)((kk * 16 * 2) >> 4);   // 32 bytes per 16-wide K step
            const uint32_t ah = aslot + (uint32_t)((kk >> 1) * 32 + (kk & 1) * 8);
            mma_f16_ta(dcol, ah, db + off, id_hi, acc);
            mma_f16_ta(dcol + RP, ah + 16, db + off, id_lo, 1u);
            acc = 1u;
          }
          mma_commit(&sfree[st]);
          if (++st == NS) { st = 0; ph ^= 1u; }
        }
        if (s_err) break;
        mma_commit(&accfull[b]);
        ++ch;
        g += n;
        kst += n;
        if (kst == ks) kst = 0;
      }
      mma_commit(&mma_done);
      if (!mbar_wait(&mma_done, 0, kWaitLimit)) s_err = 1;
    }
  } else if (warp == 15) {
    // ---------------- copier: landed Zsrc stage -> its TMEM stage slot ----------------
    if (lane == 0) {
      int sa = 0, st = 0;
      uint32_t pha = 0, ph = 0;
      int64_t n = 0;
      for (int64_t g = g0; g < g1 && !s_err; ++g) {
        if (!mbar_wait(&afull[sa], pha, limit) || !mbar_wait(&sfree[st], ph ^ 1u, limit)) {
          s_err = 1;
          break;
        }
        tc_fence_after();
        const uint32_t dst = tbase + kTA0 + (uint32_t)st * kTASlot;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const uint64_t d = sdesc_k128(sA + (size_t)sa * kStageA + b * kBoxA);
#pragma unroll
          for (int k = 0; k < 4; ++k) tmem_cp_128x256b(dst + (uint32_t)(b * 32 + k * 8), d + (uint64_t)(2 * k));
        }
        mma_commit(&cpdone[st]);   // the converters may read the slot
        mma_commit(&aempty[sa]);   // the shared-memory slot may be refilled
        ++n;
        if (++sa == NA) { sa = 0; pha ^= 1u; }
        if (++st == NS) { st = 0; ph ^= 1u; }
      }
      // the last copies have finished reading shared memory and writing TMEM
      for (int64_t j = (n > NS ? n - NS : 0); j < n; ++j)
        if (!mbar_wait(&cpdone[(int)(j % NS)], (uint32_t)((j / NS) & 1), kWaitLimit)) s_err = 1;
    }
  } else if (warp < 2 + kConvWarps) {
    // ---------------- converters: float32 stage in TMEM -> packed (h1, h2) in place ----------------
    const int q = (warp - 2) >> 2;              // 32-column half of the tile handled by this warp
    const uint32_t tlane = (uint32_t)((warp & 3) * 32) << 16;   // this warp's TMEM lane quarter
    const float zs = a.zscale ? a.zscale[0] : 1.f;
    int st = 0;
    uint32_t ph = 0;
    for (int64_t g = g0; g < g1; ++g) {
      if (__any_sync(0xffffffffu, s_err != 0)) break;
      if (!warp_wait(&cpdone[st], ph, lane, limit)) {
        if (lane == 0) s_err = 1;
        break;
      }
      tc_fence_after();
      const uint32_t ta = tbase + kTA0 + (uint32_t)st * kTASlot + tlane + (uint32_t)(q * 32);
      float xs[32];
      tmem_ld32(ta, xs);
      uint32_t h[16], l2[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        float x0 = xs[2 * k], x1 = xs[2 * k + 1];
        x0 *= zs;
        x1 *= zs;
        const float h0 = __uint_as_float(__float_as_uint(x0) & 0xFFFFE000u);
        const float h1 = __uint_as_float(__float_as_uint(x1) & 0xFFFFE000u);
        h[k] = pack_h2(h0, h1);
        l2[k] = pack_h2((x0 - h0) * kLoScale, (x1 - h1) * kLoScale);
      }
      tmem_st16(ta, h);
      tmem_st16(ta + 16, l2);
      tmem_wait_st();
      tc_fence_before();
      // the skinny tile of this stage has landed too: the MMA issuer waits on tfull alone
      if (!warp_wait(&bfull[st], ph, lane, limit)) {
        if (lane == 0) s_err = 1;
        break;
      }
      if (lane == 0) mbar_arrive(&tfull[st]);
      if (++st == NS) { st = 0; ph ^= 1u; }
    }
  } else {
    // ---------------- epilogue: TMEM -> running sums -> partial slot, tile completion ----------------
    // The four warps take every decision together (flag written between two named
    // barriers), so no warp can leave while the others wait at a barrier.
    const int et = tid - 32 * (2 + kConvWarps);
    const int q4 = warp & 3;                 // TMEM lane quarter this warp may access
    const int row = q4 * 32 + lane;          // tile row held by this thread
    const uint32_t tlane = (uint32_t)(q4 * 32) << 16;
    int ch = 0, npend = 0;
    int64_t g = g0;
    for (;;) {
      named_sync(1, BM);
      if (et == 0) s_stop = (g >= g1) || s_err;
      named_sync(1, BM);
      if (s_stop) break;
      const int64_t t = g / ks;
      const int64_t tend = ((t + 1) * ks < g1) ? (t + 1) * ks : g1;
      float y[RPp];
#pragma unroll
      for (int l = 0; l < RPp; ++l) y[l] = 0.f;
      bool failed = false;
      for (; g < tend; g = (g + kChunk < tend) ? g + kChunk : tend, ++ch) {
        if (failed) continue;                // keep the loop count; nothing more to read
        const int b = ch & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(&accfull[b], (uint32_t)((ch >> 1) & 1), limit))) {
          if (lane == 0) s_err = 1;
          failed = true;
          continue;
        }
        tc_fence_after();
        const uint32_t taddr = tbase + (uint32_t)(b * 128) + tlane;
#pragma unroll
        for (int c0 = 0; c0 < RPp; c0 += 8) {
          if (c0 < a.RP) {
            float vh[8], vl[8];
            tmem_ld8(taddr + c0, vh);
            tmem_ld8(taddr + a.RP + c0, vl);
#pragma unroll
            for (int l = 0; l < 8; ++l) y[c0 + l] += fmaf(vl[l], kLoInv, vh[l]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&accempty[b]);
      }
      named_sync(1, BM);
      if (et == 0) s_stop = s_err;
      named_sync(1, BM);
      if (s_stop) break;
      const int64_t c_first = cta_of(t * ks, S, G);
      const int nseg = (int)(cta_of((t + 1) * ks - 1, S, G) - c_first + 1);
      const int slot = (int)(c - c_first);
      float* p = a.part + ((t * a.maxseg + slot) * BM + row) * (int64_t)a.RP;
#pragma unroll
      for (int l = 0; l < RPp; l += 4)
        if (l < a.RP) *reinterpret_cast<float4*>(p + l) = make_float4(y[l], y[l + 1], y[l + 2], y[l + 3]);
      __threadfence();
      named_sync(1, BM);
      if (et == 0) s_last = (atomicAdd(&a.counters[t], 1u) == (unsigned)(nseg - 1));
      named_sync(1, BM);
      if (s_last) {
        if (et == 0) {
          if (npend < a.maxpend) a.pend[(int64_t)c * a.maxpend + npend] = (int)t;
          else s_err = 1;   // cannot happen with the host's bound; never skip silently
        }
        ++npend;
      }
    }
    if (et == 0) s_npend = npend;
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tbase, kTmemCols);
  }
  // completions: the whole CTA on each tile whose last segment was this CTA's
  const int np = s_err ? 0 : (s_npend < a.maxpend ? s_npend : a.maxpend);
  for (int k = 0; k < np; ++k) {
    const int64_t t = a.pend[(int64_t)c * a.maxpend + k];
    const int64_t c_first = cta_of(t * ks, S, G);
    const int nseg = (int)(cta_of((t + 1) * ks - 1, S, G) - c_first + 1);
    tile_finish(a, t, nseg, tid, kThreads, s_csc, s_zi);
  }
  if (s_err) poison_tiles(a.out, a.oc, a.rows, g0 / ks, (g1 - 1) / ks, tid, kThreads);
}

// Column c of a row-major rows x RP operand B -> rows c and RP + c of the split
// transposed float16 operand, scaled by the power of two 2^e_c that brings the column's
// largest magnitude into [2^9, 2^10); cscale[c] = 2^-e_c undoes it.  One block per column.
__global__ void k_split_t(const float* __restrict__ B, int64_t rows, int RP, __half* __restrict__ bt2, int64_t ldb,
                          float* __restrict__ cscale, const int* skip) {
  if (block_skip(skip)) return;
  const int col = blockIdx.x;
  __shared__ float red[32];
  __shared__ float s_scale;
  float m = 0.f;
  if (col < RP)
    for (int64_t i = threadIdx.x; i < rows; i += blockDim.x) m = fmaxf(m, fabsf(B[i * RP + col]));
  for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    float mm = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mm = fmaxf(mm, red[w]);
    int e = 0;
    if (mm > 0.f && isfinite(mm)) {
      int ex;
      frexpf(mm, &ex);   // mm in [2^(ex-1), 2^ex)
      e = 10 - ex;
      e = e < -120 ? -120 : (e > 120 ? 120 : e);
    }
    s_scale = ldexpf(1.f, e);
    if (col < RP) cscale[col] = ldexpf(1.f, -e);
  }
  __syncthreads();
  const float sc = s_scale;
  for (int64_t i = threadIdx.x; i < rows; i += blockDim.x) {
    const float v = (col < RP) ? B[i * RP + col] * sc : 0.f;
    const __half c1 = __float2half_rn(v);
    bt2[(int64_t)col * ldb + i] = c1;
    bt2[(int64_t)(RP + col) * ldb + i] = __float2half_rn((v - __half2float(c1)) * kLoScale);
  }
}

// The power of two that brings a maximum (float bits) into [2^(top-1), 2^top): its exponent.
__device__ __forceinline__ int scale_exp(unsigned mx, int top) {
  const float m = __uint_as_float(mx);
  if (!(m > 0.f) || !isfinite(m)) return 0;
  int ex;
  frexpf(m, &ex);   // m in [2^(ex-1), 2^ex)
  const int e = top - ex;
  return e < -120 ? -120 : (e > 120 ? 120 : e);
}

// max |Z| into mx[0] (blocks below gz) and max |B[:, c]| into mx[1 + c] (the others, 256 rows
// of the K x r operand each), atomic maxima of float bits.
__global__ void __launch_bounds__(256)
k_mul_stats(const float* __restrict__ Z, int64_t m, int64_t n, int64_t ldz, int gz, const float* __restrict__ B, int64_t K,
            int r, unsigned* __restrict__ mx) {
  __shared__ unsigned sm[kMaxRP];
  const int tid = threadIdx.x;
  if (tid < kMaxRP) sm[tid] = 0u;
  __syncthreads();
  if ((int)blockIdx.x >= gz) {
    const int64_t r0 = (int64_t)(blockIdx.x - gz) * 256;
    const int cnt = (int)((K - r0 < 256 ? K - r0 : 256) * r);
    const float* b = B + r0 * r;
    for (int e = tid; e < cnt; e += 256) atomicMax(&sm[e % r], __float_as_uint(fmaxf(0.f, fabsf(b[e]))));
    __syncthreads();
    if (tid < r) atomicMax(&mx[1 + tid], sm[tid]);
    return;
  }
  float v = 0.f;
  const int64_t per = (n + 15) / 16, total = m * per;   // runs of 16 columns; rows are 16-byte aligned
  for (int64_t e = (int64_t)blockIdx.x * 256 + tid; e < total; e += (int64_t)gz * 256) {
    const int64_t i = e / per, j = (e - i * per) * 16;
    const float* z = Z + i * ldz + j;
    if (j + 16 <= n) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 q = __ldg(reinterpret_cast<const float4*>(z) + u);
        v = fmaxf(v, fmaxf(fmaxf(fabsf(q.x), fabsf(q.y)), fmaxf(fabsf(q.z), fabsf(q.w))));
      }
    } else {
      for (int u = 0; j + u < n; ++u) v = fmaxf(v, fabsf(z[u]));
    }
  }
  for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((tid & 31) == 0) atomicMax(&sm[0], __float_as_uint(v));
  __syncthreads();
  if (tid == 0) atomicMax(&mx[0], sm[0]);
}

// The split transposed operand (2 RP x ldb halves) of a K x r matrix B from its column maxima
// cmax, 64 rows per block through shared memory (both sides coalesced): column c scaled by the
// power of two that brings its maximum into [2^9, 2^10), cscale[c] undoing it; columns r ..
// RP-1 zero.  zmax (nullable): block 0 also forms zscale = {s, 1/s} from it.
constexpr int SB_ROWS = 64;
__global__ void __launch_bounds__(256)
k_split_b(const float* __restrict__ B, int64_t K, int r, int RP, const unsigned* __restrict__ cmax, __half* __restrict__ bt2,
          int64_t ldb, float* __restrict__ cscale, const unsigned* __restrict__ zmax, float* __restrict__ zscale) {
  __shared__ float t[SB_ROWS][kMaxRP + 1];
  __shared__ float s_sc[kMaxRP];
  const int tid = threadIdx.x;
  const int64_t r0 = (int64_t)blockIdx.x * SB_ROWS;
  const int nr = (int)(K - r0 < SB_ROWS ? K - r0 : SB_ROWS);
  if (tid < RP) {
    const int e = tid < r ? scale_exp(cmax[tid], 10) : 0;
    s_sc[tid] = ldexpf(1.f, e);
    if (blockIdx.x == 0) cscale[tid] = ldexpf(1.f, -e);
  }
  if (blockIdx.x == 0 && tid == 0 && zmax) {
    const int e = scale_exp(zmax[0], 13);
    zscale[0] = ldexpf(1.f, e);
    zscale[1] = ldexpf(1.f, -e);
  }
  for (int e = tid; e < nr * r; e += 256) t[e / r][e % r] = B[r0 * r + e];
  __syncthreads();
  const int row = tid & 63;
  if (row < nr)
    for (int c = tid >> 6; c < RP; c += 4) {
      const float v = c < r ? t[row][c] * s_sc[c] : 0.f;
      const __half c1 = __float2half_rn(v);
      bt2[(int64_t)c * ldb + r0 + row] = c1;
      bt2[(int64_t)(RP + c) * ldb + r0 + row] = __float2half_rn((v - __half2float(c1)) * kLoScale);
    }
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

}  // namespace

// A tensor map over a row-major matrix (rows x cols, row stride ld elements) read in
// boxes of 128 bytes of columns (32 float32 or 64 float16) x box_rows rows with the
// 128-byte swizzle.
static bool make_tmap(void* map, CUtensorMapDataType dt, int esize, const void* base, int64_t rows, int64_t cols,
                      int64_t ld, int box_rows) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * esize};
  cuuint32_t box[2] = {(cuuint32_t)(128 / esize), (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  CUresult r = fn(reinterpret_cast<CUtensorMap*>(map), dt, 2, const_cast<void*>(base), dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}
bool make_tmap_f32(void* map, const float* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  return make_tmap(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, rows, cols, ld, box_rows);
}
bool make_tmap_f16(void* map, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  return make_tmap(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, base, rows, cols, ld, box_rows);
}

bool make_tmap_split(void* map, const void* base, int64_t rows, int64_t ldz, int box_rows) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {64, (cuuint64_t)(ldz / 32), (cuuint64_t)rows};
  cuuint64_t strides[2] = {128, (cuuint64_t)ldz * 4};
  cuuint32_t box[3] = {64, 1, (cuuint32_t)box_rows};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(reinterpret_cast<CUtensorMap*>(map), CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void*>(base), dims, strides,
            box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int tc_rpp(int RP) { return (RP + 15) / 16 * 16; }

void launch_split_t(const float* B, int64_t rows, int RP, void* bt2, int64_t ldb, float* cscale, cudaStream_t st,
                    const int* skip) {
  k_split_t<<<RP, 256, 0, st>>>(B, rows, RP, reinterpret_cast<__half*>(bt2), ldb, cscale, skip);
}

void launch_mul_stats(const float* Z, int64_t m, int64_t n, int64_t ldz, const float* B, int64_t K, int r, unsigned* mx,
                      int nsm, cudaStream_t st) {
  int64_t gz = Z ? (m * ((n + 15) / 16) + 255) / 256 : 0;
  if (gz > 8LL * nsm) gz = 8LL * nsm;
  k_mul_stats<<<(unsigned)(gz + (K + 255) / 256), 256, 0, st>>>(Z, m, n, ldz, (int)gz, B, K, r, mx);
}

void launch_split_b(const float* B, int64_t K, int r, int RP, const unsigned* cmax, void* bt2, int64_t ldb, float* cscale,
                    const unsigned* zmax, float* zscale, cudaStream_t st) {
  k_split_b<<<(unsigned)((K + SB_ROWS - 1) / SB_ROWS), 256, 0, st>>>(B, K, r, RP, cmax, static_cast<__half*>(bt2), ldb,
                                                                    cscale, zmax, zscale);
}

TcGeom tc_geometry(int64_t rows, int64_t K, int nsm) {
  TcGeom g;
  g.tiles = (rows + BM - 1) / BM;
  g.ks = (K + BK - 1) / BK;
  g.S = g.tiles * g.ks;
  // Leave a few SMs without a product CTA: the r x r kernels of the side stream run
  // there instead of holding an SM that a persistent CTA (which needs the whole shared
  // memory) would otherwise wait for.
  const int ncta = nsm > 16 ? nsm - 4 : nsm;
  g.G = (int)(g.S < ncta ? g.S : ncta);
  int maxseg = 1;
  for (int64_t t = 0; t < g.tiles; ++t) {
    const int64_t cf = ((t * g.ks + 1) * g.G - 1) / g.S;
    const int64_t cl = (((t + 1) * g.ks) * g.G - 1) / g.S;
    if (cl - cf + 1 > maxseg) maxseg = (int)(cl - cf + 1);
  }
  g.maxseg = maxseg;
  // tiles meeting one CTA's range (its completions are listed for the end of the kernel)
  const int64_t span = (g.S + g.G - 1) / g.G;
  g.maxpend = (int)((span + g.ks - 1) / g.ks + 1);
  return g;
}

cudaError_t prepare_tc_kernels() {
  cudaError_t e = cudaSuccess;
  for (auto k : {k_prod_tc<16>, k_prod_tc<32>, k_prod_tc<48>, k_prod_tc<64>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmem);
  return e;
}

void launch_prod_tc(const TcLaunch& l, cudaStream_t st) {
  TcArgs a;
  a.rows = l.rows;
  a.K = l.K;
  a.RP = l.RP;
  a.ks = l.geom.ks;
  a.S = l.geom.S;
  a.G = l.geom.G;
  a.maxseg = l.geom.maxseg;
  a.part = l.part;
  a.counters = l.counters;
  a.out = l.out;
  a.oc = l.out_cols ? l.out_cols : l.RP;
  a.cscale = l.cscale;
  a.zscale = l.zscale;
  a.pend = l.pend;
  a.maxpend = l.geom.maxpend;
  a.limit = l.withhold >= 0 ? kTestPolls : kWaitLimit;
  a.withhold = l.withhold;
  const CUtensorMap& A = *reinterpret_cast<const CUtensorMap*>(l.mapA);
  const CUtensorMap& B = *reinterpret_cast<const CUtensorMap*>(l.mapB);
  switch (tc_rpp(l.RP)) {
    case 16: k_prod_tc<16><<<a.G, kThreads, kTcSmem, st>>>(A, B, a); break;
    case 32: k_prod_tc<32><<<a.G, kThreads, kTcSmem, st>>>(A, B, a); break;
    case 48: k_prod_tc<48><<<a.G, kThreads, kTcSmem, st>>>(A, B, a); break;
    default: k_prod_tc<64><<<a.G, kThreads, kTcSmem, st>>>(A, B, a); break;
  }
}

}  // namespace godec
