// S-step of Algorithm 1 (eq. raw_lss): S_t = P_Omega(X - L_t) with Omega
// the nonzero subset of the k largest |X - L_t|, ties by ascending linear index.
//
// One pass over X rebuilds R = X - U diag(sigma) V^T tile by tile (k_resid.cu).  Magnitudes
// are compared through their float bit patterns (monotone for |R| >= 0).  In
// candidate mode the pass keeps every entry whose key reaches a threshold
// guessed from the previous iteration; in full mode it builds a 4096-bin
// histogram of the top 12 key bits instead.  A short radix select over the
// candidates (3 key digits, then up to 4 index digits for ties) yields the
// exact k-th key and the tie cut, and the emit step writes S as COO.
#include <cuda_bf16.h>

#include <cuda_fp16.h>

#include "godec_internal.cuh"
#include "select_util.cuh"

namespace godec {

namespace {

__device__ __forceinline__ unsigned key_of(float v) { return __float_as_uint(v) & 0x7fffffffu; }

__device__ double block_sum_double(double v) {
  __shared__ double ws[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) ws[warp] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < nw; ++w) t += ws[w];
  return t;   // valid in thread 0
}

// --------------------------------------------------------------------------------------
// Pass over a dense residual R (hard threshold without L): the histogram of the top key bits
// (full mode) or the candidates with key >= guess, staged per block and written with one
// global atomic per full buffer.  Eight columns per thread and step as two 16-byte loads.
// Bound: 4 m n bytes read (4001 x 2999: 24 -> 9 us a pass against the tiled kernel with the
// general X - U V^T arithmetic that this replaces).
// --------------------------------------------------------------------------------------
constexpr int TH_THREADS = 512, TH_STAGE = 2048;

__global__ void __launch_bounds__(TH_THREADS)
k_thresh_pass(const float* __restrict__ R, int64_t m, int64_t n, int64_t ldr, int pass, Ctl* ctl,
              unsigned* __restrict__ cand_key, long long* __restrict__ cand_idx, float* __restrict__ cand_val,
              unsigned long long cand_cap, long long k) {
  if (ctl->abort) return;
  const int mode = ctl->plan[pass];
  if (mode == PASS_NONE) return;
  const unsigned guess = max(ctl->guess[pass], 1u);   // exact zeros are never candidates
  __shared__ unsigned hist[kHistBins];                // candidate mode: the staged linear indices (low words)
  __shared__ float sval[TH_STAGE];
  __shared__ unsigned s_cnt;
  __shared__ unsigned long long s_base;
  static_assert(TH_STAGE <= kHistBins, "staged indices fit the histogram");
  const int tid = threadIdx.x;
  if (mode == PASS_FULL)
    for (int b = tid; b < kHistBins; b += TH_THREADS) hist[b] = 0u;
  if (tid == 0) s_cnt = 0u;
  __syncthreads();
  const int64_t per = (n + 7) / 8, total = m * per;
  bool bad = false;
  // every thread takes the same number of steps (the staging has block-wide barriers)
  for (int64_t e0 = (int64_t)blockIdx.x * TH_THREADS; e0 < total; e0 += (int64_t)gridDim.x * TH_THREADS) {
    const int64_t e = e0 + tid;
    float v[8];
    int64_t i = 0, j = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = 0.f;
    if (e < total) {
      i = e / per;
      j = (e - i * per) * 8;
      const float* r = R + i * ldr + j;   // rows and R are 16-byte aligned
      if (j + 8 <= n) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(r)), b = __ldg(reinterpret_cast<const float4*>(r) + 1);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (j + u < n) v[u] = r[u];
      }
    }
    if (mode == PASS_FULL) {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const unsigned key = key_of(v[u]);
        bad |= key >= 0x7f800000u;
        if (key) atomicAdd(&hist[key >> kD1Shift], 1u);
      }
      continue;
    }
    unsigned cm = 0u;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const unsigned key = key_of(v[u]);
      bad |= key >= 0x7f800000u;
      if (key >= guess) cm |= 1u << u;
    }
    // stage; when a step's candidates do not fit, the buffer goes out first (a step has at
    // most 8 TH_THREADS of them, taken TH_STAGE at a time)
    const int cnt = __popc(cm);
    unsigned tot;
    const unsigned off = block_excl_scan((unsigned)cnt, &tot);
    for (unsigned lo = 0; lo < tot; lo += TH_STAGE) {
      const unsigned have = s_cnt, part = min(tot - lo, (unsigned)TH_STAGE);
      if (have + part > TH_STAGE) {
        __syncthreads();
        if (tid == 0) s_base = atomicAdd(&ctl->cand_count, (unsigned long long)have);
        __syncthreads();
        for (unsigned q = tid; q < have; q += TH_THREADS)
          if (s_base + q < cand_cap) {
            cand_key[s_base + q] = key_of(sval[q]);
            cand_idx[s_base + q] = (long long)hist[q];
            cand_val[s_base + q] = sval[q];
          }
        __syncthreads();
        if (tid == 0) s_cnt = 0u;
        __syncthreads();
      }
      const unsigned at = s_cnt;
      unsigned pos = off;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (cm & (1u << u)) {
          if (pos >= lo && pos < lo + part) {
            sval[at + pos - lo] = v[u];
            hist[at + pos - lo] = (unsigned)(i * n + j + u);   // m n < 2^32
          }
          ++pos;
        }
      __syncthreads();
      if (tid == 0) s_cnt = at + part;
      __syncthreads();
    }
  }
  __syncthreads();
  if (mode == PASS_FULL) {
    for (int b = tid; b < kHistBins; b += TH_THREADS)
      if (hist[b]) atomicAdd(&ctl->hist[b], hist[b]);
  } else if (s_cnt) {
    if (tid == 0) s_base = atomicAdd(&ctl->cand_count, (unsigned long long)s_cnt);
    __syncthreads();
    for (unsigned q = tid; q < s_cnt; q += TH_THREADS)
      if (s_base + q < cand_cap) {
        cand_key[s_base + q] = key_of(sval[q]);
        cand_idx[s_base + q] = (long long)hist[q];
        cand_val[s_base + q] = sval[q];
      }
  }
  if (bad) ctl->nonfinite = 1;
  after_pass<TH_THREADS>(ctl, pass, mode, k, cand_cap);
}

// Bits of the selected candidates (bitmap of m n bits, clear before).
__global__ void __launch_bounds__(256)
k_mark(Ctl* ctl, const unsigned* __restrict__ cand_key, const long long* __restrict__ cand_idx,
       unsigned long long cand_cap, unsigned* __restrict__ bits) {
  if (ctl->abort || !ctl->ready || ctl->need <= 0) return;
  const unsigned long long ncand = min(ctl->cand_count, cand_cap);
  const unsigned tau = ctl->tau_key;
  const unsigned long long cut = ctl->idx_cut;
  for (unsigned long long c = (unsigned long long)blockIdx.x * 256 + threadIdx.x; c < ncand;
       c += (unsigned long long)gridDim.x * 256) {
    const unsigned key = cand_key[c];
    if (key < tau) continue;
    const unsigned long long idx = (unsigned long long)cand_idx[c];
    if (key > tau || idx <= cut) atomicOr(&bits[idx >> 5], 1u << (idx & 31));
  }
}

// --------------------------------------------------------------------------------------
// The support in ascending order from its bitmap: the entries' positions are ranks in the
// bitmap, so no sort is needed.  A block takes OB_WORDS words; per group of eight words
// (256 bits, one 32-byte sector) the write pass also leaves the rank of its first bit.
// Bound: m n / 8 bytes read twice, 12 bytes written per entry, and one random read and write
// per entry where the values come from an unordered list (10^4 x 10^4, 10^6 entries: 300 us
// as eight passes of a radix sort before).
// --------------------------------------------------------------------------------------
constexpr int OB_THREADS = 256, OB_WORDS = kOrderWords;

__global__ void __launch_bounds__(OB_THREADS)
k_bits_count(const unsigned* __restrict__ bits, long long words, unsigned* __restrict__ blocksum) {
  const long long w0 = (long long)blockIdx.x * OB_WORDS;
  unsigned c = 0;
#pragma unroll
  for (int k = 0; k < OB_WORDS / OB_THREADS / 4; ++k) {   // words: a multiple of 32, OB_WORDS of 1024
    const long long w = w0 + 4 * ((long long)k * OB_THREADS + threadIdx.x);
    if (w < words) {
      const uint4 q = __ldg(reinterpret_cast<const uint4*>(bits + w));
      c += __popc(q.x) + __popc(q.y) + __popc(q.z) + __popc(q.w);
    }
  }
  unsigned tot;
  block_excl_scan(c, &tot);
  if (threadIdx.x == 0) blocksum[blockIdx.x] = tot;
}

// blocksum := its exclusive prefix sums (one block of 1024 threads); *total = their sum.
__global__ void __launch_bounds__(1024) k_bits_scan(unsigned* __restrict__ blocksum, int nblk, unsigned* total) {
  unsigned carry = 0;
  for (int b = 0; b < nblk; b += 1024) {
    const int i = b + threadIdx.x;
    const unsigned v = i < nblk ? blocksum[i] : 0u;
    unsigned tot;
    const unsigned x = block_excl_scan(v, &tot);
    if (i < nblk) blocksum[i] = carry + x;
    carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

// idx[rank] = linear index of every set bit, below cap; with R, val[rank] = R there; rank0
// (nullable) the rank of each 256-bit group's first bit.
__global__ void __launch_bounds__(OB_THREADS)
k_bits_write(const unsigned* __restrict__ bits, long long words, const unsigned* __restrict__ blocksum,
             long long* __restrict__ idx, float* __restrict__ val, long long cap, const float* __restrict__ R, int64_t n,
             int64_t ldr, unsigned* __restrict__ rank0) {
  constexpr int WT = OB_WORDS / OB_THREADS;   // words per thread, consecutive
  const long long w0 = (long long)blockIdx.x * OB_WORDS + (long long)threadIdx.x * WT;
  unsigned w[WT];
  unsigned c = 0;
#pragma unroll
  for (int k = 0; k < WT; k += 4) {
    const uint4 q = w0 + k < words ? __ldg(reinterpret_cast<const uint4*>(bits + w0 + k)) : make_uint4(0, 0, 0, 0);
    w[k] = q.x;
    w[k + 1] = q.y;
    w[k + 2] = q.z;
    w[k + 3] = q.w;
    c += __popc(q.x) + __popc(q.y) + __popc(q.z) + __popc(q.w);
  }
  unsigned tot;
  long long pos = (long long)blocksum[blockIdx.x] + block_excl_scan(c, &tot);
  const float ninv = 1.f / (float)n;
#pragma unroll
  for (int k = 0; k < WT; ++k) {
    if (rank0 && ((w0 + k) & 7) == 0 && w0 + k < words) rank0[(w0 + k) >> 3] = (unsigned)pos;
    unsigned x = w[k];
    while (x) {
      const int b = __ffs(x) - 1;
      x &= x - 1u;
      const long long id = (w0 + k) * 32 + b;
      if (pos < cap) {
        idx[pos] = id;
        if (R) {
          long long i, j;
          split_idx(id, n, ninv, i, j);
          val[pos] = R[i * ldr + j];
        }
      }
      ++pos;
    }
  }
}

// val[rank of idx[e]] = v[e].
__global__ void __launch_bounds__(256)
k_val_order(const long long* __restrict__ idx, const float* __restrict__ v, long long nnz,
            const unsigned* __restrict__ bits, const unsigned* __restrict__ rank0, float* __restrict__ val) {
  const long long e = (long long)blockIdx.x * 256 + threadIdx.x;
  if (e >= nnz) return;
  const long long id = idx[e], w = id >> 5, g = w >> 3;
  const uint4 a = __ldg(reinterpret_cast<const uint4*>(bits + 8 * g)), b = __ldg(reinterpret_cast<const uint4*>(bits + 8 * g) + 1);
  const unsigned q[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  unsigned r = __ldg(rank0 + g);
  const int k = (int)(w & 7);
#pragma unroll
  for (int u = 0; u < 8; ++u) r += u < k ? __popc(q[u]) : (u == k ? __popc(q[u] & ((1u << (id & 31)) - 1u)) : 0u);
  val[r] = v[e];
}

// --------------------------------------------------------------------------------------
// Radix select rounds over the candidates.  Round 0..2: key digits (bits 30..19, 18..7,
// 6..0), largest first.  Rounds 3..6: 12-bit digits of the linear index of the ties,
// smallest first.  The last block to finish scans the histogram.
// --------------------------------------------------------------------------------------
constexpr int SEL_THREADS = 512, SEL_BLOCK = 2 * SEL_THREADS;

__device__ __forceinline__ void round_digit(int round, int* shift, int* bits) {
  switch (round) {
    case 0: *shift = 19; *bits = 12; break;
    case 1: *shift = 7; *bits = 12; break;
    case 2: *shift = 0; *bits = 7; break;
    default: *shift = 12 * (6 - round); *bits = 12; break;   // 36, 24, 12, 0
  }
}

__global__ void __launch_bounds__(SEL_THREADS)
k_select_round(SelectArgs a) {
  Ctl* ctl = a.ctl;
  // all of the state in one go: a load behind each test would be a round trip to L2 of its own
  const int aborted = ctl->abort, ready = ctl->ready, key_done = ctl->key_done, idx_done = ctl->idx_done;
  const long long need0 = ctl->need;
  const unsigned long long ncand = min(ctl->cand_count, a.cand_cap);
  const unsigned long long kp = ctl->key_prefix;   // key bits above this digit
  const unsigned long long ip = ctl->idx_prefix;
  const unsigned tau = ctl->tau_key;
  const int round = a.round;
  if (aborted || !ready || need0 <= 0) return;
  if (round < 3 ? key_done : (!key_done || idx_done)) return;
  // Only as many blocks as have SEL_BLOCK candidates each: every block costs a clear of its
  // histogram, a merge of it by global atomics and an arrival.  (With the same rule in the emit
  // kernel and two launches fewer: 500 x 500 at k = 12500 0.215 -> 0.204 ms an iteration.)
  const unsigned active = (unsigned)min((unsigned long long)gridDim.x, max(1ull, (ncand + SEL_BLOCK - 1) / SEL_BLOCK));
  if (blockIdx.x >= active) return;
  __shared__ unsigned h[kHistBins];
  const int tid = threadIdx.x;
  for (int b = tid; b < kHistBins; b += SEL_THREADS) h[b] = 0u;
  __syncthreads();
  int shift, bits;
  round_digit(round, &shift, &bits);
  for (unsigned long long c = (unsigned long long)blockIdx.x * SEL_THREADS + tid; c < ncand;
       c += (unsigned long long)active * SEL_THREADS) {
    unsigned key = a.cand_key[c];
    if (round < 3) {
      if (round > 0 && (key >> (shift + bits)) != kp) continue;
      atomicAdd(&h[(key >> shift) & ((1u << bits) - 1)], 1u);
    } else {
      if (key != tau) continue;
      unsigned long long idx = (unsigned long long)a.cand_idx[c];
      if ((idx >> (shift + bits)) != ip) continue;
      atomicAdd(&h[(idx >> shift) & ((1ull << bits) - 1)], 1u);
    }
  }
  __syncthreads();
  for (int b = tid; b < (1 << bits); b += SEL_THREADS)
    if (h[b]) atomicAdd(&ctl->sel_hist[b], h[b]);
  __threadfence();
  __shared__ unsigned s_last;
  __syncthreads();
  if (tid == 0) s_last = (atomicAdd(&ctl->done_ctas, 1u) == active - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // last block: copy the global histogram, clear it, find the digit
  for (int b = tid; b < kHistBins; b += SEL_THREADS) {
    h[b] = (b < (1 << bits)) ? atomicExch(&ctl->sel_hist[b], 0u) : 0u;
  }
  __syncthreads();
  // find bin (single warp-free approach: each thread scans a slice)
  __shared__ int s_bin;
  __shared__ unsigned long long s_before;
  __shared__ unsigned s_in;
  const int nb = 1 << bits;
  const bool from_top = round < 3;
  const unsigned long long need = (unsigned long long)need0;
  const int per = (nb + SEL_THREADS - 1) / SEL_THREADS;
  unsigned loc = 0;
  for (int o = tid * per; o < min(nb, tid * per + per); ++o) loc += h[from_top ? nb - 1 - o : o];
  unsigned tot;
  unsigned excl = block_excl_scan(loc, &tot);
  if (tid == 0) s_bin = -1;
  __syncthreads();
  unsigned long long run = excl;
  for (int o = tid * per; o < min(nb, tid * per + per); ++o) {
    int b = from_top ? nb - 1 - o : o;
    unsigned c = h[b];
    if (run < need && run + c >= need) { s_bin = b; s_before = run; s_in = c; }
    run += c;
  }
  __syncthreads();
  if (tid == 0) {
    ctl->done_ctas = 0u;
    const int b = s_bin;
    if (b < 0) {            // inconsistent counts: cannot happen for valid candidates
      ctl->abort = 1;
      ctl->need_bigger_cand = 1;
    } else if (round < 3) {
      ctl->key_prefix = (kp << bits) | (unsigned)b;
      ctl->need = (long long)(need - s_before);
      if (round == 2) {
        ctl->tau_key = (unsigned)ctl->key_prefix;
        ctl->key_done = 1;
        if ((unsigned long long)ctl->need == s_in) {   // every tie is taken
          ctl->idx_cut = ~0ull;
          ctl->idx_done = 1;
        }
      }
    } else {
      ctl->idx_prefix = (ip << bits) | (unsigned)b;
      ctl->need = (long long)(need - s_before);
      if (round == 6) {
        ctl->idx_cut = ctl->idx_prefix;
        ctl->idx_done = 1;
      }
    }
  }
}

// --------------------------------------------------------------------------------------
// Emit S_t, objective, and next-iteration bookkeeping (last block).
// --------------------------------------------------------------------------------------
constexpr int EMIT_THREADS = 256, EMIT_ITEMS = 8;

__global__ void __launch_bounds__(EMIT_THREADS)
k_emit(EmitArgs a) {
  Ctl* ctl = a.ctl;
  const int tid = threadIdx.x;
  // the state in one go, as in the select rounds
  const int aborted = ctl->abort, ready = ctl->ready, nb = ctl->cur ^ 1;
  const long long need = ctl->need, k_req = ctl->k_req;
  const unsigned long long ncand = (need > 0) ? min(ctl->cand_count, a.cand_cap) : 0ull;
  const unsigned tau = ctl->tau_key;
  const unsigned long long cut = ctl->idx_cut;
  if (aborted || !ready) return;
  const unsigned long long tile = (unsigned long long)EMIT_THREADS * EMIT_ITEMS;
  const unsigned active = (unsigned)min((unsigned long long)gridDim.x, max(1ull, (ncand + tile - 1) / tile));
  if (blockIdx.x >= active) return;
  long long* Sidx = a.S_idx[nb];
  float* Sval = a.S_val[nb];
  unsigned* bits = a.sbits ? a.sbits + (size_t)nb * (size_t)a.sbits_words : nullptr;   // clear until now
  double dsum = 0.0;
  __shared__ unsigned long long s_base;
  for (unsigned long long t0 = (unsigned long long)blockIdx.x * tile; t0 < ncand;
       t0 += (unsigned long long)active * tile) {
    unsigned sel = 0;
    unsigned cnt = 0;
    unsigned key[EMIT_ITEMS];
    long long idx[EMIT_ITEMS];
    float val[EMIT_ITEMS];
#pragma unroll
    for (int j = 0; j < EMIT_ITEMS; ++j) {   // all loads in flight before the first store
      const unsigned long long c = t0 + (unsigned long long)j * EMIT_THREADS + tid;
      key[j] = c < ncand ? a.cand_key[c] : 0u;
      idx[j] = c < ncand ? a.cand_idx[c] : 0ll;
      val[j] = c < ncand ? a.cand_val[c] : 0.f;
    }
#pragma unroll
    for (int j = 0; j < EMIT_ITEMS; ++j) {
      unsigned long long c = t0 + (unsigned long long)j * EMIT_THREADS + tid;
      if (c < ncand) {
        const bool s = key[j] > tau || (key[j] == tau && (unsigned long long)idx[j] <= cut);
        if (s) { sel |= 1u << j; ++cnt; }
        else dsum += (double)val[j] * (double)val[j];
      }
    }
    unsigned total;
    unsigned off = block_excl_scan(cnt, &total);
    if (tid == 0) s_base = total ? atomicAdd(&ctl->nnz_new, (unsigned long long)total) : 0ull;
    __syncthreads();
    unsigned long long pos = s_base + off;
#pragma unroll
    for (int j = 0; j < EMIT_ITEMS; ++j) {
      if (sel & (1u << j)) {
        if (pos < (unsigned long long)k_req) {   // never past the S buffers
          Sidx[pos] = idx[j];
          Sval[pos] = val[j];
          if (bits) atomicOr(&bits[idx[j] >> 5], 1u << (idx[j] & 31));
        }
        ++pos;
      }
    }
  }
  double bs = block_sum_double(dsum);
  if (tid == 0 && bs != 0.0) atomicAdd(&ctl->sumsq_cand_out, bs);
  __threadfence();
  __shared__ unsigned s_last;
  __syncthreads();
  if (tid == 0) s_last = (atomicAdd(&ctl->done_ctas2, 1u) == active - 1);
  __syncthreads();
  if (!s_last || tid != 0) return;
  __threadfence();
  // ---- last thread of the last block: commit the iteration (loads first, then stores) ----
  const double in_sum = __ldcg(&ctl->sumsq_noncand), out_sum = __ldcg(&ctl->sumsq_cand_out), nx2 = ctl->normX2;
  const unsigned long long got = __ldcg(&ctl->nnz_new);
  const double tol = ctl->tol;
  const long long nnz0 = ctl->nnz_cur, keff = ctl->k_eff;
  const int iter = ctl->iter, parity = ctl->slot_parity, passes = ctl->passes_run;
  const double obj = in_sum + out_sum;
  const double rel = nx2 > 0.0 ? obj / nx2 : 0.0;
  ctl->obj = obj;
  ctl->rel_err = rel;
  ctl->nnz_prev = nnz0;
  if (got > (unsigned long long)keff) {   // selection inconsistent: keep the old S
    ctl->need_bigger_cand = 1;
    ctl->abort = 1;
    ctl->done_ctas2 = 0u;
    return;
  }
  ctl->nnz_cur = (long long)got;
  ctl->cur = nb;
  ctl->iter = iter + 1;
  ctl->slot_parity = parity ^ 1;          // normalisers written during this iteration become current
  ctl->last_passes = passes;
  if (tol >= 0.0 && rel <= tol) {
    ctl->converged = 1;
    ctl->abort = 1;
  }
  // threshold guess for the next S-step: two digit-1 bins below the k-th key
  const int gb = (int)(tau >> kD1Shift) - 2;
  const unsigned guess = need > 0 ? (gb > 0 ? ((unsigned)gb << kD1Shift) : 1u) : 0u;
  ctl->next_guess = guess;
  // reset per-iteration state
  ctl->done_ctas2 = 0u;
  ctl->nnz_new = 0ull;
  ctl->plan[0] = guess ? PASS_CAND : PASS_FULL;
  ctl->plan[1] = PASS_NONE;
  ctl->plan[2] = PASS_NONE;
  ctl->guess[0] = guess;
  ctl->ready = 0;
  ctl->cand_count = 0ull;
  ctl->sumsq_noncand = 0.0;
  ctl->sumsq_full = 0.0;
  ctl->sumsq_cand_out = 0.0;
  ctl->k_eff = k_req;
  ctl->key_prefix = 0ull;
  ctl->idx_prefix = 0ull;
  ctl->key_done = 0;
  ctl->idx_done = 0;
  ctl->tau_key = 0u;
  ctl->idx_cut = 0ull;
  ctl->need = 0;
}

// Z := X on the entries of S_{t-1}, then Z := X - S_t on the entries of S_t.
// Z holds (X - S) zscale[0], split.  An entry whose scaled magnitude reaches kZRange
// flags range_err; the next product sees the flag, abandons that iteration before
// reading Z, and the caller rebuilds Z (setting abort here would cut this update short
// in blocks that have not started yet).
__device__ __forceinline__ void z_write(const EmitArgs& a, long long i, long long j, float z, float zs, bool& bad) {
  const float v = z * zs;
  bad |= fabsf(v) >= kZRange && isfinite(v);
  zs_put(static_cast<__half*>(a.Z), i, j, a.ldz, v);
}

__device__ __forceinline__ void z_flag(Ctl* ctl, bool bad) {
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) ctl->range_err = 1;
}

// One entry per thread (the grid covers the largest possible support, k).  The update
// also runs after the iteration that met the stop test (converged sets abort only to
// stop the iterations after it), so Z always matches the committed S.
__device__ __forceinline__ bool z_skip(const Ctl* ctl) { return ctl->abort && !ctl->converged; }

// The update of Z from S_{t-1} to S_t, one launch: entries of Omega_{t-1}
// that left the support get Z = X back, and Z = X - S_t on Omega_t.  The two sets are
// disjoint (the restore skips every entry the emit marked in the bitmap of Omega_t), so
// thread e does entry e of both lists.  The bitmap of Omega_{t-1} is cleared on the way
// (every set bit of it belongs to an entry of Omega_{t-1}, so each such entry simply
// zeroes its word).
__global__ void k_z_update(EmitArgs a) {
  Ctl* ctl = a.ctl;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (z_skip(ctl)) return;
  const long long np = ctl->nnz_prev, nc = ctl->nnz_cur;
  if ((long long)blockIdx.x * blockDim.x >= (np > nc ? np : nc)) return;
  const float zs = a.zscale ? a.zscale[0] : 1.f;
  const float ninv = 1.f / (float)a.n;
  const int cb = ctl->cur;
  bool bad = false;
  if (e < np) {
    const long long idx = a.S_idx[cb ^ 1][e];
    const unsigned* now = a.sbits ? a.sbits + (size_t)cb * (size_t)a.sbits_words : nullptr;
    if (!now || !((__ldcg(&now[idx >> 5]) >> (idx & 31)) & 1u)) {
      long long i, j;
      split_idx(idx, a.n, ninv, i, j);
      z_write(a, i, j, a.X[i * a.ldx + j], zs, bad);
    }
    if (a.sbits) a.sbits[(size_t)(cb ^ 1) * (size_t)a.sbits_words + (size_t)(idx >> 5)] = 0u;
  }
  if (e < nc) {
    const long long idx = a.S_idx[cb][e];
    long long i, j;
    split_idx(idx, a.n, ninv, i, j);
    const float v = a.S_val[cb][e];
    z_write(a, i, j, a.X[i * a.ldx + j] - v, zs, bad);
    if (a.Sd) a.Sd[i * a.ldz + j] = v;
  }
  z_flag(ctl, bad);
}

// Z = (X - S) s_Z on the entries of the committed S (vals null), or their X - S into vals.
__global__ void k_z_apply(EmitArgs a, float* vals) {
  Ctl* ctl = a.ctl;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= ctl->nnz_cur) return;
  const int cb = ctl->cur;
  long long i, j;
  split_idx(a.S_idx[cb][e], a.n, 1.f / (float)a.n, i, j);
  const float z = a.X[i * a.ldx + j] - a.S_val[cb][e];
  if (vals) vals[e] = z;
  else zs_put(static_cast<__half*>(a.Z), i, j, a.ldz, z * a.zscale[0]);
}

// The support bitmap of the committed S (bitmap ctl->cur) from its index list, one entry
// per thread; both bitmaps were cleared before (after an S-step cut short).
__global__ void k_sbits_rebuild(unsigned* sbits, long long words, long long* S0, long long* S1, const Ctl* ctl) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int cb = ctl->cur;
  if (e >= ctl->nnz_cur) return;
  const long long idx = (cb ? S1 : S0)[e];
  atomicOr(&sbits[(size_t)cb * (size_t)words + (size_t)(idx >> 5)], 1u << (idx & 31));
}

// Start of a selection over a dense matrix alone, from a zeroed control block.
__global__ void k_start_select(Ctl* ctl, long long k) {
  ctl->plan[0] = PASS_FULL;
  ctl->k_req = ctl->k_eff = k;
  ctl->tol = -1.0;
}

// Per-iteration S-step state back to "start of an iteration" (one thread).
__global__ void k_reset_iter(Ctl* ctl) {
  for (int b = threadIdx.x; b < kHistBins; b += blockDim.x) {
    ctl->hist[b] = 0u;
    ctl->sel_hist[b] = 0u;
  }
  if (threadIdx.x != 0) return;
  ctl->plan[0] = ctl->next_guess ? PASS_CAND : PASS_FULL;
  ctl->plan[1] = PASS_NONE;
  ctl->plan[2] = PASS_NONE;
  ctl->guess[0] = ctl->next_guess;
  ctl->guess[1] = ctl->guess[2] = 0u;
  ctl->passes_run = 0;
  ctl->ready = 0;
  ctl->need_bigger_cand = 0;
  ctl->cand_count = 0ull;
  ctl->k_eff = ctl->k_req;
  ctl->sumsq_noncand = ctl->sumsq_full = ctl->sumsq_cand_out = 0.0;
  ctl->done_ctas = ctl->done_ctas2 = 0u;
  ctl->key_prefix = ctl->idx_prefix = 0ull;
  ctl->need = 0;
  ctl->tau_key = 0u;
  ctl->key_done = ctl->idx_done = 0;
  ctl->idx_cut = 0ull;
  ctl->nnz_new = 0ull;
  ctl->rank_drop = 0;
  ctl->abort = 0;
  ctl->nonfinite = 0;
  ctl->chol_fail = 0;
  ctl->converged = 0;
  ctl->alarm = 0;
  ctl->timeout = 0;
}

}  // namespace

void launch_start_select(Ctl* ctl, long long k, cudaStream_t st) { k_start_select<<<1, 1, 0, st>>>(ctl, k); }

void launch_reset_iter(Ctl* ctl, cudaStream_t st) { k_reset_iter<<<1, 256, 0, st>>>(ctl); }

void launch_thresh_pass(const ResidualArgs& a, int nsm, cudaStream_t st) {
  int64_t grid = (a.m * ((a.n + 7) / 8) + TH_THREADS - 1) / TH_THREADS;
  if (grid > 4LL * nsm) grid = 4LL * nsm;
  k_thresh_pass<<<(unsigned)grid, TH_THREADS, 0, st>>>(a.X, a.m, a.n, a.ldx, a.pass, a.ctl, a.cand_key, a.cand_idx,
                                                       a.cand_val, a.cand_cap, a.k);
}

void launch_mark(const SelectArgs& a, unsigned* bits, int nsm, cudaStream_t st) {
  k_mark<<<(unsigned)(4 * nsm), 256, 0, st>>>(a.ctl, a.cand_key, a.cand_idx, a.cand_cap, bits);
}

size_t order_scratch(long long words) {
  return (size_t)((words + OB_WORDS - 1) / OB_WORDS + 1 + words / 8) * sizeof(unsigned);
}

void launch_order(const unsigned* bits, long long words, unsigned* scratch, long long* idx, float* val, long long cap,
                  const float* R, int64_t n, int64_t ldr, const long long* S_idx, const float* S_val, long long nnz,
                  unsigned* total, cudaStream_t st) {
  const int nblk = (int)((words + OB_WORDS - 1) / OB_WORDS);
  unsigned* rank0 = R ? nullptr : scratch + nblk + 1;
  k_bits_count<<<nblk, OB_THREADS, 0, st>>>(bits, words, scratch);
  k_bits_scan<<<1, 1024, 0, st>>>(scratch, nblk, total);
  k_bits_write<<<nblk, OB_THREADS, 0, st>>>(bits, words, scratch, idx, val, cap, R, n, ldr, rank0);
  if (!R && nnz > 0) k_val_order<<<(unsigned)((nnz + 255) / 256), 256, 0, st>>>(S_idx, S_val, nnz, bits, rank0, val);
}

void launch_select(SelectArgs a, int nsm, cudaStream_t st) {
  for (int d = 0; d < kNumSelRounds; ++d) {
    // an index digit that is zero for every index is not looked at (500 x 500: two of seven
    // launches, 10^4 x 10^4: one, about 1.7 us each)
    if (d >= 3 && d < 6 && 12 * (6 - d) >= a.idx_bits) continue;
    a.round = d;
    k_select_round<<<(unsigned)(2 * nsm), SEL_THREADS, 0, st>>>(a);
  }
}

void launch_emit(const EmitArgs& a, int nsm, cudaStream_t st) {
  k_emit<<<(unsigned)(2 * nsm), EMIT_THREADS, 0, st>>>(a);
}

void launch_sbits_rebuild(unsigned* sbits, long long words, long long* const S_idx[2], const Ctl* ctl,
                          long long max_nnz, cudaStream_t st) {
  const long long nb = (max_nnz + 255) / 256;
  k_sbits_rebuild<<<(unsigned)(nb > 0 ? nb : 1), 256, 0, st>>>(sbits, words, S_idx[0], S_idx[1], ctl);
}

void launch_z_apply(const EmitArgs& a, cudaStream_t st) {
  k_z_apply<<<(unsigned)(a.max_nnz > 0 ? (a.max_nnz + 255) / 256 : 1), 256, 0, st>>>(a, nullptr);
}

void launch_z_values(const EmitArgs& a, float* out, cudaStream_t st) {
  k_z_apply<<<(unsigned)(a.max_nnz > 0 ? (a.max_nnz + 255) / 256 : 1), 256, 0, st>>>(a, out);
}

void launch_z_update(const EmitArgs& a, int nsm, cudaStream_t st) {
  (void)nsm;
  const long long nb = (a.max_nnz + 255) / 256;
  const unsigned grid = (unsigned)(nb > 0 ? nb : 1);
  k_z_update<<<grid, 256, 0, st>>>(a);
}

}  // namespace godec
