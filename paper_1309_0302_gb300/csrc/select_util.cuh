// Block-wide scans of the S-step, and the decision at the end of a pass over the residual.
#pragma once

#include "godec_internal.cuh"

namespace godec {

namespace {

// Block-wide exclusive scan of one unsigned per thread (any blockDim multiple of 32).
__device__ unsigned block_excl_scan(unsigned v, unsigned* total) {
  __shared__ unsigned wsum[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  if (warp == 0) {
    unsigned w = lane < nw ? wsum[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      unsigned y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < nw) wsum[lane] = w;
  }
  __syncthreads();
  unsigned before = warp ? wsum[warp - 1] : 0u;
  *total = wsum[nw - 1];
  return before + x - v;
}

// --------------------------------------------------------------------------------------
// End of a pass over R (every thread of every block of NT threads, after its last atomic):
// the last block to arrive decides what the next pass does.  As a kernel of its own this cost
// a launch per pass, three an iteration (500 x 500: 4.9 us of 215 with the gaps; 64 problems
// in one graph: 192 of 2600 launches).  What other blocks changed is read past the L1.
// --------------------------------------------------------------------------------------
// Find the bin holding the `need`-th largest (from_top) or smallest (!from_top) element of a
// histogram of `nb` bins (nb <= 4096).  Returns the bin; *above = elements strictly before it
// in that order, *in_bin = its count.  All threads get the result.
template <int NT>
__device__ int block_find_bin(const unsigned* h, int nb, unsigned long long need, bool from_top,
                              unsigned long long* before, unsigned* in_bin,
                              unsigned long long* total_out) {
  __shared__ int s_bin;
  __shared__ unsigned long long s_before;
  __shared__ unsigned s_in;
  __shared__ unsigned long long s_total;
  const int per = (nb + NT - 1) / NT;
  const int t = threadIdx.x;
  // thread t owns ordered positions [t*per, t*per+per); position o maps to bin
  // from_top ? nb-1-o : o
  unsigned loc = 0;
  for (int o = t * per; o < min(nb, t * per + per); ++o) loc += __ldcg(&h[from_top ? nb - 1 - o : o]);
  unsigned tot32;
  unsigned excl = block_excl_scan(loc, &tot32);
  if (t == 0) { s_bin = -1; s_total = tot32; }
  __syncthreads();
  unsigned long long run = excl;
  for (int o = t * per; o < min(nb, t * per + per); ++o) {
    int b = from_top ? nb - 1 - o : o;
    unsigned c = __ldcg(&h[b]);
    if (run < need && run + c >= need) {
      s_bin = b;
      s_before = run;
      s_in = c;
    }
    run += c;
  }
  __syncthreads();
  *before = s_before;
  *in_bin = s_in;
  *total_out = s_total;
  return s_bin;
}

template <int NT>
__device__ void after_pass(Ctl* ctl, int pass, int mode, long long k, unsigned long long cap) {
  __threadfence();
  __shared__ unsigned s_last_pass;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned go = atomicAdd(&ctl->done_ctas, 1u) == gridDim.x - 1;
    if (go) {
      __threadfence();
      ctl->done_ctas = 0u;
      go = !__ldcg(&ctl->abort);   // by one thread: a wait of this pass that gave up sets it
    }
    s_last_pass = go;
  }
  __syncthreads();
  if (!s_last_pass) return;
  __threadfence();
  const int nonfinite = __ldcg(&ctl->nonfinite);
  const unsigned long long cc = __ldcg(&ctl->cand_count);
  const long long keff0 = __ldcg(&ctl->k_eff);
  const int t = threadIdx.x;
  if (mode == PASS_FULL) {
    unsigned long long before, total;
    unsigned in_bin;
    // total count first (need = 1 finds the top non-empty bin; we only want the total)
    block_find_bin<NT>(ctl->hist, kHistBins, 1ull, true, &before, &in_bin, &total);
    long long keff = (long long)((unsigned long long)k < total ? (unsigned long long)k : total);
    int bin = -1;
    if (keff > 0) bin = block_find_bin<NT>(ctl->hist, kHistBins, (unsigned long long)keff, true,
                                       &before, &in_bin, &total);
    __syncthreads();
    for (int b = t; b < kHistBins; b += NT) ctl->hist[b] = 0u;
    if (t == 0) {
      ctl->k_eff = keff;
      if (nonfinite) {
        ctl->abort = 1;
      } else if (keff == 0) {
        ctl->ready = 1;
        ctl->need = 0;
        ctl->cand_count = 0;
        ctl->sumsq_noncand = __ldcg(&ctl->sumsq_full);
      } else {
        unsigned long long ge = before + in_bin;   // keys in bins >= bin
        if (ge > cap) {
          ctl->need_bigger_cand = 1;
          ctl->abort = 1;
        } else if (pass < 2) {
          ctl->plan[pass + 1] = PASS_CAND;
          unsigned g = (unsigned)bin << kD1Shift;
          ctl->guess[pass + 1] = g ? g : 1u;
          ctl->cand_count = 0;
          ctl->sumsq_noncand = 0.0;
        } else {
          ctl->abort = 1;                          // cannot happen: FULL is never last
        }
      }
    }
  } else if (t == 0) {   // PASS_CAND
    if (nonfinite) {
      ctl->abort = 1;
    } else if (cc <= cap && (long long)cc >= keff0) {
      ctl->ready = 1;
      ctl->need = keff0;
    } else if (pass < 2) {
      ctl->plan[pass + 1] = PASS_FULL;
      ctl->cand_count = 0;
      ctl->sumsq_full = 0.0;
    } else {
      ctl->need_bigger_cand = 1;
      ctl->abort = 1;
    }
  }
  if (t == 0) ctl->passes_run = pass + 1;
}

}  // namespace

}  // namespace godec
