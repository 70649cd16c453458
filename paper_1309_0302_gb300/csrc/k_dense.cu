// Dense form of the low-rank part: L = U diag(sigma) V^T (eq. mlr_app, L = Q1 M^{1/(2q+1)}
// Q2^T, whose factors the L-step keeps).  The iteration never forms L; this kernel is for
// callers that need it as a matrix (the differentiated form's output, a dense loss).
//
// Every entry is one chain of r float32 fmas over l = 0 .. r-1 (the terms (u sigma) v, u sigma
// rounded first).  The tensor cores take two float16 terms per factor and err more: relative to
// 64 bits at 4001 x 2999 6.3e-8 here against 1.09e-7 there at r = 9, 8.0e-8 / 1.07e-7 at r = 16,
// 1.10e-7 / 1.31e-7 at r = 32, 1.36e-7 / 1.52e-7 at r = 50.
//
// A block writes a 128 x 128 tile, a thread 8 x 8 of it as packed pairs of columns (two fmas an
// instruction).  U diag(sigma) and V go through shared memory 32 columns at a time, a lane per
// row (conflict-free stores, 16-byte loads of the factors' rows).  Where L's rows are 16-byte
// aligned a thread's columns are two groups of four (16-byte stores, 256 contiguous bytes a half
// warp); elsewhere they are 16 apart, so that every store instruction still covers whole runs of
// 16 floats.  Bound: 4 m n bytes written up to about r = 16, then the m n r fmas.  A whole call
// (35 us of it beside the kernel), tiles of 64 x 128 and scalar fmas -> this: 10^4 x 10^4 at
// r = 8 129 -> 109 us, r = 24 278 -> 171 us, r = 50 595 -> 283 us; 4001 x 2999 at r = 50
// 106 -> 71 us; 76800 x 1000 at r = 3 92 -> 86 us.  The kernel alone at 10^4 x 10^4, r = 50:
// 252 us (60 us of writes, 135 us of fmas at the full rate).
#include "godec_internal.cuh"
#include "tc_util.cuh"

namespace godec {

namespace {

constexpr int DT = 128, DT_THREADS = 256, DT_K = 32, DT_LD = DT + 4;

template <bool VEC>
__global__ void __launch_bounds__(DT_THREADS, 2)
k_dense(const float* __restrict__ U, const float* __restrict__ sigma, const float* __restrict__ V, int RP, int64_t m,
        int64_t n, int r, float* __restrict__ L, int64_t ldl) {
  __shared__ __align__(16) float su[DT_K][DT_LD], sv[DT_K][DT_LD];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int64_t nbj = (n + DT - 1) / DT;
  const int64_t i0 = (int64_t)(blockIdx.x / nbj) * DT, j0 = (int64_t)(blockIdx.x % nbj) * DT;
  tc::f32x2 acc[8][4] = {};
  for (int l0 = 0; l0 < r; l0 += DT_K) {
    const int w = r - l0 < DT_K ? r - l0 : DT_K;
    if (l0) __syncthreads();
    for (int e = tid; e < DT * ((w + 3) / 4); e += DT_THREADS) {   // RP >= l0 + 4 ceil(w / 4): a multiple of 8
      const int row = e & (DT - 1), g = 4 * (e >> 7);
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
      if (i0 + row < m) a = *reinterpret_cast<const float4*>(U + (i0 + row) * RP + l0 + g);
      if (j0 + row < n) b = *reinterpret_cast<const float4*>(V + (j0 + row) * RP + l0 + g);
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        su[g + q][row] = l0 + g + q < r ? av[q] * sigma[l0 + g + q] : 0.f;
        sv[g + q][row] = bv[q];
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int l = 0; l < w; ++l) {
      const float4 u0 = *reinterpret_cast<const float4*>(&su[l][4 * ty]);
      const float4 u1 = *reinterpret_cast<const float4*>(&su[l][64 + 4 * ty]);
      const float u[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
      tc::f32x2 v[4];
      if (VEC) {
        const ulonglong2 v0 = *reinterpret_cast<const ulonglong2*>(&sv[l][4 * tx]);
        const ulonglong2 v1 = *reinterpret_cast<const ulonglong2*>(&sv[l][64 + 4 * tx]);
        v[0] = v0.x; v[1] = v0.y; v[2] = v1.x; v[3] = v1.y;
      } else {
#pragma unroll
        for (int p = 0; p < 4; ++p) v[p] = tc::pack2(sv[l][tx + 32 * p], sv[l][tx + 32 * p + 16]);
      }
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        const tc::f32x2 uu = tc::pack2(u[a], u[a]);
#pragma unroll
        for (int p = 0; p < 4; ++p) tc::fma2(acc[a][p], uu, v[p]);
      }
    }
  }
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const int64_t i = i0 + (a & 4) * 16 + 4 * ty + (a & 3);
    if (i >= m) continue;
    float* row = L + i * ldl;
    float x[8];
#pragma unroll
    for (int p = 0; p < 4; ++p) tc::unpack2(acc[a][p], x[2 * p], x[2 * p + 1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t j = j0 + 64 * h + 4 * tx;
      if (VEC && j + 4 <= n) {
        *reinterpret_cast<float4*>(row + j) = make_float4(x[4 * h], x[4 * h + 1], x[4 * h + 2], x[4 * h + 3]);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int64_t jj = VEC ? j + q : j0 + tx + 16 * (4 * h + q);
          if (jj < n) row[jj] = x[4 * h + q];
        }
      }
    }
  }
}

}  // namespace

// One block per tile, row-major over the tiles (m n < 2^32 keeps this below 2^31 blocks).
void launch_dense(const float* U, const float* sigma, const float* V, int RP, int64_t m, int64_t n, int r, float* L,
                  int64_t ldl, cudaStream_t st) {
  const unsigned tiles = (unsigned)(((n + DT - 1) / DT) * ((m + DT - 1) / DT));
  if (ldl % 4 == 0 && reinterpret_cast<uintptr_t>(L) % 16 == 0)
    k_dense<true><<<tiles, DT_THREADS, 0, st>>>(U, sigma, V, RP, m, n, r, L, ldl);
  else
    k_dense<false><<<tiles, DT_THREADS, 0, st>>>(U, sigma, V, RP, m, n, r, L, ldl);
}

}  // namespace godec
