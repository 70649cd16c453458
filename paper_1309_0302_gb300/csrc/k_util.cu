// Small helpers: zero fill, padded copies of tall factors, the scale of a matrix and ||X||_F^2.
#include <algorithm>

#include "godec_internal.cuh"
#include "tc_util.cuh"

namespace godec {

namespace {

__global__ void k_fill_zero(uint4* p, size_t n16) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += (size_t)gridDim.x * blockDim.x)
    p[i] = make_uint4(0, 0, 0, 0);
}

// 32 x 32 tiles through shared memory (padded against bank conflicts)
__global__ void k_transpose(const float* __restrict__ src, int64_t m, int64_t n, int64_t lds,
                            float* __restrict__ dst, int64_t ldd, const float* __restrict__ scale) {
  __shared__ float t[32][33];
  const int64_t i0 = (int64_t)blockIdx.y * 32, j0 = (int64_t)blockIdx.x * 32;
  const float sc = scale ? scale[0] : 1.f;
  for (int k = threadIdx.y; k < 32; k += 8) {
    const int64_t i = i0 + k, j = j0 + threadIdx.x;
    t[k][threadIdx.x] = (i < m && j < n) ? src[i * lds + j] * sc : 0.f;
  }
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += 8) {
    const int64_t j = j0 + k, i = i0 + threadIdx.x;
    if (j < n && i < m) dst[j * ldd + i] = t[threadIdx.x][k];
  }
}

// dst (row stride ldd, 16-byte aligned rows) = src (row stride lds): four columns per thread,
// scalar loads (rows of src start anywhere; neighbouring lanes share their sectors), one
// 16-byte store.  Bound: 8 m n bytes (20011 x 3003: 90 us against 185 us as a zero fill and a
// strided copy).
__global__ void __launch_bounds__(256)
k_copy_rows(const float* __restrict__ src, int64_t m, int64_t n, int64_t lds, float* __restrict__ dst, int64_t ldd) {
  const int64_t per = (n + 3) / 4, total = m * per;
  for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < total; e += (int64_t)gridDim.x * 256) {
    const int64_t i = e / per, j = (e - i * per) * 4;
    const float* s = src + i * lds + j;
    float* d = dst + i * ldd + j;
    if (j + 4 <= n) {
      const float a = s[0], b = s[1], c = s[2], f = s[3];
      *reinterpret_cast<float4*>(d) = make_float4(a, b, c, f);
    } else {
      for (int u = 0; j + u < n; ++u) d[u] = s[u];
    }
  }
}

__global__ void k_pad_copy(const float* src, int64_t rows, int cols, int64_t lds, float* dst, int RP) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < rows * RP;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t i = e / RP;
    int c = (int)(e % RP);
    dst[e] = (c < cols) ? src[i * lds + c] : 0.f;
  }
}

__global__ void k_unpad_copy(const float* src, int64_t rows, int RP, float* dst, int cols) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < rows * cols;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t i = e / cols;
    int c = (int)(e % cols);
    dst[e] = src[i * RP + c];
  }
}

// max |Z| over the matrix (non-negative floats order like their bit patterns) and, with
// sumsq, += sum of Z^2 in the same pass: float4 loads, four in flight per thread, float
// sums of sixteen squares added up in float64.  Bound: 4 rows cols bytes read from HBM.
__global__ void __launch_bounds__(256)
k_maxabs(const float* __restrict__ Z, int64_t rows, int64_t cols, int64_t ld, unsigned* out, double* sumsq, int vec) {
  float m = 0.f;
  double acc = 0.0;
  const int64_t per = (cols + 15) / 16, total = rows * per;   // runs of 16 columns
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / per, j = (e - i * per) * 16;
    const float* z = Z + i * ld + j;
    float v[16];
    if (vec && j + 16 <= cols) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 q = __ldg(reinterpret_cast<const float4*>(z) + u);
        v[4 * u] = q.x; v[4 * u + 1] = q.y; v[4 * u + 2] = q.z; v[4 * u + 3] = q.w;
      }
    } else {
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = j + u < cols ? z[u] : 0.f;
    }
    float f = 0.f;
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      m = fmaxf(m, fabsf(v[u]));
      f = fmaf(v[u], v[u], f);
    }
    if (sumsq) acc += (double)f;
  }
  for (int o = 16; o; o >>= 1) {
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (sumsq) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  }
  __shared__ float sm[8];
  __shared__ double sa[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) {
    sm[w] = m;
    sa[w] = acc;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int k = 1; k < 8; ++k) {
    m = fmaxf(m, sm[k]);
    acc += sa[k];
  }
  if (out) atomicMax(out, __float_as_uint(m));
  if (sumsq) atomicAdd(sumsq, acc);
}

__global__ void k_make_zscale(const unsigned* mx, float* zscale) {
  const float m = __uint_as_float(*mx);
  int e = 0;
  if (m > 0.f && isfinite(m)) {
    int ex;
    frexpf(m, &ex);   // m in [2^(ex-1), 2^ex)
    e = 13 - ex;
    e = e < -120 ? -120 : (e > 120 ? 120 : e);
  }
  zscale[0] = ldexpf(1.f, e);
  zscale[1] = ldexpf(1.f, -e);
}

// Self-test of the timeout path: thread 0 waits, with the pipelines' bounded polling
// helper, on a fresh mbarrier that nothing arrives on, and gives up after `polls` polls
// (each at most tc::kPollNs) as a pipeline wait does: it flags the context (timeout,
// abort) and returns.  Nothing is left in flight.
__global__ void k_wait_check(Ctl* ctl, uint32_t polls) {
  __shared__ uint64_t bar;
  if (threadIdx.x != 0) return;
  tc::mbar_init(&bar, 1);
  tc::fence_barrier_init();
  if (!tc::mbar_wait(&bar, 0u, polls)) {
    ctl->timeout = 1;
    ctl->abort = 1;
  }
}

}  // namespace

void launch_wait_check(Ctl* ctl, uint32_t polls, cudaStream_t st) { k_wait_check<<<1, 32, 0, st>>>(ctl, polls); }

void launch_fill_zero(void* p, size_t bytes, cudaStream_t st) {
  // bytes must be a multiple of 16 and p 16-byte aligned
  size_t n16 = bytes / 16;
  if (!n16) return;
  unsigned grid = (unsigned)std::min<size_t>((n16 + 255) / 256, 4096);
  k_fill_zero<<<grid, 256, 0, st>>>(reinterpret_cast<uint4*>(p), n16);
}

void launch_transpose(const float* src, int64_t m, int64_t n, int64_t lds, float* dst, int64_t ldd,
                      cudaStream_t st, const float* scale) {
  dim3 grid((unsigned)((n + 31) / 32), (unsigned)((m + 31) / 32));
  k_transpose<<<grid, dim3(32, 8), 0, st>>>(src, m, n, lds, dst, ldd, scale);
}

void launch_copy_rows(const float* src, int64_t m, int64_t n, int64_t lds, float* dst, int64_t ldd, int nsm,
                      cudaStream_t st) {
  int64_t grid = (m * ((n + 3) / 4) + 255) / 256;
  if (grid > 32LL * nsm) grid = 32LL * nsm;
  k_copy_rows<<<(unsigned)grid, 256, 0, st>>>(src, m, n, lds, dst, ldd);
}

void launch_pad_copy(const float* src, int64_t rows, int cols, int64_t lds, float* dst, int RP,
                     cudaStream_t st) {
  int64_t tot = rows * RP;
  unsigned grid = (unsigned)std::min<int64_t>((tot + 255) / 256, 4096);
  if (grid) k_pad_copy<<<grid, 256, 0, st>>>(src, rows, cols, lds, dst, RP);
}

void launch_unpad_copy(const float* src, int64_t rows, int RP, float* dst, int cols, cudaStream_t st) {
  int64_t tot = rows * cols;
  unsigned grid = (unsigned)std::min<int64_t>((tot + 255) / 256, 4096);
  if (grid) k_unpad_copy<<<grid, 256, 0, st>>>(src, rows, RP, dst, cols);
}

static void launch_maxabs(const float* Z, int64_t rows, int64_t cols, int64_t ld, unsigned* mx, double* sumsq, int nsm,
                          cudaStream_t st) {
  int64_t grid = (rows * ((cols + 15) / 16) + 255) / 256;
  if (grid > 8LL * nsm) grid = 8LL * nsm;
  const int vec = (ld % 4 == 0) && (reinterpret_cast<uintptr_t>(Z) % 16 == 0);
  k_maxabs<<<(unsigned)(grid > 0 ? grid : 1), 256, 0, st>>>(Z, rows, cols, ld, mx, sumsq, vec);
}

void launch_zscale_from(const unsigned* base, const float* extra, int64_t n_extra, unsigned* zmax, float* zscale, int nsm,
                        cudaStream_t st) {
  cudaMemcpyAsync(zmax, base, sizeof(unsigned), cudaMemcpyDeviceToDevice, st);
  if (extra && n_extra > 0) launch_maxabs(extra, 1, n_extra, n_extra, zmax, nullptr, nsm, st);
  k_make_zscale<<<1, 1, 0, st>>>(zmax, zscale);
}

void launch_sumsq(const float* X, int64_t m, int64_t n, int64_t ldx, double* out, int nsm, cudaStream_t st) {
  launch_maxabs(X, m, n, ldx, nullptr, out, nsm, st);
}

void launch_zscale(const float* Z, int64_t rows, int64_t cols, int64_t ld, unsigned* zmax, float* zscale, int nsm,
                   cudaStream_t st, double* sumsq, const float* extra, int64_t n_extra) {
  cudaMemsetAsync(zmax, 0, sizeof(unsigned), st);
  launch_maxabs(Z, rows, cols, ld, zmax, sumsq, nsm, st);
  if (extra && n_extra > 0) launch_maxabs(extra, 1, n_extra, n_extra, zmax, nullptr, nsm, st);
  k_make_zscale<<<1, 1, 0, st>>>(zmax, zscale);
}

}  // namespace godec
