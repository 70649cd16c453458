// Streaming product over the split working copy (tcgen05, sm_103a): the kernel of the power
// chain and of every other product with the working matrix Z = (X - S) s_Z.
//
//   out = op(Z) B,   op(Z) = Z (rows m, K = n)  or  Z^T (rows n, K = m),   B  K x RP
//
// Storage.  Z is kept once, already split for the tensor cores: each element is
// z = h + 2^-11 l with h = fp16(z), l = fp16((z - h) 2^11) (round to nearest; z to 2^-23
// relative), 4 bytes as a float32 copy would take.  A row holds, per 64 columns, 64 halves
// of h and then 64 of l (256 contiguous bytes), so one tensor map of 64-half blocks serves
// both directions: Z B reads the boxes as a K-major operand, Z^T C reads the same boxes as
// an M-major one (the MMA transposes on the way in).  Neither a transposed copy nor any
// conversion in the kernel is needed: the stream is TMA -> shared memory -> MMA.
//
// Arithmetic.  The skinny operand arrives split likewise, b = c1 + 2^-11 c2, as
// [c1^T; c2^T] (2 RP x K halves).  Per 16-wide K step
//   D[:, 0:2RP] += h [c1; c2]^T   and   D[:, RP:RP+RPp] += l (rows 0..RPp-1 of [c1; c2])^T,
// RPp = RP rounded up to 16 (the MMA's N granularity; columns beyond 2RP are not read), and
// out = (D[:, :RP] + 2^-11 D[:, RP:2RP]) / (s_Z s_B): the dropped l c2 is below 2^-22
// of its term.
// HALF (the precision form's chain): h alone is read, half the bytes.
//
// Work split: the (128-row tile, 64-wide K stage) space is cut into equal contiguous ranges,
// one per persistent CTA ("stream-K").  The tensor core accumulates kChunk stages in tensor
// memory (its additions are not round-to-nearest; longer runs show a bias), the epilogue
// warps drain each chunk into float32 registers, one row per thread, and write the CTA's
// share of a tile to a partial slot.  The CTA whose share arrives last hands the tile to its
// eight completion warps, which add the slots in order (deterministic), unscale, apply the
// normaliser T and write the rows, the next product's operand and the tile's Gram partial
// while the stream of the CTA's next tile goes on.
//
// A matrix larger than L2: a fixed share of its 128 x 128 blocks (spread over the matrix) is
// loaded with the evict-last policy, the rest evict-first, so every product of a chain,
// whichever direction it has, finds that share in L2.
//
// Bound: HBM, 4 m n bytes less what L2 keeps.  Measured on GB300 at 10^4 x 10^4, r = 50: a
// chain product (normaliser, operand and Gram) 94 -> 83 us between events, of which 53 us
// stream (7.5 TB/s) and about 13 us the completion of the last tiles; a plain Z^T C of it 72 us;
// at 76800 x 1000, r = 3 67-84 -> 57 us.  The form before this one kept float32 copies of Z and
// Z^T and converted every tile in the kernel.
//
// Warps: 0 TMA producer (Z and skinny tiles of a stage on one barrier), 1 MMA issuer (TMEM
// owner), 2-3 spare, 4-7 epilogue, 8-15 completion.  The MMA warp runs its loop with all
// lanes (uniform operands stay in uniform registers) and issues from one elected lane; with
// the loop on a single lane its issue rate, about 1400 cycles a stage, was the limit.  Every
// wait is bounded and ends early when another role gave up; a timeout sets ctl->timeout (without
// a control block: makes the output rows of the CTA's tiles NaN), and the CTA drains its copies
// and MMAs and returns.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "godec_internal.cuh"
#include "tc_util.cuh"

namespace godec {

namespace {

using namespace tc;

constexpr int BM = 128, BK = 64;      // rows per tile, K per stage (4 MMA steps of 16)
constexpr int kPThreads = 512;
constexpr int kHelpers = 256;         // completion threads
constexpr int kQ = 4;                 // tiles waiting for completion
constexpr int kChunk = 2;             // K stages accumulated in TMEM before a drain
constexpr int kPinOf = 64;            // classes of 128 x 128 blocks, block (i, j) in class (i + j) mod kPinOf
constexpr uint32_t kPWait = 1u << 20;
constexpr float kLoInv = 1.f / 2048.f;

// Shared memory: ring of stages (Z tile, then the skinny tile; 1024-byte aligned), the tile
// under completion (128 rows of stride RP + 1, odd: conflict-free by rows and by columns) and
// T (RP x RP).  As many stages as fit, at most kMaxNS.
constexpr int kMaxNS = 10;
constexpr size_t kSmemMax = 232448 - 1024;
__host__ __device__ constexpr uint32_t stage_bytes(int RP, bool half) { return (half ? 16384u : 32768u) + (uint32_t)RP * 256u; }
__host__ __device__ constexpr uint32_t work_bytes(int RP) { return (uint32_t)(BM * (RP + 1) + RP * RP) * 4u; }
__host__ __device__ constexpr int num_stages(int RP, bool half) {
  const int ns = (int)((kSmemMax - 1024 - work_bytes(RP)) / stage_bytes(RP, half));
  return ns < kMaxNS ? ns : kMaxNS;
}
static_assert(num_stages(kMaxRP, false) >= 3, "shared memory of the streaming product");

struct PArgs {
  int64_t rows;
  int RP;
  int64_t ks, S;            // K stages per tile, total stages
  int G, maxseg, ns;
  int pin;                  // of kPinOf classes of blocks, those kept in L2 (< 0: no cache hints)
  float* part;              // tiles x maxseg x RP x BM
  unsigned* counters;       // tiles
  float* out;               // rows x oc, oc <= RP (nullable)
  int oc;
  __half* bt2;              // 2 RP x ldb split transposed output (nullable)
  int64_t ldb;
  const float* Tn0;
  const float* Tn1;
  const float* cscale;      // per-column output factor 1 / s_B (nullable: 1)
  const float* zscale;      // {s_Z, 1 / s_Z} (nullable: 1)
  float* gram_part;         // nullable: tiles x RP x RP
  int z_prefetch;           // Z's first stages may be loaded before the programmatic wait
  uint32_t limit;           // polls after which a wait gives up
  int withhold;             // self-test: the CTA whose loads are not issued (-1: none)
  Ctl* ctl;
};

__device__ __forceinline__ int64_t cta_of(int64_t g, int64_t S, int G) { return ((g + 1) * (int64_t)G - 1) / S; }

__device__ __forceinline__ void p_timeout(Ctl* ctl, volatile int* s_err) {
  *s_err = 1;
  if (ctl) {
    ctl->timeout = 1;
    ctl->abort = 1;
  }
}

// Bounded wait that also ends (false) when another role of the CTA has given up.
__device__ __forceinline__ bool p_wait(uint64_t* bar, uint32_t parity, uint32_t limit, Ctl* ctl, volatile int* s_err) {
  for (uint32_t i = 0; i < limit; ++i) {
    if (mbar_wait(bar, parity, 1)) return true;
    if (*s_err) return false;
  }
  p_timeout(ctl, s_err);
  return false;
}

// Shared-memory matrix descriptor of an M-major operand with the 128-byte swizzle: 64
// consecutive M elements per 128-byte row, K along the rows (8-row groups 1024 bytes apart),
// the next 64 M elements lbo bytes further.
__device__ __forceinline__ uint64_t sdesc_m128(const void* p, uint32_t lbo) {
  const uint64_t a = (smem_u32(p) & 0x3FFFF) >> 4;
  return a | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// One box of 64 halves x box rows of the split matrix (block b of 64 halves, from row y).
__device__ __forceinline__ void load_block(void* dst, const CUtensorMap* map, uint64_t* bar, int b, int y,
                                           uint64_t policy, bool hint) {
  if (hint)
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %4, %5}], [%2], %6;" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(0), "r"(b), "r"(y), "l"(policy)
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(0), "r"(b), "r"(y)
        : "memory");
}

// Gram partial Y^T Y of the tile in Ps (128 rows, row stride LD) by the completion threads
// (u = 0 .. 255): the upper triangle of 8 x 8 blocks, each as two 4 x 8 halves, SPL adjacent
// lanes per half (lane sp takes the rows sp mod SPL), summed by a reduce-scatter over those
// lanes (each ends with 32 / SPL entries).  RP / 8 (RP / 8 + 1) SPL <= 256.
template <int SPL>
__device__ __forceinline__ void gram256(const float* Ps, int LD, int RP, float* gp, int u) {
  const int nb = RP / 8, sp = u % SPL;
  int rem = u / SPL;
  const bool act = rem < nb * (nb + 1);
  int ri = act ? (rem & 1) * 4 : 0, bi = 0;
  rem = act ? rem >> 1 : 0;
  while (rem >= nb - bi) {
    rem -= nb - bi;
    ++bi;
  }
  ri += 8 * bi;
  const int cj = 8 * (bi + rem);
  f32x2 w[4][4] = {};
  if (act)
#pragma unroll 2
    for (int r = sp; r < BM; r += SPL) {
      const float* x = Ps + r * LD + ri;
      const float* y = Ps + r * LD + cj;
      f32x2 yy[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) yy[j] = pack2(y[2 * j], y[2 * j + 1]);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const f32x2 xi = pack2(x[i], x[i]);
#pragma unroll
        for (int j = 0; j < 4; ++j) fma2(w[i][j], xi, yy[j]);
      }
    }
  float v[32];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) unpack2(w[i][j], v[i * 8 + 2 * j], v[i * 8 + 2 * j + 1]);
  int e0 = 0;
#pragma unroll
  for (int o = SPL / 2, h = 16; o >= 1; o >>= 1, h >>= 1) {
    const bool up = (u & o) != 0;
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (i < h) {
        const float send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    if (up) e0 += h;
  }
  if (!act) return;
  const bool mirror = (ri >> 3) != (cj >> 3);   // off the diagonal blocks
#pragma unroll
  for (int i = 0; i < 32 / SPL; ++i) {
    const int e = e0 + i, a = ri + (e >> 3), b = cj + (e & 7);
    gp[a * RP + b] = v[i];
    if (mirror) gp[b * RP + a] = v[i];
  }
}

// Completion of tile t (nseg partial slots) by the kHelpers completion threads: the slots
// added in slot order and unscaled into Ps, Y <- Y T (T upper triangular, in Ts; a warp takes
// an 8-column group of 32 RB rows, RB rows x 8 columns per thread, T read at one address per
// warp), then the rows, the next product's split transposed operand and the Gram partial.
// Bound: float32 fma issue (2 x 64 RP^2 fmas) and three memory round trips.
template <int RPp>
__device__ __forceinline__ void finish_tile(const PArgs& a, int64_t t, int nseg, int u, float* Ps, const float* Ts,
                                            bool has_t, float zi) {
  constexpr int RB = RPp > 32 ? 4 : (RPp == 32 ? 2 : 1);
  const int RP = a.RP, LD = RP + 1;
  const int64_t o0 = t * BM;
  const int nrow = (int)(a.rows - o0 < BM ? a.rows - o0 : BM);
  const float4* part = reinterpret_cast<const float4*>(a.part + t * a.maxseg * (int64_t)(BM * RP));
  // thread items (column l, rows 4 rq ..), two slots' loads in flight together
  constexpr int kIt = RPp / 8;
  float4 acc[kIt];
#pragma unroll
  for (int k = 0; k < kIt; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int s0 = 0; s0 < nseg; s0 += 2) {
    const bool two = s0 + 1 < nseg;
    const float4* p0 = part + (int64_t)s0 * (BM / 4) * RP;
    float4 v[2][kIt];
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int k = 0; k < kIt; ++k) {
        const int it = u + k * kHelpers;
        v[s][k] = (it < RP * (BM / 4) && (s == 0 || two)) ? __ldcg(p0 + (int64_t)s * (BM / 4) * RP + it)
                                                         : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int k = 0; k < kIt; ++k) {
        acc[k].x += v[s][k].x;
        acc[k].y += v[s][k].y;
        acc[k].z += v[s][k].z;
        acc[k].w += v[s][k].w;
      }
  }
#pragma unroll
  for (int k = 0; k < kIt; ++k) {
    const int it = u + k * kHelpers, l = it >> 5, r = (it & 31) * 4;
    if (l < RP) {
      const float f = (a.cscale ? __ldg(a.cscale + l) : 1.f) * zi;
      // lanes of each group of eight start at another of their four rows: no bank conflicts
      const int rot = (u >> 3) & 3;
      const float4 q = acc[k];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int j = (i + rot) & 3;
        const float x = j & 2 ? (j & 1 ? q.w : q.z) : (j & 1 ? q.y : q.x);
        Ps[(r + j) * LD + l] = r + j < nrow ? x * f : 0.f;
      }
    }
  }
  named_sync(2, kHelpers);
  if (has_t) {
    // items: 8-column group x block of 32 RB rows, one per warp (longest groups first)
    constexpr int NRB = 4 / RB;
    const int ncg = RP / 8, w = u >> 5;
    const int cg = ncg - 1 - w / NRB, r0 = (w % NRB) * 32 * RB + (u & 31);
    f32x2 o[RB][4] = {};
    if (cg >= 0) {
      const float* p = Ps + r0 * LD;
      const float* tp = Ts + cg * 8;
#pragma unroll 4
      for (int k = 0; k < cg * 8 + 8; ++k) {
        const ulonglong2 t0 = *reinterpret_cast<const ulonglong2*>(tp + k * RP);
        const ulonglong2 t1 = *reinterpret_cast<const ulonglong2*>(tp + k * RP + 4);
        const f32x2 tt[4] = {t0.x, t0.y, t1.x, t1.y};
#pragma unroll
        for (int i = 0; i < RB; ++i) {
          const float y = p[i * 32 * LD + k];
          const f32x2 yy = pack2(y, y);
#pragma unroll
          for (int j = 0; j < 4; ++j) fma2(o[i][j], yy, tt[j]);
        }
      }
    }
    named_sync(2, kHelpers);   // every read of Y done before it is overwritten
    if (cg >= 0)
#pragma unroll
      for (int i = 0; i < RB; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float* q = Ps + (r0 + 32 * i) * LD + cg * 8 + 2 * j;
          unpack2(o[i][j], q[0], q[1]);
        }
    named_sync(2, kHelpers);
  }
  if (a.out) {
    const int oc = a.oc;   // consecutive threads on consecutive floats of the output rows
    float* o = a.out + o0 * oc;
    for (int it = u; it < nrow * oc; it += kHelpers) {
      const int r = it / oc;
      o[it] = Ps[r * LD + it - r * oc];
    }
  }
  if (a.bt2) {
    // a warp writes 64 consecutive rows of one column's c1 and of its c2 (128 bytes each);
    // the row after an odd last one is zero and inside the padded stride
    const int r = (u & 63) * 2;
    if (r < nrow)
      for (int l = u >> 6; l < RP; l += kHelpers / 64) {
        const float v0 = Ps[r * LD + l] * kSkinnyScale, v1 = Ps[(r + 1) * LD + l] * kSkinnyScale;
        const __half2 c1 = __floats2half2_rn(v0, v1);
        const __half2 c2 = __floats2half2_rn((v0 - __low2float(c1)) * 2048.f, (v1 - __high2float(c1)) * 2048.f);
        __half* b = a.bt2 + (int64_t)l * a.ldb + o0 + r;
        *reinterpret_cast<__half2*>(b) = c1;
        *reinterpret_cast<__half2*>(b + (int64_t)RP * a.ldb) = c2;
      }
  }
  if (a.gram_part) {
    constexpr int SPL = RPp <= 16 ? 32 : (RPp <= 32 ? 8 : 4);
    float* gp = a.gram_part + t * (int64_t)(RP * RP);
    if (RP == 64) gram256<2>(Ps, LD, RP, gp, u);
    else gram256<SPL>(Ps, LD, RP, gp, u);
  }
  named_sync(2, kHelpers);   // Ps free again
}

__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}

template <int RPp, bool TR, bool HALF>
__global__ void __launch_bounds__(kPThreads, 1)
k_prod_split(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, PArgs a) {
  constexpr int kAccCols = RPp <= 32 ? 64 : 128, kAcc = 512 / kAccCols;
  constexpr uint32_t kA = HALF ? 16384 : 32768;
  const int NS = a.ns;
  const uint32_t limit = a.limit;
  Ctl* ctl = a.ctl;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t stage = stage_bytes(a.RP, HALF);   // bytes of a stage, a multiple of 1024
  float* Ts = reinterpret_cast<float*>(sm + (size_t)NS * stage);
  float* Ps = Ts + a.RP * a.RP;
  __shared__ uint64_t full[kMaxNS], empty[kMaxNS], accfull[kAcc], accempty[kAcc], qfull[kQ], qempty[kQ], mma_done;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int s_err;
  __shared__ volatile int s_q[kQ], s_go;
  __shared__ int s_stop, s_last;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int c = blockIdx.x, G = a.G;
  const int64_t S = a.S, ks = a.ks;
  const int64_t g0 = (int64_t)c * S / G, g1 = (int64_t)(c + 1) * S / G;
  int64_t t = 0, p = 0;                // the producer's tile and stage
  uint64_t pol_first = 0, pol_keep = 0;
  // the Z tile of stage (t, p) into slot s; the barrier expects the skinny tile too
  auto load_a = [&](int s) {
    unsigned char* d = sm + (size_t)s * stage;
    const uint64_t pol = (int)((t + (p >> 1)) & (kPinOf - 1)) < a.pin ? pol_keep : pol_first;
    const bool hint = a.pin >= 0;
    mbar_expect_tx(&full[s], stage);
    if (!TR) {
      load_block(d, &mapA, &full[s], (int)(2 * p), (int)(t * BM), pol, hint);
      if (!HALF) load_block(d + 16384, &mapA, &full[s], (int)(2 * p + 1), (int)(t * BM), pol, hint);
    } else {
      // columns 64 (2t) .. and 64 (2t + 1) .. of Z: h and l blocks each
      const int b = (int)(4 * t), y = (int)(p * BK);
      load_block(d, &mapA, &full[s], b, y, pol, hint);
      if (!HALF) load_block(d + 8192, &mapA, &full[s], b + 1, y, pol, hint);
      load_block(d + (HALF ? 8192 : 16384), &mapA, &full[s], b + 2, y, pol, hint);
      if (!HALF) load_block(d + 24576, &mapA, &full[s], b + 3, y, pol, hint);
    }
    if (++p == ks) { p = 0; ++t; }
  };
  const int nst = (int)(g1 - g0);      // this CTA's stages
  int npre = 0;
  if (tid == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapA)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapB)) : "memory");
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < kAcc; ++b) {
      mbar_init(&accfull[b], 1);
      mbar_init(&accempty[b], 4);
    }
    for (int k = 0; k < kQ; ++k) {
      mbar_init(&qfull[k], 1);
      mbar_init(&qempty[k], 1);
    }
    mbar_init(&mma_done, 1);
    fence_barrier_init();
    s_err = 0;
    pol_first = policy_evict_first();
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_keep));
    t = g0 / ks;
    p = g0 - t * ks;
    // Z is not written by the kernels before this one in the chain: its first tiles are on
    // their way before the wait for them (a free ring: no slot is waited for)
    if (a.z_prefetch)
      for (; npre < NS && npre < nst; ++npre) load_a(npre);
  }
  if (warp == 1) tmem_alloc(&tmem_base, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();   // from here on everything the preceding kernels wrote may be read
  const uint32_t tbase = tmem_base;

  if (warp == 0) {
    if (lane == 0) {
      int pb = (int)(g0 % ks), s = 0;   // K stage of the skinny tile
      uint32_t ph = 0;
      int i = 0;
      const int loads = c == a.withhold ? 0 : nst;
      for (; i < loads; ++i) {
        if (i >= npre) {
          if (!p_wait(&empty[s], ph ^ 1u, limit, ctl, &s_err)) break;
          load_a(s);
        }
        tma_load_2d(sm + (size_t)s * stage + kA, &mapB, &full[s], pb * BK, 0);
        if (++pb == (int)ks) pb = 0;
        if (++s == NS) { s = 0; ph ^= 1u; }
      }
      // every copy issued has landed before the CTA may exit
      for (int j = (i > NS ? i - NS : 0); j < i; ++j)
        if (!mbar_wait(&full[j % NS], (uint32_t)((j / NS) & 1), kPWait)) p_timeout(ctl, &s_err);
    }
  } else if (warp == 1) {
    // Iteration already abandoned, or Z outgrew its scale in the last S-step (the caller
    // rebuilds it): do nothing, and make the rest of the iteration skip too.
    bool skip = false;
    if (ctl) {
      const int ab = *reinterpret_cast<volatile int*>(&ctl->abort), re = *reinterpret_cast<volatile int*>(&ctl->range_err);
      if (re) ctl->abort = 1;
      skip = ab || re;
      if (skip) s_err = 2;
    }
    const int RP = a.RP;
    const uint32_t trb = TR ? (1u << 15) : 0u;
    const uint32_t id_hi = idesc_f16(BM, 2 * RP) | trb, id_lo = idesc_f16(BM, RPp) | trb;
    constexpr uint32_t kLbo = HALF ? 8192 : 16384;
    constexpr uint64_t kStep = TR ? (2048 >> 4) : (32 >> 4);   // 16 of K
    constexpr int kLow = TR ? 8192 : 16384;                    // l blocks after the h blocks
    const uint64_t d0 = TR ? sdesc_m128(sm, kLbo) : sdesc_k128(sm);
    const uint64_t b0 = sdesc_k128(sm + kA);
    int left = skip ? 0 : nst, kst = (int)(g0 % ks), ch = 0, s = 0;
    uint32_t ph = 0;
    while (left > 0) {
      int n = (int)ks - kst;   // this chunk: not past the end of the tile or of the range
      if (n > kChunk) n = kChunk;
      if (n > left) n = left;
      const int b = ch & (kAcc - 1);
      if (!__all_sync(0xffffffffu, p_wait(&accempty[b], (uint32_t)(((ch / kAcc) & 1) ^ 1), limit, ctl, &s_err))) break;
      const uint32_t dcol = tbase + (uint32_t)(b * kAccCols);
      bool ok = true;
      for (int e = 0; e < n; ++e) {
        ok = __all_sync(0xffffffffu, p_wait(&full[s], ph, limit, ctl, &s_err));
        if (!ok) break;
        tc_fence_after();
        const uint64_t so = (uint64_t)((uint32_t)s * (stage >> 4));
        const uint64_t dh = d0 + so, dl = dh + (kLow >> 4), db = b0 + so;
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            mma_bf16(dcol, dh + kk * kStep, db + 2 * kk, id_hi, (e > 0 || kk > 0) ? 1u : 0u);
            if (!HALF) mma_bf16(dcol + RP, dl + kk * kStep, db + 2 * kk, id_lo, 1u);
          }
          mma_commit(&empty[s]);
          if (e == n - 1) mma_commit(&accfull[b]);
        }
        __syncwarp();
        if (++s == NS) { s = 0; ph ^= 1u; }
      }
      if (!ok) break;
      ++ch;
      left -= n;
      kst += n;
      if (kst == (int)ks) kst = 0;
    }
    __syncwarp();
    // the stage commits above came from the elected lane; so does this one
    if (elect_one()) {
      mma_commit(&mma_done);
      if (!mbar_wait(&mma_done, 0, kPWait)) p_timeout(ctl, &s_err);
      pdl_launch_dependents();   // the stream is done: the next product may start its prologue
    }
    __syncwarp();
  } else if (warp >= 4 && warp < 8) {
    // ---------------- epilogue: one row per thread ----------------
    // The four warps take every decision together (flag written between two named barriers),
    // so no warp can leave while the others wait at a barrier.
    const int row = tid - 128;
    const uint32_t tlane = (uint32_t)((warp & 3) * 32) << 16;
    const int RP = a.RP;
    int ch = 0, pushed = 0;
    auto push = [&](int v) {   // one thread
      const int k = pushed % kQ;
      if (!p_wait(&qempty[k], (uint32_t)(((pushed / kQ) & 1) ^ 1), limit, ctl, &s_err)) return;
      s_q[k] = v;
      mbar_arrive(&qfull[k]);
      ++pushed;
    };
    int64_t g = g0;
    for (;;) {
      named_sync(1, BM);
      if (row == 0) s_stop = (g >= g1) || s_err;
      named_sync(1, BM);
      if (s_stop) break;
      const int64_t tt = g / ks;
      const int64_t tend = ((tt + 1) * ks < g1) ? (tt + 1) * ks : g1;
      float y[RPp];
#pragma unroll
      for (int l = 0; l < RPp; ++l) y[l] = 0.f;
      bool failed = false;
      for (; g < tend; g = (g + kChunk < tend) ? g + kChunk : tend, ++ch) {
        if (failed) continue;                // keep the loop count; nothing more to read
        const int b = ch & (kAcc - 1);
        if (!__all_sync(0xffffffffu, p_wait(&accfull[b], (uint32_t)((ch / kAcc) & 1), limit, ctl, &s_err))) {
          failed = true;
          continue;
        }
        tc_fence_after();
        const uint32_t taddr = tbase + (uint32_t)(b * kAccCols) + tlane;
#pragma unroll
        for (int c0 = 0; c0 < RPp; c0 += 16) {
          float vh[16], vl[16];
          tmem_ld8x4(taddr + c0, taddr + RP + c0, vh, vl);
#pragma unroll
          for (int l = 0; l < 16; ++l) y[c0 + l] += fmaf(vl[l], kLoInv, vh[l]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&accempty[b]);
      }
      named_sync(1, BM);
      if (row == 0) s_stop = s_err;
      named_sync(1, BM);
      if (s_stop) break;
      const int64_t c_first = cta_of(tt * ks, S, G);
      const int nseg = (int)(cta_of((tt + 1) * ks - 1, S, G) - c_first + 1);
      // partial slot, column-major (the warps' accesses are coalesced)
      float* ps = a.part + (tt * a.maxseg + (c - c_first)) * (int64_t)(BM * RP) + row;
#pragma unroll
      for (int l = 0; l < RPp; ++l)
        if (l < RP) __stcg(ps + l * BM, y[l]);
      __threadfence();
      named_sync(1, BM);
      if (row == 0) {
        const bool last = nseg == 1 || atomicAdd(&a.counters[tt], 1u) == (unsigned)(nseg - 1);
        if (last) {
          __threadfence();   // the other segments' slots: written before their counter increments
          if (nseg > 1) a.counters[tt] = 0u;
          push((int)tt);
        }
      }
    }
    if (row == 0) push(-1);
  } else if (warp >= 8) {
    // ---------------- completion ----------------
    const int u = tid - 256;
    const float* Tn = (ctl && ctl->slot_parity) ? a.Tn1 : a.Tn0;
    if (Tn)
      for (int e = u; e < a.RP * a.RP / 4; e += kHelpers)
        reinterpret_cast<float4*>(Ts)[e] = __ldg(reinterpret_cast<const float4*>(Tn) + e);
    const float zi = a.zscale ? a.zscale[1] : 1.f;
    for (int k = 0;; ++k) {
      const int q = k & (kQ - 1);
      if (u == 0) s_go = p_wait(&qfull[q], (uint32_t)((k / kQ) & 1), limit, ctl, &s_err) ? s_q[q] : -1;
      named_sync(2, kHelpers);
      const int64_t tt = s_go;
      if (tt < 0) break;
      const int nseg = (int)(cta_of((tt + 1) * ks - 1, S, G) - cta_of(tt * ks, S, G) + 1);
      finish_tile<RPp>(a, tt, nseg, u, Ps, Ts, Tn != nullptr, zi);
      if (u == 0) mbar_arrive(&qempty[q]);   // after the last barrier of finish_tile
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tbase, 512);
  }
  if (s_err && !ctl && a.out) poison_tiles(a.out, a.oc, a.rows, g0 / ks, (g1 - 1) / ks, tid, kPThreads);
}

template <int RPp, bool TR, bool HALF>
cudaError_t prep() {
  return cudaFuncSetAttribute(k_prod_split<RPp, TR, HALF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
}

// Launch with the programmatic-stream-serialization attribute when pdl is set: the kernel may
// begin (barrier set-up, tensor-memory allocation, Z prefetch) while the preceding kernel of
// the stream finishes, and waits for it in pdl_wait() before it reads anything else.
template <int RPp, bool TR, bool HALF>
void launch_one(const TcLaunch& l, const PArgs& a, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)a.G);
  cfg.blockDim = dim3(kPThreads);
  cfg.dynamicSmemBytes = (size_t)a.ns * stage_bytes(a.RP, HALF) + work_bytes(a.RP) + 1024;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = l.pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k_prod_split<RPp, TR, HALF>, *reinterpret_cast<const CUtensorMap*>(l.mapA),
                     *reinterpret_cast<const CUtensorMap*>(l.mapB), a);
}

template <bool TR>
void launch_dir(const TcLaunch& l, const PArgs& a, cudaStream_t st) {
  const int rpp = tc_rpp(l.RP);
  if (l.half_a) {
    if (rpp == 16) launch_one<16, TR, true>(l, a, st);
    else if (rpp == 32) launch_one<32, TR, true>(l, a, st);
    else if (l.ctl) cudaMemsetAsync(&l.ctl->abort, 0xff, sizeof(int), st);   // RP > 32: rejected at init
    return;
  }
  switch (rpp) {
    case 16: launch_one<16, TR, false>(l, a, st); break;
    case 32: launch_one<32, TR, false>(l, a, st); break;
    case 48: launch_one<48, TR, false>(l, a, st); break;
    default: launch_one<64, TR, false>(l, a, st); break;
  }
}

}  // namespace

cudaError_t prepare_prod_kernels() {
  cudaError_t e = cudaSuccess;
#define PREP(...) if (e == cudaSuccess) e = prep<__VA_ARGS__>()
  PREP(16, false, false); PREP(32, false, false); PREP(48, false, false); PREP(64, false, false);
  PREP(16, true, false); PREP(32, true, false); PREP(48, true, false); PREP(64, true, false);
  PREP(16, false, true); PREP(32, false, true); PREP(16, true, true); PREP(32, true, true);
#undef PREP
  return e;
}

// Classes of blocks (of kPinOf) of a matrix of `bytes` bytes asked to stay in L2; -1 (no
// hints) for a matrix that fits.  On GB300 about 40 MB stay: at 10^4 x 10^4, 25 MB asked for
// cut the DRAM reads of a product from 400 to 374 MB, 75 MB to 364 MB only, with write-backs.
static int prod_pin(double bytes) {
  if (bytes <= 96e6) return -1;
  return (int)(kPinOf * 44e6 / bytes);
}

// The split product's work split: on a whole device 20 SMs fewer than the general rule.  From
// about 110 CTAs on the stream is bound by HBM (10^4 x 10^4, r = 50: the same time at 148, 136
// and 120 CTAs), and the SMs left over run the r x r kernels of the side streams, which
// otherwise outlast the products (one iteration: 1.76 ms with 4 SMs left, 1.61 ms with 24).
// A share of the device (a batch problem's budget) up to 100 SMs follows the general rule, one
// of 100 to 120 keeps the 96 CTAs of 100, so that more SMs never get fewer CTAs.  Calls without
// side streams take the same split: with 148 CTAs Z^T C is within 2 % at eleven sizes and 9 %
// faster at 3 x 10^6 (181 -> 165 us), the gradient at 4096 x 4096, r = 20 2 % slower
// (1590 -> 1625 us).
TcGeom prod_split_geometry(int64_t rows, int64_t K, int nsm) {
  return tc_geometry(rows, K, std::max(nsm - 20, std::min(nsm, 100)));
}

void launch_prod_split(const TcLaunch& l, cudaStream_t st) {
  PArgs a;
  a.rows = l.rows;
  a.RP = l.RP;
  a.ks = l.geom.ks;
  a.S = l.geom.S;
  a.G = l.geom.G;
  a.maxseg = l.geom.maxseg;
  a.ns = num_stages(l.RP, l.half_a != 0);
  a.pin = prod_pin((double)l.rows * (double)l.K * (l.half_a ? 2.0 : 4.0));
  a.part = l.part;
  a.counters = l.counters;
  a.out = l.out;
  a.oc = l.out_cols ? l.out_cols : l.RP;
  a.bt2 = reinterpret_cast<__half*>(l.bt2);
  a.ldb = l.ldb;
  a.Tn0 = l.Tn[0];
  a.Tn1 = l.Tn[1];
  a.cscale = l.cscale;
  a.zscale = l.zscale;
  a.gram_part = l.gram_mode ? static_cast<float*>(l.gram_part) : nullptr;
  a.z_prefetch = l.z_prefetch;
  a.limit = l.withhold >= 0 ? kTestPolls : kPWait;
  a.withhold = l.withhold;
  a.ctl = l.ctl;
  if (l.trans) launch_dir<true>(l, a, st);
  else launch_dir<false>(l, a, st);
}

// ---- building the split matrix ---------------------------------------------------------
namespace {

// Rows of the split matrix from a float32 matrix: eight columns per thread (two 16-byte
// loads, one 16-byte store of h and one of l); columns n .. ldz-1 become zero.  Bound: 8 m n
// bytes of HBM traffic.
__global__ void __launch_bounds__(256)
k_split_copy(const float* __restrict__ X, int64_t m, int64_t n, int64_t ldx, __half* __restrict__ Z, int64_t ldz,
             const float* __restrict__ scale, int vec) {
  const float sc = scale[0];
  const int64_t per = ldz / 8, total = m * per;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / per, j = (e - i * per) * 8;
    const float* x = X + i * ldx + j;
    float v[8];
    if (vec && j + 8 <= n) {
      const float4 p = *reinterpret_cast<const float4*>(x), q = *reinterpret_cast<const float4*>(x + 4);
      v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w;
      v[4] = q.x; v[5] = q.y; v[6] = q.z; v[7] = q.w;
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = j + u < n ? x[u] : 0.f;
    }
    uint32_t h[4], l[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      __half h0, l0, h1, l1;
      split_z(v[2 * u] * sc, h0, l0);
      split_z(v[2 * u + 1] * sc, h1, l1);
      h[u] = (uint32_t)__half_as_ushort(h0) | ((uint32_t)__half_as_ushort(h1) << 16);
      l[u] = (uint32_t)__half_as_ushort(l0) | ((uint32_t)__half_as_ushort(l1) << 16);
    }
    __half* z = Z + zs_at(i, j, ldz);
    *reinterpret_cast<uint4*>(z) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(z + 64) = make_uint4(l[0], l[1], l[2], l[3]);
  }
}

}  // namespace

void launch_split_copy(const float* X, int64_t m, int64_t n, int64_t ldx, void* Z, int64_t ldz, const float* scale,
                       int nsm, cudaStream_t st) {
  int64_t blocks = (m * (ldz / 8) + 255) / 256;
  if (blocks > 32LL * nsm) blocks = 32LL * nsm;
  const int vec = (ldx % 4 == 0) && (reinterpret_cast<uintptr_t>(X) % 16 == 0);
  k_split_copy<<<(unsigned)(blocks > 0 ? blocks : 1), 256, 0, st>>>(X, m, n, ldx, static_cast<__half*>(Z), ldz, scale, vec);
}

}  // namespace godec
