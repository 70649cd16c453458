// Differentiated form: reverse-mode gradient with respect to X of a loss of L_T after T
// unrolled iterations of Algorithm 1 at q = 0, with the supports of S_1 .. S_{T-1} frozen.
//
// At q = 0 the L-step is L = Y1 (A2^T Y1)^{-1} Y2^T = Z P, with A2 = Z A1, Y2 = Z^T A2 and
// P = Y2 (Y2^T Y2)^{-1} Y2^T the projector on range(Y2) (Sec. 3.1, eq. lr_app); with the
// support Omega_t frozen, S_t = M_t * (X - L_t) and Z_{t+1} = (1 - M_t) * X + M_t * L_t.
// Differentiating:  dL = dZ P + Z dP,  dP = (I - P) dY2 Y2^+ + (Y2^+)^T dY2^T (I - P),
// dY2 = dZ^T Z A1 + Z^T dZ A1.  For a gradient G of L_t, with W = (Y2^T Y2)^{-1} and
// Y2p = Y2 W = (Y2^+)^T:
//     a   = G Y2p,   b = G^T (Z Y2p),   gY2 = (I - P) (Z^T a + b),
//     gZ  = a Y2^T + (Z A1) gY2^T + (Z gY2) A1^T            (rank <= 3r),
// and Z_t routes gZ to X outside Omega_{t-1} and to L_{t-1} on it:
//     dX += (1 - M_{t-1}) * gZ_t,   G_{t-1} = M_{t-1} * gZ_t   (M_0 = 0).
//
// The forward sweep recomputes and checkpoints the per-iteration factors (A2, Y2, Y2p,
// Q, Z Y2p and L_t on Omega_t; Q an orthonormal basis of range(Y2) from CholeskyQR2);
// the backward sweep reuses the Z_t kept from the forward sweep when all T of them fit in a
// quarter of the free device memory, and otherwise rebuilds them from X and the checkpointed
// values.  Each Z_t is held once, split for the tensor cores (k_prod.cu), and serves the
// products in both directions; the r x r solve is the Cholesky kernel of the L-step.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

#include "godec.h"
#include "godec_internal.cuh"

namespace godec {
void launch_spmm(const int64_t* idx, const float* val, int64_t nnz, int64_t n, const float* B, int64_t ldb, int c,
                 int trans, float* out, int64_t ldo, cudaStream_t st);
void launch_eval_lr(const int64_t* idx, int64_t nnz, int64_t n, const float* U, int64_t ldu, const float* V,
                    int64_t ldv, int K, float* vals, float* D, int64_t ldd, cudaStream_t st);
void launch_scatter_split(const int64_t* idx, const float* vals, int64_t nnz, int64_t n, void* Z, int64_t ldz,
                          const float* scale, cudaStream_t st);
void launch_outer_acc(const float* U, int64_t ldu, const float* V, int64_t ldv, int K, int64_t m, int64_t n,
                      float beta, float* D, int64_t ldd, cudaStream_t st);
void launch_pack3(const float* const u[3], const float* const v[3], int64_t m, int64_t n, int r, float* U, float* V,
                  int ld, cudaStream_t st);
void launch_axpy(const float* x, float* y, int64_t count, float alpha, cudaStream_t st);
}  // namespace godec

namespace {

using namespace godec;

constexpr int kCrossParts = 256;
constexpr int kMaxSlots = 32;

// Stream-ordered scratch of one call; freed (stream-ordered) on destruction.
struct Scratch {
  cudaStream_t st;
  int dev;
  std::vector<void*> ptrs;
  bool ok = true;
  template <typename T>
  T* get(size_t elems) {
    void* p = nullptr;
    if (!ok || scratch_alloc(&p, std::max<size_t>(elems, 1) * sizeof(T), dev, st) != cudaSuccess) {
      cudaGetLastError();   // reported by the call's status, not again by a later launch
      ok = false;
      return nullptr;
    }
    ptrs.push_back(p);
    return static_cast<T*>(p);
  }
  ~Scratch() {
    for (void* p : ptrs) cudaFreeAsync(p, st);
  }
};

// A split m x n matrix (k_prod.cu) with its tensor maps and power-of-two scale, the source of
// products in both directions (index 0: Z B, 1: Z^T C).
struct Source {
  alignas(64) unsigned char map[2][128];
  void* z = nullptr;
  float* zscale = nullptr;     // {s, 1/s} on the device
  unsigned* zmax = nullptr;
};

struct Engine {
  cudaStream_t st;
  int nsm = 0, RP = 0;
  int64_t dim[2] = {0, 0};                     // m, n
  int64_t ldb = 0;
  void* Bs = nullptr;                          // 2 RP x ldb halves (split transposed operand)
  alignas(64) unsigned char mapB[2][128];      // over Bs with K = n (index 0) and K = m (index 1)
  TcGeom geom[2];
  float *cscale = nullptr, *part = nullptr;
  unsigned* cmax = nullptr;                    // kMaxSlots column maxima, cleared together (one
  int slot = 0;                                // memset per kMaxSlots products, not one each)
  unsigned* cnt = nullptr;

  // Y (rows x c, dense) = src * B, or src^T * B with trans (B K x c, dense rows of c)
  void mul(const Source& s, int trans, const float* B, int c, float* Y) {
    const int64_t rows = dim[trans], K = dim[1 - trans];
    if (slot == 0) cudaMemsetAsync(cmax, 0, (size_t)kMaxSlots * (1 + RP) * sizeof(unsigned), st);
    unsigned* mx = cmax + (size_t)slot * (1 + RP);
    slot = (slot + 1) % kMaxSlots;
    launch_mul_stats(nullptr, 0, 0, 0, B, K, c, mx, nsm, st);
    launch_split_b(B, K, c, RP, mx + 1, Bs, ldb, cscale, nullptr, nullptr, st);
    TcLaunch l{};
    l.mapA = s.map[trans];
    l.mapB = mapB[trans];
    l.rows = rows;
    l.K = K;
    l.RP = RP;
    l.geom = geom[trans];
    l.part = part;
    l.counters = cnt;
    l.out = Y;
    l.out_cols = c;
    l.cscale = cscale;
    l.zscale = s.zscale;
    l.trans = trans;
    launch_prod_split(l, st);
  }
};

}  // namespace

extern "C" godec_status godec_backward(const float* X, int64_t m, int64_t n, int64_t ldx, const float* A1, int32_t r,
                                       int32_t T, const int64_t* const* supports, const int64_t* support_nnz,
                                       const float* gU, const float* gV, int32_t g_rank, const float* gL, int64_t ldg,
                                       float* dX, int64_t lddx, int32_t flags, void* stream) {
  const bool lowrank = gU && gV;
  if (!X || !A1 || !dX || m < 1 || n < 1 || ldx < n || lddx < n || r < 1 || r > GODEC_MAX_RANK || r > m ||
      r > n || T < 1 || (T > 1 && (!supports || !support_nnz)) || lowrank == (gL != nullptr) ||
      (lowrank && (g_rank < 1 || g_rank > GODEC_MAX_RANK)) || (gL && ldg < n) || (ldx * 4) % 16 != 0 ||
      (gL && (ldg * 4) % 16 != 0) || (flags & ~GODEC_BACKWARD_REBUILD)) {
    set_static_error("godec_backward: invalid argument");
    return GODEC_ERR_ARG;
  }
  for (int t = 0; t + 1 < T; ++t)
    if (support_nnz[t] < 0 || support_nnz[t] > m * n || (support_nnz[t] > 0 && !supports[t])) {
      set_static_error("godec_backward: invalid support %d", t + 1);
      return GODEC_ERR_ARG;
    }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      prepare_prod_kernels() != cudaSuccess || prepare_small_kernels() != cudaSuccess) {
    set_static_error("godec_backward: no CUDA device");
    return GODEC_ERR_CUDA;
  }
  const int RP = (r + 7) / 8 * 8, R3 = 3 * r, ldf = (R3 + 3) / 4 * 4;
  const int64_t mx = std::max(m, n), ldz = (n + 63) / 64 * 64;
  Scratch sc{st, dev};
  // Iterates Z_t: one copy for all t, rebuilt in the backward sweep, or (when all T of them
  // fit in a quarter of the free device memory) one per t, kept from the forward sweep.
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) free_b = 0;
  const bool keep = !(flags & GODEC_BACKWARD_REBUILD) &&
                    (double)T * (double)(m * ldz) * sizeof(float) <= 0.25 * (double)free_b;
  const int nzb = keep ? T : 1;
  std::vector<Source> src(nzb + (gL ? 1 : 0));   // Z_t copies, then the dense gradient
  for (Source& q : src) q.z = sc.get<float>((size_t)m * ldz);
  Engine E;
  E.st = st;
  E.nsm = nsm;
  E.RP = RP;
  E.ldb = (mx + 7) / 8 * 8;
  E.Bs = sc.get<unsigned short>((size_t)2 * RP * E.ldb);
  E.cmax = sc.get<unsigned>(kMaxSlots * (1 + (size_t)RP));
  E.cscale = sc.get<float>(RP);
  float* zsc = sc.get<float>(2 * src.size() + 2);      // {s, 1/s} of each source, then of X
  unsigned* zmax = sc.get<unsigned>(src.size() + 1);
  // per-iteration checkpoints (forward sweep)
  std::vector<float*> A2(T), Y2(T), Y2p(T), Qk(T), ZY2p(T), Lv(T);
  for (int t = 0; t < T; ++t) {
    A2[t] = sc.get<float>((size_t)m * r);
    Y2[t] = sc.get<float>((size_t)n * r);
    Y2p[t] = sc.get<float>((size_t)n * r);
    Qk[t] = sc.get<float>((size_t)n * r);
    ZY2p[t] = sc.get<float>((size_t)m * r);
    Lv[t] = (t + 1 < T && support_nnz[t] > 0) ? sc.get<float>((size_t)support_nnz[t]) : nullptr;
  }
  int64_t kmax = 0;
  for (int t = 0; t + 1 < T; ++t) kmax = std::max(kmax, support_nnz[t]);
  float* gv = sc.get<float>((size_t)std::max<int64_t>(kmax, 1));   // G_{t-1} on Omega_{t-1}
  float* Y2T = sc.get<float>((size_t)n * r);
  float* a = sc.get<float>((size_t)m * r);
  float* Wn = sc.get<float>((size_t)n * r);
  float* Zg = sc.get<float>((size_t)m * r);
  float* Uf = sc.get<float>((size_t)m * ldf);
  float* Vf = sc.get<float>((size_t)n * ldf);
  float* Rm = sc.get<float>((size_t)RP * RP * 4);                  // R1, T1, R2, T2 of CholeskyQR2
  double* g64 = sc.get<double>((size_t)RP * RP);
  double* Msm = sc.get<double>((size_t)GODEC_MAX_RANK * GODEC_MAX_RANK);
  double* cpart = sc.get<double>((size_t)kCrossParts * GODEC_MAX_RANK * GODEC_MAX_RANK);
  Ctl* ctl = sc.get<Ctl>(1);
  if (sc.ok) {
    E.dim[0] = m;
    E.dim[1] = n;
    E.geom[0] = prod_split_geometry(m, n, nsm);
    E.geom[1] = prod_split_geometry(n, m, nsm);
    size_t npart = 0;
    for (const TcGeom& g : E.geom) npart = std::max(npart, (size_t)g.tiles * g.maxseg * 128 * RP);
    E.part = sc.get<float>(npart);
    E.cnt = sc.get<unsigned>((size_t)std::max(E.geom[0].tiles, E.geom[1].tiles));
  }
  if (!sc.ok) {
    set_static_error("godec_backward: out of device memory");
    return GODEC_ERR_OOM;
  }
  cudaMemsetAsync(E.cnt, 0, (size_t)std::max(E.geom[0].tiles, E.geom[1].tiles) * sizeof(unsigned), st);
  cudaMemsetAsync(ctl, 0, sizeof(Ctl), st);
  bool mapped = make_tmap_f16(E.mapB[0], E.Bs, 2 * RP, n, E.ldb, 2 * RP) &&
                make_tmap_f16(E.mapB[1], E.Bs, 2 * RP, m, E.ldb, 2 * RP);
  for (size_t b = 0; b < src.size(); ++b) {
    src[b].zscale = zsc + 2 * b;
    src[b].zmax = zmax + b;
    mapped = mapped && make_tmap_split(src[b].map[0], src[b].z, m, ldz, 128) &&
             make_tmap_split(src[b].map[1], src[b].z, m, ldz, 64);
  }
  if (!mapped) {
    set_static_error("godec_backward: tensor map encoding failed");
    return GODEC_ERR_CUDA;
  }
  // Z_t = X with L_{t-1} on Omega_{t-1}, at a scale that covers both (copy slot b)
  unsigned* xmax = zmax + src.size();
  launch_zscale(X, m, n, ldx, xmax, zsc + 2 * src.size(), nsm, st);
  auto build_Z = [&](int t) {
    const Source& q = src[keep ? t : 0];
    const bool sup = t > 0 && support_nnz[t - 1] > 0;
    launch_zscale_from(xmax, sup ? Lv[t - 1] : nullptr, sup ? support_nnz[t - 1] : 0, q.zmax, q.zscale, nsm, st);
    launch_split_copy(X, m, n, ldx, q.z, ldz, q.zscale, nsm, st);
    if (sup) launch_scatter_split(supports[t - 1], Lv[t - 1], support_nnz[t - 1], n, q.z, ldz, q.zscale, st);
  };
  // ---------------- forward sweep: checkpoints ----------------
  for (int t = 0; t < T; ++t) {
    build_Z(t);
    const Source& sZ = src[keep ? t : 0];
    E.mul(sZ, 0, A1, r, A2[t]);                                // A2 = Z A1
    E.mul(sZ, 1, A2[t], r, Y2[t]);                             // Y2 = Z^T A2
    // Y2 = Q R by CholeskyQR2 (R = R2 R1), so that W = (Y2^T Y2)^{-1} = R^{-1} R^{-T} and
    // Y2p = Y2 W = Q T2^T T1^T are formed without squaring Y2's condition number
    const size_t rr = (size_t)RP * RP;
    float *R1 = Rm, *T1 = Rm + rr, *R2 = Rm + 2 * rr, *T2 = Rm + 3 * rr;
    launch_cross_gram(Y2[t], r, r, Y2[t], r, r, n, cpart, kCrossParts, g64, RP, st);
    launch_chol(g64, r, RP, R1, T1, ctl, st, 0.f);
    launch_tall_small_f(Y2[t], r, r, T1, RP, 0, r, n, 1.f, 0.f, Y2T, r, st);      // Q1 = Y2 T1
    launch_cross_gram(Y2T, r, r, Y2T, r, r, n, cpart, kCrossParts, g64, RP, st);
    launch_chol(g64, r, RP, R2, T2, ctl, st, 0.f);
    launch_tall_small_f(Y2T, r, r, T2, RP, 0, r, n, 1.f, 0.f, Qk[t], r, st);       // Q = Q1 T2
    launch_tall_small_f(Qk[t], r, r, T2, RP, 1, r, n, 1.f, 0.f, Y2T, r, st);       // Q T2^T
    launch_tall_small_f(Y2T, r, r, T1, RP, 1, r, n, 1.f, 0.f, Y2p[t], r, st);      // ... T1^T
    E.mul(sZ, 0, Y2p[t], r, ZY2p[t]);                          // Y1 W = Z Y2p
    if (t + 1 < T && support_nnz[t] > 0)                       // L_t on Omega_t
      launch_eval_lr(supports[t], support_nnz[t], n, ZY2p[t], r, Y2[t], r, r, Lv[t], nullptr, 0, st);
  }
  // ---------------- backward sweep ----------------
  if (gL) {
    const Source& q = src[nzb];
    launch_zscale(gL, m, n, ldg, q.zmax, q.zscale, nsm, st);
    launch_split_copy(gL, m, n, ldg, q.z, ldz, q.zscale, nsm, st);
  }
  for (int t = T - 1; t >= 0; --t) {
    if (!keep) build_Z(t);
    const Source& sZ = src[keep ? t : 0];
    // a = G Y2p and Wn = b = G^T (Z Y2p)
    if (t == T - 1 && gL) {
      E.mul(src[nzb], 0, Y2p[t], r, a);
      E.mul(src[nzb], 1, ZY2p[t], r, Wn);
    } else if (t == T - 1) {
      launch_cross_gram(gV, g_rank, g_rank, Y2p[t], r, r, n, cpart, kCrossParts, Msm, r, st);
      launch_tall_small_d(gU, g_rank, g_rank, Msm, r, 0, r, m, 1.f, 0.f, a, r, st);
      launch_cross_gram(gU, g_rank, g_rank, ZY2p[t], r, r, m, cpart, kCrossParts, Msm, r, st);
      launch_tall_small_d(gV, g_rank, g_rank, Msm, r, 0, r, n, 1.f, 0.f, Wn, r, st);
    } else {
      cudaMemsetAsync(a, 0, (size_t)m * r * sizeof(float), st);
      cudaMemsetAsync(Wn, 0, (size_t)n * r * sizeof(float), st);
      launch_spmm(supports[t], gv, support_nnz[t], n, Y2p[t], r, r, 0, a, r, st);
      launch_spmm(supports[t], gv, support_nnz[t], n, ZY2p[t], r, r, 1, Wn, r, st);
    }
    // Wn += Z^T a;  gY2 = (I - P) Wn = Wn - Y2p (Y2^T Wn)
    E.mul(sZ, 1, a, r, Y2T);
    launch_axpy(Y2T, Wn, (int64_t)n * r, 1.f, st);
    launch_cross_gram(Qk[t], r, r, Wn, r, r, n, cpart, kCrossParts, Msm, r, st);
    launch_tall_small_d(Qk[t], r, r, Msm, r, 0, r, n, -1.f, 1.f, Wn, r, st);     // Wn = (I - Q Q^T) Wn = gY2
    E.mul(sZ, 0, Wn, r, Zg);                                    // Z gY2
    // factors of gZ_t: [a | A2 | Z gY2] [Y2 | gY2 | A1]^T
    const float *const us[3] = {a, A2[t], Zg}, *const vs[3] = {Y2[t], Wn, A1};
    launch_pack3(us, vs, m, n, r, Uf, Vf, ldf, st);
    launch_outer_acc(Uf, ldf, Vf, ldf, R3, m, n, t == T - 1 ? 0.f : 1.f, dX, lddx, st);
    // on Omega_{t-1}: gZ_t goes to L_{t-1} (next G) instead of X
    if (t > 0 && support_nnz[t - 1] > 0)
      launch_eval_lr(supports[t - 1], support_nnz[t - 1], n, Uf, ldf, Vf, ldf, R3, gv, dX, lddx, st);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_static_error("godec_backward: %s", cudaGetErrorString(e));
    return GODEC_ERR_CUDA;
  }
  return GODEC_OK;
}
