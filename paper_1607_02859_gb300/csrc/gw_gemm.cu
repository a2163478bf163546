// Complex GEMM on CUDA cores (FP32 or FP64), used by the SIMT precisions of
// the Green's-function contraction and by the blocked Cholesky / triangular
// inverse of the screening step.  64x64 output tile per 256-thread CTA, 4x4
// complex outputs per thread on an interleaved (stride-16) pattern so that the
// shared-memory reads of a warp are broadcasts or consecutive.
#include <algorithm>

#include "gw_kernels.h"

namespace gw {

template <typename T>
struct GemmP {
  using C = typename cpx<T>::t;
  int M, N, K;
  C alpha;
  T beta;
  const C* A;
  long lda;
  const C* B;
  long ldb;
  C* Cm;
  long ldc;
  const T* kscale;
  long sA, sB, sC;
};

// chi_simt_kernel's arguments
template <typename T>
struct ChiSimt {
  using C = typename cpx<T>::t;
  const C* psi;           // [n_b][nr]
  int nr, rows, r0, n_occ, n_b;
  const T* scale;         // band factors of time z at z * s_scale
  long s_scale;
  C* out;                 // chi rows r0 .. of time z at z * s_out
  long s_out;
  T a_occ[32], a_un[32];
};

template <typename T, int AKM, bool AC, int BNK, bool BC, bool SCALE, int TRI>
__global__ void __launch_bounds__(256) cgemm_kernel(GemmP<T> p) {
  using C = typename cpx<T>::t;
  constexpr int BM = 64, BN = 64, BK = 8, PAD = 1;
  __shared__ C As[2][BK][BM + PAD];
  __shared__ C Bs[2][BK][BN + PAD];
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  if (TRI && n0 > m0 + BM - 1) return;
  p.A += blockIdx.z * p.sA;
  p.B += blockIdx.z * p.sB;
  p.Cm += blockIdx.z * p.sC;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  // FP32 sums are blocked: acc collects KBLK terms of k, then is added to tot.
  // A sequential FP32 sum over K terms has a relative rounding error growing
  // like u sqrt(K/2); blocking by ~sqrt(K) brings it to ~u K^(1/4) (4x less at
  // K = 1024) for one extra add per KBLK terms.
  constexpr int KBLK = sizeof(T) == 4 ? 32 : 0;
  C acc[4][4], tot[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = tot[i][j] = mk(T(0), T(0));
  const int kbeg = TRI == 2 ? m0 : 0;
  // the next BK terms are on their way from memory while these are summed
  C va[2], vb[2];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = tid + 256 * q;
      int ml, kl;
      if (AKM) { kl = e / BM; ml = e % BM; } else { ml = e / BK; kl = e % BK; }
      const int m = m0 + ml, k = k0 + kl;
      C v = mk(T(0), T(0));
      if (m < p.M && k < p.K) {
        v = AKM ? p.A[(long)k * p.lda + m] : p.A[(long)m * p.lda + k];
        if (AC) v = cconj(v);
        if (SCALE) v = cscale(v, p.kscale[k]);
      }
      va[q] = v;
      int nl, kb;
      if (BNK) { nl = e / BK; kb = e % BK; } else { kb = e / BN; nl = e % BN; }
      const int n = n0 + nl, kk = k0 + kb;
      C w = mk(T(0), T(0));
      if (n < p.N && kk < p.K) {
        w = BNK ? p.B[(long)n * p.ldb + kk] : p.B[(long)kk * p.ldb + n];
        if (BC) w = cconj(w);
      }
      vb[q] = w;
    }
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = tid + 256 * q;
      if (AKM) As[buf][e / BM][e % BM] = va[q];
      else As[buf][e % BK][e / BK] = va[q];
      if (BNK) Bs[buf][e % BK][e / BK] = vb[q];
      else Bs[buf][e / BN][e % BN] = vb[q];
    }
  };
  fetch(kbeg);
  put(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = kbeg; k0 < p.K; k0 += BK, buf ^= 1) {
    if (KBLK && k0 != kbeg && (k0 - kbeg) % KBLK == 0) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          tot[i][j] = cadd(tot[i][j], acc[i][j]);
          acc[i][j] = mk(T(0), T(0));
        }
    }
    const bool more = k0 + BK < p.K;
    if (more) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      C a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[buf][kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[buf][kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = cfma(a[i], b[j], acc[i][j]);
    }
    if (more) put(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int m = m0 + ty + 16 * i, n = n0 + tx + 16 * j;
      if (m >= p.M || n >= p.N) continue;
      if (TRI && m < n) continue;
      C v = cmul(p.alpha, cadd(tot[i][j], acc[i][j]));
      C* dst = p.Cm + (long)m * p.ldc + n;
      if (p.beta != T(0)) v = cadd(v, cscale(*dst, p.beta));
      *dst = v;
    }
}

// chi rows of the triangle R' <= r on CUDA cores (Eqs. Green_occ, Green_unocc and
// chi_rr in one pass): per 64 x 64 tile the sums over the occupied bands, parked in
// shared memory, then those over the unoccupied ones, and
//   out = -2 G_occ conj(G_unocc), halved on the diagonal and zero above it.
// G never goes to memory: two stored products and a product read back in the row
// transform cost 521 us of the 12^3 cell's 8 times in FP32 where this takes 360 (12.9 and
// 11.3 ms in FP64, at 1.12 TFLOP/s of its ALU).
// grid z: the times of one set of orbitals, in one launch so that the triangle's tiles
// (378 at 12^3) fill the SMs evenly.  Sums, blocking and prefetch as in cgemm_kernel.
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 1) chi_simt_kernel(const __grid_constant__ ChiSimt<T> p) {
  using C = typename cpx<T>::t;
  constexpr int BM = 64, BN = 64, BK = 8, PAD = 1;
  constexpr int KBLK = sizeof(T) == 4 ? 32 : 0;
  __shared__ C As[2][BK][BM + PAD];
  __shared__ C Bs[2][BK][BN + PAD];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* occ = reinterpret_cast<C*>(smem_raw);          // [16][256] this thread's G_occ sums
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN, z = blockIdx.z;
  if (n0 > p.r0 + m0 + BM - 1) return;              // no R' <= r in the tile
  const T* sc = p.scale + z * p.s_scale;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  C acc[4][4], tot[4][4], va[2], vb[2];
  auto fetch = [&](int k0, int k_end) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = tid + 256 * q, k = k0 + e / BM, l = e % BM;
      va[q] = vb[q] = mk(T(0), T(0));
      if (k < k_end) {
        const C* row = p.psi + (long)k * p.nr;
        if (m0 + l < p.rows) va[q] = cscale(row[p.r0 + m0 + l], sc[k]);
        if (n0 + l < p.nr) vb[q] = cconj(row[n0 + l]);
      }
    }
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = tid + 256 * q;
      As[buf][e / BM][e % BM] = va[q];
      Bs[buf][e / BN][e % BN] = vb[q];
    }
  };
  auto sums = [&](int k_beg, int k_end) {           // tot = sum over the bands k_beg .. k_end-1
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = tot[i][j] = mk(T(0), T(0));
    __syncthreads();
    fetch(k_beg, k_end);
    put(0);
    __syncthreads();
    int buf = 0;
    for (int k0 = k_beg; k0 < k_end; k0 += BK, buf ^= 1) {
      if (KBLK && k0 != k_beg && (k0 - k_beg) % KBLK == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            tot[i][j] = cadd(tot[i][j], acc[i][j]);
            acc[i][j] = mk(T(0), T(0));
          }
      }
      const bool more = k0 + BK < k_end;
      if (more) fetch(k0 + BK, k_end);
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        C a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = As[buf][kk][ty + 16 * i];
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = Bs[buf][kk][tx + 16 * j];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = cfma(a[i], b[j], acc[i][j]);
      }
      if (more) put(buf ^ 1);
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) tot[i][j] = cadd(tot[i][j], acc[i][j]);
  };
  sums(0, p.n_occ);
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) occ[(i * 4 + j) * 256 + tid] = tot[i][j];
  sums(p.n_occ, p.n_b);
  const T ao = p.a_occ[z], au = p.a_un[z];
  C* out = p.out + z * p.s_out;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int m = m0 + ty + 16 * i, n = n0 + tx + 16 * j, r = p.r0 + m;
      if (m >= p.rows || n >= p.nr) continue;
      const T f = n < r ? T(-2) : (n == r ? T(-1) : T(0));
      out[(long)m * p.nr + n] = cscale(cmulc(cscale(occ[(i * 4 + j) * 256 + tid], ao), cscale(tot[i][j], au)), f);
    }
}

template <typename T>
static gw_status run_chi_simt(gw_ctx* ctx, const GridInfo& g, int n_b, int n_occ, const void* psi, const void* scale,
                              const GreenScales* gs, int nt, int r0, int rows, void* out, long s_out, cudaStream_t st) {
  using C = typename cpx<T>::t;
  ChiSimt<T> p;
  p.psi = static_cast<const C*>(psi);
  p.nr = g.nr;
  p.rows = rows;
  p.r0 = r0;
  p.n_occ = n_occ;
  p.n_b = n_b;
  p.scale = static_cast<const T*>(scale);
  p.s_scale = (long)n_b * (8 / (long)sizeof(T));     // per-time regions of n_b 8-byte slots
  p.out = static_cast<C*>(out);
  p.s_out = s_out;
  for (int z = 0; z < nt; ++z) {
    p.a_occ[z] = (T)gs[z].amax_occ;
    p.a_un[z] = (T)gs[z].amax_unocc;
  }
  const dim3 grid((std::min(g.nr, r0 + rows) + 63) / 64, (rows + 63) / 64, nt);
  double work = 0;
  for (int m = 0; m < rows; m += 64) work += (double)std::min(64, rows - m) * std::min(g.nr, r0 + m + 64);
  const size_t smem = 16 * 256 * sizeof(C);
  gw_status rc = cuda_check(ctx, cudaFuncSetAttribute(chi_simt_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                      (int)smem),
                            "cudaFuncSetAttribute");
  if (rc) return rc;
  KTimer kt(ctx, KF_CGEMM_SIMT, 8.0 * nt * work * n_b, st);
  chi_simt_kernel<T><<<grid, 256, smem, st>>>(p);
  return launch_check(ctx, "chi_simt_kernel");
}

gw_status launch_chi_simt(gw_ctx* ctx, gw_prec prec, const GridInfo& g, int n_b, int n_occ, const void* psi,
                          const void* scale, const GreenScales* gs, int nt, int r0, int rows, void* out, long s_out,
                          cudaStream_t st) {
  if (nt < 1 || nt > 32) return fail(ctx, GW_ERR_SHAPE, "1 to 32 times per launch");
  return is_fp64(prec) ? run_chi_simt<double>(ctx, g, n_b, n_occ, psi, scale, gs, nt, r0, rows, out, s_out, st)
                       : run_chi_simt<float>(ctx, g, n_b, n_occ, psi, scale, gs, nt, r0, rows, out, s_out, st);
}

template <typename T>
static gw_status run_gemm(gw_ctx* ctx, const GemmArgs& a, cudaStream_t st) {
  using C = typename cpx<T>::t;
  GemmP<T> p;
  p.M = a.M;
  p.N = a.N;
  p.K = a.K;
  p.alpha = mk(T(a.alpha_re), T(a.alpha_im));
  p.beta = T(a.beta);
  p.A = (const C*)a.A;
  p.lda = a.lda;
  p.B = (const C*)a.B;
  p.ldb = a.ldb;
  p.Cm = (C*)a.C;
  p.ldc = a.ldc;
  p.kscale = (const T*)a.kscale;
  p.sA = a.sA;
  p.sB = a.sB;
  p.sC = a.sC;
  dim3 grid((a.N + 63) / 64, (a.M + 63) / 64, a.batch > 0 ? a.batch : 1);
  if (grid.y > 65535) return fail(ctx, GW_ERR_SHAPE, "GEMM M too large");
#define GW_GEMM_CASE(AKM, AC, BNK, BC, SC, TRI)                                                   \
  if (a.a_km == AKM && a.a_conj == AC && a.b_nk == BNK && a.b_conj == BC && (a.kscale != nullptr) == SC && \
      a.tri == TRI) {                                                                               \
    KTimer kt(ctx, KF_CGEMM_SIMT, grid.z * gemm_flops(a.M, a.N, a.K, TRI), st);                   \
    cgemm_kernel<T, AKM, AC, BNK, BC, SC, TRI><<<grid, 256, 0, st>>>(p);                           \
    return launch_check(ctx, "cgemm_kernel");                                                       \
  }
  GW_GEMM_CASE(1, false, 0, true, true, 0)    // Green's functions: psi^T diag(s) conj(psi)
  GW_GEMM_CASE(0, false, 1, true, false, 1)   // Hermitian rank-k update: C -= L21 L21^H (lower)
  GW_GEMM_CASE(0, false, 0, false, false, 0)  // triangular-inverse update: C -= L_below X_i
  GW_GEMM_CASE(1, true, 0, false, false, 2)   // L^{-H} L^{-1}, lower triangle
  GW_GEMM_CASE(0, false, 0, false, false, 1)
  GW_GEMM_CASE(0, false, 1, true, false, 0)   // A B^H (plane-wave self-energy: h c^H)
#undef GW_GEMM_CASE
  return fail(ctx, GW_ERR_UNSUPPORTED, "GEMM layout combination not compiled");
}

gw_status launch_gemm(gw_ctx* ctx, gw_prec prec, const GemmArgs& a, cudaStream_t st) {
  if (a.M <= 0 || a.N <= 0) return GW_OK;
  return is_fp64(prec) ? run_gemm<double>(ctx, a, st) : run_gemm<float>(ctx, a, st);
}

}  // namespace gw
