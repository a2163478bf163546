// Screened interaction W~ (Eqs. W_tot, bareV, die, W_correlated).
//
// With chi~ = v^{1/2} chi v^{1/2} Hermitian negative semidefinite, the matrix
// eps~ = 1 - chi~ is Hermitian positive definite with eps~ >= 1, so
//   W~ = v^{1/2} (eps~^{-1} - 1) v^{1/2}
// follows from a Cholesky factorisation without pivoting.  The identity is
// carried implicitly so that nothing is ever formed as "1 + small" and then
// subtracted again (at large omega chi~ is tiny and such a round trip would
// lose its low digits):
//   B = eps~ - 1 = -chi~,  eps~ = L L^H with L = 1 + K on the diagonal,
//   L_jj - 1 = B'_jj / (1 + sqrt(1 + B'_jj))  (B' = B after the updates),
//   L^{-1} = 1 + P,
//   eps~^{-1} - 1 = P + P^H + P^H P.
// N^3/2 complex multiply-adds in all (Cholesky, L^{-1}, P^H P: N^3/6 each),
// instead of the N^3 + N^3/6 of a solve against chi~ with N right-hand sides.
//
// The frequencies are independent, so every launch works on a batch of them
// (grid z): the chain of small sequential launches on the diagonal blocks is
// paid once per batch instead of once per frequency, and the GEMMs grow.
//  * CUDA-core precisions: 64-column panels; the trailing updates are CUDA-core
//    complex GEMMs.
//  * tensor-core precisions: 512-column panels whose 512 x 512 diagonal blocks
//    are factored and inverted on CUDA cores; everything with a 512-wide inner
//    dimension is a tcgen05 GEMM with split 16-bit products:
//      L21 = A21 (1 + P11)^H,  A22 -= L21 L21^H,
//      P_i[:, <k0] += P_ii P_i[:, <k0],  rows below -= L_li (1 + P_i),
//      X = P^H P (one frequency per launch: the largest GEMM of the step).
#include <cmath>
#include <type_traits>

#include "gw_kernels.h"
#include "gw_tc.h"

namespace gw {

constexpr int kNB = 64;     // CUDA-core panel width
constexpr int kTB = 512;    // tensor-core panel width

// One CTA per row a (and batch entry): the lower part b <= a of the row.
template <typename T>
__global__ void __launch_bounds__(256) build_eps_kernel(const typename cpx<T>::t* __restrict__ chi, long s_chi,
                                                        const double* __restrict__ vh,
                                                        typename cpx<T>::t* __restrict__ E, long s_e, int n) {
  const int a = blockIdx.x;
  const double va = vh[a];
  const auto* src = chi + blockIdx.y * s_chi + (long)a * n;
  auto* dst = E + blockIdx.y * s_e + (long)a * n;
  for (int b = threadIdx.x; b <= a; b += blockDim.x) {
    const T vv = T(va * vh[b]);
    const auto x = src[b];
    dst[b] = mk(-vv * x.x, -vv * x.y);
  }
}

// 1 / sqrt(x): the CUDA estimate with one Newton step in FP32 (the exact square
// root and division sit on the pivot chain below), the quotient in FP64.
__device__ __forceinline__ float inv_sqrt(float x) {
  const float r = rsqrtf(x);
  return fmaf(0.5f * r, fmaf(-x * r, r, 1.0f), r);
}
__device__ __forceinline__ double inv_sqrt(double x) { return 1.0 / sqrt(x); }

// Cholesky factor (K form) and inverse of the kb x kb diagonal block of every
// batch entry: L (diagonal L_jj - 1) back into A, L^{-1} - 1 into P (lower).
//
// One CTA per entry; the chain of kb pivots bounds it (FP32).  Both triangles
// live in registers, a 4 x 4 cyclic block each per thread of a 16 x 16 grid,
// and advance together: with the raw column j of the factor and the raw row j
// of the inverse published in (double-buffered) shared memory behind one
// barrier, together with 1 / L_jj from the thread that holds the pivot (a square
// root and a division of every thread would cost more FP64 issue than the updates of
// a small block), every thread scales them itself and applies
//   S -= l l^H,   X[i > j] -= l_i x_j.
// Only the 16-wide register blocks that column j touches are updated, of a short
// block only those that hold its rows.  The inverse turns the triangular solves of the panel into products (below): one
// thread per row of a solve walked 64 columns serially (68 us a panel, and 74 us
// for the inverse's rows, whatever the size).  Screening 12 frequencies of 1536
// G vectors (fp16x3) went from 7.02 to 3.79 ms, 2 x 8192 with refinement from
// 185 to 170 ms; FP64, 4 x 513, from 18.1 to 13.1 ms, FP32, 8 x 300, from 1.05 to 0.46.
template <typename T>
__global__ void __launch_bounds__(256) potrf_inv_kernel(typename cpx<T>::t* A, long lda, long s_a,
                                                        typename cpx<T>::t* P, long ldp, long s_p, int kb, int* flag,
                                                        int col0) {
  using C = typename cpx<T>::t;
  static_assert(kNB == 64, "4 x 4 blocks of a 16 x 16 thread grid");
  __shared__ C col[2][kNB], row[2][kNB];
  __shared__ T piv[2];                         // 1 / L_jj
  A += blockIdx.z * s_a;
  P += blockIdx.z * s_p;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  C S[4][4], X[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int i = ty + 16 * a, c = tx + 16 * b;
      S[a][b] = i < kb && c <= i ? A[(long)i * lda + c] : mk(T(0), T(0));
      X[a][b] = mk(T(i == c ? 1 : 0), T(0));
    }
#pragma unroll
  for (int jb = 0; jb < 4; ++jb) {
#pragma unroll 1
    for (int jj = 0; jj < 16; ++jj) {
      const int j = 16 * jb + jj;
      if (j >= kb) break;
      const int buf = j & 1;
      if (tx == jj)
#pragma unroll
        for (int a = jb; a < 4; ++a) col[buf][ty + 16 * a] = S[a][jb];
      if (ty == jj)
#pragma unroll
        for (int b = 0; b <= jb; ++b) row[buf][tx + 16 * b] = X[jb][b];
      T d = T(0);
      bool bad = false;
      if (tx == jj && ty == jj) {
        d = S[jb][jb].x;                       // eps~_jj - 1 after the updates
        bad = !(T(1) + d > T(0));
        if (bad) d = T(0);
        piv[buf] = inv_sqrt(T(1) + d);
      }
      __syncthreads();
      const T inv = piv[buf];
      C l[4], lc[4], xr[4];
#pragma unroll
      for (int a = jb; a < 4; ++a) {
        l[a] = cscale(col[buf][ty + 16 * a], inv);
        lc[a] = cscale(col[buf][tx + 16 * a], inv);
      }
#pragma unroll
      for (int b = 0; b <= jb; ++b) xr[b] = cscale(row[buf][tx + 16 * b], inv);
      if (tx == jj) {
#pragma unroll
        for (int a = jb; a < 4; ++a)
          if (ty + 16 * a > j) S[a][jb] = l[a];
        if (ty == jj) {
          S[jb][jb] = mk(d / (T(1) + sqrt(T(1) + d)), T(0));   // L_jj - 1
          if (bad && atomicCAS(flag, 0, 1) == 0) {
            flag[1] = col0 + j;
            flag[2] = blockIdx.z;
          }
        }
      }
      if (ty == jj)
#pragma unroll
        for (int b = 0; b <= jb; ++b) X[jb][b] = xr[b];
      if (ty <= jj) l[jb] = mk(T(0), T(0));    // rows up to j and columns up to j are final
      if (tx <= jj) lc[jb] = mk(T(0), T(0));
#pragma unroll
      for (int a = jb; a < 4; ++a) {
        if (16 * a >= kb) break;                // rows past a short block
        // the product first: one rounding at the size of S per update.  As two multiply-adds onto S
        // each left W~ 10 to 15% further off.
#pragma unroll
        for (int b = jb; b <= a; ++b) S[a][b] = csub(S[a][b], cmulc(l[a], lc[b]));
#pragma unroll
        for (int b = 0; b <= jb; ++b) X[a][b] = csub(X[a][b], cmul(l[a], xr[b]));
      }
    }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b <= a; ++b) {
      const int i = ty + 16 * a, c = tx + 16 * b;
      if (i >= kb || c > i) continue;
      A[(long)i * lda + c] = S[a][b];
      const T k = S[a][b].x;                   // on the diagonal: (1 + K)^{-1} - 1 = -K / (1 + K)
      P[(long)i * ldp + c] = i == c ? mk(-k / (T(1) + k), T(0)) : X[a][b];
    }
}

constexpr int kPR = 32;     // rows (columns) of a panel product per CTA

// Shared memory of the two panel products: the inverted diagonal block and the tile;
// for the right one also the diagonal block itself and the product.
template <typename T>
constexpr size_t panel_smem(bool right) {
  return (right ? 2 : 1) * sizeof(typename cpx<T>::t) * (kNB * (kNB + 1) + kPR * (kNB + 1));
}

// R x W elements of a row-major matrix on their way from memory, all in flight at
// once (256 threads; 0 outside): in a loop of loads and stores each of them was waited
// for, 13 of the 18 us of a panel.
template <int R, int W, typename C>
struct Tile {
  static constexpr int N = R * W / 256, RQ = 256 / W;
  C v[N];
  template <typename In>
  __device__ __forceinline__ void load(const C* src, long ld, In in) {
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const int i = RQ * q + (int)threadIdx.x / W, c = threadIdx.x % W;
      v[q] = C{};
      if (in(i, c)) v[q] = src[(long)i * ld + c];
    }
  }
  __device__ __forceinline__ void store(C* dst, int ld) const {
#pragma unroll
    for (int q = 0; q < N; ++q) dst[(RQ * q + (int)threadIdx.x / W) * ld + threadIdx.x % W] = v[q];
  }
};

// Rows below the diagonal block: L21 = A21 L11^{-H}, in place, kPR rows per CTA and
// 2 x 4 outputs per thread, with P11 = L11^{-1} - 1 and K11 = L11 - 1 lower triangular,
// so that the sum of each group of 16 columns stops at its last column:
//   Y = A21 + A21 P11^H,   R = A21 - Y - Y K11^H,   L21 = Y + R + R P11^H.
// The product alone leaves a residual of cond(L11) roundings of A21, which the updates
// of all later columns take up; the correction brings it back to that of a solve.
// eps~ with a largest eigenvalue of 1e5, 700 G vectors: W~ off by 3.1e-3 in FP32 with the
// product, by 2.0e-4 with a solve of every row (FP64 6.3e-12 and 2.9e-12).
template <typename T>
__global__ void __launch_bounds__(256) panel_right_kernel(typename cpx<T>::t* A, const typename cpx<T>::t* L, long lda,
                                                          long s_a, const typename cpx<T>::t* P, long ldp, long s_p,
                                                          int kb, int rows) {
  using C = typename cpx<T>::t;
  constexpr int LD = kNB + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* Ps = reinterpret_cast<C*>(smem_raw);          // [kNB][LD]
  C* Ks = Ps + kNB * LD;                            // [kNB][LD]
  C* As = Ks + kNB * LD;                            // [kPR][LD] A21, then R
  C* Ys = As + kPR * LD;                            // [kPR][LD]
  A += blockIdx.z * s_a;
  L += blockIdx.z * s_a;
  P += blockIdx.z * s_p;
  const int r0 = blockIdx.x * kPR;
  {
    auto lower = [&](int i, int c) { return i < kb && c <= i; };
    Tile<kNB, kNB, C> tp, tk;
    Tile<kPR, kNB, C> ta;
    tp.load(P, ldp, lower);
    tk.load(L, lda, lower);
    ta.load(A + (long)r0 * lda, lda, [&](int i, int c) { return r0 + i < rows && c < kb; });
    tp.store(Ps, LD);
    tk.store(Ks, LD);
    ta.store(As, LD);
  }
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  C acc[2][4], y[2][4];
  auto times = [&](const C* X, const C* W) {       // acc = this thread's elements of X W^H
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int a = 0; a < 2; ++a) acc[a][b] = mk(T(0), T(0));
#pragma unroll
    for (int pb = 0; pb < 4; ++pb) {
#pragma unroll 4
      for (int pp = 0; pp < 16; ++pp) {
        const int p = 16 * pb + pp;
        const C a0 = X[ty * LD + p], a1 = X[(ty + 16) * LD + p];
#pragma unroll
        for (int b = pb; b < 4; ++b) {
          const C w = W[(tx + 16 * b) * LD + p];
          acc[0][b] = cfmac(a0, w, acc[0][b]);
          acc[1][b] = cfmac(a1, w, acc[1][b]);
        }
      }
    }
  };
  times(As, Ps);
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int at = (ty + 16 * a) * LD + tx + 16 * b;
      y[a][b] = Ys[at] = cadd(As[at], acc[a][b]);
    }
  __syncthreads();
  times(Ys, Ks);
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      C& r = As[(ty + 16 * a) * LD + tx + 16 * b];
      r = csub(csub(r, y[a][b]), acc[a][b]);
    }
  __syncthreads();
  times(As, Ps);
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int i = ty + 16 * a;
    if (r0 + i >= rows) continue;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int c = tx + 16 * b;
      if (c < kb) A[(long)(r0 + i) * lda + c] = cadd(y[a][b], cadd(As[i * LD + c], acc[a][b]));
    }
  }
}

// One block row of P = L^{-1} - 1, left of its diagonal block: Y <- L_ii^{-1} Y =
// Y + P_ii Y for the kb rows and ncols columns at Y, in place, kPR columns per
// CTA.  CTAs past those columns set up the rows below instead: P[r][col0 ..] =
// -L[r][col0 ..] (the identity part of 1 + P in the update of those rows).
template <typename T>
__global__ void __launch_bounds__(256) panel_left_kernel(const typename cpx<T>::t* P, long ldp, long s_p,
                                                         typename cpx<T>::t* Y, int kb, int ncols,
                                                         const typename cpx<T>::t* Lb, long ldl, long s_l,
                                                         typename cpx<T>::t* Pb, int below) {
  using C = typename cpx<T>::t;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int mul_ctas = (ncols + kPR - 1) / kPR;
  if ((int)blockIdx.x >= mul_ctas) {
    Lb += blockIdx.z * s_l;
    Pb += blockIdx.z * s_p;
    const int r0 = ((int)blockIdx.x - mul_ctas) * kPR;
    for (int e = threadIdx.x; e < kPR * kNB; e += 256) {
      const int r = r0 + e / kNB, c = e % kNB;
      if (r >= below || c >= kb) continue;
      const C v = Lb[(long)r * ldl + c];
      Pb[(long)r * ldp + c] = mk(-v.x, -v.y);
    }
    return;
  }
  C* Ps = reinterpret_cast<C*>(smem_raw);          // [kNB][kNB + 1]
  C* Ys = Ps + kNB * (kNB + 1);                     // [kNB][kPR] (fits the row tile's space)
  P += blockIdx.z * s_p;
  Y += blockIdx.z * s_p;
  const int c0 = blockIdx.x * kPR;
  {
    Tile<kNB, kNB, C> tp;
    Tile<kNB, kPR, C> ty;
    tp.load(P, ldp, [&](int i, int c) { return i < kb && c <= i; });
    ty.load(Y + c0, ldp, [&](int i, int c) { return i < kb && c0 + c < ncols; });
    tp.store(Ps, kNB + 1);
    ty.store(Ys, kPR);
  }
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  C acc[4][2];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b] = mk(T(0), T(0));
#pragma unroll
  for (int pb = 0; pb < 4; ++pb) {
#pragma unroll 4
    for (int pp = 0; pp < 16; ++pp) {
      const int p = 16 * pb + pp;
      const C y0 = Ys[p * kPR + tx], y1 = Ys[p * kPR + tx + 16];
#pragma unroll
      for (int a = pb; a < 4; ++a) {
        const C w = Ps[(ty + 16 * a) * (kNB + 1) + p];
        acc[a][0] = cfma(w, y0, acc[a][0]);
        acc[a][1] = cfma(w, y1, acc[a][1]);
      }
    }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int i = ty + 16 * a;
    if (i >= kb) continue;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int c = tx + 16 * b;
      if (c0 + c < ncols) Y[(long)i * ldp + c0 + c] = cadd(Ys[i * kPR + c], acc[a][b]);
    }
  }
}

// P[rows below][col0 .. col0+kb) = -L[rows below][col0 .. col0+kb): the identity
// part of (1 + P) contributes L_li * 1 to the update of the rows below block row i.
template <typename T>
__global__ void neg_copy_kernel(const typename cpx<T>::t* __restrict__ Lm, long ldl, long s_l,
                                typename cpx<T>::t* __restrict__ P, long ldp, long s_p, int row0, int rows, int col0,
                                int kb) {
  const long r = row0 + (long)blockIdx.x;
  if ((int)blockIdx.x >= rows) return;
  Lm += blockIdx.z * s_l;
  P += blockIdx.z * s_p;
  for (int c = threadIdx.x; c < kb; c += blockDim.x) {
    const auto v = Lm[r * ldl + col0 + c];
    P[r * ldp + col0 + c] = mk(-v.x, -v.y);
  }
}

// Zero `cols` columns of `rows` rows (leading dimension ld) per batch entry.
template <typename T>
__global__ void zero_block_kernel(typename cpx<T>::t* __restrict__ P, long ld, long s_p, int cols) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= cols) return;
  P[blockIdx.z * s_p + (long)blockIdx.y * ld + b] = mk(T(0), T(0));
}

// X = P^H P + P + P^H (lower triangle, in place over P^H P); one CTA per row.
template <typename T>
__global__ void __launch_bounds__(256) assemble_kernel(typename cpx<T>::t* __restrict__ X, long s_x,
                                                       const typename cpx<T>::t* __restrict__ P, long s_p, int n) {
  const int a = blockIdx.x;
  auto* xr = X + blockIdx.y * s_x + (long)a * n;
  const auto* pr = P + blockIdx.y * s_p + (long)a * n;
  for (int b = threadIdx.x; b <= a; b += blockDim.x) {
    auto x = xr[b];
    const auto p = pr[b];
    x.x += a == b ? T(2) * p.x : p.x;
    x.y += a == b ? T(0) : p.y;
    xr[b] = x;
  }
}

// W~[a][b] = v_a X[a][b] v_b, both triangles from the lower one.  One 32 x 32
// tile pair (ta >= tb) per CTA through shared memory, so that the mirrored
// (conjugate-transposed) writes are row segments too.
template <typename T>
__global__ void __launch_bounds__(256) finalize_kernel(const typename cpx<T>::t* __restrict__ Xl, long s_x,
                                                       const double* __restrict__ vh, typename cpx<T>::t* __restrict__ W,
                                                       long s_w, int n) {
  using C = typename cpx<T>::t;
  const int ta = blockIdx.y, tb = blockIdx.x;
  if (tb > ta) return;
  __shared__ C t[32][33];
  Xl += blockIdx.z * s_x;
  W += blockIdx.z * s_w;
  const int a0 = ta * 32, b0 = tb * 32;
  for (int y = threadIdx.y; y < 32; y += blockDim.y) {
    const int a = a0 + y, b = b0 + threadIdx.x;
    C v = mk(T(0), T(0));
    if (a < n && b < n) {
      // lower element, or the mirror of one inside a diagonal tile
      v = b <= a ? Xl[(long)a * n + b] : cconj(Xl[(long)b * n + a]);
      v = cscale(v, T(vh[a] * vh[b]));
      W[(long)a * n + b] = v;
    }
    t[y][threadIdx.x] = v;
  }
  if (ta == tb) return;
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += blockDim.y) {
    const int b = b0 + y, a = a0 + threadIdx.x;
    if (a < n && b < n) W[(long)b * n + a] = cconj(t[threadIdx.x][y]);
  }
}

// y = F z in FP64 for the Hermitian F given by its lower triangle Mlow:
// F[a][b] = s_a s_b (Mlow or conj of the mirrored entry) - sub * delta_ab.
template <typename T>
__global__ void __launch_bounds__(256) hemv_probe_kernel(const typename cpx<T>::t* __restrict__ Mlow,
                                                         const double* __restrict__ sv, double sub,
                                                         const double2* __restrict__ z, double2* __restrict__ y,
                                                         int n) {
  const int a = blockIdx.x;
  double re = 0, im = 0;
  for (int b = threadIdx.x; b < n; b += blockDim.x) {
    double2 m;
    if (b <= a) {
      auto v = Mlow[(long)a * n + b];
      m = make_double2(v.x, v.y);
    } else {
      auto v = Mlow[(long)b * n + a];
      m = make_double2(v.x, -v.y);
    }
    const double s = sv ? sv[a] * sv[b] : 1.0;
    m.x *= s;
    m.y *= s;
    if (a == b) m.x -= sub;
    re += m.x * z[b].x - m.y * z[b].y;
    im += m.x * z[b].y + m.y * z[b].x;
  }
  __shared__ double sr[256], si[256];
  sr[threadIdx.x] = re;
  si[threadIdx.x] = im;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      sr[threadIdx.x] += sr[threadIdx.x + w];
      si[threadIdx.x] += si[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) y[a] = make_double2(sr[0], si[0]);
}

// A batch of B frequencies whose matrices are `ms` elements apart.
struct Batch {
  int B;
  long ms;
};

template <typename T>
static gw_status set_attrs(gw_ctx* ctx) {
  gw_status rc = cuda_check(ctx, cudaFuncSetAttribute(panel_right_kernel<T>,
                                                      cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                      (int)panel_smem<T>(true)),
                            "cudaFuncSetAttribute");
  if (!rc && panel_smem<T>(false) > 48 * 1024)
    rc = cuda_check(ctx, cudaFuncSetAttribute(panel_left_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)panel_smem<T>(false)),
                    "cudaFuncSetAttribute");
  return rc;
}

// Cholesky (lower, K form on the diagonal) of the n x n block at a (leading
// dimension lda) of every batch entry, on CUDA cores, 64-column panels; the
// inverses (minus 1) of the diagonal blocks go to the diagonal of the block at
// p, which is zeroed otherwise.
template <typename T>
static gw_status chol_simt(gw_ctx* ctx, gw_prec prec, typename cpx<T>::t* a, long lda, typename cpx<T>::t* p, long ldp,
                           int n, int col0, Batch bt, cudaStream_t st) {
  gw_status rc;
  zero_block_kernel<T><<<dim3((n + 127) / 128, n, bt.B), 128, 0, st>>>(p, ldp, bt.ms, n);
  if ((rc = launch_check(ctx, "zero_block_kernel"))) return rc;
  for (int k0 = 0; k0 < n; k0 += kNB) {
    const int kb = std::min(kNB, n - k0);
    auto* pii = p + (long)k0 * ldp + k0;
    potrf_inv_kernel<T><<<dim3(1, 1, bt.B), 256, 0, st>>>(a + (long)k0 * lda + k0, lda, bt.ms, pii, ldp, bt.ms, kb,
                                                          ctx->dflag, col0 + k0);
    if ((rc = launch_check(ctx, "potrf_inv_kernel"))) return rc;
    const int rows = n - k0 - kb;
    if (rows <= 0) break;
    panel_right_kernel<T><<<dim3((rows + kPR - 1) / kPR, 1, bt.B), 256, panel_smem<T>(true), st>>>(
        a + (long)(k0 + kb) * lda + k0, a + (long)k0 * lda + k0, lda, bt.ms, pii, ldp, bt.ms, kb, rows);
    if ((rc = launch_check(ctx, "panel_right_kernel"))) return rc;
    GemmArgs g{};
    g.M = rows;
    g.N = rows;
    g.K = kb;
    g.alpha_re = -1;
    g.beta = 1;
    g.A = a + (long)(k0 + kb) * lda + k0;
    g.lda = lda;
    g.a_km = 0;
    g.B = a + (long)(k0 + kb) * lda + k0;
    g.ldb = lda;
    g.b_nk = 1;
    g.b_conj = true;
    g.C = a + (long)(k0 + kb) * lda + k0 + kb;
    g.ldc = lda;
    g.tri = 1;
    g.batch = bt.B;
    g.sA = g.sB = g.sC = bt.ms;
    if ((rc = launch_gemm(ctx, prec, g, st))) return rc;
  }
  return GW_OK;
}

// P = L^{-1} - 1 for the n x n lower factor L (K form diagonal) at Lm, in the
// n x n block at p as chol_simt left it (the inverted diagonal blocks, zero
// elsewhere), for every batch entry (CUDA cores).
template <typename T>
static gw_status inv_simt(gw_ctx* ctx, gw_prec prec, const typename cpx<T>::t* Lm, long ldl,
                          typename cpx<T>::t* p, long ldp, int n, Batch bt, cudaStream_t st) {
  gw_status rc;
  for (int k0 = 0; k0 < n; k0 += kNB) {
    const int kb = std::min(kNB, n - k0);
    const int ncols = k0 + kb, rows = n - k0 - kb;
    const int ctas = (k0 + kPR - 1) / kPR + (rows + kPR - 1) / kPR;
    if (ctas > 0) {
      panel_left_kernel<T><<<dim3(ctas, 1, bt.B), 256, panel_smem<T>(false), st>>>(
          p + (long)k0 * ldp + k0, ldp, bt.ms, p + (long)k0 * ldp, kb, k0, Lm + (long)(k0 + kb) * ldl + k0, ldl, bt.ms,
          p + (long)(k0 + kb) * ldp + k0, rows);
      if ((rc = launch_check(ctx, "panel_left_kernel"))) return rc;
    }
    if (rows <= 0) break;
    GemmArgs g{};
    g.M = rows;
    g.N = ncols;
    g.K = kb;
    g.alpha_re = -1;
    g.beta = 1;
    g.A = Lm + (long)(k0 + kb) * ldl + k0;
    g.lda = ldl;
    g.B = p + (long)k0 * ldp;
    g.ldb = ldp;
    g.C = p + (long)(k0 + kb) * ldp;
    g.ldc = ldp;
    g.batch = bt.B;
    g.sA = g.sB = g.sC = bt.ms;
    if ((rc = launch_gemm(ctx, prec, g, st))) return rc;
  }
  return GW_OK;
}

// |eps~ X z - chi~ z| / |chi~ z| over 4 seeded probes z, in FP64, with X the
// assembled lower triangle of eps~^{-1} - 1 (one frequency) and chi intact.
template <typename T>
static gw_status residual_probe(gw_ctx* ctx, int n, const typename cpx<T>::t* chi, const double* dvh,
                                const typename cpx<T>::t* e, double2* probe, double* resid_h, cudaStream_t st) {
  gw_status rc;
  double num = 0, den = 0;
  std::vector<double2> hz(n), hu(n), hw(n), hc(n);
  for (int q = 0; q < 4; ++q) {
    uint64_t sd = 0x9E3779B97F4A7C15ull * (q + 1);
    for (int i = 0; i < n; ++i) {
      sd = sd * 6364136223846793005ull + 1442695040888963407ull;
      const double u1 = ((sd >> 11) & ((1ull << 53) - 1)) / 9007199254740992.0;
      sd = sd * 6364136223846793005ull + 1442695040888963407ull;
      const double u2 = ((sd >> 11) & ((1ull << 53) - 1)) / 9007199254740992.0;
      hz[i] = make_double2(u1 - 0.5, u2 - 0.5);
    }
    double2 *z = probe, *u = probe + n, *w = probe + 2 * n, *c = probe + 3 * n;
    if ((rc = upload(ctx, z, hz.data(), sizeof(double2) * n, st))) return rc;
    hemv_probe_kernel<T><<<n, 256, 0, st>>>(e, nullptr, 0.0, z, u, n);       // u = X z
    hemv_probe_kernel<T><<<n, 256, 0, st>>>(chi, dvh, 0.0, u, w, n);         // w = chi~ u
    hemv_probe_kernel<T><<<n, 256, 0, st>>>(chi, dvh, 0.0, z, c, n);         // c = chi~ z
    if ((rc = launch_check(ctx, "hemv_probe_kernel"))) return rc;
    ctx->launches += 2;
    cudaMemcpyAsync(hu.data(), u, sizeof(double2) * n, cudaMemcpyDeviceToHost, st);
    cudaMemcpyAsync(hw.data(), w, sizeof(double2) * n, cudaMemcpyDeviceToHost, st);
    cudaMemcpyAsync(hc.data(), c, sizeof(double2) * n, cudaMemcpyDeviceToHost, st);
    if ((rc = cuda_check(ctx, cudaStreamSynchronize(st), "probe sync"))) return rc;
    for (int i = 0; i < n; ++i) {
      const double rr = hu[i].x - hw[i].x - hc[i].x, ri = hu[i].y - hw[i].y - hc[i].y;
      num += rr * rr + ri * ri;
      den += hc[i].x * hc[i].x + hc[i].y * hc[i].y;
    }
  }
  *resid_h = den > 0 ? std::sqrt(num / den) : 0.0;
  return GW_OK;
}

// Refinement of X = eps~^{-1} - 1 in FP64 after the working-precision solve.
// With chi~ = v^1/2 chi v^1/2 and eps~ = 1 - chi~, X = eps~^{-1} chi~ solves
// eps~ X = chi~.  For an approximate X with error E, the residual
//   R = chi~ - eps~ X = chi~ - X + chi~ X
// and the update X <- X + (1 + X) R (the current 1 + X standing in for
// eps~^{-1}) leave the error -E eps~ E: Newton-Schulz, quadratic convergence,
// two N^3 FP64 GEMMs per step.
template <typename T>
__global__ void refine_expand_kernel(const typename cpx<T>::t* __restrict__ Xl, const typename cpx<T>::t* __restrict__ chi,
                                     const double* __restrict__ vh, double2* __restrict__ X, double2* __restrict__ Ct,
                                     int n) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  const int a = blockIdx.y;
  if (b >= n) return;
  const long e = (long)a * n + b;
  const auto x = b <= a ? Xl[e] : Xl[(long)b * n + a];
  X[e] = b <= a ? make_double2(x.x, x.y) : make_double2(x.x, -x.y);
  const auto c = chi[e];
  const double sc = vh[a] * vh[b];
  Ct[e] = make_double2(sc * c.x, sc * c.y);
}

__global__ void refine_resid_kernel(const double2* __restrict__ Ct, const double2* __restrict__ X, double2* R, long nn) {
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < nn; e += (long)gridDim.x * blockDim.x)
    R[e] = make_double2(Ct[e].x - X[e].x + R[e].x, Ct[e].y - X[e].y + R[e].y);
}

__global__ void refine_update_kernel(double2* X, const double2* __restrict__ R, const double2* __restrict__ XR, long nn) {
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < nn; e += (long)gridDim.x * blockDim.x)
    X[e] = make_double2(X[e].x + R[e].x + XR[e].x, X[e].y + R[e].y + XR[e].y);
}

// Lower triangle back in the working precision, Hermitian part of X.
template <typename T>
__global__ void refine_store_kernel(const double2* __restrict__ X, typename cpx<T>::t* __restrict__ Xl, int n) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  const int a = blockIdx.y;
  if (b > a || b >= n) return;
  const double2 u = X[(long)a * n + b], w = X[(long)b * n + a];
  Xl[(long)a * n + b] = mk(T(0.5 * (u.x + w.x)), T(0.5 * (u.y - w.y)));
}

template <typename T>
static gw_status refine_one(gw_ctx* ctx, int n, const typename cpx<T>::t* chi, const double* dvh,
                            typename cpx<T>::t* xl, double2* ws, int iters, cudaStream_t st) {
  const long nn = (long)n * n;
  double2* X = ws;
  double2* Ct = ws + nn;
  double2* R = ws + 2 * nn;
  double2* XR = ws + 3 * nn;
  const dim3 tb(128), gb((n + 127) / 128, n);
  const int eb = (int)std::min<long>((nn + 255) / 256, (long)ctx->num_sms * 8);
  gw_status rc;
  refine_expand_kernel<T><<<gb, tb, 0, st>>>(xl, chi, dvh, X, Ct, n);
  if ((rc = launch_check(ctx, "refine_expand_kernel"))) return rc;
  for (int it = 0; it < iters; ++it) {
    GemmArgs g{};
    g.M = g.N = g.K = n;
    g.alpha_re = 1.0;
    g.lda = g.ldb = g.ldc = n;
    g.A = Ct;                 // R = chi~ X
    g.B = X;
    g.C = R;
    if ((rc = launch_gemm(ctx, GW_FP64, g, st))) return rc;
    refine_resid_kernel<<<eb, 256, 0, st>>>(Ct, X, R, nn);
    if ((rc = launch_check(ctx, "refine_resid_kernel"))) return rc;
    g.A = X;                  // XR = X R
    g.B = R;
    g.C = XR;
    if ((rc = launch_gemm(ctx, GW_FP64, g, st))) return rc;
    refine_update_kernel<<<eb, 256, 0, st>>>(X, R, XR, nn);
    if ((rc = launch_check(ctx, "refine_update_kernel"))) return rc;
  }
  refine_store_kernel<T><<<gb, tb, 0, st>>>(X, xl, n);
  return launch_check(ctx, "refine_store_kernel");
}

// The same refinement for the tensor-core precisions, with the product chi~ X
// of the residual on the tensor cores as exact fp16 slice products (slice pairs
// up to kRefineLevels, i.e. 30 bits of the row and column maxima: the residual
// then bounds X to ~1e-9, below the FP32 storage of W~), and the correction
// X R as three fp16 split products (R is small: the correction needs only the
// working precision).  Work: X, chi~, R in FP64 and R, X R in FP32 (the last
// slot of ws); X in FP32 goes to the upper part of xl, which the final store
// overwrites with the lower triangle.
constexpr int kRefineLevels = 4;

__global__ void to_f32_kernel(const double2* __restrict__ X, float2* __restrict__ Y, long nn) {
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < nn; e += (long)gridDim.x * blockDim.x)
    Y[e] = make_float2((float)X[e].x, (float)X[e].y);
}

__global__ void refine_update_f32_kernel(double2* X, const double2* __restrict__ R, const float2* __restrict__ XR,
                                         long nn) {
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < nn; e += (long)gridDim.x * blockDim.x)
    X[e] = make_double2(X[e].x + R[e].x + (double)XR[e].x, X[e].y + R[e].y + (double)XR[e].y);
}

static gw_status refine_one_tc(gw_ctx* ctx, gw_prec prec, int n, const float2* chi, const double* dvh, float2* xl,
                               double2* ws, void* tcs, void* sls, int iters, cudaStream_t st) {
  const long nn = (long)n * n;
  double2* X = ws;
  double2* Ct = ws + nn;
  double2* R = ws + 2 * nn;
  float2* R32 = reinterpret_cast<float2*>(ws + 3 * nn);
  float2* XR32 = R32 + nn;
  const dim3 tb(128), gb((n + 127) / 128, n);
  const int eb = (int)std::min<long>((nn + 255) / 256, (long)ctx->num_sms * 8);
  int* tstat = ctx->dflag + 4;
  gw_status rc;
  refine_expand_kernel<float><<<gb, tb, 0, st>>>(xl, chi, dvh, X, Ct, n);
  if ((rc = launch_check(ctx, "refine_expand_kernel"))) return rc;
  for (int it = 0; it < iters; ++it) {
    // R = chi~ X (FP64-class), then R = chi~ - X + R
    if ((rc = tc_zgemm_sliced(ctx, n, n, n, Ct, n, X, n, R, n, kRefineLevels, tstat, sls, st))) return rc;
    refine_resid_kernel<<<eb, 256, 0, st>>>(Ct, X, R, nn);
    if ((rc = launch_check(ctx, "refine_resid_kernel"))) return rc;
    to_f32_kernel<<<eb, 256, 0, st>>>(X, xl, nn);
    to_f32_kernel<<<eb, 256, 0, st>>>(R, R32, nn);
    if ((rc = launch_check(ctx, "to_f32_kernel"))) return rc;
    ctx->launches++;
    TcGemm g;
    g.M = g.N = g.K = n;
    g.A = xl;
    g.lda = n;
    g.a_trans = g.a_conj = false;
    g.B = R32;
    g.ldb = n;
    g.b_trans = g.b_conj = false;
    g.C = XR32;
    g.ldc = n;
    g.alpha = 1.0f;
    g.accumulate = false;
    g.tri = 0;
    g.status = tstat;
    if ((rc = tc_gemm(ctx, prec, g, tcs, st))) return rc;
    refine_update_f32_kernel<<<eb, 256, 0, st>>>(X, R, XR32, nn);
    if ((rc = launch_check(ctx, "refine_update_f32_kernel"))) return rc;
  }
  refine_store_kernel<float><<<gb, tb, 0, st>>>(X, xl, n);
  return launch_check(ctx, "refine_store_kernel");
}

// One batch of frequencies: chi[B][n][n] -> W[B][n][n] (may alias chi), with
// work buffers E and P of the same shape.  tcs: tensor-core scratch (NULL for
// the CUDA-core precisions).
template <typename T>
static gw_status screen_batch(gw_ctx* ctx, gw_prec prec, int n, int B, const void* chi, const double* dvh, void* E,
                              void* Pm, void* W, double2* probe, double* resid_h, void* tcs, int refine,
                              double2* rws, void* sls, cudaStream_t st) {
  using C = typename cpx<T>::t;
  gw_status rc;
  C* e = static_cast<C*>(E);
  C* p = static_cast<C*>(Pm);
  const long nn = (long)n * n;
  const Batch bt{B, nn};
  if ((rc = set_attrs<T>(ctx))) return rc;
  build_eps_kernel<T><<<dim3(n, B), 256, 0, st>>>(static_cast<const C*>(chi), nn, dvh, e, nn, n);
  if ((rc = launch_check(ctx, "build_eps_kernel"))) return rc;
  if (!tcs) {
    // CUDA cores, 64-column panels over the whole matrix
    if ((rc = chol_simt<T>(ctx, prec, e, n, p, n, n, 0, bt, st))) return rc;
    if ((rc = inv_simt<T>(ctx, prec, e, n, p, n, n, bt, st))) return rc;
    GemmArgs g{};
    g.M = n;
    g.N = n;
    g.K = n;
    g.alpha_re = 1;
    g.beta = 0;
    g.A = p;
    g.lda = n;
    g.a_km = 1;
    g.a_conj = true;
    g.B = p;
    g.ldb = n;
    g.C = e;
    g.ldc = n;
    g.tri = 2;
    g.batch = B;
    g.sA = g.sB = g.sC = nn;
    if ((rc = launch_gemm(ctx, prec, g, st))) return rc;
  } else {
    if constexpr (std::is_same<T, float>::value) {
      int* tstat = ctx->dflag + 4;
      auto gemm = [&](int M, int N, int K, const C* A, bool at, bool ac, const C* Bm, bool btr, bool bc, C* Cm,
                      float alpha, bool acc, int tri, int batch) {
        TcGemm g;
        g.M = M;
        g.N = N;
        g.K = K;
        g.A = A;
        g.lda = n;
        g.a_trans = at;
        g.a_conj = ac;
        g.B = Bm;
        g.ldb = n;
        g.b_trans = btr;
        g.b_conj = bc;
        g.C = Cm;
        g.ldc = n;
        g.alpha = alpha;
        g.accumulate = acc;
        g.tri = tri;
        g.status = tstat;
        g.batch = batch;
        g.sA = g.sB = g.sC = nn;
        return tc_gemm(ctx, prec, g, tcs, st);
      };
      // 1. Cholesky and the inverted diagonal blocks P_kk
      for (int k0 = 0; k0 < n; k0 += kTB) {
        const int kb = std::min(kTB, n - k0);
        C* akk = e + (long)k0 * n + k0;
        C* pkk = p + (long)k0 * n + k0;
        if ((rc = chol_simt<float>(ctx, GW_FP32, akk, n, pkk, n, kb, k0, bt, st))) return rc;
        if ((rc = inv_simt<float>(ctx, GW_FP32, akk, n, pkk, n, kb, bt, st))) return rc;
        const int rows = n - k0 - kb;
        if (rows <= 0) break;
        C* a21 = e + (long)(k0 + kb) * n + k0;
        // L21 = A21 + A21 P_kk^H   (opB(k, j) = conj(P_kk[j][k]))
        if ((rc = gemm(rows, kb, kb, a21, false, false, pkk, true, true, a21, 1.0f, true, 0, B))) return rc;
        // A22 -= L21 L21^H
        if ((rc = gemm(rows, rows, kb, a21, false, false, a21, true, true, a21 + kb, -1.0f, true, 1, B))) return rc;
      }
      // 2. off-diagonal blocks of P = L^{-1} - 1, block row by block row, and
      //    the zero upper part
      for (int k0 = 0; k0 < n; k0 += kTB) {
        const int kb = std::min(kTB, n - k0);
        C* pi = p + (long)k0 * n;
        C* pkk = pi + k0;
        if (k0 > 0 && (rc = gemm(kb, k0, kb, pkk, false, false, pi, false, false, pi, 1.0f, true, 0, B))) return rc;
        const int rows = n - k0 - kb;
        if (rows <= 0) break;
        zero_block_kernel<float><<<dim3((rows + 127) / 128, kb, B), 128, 0, st>>>(pi + k0 + kb, n, nn, rows);
        if ((rc = launch_check(ctx, "zero_block_kernel"))) return rc;
        neg_copy_kernel<float><<<dim3(rows, 1, B), 256, 0, st>>>(e, n, nn, p, n, nn, k0 + kb, rows, k0, kb);
        if ((rc = launch_check(ctx, "neg_copy_kernel"))) return rc;
        if ((rc = gemm(rows, k0 + kb, kb, e + (long)(k0 + kb) * n + k0, false, false, pi, false, false,
                       p + (long)(k0 + kb) * n, -1.0f, true, 0, B)))
          return rc;
      }
      // 3. P^H P (lower) in K blocks of kTB rows of P.  P is lower triangular,
      //    so block [k1, k2) touches only the leading k2 x k2 part; going from
      //    the last block (which writes the whole lower triangle) to the first,
      //    each block is added to C by the epilogue in round-to-nearest FP32.
      //    One accumulation over all N rows would take ~3N/8 truncating
      //    tensor-core adds per element (5000 at N = 13824) and lose ~1e-4.
      for (int k1 = (n - 1) / kTB * kTB; k1 >= 0; k1 -= kTB) {
        const int k2 = std::min(n, k1 + kTB);
        if ((rc = gemm(k2, k2, k2 - k1, p + (long)k1 * n, true, true, p + (long)k1 * n, false, false, e, 1.0f,
                       k2 < n, 1, B)))
          return rc;
      }
    }
  }
  assemble_kernel<T><<<dim3(n, B), 256, 0, st>>>(e, nn, p, nn, n);
  if ((rc = launch_check(ctx, "assemble_kernel"))) return rc;
  if (refine > 0)
    for (int b = 0; b < B; ++b) {
      if constexpr (std::is_same<T, float>::value) {
        if (tcs) {
          if ((rc = refine_one_tc(ctx, prec, n, static_cast<const C*>(chi) + b * nn, dvh, e + b * nn, rws, tcs, sls,
                                  refine, st)))
            return rc;
          continue;
        }
      }
      if ((rc = refine_one<T>(ctx, n, static_cast<const C*>(chi) + b * nn, dvh, e + b * nn, rws, refine, st)))
        return rc;
    }
  if (resid_h)
    for (int b = 0; b < B; ++b)
      if ((rc = residual_probe<T>(ctx, n, static_cast<const C*>(chi) + b * nn, dvh, e + b * nn, probe, resid_h + b,
                                  st)))
        return rc;
  const int nt = (n + 31) / 32;
  finalize_kernel<T><<<dim3(nt, nt, B), dim3(32, 8), 0, st>>>(e, nn, dvh, static_cast<C*>(W), nn, n);
  return launch_check(ctx, "finalize_kernel");
}

// Tensor-core GEMM scratch of the screening: panels of kTB over a batch, and
// with refinement the full n x n x n correction product.
static size_t screen_tc_scratch(int n_chi, int bsz, bool refine) {
  const size_t a = tc_gemm_scratch(n_chi, n_chi, kTB, bsz);
  return refine ? std::max(a, tc_gemm_scratch(n_chi, n_chi, n_chi, 1)) : a;
}

// Frequencies per batch (the two work matrices of a batch within 64 GB) and
// the scratch gw_screen_W needs.
size_t screen_scratch(int n_chi, int n_omega, gw_prec prec, int* bsz_out, int* nbatch_out, bool refine) {
  const size_t es = csize(prec);
  const size_t nn = (size_t)n_chi * n_chi;
  const bool tc = prec == GW_F16X3 || prec == GW_BF16X3;
  const size_t budget = size_t(64) << 30;
  const int no = std::max(n_omega, 1);
  const int bmax = (int)std::max<size_t>(1, std::min<size_t>(no, budget / (2 * nn * es)));
  const int nbatch = (no + bmax - 1) / bmax;
  const int bsz = (no + nbatch - 1) / nbatch;
  Carver probe(nullptr);
  probe.take<double>(n_chi);
  probe.take<char>(bsz * nn * es);
  probe.take<char>(bsz * nn * es);
  probe.take<double2>(4 * (size_t)n_chi);
  if (tc) probe.take<char>(screen_tc_scratch(n_chi, bsz, refine));
  if (refine) probe.take<double2>(4 * nn);
  if (refine && tc) probe.take<char>(tc_zgemm_sliced_scratch(n_chi, n_chi, n_chi, kRefineLevels));
  if (bsz_out) *bsz_out = bsz;
  if (nbatch_out) *nbatch_out = nbatch;
  return probe.off;
}

// The screening of n_omega frequencies with v^1/2 already on the device (dvh)
// and the arena carved by cv after it: device-side memsets and kernels only
// when resid_h and first_bad are NULL (then a plan can capture it in a CUDA
// graph).  Pivot and time-out flags are left in ctx->dflag (zeroed here first).
// resid_h: the FP64 probe residuals (synchronous); first_bad: with several
// batches of frequencies, the first frequency whose factorisation failed
// (synchronises between batches).
gw_status screen_launch(gw_ctx* ctx, int n_chi, int n_omega, gw_prec prec, int refine_iters, const double* dvh,
                        const void* chi_w, void* w_w, Carver& cv, double* resid_h, int* first_bad, cudaStream_t s) {
  gw_status st;
  const size_t es = csize(prec);
  const size_t nn = (size_t)n_chi * n_chi;
  const bool tc = prec == GW_F16X3 || prec == GW_BF16X3;
  int bsz = 0, nbatch = 0;
  screen_scratch(n_chi, n_omega, prec, &bsz, &nbatch, refine_iters > 0);
  const size_t tcs_bytes = tc ? screen_tc_scratch(n_chi, bsz, refine_iters > 0) : 0;
  void* E = cv.take<char>(bsz * nn * es);
  void* M = cv.take<char>(bsz * nn * es);
  double2* pr = cv.take<double2>(4 * (size_t)n_chi);
  void* tcs = tc ? cv.take<char>(tcs_bytes) : nullptr;
  double2* rws = refine_iters > 0 ? cv.take<double2>(4 * nn) : nullptr;
  void* sls = refine_iters > 0 && tc ? cv.take<char>(tc_zgemm_sliced_scratch(n_chi, n_chi, n_chi, kRefineLevels))
                                     : nullptr;
  if ((st = cuda_check(ctx, cudaMemsetAsync(ctx->dflag, 0, 8 * sizeof(int), s), "memset flag"))) return st;
  for (int k0 = 0; k0 < n_omega; k0 += bsz) {
    const int B = std::min(bsz, n_omega - k0);
    const char* in = static_cast<const char*>(chi_w) + k0 * nn * es;
    char* out = static_cast<char*>(w_w) + k0 * nn * es;
    double* rk = resid_h ? resid_h + k0 : nullptr;
    if (is_fp64(prec))
      st = screen_batch<double>(ctx, prec, n_chi, B, in, dvh, E, M, out, pr, rk, nullptr, refine_iters, rws, nullptr, s);
    else st = screen_batch<float>(ctx, prec, n_chi, B, in, dvh, E, M, out, pr, rk, tcs, refine_iters, rws, sls, s);
    if (st) return st;
    if (first_bad && nbatch > 1 && *first_bad < 0) {
      int f[3] = {0, 0, 0};
      cudaMemcpyAsync(f, ctx->dflag, sizeof(f), cudaMemcpyDeviceToHost, s);
      if ((st = cuda_check(ctx, cudaStreamSynchronize(s), "sync"))) return st;
      if (f[0]) *first_bad = k0 + f[2];
    }
  }
  return GW_OK;
}

}  // namespace gw

using namespace gw;

extern "C" gw_status gw_workspace_size(const gw_grid* grid, int n_b, int n_occ, int n, int n_chi, int n_n,
                                       gw_prec prec, int r_block, size_t* chi0_bytes, size_t* screen_bytes,
                                       size_t* sigma_bytes) {
  GridInfo g;
  gw_status st = grid_info(nullptr, grid, &g);
  if (st) return st;
  if (!valid_prec(prec)) return fail(nullptr, GW_ERR_ARG, "bad precision");
  if (n_b < 2 || n_occ < 1 || n_occ >= n_b || n < 1 || n_chi < 1 || n_chi > g.nr || n_n < 1)
    return fail(nullptr, GW_ERR_SHAPE, "bad sizes");
  if (chi0_bytes) *chi0_bytes = chi0_omega_scratch(g, n_b, n_occ, n, n_chi, prec, r_block);
  if (screen_bytes) *screen_bytes = screen_scratch(n_chi, n, prec, nullptr, nullptr);
  if (sigma_bytes) *sigma_bytes = sigma_scratch(g, n_b, n_occ, n, n_chi, n_n, 64, prec);
  return GW_OK;
}

extern "C" gw_status gw_screen_W(gw_ctx* ctx, const gw_grid* grid, int n_chi, const int32_t* gvec_h, int n_omega,
                                 gw_prec prec, const void* chi_w, void* w_w, double* resid_h, void* stream) {
  return gw_screen_W_refine(ctx, grid, n_chi, gvec_h, n_omega, prec, 0, chi_w, w_w, resid_h, stream);
}

extern "C" gw_status gw_screen_W_refine(gw_ctx* ctx, const gw_grid* grid, int n_chi, const int32_t* gvec_h,
                                        int n_omega, gw_prec prec, int refine_iters, const void* chi_w, void* w_w,
                                        double* resid_h, void* stream) {
  if (!ctx) return fail(nullptr, GW_ERR_ARG, "ctx is NULL");
  GridInfo g;
  gw_status st = grid_info(ctx, grid, &g);
  if (st) return st;
  if (!valid_prec(prec)) return fail(ctx, GW_ERR_ARG, "bad precision");
  if (n_chi < 1 || n_chi > g.nr || n_chi > 65535) return fail(ctx, GW_ERR_SHAPE, "need 1 <= n_chi <= min(N_r, 65535)");
  if (n_omega < 0) return fail(ctx, GW_ERR_SHAPE, "n_omega < 0");
  if (n_omega == 0) return GW_OK;
  if (!gvec_h || !chi_w || !w_w) return fail(ctx, GW_ERR_ARG, "NULL pointer");
  if (refine_iters < 0 || refine_iters > 8) return fail(ctx, GW_ERR_ARG, "need 0 <= refine_iters <= 8");
  cudaStream_t s = as_stream(stream);
  std::vector<double> vh(n_chi);
  if ((st = gw_coulomb_sqrt(grid, gvec_h, n_chi, vh.data()))) return fail(ctx, st, gw_last_error(nullptr));
  if ((st = reserve(ctx, screen_scratch(n_chi, n_omega, prec, nullptr, nullptr, refine_iters > 0)))) return st;
  Carver cv(ctx->arena);
  double* dvh = cv.take<double>(n_chi);
  if ((st = upload(ctx, dvh, vh.data(), sizeof(double) * n_chi, s))) return st;
  int first_bad = -1;
  if ((st = screen_launch(ctx, n_chi, n_omega, prec, refine_iters, dvh, chi_w, w_w, cv, resid_h, &first_bad, s)))
    return st;
  int flag[8] = {0};
  if ((st = cuda_check(ctx, cudaMemcpyAsync(flag, ctx->dflag, sizeof(flag), cudaMemcpyDeviceToHost, s), "flag")))
    return st;
  if ((st = cuda_check(ctx, cudaStreamSynchronize(s), "sync"))) return st;
  if (flag[4]) return fail(ctx, GW_ERR_TIMEOUT, "tensor-core GEMM wait timed out (role " + std::to_string(flag[5]) + ")");
  if (flag[0])
    return fail(ctx, GW_ERR_NUMERIC, "eps~ not positive definite at column " + std::to_string(flag[1]) +
                                         " of frequency " + std::to_string(first_bad >= 0 ? first_bad : flag[2]));
  return GW_OK;
}
