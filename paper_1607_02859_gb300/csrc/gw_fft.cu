// Spatial transforms within the cell (Eqs. FFTX1, FFTX2, FFTW), the product of
// Eq. chi_rr of plane-wave Green's functions fused into the row transform, and the
// nonuniform time/frequency transforms (Eqs. CTX, CT_W, ST_FFT).
//
// Data stay in HBM as row-major complex matrices whose row index is a grid
// point r = (i1*n2+i2)*n3+i3 or a G-set index, and whose column index is a grid
// point R' or a G' of the set.
//  * row kernels: one CTA per row; the N_r-point row is staged in shared memory
//    (odd-padded pencil stride, so every pencil pass is bank-conflict free) and
//    transformed by three passes of fully unrolled register FFTs, over the pencils
//    that the G set and the used part of the row touch; a row too long for one CTA
//    takes a plane and a line kernel.
//  * column kernels: the transform runs over the row index for a chunk of
//    contiguous columns, so every HBM access is a coalesced row segment:
//    a "plane" kernel does the (i2,i3) 2-D FFT through shared memory and a
//    "line" kernel the i1 1-D FFT in registers.  The last i1 pass of the chi
//    chain also applies the cosine transform over all tau (Eq. CTX) before
//    anything is written, saving a full read+write of chi(G,G',tau).
#include <cooperative_groups.h>
#include <mutex>
#include <type_traits>

#include "gw_common.cuh"
#include "gw_kernels.h"
#include "gw_fft.cuh"

namespace gw {

bool grid_supported(int a, int b, int c) {
#define X(x, y, z) \
  if (a == x && b == y && c == z) return true;
  GW_GRIDS(X)
#undef X
  return false;
}

// What of the grid a G set touches, behind its inverse map on the device (set_lists):
// the (i2, i3) columns and (i1, i2) pencils that hold a point of the set, and the
// values of each axis that do.  A cutoff sphere of n_chi points touches far fewer
// than all: at 36^3 with n_chi = 8192, 489 of 1296 columns and 25 of 36 values.
template <int N1, int N2, int N3>
struct SetLists {
  int n23, n12, n1, n2, n3;
  const int *l23, *l12, *l1, *l2, *l3;
  __device__ __forceinline__ explicit SetLists(const int* __restrict__ inv) {
    const int* x = inv + N1 * N2 * N3;
    n23 = __ldg(x);
    n12 = __ldg(x + 1);
    n1 = __ldg(x + 2);
    n2 = __ldg(x + 3);
    n3 = __ldg(x + 4);
    l23 = x + kSetHead;
    l12 = l23 + N2 * N3;
    l1 = l12 + N1 * N2;
    l2 = l1 + N1;
    l3 = l2 + N2;
  }
};

// Bit i of the result: index i is in the list of n indices below 64 (whole warps call it).
__device__ __forceinline__ unsigned long long set_mask(const int* __restrict__ list, int n) {
  unsigned lo = 0, hi = 0;
  for (int e = threadIdx.x & 31; e < n; e += 32) {
    const int v = __ldg(list + e);
    if (v < 32) lo |= 1u << v;
    else hi |= 1u << (v - 32);
  }
  return (unsigned long long)__reduce_or_sync(~0u, hi) << 32 | __reduce_or_sync(~0u, lo);
}

// Rows of a Hermitian matrix x(r, R') of which only R' <= r is used: the row kernels
// take the grid index low of the launch's first row (-1: whole rows).
// Forward: elements past r are taken as zero without being read (the tensor-core
// chi pass does not write them).  Backward: the columns that the fused self-energy
// reads, i.e. up to the end of the 128-column tile that holds the diagonal of the
// row's 128-row tile; the rest of the row is not written.
__device__ __forceinline__ int low_last_fwd(int low, long row, int nr) {
  return low < 0 ? nr - 1 : low + (int)row;
}
__device__ __forceinline__ int low_last_bwd(int low, long row, int nr) {
  if (low < 0) return nr - 1;
  const int g0 = low + ((int)row & ~127);
  return min(nr - 1, (g0 + 127) / 128 * 128 + 127);
}

// Threads and CTAs per SM of the one-CTA rows (FP32): two or three CTAs on an SM, so
// that one row's loads overlap another's arithmetic.  Two rounds of pencils (N1 N2 per
// pass) for the middle grids; from 24^3, where two rows fill an SM's shared memory, as
// many threads as the registers of two CTAs allow, which hides more latency than even
// rounds: 4096 rows onto 4097 G vectors 222 -> 203 us, from them 203 -> 189, the
// triangle rows of 4 times 2.18 -> 1.90 ms.  At 20^3 and 16^3 512 threads are slower
// (triangle rows 0.91 -> 0.94, 0.24 -> 0.29 ms).  FP64 is bound by its ALU.
template <typename T, int N1, int N2, int N3>
struct RowCfg {
  static constexpr int PC = N1 * N2;
  static constexpr bool F32 = sizeof(T) == 4;
  static constexpr int NR = N1 * N2 * N3;
  static constexpr int TH = F32 ? (NR >= 13824 ? 512 : NR >= 4096 ? ((PC / 2 + 31) / 32 * 32 < 64 ? 64 : (PC / 2 + 31) / 32 * 32)
                                                           : ((PC + 31) / 32 * 32))
                                : (NR >= 4096 ? 512 : 256);
  static constexpr int MINB = F32 ? (NR >= 13824 ? 2 : (NR >= 4096 ? 3 : 4)) : 1;
};

// MODE 1: x = a, forward (+i), gather the G' set.  (Eq. FFTX1)
// MODE 2: scatter a[j] to fft positions, backward (-i), times scale.   (Eq. FFTW, 2nd step)
// VI / VO: the grid side / the G-set side (mode 1) moves as 16-byte pairs of
// elements (aligned rows of even length), four pairs in flight per thread.
// LOW: rows of a triangle (low >= 0); whole rows are compiled without its checks.
//
// The three passes over the row do only what the G set (lists) and the triangle
// (low) need: forward the planes i1 <= i1(r), of them the i3 of the set in the i2
// pass, and the set's (i2, i3) columns in the i1 pass; backward the set's (i1, i2)
// pencils, then its i1 planes, and of the i1 pass the planes up to the last one
// read.
// That is 0.44 of a whole row's pencils at 24^3 with n_chi = 4097; the rows of one
// tau went from 800 to 470 us there (scalar loads for the odd n_chi before), from
// 250 to 150 us at 20^3 with n_chi = 1536.  Bound by instruction issue.
template <typename T, int N1, int N2, int N3, int MODE, bool VI, bool VO, bool LOW>
__global__ void __launch_bounds__(RowCfg<T, N1, N2, N3>::TH, RowCfg<T, N1, N2, N3>::MINB)
    row_fft_kernel(const typename cpx<T>::t* __restrict__ a, long lda, typename cpx<T>::t* __restrict__ out, long ldo,
                   const int* __restrict__ map, const int* __restrict__ inv, int n_chi, T scale, int low) {
  using C = typename cpx<T>::t;
  using L = RowLayout<N1, N2, N3>;
  constexpr int THREADS = RowCfg<T, N1, N2, N3>::TH;
  constexpr int PL = N2 * N3;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* s = reinterpret_cast<C*>(smem_raw);
  const long row = blockIdx.x;
  const SetLists<N1, N2, N3> g(inv);
  if constexpr (MODE == 2) {
    const int i1m = LOW ? low_last_bwd(low, row, L::NR) / PL + 1 : N1;   // planes to deliver
    for (int e = threadIdx.x; e < L::TOT; e += THREADS) s[e] = mk(T(0), T(0));
    __syncthreads();
    const C* src = a + row * lda;
    for (int j0 = threadIdx.x; j0 < n_chi; j0 += 4 * THREADS) {
      C v[4];
      int m[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = j0 + u * THREADS;
        if (j < n_chi) {
          v[u] = src[j];
          m[u] = map[j];
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (j0 + u * THREADS < n_chi) s[L::pos(m[u])] = v[u];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < g.n12; e += THREADS) {
      const int o = __ldg(g.l12 + e) * L::S2;
      C x[N3];
#pragma unroll
      for (int k = 0; k < N3; ++k) x[k] = s[o + k];
      RegFFT<N3, -1>::run(x);
#pragma unroll
      for (int k = 0; k < N3; ++k) s[o + k] = x[k];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < g.n1 * N3; e += THREADS) {
      const int o = __ldg(g.l1 + e / N3) * L::S1 + e % N3;
      C x[N2];
#pragma unroll
      for (int k = 0; k < N2; ++k) x[k] = s[o + k * L::S2];
      RegFFT<N2, -1>::run(x);
#pragma unroll
      for (int k = 0; k < N2; ++k) s[o + k * L::S2] = x[k];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < PL; e += THREADS) {
      const int o = e / N3 * L::S2 + e % N3;
      C x[N1];
#pragma unroll
      for (int k = 0; k < N1; ++k) x[k] = s[o + k * L::S1];
      RegFFT<N1, -1>::run(x);
#pragma unroll
      for (int k = 0; k < N1; ++k)
        if (k < i1m) s[o + k * L::S1] = x[k];
    }
    __syncthreads();
    C* dst = out + row * ldo;
    if (VI) {
      for (int q = threadIdx.x; q < i1m * PL / 2; q += THREADS) {
        const int p = L::pos(2 * q);
        st_pair(dst + 2 * q, cscale(s[p], scale), cscale(s[p + 1], scale));
      }
    } else {
      for (int r = threadIdx.x; r < i1m * PL; r += THREADS) dst[r] = cscale(s[L::pos(r)], scale);
    }
    return;
  }
  const int last = LOW ? low_last_fwd(low, row, L::NR) : L::NR - 1;
  const int i1m = last / PL + 1;                                 // planes with an element R' <= r
  const C* pa = a + row * lda;
  if (VI) {
    const int np = i1m * PL / 2;
    for (int q0 = threadIdx.x; q0 < np; q0 += 4 * THREADS) {
      C v[4][2];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int q = q0 + u * THREADS;
        v[u][0] = v[u][1] = mk(T(0), T(0));
        if (q < np && 2 * q <= last) ld_pair(pa + 2 * q, v[u][0], v[u][1]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int q = q0 + u * THREADS;
        if (q >= np) continue;
        const int p = L::pos(2 * q);           // 2q and 2q+1 share an i3 pencil (N3 even)
        s[p] = v[u][0];
        s[p + 1] = 2 * q + 1 <= last ? v[u][1] : mk(T(0), T(0));
      }
    }
  } else {
    for (int r = threadIdx.x; r < i1m * PL; r += THREADS) s[L::pos(r)] = r <= last ? pa[r] : mk(T(0), T(0));
  }
  __syncthreads();
  for (int e = threadIdx.x; e < i1m * N2; e += THREADS) {
    const int o = e * L::S2;
    C x[N3];
#pragma unroll
    for (int k = 0; k < N3; ++k) x[k] = s[o + k];
    RegFFT<N3, +1>::run(x);
#pragma unroll
    for (int k = 0; k < N3; ++k) s[o + k] = x[k];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < i1m * g.n3; e += THREADS) {
    const int i1 = e / g.n3;
    const int o = i1 * L::S1 + __ldg(g.l3 + (e - i1 * g.n3));
    C x[N2];
#pragma unroll
    for (int k = 0; k < N2; ++k) x[k] = s[o + k * L::S2];
    RegFFT<N2, +1>::run(x);
#pragma unroll
    for (int k = 0; k < N2; ++k) s[o + k * L::S2] = x[k];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < g.n23; e += THREADS) {
    const int c = __ldg(g.l23 + e);
    const int o = c / N3 * L::S2 + c % N3;
    C x[N1];
#pragma unroll
    for (int k = 0; k < N1; ++k) x[k] = k < i1m ? s[o + k * L::S1] : mk(T(0), T(0));
    RegFFT<N1, +1>::run(x);
#pragma unroll
    for (int k = 0; k < N1; ++k) s[o + k * L::S1] = x[k];
  }
  __syncthreads();
  C* dst = out + row * ldo;
  if (VO) {
    for (int q = threadIdx.x; q < n_chi / 2; q += THREADS)
      st_pair(dst + 2 * q, s[L::pos(map[2 * q])], s[L::pos(map[2 * q + 1])]);
  } else {
    for (int j = threadIdx.x; j < n_chi; j += THREADS) dst[j] = s[L::pos(map[j])];
  }
}

// Rows too long for one CTA's shared memory (36^3 = 46656 points, 373 KB) take two
// kernels, and what passes between them is only the (i2, i3) columns that the G
// set touches (n23 of N2 N3: 489 of 1296 for 8192 G vectors at 36^3):
//   plane kernel: the (i2, i3) transforms of a few planes of one row per CTA;
//   line kernel: the i1 transforms of the set's columns of one row per CTA, with
//   the G-set side of the row in shared memory where it fits.
// Column e of the set's list of plane i1 of a row lies at
// row * t_row + i1 * t_plane + e of the workspace, which may be the grid-side
// rows themselves (t_plane = N2 N3: a plane's columns lie at the start of the
// plane).  Both kernels keep many small CTAs on an SM.  A thread-block cluster
// holding the whole row in distributed shared memory (one pass over HBM, but 76
// rows in flight, three cluster barriers and scattered remote accesses) took
// 204 ns a row of the triangle at 36^3 with n_chi = 8192, these take 118 ns
// either way; with all pencils of whole rows it was 340 ns.  With the plane filled
// into (or read from) shared memory around the i2 pass, and 128 threads per line
// CTA (12 warps per SM in flight), it was 152 ns forward and 128 ns backward.
template <typename T, int N1, int N2, int N3>
struct PlaneCfg {
  using C = typename cpx<T>::t;
  static constexpr int S2 = N3 % 2 == 0 ? N3 + 1 : N3;
  static constexpr int S1 = N2 * S2;
  static constexpr int PL = N2 * N3;
  // planes per CTA: four of 36 x 36 are 43 KB, so that MINB CTAs fit an SM; of 48 x 48, 75 KB, only two
  static constexpr int PP = N2 >= 40 ? 2 : 4;
  static constexpr int TH = (PP * N2 + 31) / 32 * 32;              // one pencil per thread and pass
  static constexpr int MINB = sizeof(T) == 4 ? (N2 >= 30 ? 4 : 6) : 2;   // a 36-point pencil takes 72 of 100 registers
  static constexpr size_t bytes = (size_t)PP * S1 * sizeof(C);
  // threads and CTAs per SM of the line kernels (forward, backward)
  static constexpr int LF = sizeof(T) == 4 ? 160 : 128, LFB = sizeof(T) == 4 ? 3 : 2;
  static constexpr int LB = sizeof(T) == 4 ? 256 : 128, LBB = 2;
  // the longest G-set row that the line kernels stage in shared memory (two CTAs per SM)
  static constexpr size_t kStage = 110 * 1024;
  // Beyond it the forward kernel scatters single values into the row in global memory, and L2 has to
  // join the 8-byte ones of FP32 to sectors before they leave: one CTA per SM (kAlone bytes of shared
  // memory keep a second one out), so that the rows in flight, 152 of 373 KB at 36^3, stay there.  1024
  // rows at 36^3 with three CTAs per SM and with one: 20000 G vectors 458 and 351 us, all 46656 1059 and
  // 680; FP64 keeps its two (512 rows, 7041 G vectors: 1700 us, 1747 with one).
  static constexpr int LFU = sizeof(T) == 4 ? 3 * LF : LF, LFUB = sizeof(T) == 4 ? 1 : LFB;
  static constexpr size_t kAlone = sizeof(T) == 4 ? 120 * 1024 : 0;
};

// One i3 pencil of a plane in shared memory, transformed in place; the elements of mask are written.
template <int N, int DIR, typename C>
__device__ __forceinline__ void plane_pencil(C* s, unsigned long long mask) {
  C x[N];
#pragma unroll
  for (int k = 0; k < N; ++k) x[k] = s[k];
  RegFFT<N, DIR>::run(x);
#pragma unroll
  for (int k = 0; k < N; ++k)
    if (mask >> k & 1) s[k] = x[k];
}

// The set's columns of up to PP planes of each of ROWS rows into the zeroed pencils of its i2, and out again.
template <int N2, int N3, int PP, int ROWS, typename G, typename C, typename F>
__device__ __forceinline__ void plane_scatter(const G& g, C* s, int s1, int s2, int np, F load) {
  const int n = np * g.n2;
  for (int t = threadIdx.x; t < ROWS * n; t += blockDim.x) {
    const int r = t / n, e = t - r * n, p = e / g.n2;
    C* z = s + (r * PP + p) * s1 + __ldg(g.l2 + (e - p * g.n2)) * s2;
#pragma unroll
    for (int k = 0; k < N3; ++k) z[k] = C{};
  }
  __syncthreads();
  for (int e = threadIdx.x; e < g.n23; e += blockDim.x) {
    const int q = __ldg(g.l23 + e);
    const int o = q / N3 * s2 + q % N3;
    C v[ROWS][PP];
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
      for (int p = 0; p < PP; ++p)
        if (p < np) v[r][p] = load(r, p, e);
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
      for (int p = 0; p < PP; ++p)
        if (p < np) s[(r * PP + p) * s1 + o] = v[r][p];
  }
  __syncthreads();
}
template <int N2, int N3, int PP, typename G, typename C, typename F>
__device__ __forceinline__ void plane_gather(const G& g, const C* s, int s1, int s2, int np, F store) {
  for (int e = threadIdx.x; e < g.n23; e += blockDim.x) {
    const int q = __ldg(g.l23 + e);
    const int o = q / N3 * s2 + q % N3;
#pragma unroll
    for (int p = 0; p < PP; ++p)
      if (p < np) store(p, e, s[p * s1 + o]);
  }
}

// MODE 1 as for row_fft_kernel: planes of a, (+i) over i2 and the set's i2 of i3,
// the set's columns to t.  MODE 2: the columns from t,
// (-i) over the set's i2 of i3 and i2, times scale, to the planes of out.
// The i2 pass meets global memory in registers (a warp's elements of one i2 lie
// side by side there), and shared memory holds the set's i2 only.
template <typename T, int N1, int N2, int N3, int MODE>
__global__ void __launch_bounds__(PlaneCfg<T, N1, N2, N3>::TH, PlaneCfg<T, N1, N2, N3>::MINB)
    row_plane_kernel(const typename cpx<T>::t* a, long lda, typename cpx<T>::t* t, long t_row, long t_plane,
                     typename cpx<T>::t* out, long ldo, const int* __restrict__ inv, T scale, int low) {
  using C = typename cpx<T>::t;
  using R = PlaneCfg<T, N1, N2, N3>;
  constexpr int PL = R::PL, S1 = R::S1, S2 = R::S2, TH = R::TH;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* s = reinterpret_cast<C*>(smem_raw);                           // [PP][N2][S2]
  const long row = blockIdx.y;
  const int p0 = blockIdx.x * R::PP;
  const int last = MODE == 2 ? low_last_bwd(low, row, N1 * PL) : low_last_fwd(low, row, N1 * PL);
  const int np = min(R::PP, last / PL + 1 - p0);                   // planes of this CTA in use
  if (np <= 0) return;
  const SetLists<N1, N2, N3> g(inv);
  const unsigned long long m2 = set_mask(g.l2, g.n2);
  C* tp = t + row * t_row + (long)p0 * t_plane;
  if constexpr (MODE == 2) {
    plane_scatter<N2, N3, R::PP, 1>(g, s, S1, S2, np, [&](int, int p, int e) { return tp[p * t_plane + e]; });
    for (int e = threadIdx.x; e < np * g.n2; e += TH)              // pencils outside the set's i2 are zero
      plane_pencil<N3, -1>(s + e / g.n2 * S1 + __ldg(g.l2 + e % g.n2) * S2, ~0ull);
    __syncthreads();
    C* dst = out + row * ldo + (long)p0 * PL;
    for (int e = threadIdx.x; e < np * N3; e += TH) {
      const int p = e / N3, i3 = e - p * N3;
      C x[N2];
#pragma unroll
      for (int k = 0; k < N2; ++k) {
        x[k] = mk(T(0), T(0));
        if (m2 >> k & 1) x[k] = s[p * S1 + i3 + k * S2];
      }
      RegFFT<N2, -1>::run(x);
#pragma unroll
      for (int k = 0; k < N2; ++k) dst[p * PL + i3 + k * N3] = cscale(x[k], scale);
    }
    return;
  }
  const int last0 = last - p0 * PL;                                // the last element in use, from the CTA's first
  const C* pa = a + row * lda + (long)p0 * PL;
  for (int e = threadIdx.x; e < np * N3; e += TH) {
    const int p = e / N3, i3 = e - p * N3, r0 = p * PL + i3;
    C x[N2];
#pragma unroll
    for (int k = 0; k < N2; ++k) {
      x[k] = mk(T(0), T(0));
      if (r0 + k * N3 <= last0) x[k] = pa[r0 + k * N3];
    }
    RegFFT<N2, +1>::run(x);
#pragma unroll
    for (int k = 0; k < N2; ++k)
      if (m2 >> k & 1) s[p * S1 + i3 + k * S2] = x[k];
  }
  __syncthreads();
  const unsigned long long m3 = set_mask(g.l3, g.n3);
  for (int e = threadIdx.x; e < np * g.n2; e += TH)
    plane_pencil<N3, +1>(s + e / g.n2 * S1 + __ldg(g.l2 + e % g.n2) * S2, m3);
  __syncthreads();
  plane_gather<N2, N3, R::PP>(g, s, S1, S2, np, [&](int p, int e, C v) { tp[p * t_plane + e] = v; });
}

// Forward line pass of one row per CTA: i1 transforms (+i) of the set's columns,
// the results to out[row][inv], in order through shared memory where STAGE.
template <typename T, int N1, int N2, int N3, bool STAGE>
__global__ void __launch_bounds__(STAGE ? PlaneCfg<T, N1, N2, N3>::LF : PlaneCfg<T, N1, N2, N3>::LFU,
                                  STAGE ? PlaneCfg<T, N1, N2, N3>::LFB : PlaneCfg<T, N1, N2, N3>::LFUB)
    row_line_fwd_kernel(const typename cpx<T>::t* t, long t_row, long t_plane, typename cpx<T>::t* __restrict__ out,
                        long ldo, const int* __restrict__ inv, int n_chi, int low) {
  using C = typename cpx<T>::t;
  constexpr int PL = N2 * N3, LT = STAGE ? PlaneCfg<T, N1, N2, N3>::LF : PlaneCfg<T, N1, N2, N3>::LFU;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* so = reinterpret_cast<C*>(smem_raw);                          // [n_chi]
  const long row = blockIdx.x;
  const int i1m = low_last_fwd(low, row, N1 * PL) / PL + 1;
  const SetLists<N1, N2, N3> g(inv);
  C* o = STAGE ? so : out + row * ldo;
  for (int e = threadIdx.x; e < g.n23; e += LT) {
    const int q = __ldg(g.l23 + e);
    C x[N1];
#pragma unroll
    for (int i1 = 0; i1 < N1; ++i1) x[i1] = i1 < i1m ? t[row * t_row + i1 * t_plane + e] : mk(T(0), T(0));
    RegFFT<N1, +1>::run(x);
#pragma unroll
    for (int i1 = 0; i1 < N1; ++i1) {
      const int j = __ldg(inv + i1 * PL + q);
      if (j >= 0) o[j] = x[i1];
    }
  }
  if (!STAGE) return;
  __syncthreads();
  for (int j = threadIdx.x; j < n_chi; j += LT) out[row * ldo + j] = so[j];
}

// Backward line pass: the row's n_chi values (through shared memory where STAGE)
// gathered through inv, i1 transforms (-i) of the set's columns, the planes in use to t.
template <typename T, int N1, int N2, int N3, bool STAGE>
__global__ void __launch_bounds__(PlaneCfg<T, N1, N2, N3>::LB, PlaneCfg<T, N1, N2, N3>::LBB)
    row_line_bwd_kernel(const typename cpx<T>::t* __restrict__ a, long lda, typename cpx<T>::t* __restrict__ t,
                        long t_row, long t_plane, const int* __restrict__ inv, int n_chi, int low, int fwd_rows) {
  using C = typename cpx<T>::t;
  constexpr int PL = N2 * N3, LT = PlaneCfg<T, N1, N2, N3>::LB;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* si = reinterpret_cast<C*>(smem_raw);                          // [n_chi]
  const long row = blockIdx.x;
  const int last = fwd_rows ? low_last_fwd(low, row, N1 * PL) : low_last_bwd(low, row, N1 * PL);
  const int i1m = last / PL + 1;
  const SetLists<N1, N2, N3> g(inv);
  const C* src = a + row * lda;
  if (STAGE) {
    for (int j = threadIdx.x; j < n_chi; j += LT) si[j] = src[j];
    __syncthreads();
    src = si;
  }
  for (int e = threadIdx.x; e < g.n23; e += LT) {
    const int q = __ldg(g.l23 + e);
    C x[N1];
#pragma unroll
    for (int i1 = 0; i1 < N1; ++i1) {
      const int j = __ldg(inv + i1 * PL + q);
      x[i1] = j >= 0 ? src[j] : mk(T(0), T(0));
    }
    RegFFT<N1, -1>::run(x);
#pragma unroll
    for (int i1 = 0; i1 < N1; ++i1)
      if (i1 < i1m) t[row * t_row + i1 * t_plane + e] = x[i1];
  }
}

// chi rows from the plane-wave form of G (the paper evaluates G in a plane-wave
// representation and transforms it to real space when needed, Sec. II.B; at one
// k point Eqs. FFT_G1, FFT_G2 are two ordinary transforms).  For each row r the
// rows a = T_unocc(r, .) and b = T_occ(r, .) over the orbitals' plane-wave set
// (the column-transformed plane-wave G, length n_pw) are expanded over the grid
// R' (backward transform), multiplied as
//   x(R') = scale a(R') conj(b(R'))            (Eq. chi_rr)
// and transformed forward onto the n_chi-long G set of chi (Eq. FFTX1): the
// backward line kernel for a and b, this kernel per plane (a few planes of both
// rows in shared memory: (i2, i3) backward, product, forward), and the forward
// line kernel.  Between them go only the columns that the sets touch, for a
// chunk of rows that stays in L2.  chi(r,R') is Hermitian: with low >= 0 only the
// planes i1 <= i1(r) are visited and the product is kept for R' <= r with half the
// diagonal; the caller adds the conjugate transpose in the end.  One tau at 36^3
// with 4224 plane waves and n_chi = 8192: 51.5 ms with a cluster of four CTAs per
// whole row, 34.7 ms with that cluster on the triangle, 15.2 ms as here (FFT
// instruction issue bounds it).
template <typename T, int N1, int N2, int N3>
struct PwPlane {
  using C = typename cpx<T>::t;
  using R = PlaneCfg<T, N1, N2, N3>;
  // two rows of as many planes as leave MINB CTAs of registers and shared memory on an SM; at 36^3, 2 tau,
  // three CTAs take 32.3 ms, one plane per CTA 35.6, as here 30.5
  static constexpr int PP = N2 >= 30 ? 2 : 4;
  static constexpr int TH = (2 * PP * (N2 > N3 ? N2 : N3) + 31) / 32 * 32;   // one pencil of the two rows per thread
  static constexpr int MINB = sizeof(T) == 4 ? (N2 >= 40 ? 2 : N2 >= 30 ? 4 : 3) : 1;
  static constexpr size_t bytes = 2 * (size_t)PP * R::S1 * sizeof(C);
};

template <typename T, int N1, int N2, int N3>
__global__ void __launch_bounds__(PwPlane<T, N1, N2, N3>::TH, PwPlane<T, N1, N2, N3>::MINB)
    row_pw_plane_kernel(const typename cpx<T>::t* __restrict__ ta, const typename cpx<T>::t* __restrict__ tb,
                        long ta_row, long ta_plane, typename cpx<T>::t* __restrict__ tx, long tx_row, long tx_plane,
                        const int* __restrict__ inv_pw, const int* __restrict__ inv_chi, T scale, int low) {
  using C = typename cpx<T>::t;
  using R = PlaneCfg<T, N1, N2, N3>;
  constexpr int PL = R::PL, S1 = R::S1, S2 = R::S2, PP = PwPlane<T, N1, N2, N3>::PP, TH = PwPlane<T, N1, N2, N3>::TH;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sa = reinterpret_cast<C*>(smem_raw);                          // [PP][N2][S2] a, then x
  C* sb = sa + PP * S1;                                            // [PP][N2][S2] b
  const long row = blockIdx.y;
  const int p0 = blockIdx.x * PP;
  const int last = low_last_fwd(low, row, N1 * PL);
  const int np = min(PP, last / PL + 1 - p0);
  if (np <= 0) return;
  const int last0 = last - p0 * PL;
  const SetLists<N1, N2, N3> gp(inv_pw), gx(inv_chi);
  {
    const C* pa = ta + row * ta_row + (long)p0 * ta_plane;
    const C* pb = tb + row * ta_row + (long)p0 * ta_plane;
    plane_scatter<N2, N3, PP, 2>(gp, sa, S1, S2, np,
                                 [&](int r, int p, int e) { return (r ? pb : pa)[p * ta_plane + e]; });
  }
  {                                                                // pencils outside the set's i2 are zero
    const int n = np * gp.n2;
    for (int t = threadIdx.x; t < 2 * n; t += TH) {
      const int e = t >= n ? t - n : t;
      plane_pencil<N3, -1>((t >= n ? sb : sa) + e / gp.n2 * S1 + __ldg(gp.l2 + e % gp.n2) * S2, ~0ull);
    }
  }
  __syncthreads();
  {
    // i2 of both rows, a column per thread; those of a stay in registers for the product of Eq. chi_rr and i2 of x
    const unsigned long long m2 = set_mask(gp.l2, gp.n2), mx = set_mask(gx.l2, gx.n2);
    const int n = np * N3, t = threadIdx.x;
    const int e = t >= n ? t - n : t, p = e / N3, i3 = e - p * N3, o = p * S1 + i3, r0 = p * PL + i3;
    C x[N2];
    if (t < 2 * n) {
      C* s = (t >= n ? sb : sa) + o;
#pragma unroll
      for (int k = 0; k < N2; ++k) {
        x[k] = mk(T(0), T(0));
        if (m2 >> k & 1) x[k] = s[k * S2];
      }
      RegFFT<N2, -1>::run(x);
      if (t >= n) {
#pragma unroll
        for (int k = 0; k < N2; ++k) s[k * S2] = x[k];
      }
    }
    __syncthreads();
    if (t < n) {
#pragma unroll
      for (int k = 0; k < N2; ++k) {
        const int r = r0 + k * N3;
        if (r <= last0) x[k] = cscale(cmulc(x[k], sb[o + k * S2]), low >= 0 && r == last0 ? scale * T(0.5) : scale);
        else x[k] = mk(T(0), T(0));
      }
      RegFFT<N2, +1>::run(x);
#pragma unroll
      for (int k = 0; k < N2; ++k)
        if (mx >> k & 1) sa[o + k * S2] = x[k];
    }
  }
  __syncthreads();
  const unsigned long long m3 = set_mask(gx.l3, gx.n3);
  for (int e = threadIdx.x; e < np * gx.n2; e += TH)
    plane_pencil<N3, +1>(sa + e / gx.n2 * S1 + __ldg(gx.l2 + e % gx.n2) * S2, m3);
  __syncthreads();
  C* px = tx + row * tx_row + (long)p0 * tx_plane;
  plane_gather<N2, N3, PP>(gx, sa, S1, S2, np, [&](int p, int e, C v) { px[p * tx_plane + e] = v; });
}

// Small grids: both rows of a grid point in one CTA's shared memory and the whole of
// the above in one launch, while two or three such CTAs share an SM (kPwOneMax: up to
// 16^3 in FP32, 12^3 in FP64).  The three kernels are bound by their launches and the
// columns' way through L2 there: 6 tau of 16^3 with 600 plane waves and 2000 G vectors
// took them 1.41 ms, this one 0.61 (a CTA per whole row 1.16); 12^3, 500 and 1728, FP32
// 0.47 and 0.17 (0.29), FP64 2.88 and 2.34 (3.68).  At 20^3, where two rows leave one
// CTA per SM, that whole-row form took 5.8 ms and the three kernels take 4.1.
template <typename T, int N1, int N2, int N3>
struct PwOne {
  using L = RowLayout<N1, N2, N3>;
  static constexpr size_t bytes = 2 * (size_t)L::TOT * sizeof(typename cpx<T>::t);
  static constexpr bool use = bytes <= kPwOneMax;
  static constexpr int PEN = N1 * (N2 > N3 ? N2 : N3);             // pencils of a pass over one row
  static constexpr int TH = PEN >= 256 ? 256 : (PEN + 31) / 32 * 32;
};

template <typename T, int N1, int N2, int N3>
__global__ void __launch_bounds__(PwOne<T, N1, N2, N3>::TH, 2)
    row_pw_one_kernel(const typename cpx<T>::t* __restrict__ ta, const typename cpx<T>::t* __restrict__ tb, long lda,
                      typename cpx<T>::t* __restrict__ out, long ldo, const int* __restrict__ inv_pw,
                      const int* __restrict__ inv_chi, int n_chi, T scale, int low) {
  using C = typename cpx<T>::t;
  using L = RowLayout<N1, N2, N3>;
  constexpr int PL = N2 * N3, S1 = L::S1, S2 = L::S2, TH = PwOne<T, N1, N2, N3>::TH;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sa = reinterpret_cast<C*>(smem_raw);                          // [N1][N2][S2] a, then x
  C* sb = sa + L::TOT;                                             // b, then the row of out
  const long row = blockIdx.x;
  const int last = low_last_fwd(low, row, N1 * PL), i1m = last / PL + 1;   // planes with an element R' <= r
  const SetLists<N1, N2, N3> gp(inv_pw), gx(inv_chi);
  auto pencils = [&](auto f) {                                     // the (i1, i2) pencils of both rows that hold plane waves
    const int n = i1m * gp.n2;
    for (int t = threadIdx.x; t < 2 * n; t += TH) {
      const int e = t >= n ? t - n : t;
      f((t >= n ? sb : sa) + e / gp.n2 * S1 + __ldg(gp.l2 + e % gp.n2) * S2);
    }
  };
  pencils([](C* s) {
#pragma unroll
    for (int k = 0; k < N3; ++k) s[k] = C{};
  });
  __syncthreads();
  for (int t = threadIdx.x; t < 2 * gp.n23; t += TH) {             // i1 (-i) of the set's columns
    const bool second = t >= gp.n23;
    const int q = __ldg(gp.l23 + (second ? t - gp.n23 : t));
    const C* src = (second ? tb : ta) + row * lda;
    C x[N1];
#pragma unroll
    for (int i1 = 0; i1 < N1; ++i1) {
      const int j = __ldg(inv_pw + i1 * PL + q);
      x[i1] = mk(T(0), T(0));
      if (j >= 0) x[i1] = __ldg(src + j);
    }
    RegFFT<N1, -1>::run(x);
    C* s = (second ? sb : sa) + q / N3 * S2 + q % N3;
#pragma unroll
    for (int i1 = 0; i1 < N1; ++i1)
      if (i1 < i1m) s[i1 * S1] = x[i1];
  }
  __syncthreads();
  pencils([](C* s) { plane_pencil<N3, -1>(s, ~0ull); });
  __syncthreads();
  {
    // i2 of both rows, the product of Eq. chi_rr and i2 of x, a column per thread
    const unsigned long long m2 = set_mask(gp.l2, gp.n2), mx = set_mask(gx.l2, gx.n2);
    for (int e = threadIdx.x; e < i1m * N3; e += TH) {
      const int i1 = e / N3, i3 = e - i1 * N3, o = i1 * S1 + i3, r0 = i1 * PL + i3;
      C x[N2], y[N2];
#pragma unroll
      for (int k = 0; k < N2; ++k) {
        x[k] = y[k] = mk(T(0), T(0));
        if (m2 >> k & 1) {
          x[k] = sa[o + k * S2];
          y[k] = sb[o + k * S2];
        }
      }
      RegFFT<N2, -1>::run(x);
      RegFFT<N2, -1>::run(y);
#pragma unroll
      for (int k = 0; k < N2; ++k) {
        const int r = r0 + k * N3;
        if (r <= last) x[k] = cscale(cmulc(x[k], y[k]), low >= 0 && r == last ? scale * T(0.5) : scale);
        else x[k] = mk(T(0), T(0));
      }
      RegFFT<N2, +1>::run(x);
#pragma unroll
      for (int k = 0; k < N2; ++k)
        if (mx >> k & 1) sa[o + k * S2] = x[k];
    }
  }
  __syncthreads();
  {
    const unsigned long long m3 = set_mask(gx.l3, gx.n3);
    for (int e = threadIdx.x; e < i1m * gx.n2; e += TH)
      plane_pencil<N3, +1>(sa + e / gx.n2 * S1 + __ldg(gx.l2 + e % gx.n2) * S2, m3);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < gx.n23; e += TH) {                 // i1 (+i) of chi's columns, in order through sb
    const int q = __ldg(gx.l23 + e), o = q / N3 * S2 + q % N3;
    C x[N1];
#pragma unroll
    for (int i1 = 0; i1 < N1; ++i1) x[i1] = i1 < i1m ? sa[o + i1 * S1] : mk(T(0), T(0));
    RegFFT<N1, +1>::run(x);
#pragma unroll
    for (int i1 = 0; i1 < N1; ++i1) {
      const int j = __ldg(inv_chi + i1 * PL + q);
      if (j >= 0) sb[j] = x[i1];
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < n_chi; j += TH) out[row * ldo + j] = sb[j];
}

// Rows too long for one CTA in the plane-wave self-energy: the CL CTAs of a
// cluster share a row's planes and columns through distributed shared memory.
template <typename T, int N1, int N2, int N3>
struct PwRow {
  using C = typename cpx<T>::t;
  static constexpr int S2 = N3 % 2 == 0 ? N3 + 1 : N3;
  static constexpr int PL = N2 * N3;
  static constexpr size_t plane_bytes(int cl) { return (size_t)(N1 / cl) * N2 * S2 * sizeof(C); }
  static constexpr int pick() {
    for (int cl : {1, 2, 3, 4, 6, 8})
      if (N1 % cl == 0 && PL % cl == 0 && 2 * plane_bytes(cl) <= 192 * 1024) return cl;
    return 0;
  }
  static constexpr int CL = pick();
  static constexpr int P = CL ? N1 / CL : 1;
  static constexpr int COLS = CL ? PL / CL : 1;
  static constexpr int WORK = P * N2 > COLS ? (P * N2 > P * N3 ? P * N2 : P * N3) : (COLS > P * N3 ? COLS : P * N3);
  static constexpr int THREADS = CL ? ((WORK + 31) / 32 * 32 > 1024 ? 1024 : (WORK + 31) / 32 * 32) : 32;
  static size_t slice_elems(int n_pw, int n_chi) {
    const size_t in = 2 * (size_t)((n_pw + CL - 1) / CL), out = (size_t)((n_chi + CL - 1) / CL);
    return in > out ? in : out;
  }
  // the sizes that the plane-wave route takes, chi and self-energy alike: two expanded rows and their
  // slices in a cluster's shared memory (chi's own row kernels use no cluster)
  static size_t smem(int n_pw, int n_chi) { return 2 * plane_bytes(CL) + slice_elems(n_pw, n_chi) * sizeof(C); }
  // row_pw_sigma_kernel: [T_occ | T_unocc | W~] slices in, hu and ho out over the last two
  static size_t sig_smem(int n_pw, int n_chi) {
    const size_t ps = (size_t)((n_pw + CL - 1) / CL), ws = (size_t)((n_chi + CL - 1) / CL);
    const size_t e = 2 * ps + ws > 3 * ps ? 2 * ps + ws : 3 * ps;
    return 2 * plane_bytes(CL) + e * sizeof(C);
  }
};

// The self-energy's rows in the same plane-wave form (first term of Eq.
// Sigma_occ_reduce with Eq. Sigma_rr): for each row r, the W~ row over chi's G
// set (wg, column-transformed, Eq. FFTW) and the rows T_unocc(r, .), T_occ(r, .)
// of the column-transformed plane-wave G are expanded over the grid R'; then
//   H(r,R') = W~(r,R') G(r,R') = W~ conj(G')            (G' the expanded T row)
// is transformed forward and gathered on the orbitals' plane waves,
//   hu / ho(r, g) = sum_R' H(r,R') e^{+i g.R'},
// so that sum_R' H(r,R') psi_n(R') = sum_g hu(r,g) c_n(g) needs only the
// plane-wave coefficients c_n of the Sigma bands.  Five transforms per row, W~
// kept expanded in the first plane buffer while the second takes G_unocc, then
// G_occ.  inv_neg: grid position -> index into the T rows (the negated set),
// inv_nat: grid position -> plane-wave index of the outputs, inv_chi: the G set.
template <typename T, int N1, int N2, int N3>
__global__ void __launch_bounds__(PwRow<T, N1, N2, N3>::THREADS)
    row_pw_sigma_kernel(const typename cpx<T>::t* __restrict__ tu, const typename cpx<T>::t* __restrict__ to,
                        long ldt, const typename cpx<T>::t* __restrict__ wg, long ldw,
                        typename cpx<T>::t* __restrict__ hu, typename cpx<T>::t* __restrict__ ho, long ldh,
                        const int* __restrict__ inv_neg, const int* __restrict__ inv_nat, int n_pw,
                        const int* __restrict__ inv_chi, int n_chi) {
  namespace cg = cooperative_groups;
  using C = typename cpx<T>::t;
  using R = PwRow<T, N1, N2, N3>;
  constexpr int P = R::P, PL = R::PL, S2 = R::S2, COLS = R::COLS, CL = R::CL;
  constexpr int TH = R::THREADS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* sa = reinterpret_cast<C*>(smem_raw);                              // W~ planes
  C* sb = reinterpret_cast<C*>(smem_raw + R::plane_bytes(CL));         // G', then H planes
  C* sl = reinterpret_cast<C*>(smem_raw + 2 * R::plane_bytes(CL));
  cg::cluster_group cluster = cg::this_cluster();
  const int c = (int)cluster.block_rank();
  const long row = blockIdx.y;
  const int n_ps = (n_pw + CL - 1) / CL, n_ws = (n_chi + CL - 1) / CL;
  // slices: [T_occ | T_unocc | W~]; outputs hu over T_unocc's, ho from 2 n_ps (both read by then)
  C* so_in = sl;
  C* su_in = sl + n_ps;
  C* sw = sl + 2 * n_ps;
  C* hu_s = sl + n_ps;
  C* ho_s = sl + 2 * n_ps;
  {
    const int j0 = c * n_ps, j1 = min(n_pw, j0 + n_ps);
    for (int j = j0 + threadIdx.x; j < j1; j += TH) {
      su_in[j - j0] = tu[row * ldt + j];
      so_in[j - j0] = to[row * ldt + j];
    }
    const int w0 = c * n_ws, w1 = min(n_chi, w0 + n_ws);
    for (int j = w0 + threadIdx.x; j < w1; j += TH) sw[j - w0] = wg[row * ldw + j];
  }
  cluster.sync();
  // backward i1 transforms of a slice-held row into every CTA's planes
  auto line_bwd = [&](const C* src, int ns, const int* inv, C* dst) {
    for (int q = c * COLS + threadIdx.x; q < (c + 1) * COLS; q += TH) {
      const int i2 = q / N3, i3 = q - i2 * N3;
      C x[N1];
      bool any = false;
#pragma unroll
      for (int i1 = 0; i1 < N1; ++i1) {
        const int j = __ldg(inv + i1 * PL + q);
        x[i1] = mk(T(0), T(0));
        if (j >= 0) {
          const int o = j / ns;
          x[i1] = cluster.map_shared_rank(src, o)[j - o * ns];
          any = true;
        }
      }
      if (__any_sync(__activemask(), any)) RegFFT<N1, -1>::run(x);   // empty columns stay zero
#pragma unroll
      for (int i1 = 0; i1 < N1; ++i1)
        cluster.map_shared_rank(dst, i1 / P)[((i1 % P) * N2 + i2) * S2 + i3] = x[i1];
    }
  };
  // forward i1 transforms of every CTA's H planes, gathered on the plane-wave set
  auto line_fwd = [&](C* out) {
    for (int q = c * COLS + threadIdx.x; q < (c + 1) * COLS; q += TH) {
      const int i2 = q / N3, i3 = q - i2 * N3;
      bool any = false;              // columns with no plane wave of the set deliver nothing
#pragma unroll
      for (int i1 = 0; i1 < N1; ++i1) any |= __ldg(inv_nat + i1 * PL + q) >= 0;
      if (!__any_sync(__activemask(), any)) continue;
      C x[N1];
#pragma unroll
      for (int i1 = 0; i1 < N1; ++i1) x[i1] = cluster.map_shared_rank(sb, i1 / P)[((i1 % P) * N2 + i2) * S2 + i3];
      RegFFT<N1, +1>::run(x);
#pragma unroll
      for (int i1 = 0; i1 < N1; ++i1) {
        const int j = __ldg(inv_nat + i1 * PL + q);
        if (j >= 0) {
          const int o = j / n_ps;
          cluster.map_shared_rank(out, o)[j - o * n_ps] = x[i1];
        }
      }
    }
  };
  auto planes_bwd = [&](C* buf) {
    pencil_pass<N3, -1>(buf, P * N2, 1, [](int q) { return q * S2; });
    __syncthreads();
    pencil_pass<N2, -1>(buf, P * N3, S2, [](int q) { return (q / N3) * (N2 * S2) + (q % N3); });
    __syncthreads();
  };
  // H = W~ conj(G') on the CTA's planes, then the forward (i2, i3) transforms
  auto product_fwd = [&]() {
    for (int e = threadIdx.x; e < P * PL; e += TH) {
      const int p = e / PL, rem = e - p * PL, i2 = rem / N3;
      const int ps = (p * N2 + i2) * S2 + (rem - i2 * N3);
      sb[ps] = cmulc(sa[ps], sb[ps]);
    }
    __syncthreads();
    pencil_pass<N2, +1>(sb, P * N3, S2, [](int q) { return (q / N3) * (N2 * S2) + (q % N3); });
    __syncthreads();
    pencil_pass<N3, +1>(sb, P * N2, 1, [](int q) { return q * S2; });
  };
  line_bwd(sw, n_ws, inv_chi, sa);
  line_bwd(su_in, n_ps, inv_neg, sb);
  cluster.sync();                  // W~ and G'_unocc planes complete; W~ and T_unocc slices free
  planes_bwd(sa);
  planes_bwd(sb);
  product_fwd();
  cluster.sync();                  // H_unocc planes final
  line_fwd(hu_s);
  cluster.sync();                  // hu complete; the second buffer free
  line_bwd(so_in, n_ps, inv_neg, sb);
  cluster.sync();
  planes_bwd(sb);
  product_fwd();
  cluster.sync();
  line_fwd(ho_s);
  cluster.sync();                  // no remote access after this point
  {
    const int j0 = c * n_ps, j1 = min(n_pw, j0 + n_ps);
    for (int j = j0 + threadIdx.x; j < j1; j += TH) {
      hu[row * ldh + j] = hu_s[j - j0];
      ho[row * ldh + j] = ho_s[j - j0];
    }
  }
}

// Columns per CTA of the plane pass: as many as leave two CTAs (FP32) in an SM's
// shared memory, at least 64 bytes of a row.
template <typename T, int N2, int N3>
constexpr int kPlaneW = N2 * N3 * 16 * sizeof(typename cpx<T>::t) <= 96 * 1024 ? 16 : 8;
template <typename T, int N2, int N3>
struct ColPlane {
  static constexpr int W = kPlaneW<T, N2, N3>;
  static constexpr size_t bytes = (size_t)N2 * N3 * W * sizeof(typename cpx<T>::t);
  static constexpr int PEN = (N2 > N3 ? N2 : N3) * W;              // pencils of a pass: one or two rounds
  static constexpr int TH = ((PEN > 288 ? PEN / 2 : PEN) + 31) / 32 * 32;
  static constexpr int MINB = sizeof(T) == 8 ? 1 : (bytes > 76 * 1024 ? 2 : 3);
};

// In-place 2-D FFT over (i2, i3) of the rows of plane i1 = blockIdx.y, for W
// contiguous columns per CTA.  PAIRS (FP32 only): rows move as 16-byte pairs
// of columns; the host takes it when ld and ncols are even (every pair then
// starts on a 16-byte boundary and lies wholly inside or outside the matrix).
// Towards the G set (DIR -1) only the (i2, i3) rows that the set touches are
// written (the i1 pass reads no others) and the i2 pass visits the set's i3;
// from it (DIR +1) only those rows are read (the others are zero) and the i3
// pass visits the set's i2.  The latency of its loads bounds it, with 18 warps on
// an SM (of 12.3 cycles between a warp's issues 5.1 wait for memory; shared-memory
// pipe 63%, DRAM 42%, issue 36%): one pass at 36^3, 8192 columns, takes 1.29 ms
// (3.3 TB/s); with all rows and one 16-column CTA per SM it took 2.28 ms.
template <typename T, int N1, int N2, int N3, int DIR, bool PAIRS>
__global__ void __launch_bounds__(ColPlane<T, N2, N3>::TH, ColPlane<T, N2, N3>::MINB)
    col_plane_kernel(typename cpx<T>::t* __restrict__ buf, long ld, int ncols, T scale, const int* __restrict__ inv) {
  using C = typename cpx<T>::t;
  constexpr int W = ColPlane<T, N2, N3>::W, TH = ColPlane<T, N2, N3>::TH;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* s = reinterpret_cast<C*>(smem_raw);
  const long i1 = blockIdx.y;
  const int c0 = blockIdx.x * W;
  C* base = buf + i1 * (N2 * N3) * ld + c0;
  const SetLists<N1, N2, N3> g(inv);
  if constexpr (DIR > 0) {
    for (int e = threadIdx.x; e < N2 * N3 * W; e += TH) s[e] = mk(T(0), T(0));
    __syncthreads();
  }
  const int n_in = DIR > 0 ? g.n23 : N2 * N3;
  auto row_in = [&](int e) { return DIR > 0 ? __ldg(g.l23 + e) : e; };
  if constexpr (PAIRS) {
    constexpr int LB = 6;                                          // loads in flight per thread
    for (int e0 = threadIdx.x; e0 < n_in * (W / 2); e0 += LB * TH) {
      C a[LB], b[LB];
      int at[LB];
#pragma unroll
      for (int u = 0; u < LB; ++u) {
        const int e = e0 + u * TH;
        a[u] = b[u] = mk(T(0), T(0));
        at[u] = -1;
        if (e < n_in * (W / 2)) {
          const int rr = row_in(e / (W / 2)), w = 2 * (e % (W / 2));
          at[u] = rr * W + w;
          if (c0 + w < ncols) ld_pair_rw(base + rr * ld + w, a[u], b[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < LB; ++u)
        if (at[u] >= 0) {
          s[at[u]] = a[u];
          s[at[u] + 1] = b[u];
        }
    }
  } else {
    for (int e = threadIdx.x; e < n_in * W; e += TH) {
      const int rr = row_in(e / W), w = e % W;
      s[rr * W + w] = (c0 + w < ncols) ? base[rr * ld + w] : mk(T(0), T(0));
    }
  }
  __syncthreads();
  const int n2 = DIR > 0 ? g.n2 : N2;
  for (int e = threadIdx.x; e < n2 * W; e += TH) {
    const int i2 = DIR > 0 ? __ldg(g.l2 + e / W) : e / W;
    const int o = i2 * (N3 * W) + e % W;
    C x[N3];
#pragma unroll
    for (int k = 0; k < N3; ++k) x[k] = s[o + k * W];
    RegFFT<N3, DIR>::run(x);
#pragma unroll
    for (int k = 0; k < N3; ++k) s[o + k * W] = x[k];
  }
  __syncthreads();
  const int n3 = DIR > 0 ? N3 : g.n3;
  for (int e = threadIdx.x; e < n3 * W; e += TH) {
    const int i3 = DIR > 0 ? e / W : __ldg(g.l3 + e / W);
    const int o = i3 * W + e % W;
    C x[N2];
#pragma unroll
    for (int k = 0; k < N2; ++k) x[k] = s[o + k * (N3 * W)];
    RegFFT<N2, DIR>::run(x);
#pragma unroll
    for (int k = 0; k < N2; ++k) s[o + k * (N3 * W)] = x[k];
  }
  __syncthreads();
  const int n_out = DIR > 0 ? N2 * N3 : g.n23;
  auto row_out = [&](int e) { return DIR > 0 ? e : __ldg(g.l23 + e); };
  if constexpr (PAIRS) {
    for (int e = threadIdx.x; e < n_out * (W / 2); e += TH) {
      const int rr = row_out(e / (W / 2)), w = 2 * (e % (W / 2));
      if (c0 + w < ncols) st_pair(base + rr * ld + w, cscale(s[rr * W + w], scale), cscale(s[rr * W + w + 1], scale));
    }
  } else {
    for (int e = threadIdx.x; e < n_out * W; e += TH) {
      const int rr = row_out(e / W), w = e % W;
      if (c0 + w < ncols) base[rr * ld + w] = cscale(s[rr * W + w], scale);
    }
  }
}

// 1-D FFT over i1 for the column c and the blockIdx.y-th (i2,i3) that the G set
// touches (l23, behind the inverse map).
// GATHER_IN: read row inv[pos] of `in` (zero if -1) instead of row pos.
// SCATTER_OUT: write row inv[pos] of `out` (skip if -1) instead of row pos.
template <typename T, int N1, int DIR, bool GATHER_IN, bool SCATTER_OUT>
__global__ void __launch_bounds__(128) col_line_kernel(const typename cpx<T>::t* __restrict__ in, long ldi,
                                                       typename cpx<T>::t* __restrict__ out, long ldo, int ncols,
                                                       int plane, const int* __restrict__ inv,
                                                       const int* __restrict__ l23, T scale) {
  using C = typename cpx<T>::t;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  const int i23 = __ldg(l23 + blockIdx.y);
  if (c >= ncols) return;
  C x[N1];
#pragma unroll
  for (int i1 = 0; i1 < N1; ++i1) {
    const long pos = (long)i1 * plane + i23;
    if (GATHER_IN) {
      const int j = inv[pos];
      x[i1] = j >= 0 ? in[(long)j * ldi + c] : mk(T(0), T(0));
    } else {
      x[i1] = in[pos * ldi + c];
    }
  }
  RegFFT<N1, DIR>::run(x);
#pragma unroll
  for (int i1 = 0; i1 < N1; ++i1) {
    const long pos = (long)i1 * plane + i23;
    if (SCATTER_OUT) {
      const int j = inv[pos];
      if (j >= 0) out[(long)j * ldo + c] = cscale(x[i1], scale);
    } else {
      out[pos * ldo + c] = cscale(x[i1], scale);
    }
  }
}

// Weighted sums of the transforms in FP32.  The weights of the time/frequency
// transforms reach |c_kj| ~ 10^2 with both signs; rounded to FP32 they alone
// would perturb sum_j c_kj x_j by ~4e-7 relative.  The FP32 path keeps each
// weight as an unevaluated pair hi + lo (hi = fl32(c), lo = fl32(c - hi)) and
// accumulates c x as fma(hi, x, fma(lo, x, s)), which removes the weight
// rounding for one extra FMA per term; the remaining FP32 accumulation error
// is below the rounding already present in the x_j themselves.  FP64 keeps the
// plain sum.  The weight arrays hold hi[n_k][n_j] and, for FP32, lo[n_k][n_j]
// right after.
//
// Two FP32 values (re, im) per 64-bit register pair: one packed multiply-add
// does both (half the issue slots of scalar FMAs at the same lane rate).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
// Weights in shared memory as (hi, hi, lo, lo), rows padded with zeros to NTB: one
// 16-byte broadcast read per term feeds the multiply-adds of several elements.
template <int NTB>
__device__ __forceinline__ void load_weights(const float* __restrict__ M, int nk, int nj, float4* w) {
  for (int e = threadIdx.x; e < nk * NTB; e += blockDim.x) {
    const int k = e / NTB, j = e - k * NTB;
    const float hi = j < nj ? M[k * nj + j] : 0.f, lo = j < nj ? M[nk * nj + k * nj + j] : 0.f;
    w[e] = make_float4(hi, hi, lo, lo);
  }
}
// s += sum_j c_kj x_j for E elements, terms in ascending j
template <int NTB, int E>
__device__ __forceinline__ void weighted(const float4* w, const f32x2 (&x)[NTB][E], f32x2 (&acc)[E]) {
#pragma unroll
  for (int u = 0; u < E; ++u) acc[u] = 0ull;
#pragma unroll
  for (int j = 0; j < NTB; ++j) {
    const ulonglong2 c = *reinterpret_cast<const ulonglong2*>(w + j);
#pragma unroll
    for (int u = 0; u < E; ++u) acc[u] = fma2(c.x, x[j][u], fma2(c.y, x[j][u], acc[u]));
  }
}

// Last column pass of the chi chain: i1 FFT (-i) of every tau slab, then
// out[k][inv[pos]][c] = sum_j cw[k][j] * slab_j(pos, c)  (Eq. CTX with the
// dV^2/Omega of Eq. FFTX2 folded into cw).  FP64: 32 columns x 8 warps per CTA.
template <typename T, int N1>
__global__ void __launch_bounds__(256) col_line_ct_kernel(const typename cpx<T>::t* __restrict__ slabs,
                                                          long slab_stride, long ld, int ntau,
                                                          const T* __restrict__ cw, int nw,
                                                          typename cpx<T>::t* __restrict__ out, long out_slice,
                                                          long ldo, const int* __restrict__ inv,
                                                          const int* __restrict__ l23, int plane, int ncols) {
  using C = typename cpx<T>::t;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* s = reinterpret_cast<C*>(smem_raw);                       // [ntau][N1][32]
  T* w = reinterpret_cast<T*>(s + (size_t)ntau * N1 * 32);      // [nw][ntau]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = blockIdx.x * 32 + lane;
  const int i23 = __ldg(l23 + blockIdx.y);
  for (int e = threadIdx.x; e < nw * ntau; e += blockDim.x) w[e] = cw[e];
  for (int j = warp; j < ntau; j += 8) {
    C x[N1];
    const C* src = slabs + (long)j * slab_stride;
#pragma unroll
    for (int i1 = 0; i1 < N1; ++i1)
      x[i1] = c < ncols ? src[((long)i1 * plane + i23) * ld + c] : mk(T(0), T(0));
    RegFFT<N1, -1>::run(x);
#pragma unroll
    for (int i1 = 0; i1 < N1; ++i1) s[(j * N1 + i1) * 32 + lane] = x[i1];
  }
  __syncthreads();
  if (c >= ncols) return;
  for (int q = warp; q < nw * N1; q += 8) {
    const int k = q / N1, i1 = q - k * N1;
    const int row = inv[(long)i1 * plane + i23];
    if (row < 0) continue;
    C acc = mk(T(0), T(0));
    for (int j = 0; j < ntau; ++j) {
      const C v = s[(j * N1 + i1) * 32 + lane];
      acc.x += w[k * ntau + j] * v.x;
      acc.y += w[k * ntau + j] * v.y;
    }
    out[(long)k * out_slice + (long)row * ldo + c] = acc;
  }
}

// The same pass in FP32 for any count of tau points up to NTB: 32 M columns per
// CTA, M so that the (tau, 32 columns) pencils fill the eight warps.  Each lane
// then keeps the values of its column at two i1 that hold a G vector in registers
// and runs over the frequencies.  At 36^3 with n_chi = 8192 and 2 tau the form
// with one warp per tau of every (i2, i3) took 7.3 to 8 ms, this one 1.0 ms.
template <int N1, int NTB>
__global__ void __launch_bounds__(256, N1 <= 24 || NTB <= 16 ? 2 : 1) col_line_ct_reg_kernel(const float2* __restrict__ slabs, long slab_stride,
                                                              long ld, int ntau, int m, const float* __restrict__ cw,
                                                              float2* __restrict__ out, long out_slice, long ldo,
                                                              const int* __restrict__ inv,
                                                              const int* __restrict__ l23, int plane, int ncols) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int act[N1], act_row[N1], n_act;
  float4* w = reinterpret_cast<float4*>(smem_raw);             // [ntau][NTB]
  float2* s = reinterpret_cast<float2*>(w + ntau * NTB);       // [ntau][N1][32 m]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int cw_cols = 32 * m;
  const int c0 = blockIdx.x * cw_cols;
  const int i23 = __ldg(l23 + blockIdx.y);
  load_weights<NTB>(cw, ntau, ntau, w);
  if (threadIdx.x == 0) {
    int n = 0;
    for (int i1 = 0; i1 < N1; ++i1) {
      const int row = __ldg(inv + (long)i1 * plane + i23);
      if (row >= 0) {
        act[n] = i1;
        act_row[n++] = row;
      }
    }
    n_act = n;
  }
  for (int t = warp; t < ntau * m; t += 8) {
    const int j = t / m, cl = (t - j * m) * 32 + lane, c = c0 + cl;
    float2 x[N1];
    const float2* src = slabs + (long)j * slab_stride;
#pragma unroll
    for (int i1 = 0; i1 < N1; ++i1)
      x[i1] = c < ncols ? src[((long)i1 * plane + i23) * ld + c] : make_float2(0.f, 0.f);
    RegFFT<N1, -1>::run(x);
#pragma unroll
    for (int i1 = 0; i1 < N1; ++i1) s[(j * N1 + i1) * cw_cols + cl] = x[i1];
  }
  __syncthreads();
  const int pairs = (n_act + 1) / 2;
  for (int t = warp; t < pairs * m; t += 8) {
    const int a = t / m, cl = (t - a * m) * 32 + lane, c = c0 + cl;
    if (c >= ncols) continue;
    const bool two = 2 * a + 1 < n_act;
    const int ia = act[2 * a], ib = two ? act[2 * a + 1] : ia;
    const long oa = (long)act_row[2 * a] * ldo + c, ob = two ? (long)act_row[2 * a + 1] * ldo + c : 0;
    f32x2 x[NTB][2];
#pragma unroll
    for (int j = 0; j < NTB; ++j) {
      x[j][0] = j < ntau ? *reinterpret_cast<const f32x2*>(s + (j * N1 + ia) * cw_cols + cl) : 0ull;
      x[j][1] = j < ntau ? *reinterpret_cast<const f32x2*>(s + (j * N1 + ib) * cw_cols + cl) : 0ull;
    }
#pragma unroll 1
    for (int k = 0; k < ntau; ++k) {
      f32x2 acc[2];
      weighted<NTB, 2>(w + k * NTB, x, acc);
      out[(long)k * out_slice + oa] = unpack2(acc[0]);
      if (two) out[(long)k * out_slice + ob] = unpack2(acc[1]);
    }
  }
}

// out[k][e] = (i if ST) sum_j M[k][j] in[j][e] in FP32: each thread keeps E
// elements of all n <= NTB slices in registers and runs over the outputs.  E = 2
// (16-byte accesses) where the slices allow it.  HBM and the multiply-add pipe
// bound it about equally at 20 points (four packed FMAs per weight and pair): 20
// slices of 2048^2 in 287 us (4.7 TB/s), 762 us with the weights in constant
// memory, whose cache the 800 of them did not fit.
template <int NTB, bool ST, int E>
__global__ void __launch_bounds__(128) ct_reg_kernel(const float2* __restrict__ in, float2* __restrict__ out,
                                                     size_t elems, int n, const float* __restrict__ M) {
  __shared__ float4 w[32 * NTB];
  load_weights<NTB>(M, n, n, w);
  __syncthreads();
  const size_t count = elems / E;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
    f32x2 x[NTB][E];
#pragma unroll
    for (int j = 0; j < NTB; ++j) {
      if constexpr (E == 2) {
        ulonglong2 v = make_ulonglong2(0ull, 0ull);
        if (j < n) v = __ldg(reinterpret_cast<const ulonglong2*>(in + (size_t)j * elems) + e);
        x[j][0] = v.x;
        x[j][1] = v.y;
      } else {
        x[j][0] = j < n ? __ldg(reinterpret_cast<const f32x2*>(in + (size_t)j * elems) + e) : 0ull;
      }
    }
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
      f32x2 acc[E];
      weighted<NTB, E>(w + k * NTB, x, acc);
      float2 v[E];
#pragma unroll
      for (int u = 0; u < E; ++u) {
        v[u] = unpack2(acc[u]);
        if (ST) v[u] = make_float2(-v[u].y, v[u].x);
      }
      float2* o = out + (size_t)k * elems + E * e;
      if constexpr (E == 2) st_pair(o, v[0], v[1]);
      else o[0] = v[0];
    }
  }
}

// FP64: out[k][e] = (i if ST) sum_j M[k][j] in[j][e]
template <bool ST>
__global__ void __launch_bounds__(256) ct_kernel(const double2* __restrict__ in, double2* __restrict__ out,
                                                 size_t elems, int n, const double* __restrict__ M) {
  __shared__ double w[32 * 32];
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) w[e] = M[e];
  __syncthreads();
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < elems; e += (size_t)gridDim.x * blockDim.x) {
    double2 x[32];
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j < n) x[j] = in[(size_t)j * elems + e];
    for (int k = 0; k < n; ++k) {
      double re = 0, im = 0;
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (j < n) {
          re += w[k * n + j] * x[j].x;
          im += w[k * n + j] * x[j].y;
        }
      out[(size_t)k * elems + e] = ST ? make_double2(-im, re) : make_double2(re, im);
    }
  }
}

template <typename T>
__global__ void hadamard_kernel(const typename cpx<T>::t* __restrict__ a, const typename cpx<T>::t* __restrict__ b,
                                typename cpx<T>::t* out, size_t count, T scale) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x)
    out[e] = cscale(cmulc(a[e], b[e]), scale);
}

// ---------------------------------------------------------------------- launchers

template <typename K>
static gw_status set_smem(gw_ctx* ctx, K kernel, size_t bytes) {
  if (bytes > 227 * 1024) return fail(ctx, GW_ERR_UNSUPPORTED, "shared-memory tile too large for this grid/precision");
  if (bytes > 48 * 1024)
    return cuda_check(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes),
                      "cudaFuncSetAttribute");
  return GW_OK;
}

template <typename T, int N1, int N2, int N3>
struct GridOps {
  using C = typename cpx<T>::t;
  using PC = PlaneCfg<T, N1, N2, N3>;
  static gw_status line_fwd(gw_ctx* ctx, const void* t, long t_row, long t_plane, void* out, long ldo, const int* inv,
                            int n_chi, int n_rows, int low, double work, int fam, cudaStream_t st) {
    const size_t bytes = (size_t)n_chi * sizeof(C);
    auto go = [&](auto kernel, size_t sm, int threads) -> gw_status {
      gw_status r = set_smem(ctx, kernel, sm);
      if (r) return r;
      KTimer kt(ctx, fam, work, st);
      kernel<<<n_rows, threads, sm, st>>>((const C*)t, t_row, t_plane, (C*)out, ldo, inv, n_chi, low);
      return launch_check(ctx, "row_line_fwd_kernel");
    };
    return bytes <= PC::kStage ? go(row_line_fwd_kernel<T, N1, N2, N3, true>, bytes, PC::LF)
                               : go(row_line_fwd_kernel<T, N1, N2, N3, false>, PC::kAlone, PC::LFU);
  }
  static gw_status line_bwd(gw_ctx* ctx, const void* a, long lda, void* t, long t_row, long t_plane, const int* inv,
                            int n_chi, int n_rows, int low, bool fwd_rows, double work, int fam, cudaStream_t st) {
    const size_t bytes = (size_t)n_chi * sizeof(C);
    auto go = [&](auto kernel, size_t sm) -> gw_status {
      gw_status r = set_smem(ctx, kernel, sm);
      if (r) return r;
      KTimer kt(ctx, fam, work, st);
      kernel<<<n_rows, PC::LB, sm, st>>>((const C*)a, lda, (C*)t, t_row, t_plane, inv, n_chi, low, fwd_rows ? 1 : 0);
      return launch_check(ctx, "row_line_bwd_kernel");
    };
    return bytes <= PC::kStage ? go(row_line_bwd_kernel<T, N1, N2, N3, true>, bytes)
                               : go(row_line_bwd_kernel<T, N1, N2, N3, false>, 0);
  }
  // planes of the launch's longest row
  static int row_planes(int low, int n_rows, bool bwd) {
    if (low < 0) return N1;
    const int g0 = low + (n_rows - 1) / 128 * 128;
    const int last = bwd ? (g0 + 127) / 128 * 128 + 127 : low + n_rows - 1;
    return std::min(N1, last / PC::PL + 1);
  }
  static gw_status row_two_pass(gw_ctx* ctx, int mode, const void* a, long lda, void* out, long ldo,
                                const int* inv, void* tmp, int n_chi, int n_rows, double scale, cudaStream_t st,
                                int low, double work) {
    constexpr int NR = N1 * N2 * N3;
    if (mode != 2 && !tmp)
      return fail(ctx, GW_ERR_UNSUPPORTED, "this grid's rows need the two-pass transform (index map and workspace)");
    if (sizeof(T) == 8 && (size_t)n_chi * sizeof(C) > 200 * 1024)
      return fail(ctx, GW_ERR_UNSUPPORTED, "G set too large for the two-pass row transform");
    constexpr int kMost = 32768;                                   // rows are the grid's y: whole 128-row tiles at a time
    for (int r = 0; n_rows > kMost && r < n_rows; r += kMost) {
      const int rows = std::min(kMost, n_rows - r);
      gw_status rc = row_two_pass(ctx, mode, (const C*)a + (long)r * lda, lda, (C*)out + (long)r * ldo, ldo, inv, tmp,
                                  n_chi, rows, scale, st, low >= 0 ? low + r : -1, work * rows / n_rows);
      if (rc || r + rows == n_rows) return rc;
    }
    const dim3 pgrid((row_planes(low, n_rows, mode == 2) + PC::PP - 1) / PC::PP, n_rows);
    auto plane = [&](auto kernel, void* t, long t_row) -> gw_status {
      gw_status r = set_smem(ctx, kernel, PC::bytes);
      if (r) return r;
      KTimer kt(ctx, KF_ROW_FFT, work, st);
      kernel<<<pgrid, PC::TH, PC::bytes, st>>>((const C*)a, lda, (C*)t, t_row, (long)PC::PL, (C*)out, ldo,
                                               inv, (T)scale, low);
      return launch_check(ctx, "row_plane_kernel");
    };
    gw_status rc;
    if (mode == 2) {
      // the columns lie in out itself, at the start of each plane
      if ((rc = line_bwd(ctx, a, lda, out, ldo, PC::PL, inv, n_chi, n_rows, low, false, 0.0, KF_ROW_FFT, st))) return rc;
      return plane(row_plane_kernel<T, N1, N2, N3, 2>, out, ldo);
    }
    if ((rc = plane(row_plane_kernel<T, N1, N2, N3, 1>, tmp, NR))) return rc;
    return line_fwd(ctx, tmp, NR, PC::PL, out, ldo, inv, n_chi, n_rows, low, 0.0, KF_ROW_FFT, st);
  }
  static gw_status row(gw_ctx* ctx, int mode, const void* a, long lda, void* out, long ldo,
                       const int* map, int n_chi, int n_rows, double scale, cudaStream_t st, const int* inv,
                       void* tmp, int low) {
    using L = RowLayout<N1, N2, N3>;
    const size_t bytes = L::TOT * sizeof(C);
    // HBM bytes of the launch: whole rows, or the triangle's share of the grid side
    double grid_el = (double)n_rows * L::NR;
    if (low >= 0) {
      grid_el = 0;
      for (int r = 0; r < n_rows; ++r) grid_el += std::min(L::NR, low + r + 1);
    }
    const double work = (grid_el + (double)n_rows * n_chi) * sizeof(C);
    auto al = [](const void* p) { return p == nullptr || reinterpret_cast<uintptr_t>(p) % 16 == 0; };
    // 16-byte pairs on the grid side (rows of a, or of out for mode 2) and on the G-set side
    const bool vi = mode == 2 ? al(out) && ldo % 2 == 0 && N3 % 2 == 0 : al(a) && lda % 2 == 0 && N3 % 2 == 0;
    const bool vo = mode != 2 && al(out) && ldo % 2 == 0 && n_chi % 2 == 0;
    if (!inv) return fail(ctx, GW_ERR_ARG, "row transform without the G set's inverse map");
    if constexpr (L::TOT * sizeof(C) > kRowSmemMax)
      return row_two_pass(ctx, mode, a, lda, out, ldo, inv, tmp, n_chi, n_rows, scale, st, low, work);
    if constexpr (L::TOT * sizeof(C) <= kRowSmemMax) {
      auto go = [&](auto kernel) -> gw_status {
        gw_status s = set_smem(ctx, kernel, bytes);
        if (s) return s;
        KTimer kt(ctx, KF_ROW_FFT, work, st);
        kernel<<<n_rows, RowCfg<T, N1, N2, N3>::TH, bytes, st>>>((const C*)a, lda, (C*)out, ldo, map, inv,
                                                                 n_chi, (T)scale, low);
        return launch_check(ctx, "row_fft_kernel");
      };
      constexpr bool E = N3 % 2 == 0;
      auto with_low = [&](auto low_c) -> gw_status {
        constexpr bool LOW = decltype(low_c)::value;
        if (mode == 1)
          return vi ? (vo ? go(row_fft_kernel<T, N1, N2, N3, 1, E, true, LOW>)
                          : go(row_fft_kernel<T, N1, N2, N3, 1, E, false, LOW>))
                    : go(row_fft_kernel<T, N1, N2, N3, 1, false, false, LOW>);
        return vi ? go(row_fft_kernel<T, N1, N2, N3, 2, E, false, LOW>)
                  : go(row_fft_kernel<T, N1, N2, N3, 2, false, false, LOW>);
      };
      if (mode == 1 || mode == 2) return low >= 0 ? with_low(std::true_type{}) : with_low(std::false_type{});
    }
    return fail(ctx, GW_ERR_ARG, "bad row transform mode");
  }
  static bool row_pw_ok(int n_pw, int n_chi) {
    using PR = PwRow<T, N1, N2, N3>;
    if constexpr (PR::CL > 0) return PR::smem(n_pw, n_chi) <= kRowSmemMax;
    return false;
  }
  static gw_status row_pw(gw_ctx* ctx, const void* a, const void* b, long lda, void* out, long ldo,
                          const int* inv_pw, int n_pw, int pw_cols, const int* inv_chi, int n_chi, int chi_cols,
                          int n_rows, double scale, cudaStream_t st, int low, void* work) {
    if (!row_pw_ok(n_pw, n_chi))
      return fail(ctx, GW_ERR_UNSUPPORTED, "plane-wave chi rows: no cluster split fits this grid and precision");
    const double nr = (double)N1 * N2 * N3;
    // ALU work: three transforms of N_r points (5 N log2 N each) and the product per row
    auto flops = [&](int rows) { return (double)rows * (3.0 * 5.0 * nr * std::log2(nr) + 6.0 * nr); };
    using P1 = PwOne<T, N1, N2, N3>;
    if constexpr (P1::use) {
      auto one = row_pw_one_kernel<T, N1, N2, N3>;
      gw_status s = set_smem(ctx, one, P1::bytes);
      if (s) return s;
      KTimer kt(ctx, KF_ROW_PW, flops(n_rows), st);
      one<<<n_rows, P1::TH, P1::bytes, st>>>(static_cast<const C*>(a), static_cast<const C*>(b), lda,
                                             static_cast<C*>(out), ldo, inv_pw, inv_chi, n_chi, (T)scale, low);
      return launch_check(ctx, "row_pw_one_kernel");
    } else {
      using PP = PwPlane<T, N1, N2, N3>;
      auto kernel = row_pw_plane_kernel<T, N1, N2, N3>;
      gw_status s = set_smem(ctx, kernel, PP::bytes);
      if (s) return s;
      const int ch = std::min(n_rows, kPwChunk);
      const long tp = pw_cols, tr = (long)N1 * tp, xp = chi_cols, xr = (long)N1 * xp;
      C* ta = static_cast<C*>(work);
      C* tb = ta + ch * tr;
      C* tx = tb + ch * tr;
      for (int r = 0; r < n_rows; r += ch) {
        const int rows = std::min(ch, n_rows - r), lo = low >= 0 ? low + r : -1;
        const C* pa = static_cast<const C*>(a) + (long)r * lda;
        const C* pb = static_cast<const C*>(b) + (long)r * lda;
        if ((s = line_bwd(ctx, pa, lda, ta, tr, tp, inv_pw, n_pw, rows, lo, true, 0.0, KF_ROW_PW, st))) return s;
        if ((s = line_bwd(ctx, pb, lda, tb, tr, tp, inv_pw, n_pw, rows, lo, true, 0.0, KF_ROW_PW, st))) return s;
        {
          const dim3 grid((row_planes(lo, rows, false) + PP::PP - 1) / PP::PP, rows);
          KTimer kt(ctx, KF_ROW_PW, flops(rows), st);             // booked on the planes
          kernel<<<grid, PP::TH, PP::bytes, st>>>(ta, tb, tr, tp, tx, xr, xp, inv_pw, inv_chi, (T)scale, lo);
          if ((s = launch_check(ctx, "row_pw_plane_kernel"))) return s;
        }
        if ((s = line_fwd(ctx, tx, xr, xp, static_cast<C*>(out) + (long)r * ldo, ldo, inv_chi, n_chi, rows, lo, 0.0,
                          KF_ROW_PW, st)))
          return s;
      }
      return GW_OK;
    }
  }
  static bool row_pw_sigma_ok(int n_pw, int n_chi) {
    using PR = PwRow<T, N1, N2, N3>;
    if constexpr (PR::CL > 0) return PR::sig_smem(n_pw, n_chi) <= kRowSmemMax;
    return false;
  }
  static gw_status row_pw_sigma(gw_ctx* ctx, const void* tu, const void* to, long ldt, const void* wg, long ldw,
                                void* hu, void* ho, long ldh, const int* inv_neg, const int* inv_nat, int n_pw,
                                const int* inv_chi, int n_chi, int n_rows, cudaStream_t st) {
    using PR = PwRow<T, N1, N2, N3>;
    if constexpr (PR::CL > 0) {
      const size_t bytes = PR::sig_smem(n_pw, n_chi);
      if (bytes > kRowSmemMax) return fail(ctx, GW_ERR_UNSUPPORTED, "plane-wave Sigma rows: G sets too large");
      auto kernel = row_pw_sigma_kernel<T, N1, N2, N3>;
      gw_status s = set_smem(ctx, kernel, bytes);
      if (s) return s;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(PR::CL, (unsigned)n_rows);
      cfg.blockDim = dim3(PR::THREADS);
      cfg.dynamicSmemBytes = bytes;
      cfg.stream = st;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = PR::CL;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      // five transforms of N_r points and two products per row
      const double nr = (double)N1 * N2 * N3;
      KTimer kt(ctx, KF_ROW_PW, (double)n_rows * (5.0 * 5.0 * nr * std::log2(nr) + 12.0 * nr), st);
      s = cuda_check(ctx, cudaLaunchKernelEx(&cfg, kernel, (const C*)tu, (const C*)to, ldt, (const C*)wg, ldw, (C*)hu,
                                             (C*)ho, ldh, inv_neg, inv_nat, n_pw, inv_chi, n_chi),
                     "cudaLaunchKernelEx(row_pw_sigma_kernel)");
      if (s) return s;
      return launch_check(ctx, "row_pw_sigma_kernel");
    } else {
      return fail(ctx, GW_ERR_UNSUPPORTED, "plane-wave Sigma rows: no cluster split fits this grid and precision");
    }
  }
  static gw_status plane(gw_ctx* ctx, int dir, void* buf, long ld, int ncols, double scale, const int* inv, int cols,
                         cudaStream_t st) {
    using CP = ColPlane<T, N2, N3>;
    dim3 grid((ncols + CP::W - 1) / CP::W, N1);
    auto go = [&](auto kernel) -> gw_status {
      gw_status s = set_smem(ctx, kernel, CP::bytes);
      if (s) return s;
      KTimer kt(ctx, KF_COL_FFT, ((double)N2 * N3 + cols) * N1 * (double)ncols * sizeof(C), st);
      kernel<<<grid, CP::TH, CP::bytes, st>>>((C*)buf, ld, ncols, (T)scale, inv);
      return launch_check(ctx, "col_plane_kernel");
    };
    const bool pairs = sizeof(T) == 4 && ld % 2 == 0 && ncols % 2 == 0 && reinterpret_cast<uintptr_t>(buf) % 16 == 0;
    if (pairs)
      return dir > 0 ? go(col_plane_kernel<T, N1, N2, N3, +1, sizeof(T) == 4>)
                     : go(col_plane_kernel<T, N1, N2, N3, -1, sizeof(T) == 4>);
    return dir > 0 ? go(col_plane_kernel<T, N1, N2, N3, +1, false>) : go(col_plane_kernel<T, N1, N2, N3, -1, false>);
  }
  static gw_status line(gw_ctx* ctx, int dir, int variant, const void* in, long ldi, void* out, long ldo, int ncols,
                        const int* inv, int cols, double scale, cudaStream_t st) {
    dim3 grid((ncols + 127) / 128, cols);
    auto go = [&](auto kernel) -> gw_status {
      KTimer kt(ctx, KF_COL_FFT, 2.0 * N1 * cols * (double)ncols * sizeof(C), st);
      kernel<<<grid, 128, 0, st>>>((const C*)in, ldi, (C*)out, ldo, ncols, N2 * N3, inv, inv + N1 * N2 * N3 + kSetHead,
                                   (T)scale);
      return launch_check(ctx, "col_line_kernel");
    };
    // variant 1: gather rows of `in` through inv; 2: scatter rows of `out` through inv
    if (variant == 1) return dir > 0 ? go(col_line_kernel<T, N1, +1, true, false>)
                                     : go(col_line_kernel<T, N1, -1, true, false>);
    return dir > 0 ? go(col_line_kernel<T, N1, +1, false, true>) : go(col_line_kernel<T, N1, -1, false, true>);
  }
  template <int NTB>
  static gw_status line_ct_reg(gw_ctx* ctx, const void* slabs, long slab_stride, long ld, int ntau, const void* cw,
                               void* out, long out_slice, long ldo, const int* inv, int cols, int ncols,
                               cudaStream_t st) {
    // columns per CTA: enough (tau, 32 columns) pencils for the eight warps
    const int m = std::max(1, std::min(8 / ntau, (ncols + 31) / 32));
    const size_t bytes = (size_t)ntau * N1 * 32 * m * sizeof(float2) + (size_t)ntau * NTB * sizeof(float4);
    auto kernel = col_line_ct_reg_kernel<N1, NTB>;
    gw_status s = set_smem(ctx, kernel, bytes);
    if (s) return s;
    dim3 grid((ncols + 32 * m - 1) / (32 * m), cols);
    KTimer kt(ctx, KF_COL_LINE_CT, ((double)ntau * N1 * cols + (double)ntau * ncols) * ncols * sizeof(float2), st);
    kernel<<<grid, 256, bytes, st>>>((const float2*)slabs, slab_stride, ld, ntau, m, (const float*)cw, (float2*)out,
                                     out_slice, ldo, inv, inv + N1 * N2 * N3 + kSetHead, N2 * N3, ncols);
    return launch_check(ctx, "col_line_ct_reg_kernel");
  }
  static gw_status line_ct(gw_ctx* ctx, const void* slabs, long slab_stride, long ld, int ntau, const void* cw,
                           void* out, long out_slice, long ldo, const int* inv, int cols, int ncols, cudaStream_t st) {
    if constexpr (std::is_same<T, float>::value) {
      auto reg = [&](auto nt) {
        return line_ct_reg<decltype(nt)::value>(ctx, slabs, slab_stride, ld, ntau, cw, out, out_slice, ldo, inv, cols,
                                                ncols, st);
      };
      if (ntau <= 8) return reg(std::integral_constant<int, 8>{});
      if (ntau <= 12) return reg(std::integral_constant<int, 12>{});
      if (ntau <= 16) return reg(std::integral_constant<int, 16>{});
      if (ntau <= 20) return reg(std::integral_constant<int, 20>{});
      if (ntau <= 24) return reg(std::integral_constant<int, 24>{});
      return reg(std::integral_constant<int, 32>{});
    } else {
      const size_t bytes = (size_t)ntau * N1 * 32 * sizeof(C) + (size_t)ntau * ntau * sizeof(T);
      auto kernel = col_line_ct_kernel<T, N1>;
      gw_status s = set_smem(ctx, kernel, bytes);
      if (s) return s;
      dim3 grid((ncols + 31) / 32, cols);
      KTimer kt(ctx, KF_COL_LINE_CT, ((double)ntau * N1 * cols + (double)ntau * ncols) * ncols * sizeof(C), st);
      kernel<<<grid, 256, bytes, st>>>((const C*)slabs, slab_stride, ld, ntau, (const T*)cw, ntau, (C*)out, out_slice,
                                       ldo, inv, inv + N1 * N2 * N3 + kSetHead, N2 * N3, ncols);
      return launch_check(ctx, "col_line_ct_kernel");
    }
  }
};

template <typename T, typename F>
static bool with_grid(const GridInfo& g, F&& f) {
#define X(a, b, c)                                 \
  if (g.n1 == a && g.n2 == b && g.n3 == c) {       \
    f(GridOps<T, a, b, c>{});                      \
    return true;                                   \
  }
  GW_GRIDS(X)
#undef X
  return false;
}

#define GW_DISPATCH(prec, g, BODY)                                                              \
  gw_status rc = GW_OK;                                                                         \
  bool found = is_fp64(prec) ? with_grid<double>(g, [&](auto ops) { using O = decltype(ops); BODY; }) \
                             : with_grid<float>(g, [&](auto ops) { using O = decltype(ops); BODY; });  \
  if (!found) return fail(ctx, GW_ERR_UNSUPPORTED, "no FFT kernels compiled for this grid");     \
  return rc;

gw_status launch_row_fft(gw_ctx* ctx, const GridInfo& g, gw_prec prec, int mode, const void* a, long lda, void* out,
                         long ldo, const int* map, int n_chi, int n_rows, double scale,
                         cudaStream_t st, const int* inv, void* tmp, int low) {
  if (n_rows <= 0) return GW_OK;
  GW_DISPATCH(prec, g, rc = O::row(ctx, mode, a, lda, out, ldo, map, n_chi, n_rows, scale, st, inv, tmp, low))
}

// shared memory of one row (RowLayout)
static size_t row_smem(const GridInfo& g, gw_prec prec) {
  return (size_t)g.n1 * g.n2 * (g.n3 % 2 == 0 ? g.n3 + 1 : g.n3) * csize(prec);
}

bool row_two_pass(const GridInfo& g, gw_prec prec) { return row_smem(g, prec) > kRowSmemMax; }

gw_status launch_row_pw_chi(gw_ctx* ctx, const GridInfo& g, gw_prec prec, const void* a, const void* b, long lda,
                            void* out, long ldo, const int* inv_pw, int n_pw, int pw_cols, const int* inv_chi,
                            int n_chi, int chi_cols, int n_rows, double scale, void* work, cudaStream_t st, int low) {
  if (n_rows <= 0) return GW_OK;
  GW_DISPATCH(prec, g, rc = O::row_pw(ctx, a, b, lda, out, ldo, inv_pw, n_pw, pw_cols, inv_chi, n_chi, chi_cols, n_rows,
                                      scale, st, low, work))
}

size_t row_pw_work(const GridInfo& g, gw_prec prec, int pw_cols, int chi_cols) {
  if (2 * row_smem(g, prec) <= kPwOneMax) return 0;               // one CTA per row
  return (size_t)std::min(g.nr, kPwChunk) * g.n1 * (2 * (size_t)pw_cols + chi_cols) * csize(prec);
}

gw_status check_row_pw(gw_ctx* ctx, const GridInfo& g, gw_prec prec, int n_pw, int n_chi) {
  GW_DISPATCH(prec, g, rc = O::row_pw_ok(n_pw, n_chi) ? GW_OK : fail(ctx, GW_ERR_UNSUPPORTED,
                                                                     "plane-wave chi rows: grid, precision and G sets "
                                                                     "beyond the sizes of the plane-wave route"))
}

gw_status launch_row_pw_sigma(gw_ctx* ctx, const GridInfo& g, gw_prec prec, const void* tu, const void* to, long ldt,
                              const void* wg, long ldw, void* hu, void* ho, long ldh, const int* inv_neg,
                              const int* inv_nat, int n_pw, const int* inv_chi, int n_chi, int n_rows,
                              cudaStream_t st) {
  if (n_rows <= 0) return GW_OK;
  GW_DISPATCH(prec, g, rc = O::row_pw_sigma(ctx, tu, to, ldt, wg, ldw, hu, ho, ldh, inv_neg, inv_nat, n_pw, inv_chi,
                                            n_chi, n_rows, st))
}

gw_status check_row_pw_sigma(gw_ctx* ctx, const GridInfo& g, gw_prec prec, int n_pw, int n_chi) {
  GW_DISPATCH(prec, g, rc = O::row_pw_sigma_ok(n_pw, n_chi) ? GW_OK : fail(ctx, GW_ERR_UNSUPPORTED,
                                                                           "plane-wave Sigma rows: this grid, "
                                                                           "precision and G sets do not fit a "
                                                                           "thread-block cluster"))
}

gw_status launch_col_plane(gw_ctx* ctx, const GridInfo& g, gw_prec prec, int dir, void* buf, long ld, int ncols,
                           double scale, const int* inv, int cols, cudaStream_t st) {
  GW_DISPATCH(prec, g, rc = O::plane(ctx, dir, buf, ld, ncols, scale, inv, cols, st))
}

gw_status launch_col_line(gw_ctx* ctx, const GridInfo& g, gw_prec prec, int dir, int variant, const void* in,
                          long ldi, void* out, long ldo, int ncols, const int* inv, int cols, double scale,
                          cudaStream_t st) {
  GW_DISPATCH(prec, g, rc = O::line(ctx, dir, variant, in, ldi, out, ldo, ncols, inv, cols, scale, st))
}

gw_status launch_col_line_ct(gw_ctx* ctx, const GridInfo& g, gw_prec prec, const void* slabs, long slab_stride,
                             long ld, int ntau, const void* cw, void* out, long out_slice, long ldo, const int* inv,
                             int cols, int ncols, cudaStream_t st) {
  GW_DISPATCH(prec, g,
              rc = O::line_ct(ctx, slabs, slab_stride, ld, ntau, cw, out, out_slice, ldo, inv, cols, ncols, st))
}

template <int NTB>
static gw_status launch_ct_reg(gw_ctx* ctx, bool st_kind, int n, const void* dM, size_t elems, const void* in,
                               void* out, cudaStream_t st) {
  KTimer kt(ctx, KF_CT, 2.0 * n * (double)elems * sizeof(float2), st);
  const bool two = elems % 2 == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0;
  const size_t items = two ? elems / 2 : elems;
  const int blocks = (int)std::min<size_t>((items + 127) / 128, (size_t)ctx->num_sms * 24);
  auto go = [&](auto kernel) -> gw_status {
    kernel<<<blocks, 128, 0, st>>>((const float2*)in, (float2*)out, elems, n, (const float*)dM);
    return launch_check(ctx, "ct_reg_kernel");
  };
  if (two) return st_kind ? go(ct_reg_kernel<NTB, true, 2>) : go(ct_reg_kernel<NTB, false, 2>);
  return st_kind ? go(ct_reg_kernel<NTB, true, 1>) : go(ct_reg_kernel<NTB, false, 1>);
}

gw_status launch_ct(gw_ctx* ctx, gw_prec prec, bool st_kind, int n, const void* dM, size_t elems, const void* in,
                    void* out, cudaStream_t st) {
  if (elems == 0) return GW_OK;
  if (!is_fp64(prec)) {
    if (n <= 4) return launch_ct_reg<4>(ctx, st_kind, n, dM, elems, in, out, st);
    if (n <= 8) return launch_ct_reg<8>(ctx, st_kind, n, dM, elems, in, out, st);
    if (n <= 12) return launch_ct_reg<12>(ctx, st_kind, n, dM, elems, in, out, st);
    if (n <= 16) return launch_ct_reg<16>(ctx, st_kind, n, dM, elems, in, out, st);
    if (n <= 20) return launch_ct_reg<20>(ctx, st_kind, n, dM, elems, in, out, st);
    if (n <= 24) return launch_ct_reg<24>(ctx, st_kind, n, dM, elems, in, out, st);
    return launch_ct_reg<32>(ctx, st_kind, n, dM, elems, in, out, st);
  }
  int blocks = (int)std::min<size_t>((elems + 255) / 256, (size_t)ctx->num_sms * 8);
  KTimer kt(ctx, KF_CT, 2.0 * n * (double)elems * sizeof(double2), st);
  if (st_kind) ct_kernel<true><<<blocks, 256, 0, st>>>((const double2*)in, (double2*)out, elems, n, (const double*)dM);
  else ct_kernel<false><<<blocks, 256, 0, st>>>((const double2*)in, (double2*)out, elems, n, (const double*)dM);
  return launch_check(ctx, "ct_kernel");
}

gw_status launch_hadamard(gw_ctx* ctx, gw_prec prec, size_t count, const void* a, const void* b, double scale,
                          void* out, cudaStream_t st) {
  if (count == 0) return GW_OK;
  int blocks = (int)std::min<size_t>((count + 255) / 256, (size_t)ctx->num_sms * 16);
  if (is_fp64(prec))
    hadamard_kernel<double><<<blocks, 256, 0, st>>>((const double2*)a, (const double2*)b, (double2*)out, count, scale);
  else
    hadamard_kernel<float><<<blocks, 256, 0, st>>>((const float2*)a, (const float2*)b, (float2*)out, count, (float)scale);
  return launch_check(ctx, "hadamard_kernel");
}

// Transform weights w * fac as FP32 pairs: hi = fl(w fac), lo = fl(w fac - hi);
// returns [hi_0 .. hi_{count-1}, lo_0 .. lo_{count-1}].
std::vector<float> split_weights(const double* w, int count, double fac) {
  std::vector<float> out(2 * (size_t)count);
  for (int e = 0; e < count; ++e) {
    const double v = w[e] * fac;
    out[e] = (float)v;
    out[count + e] = (float)(v - (double)out[e]);
  }
  return out;
}

// Upload a host array into arena memory (pageable copy; the host buffer may be
// released on return).
gw_status upload(gw_ctx* ctx, void* dst, const void* src, size_t bytes, cudaStream_t st) {
  if (bytes == 0) return GW_OK;
  return cuda_check(ctx, cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st), "upload");
}

gw_status index_maps(gw_ctx* ctx, const GridInfo& g, const int32_t* fft_index_h, int n_chi, std::vector<int>& map,
                     std::vector<int>& inv) {
  if (!fft_index_h) return fail(ctx, GW_ERR_ARG, "fft_index_h is NULL");
  if (n_chi < 1 || n_chi > g.nr) return fail(ctx, GW_ERR_SHAPE, "need 1 <= n_chi <= N_r");
  map.assign(fft_index_h, fft_index_h + n_chi);
  inv.reserve(inv_ints(g));
  inv.assign(g.nr, -1);
  for (int j = 0; j < n_chi; ++j) {
    if (map[j] < 0 || map[j] >= g.nr) return fail(ctx, GW_ERR_ARG, "fft_index out of range");
    if (inv[map[j]] >= 0) return fail(ctx, GW_ERR_ARG, "fft_index has duplicates");
    inv[map[j]] = j;
  }
  set_lists(g, inv);
  return GW_OK;
}

void set_lists(const GridInfo& g, std::vector<int>& inv) {
  inv.resize(g.nr);
  const int pl = g.n2 * g.n3, n12 = g.n1 * g.n2;
  const int sizes[5] = {pl, n12, g.n1, g.n2, g.n3};
  std::vector<char> marks((size_t)pl + n12 + g.n1 + g.n2 + g.n3, 0);
  char *c23 = marks.data(), *c12 = c23 + pl, *u1 = c12 + n12, *u2 = u1 + g.n1, *u3 = u2 + g.n2;
  // Every entry point with a G set pays for this walk over the grid, so no division and no branch per
  // point: with three of the former and five marks a call with the whole set of 24^3 took 0.09 ms longer.
  const int* at_p = inv.data();
  for (int e = 0; e < n12; ++e) {
    char* c = c23 + e % g.n2 * g.n3;
    char any = 0;
    for (int i3 = 0; i3 < g.n3; ++i3) {
      const char in = *at_p++ >= 0;
      c[i3] |= in;
      any |= in;
    }
    c12[e] = any;
    u1[e / g.n2] |= any;
  }
  for (int e = 0; e < pl; ++e) {
    u2[e / g.n3] |= c23[e];
    u3[e % g.n3] |= c23[e];
  }
  inv.resize(inv_ints(g), 0);
  int* x = inv.data() + g.nr;
  int* at = x + kSetHead;
  const char* m = c23;
  for (int v = 0; v < 5; m += sizes[v], at += sizes[v], ++v) {
    int count = 0;
    for (int i = 0; i < sizes[v]; ++i)
      if (m[i]) at[count++] = i;
    x[v] = count;
  }
}

}  // namespace gw

using namespace gw;

extern "C" gw_status gw_chi0_rtau(gw_ctx* ctx, int n_rows, int n_cols, gw_prec prec, const void* g_occ,
                                  const void* g_unocc, void* chi, void* stream) {
  if (!ctx) return fail(nullptr, GW_ERR_ARG, "ctx is NULL");
  if (!valid_prec(prec)) return fail(ctx, GW_ERR_ARG, "bad precision");
  if (n_rows < 0 || n_cols < 0) return fail(ctx, GW_ERR_SHAPE, "negative size");
  if ((size_t)n_rows * n_cols == 0) return GW_OK;
  if (!g_occ || !g_unocc || !chi) return fail(ctx, GW_ERR_ARG, "NULL pointer");
  return launch_hadamard(ctx, prec, (size_t)n_rows * n_cols, g_occ, g_unocc, -2.0, chi, as_stream(stream));
}

extern "C" gw_status gw_rr_to_GG_fft(gw_ctx* ctx, const gw_grid* grid, int direction, int stage, int n_chi,
                                     const int32_t* fft_index_h, gw_prec prec, int r0, int n_rows, const void* in,
                                     void* out, void* stream) {
  if (!ctx) return fail(nullptr, GW_ERR_ARG, "ctx is NULL");
  GridInfo g;
  gw_status st = grid_info(ctx, grid, &g);
  if (st) return st;
  if (!grid_supported(g.n1, g.n2, g.n3)) return fail(ctx, GW_ERR_UNSUPPORTED, "no FFT kernels compiled for this grid");
  if (!valid_prec(prec)) return fail(ctx, GW_ERR_ARG, "bad precision");
  if (direction != 1 && direction != -1) return fail(ctx, GW_ERR_ARG, "direction must be +1 or -1");
  if (stage != 1 && stage != 2) return fail(ctx, GW_ERR_ARG, "stage must be 1 or 2");
  if (!in || !out) return fail(ctx, GW_ERR_ARG, "NULL pointer");
  std::vector<int> map, inv;
  if ((st = index_maps(ctx, g, fft_index_h, n_chi, map, inv))) return st;
  if (stage == 1 && (n_rows < 0 || r0 < 0 || r0 + n_rows > g.nr)) return fail(ctx, GW_ERR_SHAPE, "rows out of range");
  cudaStream_t s = as_stream(stream);
  const int cols = set_columns(g, inv);
  // rows too long for shared memory need a [rows][N_r] workspace forward: so many rows at a time
  const bool work_rows = stage == 1 && direction > 0 && row_two_pass(g, prec);
  const int chunk = std::min(n_rows, 1024);
  Carver probe(nullptr);
  probe.take<int>(n_chi);
  probe.take<int>(inv_ints(g));
  if (work_rows) probe.take<char>((size_t)chunk * g.nr * csize(prec));
  if ((st = reserve(ctx, probe.off))) return st;
  Carver cv(ctx->arena);
  int* dmap = cv.take<int>(n_chi);
  int* dinv = cv.take<int>(inv_ints(g));
  void* tmp = work_rows ? cv.take<char>((size_t)chunk * g.nr * csize(prec)) : nullptr;
  if ((st = upload(ctx, dmap, map.data(), sizeof(int) * n_chi, s))) return st;
  if ((st = upload(ctx, dinv, inv.data(), sizeof(int) * inv.size(), s))) return st;
  if (stage == 1) {
    const size_t es = csize(prec);
    for (int r = 0; work_rows && r < n_rows; r += chunk)
      if ((st = launch_row_fft(ctx, g, prec, 1, static_cast<const char*>(in) + (size_t)r * g.nr * es, g.nr,
                               static_cast<char*>(out) + (size_t)r * n_chi * es, n_chi, dmap, n_chi,
                               std::min(chunk, n_rows - r), 1.0, s, dinv, tmp)))
        return st;
    if (work_rows) return GW_OK;
    if (direction > 0)
      return launch_row_fft(ctx, g, prec, 1, in, g.nr, out, n_chi, dmap, n_chi, n_rows, 1.0, s, dinv, tmp);
    return launch_row_fft(ctx, g, prec, 2, in, n_chi, out, g.nr, dmap, n_chi, n_rows, 1.0 / g.volume, s,
                          dinv);
  }
  if (direction > 0) {
    // in [N_r][n_chi] is the work buffer: (i2,i3) planes in place, then the i1 pass writes the G rows of out.
    void* work = const_cast<void*>(in);
    if ((st = launch_col_plane(ctx, g, prec, -1, work, n_chi, n_chi, 1.0, dinv, cols, s))) return st;
    return launch_col_line(ctx, g, prec, -1, 2, work, n_chi, out, n_chi, n_chi, dinv, cols, g.dv * g.dv / g.volume, s);
  }
  // W(G,G') -> W(r,G'): i1 pass gathering the G rows, then the (i2,i3) planes in place in out.
  if ((st = launch_col_line(ctx, g, prec, +1, 1, in, n_chi, out, n_chi, n_chi, dinv, cols, 1.0, s))) return st;
  return launch_col_plane(ctx, g, prec, +1, out, n_chi, n_chi, 1.0, dinv, cols, s);
}

extern "C" gw_status gw_tau_to_omega(gw_ctx* ctx, int kind, int n, const double* M_h, size_t elems, gw_prec prec,
                                     const void* in, void* out, void* stream) {
  if (!ctx) return fail(nullptr, GW_ERR_ARG, "ctx is NULL");
  if (!valid_prec(prec)) return fail(ctx, GW_ERR_ARG, "bad precision");
  if (kind != GW_CT && kind != GW_ST && kind != GW_IST) return fail(ctx, GW_ERR_ARG, "kind must be GW_CT, GW_ST or GW_IST");
  if (n < 1 || n > 32) return fail(ctx, GW_ERR_SHAPE, "need 1 <= n <= 32");
  if (!M_h || !in || !out) return fail(ctx, GW_ERR_ARG, "NULL pointer");
  if (in == out) return fail(ctx, GW_ERR_ARG, "in and out must not overlap");
  cudaStream_t s = as_stream(stream);
  gw_status st = reserve(ctx, 8 * 32 * 32);
  if (st) return st;
  std::vector<double> neg;
  if (kind == GW_IST) {             // -i sum M x = i sum (-M) x: the sine kernel with M negated
    neg.assign(M_h, M_h + (size_t)n * n);
    for (double& v : neg) v = -v;
    M_h = neg.data();
  }
  std::vector<float> m32;
  if (is_fp64(prec)) {
    if ((st = upload(ctx, ctx->arena, M_h, sizeof(double) * n * n, s))) return st;
  } else {
    m32 = split_weights(M_h, n * n, 1.0);
    if ((st = upload(ctx, ctx->arena, m32.data(), sizeof(float) * 2 * n * n, s))) return st;
  }
  return launch_ct(ctx, prec, kind != GW_CT, n, ctx->arena, elems, in, out, s);
}

// ---------------------------------------------------------------------- no-allocation variant
//
// gw_rr_to_GG_fft needs two small index maps on the device (the G set's FFT
// positions and their inverse).  The regular entry point keeps them in the
// context's scratch arena, which is created with cudaMalloc.  This variant keeps
// them instead in one fixed array in the library's own device memory, so a
// caller that may not allocate device memory at all can still run the
// transform: for example a program whose memory pool has taken the whole GPU
// and forbids any other cudaMalloc, or a serving loop that cannot afford the
// device-wide synchronisation a cudaMalloc/cudaFree may bring.  The maps are
// still uploaded on every call, by cudaMemcpyAsync from pageable host memory:
// that copy waits for the stream's earlier work before it starts, so a call
// is not free of host-side waiting, only of allocation.

namespace {

constexpr int kNoAllocMaxInts = 2 * 13824;   // n_chi + N_r for the largest compiled grid (24^3)
constexpr int kNoAllocLists = kSetHead + 2 * 24 * 24 + 3 * 24;   // and the set's lists behind its inverse map

// Holds fft_index followed by its inverse map and the set's lists (set_lists).  Every GPU that loads the
// library keeps this array until the process exits; all calls share it.
static __device__ __align__(256) int g_noalloc_maps[kNoAllocMaxInts + kNoAllocLists];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
int* g_noalloc_ptr[kMaxDevices] = {nullptr};

// Device address of g_noalloc_maps on the current device (looked up once per
// device).  In host code the symbol itself is only a host-side stand-in.
gw_status noalloc_maps_ptr(gw_ctx* err_ctx, int** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_check(err_ctx, e, "cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) return fail(err_ctx, GW_ERR_UNSUPPORTED, "device index too large");
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_maps);
    if (e != cudaSuccess) return cuda_check(err_ctx, e, "cudaGetSymbolAddress(g_noalloc_maps)");
    g_noalloc_ptr[dev] = static_cast<int*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return GW_OK;
}

}  // namespace

extern "C" gw_status gw_rr_to_GG_fft_noalloc(const gw_grid* grid, int direction, int stage, int n_chi,
                                             const int32_t* fft_index_h, gw_prec prec, int r0, int n_rows,
                                             const void* in, void* out, void* stream) {
  gw_ctx local;                       // host-only bookkeeping: no device memory behind it
  local.num_sms = 1;
  auto done = [&](gw_status st) {
    if (st) fail(nullptr, st, local.err);
    return st;
  };
  GridInfo g;
  gw_status st = grid_info(&local, grid, &g);
  if (st) return done(st);
  if (!grid_supported(g.n1, g.n2, g.n3)) return done(fail(&local, GW_ERR_UNSUPPORTED, "no FFT kernels compiled for this grid"));
  if (!valid_prec(prec)) return done(fail(&local, GW_ERR_ARG, "bad precision"));
  if (direction != 1 && direction != -1) return done(fail(&local, GW_ERR_ARG, "direction must be +1 or -1"));
  if (stage != 1 && stage != 2) return done(fail(&local, GW_ERR_ARG, "stage must be 1 or 2"));
  if (!in || !out) return done(fail(&local, GW_ERR_ARG, "NULL pointer"));
  cudaStream_t s = as_stream(stream);
  // The maps are copied from host vectors that live only for this call: a
  // captured copy would replay from freed host memory, so refuse capture.
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaError_t ce = cudaStreamIsCapturing(s, &cap);
  if (ce != cudaSuccess) return done(cuda_check(&local, ce, "cudaStreamIsCapturing"));
  if (cap != cudaStreamCaptureStatusNone)
    return done(fail(&local, GW_ERR_UNSUPPORTED,
                     "gw_rr_to_GG_fft_noalloc cannot be called while its stream is being captured"));
  std::vector<int> map, inv;
  if ((st = index_maps(&local, g, fft_index_h, n_chi, map, inv))) return done(st);
  if ((long)n_chi + g.nr > kNoAllocMaxInts)
    return done(fail(&local, GW_ERR_SHAPE, "n_chi + N_r exceeds the fixed index-map capacity of " +
                                               std::to_string(kNoAllocMaxInts) + " entries"));
  if (stage == 1 && (n_rows < 0 || r0 < 0 || r0 + n_rows > g.nr))
    return done(fail(&local, GW_ERR_SHAPE, "rows out of range"));
  const int cols = set_columns(g, inv);
  int* maps = nullptr;
  if ((st = noalloc_maps_ptr(&local, &maps))) return done(st);
  int* dmap = maps;
  int* dinv = maps + n_chi;
  // both maps are rewritten in full on every call, so nothing carries over
  if ((st = upload(&local, dmap, map.data(), sizeof(int) * n_chi, s))) return done(st);
  if ((st = upload(&local, dinv, inv.data(), sizeof(int) * inv.size(), s))) return done(st);
  if (stage == 1) {
    if (direction > 0) st = launch_row_fft(&local, g, prec, 1, in, g.nr, out, n_chi, dmap, n_chi, n_rows, 1.0, s, dinv);
    else st = launch_row_fft(&local, g, prec, 2, in, n_chi, out, g.nr, dmap, n_chi, n_rows, 1.0 / g.volume, s, dinv);
    return done(st);
  }
  if (direction > 0) {
    void* work = const_cast<void*>(in);
    if ((st = launch_col_plane(&local, g, prec, -1, work, n_chi, n_chi, 1.0, dinv, cols, s))) return done(st);
    return done(launch_col_line(&local, g, prec, -1, 2, work, n_chi, out, n_chi, n_chi, dinv, cols, g.dv * g.dv / g.volume, s));
  }
  if ((st = launch_col_line(&local, g, prec, +1, 1, in, n_chi, out, n_chi, n_chi, dinv, cols, 1.0, s))) return done(st);
  return done(launch_col_plane(&local, g, prec, +1, out, n_chi, n_chi, 1.0, dinv, cols, s));
}
