// Tensor-core (tcgen05) formation of the imaginary-time Green's functions
// (Eqs. Green_occ, Green_unocc) and of the real-space product of Eq. chi_rr.
//
// Complex products on real tensor cores.  With a(r,k) = psi_k(r) s_k and
// b(R',k) = conj(psi_k(R')), G(r,R') = sum_k a(r,k) b(R',k) is one real GEMM
//   D[r][2R'+c] = sum_k' A[r][k'] B[2R'+c][k']     (k' = 2k, 2k+1)
// where A is the complex array viewed as real (re, im interleaved along k) and B
// holds two real rows per complex column:
//   B[2R'  ] = ( br_k, -bi_k )   ->  D[r][2R'  ] = Re G(r,R')
//   B[2R'+1] = ( bi_k,  br_k )   ->  D[r][2R'+1] = Im G(r,R')
// so the FP32 accumulator in tensor memory already holds (re, im) pairs.
//
// FP32-level accuracy from 16-bit tensor cores: every operand is split as
// x = hi + lo (hi = fp16(x), lo = fp16(x - hi)) after a power-of-two scaling
// that puts max|x| near 2^15, and D = A_hi B_hi + A_hi B_lo + A_lo B_hi
// (dropping A_lo B_lo ~ 2^-22 |A||B|), accumulated in FP32.  bf16 splits are
// the same code with a coarser 2 x 8-bit representation.
//
// Tile: 128 rows r x 128 complex columns R' (MMA 128 x 256 x 16), K staged 32
// real elements at a time through a 4-stage TMA/mbarrier pipeline.  The 32 hi and
// 32 lo values of a row lie side by side (128 B, SWIZZLE_128B), one load for A and
// one for B: with hi and lo apart in 64-byte rows the loads lagged the MMAs (36^3, 4224
// bands: 133 to 138 ms for 2 tau, now 130.5, 564 TFLOP/s); the epilogue stages rows in shared memory and writes 128-byte row
// segments.  G_unocc is summed blockwise through the two 256-column halves of
// tensor memory into registers, G_occ accumulates last in one half; the
// epilogue either writes both (gw_green_tau) or their product
// chi = -2 G_occ conj(G_unocc) (gw_chi0_rtau_fused), so for chi neither G tile
// ever reaches HBM.  Warp roles: 0 = TMA producer, 1 = MMA issuer (and tensor
// memory owner), the rest = epilogue.  Every wait is bounded; on time-out the
// kernel records it in the status word, drains its own copies and MMAs, frees
// its tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cmath>
#include <mutex>
#include <type_traits>

#include "gw_tc.h"
#include "gw_tcgen05.cuh"

namespace gw {
namespace tc {

using namespace tcx;

constexpr int BM = 128;                 // rows per tile
constexpr int BNC = 128;                // complex columns per tile (MMA N = 256)
constexpr int BK = 32;                  // real K per stage: its hi and lo values make one 128-byte operand row
constexpr int STAGES = 4;
constexpr int CH = 4;                   // stages per accumulation block (128 real K)
// Epilogue warps: four per tensor-memory lane quarter (64 sums a thread, 96 registers) for the modes
// that write their tile; two (128 sums, 168 registers) for the self-energy, whose longer code spilled
// inside the K loop with 96 (36^3, 2 tau: 180 against 148 ms).  With two, the writing modes spilled
// 400 bytes a thread past the small L1 and their tile's end took 16 thousand cycles, more than the two
// accumulation blocks that the MMAs run ahead: chi rows at 20^3 with 512 bands 3.96 ms, with four 3.42
// (466 TFLOP/s), at 24^3 with 1024 bands 13.1 and 11.9 ms.
template <int MODE>
constexpr int kEpiWarps = MODE == 2 ? 8 : 16;
constexpr int A_BYTES = BM * BK * 4;            // 16 KB
constexpr int B_BYTES = 2 * BNC * BK * 4;       // 32 KB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int H_BYTES = BM * BK * 2;            // a 32-wide K chunk of H, hi or lo (64-byte rows)
constexpr int EPI_COLS = 8;                     // complex columns per epilogue round
constexpr int EPI_BYTES = 16 * 32 * EPI_COLS * 8;
constexpr int kTileTab = 256;                   // tiles of a CTA looked up in advance
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + EPI_BYTES + 4 * kTileTab + 1024 + 256;
template <int MODE>
constexpr int kThreads = 64 + 32 * kEpiWarps<MODE>;
static_assert(SMEM_BYTES <= 232448, "shared memory per CTA");

constexpr int kMaxEntries = 64;

struct Params {
  int m_rows;             // valid output rows
  int n_cols;             // valid complex output columns (N_r)
  int k_occ_steps;        // BK stages of the occupied region
  int k_un_steps;         // BK stages of the unoccupied region
  int k_un_x;             // first real K index of the unoccupied region
  float2* out0;           // chi, or G_occ
  float2* out1;           // G_unocc (green mode)
  long ldo;
  // independent products (k points, or times of one set of orbitals): entry z has its own A operand,
  // factors and output, and its own B operand and scaling unless shared
  int nb, b_shared;
  long so;                // elements between the entries' outputs
  float alpha_occ[kMaxEntries];   // A_occ (FP64 max exponential, rounded)
  float alpha_un[kMaxEntries];
  const int* dexp;        // device [nb] (or one, shared): e of the 2^e operand scaling
  int gx, gy, tiles;      // column and row tiles, tiles in use per entry
  int* status;            // device: [0] time-out flag, [1] where
  // MODE 2 (self-energy): contraction of G o W~ with psi_n on the tensor cores
  const float2* wrr;      // W~(r, R') rows of the block, [m_rows][ldw]
  long ldw;
  const float2* psi;      // psi [N_b][ldpsi]: psi_n(r) for the final sum over r
  long ldpsi;
  const int* bands;       // [n_n] device
  int n_n, np;            // bands; MMA N = 2 n_n rounded up to 16
  int r0;                 // grid row of the block's first row
  double coef;            // dV^2 / Omega
  double* acc_u;          // Sigma_unocc_nn(tau_j) at acc_u[n * acc_stride], Sigma_occ likewise
  double* acc_o;
  int acc_stride;
  // MODE 0 and 2: only tiles with R' <= r (the grid row of the tile's rows is r0 + local row).
  // chi(r,R') and G(r,R') W~(r,R') are Hermitian in (r, R'): MODE 0 writes the lower triangle with
  // the diagonal halved (T, so that the transform of chi is X + X^H with X that of T) and zeros
  // above it in the tiles on the diagonal; MODE 2 weights the strictly lower part 2 and the
  // diagonal 1 (the real quadratic form).
  int lower;
};

// Blocked accumulation.  The tensor cores add each MMA's products into the FP32
// accumulator without rounding to nearest, so the relative error of a long
// accumulation grows about linearly with the number of MMAs (3 per 16 real K
// here): ~1e-5 for a thousand bands.  G_unocc is therefore summed in blocks of
// CH stages: each block accumulates from zero in one of the two 256-column
// halves of tensor memory while the epilogue warps add the other half's
// finished block into FP32 registers (round to nearest), which keeps the
// error at the level of one block.  G_occ (the short sum over the occupied
// bands) follows as the last block and stays in tensor memory for the
// epilogue.
//
// MODE 0: out0 = -2 G_occ conj(G_unocc);  MODE 1: out0 = G_occ, out1 = G_unocc.
// MODE 2: the self-energy contraction of the tile (first term of Eq.
// Sigma_occ_reduce, Eq. Sigma_rr), with nothing written but the band sums:
//   H(r,R') = G(r,R') W~(r,R')                        (CUDA cores, FP32)
//   V_n(r)  = sum_{R' in tile} H(r,R') psi_n(R')      (tcgen05, 3 fp16 split products)
//   Sigma_unocc_nn += coef Re(conj(psi_n(r)) V_n^unocc(r)),  Sigma_occ_nn -= ... V_n^occ
// Once the tile's G is complete the pipeline stages are free: the epilogue
// writes H row by row (its own power-of-two scale per row and column half) as
// split fp16 in the 64-byte-swizzled K-major layout TMA would produce, the
// producer loads the tile's psi_n operand behind it, and the MMA warp
// accumulates V for each half of the tile's columns in the free half of
// tensor memory; unoccupied first, then occupied in the same shared memory.
// The epilogue is not overlapped with MMAs, so its length counts: W~ is loaded
// once, by TMA into the place its own H will take, for both products
// (H_occ waits in tensor memory), and the band sums are reduced by exchange.  With
// one row of W~ per lane straight from global memory, twice, and five shuffles
// and a double atomic per band, a tile's epilogue took 90 (4 bands) to 154
// (32 bands) thousand cycles, now 38 and 50; sigma at 20^3 with 512 bands 14.9 ->
// 10.4 ms, at 36^3 with 4224 bands and 2 tau 207 -> 170 ms.
template <int MODE, uint32_t FMT>
__global__ void __launch_bounds__(kThreads<MODE>, 1) green_tc_kernel(const __grid_constant__ CUtensorMap mA,
                                                                     const __grid_constant__ CUtensorMap mB,
                                                                     const __grid_constant__ CUtensorMap mP_hi,
                                                                     const __grid_constant__ CUtensorMap mP_lo,
                                                                     const __grid_constant__ CUtensorMap mW, Params p) {
  constexpr int EW = kEpiWarps<MODE>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  float2* epi = reinterpret_cast<float2*>(smem + STAGES * STAGE_BYTES);     // [16 warps][32 rows][8]
  uint32_t* tile_tab = reinterpret_cast<uint32_t*>(smem + STAGES * STAGE_BYTES + EPI_BYTES);
  uint64_t* full = reinterpret_cast<uint64_t*>(tile_tab + kTileTab);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;      // [2] block finished in tensor-memory half b
  uint64_t* tempty = tfull + 2;          // [2] half b drained by the epilogue
  uint64_t* done = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  // MODE 2
  uint64_t* hready = done + 2;           // [2] H operand of column half h written (4 warps)
  uint64_t* hfree = hready + 2;          // [2] unoccupied MMAs of half h done: its H may be overwritten
  uint64_t* vready = hfree + 2;          // [2] every V MMA of half h done
  uint64_t* psi_full = vready + 2;       // psi_n operand of the tile landed
  uint64_t* redbar = psi_full + 1;       // the epilogue warps' band sums are in shared memory
  uint64_t* done2 = redbar + 1;          // every MMA of the self-energy phase done
  uint64_t* last_mma = done2 + 1;
  uint64_t* w_full = last_mma + 1;       // W~ of the tile landed
  float* red = reinterpret_cast<float*>(epi);     // [8 warps][32][2] band sums of the warps (MODE 2 only)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Tile t: its entry, row tile and column tile.  Only tiles with some R' <= r are counted in
  // lower-triangle mode.  They go in groups of eight row tiles, column by column: the CTAs that run
  // together share B (and A) tiles in L2 instead of each reading its B from DRAM.
  struct Tile {
    int z, m0, n0;
  };
  auto cols_of = [&](int i) { return p.lower ? min(p.gx, (p.r0 + i * BM + BM - 1) / BNC + 1) : p.gx; };
  auto find_tile = [&](int t) -> Tile {
    constexpr int kGroupRows = 8;
    Tile o;
    o.z = t / p.tiles;
    int r = t - o.z * p.tiles, first = 0, rows;
    for (;; first += kGroupRows) {
      rows = min(kGroupRows, p.gy - first);
      int count = 0;
      for (int i = 0; i < rows; ++i) count += cols_of(first + i);
      if (r < count) break;
      r -= count;
    }
    const int all = cols_of(first);                     // columns that every row of the group has
    int i, c;
    if (r < rows * all) {
      i = r % rows;
      c = r / rows;
    } else {
      r -= rows * all;
      for (i = 0; r >= cols_of(first + i) - all; ++i) r -= cols_of(first + i) - all;
      c = all + r;
    }
    o.m0 = (first + i) * BM;
    o.n0 = c * BNC;
    return o;
  };
  const int n_tiles = p.tiles * p.nb;
  // the CTA's first tiles are found by all its threads at once
  for (int i = threadIdx.x; i < kTileTab && blockIdx.x + (long)i * gridDim.x < n_tiles; i += kThreads<MODE>) {
    const Tile o = find_tile(blockIdx.x + i * gridDim.x);
    tile_tab[i] = (uint32_t)o.z << 26 | (uint32_t)(o.m0 / BM) << 13 | (uint32_t)(o.n0 / BNC);
  }
  auto tile_at = [&](int t, int i) -> Tile {       // tile t, the CTA's i-th
    if (i >= kTileTab) return find_tile(t);
    const uint32_t e = tile_tab[i];
    Tile o;
    o.z = (int)(e >> 26);
    o.m0 = (int)(e >> 13 & 8191) * BM;
    o.n0 = (int)(e & 8191) * BNC;
    return o;
  };
  const int total = p.k_occ_steps + p.k_un_steps;
  const int n_un_blocks = (p.k_un_steps + CH - 1) / CH;
  const bool have_occ = p.k_occ_steps > 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], EW);
    }
    mbar_init(done, 1);
    mbar_init(last_mma, 1);
    if (MODE == 2) {
      for (int b = 0; b < 2; ++b) {
        mbar_init(&hready[b], EW / 2);
        mbar_init(&hfree[b], 1);
        mbar_init(&vready[b], 1);
      }
      mbar_init(psi_full, 1);
      mbar_init(redbar, EW);
      mbar_init(done2, 1);
      mbar_init(w_full, 1);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // MODE 2 operands in the freed pipeline stages: H hi [0, 64 KB), H lo [64, 128 KB) as eight
  // 32-wide K chunks of 128 rows; psi_n hi and lo from 128 KB, chunks of np rows.
  uint8_t* const h_hi = smem;
  uint8_t* const h_lo = smem + 8 * H_BYTES;
  uint8_t* const p_hi = smem + 16 * H_BYTES;
  const int p_chunk = MODE == 2 ? p.np * BK * 2 : 0;
  uint8_t* const p_lo = p_hi + 8 * p_chunk;
  // W~ columns 64 h + 8 k .. + 7 of the tile lie where K chunk 4 h + k % 4 of H will, hi for k < 4 and
  // lo above, swizzled alike: row r of W~ is where row r of that chunk will be, so the thread that owns
  // row r and half h overwrites only what it has read itself
  auto w_piece = [&](int h, int k) -> uint8_t* { return (k < 4 ? h_hi : h_lo) + (4 * h + (k & 3)) * H_BYTES; };

  auto timed_out = [&](int where) {
    *abort_flag = 1;
    if (atomicCAS(p.status, 0, 1) == 0) p.status[1] = where;
  };
  // bounded wait that also gives up once another role has aborted
  auto wait_or_abort = [&](uint64_t* bar, uint32_t parity) -> bool {
    const unsigned long long t0 = gtimer();
    while (!mbar_test(bar, parity)) {
      if (*abort_flag) return false;
      if (gtimer() - t0 > kWaitNs) return false;
    }
    return true;
  };

  if (warp == 0 && lane == 0) {
    // ---------------------------------------------------------- TMA producer (unoccupied K first)
    int kit = 0, ti = 0;                               // stages issued, tiles of this CTA
    for (int t = blockIdx.x; t < n_tiles && !*abort_flag; t += gridDim.x, ++ti) {
      const Tile tl = tile_at(t, ti);
      const int zb = p.b_shared ? 0 : tl.z;
      // MODE 2: the stages of the last tile held H and psi_n until its last MMA
      if (MODE == 2 && ti > 0 && !wait_or_abort(done2, (uint32_t)((ti - 1) & 1))) {
        if (!*abort_flag) timed_out(12);
        break;
      }
      for (int it = 0; it < total; ++it, ++kit) {
        const int s = kit % STAGES;
        if (kit >= STAGES && !wait_or_abort(&empty[s], (uint32_t)(((kit / STAGES) & 1) ^ 1))) {
          if (!*abort_flag) timed_out(1);
          break;
        }
        uint8_t* st = smem + s * STAGE_BYTES;
        const int x = it < p.k_un_steps ? p.k_un_x + it * BK : (it - p.k_un_steps) * BK;
        mbar_expect_tx(&full[s], STAGE_BYTES);
        tma_load_3d(st, &mA, &full[s], 2 * x, tl.m0, tl.z);
        tma_load_3d(st + A_BYTES, &mB, &full[s], 2 * x, 2 * tl.n0, zb);
      }
      if (*abort_flag) break;
      if constexpr (MODE == 2) {
        // once every MMA of the G formation has read its stages: the tile's W~, 8 columns (64 bytes a row)
        // per load, each in the place of an H chunk, then its psi_n operand
        if (wait_or_abort(done, (uint32_t)(ti & 1))) {
          mbar_expect_tx(w_full, 16 * H_BYTES);
          for (int k = 0; k < 16; ++k)
            tma_load_3d(w_piece(k >> 3, k & 7), &mW, w_full, 2 * tl.n0 + 16 * k, tl.m0, 0);
          mbar_expect_tx(psi_full, (uint32_t)(16 * p_chunk));
          for (int cc = 0; cc < 8; ++cc) {
            tma_load_3d(p_hi + cc * p_chunk, &mP_hi, psi_full, 2 * tl.n0 + cc * BK, 0, 0);
            tma_load_3d(p_lo + cc * p_chunk, &mP_lo, psi_full, 2 * tl.n0 + cc * BK, 0, 0);
          }
          mbar_wait(w_full, (uint32_t)(ti & 1));      // our copies land before the CTA can exit
          mbar_wait(psi_full, (uint32_t)(ti & 1));
        } else if (!*abort_flag) {
          timed_out(6);
        }
      }
    }
    if (*abort_flag)
      // let our own copies land before the CTA exits
      for (int it = kit - STAGES < 0 ? 0 : kit - STAGES; it < kit; ++it)
        mbar_wait(&full[it % STAGES], (uint32_t)((it / STAGES) & 1));
  } else if (warp == 1 && lane == 0) {
    // ---------------------------------------------------------- MMA issuer
    constexpr uint32_t idesc = make_idesc(FMT, 2 * BNC, BM);
    const int n_blocks = n_un_blocks + (have_occ ? 1 : 0);
    int kit = 0, bc = 0, ti = 0;                       // stages used, accumulation blocks, tiles
    bool ok = true;
    for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++ti) {
      // MODE 2: the last tile's V sums have been read from tensor memory
      if (MODE == 2 && ti > 0 && !wait_or_abort(redbar, (uint32_t)((ti - 1) & 1))) {
        if (!*abort_flag) timed_out(13);
        ok = false;
        break;
      }
      int it = 0;
      for (int c = 0; c < n_blocks && ok; ++c, ++bc) {
        const int b = bc & 1, use = bc >> 1;
        const int first = c < n_un_blocks ? c * CH : p.k_un_steps;
        const int last = c < n_un_blocks ? min(p.k_un_steps, (c + 1) * CH) : total;
        if (use > 0 && !wait_or_abort(&tempty[b], (uint32_t)((use - 1) & 1))) {
          if (!*abort_flag) timed_out(4);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(b * 256);
        for (; it < last; ++it, ++kit) {
          const int s = kit % STAGES;
          if (!wait_or_abort(&full[s], (uint32_t)((kit / STAGES) & 1))) {
            if (!*abort_flag) timed_out(2);
            ok = false;
            break;
          }
          tc_fence_after();
          uint8_t* st = smem + s * STAGE_BYTES;
          const uint64_t ah = sw128_desc(st), al = ah + (64 >> 4);      // lo: 64 bytes along the row
          const uint64_t bh = sw128_desc(st + A_BYTES), bl = bh + (64 >> 4);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            const uint64_t off = (uint64_t)(kk * 32) >> 4;    // 16 elements = 32 bytes along K
            umma(d, ah + off, bh + off, idesc, (it > first || kk > 0) ? 1u : 0u);
            umma(d, ah + off, bl + off, idesc, 1u);
            umma(d, al + off, bh + off, idesc, 1u);
          }
          umma_commit(&empty[s]);
        }
        if (ok) umma_commit(&tfull[b]);
      }
      if constexpr (MODE == 2) {
        umma_commit(done);     // arrives once every MMA issued above has completed
        // V accumulators [occ][half] of np columns each in the half that G_occ does not hold (the last
        // G_unocc block's, drained before the epilogue signals hready)
        const uint32_t vbase = tmem + (uint32_t)((bc & 1) * 256);
        const uint32_t idesc2 = make_idesc(FMT, p.np, BM);
        bool go = ok && wait_or_abort(psi_full, (uint32_t)(ti & 1));
        if (!go && !*abort_flag) timed_out(7);
        for (int o = 0; o < 2 && go; ++o) {
          for (int h = 0; h < 2 && go; ++h) {
            if (!wait_or_abort(&hready[h], (uint32_t)o)) {
              if (!*abort_flag) timed_out(8);
              go = false;
              break;
            }
            tc_fence_after();
            const uint32_t d = vbase + (uint32_t)((2 * o + h) * p.np);
#pragma unroll 1
            for (int cc = 4 * h; cc < 4 * h + 4; ++cc) {
              const uint64_t ah = sw64_desc(h_hi + cc * H_BYTES), al = sw64_desc(h_lo + cc * H_BYTES);
              const uint64_t bh = sw64_desc(p_hi + cc * p_chunk), bl = sw64_desc(p_lo + cc * p_chunk);
#pragma unroll
              for (int kk = 0; kk < BK / 16; ++kk) {
                const uint64_t off = (uint64_t)(kk * 32) >> 4;
                umma(d, ah + off, bh + off, idesc2, (cc > 4 * h || kk > 0) ? 1u : 0u);
                umma(d, ah + off, bl + off, idesc2, 1u);
                umma(d, al + off, bh + off, idesc2, 1u);
              }
            }
            umma_commit(o == 0 ? &hfree[h] : &vready[h]);
          }
        }
        ok = ok && go;
        umma_commit(done2);
      }
    }
    umma_commit(last_mma);     // every MMA of this CTA has completed before tensor memory is freed
    if (!mbar_wait(last_mma, 0)) timed_out(5);
  } else if (warp >= 2) {
    // ---------------------------------------------------------- epilogue
    constexpr int CW = 1024 / EW;                 // real columns of a warp
    constexpr int NC = CW / 2;                    // complex columns
    const int ew = warp - 2;
    const int q = warp & 3;                       // tensor-memory lane quarter of this warp
    const int cg = ew >> 2;                       // column group: complex columns cg*NC .. of the tile
    const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
    const int row = q * 32 + lane;                // tensor-memory lane = tile row
    const int swz = (row >> 1) & 3;               // 64-byte swizzle key of the row
    int bc = 0, ti = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++ti) {
      const Tile tl = tile_at(t, ti);
      const int m0 = tl.m0, n0 = tl.n0;
      const int c0 = n0 + cg * NC;                  // first complex column of this warp
      const int grow0 = p.r0 + m0;                  // grid row of the tile's first row
      const int dr = grow0 + row - c0;              // column (from c0) of this row's diagonal element
      if (MODE == 2 && p.ldw % 2 == 0 && (reinterpret_cast<uintptr_t>(p.wrr) & 15) == 0) {
        // this warp's block of W~ on its way into L2 while the K loop runs
        const int gr = m0 + row;
        const int bytes = gr < p.m_rows ? min(NC, p.n_cols - c0) * 8 & ~15 : 0;
        if (bytes > 0) prefetch_l2(p.wrr + (long)gr * p.ldw + c0, bytes);
      }
      float tot[CW];                                // this thread's part of its row of G_unocc, FP32 round-to-nearest sums
#pragma unroll
      for (int i = 0; i < CW; ++i) tot[i] = 0.f;
      for (int c = 0; c < n_un_blocks; ++c, ++bc) {
        const int b = bc & 1;
        const bool got = wait_or_abort(&tfull[b], (uint32_t)((bc >> 1) & 1));
        if (!__all_sync(0xffffffffu, got)) {
          if (lane == 0 && !*abort_flag) timed_out(3);
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t base = tmem + lane_addr + (uint32_t)(b * 256 + cg * CW);
#pragma unroll
        for (int u = 0; u < CW / 16; ++u) {
          uint32_t x[16];
          tmem_ld16(base + 16 * u, x);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; ++i) tot[16 * u + i] += __uint_as_float(x[i]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[b]);
      }
      const int bo = bc & 1;
      if (ok && have_occ) {
        const bool got = wait_or_abort(&tfull[bo], (uint32_t)((bc >> 1) & 1));
        if (!__all_sync(0xffffffffu, got)) {
          if (lane == 0 && !*abort_flag) timed_out(3);
          ok = false;
        }
        tc_fence_after();
      }
      // tcgen05.ld is warp-collective: the whole warp takes the same branch
      ok = __all_sync(0xffffffffu, ok && !*abort_flag);
      if (ok) {
        const float sc = ldexpf(1.0f, -2 * p.dexp[p.b_shared ? 0 : tl.z]);
        const float ao = p.alpha_occ[tl.z] * sc, au = p.alpha_un[tl.z] * sc;
        const uint32_t occ = tmem + lane_addr + (uint32_t)(bo * 256 + cg * CW);
        // the half that G_occ holds may take the next tile's sums
        auto free_occ = [&]() {
          tc_fence_before();
          __syncwarp();
          if (have_occ && lane == 0) mbar_arrive(&tempty[bo]);
        };
        if constexpr (MODE == 2) {
          // ---------------------------------------------- self-energy contraction of the tile
          const bool rvalid = m0 + row < p.m_rows;
          const int h = cg;                             // the warp's column half
          const long grow = grow0 + row;                // grid row r of this thread
          bool fine = wait_or_abort(w_full, (uint32_t)(ti & 1));
          ok = __all_sync(0xffffffffu, fine);
          if (!ok) {
            if (lane == 0 && !*abort_flag) timed_out(14);
            break;
          }
          // H = w G o W~ for G_unocc in registers and for G_occ in tensor memory (in place); returns the
          // powers of two that put the rows' maxima below 2^15
          float mu = 0.f, mo = 0.f;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint8_t* wp = w_piece(h, k) + row * 64;
#pragma unroll
            for (int hs = 0; hs < 2; ++hs) {
              uint32_t x[8];
              tmem_ld8(occ + 16 * k + 8 * hs, x);
              float4 w2[2];
#pragma unroll
              for (int s = 0; s < 2; ++s) w2[s] = *reinterpret_cast<const float4*>(wp + (((2 * hs + s) ^ swz) << 4));
              tmem_wait_ld();
#pragma unroll
              for (int s = 0; s < 2; ++s) {
                const float4 w = w2[s];
                const int c = 8 * k + 4 * hs + 2 * s;
                // weight of (r, R'): 2 below the diagonal, 1 on it, 0 above (lower-triangle mode)
                float wa = 1.f, wb = 1.f;
                if (p.lower) {
                  wa = c < dr ? 2.f : (c == dr ? 1.f : 0.f);
                  wb = c + 1 < dr ? 2.f : (c + 1 == dr ? 1.f : 0.f);
                }
                {
                  const float ar = tot[2 * c] * au * wa, ai = tot[2 * c + 1] * au * wa;
                  const float br = tot[2 * c + 2] * au * wb, bi = tot[2 * c + 3] * au * wb;
                  tot[2 * c] = ar * w.x - ai * w.y;
                  tot[2 * c + 1] = ar * w.y + ai * w.x;
                  tot[2 * c + 2] = br * w.z - bi * w.w;
                  tot[2 * c + 3] = br * w.w + bi * w.z;
                  mu = fmaxf(mu, fmaxf(fmaxf(fabsf(tot[2 * c]), fabsf(tot[2 * c + 1])),
                                       fmaxf(fabsf(tot[2 * c + 2]), fabsf(tot[2 * c + 3]))));
                }
                {
                  const float g0 = __uint_as_float(x[4 * s]), g1 = __uint_as_float(x[4 * s + 1]);
                  const float g2 = __uint_as_float(x[4 * s + 2]), g3 = __uint_as_float(x[4 * s + 3]);
                  const float ar = g0 * ao * wa, ai = g1 * ao * wa;
                  const float br = g2 * ao * wb, bi = g3 * ao * wb;
                  const float y0 = ar * w.x - ai * w.y, y1 = ar * w.y + ai * w.x;
                  const float y2 = br * w.z - bi * w.w, y3 = br * w.w + bi * w.z;
                  mo = fmaxf(mo, fmaxf(fmaxf(fabsf(y0), fabsf(y1)), fmaxf(fabsf(y2), fabsf(y3))));
                  x[4 * s] = __float_as_uint(y0);
                  x[4 * s + 1] = __float_as_uint(y1);
                  x[4 * s + 2] = __float_as_uint(y2);
                  x[4 * s + 3] = __float_as_uint(y3);
                }
              }
              tmem_st8(occ + 16 * k + 8 * hs, x);
            }
          }
          tmem_wait_st();
          auto exponent = [](float m) -> int {
            int ex = 0;
            if (m > 0.f) frexpf(m, &ex);
            return m > 0.f ? 14 - ex : 0;
          };
          // this row of H, scaled by 2^sh and split in two 16-bit parts, into K chunks
          // 4h..4h+3: row `row` of a chunk is 64 bytes at (row/8)*512 + (row%8)*64, its
          // 16-byte segment s stored at s ^ ((row/2) % 4) (the 64-byte swizzle of TMA)
          auto store_h = [&](int sh) {
            // 2^sh in two factors: a row of tiny H (W~ of a large tau decays like exp(-omega tau))
            // can need sh above 127, where one FP32 power of two would overflow
            const float s1 = ldexpf(1.0f, sh >> 1), s2 = ldexpf(1.0f, sh - (sh >> 1));
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int base = (4 * h + j) * H_BYTES + (row >> 3) * 512 + (row & 7) * 64;
#pragma unroll
              for (int sg = 0; sg < 4; ++sg) {
                uint32_t hw[4], lw[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                  const int c = 16 * j + 4 * sg + t;
                  split2<FMT>(tot[2 * c] * s1 * s2, tot[2 * c + 1] * s1 * s2, hw[t], lw[t]);
                }
                const int off = base + ((sg ^ swz) << 4);
                *reinterpret_cast<uint4*>(h_hi + off) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                *reinterpret_cast<uint4*>(h_lo + off) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
              }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // visible to the tensor cores
            __syncwarp();
          };
          const int shu = exponent(mu), sho = exponent(mo);
          store_h(shu);
          if (lane == 0) mbar_arrive(&hready[h]);
          // H_occ of this row and half from tensor memory
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            uint32_t x[16];
            tmem_ld16(occ + 16 * u, x);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) tot[16 * u + i] = __uint_as_float(x[i]);
          }
          free_occ();
          fine = wait_or_abort(&hfree[h], (uint32_t)(ti & 1));   // the unoccupied MMAs have read this half
          if (__all_sync(0xffffffffu, fine)) {
            tc_fence_after();
            store_h(sho);
            if (lane == 0) mbar_arrive(&hready[h]);
            fine = wait_or_abort(&vready[h], (uint32_t)(ti & 1));
          }
          if (__all_sync(0xffffffffu, fine)) {
            tc_fence_after();
            const uint32_t vb = tmem + lane_addr + (uint32_t)((1 - bo) * 256);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              if (16 * u < p.np) {                      // np is the same for the whole warp
                uint32_t x[16], y[16];
                tmem_ld16(vb + (uint32_t)(h * p.np + 16 * u), x);
                tmem_ld16(vb + (uint32_t)((2 + h) * p.np + 16 * u), y);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                  tot[16 * u + i] = __uint_as_float(x[i]);
                  tot[64 + 16 * u + i] = __uint_as_float(y[i]);
                }
              }
            }
            // 2^-(sh + e) in two factors as well, applied one after the other, so that the
            // tiny rows come back as normal FP32 numbers where they are representable
            const int e = p.dexp[0], ku = shu + e, ko = sho + e;
            const float fu1 = ldexpf(1.0f, -(ku >> 1)), fu2 = ldexpf(1.0f, -(ku - (ku >> 1)));
            const float fo1 = ldexpf(1.0f, -(ko >> 1)), fo2 = ldexpf(1.0f, -(ko - (ko >> 1)));
            // Re(conj(psi_n) V_n) of the row for NB >= n_n bands, then the sums over the warp's rows: at
            // each of the five exchange steps a lane keeps half of its sums and hands over the other
            // half, so that 62 shuffles leave lane l with sums l-th of 2 NB (the pairs added are those
            // of a butterfly over each sum)
            const int my_band = lane < p.n_n ? __ldg(p.bands + lane) : 0;
            tc_fence_before();                          // V is read: the next tile may sum over it (redbar)
            auto bands = [&](auto nb_c) {
              constexpr int NB = decltype(nb_c)::value;
#pragma unroll
              for (int b0 = 0; b0 < NB; b0 += 8) {
                float2 ps[8];
#pragma unroll
                for (int i = 0; i < 8 && b0 + i < NB; ++i) {
                  const int n = b0 + i;
                  const long at = (long)__shfl_sync(0xffffffffu, my_band, n) * p.ldpsi + grow;
                  ps[i] = rvalid && n < p.n_n ? __ldg(p.psi + at) : make_float2(0.f, 0.f);
                }
#pragma unroll
                for (int i = 0; i < 8 && b0 + i < NB; ++i) {
                  const int n = b0 + i;
                  const float su = (ps[i].x * tot[2 * n] + ps[i].y * tot[2 * n + 1]) * fu1 * fu2;
                  const float so = (ps[i].x * tot[64 + 2 * n] + ps[i].y * tot[64 + 2 * n + 1]) * fo1 * fo2;
                  tot[2 * n] = su;
                  tot[2 * n + 1] = so;
                }
              }
              int nv = 2 * NB;
#pragma unroll
              for (int off = 16; off > 0; off >>= 1) {
                if (nv > 1) {
                  nv >>= 1;
                  const bool up = (lane & off) != 0;
#pragma unroll
                  for (int i = 0; i < NB; ++i)
                    if (i < nv) {
                      const float keep = up ? tot[i + nv] : tot[i], send = up ? tot[i] : tot[i + nv];
                      tot[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
                    }
                } else {
                  tot[0] += __shfl_xor_sync(0xffffffffu, tot[0], off);
                }
              }
              // lane l: sums (l * 2 NB) / 32 .. of [su_0, so_0, su_1, ...]
              float* rw = red + ew * 64;
              if (NB == 32) {
                rw[2 * lane] = tot[0];
                rw[2 * lane + 1] = tot[1];
              } else if (lane % (NB < 16 ? 16 / NB : 1) == 0) {
                rw[lane * NB / 16] = tot[0];
              }
            };
            if (p.n_n <= 4) bands(std::integral_constant<int, 4>{});
            else if (p.n_n <= 8) bands(std::integral_constant<int, 8>{});
            else if (p.n_n <= 16) bands(std::integral_constant<int, 16>{});
            else bands(std::integral_constant<int, 32>{});
            __syncwarp();
            if (lane == 0) mbar_arrive(redbar);
          } else {
            if (lane == 0 && !*abort_flag) timed_out(10);
            ok = false;
          }
          // one warp adds the CTA's band sums into Sigma_unocc_nn(tau_j), Sigma_occ_nn(-tau_j)
          if (ew == 0) {
            const bool got = wait_or_abort(redbar, (uint32_t)(ti & 1));
            if (got && lane < p.n_n) {
              double su = 0.0, so = 0.0;
#pragma unroll
              for (int w = 0; w < EW; ++w) {
                su += (double)red[w * 64 + 2 * lane];
                so += (double)red[w * 64 + 2 * lane + 1];
              }
              atomicAdd(&p.acc_u[(long)lane * p.acc_stride], p.coef * su);
              atomicAdd(&p.acc_o[(long)lane * p.acc_stride], -p.coef * so);
            } else if (!got && lane == 0 && !*abort_flag) {
              timed_out(11);
            }
          }
        } else {
          // MODE 0 forms chi over G_unocc in registers at once, which frees G_occ's tensor memory: the
          // MMAs of the next tile run while this one is written.  MODE 1 writes G_occ first.
          if (MODE == 0) {
            const bool diag_tile = p.lower && n0 + BNC > grow0;   // the tile meets the diagonal
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              uint32_t ro[16];
              if (have_occ) {
                tmem_ld16(occ + 16 * u, ro);
                tmem_wait_ld();
              } else {
#pragma unroll
                for (int i = 0; i < 16; ++i) ro[i] = 0u;
              }
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const float gor = __uint_as_float(ro[2 * j]) * ao, goi = __uint_as_float(ro[2 * j + 1]) * ao;
                const float gur = tot[16 * u + 2 * j] * au, gui = tot[16 * u + 2 * j + 1] * au;
                float2 v = make_float2(-2.0f * (gor * gur + goi * gui), -2.0f * (goi * gur - gor * gui));
                if (diag_tile) {
                  const float f = 8 * u + j < dr ? 1.f : (8 * u + j == dr ? 0.5f : 0.f);
                  v.x *= f;
                  v.y *= f;
                }
                tot[16 * u + 2 * j] = v.x;
                tot[16 * u + 2 * j + 1] = v.y;
              }
            }
            free_occ();
          }
          // 32 rows x 8 columns at a time through shared memory as pairs of columns (pair s of row r at
          // s ^ (r/2) % 4), then 64-byte row segments out
          float4* stg = reinterpret_cast<float4*>(epi + ew * 32 * EPI_COLS);
          float4* const st_w = stg + lane * 4;                               // this lane's row
          const int rrow = lane >> 2, rpair = lane & 3;                      // written out: row rrow + 8 i
          const float4* const st_r = stg + rrow * 4 + (rpair ^ (rrow >> 1 & 3));
#pragma unroll
          for (int pass = 0; pass < (MODE == 0 ? 1 : 2); ++pass) {
            const int ldo = (int)p.ldo;
            float2* outp = (MODE == 0 || pass == 0 ? p.out0 : p.out1) + tl.z * p.so + (long)(m0 + q * 32) * ldo + c0 +
                           rrow * ldo + rpair * 2;
            const int rows_left = p.m_rows - m0 - q * 32 - rrow, cols_left = p.n_cols - c0 - rpair * 2;
            const bool vec = (ldo & 1) == 0 && (reinterpret_cast<uintptr_t>(outp) & 15) == 0;
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
              uint32_t ro[16];
              if (MODE == 1 && pass == 0) {
                if (have_occ) {
                  tmem_ld16(occ + 16 * cc, ro);
                  tmem_wait_ld();
                } else {
#pragma unroll
                  for (int i = 0; i < 16; ++i) ro[i] = 0u;
                }
              }
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                float4 v;
                if (MODE == 1 && pass == 0)
                  v = make_float4(__uint_as_float(ro[4 * j]) * ao, __uint_as_float(ro[4 * j + 1]) * ao,
                                  __uint_as_float(ro[4 * j + 2]) * ao, __uint_as_float(ro[4 * j + 3]) * ao);
                else {
                  const int c = 16 * cc + 4 * j;
                  const float f = MODE == 0 ? 1.f : au;
                  v = make_float4(tot[c] * f, tot[c + 1] * f, tot[c + 2] * f, tot[c + 3] * f);
                }
                st_w[j ^ swz] = v;
              }
              __syncwarp();
              float2* o = outp + 8 * cc;
#pragma unroll
              for (int i = 0; i < 4; ++i, o += 8 * ldo) {
                if (8 * i >= rows_left || 8 * cc >= cols_left) continue;
                const float4 v = st_r[8 * i * 4];
                if (vec && 8 * cc + 1 < cols_left) {
                  *reinterpret_cast<float4*>(o) = v;
                } else {
                  o[0] = make_float2(v.x, v.y);
                  if (8 * cc + 1 < cols_left) o[1] = make_float2(v.z, v.w);
                }
              }
              __syncwarp();
            }
            if (MODE == 1 && pass == 0) free_occ();
          }
        }
      }
      if (have_occ) ++bc;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// ---------------------------------------------------------------------- operand preparation

// max |component| of the n elements of entry blockIdx.y (stride sx)
__global__ void maxabs_kernel(const float2* __restrict__ x, size_t n, long sx, unsigned int* __restrict__ out) {
  x += blockIdx.y * sx;
  out += blockIdx.y;
  float m = 0.f;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    m = fmaxf(m, fmaxf(fabsf(x[i].x), fabsf(x[i].y)));
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));   // non-negative floats order as uints
}

// e such that max|x| * 2^e lies in [2^14, 2^15), one thread per entry
__global__ void exponent_kernel(const unsigned int* __restrict__ maxbits, int* __restrict__ e) {
  const float m = __uint_as_float(maxbits[threadIdx.x]);
  int ex = 0;
  if (m > 0.f) {
    frexpf(m, &ex);        // m = f * 2^ex, f in [0.5, 1)
    e[threadIdx.x] = 15 - ex;
  } else {
    e[threadIdx.x] = 0;
  }
}

// Operand rows from psi [N_b][N_r] (band-major), transposed to K-major through a
// 32 x 32 shared tile.  Band k goes to real column kcol(k) = 2k (occupied) or
// k_un_x + 2(k - n_occ) (unoccupied); padding columns are written as zero.
//  A: row r (rows r0..r0+rows-1):  (ar, ai) * s_k * 2^e
//  B: rows 2R', 2R'+1:             (br, -bi) and (bi, br) of conj(psi) * 2^e
// Entry blockIdx.z: orbitals sx elements apart, its own factors s_k, scaling (unless
// e_shared) and operand.
template <bool IS_B, uint32_t FMT>
__global__ void __launch_bounds__(256) prep_kernel(const float2* __restrict__ psi, int n_b, int n_occ, int nr, int r0,
                                                   int rows, const float* __restrict__ sk,
                                                   const int* __restrict__ dexp, int k_occ_pad, int k_un_x,
                                                   int kpad, uint16_t* __restrict__ op, long sx, int e_shared) {
  __shared__ float2 t[32][33];
  const int z = blockIdx.z;
  psi += z * sx;
  sk += (long)z * n_b;
  op += (long)z * (IS_B ? 2 : 1) * rows * 2 * kpad;
  const int kb = blockIdx.y * 32;       // band tile (covers padded band slots)
  const int rb = blockIdx.x * 32;       // row tile
  const float sc = ldexpf(1.0f, dexp[e_shared ? 0 : z]);
  // band slot -> band index (or -1 for padding)
  const int occ_slots = k_occ_pad / 2, un_slots = (kpad - k_un_x) / 2;
  auto band_of = [&](int slot) -> int {
    if (slot < occ_slots) return slot < n_occ ? slot : -1;
    const int u = slot - occ_slots;
    return (u < un_slots && n_occ + u < n_b) ? n_occ + u : -1;
  };
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int band = band_of(kb + i);
    const int r = r0 + rb + threadIdx.x;
    float2 v = make_float2(0.f, 0.f);
    if (band >= 0 && rb + threadIdx.x < rows) {
      v = psi[(long)band * nr + r];
      const float s = IS_B ? sc : sc * sk[band];
      v.x *= s;
      v.y *= s;
    }
    t[i][threadIdx.x] = v;
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int rr = rb + i;
    if (rr >= rows) continue;
    const int slot = kb + threadIdx.x;
    const int col = slot < occ_slots ? 2 * slot : k_un_x + 2 * (slot - occ_slots);
    if (col >= kpad) continue;
    const int at = col / BK * (2 * BK) + col % BK;      // hi of the stage's 32 values, lo 32 further
    const float2 v = t[threadIdx.x][i];
    uint32_t h, l;
    if (!IS_B) {
      split2<FMT>(v.x, v.y, h, l);
      uint16_t* o = op + (long)rr * 2 * kpad + at;
      *reinterpret_cast<uint32_t*>(o) = h;
      *reinterpret_cast<uint32_t*>(o + BK) = l;
    } else {
      // b = conj(psi): br = v.x, bi = -v.y;  row 2R': (br, -bi) = (v.x, v.y); row 2R'+1: (bi, br) = (-v.y, v.x)
      split2<FMT>(v.x, v.y, h, l);
      uint16_t* o = op + (long)(2 * rr) * 2 * kpad + at;
      *reinterpret_cast<uint32_t*>(o) = h;
      *reinterpret_cast<uint32_t*>(o + BK) = l;
      split2<FMT>(-v.y, v.x, h, l);
      o += 2 * kpad;
      *reinterpret_cast<uint32_t*>(o) = h;
      *reinterpret_cast<uint32_t*>(o + BK) = l;
    }
  }
}

// The psi_n operand of the self-energy contraction (MODE 2): B rows 2n and 2n+1
// hold (br, -bi) and (bi, br) of b = psi_{bands[n]}(R') * 2^e along real K =
// 2R', 2R'+1, so that D[r][2n + c] = (Re, Im) sum_R' H(r,R') psi_n(R').  Rows of
// band slots n >= n_n (up to np/2) are zero.  One thread per (R', n).
template <uint32_t FMT>
__global__ void __launch_bounds__(256) prep_psin_kernel(const float2* __restrict__ psi, int nr,
                                                        const int* __restrict__ bands, int n_n, int kp,
                                                        const int* __restrict__ dexp, uint16_t* __restrict__ hi,
                                                        uint16_t* __restrict__ lo) {
  const int rp = blockIdx.x * 256 + threadIdx.x;
  const int n = blockIdx.y;
  if (2 * rp >= kp) return;
  float2 v = make_float2(0.f, 0.f);
  if (n < n_n && rp < nr) {
    v = psi[(long)bands[n] * nr + rp];
    const float sc = ldexpf(1.0f, *dexp);
    v.x *= sc;
    v.y *= sc;
  }
  uint16_t h0, l0, h1, l1, h2, l2;
  split<FMT>(v.x, h0, l0);
  split<FMT>(-v.y, h1, l1);
  split<FMT>(v.y, h2, l2);
  const long o0 = (long)(2 * n) * kp + 2 * rp, o1 = o0 + kp;
  reinterpret_cast<uint32_t*>(hi + o0)[0] = (uint32_t)h0 | ((uint32_t)h1 << 16);
  reinterpret_cast<uint32_t*>(lo + o0)[0] = (uint32_t)l0 | ((uint32_t)l1 << 16);
  reinterpret_cast<uint32_t*>(hi + o1)[0] = (uint32_t)h2 | ((uint32_t)h0 << 16);
  reinterpret_cast<uint32_t*>(lo + o1)[0] = (uint32_t)l2 | ((uint32_t)l0 << 16);
}

// ---------------------------------------------------------------------- host side

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeFn encoder(gw_ctx* ctx, gw_status* st) {
  static std::mutex mu;
  static EncodeFn fn = nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !p) {
      *st = fail(ctx, GW_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
      return nullptr;
    }
    fn = reinterpret_cast<EncodeFn>(p);
  }
  *st = GW_OK;
  return fn;
}

}  // namespace tc

gw_status tc_make_map3(gw_ctx* ctx, CUtensorMap* m, const void* base, int kpad, long rows, int batch, int box_rows,
                       uint32_t fmt, int box_k) {
  using namespace tc;
  gw_status st;
  EncodeFn enc = encoder(ctx, &st);
  if (!enc) return st;
  cuuint64_t dims[3] = {(cuuint64_t)kpad, (cuuint64_t)rows, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)kpad * 2, (cuuint64_t)kpad * 2 * (cuuint64_t)rows};
  cuuint32_t box[3] = {(cuuint32_t)box_k, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  if (box_k != 64 && box_k != 32) return fail(ctx, GW_ERR_ARG, "TMA box along K must be 32 or 64 elements");
  CUresult r = enc(m, fmt == 0 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
                   const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   box_k == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(ctx, GW_ERR_CUDA, "cuTensorMapEncodeTiled (3-D) failed (" + std::to_string((int)r) + ")");
  return GW_OK;
}

namespace tc {

// Map over W~ rows [rows][ldw] as FP32 pairs, box 8 complex x 128 rows, 64-byte swizzle; what lies
// past the grid or the block reads as zero.
static gw_status w_map(gw_ctx* ctx, CUtensorMap* m, const float2* base, int nr, long ldw, int rows) {
  gw_status st;
  EncodeFn enc = encoder(ctx, &st);
  if (!enc) return st;
  if (ldw % 2 || reinterpret_cast<uintptr_t>(base) % 16)
    return fail(ctx, GW_ERR_UNSUPPORTED, "fused self-energy: W~ rows must be 16-byte aligned");
  cuuint64_t dims[3] = {(cuuint64_t)2 * nr, (cuuint64_t)rows, 1};
  cuuint64_t strides[2] = {(cuuint64_t)ldw * 8, (cuuint64_t)ldw * 8 * (cuuint64_t)rows};
  cuuint32_t box[3] = {16, BM, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float2*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(ctx, GW_ERR_CUDA, "cuTensorMapEncodeTiled (W~) failed (" + std::to_string((int)r) + ")");
  return GW_OK;
}

struct Layout {
  int k_occ_pad, k_un_pad, k_un_x, kpad;
};
static Layout layout(int n_b, int n_occ) {
  Layout L;
  L.k_occ_pad = (2 * n_occ + BK - 1) / BK * BK;
  L.k_un_pad = (2 * (n_b - n_occ) + BK - 1) / BK * BK;
  L.k_un_x = L.k_occ_pad;
  L.kpad = L.k_occ_pad + L.k_un_pad;
  return L;
}

// MMA N of the self-energy contraction for n_sig bands, and the padded real K of its operand
static int sig_np(int n_sig) { return (2 * n_sig + 15) / 16 * 16; }
static int sig_kp(const GridInfo& g) { return (2 * g.nr + BK - 1) / BK * BK; }

// Words at the start of the scratch: [2..3] time-out status, then the entries' maxima and exponents.
constexpr int kWords = 64 + 2 * kMaxEntries;

static size_t scratch_bytes(const GridInfo& g, int n_b, int n_occ, int n_rows, bool with_tmp, int n_sig, int nb,
                            bool b_shared) {
  const Layout L = layout(n_b, n_occ);
  const size_t nbb = b_shared ? 1 : nb;
  Carver probe(nullptr);
  probe.take<unsigned int>(kWords);
  probe.take<uint16_t>(nbb * 2 * g.nr * 2 * L.kpad);
  if (n_sig > 0) {
    probe.take<uint16_t>((size_t)sig_np(n_sig) * sig_kp(g));
    probe.take<uint16_t>((size_t)sig_np(n_sig) * sig_kp(g));
  }
  probe.take<float>((size_t)nb * n_b);
  probe.take<uint16_t>((size_t)nb * n_rows * 2 * L.kpad);
  if (with_tmp) probe.take<float2>((size_t)n_rows * g.nr);
  return Carver::round(probe.off);
}

static int* status_words(void* scratch) { return static_cast<int*>(scratch) + 2; }

// One G/chi formation for rows r0 .. r0+n_rows-1 using `scratch` (of at least
// scratch_bytes()).  mode 0: chi into out0; mode 1: G_occ into out0 and G_unocc
// into out1 (a NULL one goes to scratch).  prep_b = false reuses the B operand
// and the operand scaling left in the same scratch by an earlier call for the
// same psi.
static gw_status run(gw_ctx* ctx, const GridInfo& g, int n_b, int n_occ, const void* psi, const GreenScales* gs,
                     int r0, int n_rows, gw_prec prec, int mode, void* out0, void* out1, void* scratch, bool prep_b,
                     cudaStream_t st, const float* sk_dev = nullptr, int* status_dev = nullptr,
                     const TcSigma* sig = nullptr, bool lower = false, const TcEntries& en = TcEntries{}) {
  const uint32_t fmt = prec == GW_BF16X3 ? 1u : 0u;
  const Layout L = layout(n_b, n_occ);
  gw_status rc;
  const int nb = en.n;
  const bool b_shared = en.psi_stride == 0;
  const size_t nbb = b_shared ? 1 : nb;
  if (nb < 1 || nb > kMaxEntries) return fail(ctx, GW_ERR_SHAPE, "1 to 64 entries per G formation");
  const bool need_tmp = mode == 1 && (!out0 || !out1);
  Carver cv(scratch);
  unsigned int* words = cv.take<unsigned int>(kWords);
  unsigned int* dmax = words + 64;
  int* dexp = reinterpret_cast<int*>(words + 64 + kMaxEntries);
  // time-out status: in the scratch, or in a word the caller owns (kept past later uses of the scratch)
  int* status = status_dev ? status_dev : status_words(scratch);
  uint16_t* bop = cv.take<uint16_t>(nbb * 2 * g.nr * 2 * L.kpad);
  // these operands are prepared by the first call and read by later ones: their place must not
  // depend on this call's number of rows or entries, so they come before what does
  const int np = mode == 2 ? sig_np(sig->n_n) : 0, kps = sig_kp(g);
  uint16_t* phi = mode == 2 ? cv.take<uint16_t>((size_t)np * kps) : nullptr;
  uint16_t* plo = mode == 2 ? cv.take<uint16_t>((size_t)np * kps) : nullptr;
  float* dsk = cv.take<float>((size_t)nb * n_b);
  uint16_t* aop = cv.take<uint16_t>((size_t)nb * n_rows * 2 * L.kpad);
  float2* tmp = need_tmp ? cv.take<float2>((size_t)n_rows * g.nr) : nullptr;
  if (mode == 1) {
    if (!out0) out0 = tmp;
    if (!out1) out1 = tmp;
  }
  // per-band factors: uploaded here, or already on the device (sk_dev: no host-to-device copy in this call)
  const float* sk = sk_dev;
  if (!sk) {
    std::vector<float> skf;
    for (int z = 0; z < nb; ++z) skf.insert(skf.end(), gs[z].s.begin(), gs[z].s.end());
    if ((rc = upload(ctx, dsk, skf.data(), sizeof(float) * skf.size(), st))) return rc;
    sk = dsk;
  }
  const dim3 tb(32, 8);
  const int slots = L.kpad / 2;
  if (prep_b) {
    if ((rc = cuda_check(ctx, cudaMemsetAsync(dmax, 0, nbb * sizeof(unsigned int), st), "memset"))) return rc;
    const size_t nel = (size_t)n_b * g.nr;
    maxabs_kernel<<<dim3((unsigned)std::min<size_t>((nel + 255) / 256, (size_t)ctx->num_sms * 8 / nbb + 1), nbb), 256, 0,
                    st>>>(static_cast<const float2*>(psi), nel, en.psi_stride, dmax);
    if ((rc = launch_check(ctx, "maxabs_kernel"))) return rc;
    exponent_kernel<<<1, (unsigned)nbb, 0, st>>>(dmax, dexp);
    if ((rc = launch_check(ctx, "exponent_kernel"))) return rc;
    const dim3 gbB((g.nr + 31) / 32, (slots + 31) / 32, nbb);
    if (fmt == 0)
      prep_kernel<true, 0><<<gbB, tb, 0, st>>>((const float2*)psi, n_b, n_occ, g.nr, 0, g.nr, sk, dexp,
                                                L.k_occ_pad, L.k_un_x, L.kpad, bop, en.psi_stride, b_shared);
    else
      prep_kernel<true, 1><<<gbB, tb, 0, st>>>((const float2*)psi, n_b, n_occ, g.nr, 0, g.nr, sk, dexp,
                                                L.k_occ_pad, L.k_un_x, L.kpad, bop, en.psi_stride, b_shared);
    if ((rc = launch_check(ctx, "prep_kernel(B)"))) return rc;
    if (mode == 2) {
      const dim3 gp((kps / 2 + 255) / 256, np / 2);
      if (fmt == 0)
        prep_psin_kernel<0><<<gp, 256, 0, st>>>((const float2*)psi, g.nr, sig->bands, sig->n_n, kps, dexp, phi, plo);
      else
        prep_psin_kernel<1><<<gp, 256, 0, st>>>((const float2*)psi, g.nr, sig->bands, sig->n_n, kps, dexp, phi, plo);
      if ((rc = launch_check(ctx, "prep_psin_kernel"))) return rc;
    }
  }
  const dim3 gbA((n_rows + 31) / 32, (slots + 31) / 32, nb);
  if (fmt == 0)
    prep_kernel<false, 0><<<gbA, tb, 0, st>>>((const float2*)psi, n_b, n_occ, g.nr, r0, n_rows, sk, dexp,
                                               L.k_occ_pad, L.k_un_x, L.kpad, aop, en.psi_stride, b_shared);
  else
    prep_kernel<false, 1><<<gbA, tb, 0, st>>>((const float2*)psi, n_b, n_occ, g.nr, r0, n_rows, sk, dexp,
                                               L.k_occ_pad, L.k_un_x, L.kpad, aop, en.psi_stride, b_shared);
  if ((rc = launch_check(ctx, "prep_kernel(A)"))) return rc;
  CUtensorMap ma, mb, mph, mpl, mw;
  if ((rc = tc_make_map3(ctx, &ma, aop, 2 * L.kpad, n_rows, nb, BM, fmt, 2 * BK))) return rc;
  if ((rc = tc_make_map3(ctx, &mb, bop, 2 * L.kpad, 2L * g.nr, (int)nbb, 2 * BNC, fmt, 2 * BK))) return rc;
  if (mode == 2) {
    if ((rc = tc_make_map3(ctx, &mph, phi, kps, np, 1, np, fmt, BK))) return rc;
    if ((rc = tc_make_map3(ctx, &mpl, plo, kps, np, 1, np, fmt, BK))) return rc;
    if ((rc = w_map(ctx, &mw, sig->wrr, g.nr, sig->ldw, n_rows))) return rc;
  } else {
    mph = ma;                                    // unused outside the self-energy mode
    mpl = ma;
    mw = ma;
  }
  Params P;
  P.m_rows = n_rows;
  P.n_cols = g.nr;
  P.k_occ_steps = L.k_occ_pad / BK;
  P.k_un_steps = L.k_un_pad / BK;
  P.k_un_x = L.k_un_x;
  P.out0 = static_cast<float2*>(out0);
  P.out1 = static_cast<float2*>(mode == 1 ? out1 : out0);
  P.ldo = g.nr;
  for (int z = 0; z < nb; ++z) {
    P.alpha_occ[z] = (float)gs[z].amax_occ;
    P.alpha_un[z] = (float)gs[z].amax_unocc;
  }
  P.nb = nb;
  P.b_shared = b_shared ? 1 : 0;
  P.so = en.out_stride;
  P.dexp = dexp;
  P.status = status;
  P.wrr = nullptr;
  P.ldw = 0;
  P.psi = static_cast<const float2*>(psi);
  P.ldpsi = g.nr;
  P.bands = nullptr;
  P.n_n = 0;
  P.np = np;
  P.r0 = r0;
  P.coef = 0.0;
  P.acc_u = P.acc_o = nullptr;
  P.acc_stride = 0;
  P.lower = (mode != 1 && lower) ? 1 : 0;
  if (mode == 2) {
    P.wrr = sig->wrr;
    P.ldw = sig->ldw;
    P.bands = sig->bands;
    P.n_n = sig->n_n;
    P.coef = sig->coef;
    P.acc_u = sig->acc_u;
    P.acc_o = sig->acc_o;
    P.acc_stride = sig->acc_stride;
  }
  // tiles per entry: all, or those meeting R' <= r
  P.gx = (g.nr + BNC - 1) / BNC;
  P.gy = (n_rows + BM - 1) / BM;
  P.tiles = 0;
  for (int i = 0; i < P.gy; ++i) P.tiles += P.lower ? std::min(P.gx, (r0 + i * BM + BM - 1) / BNC + 1) : P.gx;
  const double tile_frac = nb * (double)P.tiles / ((double)P.gx * P.gy);
  // persistent: one CTA per SM walks the tiles, so that the TMA loads and MMAs of a tile start while the
  // last one's epilogue runs (modes 0 and 1) and no tile pays for a CTA's set-up
  const unsigned grid = (unsigned)std::min<long>((long)P.tiles * nb, ctx->num_sms);
  const int threads = mode == 2 ? kThreads<2> : kThreads<0>;
  auto go = [&](auto kernel) -> gw_status {
    gw_status r = cuda_check(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES),
                             "cudaFuncSetAttribute");
    if (r) return r;
    const double work =
        tile_frac * (8.0 * n_rows * (double)g.nr * n_b + (mode == 2 ? 16.0 * n_rows * (double)g.nr * P.n_n : 0.0));
    KTimer kt(ctx, KF_GREEN_TC, work, st);
    kernel<<<grid, threads, SMEM_BYTES, st>>>(ma, mb, mph, mpl, mw, P);
    return launch_check(ctx, "green_tc_kernel");
  };
  if (mode == 0) rc = fmt == 0 ? go(green_tc_kernel<0, 0>) : go(green_tc_kernel<0, 1>);
  else if (mode == 1) rc = fmt == 0 ? go(green_tc_kernel<1, 0>) : go(green_tc_kernel<1, 1>);
  else rc = fmt == 0 ? go(green_tc_kernel<2, 0>) : go(green_tc_kernel<2, 1>);
  if (!rc && ctx->inject_timeout > 0 && --ctx->inject_timeout == 0)
    rc = cuda_check(ctx, cudaMemsetAsync(status, 1, 2 * sizeof(int), st), "memset");
  return rc;
}

// Reads the status word the kernels' bounded waits write (synchronises the stream).
static gw_status check_status(gw_ctx* ctx, void* scratch, cudaStream_t st) {
  int hs[2] = {0, 0};
  const int* status = status_words(scratch);
  gw_status rc;
  if ((rc = cuda_check(ctx, cudaMemcpyAsync(hs, status, sizeof(hs), cudaMemcpyDeviceToHost, st), "status"))) return rc;
  if ((rc = cuda_check(ctx, cudaStreamSynchronize(st), "tensor-core GEMM"))) return rc;
  if (hs[0]) return fail(ctx, GW_ERR_TIMEOUT, "tensor-core pipeline wait timed out (role " + std::to_string(hs[1]) + ")");
  return GW_OK;
}

}  // namespace tc

size_t tc_scratch_bytes(const GridInfo& g, int n_b, int n_occ, int n_rows, bool with_tmp, int n_sig, int n_entries,
                        bool one_psi) {
  return tc::scratch_bytes(g, n_b, n_occ, n_rows, with_tmp, n_sig, n_entries, one_psi);
}

gw_status tc_begin(gw_ctx* ctx, void* scratch, cudaStream_t st, int* status_dev) {
  return cuda_check(ctx, cudaMemsetAsync(status_dev ? status_dev : tc::status_words(scratch), 0, 2 * sizeof(int), st),
                    "memset");
}

gw_status tc_sigma_rows(gw_ctx* ctx, const GridInfo& g, int n_b, int n_occ, const void* psi, const GreenScales& gs,
                        int r0, int n_rows, gw_prec prec, const TcSigma& sig, void* scratch, bool prep_b,
                        cudaStream_t st) {
  if (sig.n_n < 1 || sig.n_n > 32) return fail(ctx, GW_ERR_SHAPE, "fused self-energy contraction takes 1..32 bands");
  return tc::run(ctx, g, n_b, n_occ, psi, &gs, r0, n_rows, prec, 2, nullptr, nullptr, scratch, prep_b, st, sig.sk,
                 nullptr, &sig, true);
}

gw_status tc_green_rows(gw_ctx* ctx, const GridInfo& g, int n_b, int n_occ, const void* psi, const GreenScales* gs,
                        int r0, int n_rows, gw_prec prec, void* g_occ, void* g_unocc, void* scratch, bool prep_b,
                        cudaStream_t st, const float* sk_dev, const TcEntries& en) {
  return tc::run(ctx, g, n_b, n_occ, psi, gs, r0, n_rows, prec, 1, g_occ, g_unocc, scratch, prep_b, st, sk_dev, nullptr,
                 nullptr, false, en);
}

gw_status tc_chi_rows(gw_ctx* ctx, const GridInfo& g, int n_b, int n_occ, const void* psi, const GreenScales* gs,
                      int r0, int n_rows, gw_prec prec, void* chi, void* scratch, bool prep_b, cudaStream_t st,
                      const float* sk_dev, int* status_dev, bool lower, const TcEntries& en) {
  return tc::run(ctx, g, n_b, n_occ, psi, gs, r0, n_rows, prec, 0, chi, nullptr, scratch, prep_b, st, sk_dev,
                 status_dev, nullptr, lower, en);
}

gw_status tc_check_status(gw_ctx* ctx, const int* status_dev, cudaStream_t st) {
  int hs[2] = {0, 0};
  gw_status rc;
  if ((rc = cuda_check(ctx, cudaMemcpyAsync(hs, status_dev, sizeof(hs), cudaMemcpyDeviceToHost, st), "status"))) return rc;
  if ((rc = cuda_check(ctx, cudaStreamSynchronize(st), "tensor-core GEMM"))) return rc;
  if (hs[0]) return fail(ctx, GW_ERR_TIMEOUT, "tensor-core pipeline wait timed out (role " + std::to_string(hs[1]) + ")");
  return GW_OK;
}

gw_status tc_check(gw_ctx* ctx, void* scratch, cudaStream_t st) { return tc::check_status(ctx, scratch, st); }

}  // namespace gw
