// k_ozpotrf.cu -- FP64 Cholesky factorisation with its trailing updates on the
// BF16 tensor cores, by splitting into exact slices (Ozaki, Ogita, Oishi and Rump 2012,
// "Error-free transformations of matrix multiplication by using fast routines of
// matrix multiplication and its applications").
//
// FP64 units on this GPU do 2 FMA per clock and SM (about 1.1 TFLOP/s in all),
// the BF16 tensor cores three orders of magnitude more, so C -= P P^T is formed
// from integer slices: every row i of the panel P is scaled by 2^-e_i
// (|p_ik| 2^-e_i < 1) and cut into S = 7 balanced base-256 digits,
//     p_ik 2^-e_i = sum_s d_s 2^-(7 + 8 s) + r,   |d_s| <= 128,  |r| <= 2^-56,
// which BF16 holds exactly.  Pairs a + b = d <= 6 share one FP32 accumulator in
// TMEM per level d; over a window of WIN * 64 values of k a level's partial sums
// stay exact integers below 2^24 (levels 0..4; the last two may round their
// lowest bit, 2^-54 of the row scales, in the worst case).  Each window is added
// into one 64-bit integer per output; a single conversion to FP64 and one
// subtraction from C end the update.  What is cut off is relative to a row's largest
// entry, so this stands in for FMAs where the rows' large entries meet (flat rows,
// ozslice.cuh); entries of other rows, the sparse and the decaying ones, take FMAs.
// Error of the factor against double-double (root mean square), CUDA-core route / this:
// n = 65 1.4e-16 / 1.4e-16, n = 1024 kappa = 10 2.2e-16 / 1.8e-16, n = 2500 kappa = 1e4
// 6.1e-15 / 4.0e-15.
//
// Two-level right-looking blocking: panels of 64 columns inside blocks of NB = 512,
// one update of the block's remaining columns per panel (depth 64) and one of the
// whole trailing matrix per block (depth 512, sliced again with one exponent per
// row over the block); the CTA that updates the next diagonal block factors it in
// the same launch, so a panel is two launches.  Factor alone on one GB300, FP64
// CUDA-core updates -> here: n = 1024 3.66 -> 1.16 ms, 3000 18.6 -> 3.7, 5000
// 53 -> 7.2, 16384 1260 -> 66.8 ms (there the tensor cores do 28 products of slices
// for one of FP64: 620 TFLOP/s over the whole factorisation; blocks of 256 columns
// 71.2).  Per panel, small trailing matrix: 51 us tile + diagonal block, 19 us panel
// solve.
#include <algorithm>

#include "kernels.h"
#include "ozslice.cuh"
#include "rcp64.cuh"
#include "tc_ptx.cuh"

namespace jmg {
namespace ozf {
constexpr int BM = 128;        // rows of an output tile
constexpr int BN = 64;         // columns of an output tile
constexpr int BK = 64;         // K per block: 64 BF16 = one 128-byte swizzle row
constexpr int WIN = 3;         // K blocks per exact accumulation window
constexpr int ASTAGES = 6;     // ring of row-slice tiles
constexpr int THREADS = 576;   // warps 0-1 producer / MMA, 2-17 epilogue (16 columns each)
constexpr int A_TILE = BM * BK * 2;  // 16 KiB
constexpr int B_TILE = BN * BK * 2;  // 8 KiB
constexpr int B_BUF = S * B_TILE;
constexpr int SMEM = 2 * B_BUF + ASTAGES * A_TILE + 1024 + 256;
constexpr uint32_t TCOLS = 512;      // 7 levels x 64 columns, rounded up
constexpr int PW = 64;               // panel width
constexpr int PT = 256;              // threads of the panel solve
constexpr int GROUP = 8;             // row tiles per raster group

// Tile b of the lower trapezoid {(ti, tj): ti < TI, tj < TJ, 64 tj <= 128 ti + 127}
// in groups of GROUP row tiles, column by column within a group, so that the
// CTAs that run together share few rows and few columns of the operand.  Tiles
// above the diagonal are enumerated too (false: skip).
JMG_DEV bool tile_of(int b, int TI, int TJ, int& ti, int& tj) {
  // group g holds GROUP * min(TJ, 2 GROUP (g + 1)) tiles
  constexpr int W = 2 * GROUP;
  const int gt = TJ / W;  // groups 0 .. gt-1 have W (g + 1) columns
  const long long tri = (long long)GROUP * W * gt * (gt + 1) / 2;
  int g, rem;
  if (b < tri) {
    const int q = b / (GROUP * W);
    g = (int)((sqrtf(8.0f * (float)q + 1.0f) - 1.0f) * 0.5f);
    while ((long long)g * (g + 1) / 2 > q) --g;
    while ((long long)(g + 1) * (g + 2) / 2 <= q) ++g;
    rem = b - GROUP * W * (g * (g + 1) / 2);
  } else {
    const int r = (int)(b - tri);
    g = gt + r / (GROUP * TJ);
    rem = r % (GROUP * TJ);
  }
  ti = g * GROUP + rem % GROUP;
  tj = rem / GROUP;
  return ti < TI && tj * BN < (ti + 1) * BM;
}
static long long tile_count(int TI, int TJ) {
  const int W = 2 * GROUP, gt = std::min(TJ / W, cdiv(TI, GROUP)), G = cdiv(TI, GROUP);
  return (long long)GROUP * W * gt * (gt + 1) / 2 + (long long)(G - gt) * GROUP * TJ;
}

// ---------------------------------------------------------------------------
// Diagonal block of kb <= 64 columns, in place, by one CTA of THREADS threads, in two
// halves of 32: a column updates its own half at once, the first half updates the second
// with one sum of 32 products per entry.  (Against updating all columns at once: half the
// trailing work beside the chain, and an entry of the second half is rounded 32 times
// less: error of L at n = 65 1.8e-16 -> 1.4e-16, n = 1024 2.0e-16 -> 1.8e-16, in the same
// time.)
// A dependent FP64 instruction waits 68 clocks and the pivots are a serial chain:
// warp 0 keeps column j in registers (two rows per lane) and in
// step j updates column j+1, takes pivot j+1 (its reciprocal in integers) and hands
// u_j = column j / a_jj to the trailing warps (named barrier 1); those apply
// a_rc -= a_rj u_c to columns j+2 .. of the half, column j+2 first, which they release
// (named barrier 2: the chain's input of step j+1).  Each barrier is passed the same
// number of times on both sides, and nothing leaves the loop early: the first pivot that
// is not positive is recorded and the columns from it on are dropped.
namespace diag64 {
constexpr int HB = 32;      // columns of a half
constexpr int TRAIL = 384;  // trailing threads
constexpr int BAR = 32 + TRAIL;
constexpr int LD = PW + 1;
constexpr int NEL = PW * (PW + 1) / 2;
constexpr int SMEM = (PW * LD + 2 * PW + 2 * PW) * 8 + NEL * 2;
}  // namespace diag64

JMG_DEV void bar_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
JMG_DEV void bar_arrive(int id, int count) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}

JMG_DEV void diag_body(double* sm_d64, double* __restrict__ A, int lda, int kb, int koff,
                       int* __restrict__ info) {
  using namespace diag64;
  constexpr int TH = THREADS;
  double* s64 = sm_d64;                 // s64[c * LD + r] = a_rc
  double* s_u = s64 + PW * LD;          // [2][PW]
  double* s_l = s_u + 2 * PW;           // [PW]
  double* s_il = s_l + PW;              // [PW]
  unsigned short* s_rc = reinterpret_cast<unsigned short*>(s_il + PW);  // packed -> (c, r)
  __shared__ int fail;
  const int t = threadIdx.x, warp = t / 32, lane = t % 32;
  if (t == 0) fail = *(volatile int*)info;
  __syncthreads();
  if (fail != 0) return;  // an earlier block already failed
  {
    constexpr int Q = (PW * PW + TH - 1) / TH;
    double v[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {  // all loads first
      const int idx = t + TH * q, r = idx % PW, c = idx / PW;
      v[q] = (idx < PW * PW && r < kb && c <= r) ? A[(size_t)c * lda + r] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int idx = t + TH * q;
      if (idx < PW * PW) s64[(idx / PW) * LD + idx % PW] = v[q];
    }
  }
  for (int c = warp; c < PW; c += TH / 32) {
    const int base = c * PW - c * (c - 1) / 2;  // column c starts here in packed order
    for (int r = c + lane; r < PW; r += 32) s_rc[base + r - c] = (unsigned short)((c << 8) | r);
  }
  __syncthreads();
  auto column = [](int c) { return c * PW - c * (c - 1) / 2; };  // its start in packed order
  int fj = -1;  // first failing column (chain warp)
  for (int p = 0; p < kb; p += HB) {
    const int pe = min(kb, p + HB);
    if (warp == 0) {
      double lo = s64[p * LD + lane], hi = s64[p * LD + lane + 32];  // column j, two rows
      bool bad = false;
      double w = pivot_rcp(__shfl_sync(0xffffffffu, p ? hi : lo, 0), &bad);
      if (bad && fj < 0) fj = p;
      for (int j = p; j + 1 < pe; ++j) {
        const int j1 = j + 1;
        const double a1 = __shfl_sync(0xffffffffu, j1 < 32 ? lo : hi, j1 & 31);
        const double v = a1 * w;  // u of row j+1
        if (j > p) bar_sync(2, BAR);  // column j+1 done to j-1
        double* cn = &s64[j1 * LD];
        double nlo = cn[lane], nhi = cn[lane + 32];
        double* u = &s_u[(j & 1) * PW];
        bad = false;
        if (j1 < 32) {
          nlo = fma(-lo, v, nlo);
          const double d = __shfl_sync(0xffffffffu, nlo, j1);
          const double uhi = hi * w;
          u[lane] = lo * w;
          nhi = fma(-hi, v, nhi);
          cn[lane] = nlo;
          cn[lane + 32] = nhi;
          s64[(lane + 32) * LD + j] = uhi;  // kept for the second half
          __syncwarp();
          bar_arrive(1, BAR);
          w = pivot_rcp(d, &bad);
        } else {
          nhi = fma(-hi, v, nhi);
          const double d = __shfl_sync(0xffffffffu, nhi, j1 - 32);
          u[lane + 32] = hi * w;
          cn[lane + 32] = nhi;
          __syncwarp();
          bar_arrive(1, BAR);
          w = pivot_rcp(d, &bad);
        }
        if (bad && fj < 0) fj = j1;
        lo = nlo;
        hi = nhi;
      }
      if (p == 0) s64[(lane + 32) * LD + pe - 1] = hi * w;
      if (lane == 0 && fj >= 0) fail = fj + 1;
    } else if (warp <= TRAIL / 32) {
      const int tq = t - 32;  // index among the trailing threads
      for (int j = p; j + 1 < pe; ++j) {
        __syncwarp();
        bar_sync(1, BAR);  // u_j and column j in place
        const double* cj = &s64[j * LD];
        const double* uj = &s_u[(j & 1) * PW];
        if (j + 2 < pe) {
          if (tq >= j + 2 && tq < kb) {
            double* c2 = &s64[(j + 2) * LD];
            c2[tq] = fma(-cj[tq], uj[j + 2], c2[tq]);
          }
          __syncwarp();
          bar_arrive(2, BAR);
        }
        const int e2 = column(pe);
        for (int e = column(min(j + 3, pe)) + tq; e < e2; e += TRAIL) {
          const int rc = s_rc[e], c = rc >> 8, r = rc & 255;
          if (r >= kb) continue;
          s64[c * LD + r] = fma(-cj[r], uj[c], s64[c * LD + r]);
        }
      }
    }
    __syncthreads();
    if (pe == kb) break;
    const int e = column(HB) + t;  // second half: 528 entries, one per thread
    if (e < NEL) {
      const int rc = s_rc[e], c = rc >> 8, r = rc & 255;
      double sum = s64[r] * s64[c * LD];
#pragma unroll 8
      for (int j = 1; j < HB; ++j) sum = fma(s64[j * LD + r], s64[c * LD + j], sum);
      s64[c * LD + r] -= sum;
    }
    __syncthreads();
  }
  const int jdone = fail ? fail - 1 : kb;  // columns that are final
  if (t < jdone) {  // l_cc = sqrt(a_cc), l_rc = a_rc / l_cc
    const double l = sqrt(s64[t * LD + t]);
    s_l[t] = l;
    s_il[t] = 1.0 / l;
  }
  __syncthreads();
  for (int c = warp; c < jdone; c += TH / 32)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = lane + 32 * h;
      if (r >= c && r < kb) A[(size_t)c * lda + r] = r == c ? s_l[c] : s64[c * LD + r] * s_il[c];
    }
  if (t == 0 && fail) atomicCAS(info, 0, koff + fail);
}

// The first block; any: nany flags of the factorisation's updates, cleared here.
__global__ void __launch_bounds__(THREADS) k_oz_diag(double* __restrict__ A, int lda, int kb,
                                                     int koff, int* __restrict__ info,
                                                     int* __restrict__ any, int nany) {
  for (int i = threadIdx.x; i < nany; i += THREADS) any[i] = 0;
  extern __shared__ __align__(16) double sm_diag64[];
  diag_body(sm_diag64, A, lda, kb, koff, info);
}

// ---------------------------------------------------------------------------
// C (m x ncols) -= P Q^T, P and Q given by their slices and row exponents: row r of
// slice s is row s * nA + rA + r of P's map (nB, rB: Q's).
//  * RECT = false, the factorisation: Q is P's head, only the lower part is updated, and
//    CTA 0 takes tile 0 alone and then factors the diagonal block it has just updated
//    (kb_diag columns), while the others work through the rest of the update;
//  * RECT = true, the blocked solves: the whole rectangle.
// info may be null when RECT; err (RECT only) is the solve's error word.
// Entries whose row or column is spread (ozslice.cuh; the rows' words are exA and exB,
// `flat` the count that makes a flat one) take FP64 FMAs over `F` instead: 32 x 32 entries
// at a time, two columns per epilogue warp, shared out over all CTAs whoever did the slices
// of the tile (its entries are others).  Bound by the FP64 pipe (16 clocks a warp
// instruction): 0.14 ms for 32 x 32 at depth 512.  *any is set by the kernels that made the
// words when one of them is spread, so that a launch without only tests its words: factor at
// n = 5000 7.13 -> 7.20 ms, 16384 66.2 -> 66.8, solves at 16384, 64 11.2 -> 11.5.  With next
// to every row spread (exponential covariance of a 2-D grid of 5000 sites, range 0.5) the
// factor takes 48.7 ms and 64 right-hand sides 6.7 (CUDA-core kernels: 53.1, 10.4).
struct Fma {            // the operands in FP64: P(row, k) = P[row prs + k pks], k < kv;
  const double *P, *Q;  // Q(column, k) = Q[column qcs + k qks]
  size_t prs, pks, qcs, qks;
  int kv;
};

template <bool RECT>
__global__ void __launch_bounds__(THREADS, 1)
    k_oz_update(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                double* __restrict__ C, int ldc, int nA, int rA, int nB, int rB, int m, int ncols,
                int nkb, const int* __restrict__ exA, const int* __restrict__ exB, int flat,
                const int* __restrict__ any, const Fma F, int TI, int TJ,
                int ntiles, int kb_diag, int koff, int* __restrict__ info, int* __restrict__ err,
                unsigned long long wait_ns, int hold) {
  using namespace tc;
  extern __shared__ __align__(1024) unsigned char sm_raw_ozf[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(sm_raw_ozf) + 1023) & ~uintptr_t(1023));
  unsigned char* bbuf = smem;              // [2][S][B_TILE]
  unsigned char* abuf = smem + 2 * B_BUF;  // [ASTAGES][A_TILE]
  uint64_t* bars = reinterpret_cast<uint64_t*>(abuf + ASTAGES * A_TILE);
  uint64_t* bfull = bars;       // 2
  uint64_t* bempty = bars + 2;  // 2
  uint64_t* afull = bars + 4;   // ASTAGES
  uint64_t* aempty = afull + ASTAGES;
  uint64_t* accf = aempty + ASTAGES;
  uint64_t* acce = accf + 1;
  uint64_t* drain = acce + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  __shared__ int s_fail, s_info, s_any;

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  // this CTA's tiles: first, first + step, ...
  const int first = blockIdx.x,
            step = RECT ? (int)gridDim.x : (blockIdx.x == 0 ? ntiles : (int)gridDim.x - 1);
  auto tile = [&](int b, int& ti, int& tj) -> bool {
    if (!RECT) return tile_of(b, TI, TJ, ti, tj);
    ti = b / TJ, tj = b % TJ;
    return true;
  };
  if (threadIdx.x == 0) {
    s_fail = 0;
    s_any = *any;
    s_info = info ? *(volatile int*)info : 0;
    if (RECT && *(volatile int*)err != 0) s_info = 1;  // an earlier launch gave up
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bfull[i], 1);
      mbar_init(&bempty[i], 1);
    }
    for (int i = 0; i < ASTAGES; ++i) {
      mbar_init(&afull[i], 1);
      mbar_init(&aempty[i], 1);
    }
    mbar_init(accf, 1);
    mbar_init(acce, 16);
    mbar_init(drain, 1);
    fence_mbar_init();
    prefetch_tmap(&tmA);
    prefetch_tmap(&tmB);
  }
  __syncthreads();
  // an earlier block already failed, or this CTA is here for spread entries only
  if (s_info != 0 || (first >= ntiles && !s_any)) return;
  if (warp == 1) {
    tmem_alloc(tmem_slot, TCOLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  long long b_issued = 0, a_issued = 0;
  if (warp == 0) {
    // hold (a test hook) keeps the producer idle: the MMA warp's first wait runs out
    if (lane == 0 && !hold) {
      bool ok = true;
      for (int b = first; b < ntiles && ok; b += step) {
        int ti, tj;
        if (!tile(b, ti, tj)) continue;
        for (int kb = 0; kb < nkb && ok; ++kb) {
          const int bs = (int)(b_issued & 1);
          if (b_issued >= 2 &&
              !mbar_wait(&bempty[bs], (uint32_t)((b_issued >> 1) - 1) & 1, wait_ns)) {
            ok = false;
            break;
          }
          if (ld_shared_volatile(&s_fail)) {
            ok = false;
            break;
          }
          mbar_expect_tx(&bfull[bs], B_BUF);
          for (int s = 0; s < S; ++s)
            tma_load_2d(bbuf + bs * B_BUF + s * B_TILE, &tmB, kb * BK, s * nB + rB + tj * BN,
                        &bfull[bs]);
          ++b_issued;
          for (int s = 0; s < S; ++s) {
            const int st = (int)(a_issued % ASTAGES);
            if (a_issued >= ASTAGES &&
                !mbar_wait(&aempty[st], (uint32_t)((a_issued / ASTAGES) - 1) & 1, wait_ns)) {
              ok = false;
              break;
            }
            mbar_expect_tx(&afull[st], A_TILE);
            tma_load_2d(abuf + st * A_TILE, &tmA, kb * BK, s * nA + rA + ti * BM, &afull[st]);
            ++a_issued;
          }
        }
      }
      if (!ok) atomicExch(&s_fail, 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr int GMAX = 256 / BN;  // B slices per MMA
      long long ga = 0, gb = 0, gw = 0;
      bool ok = true;
      for (int b = first; b < ntiles && ok; b += step) {
        int ti, tj;
        if (!tile(b, ti, tj)) continue;
        for (int kw = 0; kw < nkb && ok; kw += WIN, ++gw) {
          if (gw >= 1 && !mbar_wait(acce, (uint32_t)(gw - 1) & 1, wait_ns)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const int ke = min(nkb, kw + WIN);
          for (int kb = kw; kb < ke && ok; ++kb, ++gb) {
            const int bs = (int)(gb & 1);
            if (!mbar_wait(&bfull[bs], (uint32_t)(gb >> 1) & 1, wait_ns)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t sb = smem_u32(bbuf + bs * B_BUF);
            for (int a = 0; a < S; ++a, ++ga) {
              const int st = (int)(ga % ASTAGES);
              if (!mbar_wait(&afull[st], (uint32_t)(ga / ASTAGES) & 1, wait_ns)) {
                ok = false;
                break;
              }
              tc_fence_after();
              const uint32_t sa = smem_u32(abuf + st * A_TILE);
              // row slice a meets column slices 0 .. S-1-a (levels a .. S-1): they
              // lie one after another in shared memory and their levels one after
              // another in TMEM, so up to four make one MMA of 256 columns
              for (int b0 = 0; b0 < S - a; b0 += GMAX) {
                const int cnt = min(GMAX, S - a - b0);
                const uint32_t idesc_g = idesc_f16(BM, BN * cnt, 1);
                const uint32_t dacc = tmem + (uint32_t)((a + b0) * BN);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                  const bool first = (kb == kw) && (a == 0) && (kk == 0);
                  tc_mma_f16(dacc, sdesc_sw128(sa + kk * 32),
                             sdesc_sw128(sb + b0 * B_TILE + kk * 32), idesc_g, first ? 0u : 1u);
                }
              }
              tc_commit(&aempty[st]);
            }
            tc_commit(&bempty[bs]);
          }
          if (!ok) atomicExch(&s_fail, 1);
          tc_commit(accf);
        }
      }
      if (!ok) atomicExch(&s_fail, 1);
    }
  } else {
    // epilogue: warp w reads TMEM lane group q = w % 4 and 16 columns of every
    // level.  acc holds sum_d level_d 2^(SH - 8 d), SH fractional bits chosen so
    // that K products of at most 2^14 stay below 2^62.
    constexpr int CW = 16;
    const int q = warp & 3, ch = ((warp - 2) >> 2) * CW;
    const int sh = nkb * BK <= 256 ? 40 : (nkb * BK <= 512 ? 39 : 38);
    const long long half = 1ll << (47 - sh);
    long long gw = 0;
    bool ok = true;
    for (int b = first; b < ntiles && ok; b += step) {
      int ti, tj;
      if (!tile(b, ti, tj)) continue;
      const int row = ti * BM + q * 32 + lane;
      const int c0 = tj * BN + ch;
      // columns c < jn of this thread are in range (and on or below the diagonal)
      const int jn = row < m ? max(0, min(CW, min(ncols - c0, RECT ? CW : row - c0 + 1))) : 0;
      // the words of the row, and of column c0 + lane; put: the columns done here
      const bool col = lane < CW && c0 + lane < ncols;
      const int wr = row < m ? exA[row] : 0, wc = col ? exB[c0 + lane] : 0;
      const unsigned cs = __ballot_sync(0xffffffffu, col && word_spread(wc, flat));
      const unsigned put = word_spread(wr, flat) ? 0u : ((1u << jn) - 1) & ~cs;
      unsigned long long acc[CW];  // (unsigned: rows and columns past the end wrap, never trap)
#pragma unroll
      for (int c = 0; c < CW; ++c) acc[c] = 0ull;
      for (int kw = 0; kw < nkb; kw += WIN, ++gw) {
        // (one answer for the warp: what follows is aligned across its lanes)
        if (!__all_sync(0xffffffffu, mbar_wait(accf, (uint32_t)gw & 1, wait_ns) &&
                                         !ld_shared_volatile(&s_fail))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t tacc = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)ch;
#pragma unroll
        for (int d = 0; d < 5; ++d) {
          uint32_t v[16];
          tmem_ld16(tacc + (uint32_t)(d * BN), v);
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < CW; ++c)
            acc[c] += (unsigned long long)((long long)__float2int_rn(__uint_as_float(v[c]))
                                           << (sh - 8 * d));
        }
        {
          uint32_t v[16], w[16];
          tmem_ld16(tacc + (uint32_t)(5 * BN), v);
          tmem_ld16(tacc + (uint32_t)(6 * BN), w);
          tmem_ld_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acce);
#pragma unroll
          for (int c = 0; c < CW; ++c) {
            const long long lo = ((long long)__float2int_rn(__uint_as_float(v[c])) << 8) +
                                 (long long)__float2int_rn(__uint_as_float(w[c]));
            acc[c] += (unsigned long long)((lo + half) >> (48 - sh));
          }
        }
      }
      if (!ok) {
        atomicExch(&s_fail, 1);
        break;
      }
      double* cp = C + (size_t)c0 * ldc + row;
      const int er = word_exp(wr) - 14 - sh;
      double old[CW];
#pragma unroll
      for (int c = 0; c < CW; ++c) old[c] = put >> c & 1u ? cp[(size_t)c * ldc] : 0.0;
#pragma unroll
      for (int c = 0; c < CW; ++c) {
        const int ec = word_exp(__shfl_sync(0xffffffffu, wc, c));
        if (put >> c & 1u) cp[(size_t)c * ldc] = old[c] - scaled_double((long long)acc[c], er + ec);
      }
    }
    if (s_any && ok) {
      // (factorisation: CTA 0 does its share of tile 0, which holds the diagonal block)
      const bool head = !RECT && blockIdx.x == 0;
      const int u0 = RECT || head ? blockIdx.x : 7 + blockIdx.x;
      const int ue = head ? 8 : 8 * ntiles, us = head ? 1 : (RECT ? gridDim.x : gridDim.x - 1);
      for (int u = u0; u < ue; u += us) {
        int ti, tj;
        if (!tile(u >> 3, ti, tj)) continue;
        const int row = ti * BM + (u & 3) * 32 + lane, c0 = tj * BN + (u & 4) * 8 + 2 * (warp - 2);
        const int jn = row < m ? min(2, min(ncols - c0, RECT ? 2 : row - c0 + 1)) : 0;
        const bool rs = jn > 0 && word_spread(exA[row], flat);
        const bool s0 = jn > 0 && (rs || word_spread(exB[c0], flat));
        const bool s1 = jn > 1 && (rs || word_spread(exB[c0 + 1], flat));
        if (!__any_sync(0xffffffffu, s0 || s1)) continue;
        const double* p = F.P + (size_t)min(row, m - 1) * F.prs;
        const double* q0 = F.Q + (size_t)min(c0, ncols - 1) * F.qcs;
        const double* q1 = F.Q + (size_t)min(c0 + 1, ncols - 1) * F.qcs;
        double a0 = 0.0, a1 = 0.0;
#pragma unroll 8
        for (int k = 0; k < F.kv; ++k) {
          const double x = p[k * F.pks];
          a0 = fma(x, q0[k * F.qks], a0);
          a1 = fma(x, q1[k * F.qks], a1);
        }
        double* cp = C + (size_t)c0 * ldc + row;
        if (s0) cp[0] -= a0;
        if (s1) cp[ldc] -= a1;
      }
    }
  }
  __syncwarp();
  __syncthreads();
  if (ld_shared_volatile(&s_fail)) {
    if (warp == 0 && lane == 0) {
      for (long long u = (b_issued > 2 ? b_issued - 2 : 0); u < b_issued; ++u)
        (void)mbar_wait(&bfull[u & 1], (uint32_t)(u >> 1) & 1, wait_ns);
      for (long long g = (a_issued > ASTAGES ? a_issued - ASTAGES : 0); g < a_issued; ++g)
        (void)mbar_wait(&afull[g % ASTAGES], (uint32_t)(g / ASTAGES) & 1, wait_ns);
      if (info) atomicCAS(info, 0, -1);
      if (RECT) atomicExch(err, JMG_ERR_TIMEOUT);
    }
    if (warp == 1 && lane == 0) mma_drain(drain, wait_ns);
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, TCOLS);
  if (!RECT && blockIdx.x == 0 && !ld_shared_volatile(&s_fail)) {
    __syncthreads();  // tile 0 is in global memory, the rings are idle
    diag_body(reinterpret_cast<double*>(smem), C, ldc, kb_diag, koff, info);
  }
}

// ---------------------------------------------------------------------------
// Panel solve X L_kk^T = A21 (64 columns) and its slices.  G lanes share a row,
// each holding the column pairs {2 (g + G i), 2 (g + G i) + 1}; an SM's FP64 pipe
// takes one warp instruction per 16 clocks and a dependent one waits 68, so the row
// is spread over just enough lanes to fill the chip with eight warps per SM (four left
// half the pipe idle).  The solve runs on unscaled columns with Lh[j][l] = L_lj / L_jj
// (a_l -= a_j Lh[j][l]), the scaling by 1 / L_jj comes last: one FP64 instruction per
// element and step, nothing else.
template <int G>
__global__ void __launch_bounds__(PT) k_oz_panel(double* __restrict__ A, int lda, int n, int k,
                                                  __nv_bfloat16* __restrict__ SP,
                                                  int* __restrict__ ex,
                                                  unsigned long long* __restrict__ rowmax,
                                                  int* __restrict__ ex_block, int first, int last,
                                                  int* __restrict__ any,
                                                  const int* __restrict__ info) {
  constexpr int NP = 32 / G;     // column pairs per lane
  constexpr int RW = 32 / G;     // rows per warp
  constexpr int RB = PT / 32 * RW;  // rows per CTA
  __shared__ __align__(16) double Lh[PW * PW];
  __shared__ double rinv[PW];
  if (*(volatile const int*)info != 0) return;
  const int t = threadIdx.x, lane = t % 32, warp = t / 32;
  const double* Lkk = A + (size_t)k * lda + k;
  {
    constexpr int Q = PW * PW / PT;
    double v[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const int idx = t + PT * i, l = idx % PW, j = idx / PW;
      v[i] = l >= j ? Lkk[(size_t)j * lda + l] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) Lh[t + PT * i] = v[i];
  }
  const int g = lane % G, rl = warp * RW + lane / G;
  const int row = k + PW + blockIdx.x * RB + rl;
  double x[2 * NP];
#pragma unroll
  for (int i = 0; i < NP; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      x[2 * i + h] = row < n ? A[(size_t)(k + 2 * (g + G * i) + h) * lda + row] : 0.0;
  __syncthreads();
  if (t < PW) rinv[t] = 1.0 / Lh[t * PW + t];
  __syncthreads();
#pragma unroll 4
  for (int i = 0; i < PW * PW / PT; ++i) {
    const int idx = t + PT * i, l = idx % PW, j = idx / PW;
    if (l > j) Lh[idx] *= rinv[j];
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < PW; ++j) {
    const int go = (j / 2) % G, io = (j / 2) / G;  // owner lane and register of column j
    const double aj = G == 1 ? x[j] : __shfl_sync(0xffffffffu, x[2 * io + (j & 1)], go, G);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      if (2 * (G - 1 + G * i) + 1 <= j) continue;  // every lane's pair is done
      const double2 l2 = *reinterpret_cast<const double2*>(&Lh[j * PW + 2 * (g + G * i)]);
      const int l = 2 * (g + G * i);
      if (l > j) x[2 * i] = fma(-aj, l2.x, x[2 * i]);
      if (l + 1 > j) x[2 * i + 1] = fma(-aj, l2.y, x[2 * i + 1]);
    }
  }
  unsigned long long mx = 0;
#pragma unroll
  for (int i = 0; i < NP; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = 2 * (g + G * i) + h;
      x[2 * i + h] *= rinv[c];
      if (row < n) A[(size_t)(k + c) * lda + row] = x[2 * i + h];
      const unsigned long long b =
          (unsigned long long)__double_as_longlong(x[2 * i + h]) & 0x7FFFFFFFFFFFFFFFull;
      mx = b > mx ? b : mx;
    }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) {
    const unsigned long long b = __shfl_xor_sync(0xffffffffu, mx, o, G);
    mx = b > mx ? b : mx;
  }
  int near = 0;
#pragma unroll
  for (int i = 0; i < 2 * NP; ++i)
    near += near_max(abs_bits(x[i]), mx);
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) near += __shfl_xor_sync(0xffffffffu, near, o, G);
  if (row >= n) return;
  const int e = scale_exp_bits(mx);
  if (g == 0) {
    const int word = row_word(mx, near);
    ex[row] = word;
    if (word_spread(word, flat_count(PW))) *any = 1;
    unsigned long long bm = mx;  // of the block so far
    if (!first && rowmax[row] > bm) bm = rowmax[row];
    rowmax[row] = bm;
    if (last) ex_block[row] = row_word(bm, 0);  // (k_oz_strip adds the count)
  }
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    int d0[S], d1[S];
    digits7(x[2 * i], e, d0);
    digits7(x[2 * i + 1], e, d1);
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const __nv_bfloat162 p = __floats2bfloat162_rn((float)d0[s], (float)d1[s]);
      *reinterpret_cast<__nv_bfloat162*>(&SP[((size_t)s * n + row) * PW + 2 * (g + G * i)]) = p;
    }
  }
}

// Slices of the finished block column k0 .. k0 + K - 1 (rows from r0 on) with one
// exponent per row over the whole block; the rows' words in ex gain the entries near the
// maximum, and *any is set when a row turns out to be spread.  grid = (32-row tiles, K / 64).
__global__ void __launch_bounds__(256) k_oz_strip(const double* __restrict__ A, int lda, int n,
                                                  int k0, int r0, int K,
                                                  const unsigned long long* __restrict__ rowmax,
                                                  __nv_bfloat16* __restrict__ SP,
                                                  int* __restrict__ ex, int* __restrict__ any,
                                                  const int* __restrict__ info) {
  __shared__ double T[64][33];
  if (info && *(volatile const int*)info != 0) return;
  const int t = threadIdx.x;
  const int rb = r0 + blockIdx.x * 32, kc = blockIdx.y * 64;
  {
    double v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int r = rb + t % 32, c = t / 32 + 8 * q;
      v[q] = r < n ? A[(size_t)(k0 + kc + c) * lda + r] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) T[t / 32 + 8 * q][t % 32] = v[q];
  }
  __syncthreads();
  const int rr = t / 8, cc = 8 * (t % 8), row = rb + rr;
  const unsigned long long mx = row < n ? rowmax[row] : 0;
  int near = 0;
#pragma unroll
  for (int u = 0; u < 8; ++u)
    near += near_max(abs_bits(T[cc + u][rr]), mx);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) near += __shfl_xor_sync(0xffffffffu, near, o);
  if (row >= n) return;
  const int e = scale_exp_bits(mx);
  if (cc == 0) {
    const int add = (can_be_flat(mx) ? near << 16 : 0) + (1 << 26);
    const int word = atomicAdd(&ex[row], add) + add;
    if (word >> 26 == (int)gridDim.y && word_spread(word, flat_count(K))) *any = 1;
  }
  uint32_t w[S][4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    int d0[S], d1[S];
    digits7(T[cc + 2 * u][rr], e, d0);
    digits7(T[cc + 2 * u + 1][rr], e, d1);
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const __nv_bfloat162 p = __floats2bfloat162_rn((float)d0[s], (float)d1[s]);
      w[s][u] = *reinterpret_cast<const uint32_t*>(&p);
    }
  }
#pragma unroll
  for (int s = 0; s < S; ++s)
    *reinterpret_cast<uint4*>(&SP[((size_t)s * n + row) * K + kc + cc]) =
        make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

// ---------------------------------------------------------------------------
// The blocked solves' operands.

// Row maxima (abs_bits order) of every SK-wide block column of the lower L, diagonal
// blocks included: out[b * n + i], and the rows' words for the strips, still without their
// counts, ex[b * n + i].  grid = (rows / 256, blocks); a thread walks its row, coalesced
// across the threads.  any: two flags per block, cleared here.
constexpr int SK = 512;
__global__ void __launch_bounds__(256) k_oz_block_max(const double* __restrict__ L, int lda, int n,
                                                      unsigned long long* __restrict__ out,
                                                      int* __restrict__ ex,
                                                      int* __restrict__ any) {
  if (blockIdx.x == 0 && threadIdx.x < 2) any[2 * blockIdx.y + threadIdx.x] = 0;
  const int i = blockIdx.x * 256 + threadIdx.x, k0 = blockIdx.y * SK;
  if (i >= n) return;
  unsigned long long mx = 0;
  const int ke = min(k0 + SK, i + 1);
#pragma unroll 8
  for (int k = k0; k < ke; ++k) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(L[(size_t)k * lda + i]) &
                                 0x7FFFFFFFFFFFFFFFull;
    mx = b > mx ? b : mx;
  }
  out[(size_t)blockIdx.y * n + i] = mx;
  ex[(size_t)blockIdx.y * n + i] = row_word(mx, 0);
}
// sc[i] = the exponent of row i of L over all its blocks
__global__ void k_oz_row_scale(int n, int nb, const unsigned long long* __restrict__ bmax,
                               int* __restrict__ sc) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  unsigned long long mx = 0;
  for (int b = 0; b < nb; ++b) {
    const unsigned long long v = bmax[(size_t)b * n + i];
    mx = v > mx ? v : mx;
  }
  sc[i] = scale_exp_bits(mx);
}

// x 2^e by integer addition to the exponent field where it stays normal
JMG_DEV double mul_pow2(double x, int e) {
  const int E = (__double2hiint(x) >> 20) & 0x7FF;
  if (E == 0 || E == 0x7FF || E + e < 1 || E + e > 0x7FE) return ldexp(x, e);
  return __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x));
}

// Slices of the columns of a column-major P (kv <= SK rows, ncols columns), one
// exponent per column (its word in ex): slice s, column c, row k at
// SP[(s * ncols + c) * SK + k] (zero past kv).  Row k is scaled by 2^(sign sc[k]) first (sign 0: not).  One warp per
// column.
__global__ void __launch_bounds__(256) k_oz_cut_cols(const double* __restrict__ P, int ld, int kv,
                                                     int ncols, const int* __restrict__ sc,
                                                     int sign, __nv_bfloat16* __restrict__ SP,
                                                     int* __restrict__ ex, int* __restrict__ any) {
  const int c = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
  if (c >= ncols) return;
  constexpr int Q = SK / 64;
  double x[2 * Q];
#pragma unroll
  for (int q = 0; q < Q; ++q)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = 64 * q + 2 * lane + h;
      x[2 * q + h] = k < kv ? P[(size_t)c * ld + k] : 0.0;
    }
  unsigned long long mx = 0;
#pragma unroll
  for (int i = 0; i < 2 * Q; ++i) {
    const int k = 64 * (i / 2) + 2 * lane + (i & 1);
    if (sign != 0 && k < kv) x[i] = mul_pow2(x[i], sign * sc[k]);
    const unsigned long long b =
        (unsigned long long)__double_as_longlong(x[i]) & 0x7FFFFFFFFFFFFFFFull;
    mx = b > mx ? b : mx;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long b = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = b > mx ? b : mx;
  }
  int near = 0;
#pragma unroll
  for (int i = 0; i < 2 * Q; ++i)
    near += 64 * (i / 2) + 2 * lane + (i & 1) < kv &&
            near_max(abs_bits(x[i]), mx);
  near = __reduce_add_sync(0xffffffffu, near);
  const int e = scale_exp_bits(mx);
  if (lane == 0) {
    const int word = row_word(mx, near);
    ex[c] = word;
    if (word_spread(word, flat_count(kv))) *any = 1;
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    int d0[S], d1[S];
    digits7(x[2 * q], e, d0);
    digits7(x[2 * q + 1], e, d1);
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<__nv_bfloat162*>(&SP[((size_t)s * ncols + c) * SK + 64 * q + 2 * lane]) =
          __floats2bfloat162_rn((float)d0[s], (float)d1[s]);
  }
}

static int map_slices(CUtensorMap* map, const void* base, int n, int K, int box_rows) {
  return make_tmap_2d(map, base, (unsigned long long)K, (unsigned long long)S * n,
                      (unsigned long long)K * 2, BK, (unsigned)box_rows,
                      CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, CU_TENSOR_MAP_SWIZZLE_128B);
}
}  // namespace ozf

// ---------------------------------------------------------------------------
// host side

namespace {
struct OzfPlan {
  int NB;
  int nany;  // one flag per panel, one per block
  size_t panel, strip, exp_in, exp_out, rowmax, any, total;
};
OzfPlan ozf_plan(int n) {
  OzfPlan p{};
  p.NB = (int)std::min<size_t>(512, round_up((size_t)n, ozf::PW));
  size_t off = 0;
  auto take = [&](size_t b) {
    const size_t at = off;
    off = round_up(off + b, 256);
    return at;
  };
  p.panel = take((size_t)ozf::S * n * ozf::PW * 2);
  p.strip = take(n > p.NB ? (size_t)ozf::S * n * p.NB * 2 : 0);
  p.exp_in = take(sizeof(int) * (size_t)n);
  p.exp_out = take(sizeof(int) * (size_t)n);
  p.rowmax = take(sizeof(unsigned long long) * (size_t)n);
  p.nany = cdiv(n, ozf::PW) + cdiv(n, p.NB);
  p.any = take(sizeof(int) * (size_t)p.nany);
  p.total = off;
  return p;
}
}  // namespace

size_t ozf_workspace(int n) { return n > ozf::PW ? ozf_plan(n).total : 0; }

int potrf_split(int n, double* A, int lda, int* info, void* work, cudaStream_t s, int hold) {
  using namespace ozf;
  const OzfPlan p = ozf_plan(n);
  char* w = static_cast<char*>(work);
  __nv_bfloat16* panel = reinterpret_cast<__nv_bfloat16*>(w + p.panel);
  __nv_bfloat16* strip = reinterpret_cast<__nv_bfloat16*>(w + p.strip);
  int* e_in = reinterpret_cast<int*>(w + p.exp_in);
  int* e_out = reinterpret_cast<int*>(w + p.exp_out);
  unsigned long long* rowmax = reinterpret_cast<unsigned long long*>(w + p.rowmax);
  int* any = reinterpret_cast<int*>(w + p.any);
  int dev = 0, nsm = 152;
  JMG_CUDA(cudaGetDevice(&dev));
  JMG_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  JMG_TRY(ensure_smem(k_oz_update<false>, SMEM));
  JMG_TRY(ensure_smem(k_oz_diag, diag64::SMEM));
  CUtensorMap pa, pb, oa, ob;
  JMG_TRY(map_slices(&pa, panel, n, PW, BM));
  JMG_TRY(map_slices(&pb, panel, n, PW, BN));
  if (n > p.NB) {
    JMG_TRY(map_slices(&oa, strip, n, p.NB, BM));
    JMG_TRY(map_slices(&ob, strip, n, p.NB, BN));
  }
  // P: columns k0 .. of L, K of them
  auto update = [&](const CUtensorMap& ma, const CUtensorMap& mb, int r0, int ncols, int k0, int K,
                    const int* ex, const int* spread) -> int {
    const double* P = A + (size_t)k0 * lda + r0;
    const Fma F{P, P, 1, (size_t)lda, 1, (size_t)lda, K};
    const int TI = cdiv(n - r0, BM), TJ = cdiv(ncols, BN);
    const long long nt = tile_count(TI, TJ);
    k_oz_update<false><<<(int)std::min<long long>(8 * nt, nsm), THREADS, SMEM, s>>>(
        ma, mb, A + (size_t)r0 * lda + r0, lda, n, r0, n, r0, n - r0, ncols, K / BK, ex + r0,
        ex + r0, flat_count(K), spread, F, TI, TJ, (int)nt, std::min(PW, n - r0), r0, info, nullptr,
        g_wait_ns, hold);
    return launched();
  };
  // the first diagonal block; every update leaves the next one factored
  k_oz_diag<<<1, THREADS, diag64::SMEM, s>>>(A, lda, std::min(PW, n), 0, info, any, p.nany);
  JMG_TRY(launched());
  for (int k0 = 0; k0 < n; k0 += p.NB) {
    const int kend = std::min(k0 + p.NB, n);
    for (int k = k0; k < kend; k += PW) {
      const int kb = std::min(PW, n - k), m = n - k - kb;
      if (m <= 0) return JMG_OK;
      const int first = k == k0, last = k + PW >= kend;
      // lanes per row: enough rows per pass for the eight warps of every SM
      auto panel_solve = [&](auto kern, int rows) {
        kern<<<cdiv(m, rows), PT, 0, s>>>(A, lda, n, k, panel, e_in, rowmax, e_out, first, last,
                                          any + k / PW, info);
      };
      if (m <= 16 * nsm)
        panel_solve(k_oz_panel<16>, 16);
      else if (m <= 32 * nsm)
        panel_solve(k_oz_panel<8>, 32);
      else if (m <= 64 * nsm)
        panel_solve(k_oz_panel<4>, 64);
      else
        panel_solve(k_oz_panel<2>, 128);
      JMG_TRY(launched());
      if (k + PW < kend) JMG_TRY(update(pa, pb, k + PW, kend - (k + PW), k, PW, e_in, any + k / PW));
    }
    if (kend >= n) break;
    int* block_any = any + cdiv(n, PW) + k0 / p.NB;
    k_oz_strip<<<dim3(cdiv(n - kend, 32), p.NB / 64), 256, 0, s>>>(A, lda, n, k0, kend, p.NB,
                                                                  rowmax, strip, e_out,
                                                                  block_any, info);
    JMG_TRY(launched());
    JMG_TRY(update(oa, ob, kend, n - kend, k0, p.NB, e_out, block_any));
  }
  return JMG_OK;
}

// ---------------------------------------------------------------------------
// Solves with many right-hand sides: (L L^T) X = B, FP64.  Blocks of SK rows: the
// diagonal block by the one-launch substitution (k_trsv.cu), everything behind it by
// one tensor-core update from exact slices,
//   forward   B_rest -= L[rest, block] Y_block,
//   backward  B_rest -= L[block, rest]^T X_block,
// in place of FP64 products on the CUDA cores, which bound the one-launch solves from
// about 16 right-hand sides on.  In the backward direction row k of the block is scaled
// by 2^-sc[k] in L and 2^sc[k] in X (sc: the row's exponent), so that a badly scaled A =
// D G D costs nothing (the forward one is scaled by rows already).
namespace {
struct SolvePlan {
  int nb;
  size_t strip, exr, cols, exc, bmax, sc, any, total;
};
SolvePlan solve_plan(int n, int nrhs) {
  SolvePlan p{};
  p.nb = cdiv(n, ozf::SK);
  size_t off = 0;
  auto take = [&](size_t b) {
    const size_t at = off;
    off = round_up(off + b, 256);
    return at;
  };
  p.strip = take((size_t)ozf::S * n * ozf::SK * 2);
  p.exr = take(sizeof(int) * (size_t)n * p.nb);
  p.cols = take((size_t)ozf::S * nrhs * ozf::SK * 2);
  p.exc = take(sizeof(int) * round_up((size_t)nrhs, 64));
  p.bmax = take(sizeof(unsigned long long) * (size_t)n * p.nb);
  p.sc = take(sizeof(int) * (size_t)n);
  p.any = take(sizeof(int) * 2 * (size_t)p.nb);  // forward and backward update of each block
  p.total = off;
  return p;
}
}  // namespace

size_t ozs_workspace(int n, int nrhs) {
  // Worth it where the one-launch solves are bound by their products.  Both directions,
  // one launch each / blocked: n = 4100, 64 right-hand sides 2.74 / 2.59 ms; 8192, 33:
  // 7.25 / 5.04; 16384, 16: 10.6 / 10.9; 16384, 20: 17.9 / 10.9; 16384, 64: 35.2 / 11.1;
  // 12001, 100: 37.1 / 8.3.  Smaller orders with many right-hand sides: 600, 500 0.73 / 0.78;
  // 600, 1000 1.48 / 1.35; 1000, 100 0.44 / 0.53; 1000, 200 0.74 / 0.62; 2000, 300 3.43 / 1.62;
  // 4000, 200 8.1 / 2.8; 4000, 500 19.7 / 5.4.
  if (nrhs <= 16) return 0;
  const long long size = (long long)n * nrhs;
  const bool many = nrhs > 100 && n > ozf::SK && size >= (n < 1000 ? 600000 : 150000);
  if (!many && (n < 4096 || (n < 8192 && size < 250000))) return 0;
  return solve_plan(n, nrhs).total;
}

int solve_split(int n, int nrhs, const double* L, int lda, double* B, int ldb, int* sync,
                int* info, void* work, cudaStream_t s, int hold) {
  using namespace ozf;
  const SolvePlan p = solve_plan(n, nrhs);
  char* w = static_cast<char*>(work);
  __nv_bfloat16* strip = reinterpret_cast<__nv_bfloat16*>(w + p.strip);
  __nv_bfloat16* cols = reinterpret_cast<__nv_bfloat16*>(w + p.cols);
  int* exr = reinterpret_cast<int*>(w + p.exr);
  int* exc = reinterpret_cast<int*>(w + p.exc);
  unsigned long long* bmax = reinterpret_cast<unsigned long long*>(w + p.bmax);
  int* sc = reinterpret_cast<int*>(w + p.sc);
  int* any = reinterpret_cast<int*>(w + p.any);
  int dev = 0, nsm = 152;
  JMG_CUDA(cudaGetDevice(&dev));
  JMG_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  JMG_TRY(ensure_smem(k_oz_update<true>, SMEM));
  CUtensorMap mq;
  JMG_TRY(map_slices(&mq, cols, nrhs, SK, BN));
  k_oz_block_max<<<dim3(cdiv(n, 256), p.nb), 256, 0, s>>>(L, lda, n, bmax, exr, any);
  JMG_TRY(launched());
  k_oz_row_scale<<<cdiv(n, 256), 256, 0, s>>>(n, p.nb, bmax, sc);
  JMG_TRY(launched());
  // C (m x nrhs, head of B + row0) -= strip cols^T; strip rows rA.. of nA per slice
  auto update = [&](const CUtensorMap& mp, int nA, int rA, int row0, int m, const int* ex,
                    const int* spread, const Fma& F) -> int {
    const int TI = cdiv(m, BM), TJ = cdiv(nrhs, BN), nt = TI * TJ;
    k_oz_update<true><<<std::min(8 * nt, nsm), THREADS, SMEM, s>>>(
        mp, mq, B + row0, ldb, nA, rA, nrhs, 0, m, nrhs, SK / BK, ex, exc, flat_count(F.kv),
        spread, F, TI, TJ, nt, 0, 0, info, sync, g_wait_ns, hold);
    return launched();
  };
  CUtensorMap mp;
  JMG_TRY(map_slices(&mp, strip, n, SK, BM));
  for (int b = 0; b < p.nb; ++b) {
    const int k0 = b * SK, kb = std::min(SK, n - k0), k1 = k0 + kb;
    JMG_TRY(trsv_block(kb, nrhs, L + (size_t)k0 * lda + k0, lda, B + k0, ldb, 0, b > 0, sync,
                       info, s));
    if (k1 >= n) break;
    k_oz_strip<<<dim3(cdiv(n - k1, 32), SK / 64), 256, 0, s>>>(L, lda, n, k0, k1, SK,
                                                              bmax + (size_t)b * n, strip,
                                                              exr + (size_t)b * n, any + 2 * b,
                                                              info);
    JMG_TRY(launched());
    k_oz_cut_cols<<<cdiv(nrhs, 8), 256, 0, s>>>(B + k0, ldb, kb, nrhs, sc, 0, cols, exc,
                                                any + 2 * b);
    JMG_TRY(launched());
    JMG_TRY(update(mp, n, k1, k1, n - k1, exr + (size_t)b * n + k1, any + 2 * b,
                   Fma{L + (size_t)k0 * lda + k1, B + k0, 1, (size_t)lda, (size_t)ldb, 1, kb}));
  }
  for (int b = p.nb - 1; b >= 0; --b) {
    const int k0 = b * SK, kb = std::min(SK, n - k0);
    JMG_TRY(trsv_block(kb, nrhs, L + (size_t)k0 * lda + k0, lda, B + k0, ldb, 1, 1, sync,
                       info, s));
    if (k0 == 0) break;
    int* spread = any + 2 * b + 1;
    k_oz_cut_cols<<<cdiv(k0, 8), 256, 0, s>>>(L + k0, lda, kb, k0, sc + k0, -1, strip, exr, spread);
    JMG_TRY(launched());
    k_oz_cut_cols<<<cdiv(nrhs, 8), 256, 0, s>>>(B + k0, ldb, kb, nrhs, sc + k0, 1, cols, exc,
                                                spread);
    JMG_TRY(launched());
    CUtensorMap mt;
    JMG_TRY(map_slices(&mt, strip, k0, SK, BM));
    JMG_TRY(update(mt, k0, 0, 0, k0, exr, spread,
                   Fma{L + k0, B + k0, (size_t)lda, 1, (size_t)ldb, 1, kb}));
  }
  return JMG_OK;
}

}  // namespace jmg
