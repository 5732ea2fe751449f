// k_ozpotrf.cu -- FP64 Cholesky factorisation with its trailing updates on the
// BF16 tensor cores, by error-free splitting (Ozaki, Ogita, Oishi and Rump 2012,
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
// subtraction from C end the update.  Against the FP64 CUDA-core update this
// keeps the same 2^-53 relative to the rows of P and rounds C once per update
// instead of once per product: over random Gram matrices of order 100 .. 3000 the
// factor's error is 0.8-0.95 of the CUDA-core route's.
//
// Two-level right-looking blocking: panels of 64 columns inside blocks of NB = 512,
// one update of the block's remaining columns per panel (depth 64) and one of the
// whole trailing matrix per block (depth 512, sliced again with one exponent per
// row over the block).  Factor alone on one GB300, before -> now: n = 1024
// 3.66 -> 1.92 ms, 3000 18.6 -> 6.1, 5000 53 -> 11.2, 16384 1260 -> 84 ms (there the
// tensor cores do 28 products of slices for one of FP64: 490 TFLOP/s over the
// whole factorisation).
#include <algorithm>

#include "kernels.h"
#include "tc_ptx.cuh"

namespace jmg {
namespace ozf {
constexpr int S = 7;           // slices per operand
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
constexpr int GROUP = 8;             // row tiles per raster group
constexpr int E_BAD = 1 << 20;       // exponent of a row that is not finite

// exponent e with |x| 2^-e < 1 for every |x| <= m (m as the bits of |x|);
// 0 for m == 0, E_BAD for infinities and NaN
JMG_DEV int scale_exp_bits(unsigned long long mb) {
  if (mb == 0) return 0;
  const int ex = (int)(mb >> 52);
  if (ex >= 0x7FF) return E_BAD;
  if (ex) return ex - 1022;
  return -1010 - __clzll((long long)mb);  // subnormal: m = mb 2^-1074, mb < 2^(64-clz)
}

// The digits of x 2^-e (|x 2^-e| < 1): V = rint(x 2^(55-e)), |V| <= 2^55, cut into
// balanced base-256 digits from the bottom; integer operations only.
JMG_DEV void digits7(double x, int e, int (&d)[S]) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  int ex = (int)((b >> 52) & 0x7FF);
  unsigned long long M = b & ((1ull << 52) - 1);
  if (ex)
    M |= 1ull << 52;
  else
    ex = 1;
  const int sh = ex - 1020 - e;  // V = M 2^sh
  unsigned long long V = 0;
  if (sh >= 0) {
    V = sh <= 60 ? M << sh : 0ull;  // (below 2^55 for every finite row; subnormals shift far)
  } else if (sh > -64) {
    const int k = -sh;
    V = (M >> k) + ((M >> (k - 1)) & 1ull);  // to nearest, ties away
  }
  long long W = (b >> 63) ? -(long long)V : (long long)V;
#pragma unroll
  for (int s = S - 1; s >= 1; --s) {
    const int k = (int)(signed char)(W & 255);
    d[s] = k;
    W = (W - k) >> 8;
  }
  d[0] = (int)W;  // |W| <= 128
}

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

// c - v 2^ex with one FP64 subtraction: v is rounded once to FP64 and its
// exponent field is moved by integer addition where it stays normal.
JMG_DEV double sub_scaled(double c, long long v, int ex) {
  if (v == 0) return c;
  double d = (double)v;
  const int E = ((__double2hiint(d) >> 20) & 0x7FF) + ex;
  if (E > 0 && E < 0x7FF)
    d = __hiloint2double(__double2hiint(d) + (ex << 20), __double2loint(d));
  else
    d = ldexp(d, ex);
  return c - d;
}

// C (rows and columns from r0 on, columns below r0 + ncols, lower part) -=
// P P^T, P given by its slices: row r of slice s is row s * n + r of the map.
__global__ void __launch_bounds__(THREADS, 1)
    k_oz_syrk(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              double* __restrict__ C, int ldc, int n, int r0, int ncols, int nkb,
              const int* __restrict__ ex, int TI, int TJ, int ntiles, int* __restrict__ info,
              unsigned long long wait_ns) {
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
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acce + 1);
  __shared__ int s_fail, s_info;

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    s_fail = 0;
    s_info = *(volatile int*)info;
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
    fence_mbar_init();
    prefetch_tmap(&tmA);
    prefetch_tmap(&tmB);
  }
  __syncthreads();
  if (s_info != 0) return;  // an earlier block already failed
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
    if (lane == 0) {
      bool ok = true;
      for (int b = blockIdx.x; b < ntiles && ok; b += gridDim.x) {
        int ti, tj;
        if (!tile_of(b, TI, TJ, ti, tj)) continue;
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
            tma_load_2d(bbuf + bs * B_BUF + s * B_TILE, &tmB, kb * BK, s * n + r0 + tj * BN,
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
            tma_load_2d(abuf + st * A_TILE, &tmA, kb * BK, s * n + r0 + ti * BM, &afull[st]);
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
      for (int b = blockIdx.x; b < ntiles && ok; b += gridDim.x) {
        int ti, tj;
        if (!tile_of(b, TI, TJ, ti, tj)) continue;
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
    for (int b = blockIdx.x; b < ntiles && ok; b += gridDim.x) {
      int ti, tj;
      if (!tile_of(b, TI, TJ, ti, tj)) continue;
      const int row = r0 + ti * BM + q * 32 + lane;
      const int c0 = r0 + tj * BN + ch;
      // columns c < jn of this thread are in range and on or below the diagonal
      const int jn = row < n ? min(CW, min(r0 + ncols - c0, row - c0 + 1)) : 0;
      unsigned long long acc[CW];  // (unsigned: rows and columns past the end wrap, never trap)
#pragma unroll
      for (int c = 0; c < CW; ++c) acc[c] = 0ull;
      for (int kw = 0; kw < nkb; kw += WIN, ++gw) {
        if (!mbar_wait(accf, (uint32_t)gw & 1, wait_ns) || ld_shared_volatile(&s_fail)) {
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
      if (jn > 0) {
        double* cp = C + (size_t)c0 * ldc + row;
        const int er = ex[row];
        double old[CW];
#pragma unroll
        for (int c = 0; c < CW; ++c) old[c] = c < jn ? cp[(size_t)c * ldc] : 0.0;
#pragma unroll
        for (int c = 0; c < CW; ++c)
          if (c < jn) {
            const int ec = ex[c0 + c];
            double r = sub_scaled(old[c], (long long)acc[c], er + ec - 14 - sh);
            if (er == E_BAD || ec == E_BAD) r = __longlong_as_double(0x7FF8000000000000ll);
            cp[(size_t)c * ldc] = r;
          }
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
      atomicCAS(info, 0, -1);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, TCOLS);
}

// ---------------------------------------------------------------------------
// Panel solve X L_kk^T = A21 (64 columns) and its slices.  G lanes share a row,
// each holding the column pairs {2 (g + G i), 2 (g + G i) + 1}; the FP64 pipe
// takes one warp instruction per ~64 clocks and SM quarter, so the row is spread
// over just enough lanes to fill the chip.  The solve runs on unscaled columns
// with Lh[j][l] = L_lj / L_jj (a_l -= a_j Lh[j][l]), the scaling by 1 / L_jj
// comes last: one FP64 instruction per element and step, nothing else.
template <int G>
__global__ void __launch_bounds__(128) k_oz_panel(double* __restrict__ A, int lda, int n, int k,
                                                  __nv_bfloat16* __restrict__ SP,
                                                  int* __restrict__ ex,
                                                  unsigned long long* __restrict__ rowmax,
                                                  int first, const int* __restrict__ info) {
  constexpr int NP = 32 / G;     // column pairs per lane
  constexpr int RW = 32 / G;     // rows per warp
  constexpr int RB = 4 * RW;     // rows per CTA
  __shared__ __align__(16) double Lh[PW * PW];
  __shared__ double rinv[PW];
  if (*(volatile const int*)info != 0) return;
  const int t = threadIdx.x, lane = t % 32, warp = t / 32;
  const double* Lkk = A + (size_t)k * lda + k;
  {
    double v[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const int idx = t + 128 * i, l = idx % PW, j = idx / PW;
      v[i] = l >= j ? Lkk[(size_t)j * lda + l] : 0.0;
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) Lh[t + 128 * i] = v[i];
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
  for (int i = 0; i < 32; ++i) {
    const int idx = t + 128 * i, l = idx % PW, j = idx / PW;
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
  if (row >= n) return;
  const int e = scale_exp_bits(mx);
  if (g == 0) {
    ex[row] = e;
    rowmax[row] = first ? mx : (mx > rowmax[row] ? mx : rowmax[row]);
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
// exponent per row over the whole block.  grid = (32-row tiles, K / 64).
__global__ void __launch_bounds__(256) k_oz_strip(const double* __restrict__ A, int lda, int n,
                                                  int k0, int r0, int K,
                                                  const unsigned long long* __restrict__ rowmax,
                                                  __nv_bfloat16* __restrict__ SP,
                                                  int* __restrict__ ex,
                                                  const int* __restrict__ info) {
  __shared__ double T[64][33];
  if (*(volatile const int*)info != 0) return;
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
  if (row >= n) return;
  const int e = scale_exp_bits(rowmax[row]);
  if (kc == 0 && cc == 0) ex[row] = e;
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
  size_t panel, strip, exp_in, exp_out, rowmax, total;
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
  p.total = off;
  return p;
}
}  // namespace

size_t ozf_workspace(int n) { return n > ozf::PW ? ozf_plan(n).total : 0; }

int potrf_split(int n, double* A, int lda, int* info, void* work, cudaStream_t s) {
  using namespace ozf;
  const OzfPlan p = ozf_plan(n);
  char* w = static_cast<char*>(work);
  __nv_bfloat16* panel = reinterpret_cast<__nv_bfloat16*>(w + p.panel);
  __nv_bfloat16* strip = reinterpret_cast<__nv_bfloat16*>(w + p.strip);
  int* e_in = reinterpret_cast<int*>(w + p.exp_in);
  int* e_out = reinterpret_cast<int*>(w + p.exp_out);
  unsigned long long* rowmax = reinterpret_cast<unsigned long long*>(w + p.rowmax);
  int dev = 0, nsm = 152;
  JMG_CUDA(cudaGetDevice(&dev));
  JMG_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  JMG_TRY(ensure_smem(k_oz_syrk, SMEM));
  CUtensorMap pa, pb, oa, ob;
  JMG_TRY(map_slices(&pa, panel, n, PW, BM));
  JMG_TRY(map_slices(&pb, panel, n, PW, BN));
  if (n > p.NB) {
    JMG_TRY(map_slices(&oa, strip, n, p.NB, BM));
    JMG_TRY(map_slices(&ob, strip, n, p.NB, BN));
  }
  auto update = [&](const CUtensorMap& ma, const CUtensorMap& mb, int r0, int ncols, int nkb,
                    const int* ex) -> int {
    const int TI = cdiv(n - r0, BM), TJ = cdiv(ncols, BN);
    const long long nt = tile_count(TI, TJ);
    k_oz_syrk<<<(int)std::min<long long>(nt, nsm), THREADS, SMEM, s>>>(
        ma, mb, A, lda, n, r0, ncols, nkb, ex, TI, TJ, (int)nt, info, g_wait_ns);
    return launched();
  };
  for (int k0 = 0; k0 < n; k0 += p.NB) {
    const int kend = std::min(k0 + p.NB, n);
    for (int k = k0; k < kend; k += PW) {
      const int kb = std::min(PW, n - k), m = n - k - kb;
      JMG_TRY(launch_potf2(A + (size_t)k * lda + k, lda, kb, k, info, s));
      if (m <= 0) return JMG_OK;
      const int first = k == k0;
      // lanes per row: enough rows per pass for the 4 quarters of every SM
      if (m <= 32 * nsm)
        k_oz_panel<4><<<cdiv(m, 32), 128, 0, s>>>(A, lda, n, k, panel, e_in, rowmax, first, info);
      else if (m <= 64 * nsm)
        k_oz_panel<2><<<cdiv(m, 64), 128, 0, s>>>(A, lda, n, k, panel, e_in, rowmax, first, info);
      else
        k_oz_panel<1><<<cdiv(m, 128), 128, 0, s>>>(A, lda, n, k, panel, e_in, rowmax, first, info);
      JMG_TRY(launched());
      if (k + PW < kend) JMG_TRY(update(pa, pb, k + PW, kend - (k + PW), 1, e_in));
    }
    if (kend >= n) break;
    k_oz_strip<<<dim3(cdiv(n - kend, 32), p.NB / 64), 256, 0, s>>>(A, lda, n, k0, kend, p.NB,
                                                                  rowmax, strip, e_out, info);
    JMG_TRY(launched());
    JMG_TRY(update(oa, ob, kend, n - kend, p.NB / 64, e_out));
  }
  return JMG_OK;
}

}  // namespace jmg
