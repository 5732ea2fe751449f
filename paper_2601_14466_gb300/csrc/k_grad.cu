// k_grad.cu -- adjoint of the SPD solve X = A^{-1} B with respect to A:
//
//     Abar = -(Bbar X^T + X Bbar^T) / 2          (full symmetric, FP64)
//
// where Bbar = A^{-1} Xbar comes from the solve with the stored factor.  The
// paper exposes potrs as a primitive that composes with the framework's
// transformations ("Summary"); reverse-mode differentiation is one of them, and
// this is its matrix-calculus form for a symmetric A read from one triangle.
//
// Few right-hand sides: one CTA per 64 x 64 lower tile (ti >= tj); the rank-2 nrhs
// products run on the FP64 CUDA cores (4 x 4 register tile per thread).  The tile is written
// to (ti, tj) directly and to the mirror (tj, ti) through a shared-memory
// transpose so that both stores coalesce down columns; on diagonal tiles the
// upper half is the mirror of the lower half, so Abar is exactly symmetric.
#include "kernels.h"
#include "ozslice.cuh"
#include "tc_ptx.cuh"

namespace jmg {

namespace grad {
constexpr int TB = 64, KC = 16;
}

__global__ void __launch_bounds__(256) k_sym_grad(int n, int nrhs, const double* __restrict__ Bb,
                                                  int ldb, const double* __restrict__ X, int ldx,
                                                  double* __restrict__ G, int ldg) {
  using namespace grad;
  int ti, tj;
  tri_index(blockIdx.x, ti, tj);
  const int i0 = ti * TB, j0 = tj * TB;
  // the four K slices and, after the K loop, the output tile share one buffer
  // (4 * KC * (TB + 1) == TB * (TB + 1) doubles, 33 KB)
  __shared__ double sbuf[TB * (TB + 1)];
  double(*Bi)[TB + 1] = reinterpret_cast<double(*)[TB + 1]>(sbuf);
  double(*Xi)[TB + 1] = Bi + KC;
  double(*Bj)[TB + 1] = Bi + 2 * KC;
  double(*Xj)[TB + 1] = Bi + 3 * KC;
  double(*T)[TB + 1] = reinterpret_cast<double(*)[TB + 1]>(sbuf);
  static_assert(4 * KC == TB, "slices and tile share the buffer");
  const int t = threadIdx.x, tx = t % 16, ty = t / 16;  // rows tx + 16q, cols ty + 16p
  double acc[4][4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int p = 0; p < 4; ++p) acc[q][p] = 0.0;
  for (int k0 = 0; k0 < nrhs; k0 += KC) {
    // 4 x (64 x 16) values: 4 per thread per slice
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int idx = t + 256 * q;
      const int r = idx % TB, k = idx / TB;
      const int gk = k0 + k;
      const bool kin = gk < nrhs;
      const int gi = i0 + r, gj = j0 + r;
      Bi[k][r] = (kin && gi < n) ? Bb[(size_t)gk * ldb + gi] : 0.0;
      Xi[k][r] = (kin && gi < n) ? X[(size_t)gk * ldx + gi] : 0.0;
      Bj[k][r] = (kin && gj < n) ? Bb[(size_t)gk * ldb + gj] : 0.0;
      Xj[k][r] = (kin && gj < n) ? X[(size_t)gk * ldx + gj] : 0.0;
    }
    __syncthreads();
    const int kn = min(KC, nrhs - k0);
#pragma unroll 4
    for (int k = 0; k < kn; ++k) {
      double bi[4], xi[4], bj[4], xj[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        bi[q] = Bi[k][tx + 16 * q];
        xi[q] = Xi[k][tx + 16 * q];
        bj[q] = Bj[k][ty + 16 * q];
        xj[q] = Xj[k][ty + 16 * q];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[q][p] = fma(bi[q], xj[p], fma(xi[q], bj[p], acc[q][p]));
    }
    __syncthreads();
  }
  // (the K loop ended with a barrier, so the slices are free)
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const double v = -0.5 * acc[q][p];
      const int r = tx + 16 * q, c = ty + 16 * p;
      T[r][c] = v;
      // diagonal tiles: lower half here, the upper half is its mirror (below), so
      // the result is symmetric bit for bit
      if (i0 + r < n && j0 + c < n && (ti != tj || r >= c)) G[(size_t)(j0 + c) * ldg + i0 + r] = v;
    }
  __syncthreads();
  // mirror: G[j0 + c', i0 + r'] = T[r'][c'], written down columns i0 + r'
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int idx = t + 256 * q;
    const int c = idx % TB, r = idx / TB;  // row j0 + c of G, column i0 + r
    if (j0 + c < n && i0 + r < n && (ti != tj || r > c)) G[(size_t)(i0 + r) * ldg + j0 + c] = T[r][c];
  }
}

// ---------------------------------------------------------------------------
// The same on the tensor cores, from exact slices (k_ozpotrf.cu): 2 nrhs FP64 FMAs per
// entry hold the FP64 pipe for nrhs clocks and SM, the slices of a chunk of KC = 16
// right-hand sides cost a tile the same whatever the FP64 work.  One CTA per 128 x 64
// tile of the lower trapezoid; per chunk the two products Bbar_i X_j^T and X_i Bbar_j^T
// one after the other: stage 16 columns of both operands, cut every row into seven
// digits straight into the swizzled operand tiles, 28 slice products into seven TMEM
// levels (exact: |sum| <= 7 16 2^14 < 2^24), one conversion and one FP64 addition per
// entry.  Column k of the pair is scaled by 2^s_k and 2^-s_k first (s_k from the tile's
// column maxima), so that a pair with a large Bbar and a small X next to one with the
// opposite costs no digits.
//
// Rows of either operand that are spread all the same (ozslice.cuh) take FP64 FMAs from
// the staged columns, two rows by 16 columns of a warp at a time.  So does the whole
// product when more than a quarter of its rows are spread, in a chunk of fewer than six
// right-hand sides (sizes differ by chance there, and the FMAs are few), when an entry is
// not finite, and after a wait that ran out.
// n = 8192, 16 right-hand sides: 1829 us with FMAs alone -> 735 (a tile's phases, not
// pipelined, take ~26 us; the 537 MB written would take 80), error against 64 bits 0.4 of
// the FMAs'; 2100 when next to every row is spread (128 x 64 tiles, one CTA per SM).
namespace grad {
constexpr int BM = 128, BN = 64, TH = 512;
constexpr int A_TILE = BM * 128, B_TILE = BN * 128;  // rows of 128 bytes, 16 BF16 of them used
constexpr int LDT = BM + 1;
constexpr int SMEM = ozf::S * (A_TILE + B_TILE) + KC * (BM + BN) * 8 + 1024;
static_assert(BN * LDT * 8 <= ozf::S * A_TILE, "the output tile lies over the operand tiles");
}  // namespace grad

__global__ void __launch_bounds__(grad::TH, 1)
    k_sym_grad_tc(int n, int nrhs, const double* __restrict__ Bb, int ldb,
                  const double* __restrict__ X, int ldx, double* __restrict__ G, int ldg,
                  unsigned long long wait_ns, int hold) {
  using namespace grad;
  using namespace tc;
  using ozf::S;
  extern __shared__ __align__(1024) unsigned char sm_raw_grad[];
  unsigned char* abuf = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(sm_raw_grad) + 1023) & ~uintptr_t(1023));
  unsigned char* bbuf = abuf + S * A_TILE;
  double* sP = reinterpret_cast<double*>(bbuf + S * B_TILE);  // [KC][BM]
  double* sQ = sP + KC * BM;                                  // [KC][BN]
  __shared__ uint64_t bar, drain;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_ep[BM], s_eq[BN], s_k[KC];  // rows' exponents (2 e + spread), column shifts
  const int t = threadIdx.x, warp = t / 32, lane = t % 32;
  // tile b: row tile ti has the column tiles 0 .. 2 ti + 1
  int ti = (int)((sqrtf(4.0f * (float)blockIdx.x + 1.0f) - 1.0f) * 0.5f);
  while ((long long)ti * (ti + 1) > (long long)blockIdx.x) --ti;
  while ((long long)(ti + 1) * (ti + 2) <= (long long)blockIdx.x) ++ti;
  const int tj = (int)(blockIdx.x - (long long)ti * (ti + 1));
  const int i0 = ti * BM, j0 = tj * BN;
  if (j0 >= n) return;
  if (t == 0) {
    mbar_init(&bar, 1);
    mbar_init(&drain, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(&tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  constexpr int CW = 16;
  const int q = warp & 3, ch = (warp >> 2) * CW;  // TMEM lane quarter, columns of this warp
  const int r = q * 32 + lane;
  double v[CW];
#pragma unroll
  for (int c = 0; c < CW; ++c) v[c] = 0.0;
  bool ok = true;  // uniform over the CTA
  uint32_t phase = 0;
  for (int k0 = 0; k0 < nrhs; k0 += KC) {
    const int kn = min(KC, nrhs - k0);
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      const double* P = half ? X : Bb;
      const double* Q = half ? Bb : X;
      const int ldp = half ? ldx : ldb, ldq = half ? ldb : ldx;
      bool fin = true;
      {
        double a[6];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int k = t / BM + 4 * u, gi = i0 + t % BM;
          a[u] = (k0 + k < nrhs && gi < n) ? P[(size_t)(k0 + k) * ldp + gi] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int k = t / BN + 8 * u, gj = j0 + t % BN;
          a[4 + u] = (k0 + k < nrhs && gj < n) ? Q[(size_t)(k0 + k) * ldq + gj] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 6; ++u)
          fin = fin && ((unsigned)__double2hiint(a[u]) & 0x7ff00000u) != 0x7ff00000u;
#pragma unroll
        for (int u = 0; u < 4; ++u) sP[(t / BM + 4 * u) * BM + t % BM] = a[u];
#pragma unroll
        for (int u = 0; u < 2; ++u) sQ[(t / BN + 8 * u) * BN + t % BN] = a[4 + u];
      }
      bool slices = __syncthreads_and(fin) && ok && kn >= 6;
      if (slices) {
        {  // column k = warp: shift by half the difference of the maxima's exponents
          unsigned mp = 0, mq = 0;
#pragma unroll
          for (int u = 0; u < BM / 32; ++u)
            mp = max(mp, (unsigned)__double2hiint(sP[warp * BM + lane + 32 * u]) & 0x7fffffffu);
#pragma unroll
          for (int u = 0; u < BN / 32; ++u)
            mq = max(mq, (unsigned)__double2hiint(sQ[warp * BN + lane + 32 * u]) & 0x7fffffffu);
          mp = __reduce_max_sync(0xffffffffu, mp);
          mq = __reduce_max_sync(0xffffffffu, mq);
          if (lane == 0) s_k[warp] = ((int)(mq >> 20) - (int)(mp >> 20)) / 2;
        }
        __syncthreads();
        // eight values of a row of P (t < 256) or Q (t < 384)
        const bool isq = t >= 2 * BM;
        const int w = isq ? t - 2 * BM : t, row = w / 2, h = 8 * (w & 1);
        double x[8];
        int sk[8], e = -(1 << 20);
        bool spread = false;
        if (t < 2 * (BM + BN)) {
          const double* src = isq ? sQ + row : sP + row;
          const int ld = isq ? BN : BM;
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            x[u] = src[(h + u) * ld];
            sk[u] = isq ? -s_k[h + u] : s_k[h + u];
            const unsigned long long b =
                (unsigned long long)__double_as_longlong(x[u]) & 0x7FFFFFFFFFFFFFFFull;
            if (b) e = max(e, max((int)(b >> 52), 1) - 1022 + sk[u]);
          }
          e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
          int near = 0;  // entries near the row's largest (subnormal ones never)
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int f = (__double2hiint(x[u]) >> 20) & 0x7FF;
            near += f > 0 && f - 1022 + sk[u] + ozf::NEAR >= e;
          }
          near += __shfl_xor_sync(0xffffffffu, near, 1);
          spread = e > -(1 << 20) && near < ozf::flat_count(kn);
          if (h == 0) (isq ? s_eq : s_ep)[row] = 2 * e + (spread ? 1 : 0);
        }
        slices = __syncthreads_count(spread) <= (BM + BN) / 2;  // (two threads per row)
        if (slices && t < 2 * (BM + BN)) {
          uint32_t d4[S][4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            int d0[S], d1[S];
            ozf::digits7(x[2 * u], e - sk[2 * u], d0);
            ozf::digits7(x[2 * u + 1], e - sk[2 * u + 1], d1);
#pragma unroll
            for (int s = 0; s < S; ++s) {
              const __nv_bfloat162 p = __floats2bfloat162_rn((float)d0[s], (float)d1[s]);
              d4[s][u] = *reinterpret_cast<const uint32_t*>(&p);
            }
          }
          unsigned char* dst = (isq ? bbuf : abuf) + row * 128 + (((h >> 3) ^ (row & 7)) << 4);
          const int tile = isq ? B_TILE : A_TILE;
#pragma unroll
          for (int s = 0; s < S; ++s)
            *reinterpret_cast<uint4*>(dst + s * tile) =
                make_uint4(d4[s][0], d4[s][1], d4[s][2], d4[s][3]);
          fence_proxy_async();
        }
      }
      if (slices) {
        tc_fence_before();
        __syncthreads();
        if (t == 0 && !hold) {  // (hold, a test hook: no products, the wait below runs out)
          tc_fence_after();
          constexpr int GMAX = 256 / BN;
          for (int a = 0; a < S; ++a)
            for (int b0 = 0; b0 < S - a; b0 += GMAX) {
              const int cnt = min(GMAX, S - a - b0);
              tc_mma_f16(tmem + (uint32_t)((a + b0) * BN), sdesc_sw128(smem_u32(abuf + a * A_TILE)),
                         sdesc_sw128(smem_u32(bbuf + b0 * B_TILE)), idesc_f16(BM, BN * cnt, 1),
                         a == 0 ? 0u : 1u);
            }
          tc_commit(&bar);
        }
        __syncwarp();
        ok = __syncthreads_and(mbar_wait(&bar, phase, wait_ns));
        phase ^= 1;
      }
      if (slices && ok) {
        tc_fence_after();
        const uint32_t tacc = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)ch;
        constexpr int sh = 40;
        long long acc[CW];
#pragma unroll
        for (int c = 0; c < CW; ++c) acc[c] = 0;
#pragma unroll
        for (int d = 0; d < S; ++d) {
          uint32_t w[16];
          tmem_ld16(tacc + (uint32_t)(d * BN), w);
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < CW; ++c) {
            const long long y = __float2int_rn(__uint_as_float(w[c]));
            acc[c] += d < 6 ? y << (sh - 8 * (d < 6 ? d : 0)) : (y + (1 << 7)) >> 8;
          }
        }
        const int er = s_ep[r];
        const unsigned cols = __ballot_sync(0xffffffffu, lane < CW && (s_eq[ch + (lane & 15)] & 1));
        unsigned rows = __ballot_sync(0xffffffffu, er & 1);  // spread ones of this warp
#pragma unroll
        for (int c = 0; c < CW; ++c)
          if (!(er & 1) && !(cols >> c & 1u))
            v[c] += ozf::scaled_double(acc[c], (er >> 1) + (s_eq[ch + c] >> 1) - 14 - sh);
        if (cols)
          for (int k = 0; k < kn; ++k) {
            const double x = sP[k * BM + r];
#pragma unroll
            for (int c = 0; c < CW; ++c)
              if (cols >> c & 1u) v[c] = fma(x, sQ[k * BN + ch + c], v[c]);
          }
        while (rows) {  // lanes 0-15: columns of row r0, lanes 16-31: of row r1
          const int r0 = __ffs(rows) - 1;
          rows &= rows - 1;
          const int r1 = rows ? __ffs(rows) - 1 : r0;
          rows &= rows - 1;
          const double* p = sP + q * 32 + (lane < 16 ? r0 : r1);
          const double* x = sQ + ch + (lane & 15);
          double s = 0.0;
          for (int k = 0; k < kn; ++k) s = fma(p[k * BM], x[k * BN], s);
#pragma unroll
          for (int c = 0; c < CW; ++c) {
            const double y = __shfl_sync(0xffffffffu, s, lane == r0 ? c : 16 + c);
            if ((lane == r0 || lane == r1) && !(cols >> c & 1u)) v[c] += y;
          }
        }
      } else {
        for (int k = 0; k < kn; ++k)
#pragma unroll
          for (int c = 0; c < CW; ++c) v[c] = fma(sP[k * BM + r], sQ[k * BN + ch + c], v[c]);
      }
      tc_fence_before();
      __syncthreads();  // accumulators and staged columns are free
    }
  }
  if (!ok && t == 0) mma_drain(&drain, wait_ns);  // the products still under way
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 512);
  const int row = i0 + r;
  double* T = reinterpret_cast<double*>(abuf);  // T[c * LDT + r]
#pragma unroll
  for (int c = 0; c < CW; ++c) {
    const double g = -0.5 * v[c];
    const int col = j0 + ch + c;
    T[(ch + c) * LDT + r] = g;
    if (row < n && col <= row) G[(size_t)col * ldg + row] = g;
  }
  __syncthreads();
  for (int i = warp; i < BM; i += TH / 32)  // column i0 + i of G, rows j0 ..
#pragma unroll
    for (int h = 0; h < BN; h += 32) {
      const int col = i0 + i, gj = j0 + h + lane;
      if (col < n && gj < col) G[(size_t)col * ldg + gj] = T[(h + lane) * LDT + i];
    }
}

int launch_sym_grad(int n, int nrhs, const double* Bb, int ldb, const double* X, int ldx, double* G,
                    int ldg, cudaStream_t s, int hold) {
  if (n <= 0) return JMG_OK;
  if (nrhs <= 0) {
    JMG_CUDA(cudaMemset2DAsync(G, sizeof(double) * ldg, 0, sizeof(double) * n, n, s));
    return JMG_OK;
  }
  // FP64 work grows with nrhs, a chunk on the tensor cores costs about the same from 6 to
  // 16 (a little more with few, where more rows are spread by chance): n = 8192 nrhs 6 744
  // / 830 us, 7 860 / 750, 8 970 / 790; n = 2048 6 60 / 75, 8 77 / 69; one wave of tiles (n
  // <= 1024) 11 31 / 32, 8 24 / 32.
  if (nrhs >= (n <= 1024 ? 12 : 7)) {
    using namespace grad;
    JMG_TRY(ensure_smem(k_sym_grad_tc, SMEM));
    const long long TI = cdiv(n, BM);
    k_sym_grad_tc<<<(unsigned)(TI * (TI + 1)), TH, SMEM, s>>>(n, nrhs, Bb, ldb, X, ldx, G, ldg,
                                                             g_wait_ns, hold);
    return launched();
  }
  k_sym_grad<<<(unsigned)tri_tiles(cdiv(n, grad::TB)), 256, 0, s>>>(n, nrhs, Bb, ldb, X, ldx, G,
                                                                      ldg);
  return launched();
}

}  // namespace jmg
