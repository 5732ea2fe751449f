// potrf_diag.cuh -- the diagonal-block factorisation as a device function of one CTA,
// for kernels that factor a block behind an update of it (k_dense.cu, k_tc.cu).
#pragma once
#include "kernels.h"

namespace jmg {

// ============================================================================
// Diagonal-block factorisation L_kk L_kk^T = A_kk (kb <= 128), in place, as a
// blocked right-looking Cholesky over 32-column sub-blocks, one CTA:
//
//  1. the 32 x 32 diagonal sub-block is factored in FP64 whatever the storage
//     type T (double for the plain path, float for the FP32 working matrix of
//     the mixed path).  Its 528 lower elements sit in shared memory as FP64;
//     step j applies a_rc -= a_rj * a_cj / a_jj (= l_rj * l_cj) to every
//     element with c > j, handing the trailing triangle's elements (a range of
//     the packed column-major order) to consecutive threads so that FP64 work
//     is issued by full warps only; each column costs one barrier.  The owner
//     of a_(j+1)(j+1) forms 1 / a_(j+1)(j+1) in step j, the only operation on
//     the serial chain besides the updates (exact for the plain path; an FP32
//     seed plus one step of Newton's method for the mixed path, whose output is
//     rounded to FP32 anyway); sqrt(a_jj) and its reciprocal follow after the
//     last column;
//  2. the rows of the block below it solve x L_qq^T = a (triangular solve, one
//     thread per row, in T);
//  3. the rest of the block takes the symmetric rank-32 update C -= X X^T (in
//     T, 4 x 4 register tiles).
//
// In the mixed path only step 1 runs in FP64: steps 2 and 3 are the panel's
// share of the trailing update, which the tensor-core path rounds further
// anyway, and FP64 runs at 1/64 of the FP32 rate on this GPU.  A pivot that is
// not > 0 (or NaN) records info = koff + j + 1; the columns before it are
// written, the rest keep their input.
// ============================================================================
namespace pdiag {
constexpr int KB = 128;                  // largest diagonal block
constexpr int BS = 32;                   // FP64 sub-block
constexpr int TH = 256;
constexpr int LD = KB + 4;               // shared leading dimension: 16-byte aligned columns
constexpr int NEL = BS * (BS + 1) / 2;   // lower elements of a sub-block
static_assert(TH == 256, "the FP64 step's warp roles and its named barrier (224 threads) assume 8 warps");

// 1/d to about 44 bits for positive normal d with |log2 d| <= 100: the leading
// bits of d as an FP32 number (exponent rebiased, mantissa truncated, with
// integer operations that stay off the FP64 pipe, where a conversion costs as
// much as an FMA), rcp.approx on it, the FP32 result widened the same way, and
// one step of Newton's method for 1/d in FP64.
JMG_DEV double rcp_seeded(double d) {
  const int hi = __double2hiint(d);
  const unsigned lo = (unsigned)__double2loint(d);
  const int fb = ((((hi >> 20) & 0x7ff) - 896) << 23) | ((hi & 0xfffff) << 3) | (int)(lo >> 29);
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__int_as_float(fb)));
  const int yb = __float_as_int(y);
  const double y0 =
      __hiloint2double(((((yb >> 23) & 0xff) + 896) << 20) | ((yb & 0x7fffff) >> 3), (yb & 7) << 29);
  return fma(y0, fma(-d, y0, 1.0), y0);
}

// 1 / d for the updates of step j (exact division for the plain path; for the
// mixed path the seeded Newton step above, whose result is rounded to FP32
// anyway).  Only this reciprocal sits on the serial chain of the steps; sqrt(d)
// is taken after the last step.  *bad is set when d is not positive (or NaN);
// the result is then finite garbage or non-finite, never a trap.
JMG_DEV double pivot_w(double d, bool exact, bool* bad) {
  const int hi = __double2hiint(d), e = (hi >> 20) & 0x7ff;
  if (!exact && hi >= 0 && e >= 1023 - 100 && e <= 1023 + 100) return rcp_seeded(d);
  *bad = !(d > 0.0);
  return 1.0 / d;
}

template <typename T>
JMG_DEV void load4(const T* p, T (&v)[4]);
template <>
JMG_DEV void load4<float>(const float* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
}
template <>
JMG_DEV void load4<double>(const double* p, double (&v)[4]) {
  const double2 q0 = reinterpret_cast<const double2*>(p)[0];
  const double2 q1 = reinterpret_cast<const double2*>(p)[1];
  v[0] = q0.x, v[1] = q0.y, v[2] = q1.x, v[3] = q1.y;
}
}  // namespace pdiag

// LOADED: the block's lower part is in shared memory already (in the layout below; the
// caller's barrier lies between), A is only written.
template <typename T, bool LOADED = false>
JMG_DEV void potrf_diag_body(T* __restrict__ A, int lda, int kb, int koff,
                             int* __restrict__ info) {
  using namespace pdiag;
  extern __shared__ __align__(16) unsigned char sm_diag[];
  T* sa = reinterpret_cast<T*>(sm_diag);  // kb columns, LD apart: sa[c * LD + r] = a_rc
  __shared__ double s_l[BS], s_il[BS], s_u[2][BS];
  __shared__ T s_rinv[BS];
  __shared__ int fail;
  constexpr bool kExact = sizeof(T) == 8;
  const int t = threadIdx.x;
  if (t == 0) fail = *(volatile int*)info;  // one read, so every thread takes the same exit
  __syncthreads();
  if (fail != 0) return;  // an earlier block already failed
  for (int base = 0; !LOADED && base < kb * kb; base += TH * 16) {  // 16 independent loads per thread
    T v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int idx = base + t + TH * q;
      const int i = idx % kb, j = idx / kb;
      v[q] = (idx < kb * kb && i >= j) ? A[(size_t)j * lda + i] : T(0);
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int idx = base + t + TH * q;
      if (idx < kb * kb) sa[(idx / kb) * LD + idx % kb] = v[q];
    }
  }
  // packed column-major lower order of a sub-block: element e <-> (row, column)
  __shared__ unsigned short s_rc[NEL];
  __shared__ double s64[BS * (BS + 1)];  // the FP64 sub-block: s64[c * (BS+1) + r]
  for (int e = t; e < NEL; e += TH) {
    int r = e, c = 0;
    while (r >= BS - c) r -= BS - c++;
    s_rc[e] = (unsigned short)((c << 8) | (c + r));
  }
  __syncthreads();

  for (int p = 0; p < kb; p += BS) {
    const int bs = min(BS, kb - p);
    // ---- 1. FP64 factor of the sub-block.  Step j updates every element
    // (r, c), c > j, of the trailing triangle: a_rc -= a_rj u_c with
    // u_c = a_cj w_j, w_j = 1/a_jj.  A warp-wide FP64 instruction occupies its
    // SM sub-partition's FP64 pipe for ~64 cycles whatever the active lanes,
    // and the pivots form a serial chain, so the work is split by warp and
    // the chain runs one column ahead of the rest:
    //  * warp 0 (the chain) keeps column j and w_j in registers (one lane per
    //    row); in step j it forms u, hands it to the trailing warps (named
    //    barrier U), finishes column j+1 (its update by column j) and takes
    //    pivot j+1 on every lane;
    //  * warps 1-3 and 5-7 (trailing) take u_j and update column j+2 first,
    //    release it (named barrier Y: the chain's input of step j+1), then
    //    the columns j+3.. (packed indices on consecutive threads);
    //  * warp 4, which shares warp 0's FP64 pipe, stays out.
    // The last step has no work, so both sides run steps 0..bs-2.  Each
    // barrier is passed the same number of times on both sides (U: bs-1,
    // Y: bs-2), and every arrival waits, through the other barrier, for the
    // other side to have passed the previous instance, so no instance can
    // count an arrival meant for the next.  Nothing leaves the loop early: a
    // pivot that is not positive is recorded (the first one wins) and the
    // columns from it on are dropped after the loop.  u alternates between
    // two buffers; the chain writes buffer j&1 only after passing Y of step
    // j-1, i.e. after the trailing warps have finished step j-2.
    for (int e = t; e < NEL; e += TH) {
      const int rc = s_rc[e], c = rc >> 8, r = rc & 255;
      if (r < bs) s64[c * (BS + 1) + r] = (double)sa[(p + c) * LD + p + r];
    }
    __syncthreads();
    const int warp = t >> 5, lane = t & 31;
    if (warp == 0) {
      const bool row = lane < bs;
      double colj = row ? s64[lane] : 0.0;  // column 0
      bool bad = false;
      double w = pivot_w(__shfl_sync(0xffffffffu, colj, 0), kExact, &bad);
      int fj = bad ? 0 : -1;  // first failing column of the sub-block
      for (int j = 0; j + 1 < bs; ++j) {
        const bool own = row && lane > j;  // rows below the diagonal of column j
        __syncwarp();
        if (j > 0) asm volatile("bar.sync 2, 224;" ::: "memory");  // column j+1 done to j-1
        double nxt = own ? s64[(j + 1) * (BS + 1) + lane] : 0.0;
        const double u = own ? colj * w : 0.0;
        if (own) s_u[j & 1][lane] = u;
        __syncwarp();
        asm volatile("bar.arrive 1, 224;" ::: "memory");
        nxt = fma(-colj, __shfl_sync(0xffffffffu, u, j + 1), nxt);
        if (own) s64[(j + 1) * (BS + 1) + lane] = nxt;
        bad = false;
        const double wn = pivot_w(__shfl_sync(0xffffffffu, nxt, j + 1), kExact, &bad);
        if (bad && fj < 0) fj = j + 1;
        colj = nxt;
        w = wn;
      }
      if (lane == 0 && fj >= 0) fail = p + fj + 1;
    } else if (warp != 4) {
      const int tq = warp < 4 ? t - 32 : t - 64;  // index among the trailing warps
      for (int j = 0; j + 1 < bs; ++j) {
        __syncwarp();
        asm volatile("bar.sync 1, 224;" ::: "memory");  // u_j and column j in place
        const double* cj = &s64[j * (BS + 1)];
        const double* uj = s_u[j & 1];
        if (j + 2 < bs) {
          if (tq >= j + 2 && tq < bs) {
            double* c2 = &s64[(j + 2) * (BS + 1)];
            c2[tq] = fma(-cj[tq], uj[j + 2], c2[tq]);
          }
          __syncwarp();
          asm volatile("bar.arrive 2, 224;" ::: "memory");
        }
        // first packed index of column j+3: sum of the column lengths before it
        const int c3 = j + 3;
        const int e3 = c3 >= BS ? NEL : c3 * BS - c3 * (c3 - 1) / 2;
        for (int e = e3 + tq; e < NEL; e += TH - 64) {
          const int rc = s_rc[e], c = rc >> 8, r = rc & 255;
          if (r >= bs) continue;
          s64[c * (BS + 1) + r] = fma(-cj[r], uj[c], s64[c * (BS + 1) + r]);
        }
      }
    }
    __syncthreads();
    const int jdone = fail ? fail - 1 - p : bs;  // columns of the sub-block that are final
    // L of the sub-block: l_cc = sqrt(a_cc), l_rc = a_rc / l_cc
    if (t < jdone) {
      const int c = t;
      const double a = s64[c * (BS + 1) + c];
      double l, il;
      if (kExact || a < 1e-30) {
        l = sqrt(a);
        il = 1.0 / l;
      } else {
        const double y0 = (double)rsqrtf((float)a);
        il = y0 * fma(-0.5 * a, y0 * y0, 1.5);  // one Newton step for d^{-1/2}
        l = a * il;
      }
      s_l[c] = l;
      s_il[c] = il;
    }
    __syncthreads();
    for (int e = t; e < NEL; e += TH) {
      const int rc = s_rc[e], c = rc >> 8, r = rc & 255;
      if (r < bs && c < jdone) {
        const T v = (T)(r == c ? s_l[c] : s64[c * (BS + 1) + r] * s_il[c]);
        sa[(p + c) * LD + p + r] = v;
        A[(size_t)(p + c) * lda + p + r] = v;
        if (r == c) s_rinv[c] = kExact ? (T)s_il[c] : (T)__frcp_rn((float)v);
      }
    }
    if (jdone < bs) break;  // (uniform: every thread read the same flag after the barrier)
    const int mr = kb - p - BS;
    if (mr <= 0) break;
    __syncthreads();

    // ---- 2. rows below the sub-block: x L_qq^T = a, one thread per row
    if (t < mr) {
      const int r = p + BS + t;
      T x[BS];
#pragma unroll
      for (int c = 0; c < BS; ++c) x[c] = sa[(p + c) * LD + r];
#pragma unroll
      for (int j = 0; j < BS; ++j) {
        x[j] *= s_rinv[j];
#pragma unroll
        for (int l = j + 1; l < BS; ++l) x[l] = fma(-x[j], sa[(p + j) * LD + p + l], x[l]);
      }
#pragma unroll
      for (int c = 0; c < BS; ++c) {
        sa[(p + c) * LD + r] = x[c];
        A[(size_t)(p + c) * lda + r] = x[c];
      }
    }
    __syncthreads();

    // ---- 3. trailing part of the block: C -= X X^T on 4 x 4 tiles (lower)
    {
      const int q0 = p + BS, nt = (mr + 3) / 4, ntiles = nt * (nt + 1) / 2;
      for (int tile = t; tile < ntiles; tile += TH) {
        int I = (int)((sqrtf(8.0f * (float)tile + 1.0f) - 1.0f) * 0.5f);
        while (I * (I + 1) / 2 > tile) --I;
        while ((I + 1) * (I + 2) / 2 <= tile) ++I;
        const int J = tile - I * (I + 1) / 2;
        const int r0 = q0 + 4 * I, c0 = q0 + 4 * J;
        T acc[4][4] = {};
#pragma unroll 8
        for (int k = 0; k < BS; ++k) {
          T xr[4], xc[4];
          load4(&sa[(p + k) * LD + r0], xr);  // rows past kb read padding, never stored
          load4(&sa[(p + k) * LD + c0], xc);
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) acc[i][jj] = fma(xr[i], xc[jj], acc[i][jj]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const int r = r0 + i, c = c0 + jj;
            if (r < kb && r >= c) sa[c * LD + r] -= acc[i][jj];
          }
      }
    }
    __syncthreads();
  }
  if (t == 0 && fail) atomicCAS(info, 0, koff + fail);
}

}  // namespace jmg
