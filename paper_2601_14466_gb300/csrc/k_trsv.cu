// k_trsv.cu -- blocked triangular solves with an FP64 Cholesky factor, one launch
// per direction (paper: "Software design", the solve step of potrs):
//
//   forward   L Y = B :  Y_b = L_bb^{-1} (B_b - sum_{j<b} L_bj Y_j)
//   backward  L^T X = Y: X_b = L_bb^{-T} (Y_b - sum_{j>b} L_jb^T X_j)
//
// Block rows of 32, taken in dependency order d = 0, 1, ... (b = d forward,
// b = nblk-1-d backward).  The serial chain of NR right-hand sides runs in ONE
// CTA, a leader; every other CTA is a helper of a group of up to 16 right-hand
// sides (all its leaders): block d >= LAG gets
//     P_d = B_d - sum_{j <= d-LAG} L_dj Y_j
// from the published rows as they appear (acquire loads of the leaders' counters,
// bounded by globaltimer), written in place over B_d, and flags it (release).  A
// leader multiplies the last LAG-1 finished blocks itself, so it never waits for
// another SM's use of them, only for P_d, which the helpers finish LAG-1 blocks
// ahead.
//
// The chain is bound by latency (FP64: 68 clocks for a dependent FMA, while the SM's
// one FP64 pipe takes an independent warp instruction every 16), so a leader keeps
// only what must be serial on it.  Per right-hand side one chain
// warp (lane = row) subtracts the product with block d-1 and substitutes
// (31 steps of s_k -= (L_ki / L_ii) s_i on unscaled values, one scaling by 1 / L_kk
// at the end, so a step is one shuffle and one FMA); aux warps
// form the products with blocks d-2 .. d-LAG+1 beforehand, prep warps scale the
// diagonal blocks, loaders bring L through a four-step ring, and a fetching and
// a publishing warp keep global round trips off the chain.  The roles meet
// through counters in shared memory, no CTA-wide barrier.  A step takes 3.9 us up to
// 16 right-hand sides (28-32 us with one lane per right-hand side substituting and
// barriers between the phases): both directions at n = 12288, 8 right-hand sides,
// 24.3 -> 3.6 ms.  From 17 right-hand sides on the helpers' products bound it
// (n = 16384, 64: 42.8 -> 33.6 ms, 1.02 TFLOP/s of 1.1); large solves then run blocked,
// with their products on the tensor cores (solve_split in k_ozpotrf.cu).
//
// Roles come from an atomic ticket in order (tickets below the number of leaders
// NL lead; ticket t helps block LAG + t - NL), so the leaders are running before
// any helper, and a helper of block d depends only on the leaders, which depend
// only on helpers of lower blocks, all of which took their tickets earlier: no
// co-residency assumption beyond the leaders'.  Groups (grid.y) run independently.
#include <algorithm>

#include "kernels.h"
#include "rcp64.cuh"

namespace jmg {

namespace trsv {
constexpr int NBK = 32;    // block rows
constexpr int GR = 16;     // right-hand sides per group
constexpr int TH = 512;    // 16 warps
constexpr int LDB = 33;    // row stride of a block of L in shared memory
constexpr int RING = 4;    // leader: steps of L in flight or in use
constexpr int SR = 8;      // leader: slots of the per-step rings (> LAG)
constexpr int HRING = 16;  // helper: blocks of L in flight or in use
constexpr int KCH = 8;     // finished blocks a helper multiplies per step (at most)

// leader shapes: blocks the leader multiplies itself (d-1 .. d-LAG+1), so many that
// the helpers' round trip (~6 us) does not hold the chain up.
template <typename T, int NR>
struct Cfg;
template <>
struct Cfg<double, 1> { static constexpr int LAG = 5, NAUX = 3; };
template <>
struct Cfg<double, 4> { static constexpr int LAG = 3, NAUX = 1; };

template <typename T>
struct Helper {
  T Ls[HRING][NBK][LDB];  // blocks of L: Ls[slot][k][i] = factor entry (row i, column k)
  T Ys[KCH][NBK][GR + 4];  // finished rows of Y (padded; four columns load as one vector)
  T red[16][4][NBK];       // partial sums of the k parts
};
template <typename T, int NR>
struct Leader {
  static constexpr int LAG = Cfg<T, NR>::LAG, NAUX = Cfg<T, NR>::NAUX;
  T Lo[RING][LAG - 1][NBK][LDB];  // off-diagonal blocks, [k][i]
  T Ld[RING][NBK][LDB];           // diagonal block: Ld[i][l] = L_li, then L_li / L_ii (l > i)
  T rinv[RING][NBK];
  T Y[SR][NR][NBK];               // solved blocks
  T P[SR][NR][NBK];               // P_d
  T Q[SR][NR][NAUX][NBK];         // P_d minus the products of aux warps NAUX-1 .. a
  int y_done[NR], q_done[NR][NAUX], p_done, prep_done, load_done[4];
};
template <typename T, int NR>
struct Smem {
  union {
    Helper<T> h;
    Leader<T, NR> l;
  };
  int ticket, ready, abort;
};

JMG_DEV int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
JMG_DEV void st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
JMG_DEV int ld_acquire_sm(const int* p) {
  int v;
  asm volatile("ld.acquire.cta.shared.b32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
JMG_DEV void st_release_sm(int* p, int v) {
  asm volatile("st.release.cta.shared.b32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
// asynchronous global -> shared copies of one element (L is final while the
// kernel runs, so caching it in L1 is safe)
JMG_DEV void cp_async_elem(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src)
               : "memory");
}
JMG_DEV void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// wait until at most n of the most recent groups are pending
JMG_DEV void cp_async_wait(int n) {
  switch (n) {
    case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
    case 3: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
    case 4: asm volatile("cp.async.wait_group 4;" ::: "memory"); break;
    case 5: asm volatile("cp.async.wait_group 5;" ::: "memory"); break;
    case 6: asm volatile("cp.async.wait_group 6;" ::: "memory"); break;
    case 7: asm volatile("cp.async.wait_group 7;" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 8;" ::: "memory"); break;
  }
}

// Raise the error word and this CTA's abort flag.
template <typename SM>
JMG_DEV void give_up(int* err, int* info, SM& S) {
  atomicExch(&S.abort, 1);
  atomicExch(err, JMG_ERR_TIMEOUT);
  if (info) atomicCAS(info, 0, -1);
}

// Bounded spin of one thread until *p > d (acquire); returns the value.  On
// expiry (limit_ns of %globaltimer), or when another CTA raised the error word,
// flags the abort: the solve is then incomplete.
template <typename SM>
JMG_DEV int wait_gt(const int* p, int d, int* err, int* info, SM& S, uint64_t limit_ns) {
  int have = ld_acquire(p);
  if (have <= d) {
    const uint64_t t0 = globaltimer_ns();
    while ((have = ld_acquire(p)) <= d) {
      if (globaltimer_ns() - t0 > limit_ns || *(volatile int*)err ||
          ld_shared_volatile(&S.abort)) {
        give_up(err, info, S);
        break;
      }
    }
  }
  return have;
}

// Bounded spin of a warp on a counter in shared memory (each lane its own p, or all
// the same) until every one is >= want; false, on every lane, on abort or expiry.  The
// vote orders no memory between the lanes; the __syncwarp puts what any lane reads next
// after the acquires of all of them.
template <typename SM>
JMG_DEV bool wait_sm(const int* p, int want, int* err, int* info, SM& S, uint64_t limit_ns) {
  if (__all_sync(0xffffffffu, ld_acquire_sm(p) >= want)) {
    __syncwarp();
    return true;
  }
  const uint64_t t0 = globaltimer_ns();
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (__all_sync(0xffffffffu, ld_acquire_sm(p) >= want)) {
        __syncwarp();
        return true;
      }
    if (__any_sync(0xffffffffu, ld_shared_volatile(&S.abort))) return false;
    if (__any_sync(0xffffffffu, globaltimer_ns() - t0 > limit_ns)) {
      give_up(err, info, S);
      return false;
    }
  }
}

// Start the copy of the 32 x 32 block of L that multiplies block row bd with the
// solved block bj into dst[k][i]: i counts the rows of bd, k those of bj, both in
// the order of the solve (backward: from the block's last row up); warp w of NW.
// Lanes run down a column of L (rows i forward, rows k backward).  Rows past the
// end are zero.  DIAG: bd == bj, only k <= i (L_ii and what it multiplies).
template <int NW, bool DIAG, typename T>
JMG_DEV void copy_block(T (*dst)[LDB], const T* L, int lda, int n, int bd, int bj, int trans,
                        int w, int lane) {
  const int r0 = bd * NBK, rows = min(NBK, n - r0), j0 = bj * NBK, jr = min(NBK, n - j0);
  const T* p = trans ? L + (size_t)(r0 + rows - 1 - w) * lda + j0 + jr - 1 - lane
                     : L + (size_t)(j0 + w) * lda + r0 + lane;
  T* q = trans ? &dst[lane][w] : &dst[w][lane];
  const ptrdiff_t ps = trans ? -(ptrdiff_t)NW * lda : (ptrdiff_t)NW * lda;
  const int qs = trans ? NW : NW * LDB;
  const bool full = rows == NBK && jr == NBK;
#pragma unroll
  for (int u = 0; u < NBK / NW; ++u) {
    const int s = w + NW * u;
    const int i = trans ? s : lane, k = trans ? lane : s;
    if ((full || (i < rows && k < jr)) && (!DIAG || k <= i))
      cp_async_elem(q + u * qs, p + u * ps);
    else
      q[u * qs] = T(0);
  }
}

// sum_k Lo[k][lane] y[k] over one block, in four sums (a dependent FP64 FMA waits
// for 68 clocks, an independent one 16)
template <typename T>
JMG_DEV T block_dot(const T (*Lo)[LDB], const T* y, int lane) {
  T a[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
  for (int k = 0; k < NBK; k += 4)
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] = fma(Lo[k + q][lane], y[k + q], a[q]);
  return (a[0] + a[1]) + (a[2] + a[3]);
}
}  // namespace trsv

template <typename T, int NR>
__global__ void __launch_bounds__(trsv::TH, 1)
    k_trsv_persist(int n, int nrhs, const T* __restrict__ L, int lda, T* __restrict__ B, int ldb,
                   int trans, int g0, int slots, int* __restrict__ tickets, int* __restrict__ done,
                   int* __restrict__ pflag, int* __restrict__ err, int* __restrict__ info,
                   unsigned long long wait_ns, int hold) {
  using namespace trsv;
  constexpr int LAG = Cfg<T, NR>::LAG, NAUX = Cfg<T, NR>::NAUX;
  extern __shared__ __align__(16) unsigned char sm_raw_trsv[];
  Smem<T, NR>& S = *reinterpret_cast<Smem<T, NR>*>(sm_raw_trsv);
  const int nblk = cdiv_dev(n, NBK);
  const int grp = g0 + blockIdx.y;
  const int ncol_g = min(GR, nrhs - grp * GR);  // right-hand sides of the group
  const int NL = cdiv_dev(ncol_g, NR);          // leaders of the group
  int* cnt = done + (size_t)grp * slots;        // finished blocks, one counter per leader
  int* pf = pflag + (size_t)grp * nblk;
  const int t = threadIdx.x, lane = t % 32, warp = t / 32;
  auto blk = [&](int d) { return trans ? nblk - 1 - d : d; };
  // row of B that lane l of block row b stands for (the solve's order)
  auto row_of = [&](int b, int rows, int l) { return b * NBK + (trans ? rows - 1 - l : l); };

  if (t == 0) {
    // no factor (info), or the other direction gave up (err): leave B alone
    const bool skip = (info && *(volatile int*)info != 0) || *(volatile int*)err != 0;
    S.ticket = skip ? -1 : atomicAdd(&tickets[grp], 1) + (hold ? NL : 0);
    S.abort = 0;
  }
  __syncthreads();
  if (S.ticket < 0) return;
  if (S.ticket < NL) {
    // ================================================================ leader
    Leader<T, NR>& M = S.l;
    const int c0 = grp * GR + S.ticket * NR;
    const int ncol = min(NR, nrhs - c0);
    int* my_cnt = cnt + S.ticket;
    if (t < NR) M.y_done[t] = 0;
    if (t < NR * NAUX) (&M.q_done[0][0])[t] = 0;
    if (t == 0) M.p_done = M.prep_done = 0;
    if (t < 4) M.load_done[t] = 0;
    __syncthreads();
    auto wsm = [&](const int* p, int want) { return wait_sm(p, want, err, info, S, wait_ns); };
    auto signal = [&](int* p, int v) {
      __syncwarp();
      if (lane == 0) st_release_sm(p, v);
    };
    constexpr int AUX0 = NR == 1 ? 1 : 4;   // first aux warp: (column, part)
    constexpr int PREP = 10, LOAD0 = 12;
    // 1 / x on the integer pipe, off the one the chain uses
    auto inverse = [](T x) -> T {
      bool bad = false;
      const T r = pivot_rcp(x < T(0) ? -x : x, &bad);
      return x < T(0) ? -r : r;
    };
    if (warp < NR) {
      // ---- chain warp of right-hand side c0 + warp
      const int c = warp;
      if (c < ncol) {
        for (int d = 0; d < nblk; ++d) {
          const int b = blk(d), rows = min(NBK, n - b * NBK), slot = d % RING;
          if (!wsm(&M.prep_done, d + 1) || !wsm(&M.q_done[c][0], d + 1)) break;
          T s = M.Q[d % SR][c][0][lane];
          if (d >= 1) {
            s -= block_dot<T>(M.Lo[slot][0], M.Y[(d - 1) % SR][c], lane);
          }
          const T(*Ld)[LDB] = M.Ld[slot];
#pragma unroll
          for (int i = 0; i < NBK - 1; ++i) {
            const T si = __shfl_sync(0xffffffffu, s, i);
            if (lane > i) s = fma(-Ld[i][lane], si, s);
          }
          const T y = s * M.rinv[slot][lane];
          M.Y[d % SR][c][lane] = lane < rows ? y : T(0);
          if (lane < rows) B[(size_t)(c0 + c) * ldb + row_of(b, rows, lane)] = y;
          signal(&M.y_done[c], d + 1);
        }
      }
    } else if (warp >= AUX0 && warp < AUX0 + NR * NAUX) {
      // ---- aux warp a of column c: products with blocks d-2-a, d-2-a-NAUX, ...; the
      // warps pass P_d minus what has been multiplied so far from the last one (the
      // oldest blocks) to the first, and that to the chain
      const int c = (warp - AUX0) % NR, a = (warp - AUX0) / NR;
      if (c < ncol) {
        for (int d = 0; d < nblk; ++d) {
          if (!wsm(&M.load_done[lane & 3], d + 1)) break;  // every loader's part
          T s = T(0);
          bool ok = true;
          constexpr int NE = (LAG - 2 + NAUX - 1) / NAUX;
#pragma unroll
          for (int q = NE - 1; q >= 0; --q) {  // the newest block last
            const int e = 2 + a + q * NAUX;
            if (e >= LAG || d - e < 0) continue;
            if (!wsm(&M.y_done[c], d - e + 1)) {
              ok = false;
              break;
            }
            s -= block_dot<T>(M.Lo[d % RING][e - 1], M.Y[(d - e) % SR][c], lane);
          }
          if (!ok) break;
          if (a == NAUX - 1) {
            if (!wsm(&M.p_done, d + 1)) break;
            s += M.P[d % SR][c][lane];
          } else {
            if (!wsm(&M.q_done[c][a + 1], d + 1)) break;
            s += M.Q[d % SR][c][a + 1][lane];
          }
          M.Q[d % SR][c][a][lane] = s;
          signal(&M.q_done[c][a], d + 1);
        }
      }
    } else if (warp == PREP) {
      // ---- prep warp: 1 / L_ii and the scaled columns of the diagonal block
      for (int d = 0; d < nblk; ++d) {
        const int slot = d % RING, rows = min(NBK, n - blk(d) * NBK);
        if (!wsm(&M.load_done[lane & 3], d + 1)) break;  // every loader's part
        T(*Ld)[LDB] = M.Ld[slot];
        const T r = lane < rows ? inverse(Ld[lane][lane]) : T(0);
        M.rinv[slot][lane] = r;
#pragma unroll 8
        for (int i = 0; i < NBK - 1; ++i) {
          const T ri = __shfl_sync(0xffffffffu, r, i);
          if (lane > i) Ld[i][lane] *= ri;
        }
        signal(&M.prep_done, d + 1);
      }
    } else if (warp == 8) {
      // ---- fetching warp: P_d (after its flag) into P[d % SR]
      for (int d = 0; d < nblk; ++d) {
        bool ok = true;
        for (int c = 0; c < ncol; ++c) ok = ok && wsm(&M.y_done[c], d - SR + 1);  // slot free
        if (!ok) break;
        if (d >= LAG) {
          if (lane == 0) (void)wait_gt(&pf[d], 0, err, info, S, wait_ns);
          __syncwarp();
          if (ld_shared_volatile(&S.abort)) break;
        }
        const int b = blk(d), rows = min(NBK, n - b * NBK);
        T v[NR];
#pragma unroll
        for (int c = 0; c < NR; ++c)
          v[c] = (lane < rows && c < ncol)
                     ? __ldcg(&B[(size_t)(c0 + c) * ldb + row_of(b, rows, lane)])
                     : T(0);
#pragma unroll
        for (int c = 0; c < NR; ++c) M.P[d % SR][c][lane] = v[c];
        signal(&M.p_done, d + 1);
      }
    } else if (warp == 9) {
      // ---- publishing warp: Y_d is in global memory (stored by the chain warps)
      for (int d = 0; d < nblk; ++d) {
        bool ok = true;
        for (int c = 0; c < ncol; ++c) ok = ok && wsm(&M.y_done[c], d + 1);
        if (!ok) break;
        if (lane == 0) {
          __threadfence();
          st_release(my_cnt, d + 1);
        }
        __syncwarp();
      }
    } else if (warp >= LOAD0) {
      // ---- loaders: step d's blocks of L into slot d % RING, two steps in flight
      for (int d = 0; d <= nblk; ++d) {
        if (d < nblk) {
          bool ok = true;
          for (int c = 0; c < ncol; ++c) ok = ok && wsm(&M.y_done[c], d - RING + 1);
          if (!ok) break;
          const int b = blk(d), slot = d % RING, w = warp - LOAD0;
          copy_block<4, true>(M.Ld[slot], L, lda, n, b, b, trans, w, lane);
#pragma unroll 1
          for (int e = 1; e < LAG; ++e)
            if (d - e >= 0)
              copy_block<4, false>(M.Lo[slot][e - 1], L, lda, n, b, blk(d - e), trans, w, lane);
          cp_async_commit();
        }
        if (d >= 1) {
          cp_async_wait(d < nblk ? 1 : 0);  // step d-1 has landed
          signal(&M.load_done[warp - LOAD0], d);
        }
      }
      cp_async_wait(0);  // nothing of ours may land after the CTA ends
    }
    return;
  }

  // ================================================================ helpers
  Helper<T>& H = S.h;
  const int c0 = grp * GR;
  // a warp multiplies tq right-hand sides (4, or 2 or 1 of a narrow group) with its
  // part of the 32 columns of a block: one value of L feeds tq products
  const int tq = ncol_g > 2 ? 4 : ncol_g, nq = cdiv_dev(ncol_g, tq);
  int nqp = 1;
  while (nqp < nq) nqp *= 2;
  const int hq = warp % nqp, part = warp / nqp, parts = 16 / nqp, kper = NBK / parts;
  while (true) {
    const int d = LAG + S.ticket - NL;  // block (in dependency order) of this ticket
    if (d >= nblk) break;
    const int b = blk(d), rows = min(NBK, n - b * NBK);
    const int ndep = d - LAG + 1;  // dependencies j = 0 .. d-LAG
    auto issue_L = [&](int j) {
      copy_block<16, false>(H.Ls[j % HRING], L, lda, n, b, blk(j), trans, warp, lane);
      cp_async_commit();
    };
    T acc[4] = {T(0), T(0), T(0), T(0)};
    int pfd = 0;  // blocks of L issued
    for (; pfd < min(ndep, HRING - KCH); ++pfd) issue_L(pfd);
    for (int j = 0; j < ndep;) {
      if (warp == 0) {
        int r = 0x7fffffff;
        if (lane < NL) r = wait_gt(cnt + lane, j, err, info, S, wait_ns);
        for (int o = 8; o > 0; o >>= 1) r = min(r, __shfl_xor_sync(0xffffffffu, r, o));
        if (lane == 0) S.ready = r;
      }
      __syncthreads();
      if (S.abort) break;
      const int ready = min(min(S.ready, ndep), j + KCH);
      {  // this warp's column of the finished blocks (all loads first, then the stores)
        T v[KCH];
#pragma unroll
        for (int q = 0; q < KCH; ++q) {
          const int jb = blk(j + q), jr = min(NBK, n - jb * NBK);
          v[q] = (q < ready - j && lane < jr && warp < ncol_g)
                     ? __ldcg(&B[(size_t)(c0 + warp) * ldb + row_of(jb, jr, lane)])
                     : T(0);
        }
#pragma unroll
        for (int q = 0; q < KCH; ++q) H.Ys[q][lane][warp] = v[q];
      }
      for (; pfd < min(ndep, ready + HRING - KCH); ++pfd) issue_L(pfd);
      cp_async_wait(pfd - ready);  // blocks j .. ready-1 have landed
      __syncthreads();
      for (int q = 0; q < ready - j; ++q) {
        const T(*Lq)[LDB] = H.Ls[(j + q) % HRING];
        const T(*Yq)[GR + 4] = H.Ys[q];
        if (tq == 4) {
#pragma unroll 8
          for (int k = part * kper; k < (part + 1) * kper; ++k) {
            const T l = Lq[k][lane];
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[c] = fma(l, Yq[k][4 * hq + c], acc[c]);
          }
        } else {
          for (int k = part * kper; k < (part + 1) * kper; ++k) {
            const T l = Lq[k][lane];
            acc[0] = fma(l, Yq[k][0], acc[0]);
            if (tq == 2) acc[1] = fma(l, Yq[k][1], acc[1]);
          }
        }
      }
      __syncthreads();  // the ring slots and Ys are free again
      j = ready;
    }
    cp_async_wait(0);  // no copy of ours may land after the CTA moves on
    if (S.abort) break;
    // P_d over B_d, then the flag
#pragma unroll
    for (int c = 0; c < 4; ++c) H.red[warp][c][lane] = acc[c];
    __syncthreads();
    if (warp < ncol_g && lane < rows) {
      const int wq = warp / tq, wc = warp % tq;
      T sum = H.red[wq][wc][lane];
      for (int p = 1; p < parts; ++p) sum += H.red[wq + p * nqp][wc][lane];
      T* p = &B[(size_t)(c0 + warp) * ldb + row_of(b, rows, lane)];
      *p = __ldcg(p) - sum;
    }
    __syncthreads();
    if (t == 0) {
      __threadfence();
      st_release(&pf[d], 1);
      S.ticket = atomicAdd(&tickets[grp], 1) + (hold ? NL : 0);
    }
    __syncthreads();
  }
}

// Groups per launch.  Every launch keeps all of its CTAs resident (a leader waits for its
// helpers), so more groups at once leave fewer SMs to help: with gb of them a launch takes
// about the longer of its chain, 3.9 us a step, and the helpers' products, 4.3 us for 32 x
// 32 times 16 right-hand sides on one SM, over nsm - gb nl SMs, and 0.6 of the shorter (n =
// 8000: 4.5 ms modelled and measured for 4 groups at once, 2.45 for 2).  The gb with the
// least time in all launches.  Both directions, as many groups as fit with one helper each
// / this: n = 500, 1000 right-hand sides 2.00 / 1.07 ms; 1000, 1000 8.28 / 3.58; 4000, 300
// 16.8 / 11.9; 8000, 500 270 / 71; up to 64 right-hand sides as before.  Blocks up to LAG
// have no helpers to wait for: all groups in one launch.
static int trsv_batch(int groups, int nblk, int lag, int nl, int nsm) {
  if (nblk <= lag) return std::min(groups, 65535);
  int best = 1;
  double least = 0.0;
  for (int gb = std::min(groups, std::max(1, nsm / (nl + 1))); gb >= 1; --gb) {
    const double chain = 3.9 * nblk,
                 products = 4.3 * gb * 0.5 * nblk * nblk / std::max(1, nsm - gb * nl);
    const double time = cdiv(groups, gb) * (std::max(chain, products) +
                                            0.6 * std::min(chain, products) + 6.0);
    if (least == 0.0 || time < least) least = time, best = gb;
  }
  return best;
}

// leaders a group can have (see launch_trsv_persist)
static int trsv_slots(int nrhs) { return nrhs <= trsv::GR ? trsv::GR : trsv::GR / 4; }

size_t trsv_sync_ints(int n, int nrhs) {
  // the error word first; then per group of 16 right-hand sides a ticket counter,
  // a counter of finished blocks per leader and one flag per block (P_d ready)
  const int groups = cdiv(std::max(nrhs, 1), trsv::GR);
  return 1 + (size_t)groups * (1 + trsv_slots(nrhs) + cdiv(std::max(n, 1), trsv::NBK));
}

// keep_err: the error word stays as the launches before left it
template <typename T, int NR>
static int trsv_launch(int n, int nrhs, const T* L, int lda, T* B, int ldb, int trans, int keep_err,
                       int* sync, int* info, cudaStream_t s, int hold) {
  const int groups = cdiv(nrhs, trsv::GR), nblk = cdiv(n, trsv::NBK);
  int* err = sync;
  int* tickets = sync + 1;
  int* done = tickets + groups;
  const int slots = trsv_slots(nrhs);
  int* pflag = done + (size_t)groups * slots;
  JMG_CUDA(cudaMemsetAsync(sync + keep_err, 0,
                           sizeof(int) * (trsv_sync_ints(n, nrhs) - keep_err), s));
  const size_t smem = sizeof(trsv::Smem<T, NR>);
  auto k = k_trsv_persist<T, NR>;
  JMG_TRY(ensure_smem(k, (int)smem));
  // the leaders plus one helper per block when they all fit; the tickets keep the
  // dependency order either way.
  int dev = 0, nsm = 152;
  JMG_CUDA(cudaGetDevice(&dev));
  JMG_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const int nl = cdiv(std::min(nrhs, trsv::GR), NR);
  const int want = nl + std::max(0, nblk - trsv::Cfg<T, NR>::LAG);
  const int batch = trsv_batch(groups, nblk, trsv::Cfg<T, NR>::LAG, nl, nsm);
  for (int g0 = 0; g0 < groups; g0 += batch) {
    const int gn = std::min(batch, groups - g0);
    const int gx = want == nl ? nl : std::max(nl + 1, std::min(want, nsm / gn));
    k<<<dim3(gx, gn), trsv::TH, smem, s>>>(n, nrhs, L, lda, B, ldb, trans, g0, slots, tickets, done,
                                           pflag, err, info, g_wait_ns, hold);
    JMG_TRY(launched());
  }
  return JMG_OK;
}

int trsv_block(int n, int nrhs, const double* L, int lda, double* B, int ldb, int trans,
               int keep_err, int* sync, int* info, cudaStream_t s, int hold) {
  if (n <= 0 || nrhs <= 0) return JMG_OK;
  // Up to 16 right-hand sides every one gets a leader of its own (the chain sets
  // the time); beyond, the helpers' products do, and four share a leader.
  if (nrhs <= trsv::GR)
    return trsv_launch<double, 1>(n, nrhs, L, lda, B, ldb, trans, keep_err, sync, info, s, hold);
  return trsv_launch<double, 4>(n, nrhs, L, lda, B, ldb, trans, keep_err, sync, info, s, hold);
}

// the forward solve clears the error word with the rest; the backward solve keeps
// it, so that it returns at once after a forward solve that gave up
template <>
int launch_trsv_persist<double>(int n, int nrhs, const double* L, int lda, double* B, int ldb,
                                int trans, int* sync, int* info, cudaStream_t s, int hold) {
  return trsv_block(n, nrhs, L, lda, B, ldb, trans, trans ? 1 : 0, sync, info, s, hold);
}

}  // namespace jmg
