// k_dense.cu -- CUDA-core kernels of the blocked Cholesky solver (sm_103a):
// diagonal-block factorisation, panel TRSM, tiled GEMM / SYRK / SYMM, blocked
// triangular solves, FP64 residual and the small helpers of the refinement loop.
//
// Paper: "Software design" -- potrs solves A x = b for SPD A by a Cholesky
// factorisation followed by the triangular solves.  The paper delegates both to
// cuSOLVERMp; the blocking below is the textbook right-looking scheme (factor
// the diagonal block, solve the panel below it, update the trailing matrix).
#include <map>
#include <mutex>
#include <utility>

#include "kernels.h"
#include "potrf_diag.cuh"

namespace jmg {

long long g_launches = 0;
unsigned long long g_wait_ns = 2000000000ull;

int ensure_smem_raw(const void* func, int bytes) {
  int dev = 0;
  JMG_CUDA(cudaGetDevice(&dev));
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, int> raised;
  std::lock_guard<std::mutex> lock(mu);
  const auto key = std::make_pair(func, dev);
  const auto it = raised.find(key);
  if (it != raised.end() && it->second >= bytes) return JMG_OK;
  JMG_CUDA(cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  raised[key] = bytes;
  return JMG_OK;
}

template <typename T>
__global__ void __launch_bounds__(pdiag::TH) k_potrf_diag(T* __restrict__ A, int lda, int kb,
                                                          int koff, int* __restrict__ info) {
  potrf_diag_body<T>(A, lda, kb, koff, info);
}

// Batched: CTA b factors the n x n FP32 system A + b * sA (n <= 128) with info[b].
__global__ void __launch_bounds__(pdiag::TH) k_potrf_diag_batched(float* __restrict__ A, int lda,
                                                                  long long sA, int n,
                                                                  int* __restrict__ info) {
  potrf_diag_body<float>(A + (size_t)blockIdx.x * sA, lda, n, 0, info + blockIdx.x);
}
int launch_potf2_batched(int n, int batch, float* A, int lda, long long sA, int* info,
                         cudaStream_t s) {
  JMG_TRY(ensure_smem(k_potrf_diag_batched, (int)(pdiag::KB * pdiag::LD * sizeof(float))));
  k_potrf_diag_batched<<<batch, pdiag::TH, (size_t)n * pdiag::LD * sizeof(float), s>>>(A, lda, sA,
                                                                                      n, info);
  return launched();
}

template <typename T>
static int potf2_impl(T* A, int lda, int kb, int koff, int* info, cudaStream_t s) {
  if (kb > pdiag::KB) return JMG_ERR_UNSUPPORTED;
  const size_t smem = (size_t)kb * pdiag::LD * sizeof(T);
  auto k = k_potrf_diag<T>;
  JMG_TRY(ensure_smem(k, (int)(pdiag::KB * pdiag::LD * sizeof(T))));
  k<<<1, pdiag::TH, smem, s>>>(A, lda, kb, koff, info);
  return launched();
}
int launch_potf2(double* A, int lda, int kb, int koff, int* info, cudaStream_t s) {
  return potf2_impl(A, lda, kb, koff, info, s);
}
int launch_potf2(float* A, int lda, int kb, int koff, int* info, cudaStream_t s) {
  return potf2_impl(A, lda, kb, koff, info, s);
}

// ============================================================================
// Panel TRSM: A21 (m x kb) <- A21 * Lkk^{-T}, in place.  Each CTA owns BR rows;
// row r of the result solves x_r Lkk^T = a_r by forward substitution over the
// columns j (x_rj = a_rj / L_jj, then a_rl -= x_rj L_lj for l > j).  Lkk sits in
// shared memory; threads are (row, column-group) pairs.
// ============================================================================
__global__ void __launch_bounds__(256) k_trsm(double* __restrict__ A21, int lda, int m, int kb,
                                              const double* __restrict__ Lkk,
                                              const int* __restrict__ info) {
  using T = double;
  constexpr int BR = 32;
  if (*(volatile const int*)info != 0) return;
  extern __shared__ __align__(16) unsigned char sm_trsm[];
  T* Ls = reinterpret_cast<T*>(sm_trsm);  // kb x (kb+1), column-major
  const int ldl = kb + 1;
  T* Xs = Ls + (size_t)kb * ldl;  // kb columns x (BR+1)
  const int ldx = BR + 1;
  const int t = threadIdx.x;
  const int r0 = blockIdx.x * BR;
  for (int base = 0; base < kb * kb; base += 256 * 16) {  // 16 independent loads per thread
    T v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int idx = base + t + 256 * q;
      const int i = idx % kb, j = idx / kb;
      v[q] = (idx < kb * kb && i >= j) ? Lkk[(size_t)j * lda + i] : T(0);
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int idx = base + t + 256 * q;
      if (idx < kb * kb) Ls[(idx / kb) * ldl + idx % kb] = v[q];
    }
  }
  for (int base = 0; base < BR * kb; base += 256 * 16) {
    T v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int idx = base + t + 256 * q;
      const int i = idx % BR, j = idx / BR;
      v[q] = (idx < BR * kb && r0 + i < m) ? A21[(size_t)j * lda + r0 + i] : T(0);
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int idx = base + t + 256 * q;
      if (idx < BR * kb) Xs[(idx / BR) * ldx + idx % BR] = v[q];
    }
  }
  __syncthreads();
  constexpr int G = 256 / BR;
  const int r = t % BR, g = t / BR;
  for (int j = 0; j < kb; ++j) {
    if (g == 0) Xs[j * ldx + r] = Xs[j * ldx + r] / Ls[j * ldl + j];
    __syncthreads();
    const T xrj = Xs[j * ldx + r];
    for (int l = j + 1 + g; l < kb; l += G) Xs[l * ldx + r] -= xrj * Ls[j * ldl + l];
    __syncthreads();
  }
  for (int idx = t; idx < BR * kb; idx += blockDim.x) {
    int i = idx % BR, j = idx / BR;
    if (r0 + i < m) A21[(size_t)j * lda + r0 + i] = Xs[j * ldx + i];
  }
}

int launch_trsm(double* A21, int lda, int m, int kb, const double* Lkk, const int* info,
                cudaStream_t s) {
  if (m <= 0) return JMG_OK;
  const size_t smem = ((size_t)kb * (kb + 1) + (size_t)kb * 33) * sizeof(double);
  JMG_TRY(ensure_smem(k_trsm, (int)smem));
  k_trsm<<<cdiv(m, 32), 256, smem, s>>>(A21, lda, m, kb, Lkk, info);
  return launched();
}
// 16-bit words of the mixed path's tensor-core operands
// word pairs (a, b) with a + b < words, ordered by significance
__constant__ int c_pair_a[6] = {0, 0, 1, 0, 1, 2};
__constant__ int c_pair_b[6] = {0, 1, 0, 2, 1, 0};
int split_pairs(int words) { return words <= 1 ? 1 : (words == 2 ? 3 : 6); }
template <typename H>
JMG_DEV H to16(float v);
template <>
JMG_DEV __nv_bfloat16 to16<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}
template <>
JMG_DEV __half to16<__half>(float v) {
  return __float2half_rn(v);
}
template <typename H>
JMG_DEV float from16(H v);
template <>
JMG_DEV float from16<__nv_bfloat16>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}
template <>
JMG_DEV float from16<__half>(__half v) {
  return __half2float(v);
}
template <typename H>
struct alignas(4) Two16 {
  H x, y;
};

// FP32 panel TRSM (kb == KB): row r of the panel solves x Lkk^T = a, G lanes per row,
// each holding the column pairs {2 (g + G i), 2 (g + G i) + 1}: step j shuffles a_j to
// the row's lanes, x_j = a_j / L_jj (by the reciprocal), a_l -= x_j L_lj for l > j, in
// this order whatever G is.  32-row tiles go through shared memory (coalesced down
// the columns of L21), a resident grid keeps L_kk.  Bound by issue: about 20
// instructions per step for 4 rows.
//
// With PA the same pass writes the rows' 16-bit words w0 = rn(x), w1 = rn(x - w0), ...
// into the row-major extended operands of the update: pair p of the pair table takes
// PA[:, p KB + c] = word a_p, PB[:, p KB + c] = word b_p (PB may be null).
// Panel of 128 columns with FP16 words, n = 16384: 28 us a panel on average against
// 25.4 + 8.6 us with the words in a pass of their own.
namespace ptrsm {
constexpr int RB = 32, TH = 256, G = 8, LDX = RB + 1;
template <int KB>
constexpr size_t smem() {
  return sizeof(float) * ((size_t)KB * KB + (size_t)KB * LDX + KB);
}
}  // namespace ptrsm

template <int KB, typename H>
__global__ void __launch_bounds__(ptrsm::TH, 2) k_trsm_rows(float* __restrict__ A21, int lda, int m,
                                                            const float* __restrict__ Lkk,
                                                            const int* __restrict__ info,
                                                            int npairs, H* __restrict__ PA,
                                                            H* __restrict__ PB, int ldp) {
  using namespace ptrsm;
  constexpr int NP = KB / 2 / G;
  if (*(volatile const int*)info != 0) return;
  extern __shared__ __align__(16) float sm_trows[];
  float* Lt = sm_trows;        // Lt[j * KB + l] = L_lj, l >= j
  float* Xt = Lt + KB * KB;    // the tile: Xt[c * LDX + r]
  float* rinv = Xt + KB * LDX;
  const int t = threadIdx.x, lane = t % 32, warp = t / 32;
  for (int base = 0; base < KB * KB; base += TH * 16) {  // 16 independent loads per thread
    float v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int idx = base + t + TH * q, l = idx % KB, j = idx / KB;
      v[q] = l >= j ? Lkk[(size_t)j * lda + l] : 0.0f;
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) Lt[base + t + TH * q] = v[q];
  }
  __syncthreads();
  if (t < KB) rinv[t] = 1.0f / Lt[t * KB + t];
  const int g = lane % G, rl = warp * (32 / G) + lane / G;
  for (int r0 = blockIdx.x * RB; r0 < m; r0 += gridDim.x * RB) {
    __syncthreads();  // Lt, rinv are in place; the previous tile is stored
    {
      constexpr int Q = KB * RB / TH;
      float v[Q];
#pragma unroll
      for (int q = 0; q < Q; ++q)
        v[q] = r0 + lane < m ? A21[(size_t)(warp + 8 * q) * lda + r0 + lane] : 0.0f;
#pragma unroll
      for (int q = 0; q < Q; ++q) Xt[(warp + 8 * q) * LDX + lane] = v[q];
    }
    __syncthreads();
    float x[2 * NP];
#pragma unroll
    for (int i = 0; i < NP; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h) x[2 * i + h] = Xt[(2 * (g + G * i) + h) * LDX + rl];
#pragma unroll
    for (int j = 0; j < KB; ++j) {
      const int go = (j / 2) % G, io = (j / 2) / G;  // owner lane and register of column j
      const float xj = __shfl_sync(0xffffffffu, x[2 * io + (j & 1)], go, G) * rinv[j];
      if (g == go) x[2 * io + (j & 1)] = xj;
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        if (2 * (G - 1 + G * i) + 1 <= j) continue;  // every lane's pair is done
        const int l = 2 * (g + G * i);
        const float2 l2 = *reinterpret_cast<const float2*>(&Lt[j * KB + l]);
        if (l > j) x[2 * i] = fmaf(-xj, l2.x, x[2 * i]);
        if (l + 1 > j) x[2 * i + 1] = fmaf(-xj, l2.y, x[2 * i + 1]);
      }
    }
#pragma unroll
    for (int i = 0; i < NP; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = 2 * (g + G * i) + h;
        Xt[c * LDX + rl] = x[2 * i + h];
      }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < KB * RB / TH; ++q)
      if (r0 + lane < m) A21[(size_t)(warp + 8 * q) * lda + r0 + lane] = Xt[(warp + 8 * q) * LDX + lane];
    if (!PA) continue;
#pragma unroll
    for (int rr = 0; rr < RB / 8; ++rr) {  // a warp writes whole rows
      const int rw = warp * (RB / 8) + rr, r = r0 + rw;
      if (r >= m) break;
#pragma unroll
      for (int cb = 0; cb < KB; cb += 64) {
        const int c = cb + 2 * lane;
        float e0 = Xt[c * LDX + rw], e1 = Xt[(c + 1) * LDX + rw];
        Two16<H> w[3];
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          w[u].x = to16<H>(e0);
          w[u].y = to16<H>(e1);
          e0 -= from16<H>(w[u].x);
          e1 -= from16<H>(w[u].y);
        }
        for (int p = 0; p < npairs; ++p) {
          const size_t at = (size_t)r * ldp + p * KB + c;
          const int a = c_pair_a[p], b = c_pair_b[p];
          *reinterpret_cast<Two16<H>*>(&PA[at]) = a == 0 ? w[0] : (a == 1 ? w[1] : w[2]);
          if (PB) *reinterpret_cast<Two16<H>*>(&PB[at]) = b == 0 ? w[0] : (b == 1 ? w[1] : w[2]);
        }
      }
    }
  }
}

template <int KB, typename H>
static int trsm_rows_launch(float* A21, int lda, int m, const float* Lkk, const int* info, int np,
                            void* PA, void* PB, int ldp, cudaStream_t s) {
  auto k = k_trsm_rows<KB, H>;
  JMG_TRY(ensure_smem(k, (int)ptrsm::smem<KB>()));
  int dev = 0, nsm = 152;
  JMG_CUDA(cudaGetDevice(&dev));
  JMG_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const int grid = std::min(cdiv(m, ptrsm::RB), 2 * nsm);
  k<<<grid, ptrsm::TH, ptrsm::smem<KB>(), s>>>(A21, lda, m, Lkk, info, np, (H*)PA, (H*)PB, ldp);
  return launched();
}

int launch_trsm(float* A21, int lda, int m, int kb, const float* Lkk, const int* info,
                cudaStream_t s) {
  if (m <= 0) return JMG_OK;
  if (kb == 128)
    return trsm_rows_launch<128, __half>(A21, lda, m, Lkk, info, 0, nullptr, nullptr, 0, s);
  if (kb == 64)
    return trsm_rows_launch<64, __half>(A21, lda, m, Lkk, info, 0, nullptr, nullptr, 0, s);
  return JMG_ERR_UNSUPPORTED;  // (a panel with rows below it is always full)
}

int launch_trsm_words(float* A21, int lda, int m, int kb, const float* Lkk, const int* info,
                      int prec, int words, void* PA, void* PB, int ldp, cudaStream_t s) {
  if (m <= 0) return JMG_OK;
  const int np = split_pairs(words);
  if (np == 1) PB = nullptr;
  const bool half = prec == JMG_PREC_FP16;
  if (kb == 128)
    return half ? trsm_rows_launch<128, __half>(A21, lda, m, Lkk, info, np, PA, PB, ldp, s)
                : trsm_rows_launch<128, __nv_bfloat16>(A21, lda, m, Lkk, info, np, PA, PB, ldp, s);
  if (kb == 64)
    return half ? trsm_rows_launch<64, __half>(A21, lda, m, Lkk, info, np, PA, PB, ldp, s)
                : trsm_rows_launch<64, __nv_bfloat16>(A21, lda, m, Lkk, info, np, PA, PB, ldp, s);
  return JMG_ERR_UNSUPPORTED;  // (a panel with rows below it is always full)
}

// ============================================================================
// FP32 trailing update of the plain path, C -= P P^T (lower part, P = L21, K = kb
// columns), and the next diagonal block in the same launch: CTA 0 takes the tile at
// the diagonal's head and then factors it (kn x kn) while the others work through
// the rest, so the block's serial chain (63 us at 128 columns) hides behind the
// update.  128 x 128 tiles, 8 x 8 per thread, two 16-deep stages of P in shared
// memory: 6 shared-memory wavefronts per 64 FMAs of a warp, bound by the FP32 pipe.  Every
// element sums its products in order from zero and is subtracted from C once, as
// the 64 x 64 kernel (k_gemm) does: the bits are the same.  n = 8192, all updates and
// diagonal blocks: 7.2 + 4.0 -> 7.8 ms.
// ============================================================================
namespace syrk32 {
constexpr int BT = 128, BK = 16, TH = 256, LDS = BT + 4;
constexpr size_t STAGE = sizeof(float) * 2 * BK * LDS;  // rows' and columns' operand
constexpr size_t SMEM = 2 * STAGE > sizeof(float) * pdiag::KB * pdiag::LD
                            ? 2 * STAGE
                            : sizeof(float) * pdiag::KB * pdiag::LD;
}  // namespace syrk32

__global__ void __launch_bounds__(syrk32::TH, 2) k_syrk_f32(int m, int kb, int kn, int koff,
                                                            const float* __restrict__ P,
                                                            float* C, int lda, int* info) {
  using namespace syrk32;
  extern __shared__ __align__(16) unsigned char sm_diag[];
  __shared__ int s_info;  // (one read: CTA 0 may report a pivot while others start)
  if (threadIdx.x == 0) s_info = *(volatile const int*)info;
  __syncthreads();
  if (s_info != 0) return;
  float* st = reinterpret_cast<float*>(sm_diag);  // [stage][rows | columns][BK][LDS]
  int ti, tj;
  tri_index(blockIdx.x, ti, tj);
  const int i0 = ti * BT, j0 = tj * BT;
  const int t = threadIdx.x, tx = t % 16, ty = t / 16;
  const bool diag = ti == tj;
  float acc[8][8];
#pragma unroll
  for (int q = 0; q < 8; ++q)
#pragma unroll
    for (int p = 0; p < 8; ++p) acc[q][p] = 0.0f;
  // a stage: 16 columns of P, 128 rows each; 8 elements per thread and operand
  float ra[8], rb[8];
  const int r = t % BT, l0 = t / BT;
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const size_t col = (size_t)(k0 + l0 + 2 * q) * lda;
      ra[q] = i0 + r < m ? P[col + i0 + r] : 0.0f;
      if (!diag) rb[q] = j0 + r < m ? P[col + j0 + r] : 0.0f;
    }
  };
  auto store = [&](int s) {
    float* a = st + s * 2 * BK * LDS;
    float* b = a + BK * LDS;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      a[(l0 + 2 * q) * LDS + r] = ra[q];
      b[(l0 + 2 * q) * LDS + r] = diag ? ra[q] : rb[q];
    }
  };
  fetch(0);
  store(0);
  __syncthreads();
  for (int k0 = 0, s = 0; k0 < kb; k0 += BK, s ^= 1) {
    const bool more = k0 + BK < kb;
    if (more) fetch(k0 + BK);
    const float* a = st + s * 2 * BK * LDS;
    const float* b = a + BK * LDS;
#pragma unroll
    for (int l = 0; l < BK; ++l) {
      // rows 4 tx + {0..3}, 64 + 4 tx + {0..3}; columns likewise by ty
      const float4 a0 = *reinterpret_cast<const float4*>(&a[l * LDS + 4 * tx]);
      const float4 a1 = *reinterpret_cast<const float4*>(&a[l * LDS + 64 + 4 * tx]);
      const float4 b0 = *reinterpret_cast<const float4*>(&b[l * LDS + 4 * ty]);
      const float4 b1 = *reinterpret_cast<const float4*>(&b[l * LDS + 64 + 4 * ty]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int p = 0; p < 8; ++p) acc[q][p] = fmaf(av[q], bv[p], acc[q][p]);
    }
    if (more) store(s ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const int gj = j0 + (p < 4 ? 0 : 60) + 4 * ty + p;
    if (gj >= m) continue;
    float* cp = C + (size_t)gj * lda;
    float old[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int gi = i0 + (q < 4 ? 0 : 60) + 4 * tx + q;
      old[q] = gi < m && gi >= gj ? cp[gi] : 0.0f;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int gi = i0 + (q < 4 ? 0 : 60) + 4 * tx + q;
      if (gi < m && gi >= gj) cp[gi] = old[q] - acc[q][p];
    }
  }
  if (blockIdx.x == 0) {
    __syncthreads();  // the block is in global memory, the stages are idle
    potrf_diag_body<float>(C, lda, kn, koff, info);
  }
}

int launch_syrk_f32(int m, int kb, int kn, int koff, const float* P, float* C, int lda, int* info,
                    cudaStream_t s) {
  if (m <= 0) return JMG_OK;
  if (kb % syrk32::BK) return JMG_ERR_UNSUPPORTED;
  JMG_TRY(ensure_smem(k_syrk_f32, (int)syrk32::SMEM));
  k_syrk_f32<<<(unsigned)tri_tiles(cdiv(m, syrk32::BT)), syrk32::TH, syrk32::SMEM, s>>>(
      m, kb, kn, koff, P, C, lda, info);
  return launched();
}

// ============================================================================
// Tiled GEMM on the CUDA cores: C -= op(A) op(B) with 64 x BN output tiles,
// BK = 16, 256 threads, each thread a 4 x (BN/16) register tile.  Rows of a
// thread are tx + 16 q and columns ty + 16 q' so that shared-memory reads are
// conflict-free and global stores coalesce along a column.
// ============================================================================
constexpr int GBM = 64, GBK = 16;

template <typename T, int AMODE>
JMG_DEV T load_a(const T* __restrict__ A, int lda, int i, int l) {
  if (AMODE == MODE_N) return A[(size_t)l * lda + i];
  if (AMODE == MODE_T) return A[(size_t)i * lda + l];
  return (i >= l) ? A[(size_t)l * lda + i] : A[(size_t)i * lda + l];
}

template <typename T, int BN, int AMODE, int BMODE, int OUT>
__global__ void __launch_bounds__(256) k_gemm(int m, int n, int k, const T* __restrict__ A, int lda,
                                              const T* __restrict__ B, int ldb, T* __restrict__ C,
                                              int ldc, int kchunk, const int* __restrict__ info) {
  if (info && *(volatile const int*)info != 0) return;
  constexpr int TN = BN / 16;
  __shared__ T As[GBK][GBM + 1];
  __shared__ T Bs[GBK][BN + 1];
  int ti, tj;
  if (OUT == OUT_SUB_LOWER) {
    tri_index(blockIdx.x, ti, tj);
  } else {
    ti = blockIdx.x;
    tj = blockIdx.y;
  }
  const int i0 = ti * GBM, j0 = tj * BN;
  const int kbeg = (OUT == OUT_PART) ? blockIdx.z * kchunk : 0;
  const int kend = (OUT == OUT_PART) ? min(k, kbeg + kchunk) : k;
  const int t = threadIdx.x, tx = t % 16, ty = t / 16;
  T acc[4][TN];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int p = 0; p < TN; ++p) acc[q][p] = T(0);

  for (int l0 = kbeg; l0 < kend; l0 += GBK) {
    // ---- A tile: GBM x GBK
    // coalesce along the stored column: rows for N (and S tiles that reach the
    // lower triangle), k for T (and S tiles wholly above the diagonal)
    const bool a_rowfast = (AMODE == MODE_N) || (AMODE == MODE_S && !(i0 + GBM - 1 < l0));
#pragma unroll
    for (int q = 0; q < (GBM * GBK) / 256; ++q) {
      int idx = t + 256 * q;
      int ii, ll;
      if (a_rowfast) {
        ii = idx % GBM;
        ll = idx / GBM;
      } else {
        ll = idx % GBK;
        ii = idx / GBK;
      }
      int gi = i0 + ii, gl = l0 + ll;
      As[ll][ii] = (gi < m && gl < kend) ? load_a<T, AMODE>(A, lda, gi, gl) : T(0);
    }
    // ---- B tile: GBK x BN
#pragma unroll
    for (int q = 0; q < (GBK * BN + 255) / 256; ++q) {
      int idx = t + 256 * q;
      if (idx < GBK * BN) {
        int ll, jj;
        if (BMODE == MODE_N) {
          ll = idx % GBK;
          jj = idx / GBK;
        } else {
          jj = idx % BN;
          ll = idx / BN;
        }
        int gl = l0 + ll, gj = j0 + jj;
        T v = T(0);
        if (gl < kend && gj < n)
          v = (BMODE == MODE_N) ? B[(size_t)gj * ldb + gl] : B[(size_t)gl * ldb + gj];
        Bs[ll][jj] = v;
      }
    }
    __syncthreads();
#pragma unroll
    for (int l = 0; l < GBK; ++l) {
      T a[4], b[TN];
#pragma unroll
      for (int q = 0; q < 4; ++q) a[q] = As[l][tx + 16 * q];
#pragma unroll
      for (int p = 0; p < TN; ++p) b[p] = Bs[l][ty + 16 * p];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int p = 0; p < TN; ++p) acc[q][p] = fma(a[q], b[p], acc[q][p]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int gi = i0 + tx + 16 * q;
    if (gi >= m) continue;
#pragma unroll
    for (int p = 0; p < TN; ++p) {
      int gj = j0 + ty + 16 * p;
      if (gj >= n) continue;
      if (OUT == OUT_PART) {
        C[(size_t)blockIdx.z * ldc * n + (size_t)gj * ldc + gi] = acc[q][p];
      } else {
        if (OUT == OUT_SUB_LOWER && gi < gj) continue;
        C[(size_t)gj * ldc + gi] -= acc[q][p];
      }
    }
  }
}

template <typename T, int BN, int AMODE, int BMODE, int OUT>
static int gemm_launch4(int m, int n, int k, const T* A, int lda, const T* B, int ldb, T* C,
                        int ldc, int splits, const int* info, cudaStream_t s) {
  dim3 grid;
  int kchunk = k;
  if (OUT == OUT_SUB_LOWER) {
    long long tiles = tri_tiles(cdiv(m, GBM));
    grid = dim3((unsigned)tiles, 1, 1);
  } else {
    grid = dim3(cdiv(m, GBM), cdiv(n, BN), 1);
    if (OUT == OUT_PART) {
      kchunk = (int)round_up((size_t)cdiv(k, splits), GBK);
      grid.z = cdiv(k, kchunk);
    }
  }
  k_gemm<T, BN, AMODE, BMODE, OUT><<<grid, 256, 0, s>>>(m, n, k, A, lda, B, ldb, C, ldc, kchunk,
                                                        info);
  return launched();
}

template <typename T, int AMODE, int BMODE, int OUT>
static int gemm_bn(int m, int n, int k, const T* A, int lda, const T* B, int ldb, T* C, int ldc,
                   int splits, const int* info, cudaStream_t s) {
  if (OUT == OUT_SUB_LOWER || n > 32)
    return gemm_launch4<T, 64, AMODE, BMODE, OUT>(m, n, k, A, lda, B, ldb, C, ldc, splits, info, s);
  if (n > 16)
    return gemm_launch4<T, 32, AMODE, BMODE, OUT>(m, n, k, A, lda, B, ldb, C, ldc, splits, info, s);
  return gemm_launch4<T, 16, AMODE, BMODE, OUT>(m, n, k, A, lda, B, ldb, C, ldc, splits, info, s);
}

template <typename T>
int launch_gemm(int m, int n, int k, const T* A, int lda, int amode, const T* B, int ldb,
                int bmode, T* C, int ldc, int out, int splits, const int* info, cudaStream_t s) {
  if (m <= 0 || n <= 0 || k <= 0) return JMG_OK;
#define JMG_G(AM, BM, OU) \
  if (amode == AM && bmode == BM && out == OU) \
    return gemm_bn<T, AM, BM, OU>(m, n, k, A, lda, B, ldb, C, ldc, splits, info, s);
  JMG_G(MODE_N, MODE_T, OUT_SUB_LOWER)  // SYRK: C -= P P^T
  JMG_G(MODE_N, MODE_N, OUT_SUB)        // forward-solve update: B -= L Y
  JMG_G(MODE_T, MODE_N, OUT_SUB)        // back-solve update: B -= L^T X
  JMG_G(MODE_S, MODE_N, OUT_PART)       // symmetric residual partials
  JMG_G(MODE_N, MODE_T, OUT_SUB)        // general C -= A B^T
#undef JMG_G
  return JMG_ERR_UNSUPPORTED;
}
template int launch_gemm<double>(int, int, int, const double*, int, int, const double*, int, int,
                                 double*, int, int, int, const int*, cudaStream_t);

// ============================================================================
// FP64 residual R = B - A X (A symmetric, lower stored): split-K partial sums of
// A X through the tiled GEMM (mode S), then a fixed-order reduction that also
// records the per-column infinity norms of r, x and b.
// ============================================================================
int residual_splits(int n, int nrhs) {
  // enough CTAs for ~8 per SM on 152 SMs, never chunks shorter than 256
  long long tiles = (long long)cdiv(n, GBM) * cdiv(nrhs, nrhs > 32 ? 64 : (nrhs > 16 ? 32 : 16));
  long long want = 152LL * 8;
  int splits = (int)((want + tiles - 1) / tiles);
  int maxs = max(1, n / 256);
  return max(1, min(splits, maxs));
}

__global__ void k_resid_reduce(int n, int nrhs, int splits, const double* __restrict__ part,
                               const double* __restrict__ X, int ldx, const double* __restrict__ B,
                               int ldb, double* __restrict__ R, int ldr, double* __restrict__ colmax) {
  const int c = blockIdx.y;
  double rm = 0.0, xm = 0.0, bm = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int z = 0; z < splits; ++z) acc += part[(size_t)z * n * nrhs + (size_t)c * n + i];
    // B == nullptr: plain product (PCG's Q = A P) instead of the residual
    double b = B ? B[(size_t)c * ldb + i] : 0.0;
    double r = B ? b - acc : acc;
    R[(size_t)c * ldr + i] = r;
    double x = X[(size_t)c * ldx + i];
    rm = (isnan(r) || isnan(rm)) ? NAN : fmax(rm, fabs(r));
    xm = (isnan(x) || isnan(xm)) ? NAN : fmax(xm, fabs(x));
    bm = fmax(bm, fabs(b));
  }
  // warp then block max
  for (int o = 16; o > 0; o >>= 1) {
    double a = __shfl_xor_sync(0xffffffffu, rm, o);
    rm = (isnan(a) || isnan(rm)) ? NAN : fmax(rm, a);
    a = __shfl_xor_sync(0xffffffffu, xm, o);
    xm = (isnan(a) || isnan(xm)) ? NAN : fmax(xm, a);
    bm = fmax(bm, __shfl_xor_sync(0xffffffffu, bm, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomic_max_nonneg(&colmax[c], rm);
    atomic_max_nonneg(&colmax[nrhs + c], xm);
    atomic_max_nonneg(&colmax[2 * nrhs + c], bm);
  }
}

int launch_resid_reduce(int n, int nrhs, int used, const double* part, const double* X, int ldx,
                        const double* B, int ldb, double* R, int ldr, double* colmax,
                        cudaStream_t s) {
  dim3 grid(min(cdiv(n, 256), 64), nrhs);
  k_resid_reduce<<<grid, 256, 0, s>>>(n, nrhs, used, part, X, ldx, B, ldb, R, ldr, colmax);
  return launched();
}

int launch_residual(int n, int nrhs, const double* A, int lda, const double* X, int ldx,
                    const double* B, int ldb, double* R, int ldr, double* colmax, double* part,
                    int splits, cudaStream_t s, cudaEvent_t ev0, cudaEvent_t ev1) {
  if (n <= 0 || nrhs <= 0) return JMG_OK;
  JMG_CUDA(cudaMemsetAsync(colmax, 0, sizeof(double) * 3 * nrhs, s));
  if (ev0) JMG_CUDA(cudaEventRecord(ev0, s));
  JMG_TRY(launch_gemm<double>(n, nrhs, n, A, lda, MODE_S, X, ldx, MODE_N, part, n, OUT_PART, splits,
                              nullptr, s));
  if (ev1) JMG_CUDA(cudaEventRecord(ev1, s));
  // number of splits actually used by the GEMM grid
  int kchunk = (int)round_up((size_t)cdiv(n, splits), GBK);
  int used = cdiv(n, kchunk);
  dim3 grid(min(cdiv(n, 256), 64), nrhs);
  k_resid_reduce<<<grid, 256, 0, s>>>(n, nrhs, used, part, X, ldx, B, ldb, R, ldr, colmax);
  return launched();
}

// Row statistics of the symmetric A from its lower triangle:
//   rowsum[i] = sum_j |a_ij|   (NaN propagates; ||A||_inf = max_i rowsum[i])
//   rowmax[i] = max_j |a_ij| truncated to its upper 32 bits (sign, exponent
//               and 20 leading fraction bits): the same binary exponent as the
//               maximum, which is all the row scales of the split residual use
// over the full row j = 0..n-1.  One CTA per strip of 16 columns j reads them
// down from the diagonal in 1024-row chunks (long contiguous runs of each
// column, 16 loads in flight per thread).  Entry a_rj (r > j) adds to row r --
// kept per thread for its four rows of the chunk and flushed with one atomic
// per row and chunk -- and to row j (its mirror), kept per thread for the
// strip's 16 columns and reduced across the CTA at the end; a_jj adds once.
// The maxima are taken on the upper 32 bits of |a| as unsigned integers,
// which order like the values (NaN above every finite value).
// Bound by the FP64 pipe (one warp instruction per 16 clocks and SM), so an entry
// costs its two additions and nothing else there (its sign is cleared in the upper
// word), and strips of 16 columns let two CTAs share an SM: n = 16384 1326 -> 607 us
// (strips of 32, one CTA, a third FP64 operation for the sign).
constexpr int STATS_W = 16;
__global__ void __launch_bounds__(256, 2) k_row_stats(int n, const double* __restrict__ A,
                                                      int lda, double* __restrict__ rowsum,
                                                      double* __restrict__ rowmax) {
  constexpr int W = STATS_W, U = 4, TH = 256, JB = 4;
  __shared__ double red_s[TH / 32][W];
  __shared__ unsigned red_m[TH / 32][W];
  const int j0 = blockIdx.x * W;
  const int jn = min(W, n - j0);
  const int t = threadIdx.x, lane = t % 32, warp = t / 32;
  double cs[W];
  unsigned cm[W];
#pragma unroll
  for (int jj = 0; jj < W; ++jj) cs[jj] = 0.0, cm[jj] = 0u;
  for (int rb = j0; rb < n; rb += TH * U) {
    double rs[U];
    unsigned rm[U];
#pragma unroll
    for (int u = 0; u < U; ++u) rs[u] = 0.0, rm[u] = 0u;
    const double* col = A + (size_t)j0 * lda + rb + t;  // (column j0, row rb + t)
    const bool inner = rb >= j0 + W && rb + TH * U <= n;  // all rows below the strip's diagonal
    const int rt = rb + t - j0, rows = n - (rb + t);      // row in the strip, rows left
#pragma unroll
    for (int jb = 0; jb < W; jb += JB) {
      double v[JB][U];
#pragma unroll
      for (int q = 0; q < JB; ++q) {  // JB x U independent loads
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = TH * u;
          v[q][u] = (inner && jn == W) || (jb + q < jn && rt + i >= jb + q && i < rows) ? col[i] : 0.0;
        }
        col += lda;
      }
#pragma unroll
      for (int q = 0; q < JB; ++q)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const unsigned hi = (unsigned)__double2hiint(v[q][u]) & 0x7fffffffu;
          const double av = __hiloint2double((int)hi, __double2loint(v[q][u]));
          rs[u] += av;
          rm[u] = max(rm[u], hi);
          if (inner || rt + TH * u > jb + q) {
            cs[jb + q] += av;
            cm[jb + q] = max(cm[jb + q], hi);
          }
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int r = rb + t + TH * u;
      if (r < n) {
        if (rowsum) atomicAdd(&rowsum[r], rs[u]);
        if (rowmax) atomicMax(reinterpret_cast<unsigned*>(&rowmax[r]) + 1, rm[u]);
      }
    }
  }
  // the mirrored part of the strip's rows: reduce the column sums over the CTA
#pragma unroll
  for (int jj = 0; jj < W; ++jj) {
    double a = cs[jj];
    unsigned m = cm[jj];
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
    if (lane == jj) {
      red_s[warp][jj] = a;
      red_m[warp][jj] = m;
    }
  }
  __syncthreads();
  if (t < jn) {
    double a = 0.0;
    unsigned m = 0u;
#pragma unroll
    for (int w = 0; w < TH / 32; ++w) {
      a += red_s[w][t];
      m = max(m, red_m[w][t]);
    }
    if (rowsum) atomicAdd(&rowsum[j0 + t], a);
    if (rowmax) atomicMax(reinterpret_cast<unsigned*>(&rowmax[j0 + t]) + 1, m);
  }
}

int launch_row_stats(int n, const double* A, int lda, double* rowsum, double* rowmax,
                     cudaStream_t s) {
  if (n <= 0) return JMG_OK;
  if (rowsum) JMG_CUDA(cudaMemsetAsync(rowsum, 0, sizeof(double) * n, s));
  if (rowmax) JMG_CUDA(cudaMemsetAsync(rowmax, 0, sizeof(double) * n, s));
  k_row_stats<<<cdiv(n, STATS_W), 256, 0, s>>>(n, A, lda, rowsum, rowmax);
  return launched();
}

__global__ void k_max_reduce(int n, const double* __restrict__ v, double* __restrict__ out) {
  double m = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    m = (isnan(v[i]) || isnan(m)) ? NAN : fmax(m, v[i]);
  for (int o = 16; o > 0; o >>= 1) {
    double a = __shfl_xor_sync(0xffffffffu, m, o);
    m = (isnan(a) || isnan(m)) ? NAN : fmax(m, a);
  }
  if ((threadIdx.x & 31) == 0) atomic_max_nonneg(out, m);
}

int launch_max_reduce(int n, const double* v, double* out, cudaStream_t s) {
  JMG_CUDA(cudaMemsetAsync(out, 0, sizeof(double), s));
  if (n <= 0) return JMG_OK;
  k_max_reduce<<<min(cdiv(n, 256), 152), 256, 0, s>>>(n, v, out);
  return launched();
}

int launch_norm_inf(int n, const double* A, int lda, double* rowsum, double* out,
                    cudaStream_t s) {
  JMG_TRY(launch_row_stats(n, A, lda, rowsum, nullptr, s));
  return launch_max_reduce(n, rowsum, out, s);
}

__global__ void k_eta(int nrhs, const double* __restrict__ colmax, const double* __restrict__ anorm,
                      double* __restrict__ eta) {
  // single warp
  double worst = 0.0;
  for (int c = threadIdx.x; c < nrhs; c += 32) {
    double rn = colmax[c], xn = colmax[nrhs + c], bn = colmax[2 * nrhs + c];
    double den = (*anorm) * xn + bn;
    double e = den > 0.0 ? rn / den : (rn > 0.0 ? INFINITY : 0.0);
    if (isnan(rn) || isnan(xn)) e = NAN;
    eta[1 + c] = e;
    worst = (isnan(e) || isnan(worst)) ? NAN : fmax(worst, e);
  }
  for (int o = 16; o > 0; o >>= 1) {
    double a = __shfl_xor_sync(0xffffffffu, worst, o);
    worst = (isnan(a) || isnan(worst)) ? NAN : fmax(worst, a);
  }
  if (threadIdx.x == 0) eta[0] = worst;
}

int launch_eta(int nrhs, const double* colmax, const double* anorm, double* eta_out,
               cudaStream_t s) {
  k_eta<<<1, 32, 0, s>>>(nrhs, colmax, anorm, eta_out);
  return launched();
}

// ============================================================================
// Conversions used by the mixed-precision path.
// ============================================================================
__global__ void k_lower_to_f32(int n, const double* __restrict__ A, int lda, float* __restrict__ W,
                               int ldw, double shift) {
  // one CTA per column, rows j..n-1
  const int j = blockIdx.x;
  for (int i = j + threadIdx.x; i < n; i += blockDim.x) {
    double v = A[(size_t)j * lda + i];
    if (i == j) v += shift;
    W[(size_t)j * ldw + i] = (float)v;
  }
}

int launch_lower_to_f32(int n, const double* A, int lda, float* W, int ldw, double shift,
                        cudaStream_t s) {
  if (n <= 0) return JMG_OK;
  k_lower_to_f32<<<n, 256, 0, s>>>(n, A, lda, W, ldw, shift);
  return launched();
}

__global__ void k_scale_to_f32(int n, const double* __restrict__ R, int ldr,
                               const double* __restrict__ colmax_r, float* __restrict__ D, int ldd) {
  const int c = blockIdx.y;
  double sc = colmax_r[c];
  double inv = (sc > 0.0 && isfinite(sc)) ? 1.0 / sc : 1.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    D[(size_t)c * ldd + i] = (float)(R[(size_t)c * ldr + i] * inv);
}

int launch_scale_to_f32(int n, int nrhs, const double* R, int ldr, const double* colmax_r,
                        float* D, int ldd, cudaStream_t s) {
  dim3 grid(min(cdiv(n, 256), 64), nrhs);
  k_scale_to_f32<<<grid, 256, 0, s>>>(n, R, ldr, colmax_r, D, ldd);
  return launched();
}

__global__ void k_axpy_f32(int n, const float* __restrict__ D, int ldd,
                           const double* __restrict__ colmax_r, double* __restrict__ X, int ldx) {
  const int c = blockIdx.y;
  double sc = colmax_r[c];
  if (!(sc > 0.0 && isfinite(sc))) sc = 1.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    X[(size_t)c * ldx + i] += sc * (double)D[(size_t)c * ldd + i];
}

int launch_axpy_f32(int n, int nrhs, const float* D, int ldd, const double* colmax_r, double* X,
                    int ldx, cudaStream_t s) {
  dim3 grid(min(cdiv(n, 256), 64), nrhs);
  k_axpy_f32<<<grid, 256, 0, s>>>(n, D, ldd, colmax_r, X, ldx);
  return launched();
}

int launch_copy2d(int n, int nrhs, const double* src, int lds, double* dst, int ldd,
                  cudaStream_t s) {
  JMG_CUDA(cudaMemcpy2DAsync(dst, sizeof(double) * ldd, src, sizeof(double) * lds,
                             sizeof(double) * n, nrhs, cudaMemcpyDeviceToDevice, s));
  return JMG_OK;
}

int launch_zero(double* p, size_t n, cudaStream_t s) {
  JMG_CUDA(cudaMemsetAsync(p, 0, sizeof(double) * n, s));
  return JMG_OK;
}

}  // namespace jmg

namespace jmg {

// ============================================================================
// Vector kernels of the preconditioned conjugate gradient refinement (FP64,
// one right-hand side per column, columns independent).
// ============================================================================

// out[c] = sum_i U[i,c] V[i,c]; one CTA per column, fixed reduction order.
__global__ void __launch_bounds__(256) k_dot_cols(int n, const double* __restrict__ U, int ldu,
                                                  const double* __restrict__ V, int ldv,
                                                  double* __restrict__ out) {
  __shared__ double part[256];
  const int c = blockIdx.x;
  double a = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) a = fma(U[(size_t)c * ldu + i], V[(size_t)c * ldv + i], a);
  part[threadIdx.x] = a;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[c] = part[0];
}

int launch_dot_cols(int n, int nrhs, const double* U, int ldu, const double* V, int ldv,
                    double* out, cudaStream_t s) {
  k_dot_cols<<<nrhs, 256, 0, s>>>(n, U, ldu, V, ldv, out);
  return launched();
}

// alpha_c = rz_c / pq_c (0 when pq_c <= 0, which also raises *bad);
// X += alpha P, R -= alpha Q; colmax[0..nrhs) = ||R||, [nrhs..2nrhs) = ||X||.
__global__ void k_pcg_step(int n, const double* __restrict__ P, const double* __restrict__ Q,
                           const double* __restrict__ rz, const double* __restrict__ pq,
                           double* __restrict__ X, double* __restrict__ R, int nrhs,
                           double* __restrict__ colmax, int* __restrict__ bad) {
  const int c = blockIdx.y;
  const double den = pq[c];
  double alpha = 0.0;
  if (den > 0.0 && isfinite(den)) {
    alpha = rz[c] / den;
  } else if (rz[c] != 0.0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(bad, 1);
  }
  double rm = 0.0, xm = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const size_t o = (size_t)c * n + i;
    const double x = fma(alpha, P[o], X[o]);
    const double r = fma(-alpha, Q[o], R[o]);
    X[o] = x;
    R[o] = r;
    rm = (isnan(r) || isnan(rm)) ? NAN : fmax(rm, fabs(r));
    xm = (isnan(x) || isnan(xm)) ? NAN : fmax(xm, fabs(x));
  }
  for (int o = 16; o > 0; o >>= 1) {
    double a = __shfl_xor_sync(0xffffffffu, rm, o);
    rm = (isnan(a) || isnan(rm)) ? NAN : fmax(rm, a);
    a = __shfl_xor_sync(0xffffffffu, xm, o);
    xm = (isnan(a) || isnan(xm)) ? NAN : fmax(xm, a);
  }
  if ((threadIdx.x & 31) == 0) {
    atomic_max_nonneg(&colmax[c], rm);
    atomic_max_nonneg(&colmax[nrhs + c], xm);
  }
}

int launch_pcg_step(int n, int nrhs, const double* P, const double* Q, const double* rz,
                    const double* pq, double* X, double* R, double* colmax, int* bad,
                    cudaStream_t s) {
  JMG_CUDA(cudaMemsetAsync(colmax, 0, sizeof(double) * 2 * nrhs, s));
  dim3 grid(std::min(cdiv(n, 256), 64), nrhs);
  k_pcg_step<<<grid, 256, 0, s>>>(n, P, Q, rz, pq, X, R, nrhs, colmax, bad);
  return launched();
}

// P = Z + (rz_new / rz_old) P   (beta = 0 when rz_old == 0); then rz_old = rz_new
__global__ void k_pcg_dir(int n, const double* __restrict__ Z, double* __restrict__ P,
                          const double* __restrict__ rz_new, const double* __restrict__ rz_old) {
  const int c = blockIdx.y;
  const double beta = (rz_old[c] != 0.0) ? rz_new[c] / rz_old[c] : 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const size_t o = (size_t)c * n + i;
    P[o] = fma(beta, P[o], Z[o]);
  }
}

int launch_pcg_dir(int n, int nrhs, const double* Z, double* P, const double* rz_new,
                   const double* rz_old, cudaStream_t s) {
  dim3 grid(std::min(cdiv(n, 256), 64), nrhs);
  k_pcg_dir<<<grid, 256, 0, s>>>(n, Z, P, rz_new, rz_old);
  return launched();
}

// Z = scale_c * D32 (FP64 from the FP32 preconditioner output)
__global__ void k_scale_from_f32(int n, const float* __restrict__ D, int ldd,
                                 const double* __restrict__ colmax_r, double* __restrict__ Z) {
  const int c = blockIdx.y;
  double sc = colmax_r[c];
  if (!(sc > 0.0 && isfinite(sc))) sc = 1.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    Z[(size_t)c * n + i] = sc * (double)D[(size_t)c * ldd + i];
}

int launch_scale_from_f32(int n, int nrhs, const float* D, int ldd, const double* colmax_r,
                          double* Z, cudaStream_t s) {
  dim3 grid(std::min(cdiv(n, 256), 64), nrhs);
  k_scale_from_f32<<<grid, 256, 0, s>>>(n, D, ldd, colmax_r, Z);
  return launched();
}

// max_i A_ii (A_ii > 0 expected; NaN wins) into *out (must be zeroed)
__global__ void k_diag_max(int n, const double* __restrict__ A, int lda, double* __restrict__ out) {
  double m = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double v = A[(size_t)i * lda + i];
    m = (isnan(v) || isnan(m)) ? NAN : fmax(m, fabs(v));
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double a = __shfl_xor_sync(0xffffffffu, m, o);
    m = (isnan(a) || isnan(m)) ? NAN : fmax(m, a);
  }
  if ((threadIdx.x & 31) == 0) atomic_max_nonneg(out, m);
}

int launch_diag_max(int n, const double* A, int lda, double* out, cudaStream_t s) {
  JMG_CUDA(cudaMemsetAsync(out, 0, sizeof(double), s));
  k_diag_max<<<std::max(1, std::min(cdiv(n, 256), 64)), 256, 0, s>>>(n, A, lda, out);
  return launched();
}

}  // namespace jmg

#include <cuda_fp8.h>

namespace jmg {

// ============================================================================
// FP8 quantisation of the panel with one power-of-two scale per 128-row tile
// (the 128 x 128 tiles of a 128-wide panel): one CTA per tile finds amax,
// picks e = floor(log2(448 / amax)) (448 = largest finite e4m3) clamped to
// [-126, 126], and writes q = e4m3_rn_satfinite(x * 2^e) row-major.
// ============================================================================
__global__ void __launch_bounds__(256) k_quant_fp8(int m, int kb, const float* __restrict__ L21,
                                                   int ldw, unsigned char* __restrict__ Q, int ldq,
                                                   signed char* __restrict__ ex) {
  // the tile goes through shared memory (column c at c * 129): read along the
  // columns of L21 (coalesced, 16 loads in flight per thread, amax on the way),
  // written along the rows of Q (four codes per 32-bit store)
  extern __shared__ float qtile[];
  constexpr int LDT = 129;
  __shared__ float red[8];
  __shared__ int s_e;
  const int r0 = blockIdx.x * 128;
  const int rows = min(128, m - r0);
  const int t = threadIdx.x;
  float amax = 0.0f;
  for (int base = 0; base < 128 * kb; base += 256 * 16) {
    float v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int idx = base + t + 256 * q, i = idx & 127, c = idx >> 7;
      v[q] = (idx < 128 * kb && i < rows) ? L21[(size_t)c * ldw + r0 + i] : 0.0f;
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int idx = base + t + 256 * q;
      if (idx < 128 * kb) {
        qtile[(idx >> 7) * LDT + (idx & 127)] = v[q];
        amax = fmaxf(amax, fabsf(v[q]));
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  if ((t & 31) == 0) red[t / 32] = amax;
  __syncthreads();
  if (t == 0) {
    float a = red[0];
    for (int w = 1; w < 8; ++w) a = fmaxf(a, red[w]);
    int e = 0;
    if (a > 0.0f && isfinite(a)) {
      e = (int)floorf(log2f(448.0f / a));
      // guard the rounding of log2f: keep a * 2^e <= 448
      while (e > -126 && ldexpf(a, e) > 448.0f) --e;
      e = max(-126, min(126, e));
    }
    s_e = e;
    ex[blockIdx.x] = (signed char)e;
  }
  __syncthreads();
  const int e = s_e, kq = kb / 4;
  for (int idx = t; idx < rows * kq; idx += 256) {
    const int i = idx / kq, c = (idx % kq) * 4;
    unsigned int w = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float v = ldexpf(qtile[(c + u) * LDT + i], e);
      w |= (unsigned int)(unsigned char)__nv_cvt_float_to_fp8(v, __NV_SATFINITE, __NV_E4M3)
           << (8 * u);
    }
    *reinterpret_cast<unsigned int*>(Q + (size_t)(r0 + i) * ldq + c) = w;
  }
}

int launch_quant_fp8(int m, int kb, const float* L21, int ldw, void* Q, int ldq, signed char* e,
                     cudaStream_t s) {
  if (m <= 0) return JMG_OK;
  if (kb % 4 || ldq % 4 || (reinterpret_cast<uintptr_t>(Q) & 3)) return JMG_ERR_ALIGN;
  const int smem = (int)sizeof(float) * kb * 129;
  JMG_TRY(ensure_smem(k_quant_fp8, smem));
  k_quant_fp8<<<cdiv(m, 128), 256, smem, s>>>(m, kb, L21, ldw, (unsigned char*)Q, ldq, e);
  return launched();
}

}  // namespace jmg
