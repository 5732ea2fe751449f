// k_batched.cu -- many small independent systems A_b X_b = B_b (n <= 128), one CTA
// per system (paper: "Summary", potrs under vectorisation over a batch).
#include <type_traits>

#include "kernels.h"
#include "rcp64.cuh"

namespace jmg {

// ============================================================================
// Factor and solve in one kernel, FP64 arithmetic on T storage.  The factor is
// kept unscaled: column j holds a_rj, w_j = 1 / a_jj, and u_rj = a_rj w_j goes to
// the mirrored place above the diagonal, so that
//   update     a_rc -= a_rj u_cj        (one FMA per element, full warps: columns
//                                        j1 .. j2 are a range of the packed column-major
//                                        order)
//   forward    b_k  -= b_j u_kj         (k > j)
//   backward   x_k   = b_k w_k - sum_{i > k} u_ik x_i
// need one FP64 instruction per element and no division (the pivot's reciprocal
// runs on the integer pipe); l_rc = a_rc / sqrt(a_cc) is formed once at the end.
// Columns come in blocks of JB: a column updates its own block at once, the columns
// behind it with the block's other columns, as one sum of products subtracted from a_rc
// once.  An entry is then rounded n / JB + JB times at its own size instead of n times,
// which set the error (root mean square, of the largest entry): L at order 128 2.8e-16
// with a rounding per column, 1.6e-16 with blocks of 32, 1.3e-16 with 16, X 9.4e-16, 6.7e-16
// and 6.2e-16; L at order 48 1.7e-16, 1.5e-16 and 1.2e-16, X 5.9e-16, 5.1e-16 and 4.5e-16 (the
// blocked kernels before: 1.6, 6.9, 1.5 and 5.4e-16).  Time in the same order, one
// right-hand side: 1000 systems of order 48 78, 80 and 84 us, 20000 - , 1436 and 1413; 1000
// of order 128 1302, 1339 and 1348.
// Bound by the FP64 pipe (one warp instruction per ~16 clocks and SM) with enough
// systems resident per SM to cover the column chain: two barriers per column, none
// in the solve.  1000 FP64 systems, one right-hand side: order 16 21 us, 48 83, 128
// 1348 (83, 611 and 8877 us with a factor kernel of 256 threads and a solve with one
// thread per right-hand side).
// The solve spreads 32 / KG right-hand sides over a warp, KG lanes each (as many
// lanes as fill the warps, from 32 for one right-hand side per warp down to 4): the
// fewer lanes share a right-hand side, the fewer of them idle past the diagonal.
// ============================================================================
namespace bat {
constexpr int NMAX = 128;
constexpr int JB = 16;  // columns per block
// Pivots at the ends of T's range, whose reciprocal is not a normal number of T.  The fast
// path multiplies by it; this one (not inlined: nothing of it is to cost the fast one
// registers) divides, with the finished factor, one thread per right-hand side.
template <typename T>
JMG_DEV bool out_of_range(T w) {
  constexpr T least = sizeof(T) == 8 ? (T)0x1p-1022 : (T)0x1p-126f;
  return !(w >= least && w <= 1 / least);
}
template <typename T>
__device__ __noinline__ void solve_by_division(const T* L, int lda, int n, int nrhs, T* B, int ldb) {
  for (int q = threadIdx.x; q < nrhs; q += blockDim.x) {
    T* b = B + (size_t)q * ldb;
    for (int j = 0; j < n; ++j) {
      const T y = b[j] / L[(size_t)j * lda + j];
      b[j] = y;
      for (int k = j + 1; k < n; ++k) b[k] -= L[(size_t)j * lda + k] * y;
    }
    for (int j = n - 1; j >= 0; --j) {
      T x = b[j];
      for (int k = j + 1; k < n; ++k) x -= L[(size_t)j * lda + k] * b[k];
      b[j] = x / L[(size_t)j * lda + j];
    }
  }
}
// v (component k = g + KG h on lane g of the right-hand side's KG) <- U^-T D^-1 U^-1 v
// with u_kj = U[k * ld + j], j < k, and w_k = 1 / d_k
template <typename T, int KG, int H>
JMG_DEV void solve_one(const T* U, int ld, const T* w, int n, T (&v)[H], int g) {
#pragma unroll
  for (int hj = 0; hj < H; ++hj) {  // forward
    const int je = min(KG, n - KG * hj);
#pragma unroll 1
    for (int jj = 0; jj < je; ++jj) {
      const T bj = __shfl_sync(0xffffffffu, v[hj], jj, KG);
      const int j = KG * hj + jj;
#pragma unroll
      for (int h = hj; h < H; ++h) {
        const int k = g + KG * h;
        if (k > j && k < n) v[h] = fma(-U[k * ld + j], bj, v[h]);
      }
    }
  }
#pragma unroll
  for (int h = 0; h < H; ++h)
    if (g + KG * h < n) v[h] *= w[g + KG * h];
#pragma unroll
  for (int hj = H - 1; hj >= 0; --hj) {  // backward
#pragma unroll 1
    for (int jj = min(KG, n - KG * hj) - 1; jj >= 0; --jj) {
      const T xi = __shfl_sync(0xffffffffu, v[hj], jj, KG);
      const int i = KG * hj + jj;
#pragma unroll
      for (int h = 0; h <= hj; ++h) {
        const int k = g + KG * h;
        if (k < i) v[h] = fma(-U[i * ld + k], xi, v[h]);
      }
    }
  }
}
// every right-hand side of one system; warp w0 takes the first ones
template <typename T, int KG, int H>
JMG_DEV void solve_all(const T* U, int ld, const T* w, int n, int nrhs, T* B, int ldb, int w0,
                       int nw, int lane) {
  constexpr int RG = 32 / KG;
  const int g = lane % KG;
  for (int q0 = w0 * RG; q0 < nrhs; q0 += nw * RG) {
    const int q = q0 + lane / KG;
    T v[H];
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const int k = g + KG * h;
      v[h] = k < n && q < nrhs ? B[(size_t)q * ldb + k] : T(0);
    }
    solve_one<T, KG, H>(U, ld, w, n, v, g);
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const int k = g + KG * h;
      if (k < n && q < nrhs) B[(size_t)q * ldb + k] = v[h];
    }
  }
}
}  // namespace bat

// n <= KG * H.  FP32 storage: the solve runs in FP32 on u and w rounded once.
template <typename T, int KG, int H>
__global__ void __launch_bounds__(KG* H <= 64 ? 128 : 512) k_posv_batched(int n, int nrhs, T* __restrict__ A, int lda, long long sA,
                               T* __restrict__ B, int ldb, long long sB, int* __restrict__ info) {
  extern __shared__ __align__(16) double sm_bat[];
  const int ld = n | 1;  // odd: rows and columns are free of bank conflicts
  double* s = sm_bat;             // s[c * ld + r] = a_rc (r >= c), u_cr (r < c)
  double* s_w = s + n * ld;       // 1 / a_jj
  double* s_l = s_w + n;          // sqrt(a_jj)
  double* s_il = s_l + n;         // 1 / sqrt(a_jj)
  unsigned short* s_rc = reinterpret_cast<unsigned short*>(s_il + n);  // packed -> (c, r)
  T* Ab = A + (size_t)blockIdx.x * sA;
  const int t = threadIdx.x, nt = blockDim.x, lane = t % 32, warp = t / 32, nw = nt / 32;
  for (int c = warp; c < n; c += nw) {
    const int base = c * n - c * (c - 1) / 2;
    for (int r = c + lane; r < n; r += 32) {
      s[c * ld + r] = (double)Ab[(size_t)c * lda + r];
      s_rc[base + r - c] = (unsigned short)((c << 8) | r);
    }
  }
  __syncthreads();
  const int nel = n * (n + 1) / 2;
  int fail = n;  // first failing column
  auto column = [&](int c) { return c * n - c * (c - 1) / 2; };  // its start in packed order
  for (int p = 0; p < n && fail == n; p += bat::JB) {
    const int pe = min(n, p + bat::JB), e2 = column(pe);
    for (int j = p; j < pe; ++j) {
      const double d = s[j * ld + j];
      bool bad = false;
      // u_j: the warps that hold rows below j (and the first one, for w_j)
      if (32 * warp < n - 1 - j || warp == 0) {
        const double w = pivot_rcp(d, &bad);
        if (t == 0) s_w[j] = w;
          for (int r = j + 1 + t; r < n; r += nt) s[r * ld + j] = s[j * ld + r] * w;
      }
      if (!(d > 0.0)) {  // (the same value on every thread)
        fail = j;
        break;
      }
      __syncthreads();
      if (j + 1 == pe) break;
      for (int e = column(j + 1) + t; e < e2; e += nt) {
        const int rc = s_rc[e], c = rc >> 8, r = rc & 255;
        s[c * ld + r] = fma(-s[j * ld + r], s[c * ld + j], s[c * ld + r]);
      }
      __syncthreads();
    }
    if (fail < n || pe == n) break;  // (a block with columns behind it is a full one)
    for (int e = e2 + t; e < nel; e += nt) {
      const int rc = s_rc[e], c = rc >> 8, r = rc & 255;
      const double *a = s + p * ld + r, *u = s + c * ld + p;
      double sum = a[0] * u[0];
#pragma unroll
      for (int j = 1; j < bat::JB; ++j) sum = fma(a[j * ld], u[j], sum);
      s[c * ld + r] -= sum;
    }
    __syncthreads();
  }
  bool odd = false;
  if (t < fail) {
    s_l[t] = sqrt(s[t * ld + t]);
    s_il[t] = 1.0 / s_l[t];
    odd = bat::out_of_range((T)s_w[t]);
  }
  odd = __syncthreads_or(odd);
  for (int c = warp; c < fail; c += nw)
    for (int r = c + lane; r < n; r += 32)
      Ab[(size_t)c * lda + r] = (T)(r == c ? s_l[c] : s[c * ld + r] * s_il[c]);
  if (t == 0) info[blockIdx.x] = fail < n ? fail + 1 : 0;
  if (fail < n) return;
  T* Bb = B + (size_t)blockIdx.x * sB;
  if (odd) {
    __syncthreads();  // the factor is in global memory
    bat::solve_by_division(Ab, lda, n, nrhs, Bb, ldb);
    return;
  }
  const int w0 = (warp + blockIdx.x) % nw;  // the first right-hand side takes turns over the quarters
  if constexpr (sizeof(T) == 8) {
    bat::solve_all<T, KG, H>(s, ld, s_w, n, nrhs, Bb, ldb, w0, nw, lane);
  } else {
    float* U = reinterpret_cast<float*>(s_rc + (nel + 1) / 2 * 2);
    float* w = U + n * ld;
    for (int r = 1 + warp; r < n; r += nw)
      for (int c = lane; c < r; c += 32) U[r * ld + c] = (float)s[r * ld + c];
    if (t < n) w[t] = (float)s_w[t];
    __syncthreads();
    bat::solve_all<T, KG, H>(U, ld, w, n, nrhs, Bb, ldb, w0, nw, lane);
  }
}

// ============================================================================
// FP32 storage above order 48: the factors come from k_potrf_diag_batched (k_dense.cu:
// FP64 in the 32 x 32 diagonal sub-blocks only), the solve runs in FP32 on them, four
// warps per system, eight above 32 right-hand sides.  U lies behind w: in front of them
// the same loops took 1.2-1.3 times as long from 32 right-hand sides on (1000 systems of
// order 56, 70 right-hand sides: 274 -> 205 us, 264 with one thread per right-hand side).
// ============================================================================
template <int KG, int H>
__global__ void __launch_bounds__(256) k_potrs_batched_f32(int n, int nrhs,
                                                           const float* __restrict__ L, int lda,
                                                           long long sA, float* __restrict__ B,
                                                           int ldb, long long sB,
                                                           const int* __restrict__ info) {
  extern __shared__ __align__(16) float sm_bat32[];
  if (info[blockIdx.x] != 0) return;
  const int ld = n | 1;
  float* w = sm_bat32;  // 1 / l_cc^2
  float* s_l = w + n;   // l_cc
  float* U = s_l + n;   // U[r * ld + c] = l_rc / l_cc
  const float* Lb = L + (size_t)blockIdx.x * sA;
  const int t = threadIdx.x, nt = blockDim.x, lane = t % 32, warp = t / 32, nw = nt / 32;
  bool odd = false;
  for (int c = t; c < n; c += nt) {
    const float l = Lb[(size_t)c * lda + c];
    s_l[c] = l;
    w[c] = 1.0f / l / l;
    odd |= bat::out_of_range(w[c]);
  }
  if (__syncthreads_or(odd)) {
    bat::solve_by_division(Lb, lda, n, nrhs, B + (size_t)blockIdx.x * sB, ldb);
    return;
  }
  for (int c = warp; c < n; c += nw)
    for (int r = c + 1 + lane; r < n; r += 32) U[r * ld + c] = Lb[(size_t)c * lda + r] / s_l[c];
  __syncthreads();
  bat::solve_all<float, KG, H>(U, ld, w, n, nrhs, B + (size_t)blockIdx.x * sB, ldb, warp, nw, lane);
}

// f(KG, H) for a system of order n and `per` right-hand sides per warp
template <typename F>
static int by_shape(int n, int per, F f) {
  using std::integral_constant;
#define JMG_B(KG)                                                                              \
  return n <= 32 ? f(integral_constant<int, KG>(), integral_constant<int, 32 / KG>())          \
                 : (n <= 64 ? f(integral_constant<int, KG>(), integral_constant<int, 64 / KG>()) \
                            : f(integral_constant<int, KG>(), integral_constant<int, 128 / KG>()))
  if (per <= 1) JMG_B(32);
  if (per <= 2) JMG_B(16);
  if (per <= 4 || n > 64) JMG_B(8);  // (4 lanes above order 64: 32 registers, slower than 8)
  JMG_B(4);
#undef JMG_B
}

template <typename T>
static int fused_launch(int n, int nrhs, int batch, T* A, int lda, long long sA, T* B, int ldb,
                        long long sB, int* info, cudaStream_t s) {
  const size_t nel = (size_t)n * (n + 1) / 2;
  const size_t smem = sizeof(double) * ((size_t)n * (n | 1) + 3 * n) + sizeof(short) * ((nel + 1) / 2 * 2) +
                      (sizeof(T) == 4 ? sizeof(float) * ((size_t)n * (n | 1) + n) : 0);
  // threads: enough for a column's rows and the trailing triangle of the first columns,
  // few enough for many systems per SM.  1000 FP64 systems, one right-hand side, half as
  // many / these / twice as many: order 24 38 / 31 / 30 us, 48 87 / 83 / 128, 80 403 / 365 /
  // 360, 128 1408 / 1349 / - (order 64 215 / 209 / 181, 96 656 / 610 / 572).
  const int nt = n <= 24 ? 64 : (n <= 64 ? 128 : (n <= 96 ? 256 : 512));
  return by_shape(n, cdiv(nrhs, nt / 32), [&](auto kg, auto h) -> int {
    auto k = k_posv_batched<T, decltype(kg)::value, decltype(h)::value>;
    JMG_TRY(ensure_smem(k, (int)smem));
    k<<<batch, nt, smem, s>>>(n, nrhs, A, lda, sA, B, ldb, sB, info);
    return launched();
  });
}

template <>
int posv_small_batched<double>(int n, int nrhs, int batch, double* A, int lda, long long sA,
                               double* B, int ldb, long long sB, int* info, cudaStream_t s) {
  if (n > bat::NMAX) return JMG_ERR_UNSUPPORTED;
  if (n == 0 || batch == 0) {
    JMG_CUDA(cudaMemsetAsync(info, 0, sizeof(int) * (size_t)batch, s));
    return JMG_OK;
  }
  return fused_launch<double>(n, nrhs, batch, A, lda, sA, B, ldb, sB, info, s);
}

template <>
int posv_small_batched<float>(int n, int nrhs, int batch, float* A, int lda, long long sA,
                              float* B, int ldb, long long sB, int* info, cudaStream_t s) {
  if (n > bat::NMAX) return JMG_ERR_UNSUPPORTED;
  // up to order 48 the factor in FP64 throughout (k_posv_batched): half the error of the
  // factor of larger orders (L at order 48 2.5e-8 / 4.9e-8).  1000 systems, one right-hand
  // side, this / that: order 25 31 / 47 us, 40 61 / 68, 48 88 / 82, 56 164 / 91.
  if (n > 0 && batch > 0 && n <= 48)
    return fused_launch<float>(n, nrhs, batch, A, lda, sA, B, ldb, sB, info, s);
  JMG_CUDA(cudaMemsetAsync(info, 0, sizeof(int) * (size_t)batch, s));
  if (n == 0 || batch == 0) return JMG_OK;
  JMG_TRY(launch_potf2_batched(n, batch, A, lda, sA, info, s));
  if (nrhs == 0) return JMG_OK;
  const size_t smem = sizeof(float) * ((size_t)n * (n | 1) + 2 * n);
  const int nt = nrhs <= 32 ? 128 : 256;
  return by_shape(n, cdiv(nrhs, nt / 32), [&](auto kg, auto h) -> int {
    auto k = k_potrs_batched_f32<decltype(kg)::value, decltype(h)::value>;
    JMG_TRY(ensure_smem(k, (int)smem));
    k<<<batch, nt, smem, s>>>(n, nrhs, A, lda, sA, B, ldb, sB, info);
    return launched();
  });
}

}  // namespace jmg
