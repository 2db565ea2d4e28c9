// FP64 GEMM on the DFMA pipe: the "native FP64" path of the Gram product
// G = J~^T J~ (Methods, "Second-order Optimizer"), the CCF Hilbert contraction
// J_U = K J_g, and the trailing updates of the blocked Cholesky factorisation.
//
// GB300 executes FP64 at roughly 1/60 of its FP32 rate (one warp instruction per 17 clocks and
// SM, 1.19 TFLOP/s in all), so every shape used here is bound by that pipe and by how evenly the
// output tiles fill the 152 SMs; shared-memory and L2 traffic are far below their limits even for
// 16 x 16 tiles.  K is staged through shared memory 16 at a time with a register prefetch of the
// next stage.  Operand layouts are template parameters so that J~ (row-major, rows x P') serves as
// both J~^T and J~ without a transpose copy.
#include "gn_internal.cuh"

namespace gn {
namespace {

constexpr int BK = 16;

// T x T output tile, each thread R x R outputs (rows ty + NT i, columns tx + NT j), K staged 16 at
// a time.  KG groups of (T / R)^2 threads share the tile: group g takes every KG-th K stage, and
// the groups' sums are added in group order at the end.
template <int T, int R, int KG, bool AK, bool BKC>
__global__ void __launch_bounds__(KG * (T / R) * (T / R)) dgemm_kernel(int64_t m, int64_t n, int64_t k, double alpha,
                                                                       const double* __restrict__ A, int64_t lda,
                                                                       const double* __restrict__ B, int64_t ldb,
                                                                       double beta, double* C, int64_t ldc, int lower,
                                                                       const double* __restrict__ rowscale) {
  constexpr int NT = T / R, THREADS = NT * NT;
  constexpr int KR = THREADS / BK;      // operand rows loaded per pass, K contiguous in memory
  constexpr int MR = THREADS / T;       // K steps loaded per pass, rows contiguous in memory
  constexpr int LD = T * BK / THREADS;  // elements of one operand per thread and stage
  const int bm = blockIdx.y, bn = blockIdx.x;
  if (lower && bn > bm) return;
  __shared__ double Asm[KG][BK][T + 1];
  __shared__ double Bsm[KG][BK][T + 1];
  const int t = threadIdx.x % THREADS, kg = threadIdx.x / THREADS;
  double (*As)[T + 1] = Asm[kg];
  double (*Bs)[T + 1] = Bsm[kg];
  const int tx = t % NT, ty = t / NT;
  const int64_t m0 = (int64_t)bm * T, n0 = (int64_t)bn * T;
  double acc[R][R];
#pragma unroll
  for (int i = 0; i < R; i++)
#pragma unroll
    for (int j = 0; j < R; j++) acc[i][j] = 0.0;
  double ra[LD], rb[LD];
  auto load = [&](int64_t k0) {
#pragma unroll
    for (int r = 0; r < LD; r++) {
      const int mm = AK ? t / BK + KR * r : t % T, kk = AK ? t % BK : t / T + MR * r;
      const int64_t gm = m0 + mm, gk = k0 + kk;
      ra[r] = (gm < m && gk < k) ? (AK ? A[gm * lda + gk] : A[gk * lda + gm]) : 0.0;
      const int nn = BKC ? t / BK + KR * r : t % T, kb = BKC ? t % BK : t / T + MR * r;
      const int64_t gn = n0 + nn, gkb = k0 + kb;
      rb[r] = (gn < n && gkb < k) ? (BKC ? B[gn * ldb + gkb] : B[gkb * ldb + gn]) : 0.0;
    }
  };
  auto store = [&]() {
#pragma unroll
    for (int r = 0; r < LD; r++) {
      if (AK) As[t % BK][t / BK + KR * r] = ra[r];
      else As[t / T + MR * r][t % T] = ra[r];
      if (BKC) Bs[t % BK][t / BK + KR * r] = rb[r];
      else Bs[t / T + MR * r][t % T] = rb[r];
    }
  };
  load((int64_t)kg * BK);
  store();
  __syncthreads();
  for (int64_t k0 = 0; k0 < k; k0 += KG * BK) {   // the same stages for every group (zeros past k)
    const bool more = k0 + KG * BK < k;
    if (more) load(k0 + (KG + kg) * BK);
#pragma unroll
    for (int kk = 0; kk < BK; kk++) {
      double a[R], b[R];
#pragma unroll
      for (int i = 0; i < R; i++) a[i] = As[kk][ty + NT * i];
#pragma unroll
      for (int j = 0; j < R; j++) b[j] = Bs[kk][tx + NT * j];
#pragma unroll
      for (int i = 0; i < R; i++)
#pragma unroll
        for (int j = 0; j < R; j++) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
    if (more) {
      store();
      __syncthreads();
    }
  }
  if constexpr (KG > 1) {   // group 0 collects the sums, in group order (operand buffers are free)
    static_assert(THREADS * R * R <= KG * BK * (T + 1), "a group's sums fit the operand buffer");
    double* part = &Asm[0][0][0];
    for (int g = 1; g < KG; g++) {
      if (kg == g)
#pragma unroll
        for (int q = 0; q < R * R; q++) part[q * THREADS + t] = acc[q / R][q % R];
      __syncthreads();
      if (kg == 0)
#pragma unroll
        for (int q = 0; q < R * R; q++) acc[q / R][q % R] += part[q * THREADS + t];
      __syncthreads();
    }
    if (kg > 0) return;
  }
#pragma unroll
  for (int i = 0; i < R; i++) {
    const int64_t r = m0 + ty + NT * i;
    if (r >= m) continue;
    const double rs = rowscale ? rowscale[r] * alpha : alpha;
#pragma unroll
    for (int j = 0; j < R; j++) {
      const int64_t c = n0 + tx + NT * j;
      if (c >= n) continue;
      double v = rs * acc[i][j];
      if (beta != 0.0) v = fma(beta, C[r * ldc + c], v);
      C[r * ldc + c] = v;
    }
  }
}

template <int T, int R, int KG>
void launch_tiles(int64_t m, int64_t n, int64_t k, double alpha, const double* A, int64_t lda, bool a_kcontig,
                  const double* B, int64_t ldb, bool b_kcontig, double beta, double* C, int64_t ldc, bool lower,
                  const double* rowscale, cudaStream_t st) {
  const dim3 grid((unsigned)((n + T - 1) / T), (unsigned)((m + T - 1) / T));
  constexpr int THREADS = KG * (T / R) * (T / R);
  // k <= 0 is valid: the kernel then only applies C = beta C
  if (a_kcontig && b_kcontig)
    dgemm_kernel<T, R, KG, true, true><<<grid, THREADS, 0, st>>>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, lower,
                                                             rowscale);
  else if (a_kcontig && !b_kcontig)
    dgemm_kernel<T, R, KG, true, false><<<grid, THREADS, 0, st>>>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, lower,
                                                              rowscale);
  else if (!a_kcontig && b_kcontig)
    dgemm_kernel<T, R, KG, false, true><<<grid, THREADS, 0, st>>>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, lower,
                                                              rowscale);
  else
    dgemm_kernel<T, R, KG, false, false><<<grid, THREADS, 0, st>>>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, lower,
                                                               rowscale);
  count_launch();
}

}  // namespace

cudaError_t dgemm(int64_t m, int64_t n, int64_t k, double alpha, const double* A, int64_t lda, bool a_kcontig,
                  const double* B, int64_t ldb, bool b_kcontig, double beta, double* C, int64_t ldc, bool lower,
                  const double* rowscale, cudaStream_t st) {
  if (m <= 0 || n <= 0) return cudaSuccess;
  auto tiles = [&](int64_t t) {
    const int64_t gm = (m + t - 1) / t, gn = (n + t - 1) / t;
    return lower ? gm * (gm + 1) / 2 : gm * gn;
  };
  if ((m + 63) / 64 > 65535) return cudaErrorInvalidValue;
  // Tiles: 64 x 64 once they make a dozen per SM (0.97 of the pipe at n = 8514).  Fewer leave SMs
  // idle in the last round, so 32 x 32 down to four tiles per SM, then 16 x 16.  A long K with few
  // tiles per SM exposes the FP64 latency (63 clocks), so the groups of a block split it: 4 or 8
  // groups once each has a few stages.  Symmetric product, one launch, K = 1025, TFLOP/s of the
  // lower half with 64 x 64 tiles only -> with this rule: n = 98 0.009 -> 0.115, n = 482 0.225 ->
  // 0.755, n = 1154 0.437 -> 0.99 (3.13 -> 1.38 ms), n = 3402 1.145 -> 1.12.  At n = 1154 and K = 1025
  // 16 x 16 tiles take 1.39 ms and 32 x 32 without groups 2.10 ms, which sets the two lines; with
  // K = 64 (the factorisation's updates) the groups cost more than they hide.
  const bool longk = k >= 256;
#define GN_DGEMM(T, R, KG) \
  launch_tiles<T, R, KG>(m, n, k, alpha, A, lda, a_kcontig, B, ldb, b_kcontig, beta, C, ldc, lower, rowscale, st)
  if (tiles(64) >= 152 * 12) GN_DGEMM(64, 4, 1);
  else if (tiles(32) >= 152 * 4 && longk) GN_DGEMM(32, 4, 4);
  else if (tiles(32) >= 152 * 4) GN_DGEMM(32, 4, 1);
  else if (longk) GN_DGEMM(16, 2, 8);
  else GN_DGEMM(16, 2, 1);
#undef GN_DGEMM
  return cudaGetLastError();
}

}  // namespace gn
