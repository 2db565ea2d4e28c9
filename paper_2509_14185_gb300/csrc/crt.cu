// The split Gram G = J^T J at six slices (48-bit operands) by residues: the exact integer product
// from 13 BF16 matrix products instead of 21 slice products (Methods, "Second-order Optimizer").
//
// ozaki.cu multiplies the base-256 digits of the 48-bit integers v = round(x 2^(48 - e)) pairwise: 21
// products for six slices, less the levels it drops, the lower levels summed in FP32 over the
// whole contraction.  Here the same integers enter through their residues (Ozaki scheme II: Ozaki,
// Uchino & Imamura, "Ozaki Scheme II: A GEMM-oriented emulation of floating-point matrix
// multiplication using an integer modular technique", 2025): for 13 pairwise coprime moduli p <= 417,
//   1. residues: r_p = v mod p, balanced, |r_p| <= 208: exact in BF16;
//   2. products: C_p = R_p^T R_p on the tensor cores.  384 products of magnitude <= 208^2 sum to less than
//      2^24, so the FP32 accumulation is exact over 384 rows; after each such chunk the epilogue
//      reduces the accumulator modulo p (FP32 operations, exact) and carries it in a register;
//   3. reconstruction: the Chinese remainder theorem gives the exact integer X = sum_k v_ki v_kj from its
//      13 residues (their product M = 2^112.4 exceeds 2 |X| <= 2 K 2^96 for K <= 32768 rows; more rows are
//      several products), and G_ij = X 2^(e_i + e_j - 96) is rounded once.
// The moduli trade the number of products against the chunk: 13 moduli up to 511 need a reduction
// every 256 rows, which takes longer than the products it should hide behind.
// So the only error is that of the 48-bit operands, 2^-49 (|x_i|_1 + |x_j|_1) in units of 2^(e_i + e_j), the first term
// of ozaki.cu's bound.
//
// The product kernel: 256 x 256 outputs per pair of CTAs (cta_group::2, each CTA fetches 128 rows of A
// and of B per 64-wide K stage), two 256-column accumulators so that one chunk's products run while
// the last is reduced, persistent pairs over the (modulus, tile) items.  It wants the full shared-memory
// bandwidth (64 bytes per clock of operand reads, 64 of copies), so its waits suspend instead of polling
// (tc.cuh) and its loops keep to the 512 clocks of a stage.  8514 columns, 16385 rows: 10.6 ms = 1.57 PFLOP/s
// (2501 rows of 4850 columns: tensor pipe 57 % busy); first version 16.9 ms.  Clusters of two pairs
// sharing B by multicast cut the L2 reads by a fifth and took 11.8 ms: they fill only 144 of the 152 SMs.
// Whole Gram, slices -> residues: 16.84 -> 13.35 ms there (0.17 column maxima, 1.14 residues, 10.6 products, 0.46
// reconstruction), 1154 x 4097 0.303 -> 0.211 ms, 322 x 1025 0.110 -> 0.066 ms; error against 64 bits 3e-10 -> 2.6e-15 (the
// slices sum their lower levels in FP32 over all rows).
#include <cuda.h>
#include <cuda_bf16.h>

#include <cmath>
#include <cstdio>
#include <cstring>

#include "gn_internal.cuh"
#include "tc.cuh"

namespace gn {
namespace {

constexpr int NP = 13;                     // moduli
constexpr int kModuli[NP] = {417, 415, 413, 412, 409, 407, 403, 401, 397, 391, 389, 383, 379};
constexpr int CT = 256;                    // output tile
constexpr int KS = 64;                     // contraction per stage (128-byte rows, SWIZZLE_128B)
constexpr int SPC = 6;                     // stages per exact chunk (384 rows)
constexpr int NST = 6;                     // stages in the ring
constexpr int HALF_BYTES = 128 * KS * 2;   // 128 operand rows of one stage: 16 KB
constexpr int STAGE_BYTES = 2 * HALF_BYTES;
constexpr int THREADS = 384;               // warp 0 TMA, warp 1 MMA, warps 4..11 epilogue
constexpr size_t SMEM = (size_t)NST * STAGE_BYTES + 1024 + 256;
constexpr int64_t kMaxRows = 32768;        // |X| <= K 2^96 <= 0.38 M / 2

struct CrtMod {
  float p[NP], inv[NP];
};

// ---- PTX of a CTA pair ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// the address of this CTA's shared variable in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void remote_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tma_pair(void* dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
// K-major operand rows of 128 bytes with the 128-byte swizzle; 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t desc128(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// kind::f16: D = F32, A = B = BF16, both K-major, M = 256, N = 256
constexpr uint32_t kIdesc =
    (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(CT >> 3) << 17) | ((uint32_t)(CT >> 4) << 24);
__device__ __forceinline__ void mma_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(kIdesc), "r"(acc));
}
__device__ __forceinline__ void commit_pair(uint64_t* bar) {   // arrives at this barrier of both CTAs
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  return (uint64_t)__float_as_uint(a) | ((uint64_t)__float_as_uint(b) << 32);
}
constexpr float kRound = 12582912.0f;   // 1.5 2^23: (x + kRound) - kRound rounds |x| < 2^22 to an integer

// lower-triangular tile t, row by row, column by column (the first c mt - c (c - 1) / 2 are the tile
// columns < c), or (order 2) in square super-blocks of kSB: the pairs in flight share few row bands
constexpr int64_t kSB = 9;
__device__ __forceinline__ void tri(int64_t t, int64_t& i, int64_t& j) {
  i = (int64_t)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= t) i++;
  while (i * (i + 1) / 2 > t) i--;
  j = t - i * (i + 1) / 2;
}
__device__ __forceinline__ void crt_tile(int64_t t, int64_t mt, int colmajor, int64_t& ti, int64_t& tj) {
  if (colmajor) {   // the triangle reflected about its anti-diagonal, read backwards
    int64_t a, b;
    tri(mt * (mt + 1) / 2 - 1 - t, a, b);
    ti = mt - 1 - b;
    tj = mt - 1 - a;
    return;
  }
  for (int64_t I = 0;; I++) {   // super-row I: I blocks of hh x kSB tiles, then the diagonal block
    const int64_t hh = mt - I * kSB < kSB ? mt - I * kSB : kSB;
    const int64_t cnt = I * hh * kSB + hh * (hh + 1) / 2;
    if (t < cnt) {
      if (t < I * hh * kSB) {
        const int64_t J = t / (hh * kSB), v = t % (hh * kSB);
        ti = I * kSB + v / kSB;
        tj = J * kSB + v % kSB;
      } else {
        tri(t - I * hh * kSB, ti, tj);
        ti += I * kSB;
        tj += I * kSB;
      }
      return;
    }
    t -= cnt;
  }
}

struct CrtArgs {
  int64_t npad;             // operand rows per modulus
  int nk;                   // stages of the contraction
  int64_t mt, tile0, ntiles;
  int colmajor;
  uint16_t* res;            // [tile][modulus][256][256]: residue + 256
  int* flag;
  unsigned long long wait_ns;
  int starve;               // testing: the producer issues no copy
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    crt_gemm(const __grid_constant__ CUtensorMap tm, const __grid_constant__ CrtMod md, const CrtArgs p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t full[NST], empty[NST], acc_full[2], acc_empty[2], done;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_cta;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cta_rank();
  const int64_t items = p.ntiles * NP, pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  const int nchunk = (p.nk + SPC - 1) / SPC;
  int* flag = p.flag;
  if (threadIdx.x == 0) {
    abort_cta = 0;
    for (int i = 0; i < NST; i++) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int b = 0; b < 2; b++) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 16);   // eight epilogue warps of either CTA
    }
    mbar_init(&done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "n"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();   // the pair's barriers are initialised before either CTA signals the other
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == 0) {
    // ---------------- TMA producer: this CTA's 128 rows of A and of B; bytes counted by the leader's barrier
    if (lane == 0) {
      // The loop of one stage has 512 clocks (four MMAs); counters run instead of being divided out of a
      // stage number, whose 64-bit remainders alone kept the tensor pipe at 0.62.
      int st = 0, issued = 0;
      uint32_t par = 1;   // an unused ring passes its first wait
      bool ok = true;
      const uint32_t full0 = mapa(smem_u32(&full[0]), 0);
      for (int64_t it = pair; it < items && ok && !p.starve; it += pairs) {
        int64_t ti, tj;
        crt_tile(p.tile0 + it % p.ntiles, p.mt, p.colmajor, ti, tj);
        const int base = (int)(it / p.ntiles * p.npad + 128 * rank);
        const int ra = base + (int)(ti * CT), rb = base + (int)(tj * CT);
        for (int kt = 0; kt < p.nk; kt++) {
          if (!mbar_wait(&empty[st], par, flag, p.wait_ns) || *(volatile int*)&abort_cta) {
            ok = false;
            break;
          }
          unsigned char* dst = smem + st * STAGE_BYTES;
          const uint32_t bar = full0 + st * 8;
          if (rank == 0) mbar_expect_tx(&full[st], 2 * STAGE_BYTES);
          tma_pair(dst, &tm, kt * KS, ra, bar);
          tma_pair(dst + HALF_BYTES, &tm, kt * KS, rb, bar);
          if (issued < NST) issued++;
          if (++st == NST) {
            st = 0;
            par ^= 1;
          }
        }
      }
      if (!ok) abort_cta = 1;
      // drain (leader): every copy issued must land before the pair may exit
      if (rank == 0)
        for (; issued > 0; issued--) {   // the last stages, newest first
          if (--st < 0) {
            st = NST - 1;
            par ^= 1;
          }
          if (!mbar_wait(&full[st], par ^ 1, flag, p.wait_ns)) atomicOr(flag, 4);
        }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader CTA only) ----------------
    if (rank == 0 && lane == 0) {
      int st = 0, buf = 0;
      uint32_t par = 0, apar = 1;   // the accumulators' first use passes its wait
      const uint64_t d0 = desc128(smem_u32(smem));
      bool ok = true, any = false;
      for (int64_t it = pair; it < items && ok; it += pairs) {
        int q = 0;
        for (int kt = 0; kt < p.nk; kt++) {
          if ((q == 0 && !mbar_wait(&acc_empty[buf], apar, flag, p.wait_ns)) ||
              !mbar_wait(&full[st], par, flag, p.wait_ns)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t a = d0 + (uint32_t)(st * (STAGE_BYTES >> 4));
#pragma unroll
          for (int kk = 0; kk < KS / 16; kk++)
            mma_pair(tmem + buf * CT, a + kk * 2, a + (HALF_BYTES >> 4) + kk * 2, (q == 0 && kk == 0) ? 0u : 1u);
          any = true;
          commit_pair(&empty[st]);
          if (++st == NST) {
            st = 0;
            par ^= 1;
          }
          if (++q == SPC || kt == p.nk - 1) {
            commit_pair(&acc_full[buf]);
            q = 0;
            buf ^= 1;
            if (buf == 0) apar ^= 1;
          }
        }
      }
      if (!ok) abort_cta = 1;
      if (any) {   // every MMA issued must complete before tensor memory is released
        commit_pair(&done);
        if (!mbar_wait(&done, 0, flag, p.wait_ns)) atomicOr(flag, 4);
      }
    }
  } else if (warp >= 4) {
    // ---------------- epilogue: 8 warps, 128 columns per thread ----------------
    const int quad = warp & 3, half = (warp - 4) >> 2;
    const int row = quad * 32 + lane;
    const uint32_t lbase = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * 128);
    const uint32_t eb[2] = {mapa(smem_u32(&acc_empty[0]), 0), mapa(smem_u32(&acc_empty[1]), 0)};
    int64_t ch = 0;
    bool ok = true;
    for (int64_t it = pair; it < items && ok; it += pairs) {
      const int m = (int)(it / p.ntiles);
      const uint64_t inv = pack2(md.inv[m], md.inv[m]), neg = pack2(-md.p[m], -md.p[m]);
      const uint64_t up = pack2(kRound, kRound), down = pack2(-kRound, -kRound);
      uint64_t s[64];
#pragma unroll
      for (int i = 0; i < 64; i++) s[i] = 0;
      for (int c = 0; c < nchunk; c++, ch++) {
        const int buf = (int)(ch & 1);
        if (!epilogue_all(mbar_wait(&acc_full[buf], (uint32_t)(ch >> 1) & 1, flag, p.wait_ns))) {
          ok = false;
          break;
        }
        tc_fence_after();
        // the next 32 columns load while these are reduced
        uint32_t r[2][32];
        tmem_ld32(lbase + (uint32_t)(buf * CT), r[0]);
#pragma unroll
        for (int b = 0; b < 4; b++) {
          tmem_wait32(r[b & 1]);
          if (b < 3) tmem_ld32(lbase + (uint32_t)(buf * CT + b * 32 + 32), r[(b + 1) & 1]);
#pragma unroll
          for (int i = 0; i < 16; i++) {
            const uint64_t v =
                add2(s[b * 16 + i], (uint64_t)r[b & 1][2 * i] | ((uint64_t)r[b & 1][2 * i + 1] << 32));
            s[b * 16 + i] = fma2(neg, add2(fma2(v, inv, up), down), v);   // v - p round(v / p)
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) remote_arrive(eb[buf]);
      }
      if (!ok) break;
      // residues + 256, 128 columns of one row per thread
      uint16_t* out = p.res + (((it % p.ntiles) * NP + m) * CT + 128 * rank + row) * CT + half * 128;
#pragma unroll
      for (int b = 0; b < 16; b++) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const uint64_t v = s[b * 4 + i];   // float(r) + 1.5 2^23 + 256 holds r + 256 in its low bits
          const uint32_t lo = __float_as_uint(__uint_as_float((uint32_t)v) + (kRound + 256.0f));
          const uint32_t hi = __float_as_uint(__uint_as_float((uint32_t)(v >> 32)) + (kRound + 256.0f));
          w[i] = (lo & 0xffffu) | (hi << 16);
        }
        *reinterpret_cast<uint4*>(out + b * 8) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    if (!ok) abort_cta = 1;
  }
  tc_fence_before();
  __syncthreads();
  // the pair's last commit signals here as well: nothing arrives at this CTA's barriers after it
  if (rank == 1 && threadIdx.x == 0 && !p.starve) mbar_wait(&done, 0, flag, p.wait_ns);
  __syncthreads();
  cluster_sync();   // no CTA leaves while the other may still signal it or use its tensor memory
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(512));
  }
}

// ---- residues of the operand ------------------------------------------------------------------------
// 64 rows x 32 columns of J per block: v = round(x 2^(48 - e)) as d0 + 2^18 d1 + 2^33 d2 (|d0| <= 2^17,
// |d1| <= 2^14, |d2| <= 2^15), the residue of the digits' weighted sum (below 2^24: exact FP32), transposed through shared memory into the
// K-major planes.
struct CrtPrep {
  float p[NP], inv[NP];
  float c[NP][2];           // 2^18, 2^33 mod p, balanced
};
// x 2^(48 - e) to the nearest integer (ties away from zero), 2^e > |x|, on the bits of x
__device__ __forceinline__ long long rint48(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  if (ex > 0) m |= 1ull << 52;
  const int r = 1027 + e - (ex > 0 ? ex : 1);   // >= 5
  // (a non-finite column has e = 0, and r below 5 for its large entries: any digits will do)
  const unsigned long long v = r > 54 ? 0ull : r < 1 ? m : (m + (1ull << (r - 1))) >> r;
  return (b >> 63) ? -(long long)v : (long long)v;
}
constexpr int kPitch = 66;   // 33 words: the column-wise stores hit 32 banks
constexpr size_t kPrepSmem = (size_t)NP * 32 * kPitch * 2;
__global__ void __launch_bounds__(256) crt_residues(const double* __restrict__ X, int64_t ld, int64_t nrows,
                                                    int64_t ncols, const int* __restrict__ e, int64_t npad,
                                                    int64_t kpad, __nv_bfloat16* out,
                                                    const __grid_constant__ CrtPrep md) {
  extern __shared__ uint16_t sl[];   // [NP][32][kPitch]
  const int t = threadIdx.x, jj = t & 31;
  const int64_t k0 = (int64_t)blockIdx.x * 64, j0 = (int64_t)blockIdx.y * 32, j = j0 + jj;
  const int ex = e[j];
#pragma unroll 2
  for (int r = 0; r < 8; r++) {
    const int kk = (t >> 5) + 8 * r;
    const int64_t k = k0 + kk;
    const double x = (k < nrows && j < ncols) ? X[k * ld + j] : 0.0;
    const long long u = rint48(x, ex) + 0x100020000ll;   // digit biases of the low two
    const float d0 = (float)((int)(u & 0x3ffff) - 0x20000), d1 = (float)((int)((u >> 18) & 0x7fff) - 0x4000),
                d2 = (float)(int)(u >> 33);
#pragma unroll
    for (int m = 0; m < NP; m++) {
      const float v = fmaf(d2, md.c[m][1], fmaf(d1, md.c[m][0], d0));
      const float q = fmaf(v, md.inv[m], kRound) - kRound;
      sl[(m * 32 + jj) * kPitch + kk] = (uint16_t)(__float_as_uint(fmaf(-md.p[m], q, v)) >> 16);   // exact in BF16
    }
  }
  __syncthreads();
  for (int idx = t; idx < NP * 32 * 8; idx += 256) {
    const int m = idx / 256, c = (idx >> 3) & 31, seg = idx & 7;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(sl + (m * 32 + c) * kPitch + seg * 8);
    *reinterpret_cast<uint4*>(out + ((int64_t)m * npad + j0 + c) * kpad + k0 + seg * 8) =
        make_uint4(src[0], src[1], src[2], src[3]);
  }
}

// ---- reconstruction -------------------------------------------------------------------------------------
// X = sum_m (u_m - 256) W_m mod M with W_m = 1 mod p_m and 0 mod the others; u_m <= 512 in nine bits, so
// each 32-bit word of W_m accumulates in 64 bits without a carry.  The multiple of M to subtract
// comes from the FP32 sum of (u_m - 256) W_m / M (error ~1e-3; |X / M| <= 0.38).
struct CrtRec {
  uint32_t W[NP][4], M[4];
  uint32_t off[4];          // 256 sum W_m mod 2^128
  float g[NP], goff;        // W_m / M and 256 times their sum
};
__global__ void __launch_bounds__(256, 4) crt_reconstruct(const uint16_t* __restrict__ res, int64_t mt, int64_t tile0,
                                                       int colmajor, const int* __restrict__ e, int64_t n, double* G,
                                                       int64_t ld, int add, const __grid_constant__ CrtRec md) {
  int64_t ti, tj;
  crt_tile(tile0 + blockIdx.x, mt, colmajor, ti, tj);
  const int c0 = (threadIdx.x & 127) * 2;
  const int64_t gj = tj * CT + c0;
  const int ej[2] = {e[gj], e[gj + 1]};
  const uint16_t* src = res + (int64_t)blockIdx.x * NP * CT * CT + c0;
#pragma unroll 1
  for (int rr = 0; rr < 4; rr++) {
    const int r = blockIdx.y * 8 + rr * 2 + (threadIdx.x >> 7);
    const int64_t gi = ti * CT + r;
    if (gi >= n || gj > gi) continue;   // the lower triangle
    uint32_t u[NP];
#pragma unroll
    for (int m = 0; m < NP; m++) u[m] = *reinterpret_cast<const uint32_t*>(src + ((int64_t)m * CT + r) * CT);
    const int ei = e[gi];
#pragma unroll 1   // (one element's words at a time: 64 registers, four blocks per SM)
    for (int h = 0; h < 2; h++) {
      if (gj + h > gi) continue;
      unsigned long long a0 = 0, a1 = 0, a2 = 0, a3 = 0;
      float q = -md.goff;
#pragma unroll
      for (int m = 0; m < NP; m++) {
        const uint32_t v = h ? u[m] >> 16 : u[m] & 0xffffu;
        a0 += (unsigned long long)v * md.W[m][0];
        a1 += (unsigned long long)v * md.W[m][1];
        a2 += (unsigned long long)v * md.W[m][2];
        a3 += (unsigned long long)v * md.W[m][3];
        q = fmaf((float)v, md.g[m], q);
      }
      const long long Q = (long long)rintf(q);
      // 128-bit X = a - off - Q M, as two 64-bit halves
      unsigned __int128 X = (unsigned __int128)a0 + ((unsigned __int128)a1 << 32) + ((unsigned __int128)a2 << 64) +
                            ((unsigned __int128)a3 << 96);
      const unsigned __int128 off = ((unsigned __int128)(((unsigned long long)md.off[3] << 32) | md.off[2]) << 64) |
                                    (((unsigned long long)md.off[1] << 32) | md.off[0]);
      const unsigned __int128 M = ((unsigned __int128)(((unsigned long long)md.M[3] << 32) | md.M[2]) << 64) |
                                  (((unsigned long long)md.M[1] << 32) | md.M[0]);
      X -= off;
      X -= (unsigned __int128)(__int128)Q * M;
      const bool neg = (long long)(unsigned long long)(X >> 64) < 0;
      if (neg) X = -X;
      double v = 0.0;
      const unsigned long long hi = (unsigned long long)(X >> 64), lo = (unsigned long long)X;
      if (hi | lo) {
        const int lz = hi ? __clzll((long long)hi) : 64 + __clzll((long long)lo);
        X <<= lz;
        const unsigned long long top = (unsigned long long)(X >> 64);
        // round to nearest even at bit 11 of the top half; the low half is sticky
        const unsigned long long rem = (top & 0x7ff) | ((unsigned long long)X ? 1ull : 0ull);
        const int ex = 1023 + 127 - lz + ei + ej[h] - 96;
        if (ex > 0 && ex < 2046) {
          unsigned long long b = ((unsigned long long)(ex - 1) << 52) + (top >> 11);
          if (rem > 0x400 || (rem == 0x400 && (b & 1))) b++;
          v = __longlong_as_double((long long)b);
        } else {   // outside the normal range: scale the rounded significand
          v = ldexp((double)(top >> 11) + (rem > 0x400 ? 1.0 : 0.0), ex - 1023 - 52);
        }
        if (neg) v = -v;
      }
      double* dst = G + gi * ld + gj + h;
      *dst = add ? *dst + v : v;
    }
  }
}

int64_t rup(int64_t v, int64_t m) { return (v + m - 1) / m * m; }

struct CrtTables {
  CrtMod mod;
  CrtPrep prep;
  CrtRec rec;
};
const CrtTables& tables() {
  static const CrtTables t = [] {
    CrtTables r;
    memset(&r, 0, sizeof(r));
    unsigned __int128 M = 1, sum = 0;
    for (int m = 0; m < NP; m++) M *= (unsigned)kModuli[m];
    auto words = [](unsigned __int128 v, uint32_t* w) {
      for (int i = 0; i < 4; i++) w[i] = (uint32_t)(v >> (32 * i));
    };
    auto balanced = [](long long v, int p) { return (float)(v > p / 2 ? v - p : v); };
    double gs = 0.0;
    for (int m = 0; m < NP; m++) {
      const int p = kModuli[m];
      const unsigned __int128 q = M / (unsigned)p;
      int inv = 1;
      while ((unsigned)((q % (unsigned)p) * (unsigned)inv % (unsigned)p) != 1u) inv++;
      const unsigned __int128 W = q * (unsigned)inv;
      words(W, r.rec.W[m]);
      sum += W * 256u;
      const double g = (double)inv / p;   // W / M
      r.rec.g[m] = (float)g;
      gs += 256.0 * (double)r.rec.g[m];
      r.mod.p[m] = r.prep.p[m] = (float)p;
      r.mod.inv[m] = r.prep.inv[m] = 1.0f / (float)p;
      for (int i = 0; i < 2; i++) r.prep.c[m][i] = balanced((1ll << (18 + 15 * i)) % p, p);
    }
    words(M, r.rec.M);
    words(sum, r.rec.off);
    r.rec.goff = (float)gs;
    return r;
  }();
  return t;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

}  // namespace

// Sizes of a residue Gram of n columns: how many of nrows rows go into one product (the planes stay
// within what the six slices of ozaki.cu would take, or 6 GB), the tiles whose residues are kept at once, and
// the bytes of all that.  The bytes never fall as nrows grows, so a workspace for the largest row block serves
// the shorter ones.
CrtPlan crt_plan(int64_t n, int64_t nrows) {
  CrtPlan pl;
  pl.npad = rup(n > 0 ? n : 1, CT);
  const int64_t all = rup(nrows > 0 ? nrows : 1, KS);
  int64_t cap = 6 * pl.npad * all * 2;
  if (cap < (int64_t)6 << 30) cap = (int64_t)6 << 30;
  int64_t k = cap / (NP * pl.npad * 2) / KS * KS;
  if (k < KS) k = KS;
  if (k > kMaxRows) k = kMaxRows;
  // the last product takes what is left: products of equal size would need less memory for slightly more rows
  pl.krows = k < all ? k : all;
  const int64_t mt = pl.npad / CT, tiles = mt * (mt + 1) / 2;
  pl.batch = tiles < 8 * 76 ? tiles : 8 * 76;
  pl.planes = rup(NP * pl.npad * pl.krows * 2, 1024);
  pl.res = rup(pl.batch * NP * CT * CT * 2, 1024);
  pl.bytes = (size_t)(pl.planes + pl.res + rup(pl.npad * 4, 1024));
  return pl;
}

// Exponents and residue planes of rows [0, k) of J (k <= pl.krows); part: the scratch of colmax.
int crt_prepare(const CrtPlan& pl, const double* J, int64_t ld, int64_t k, int64_t n, void* ws, double* part,
                cudaStream_t st) {
  int* e = reinterpret_cast<int*>(static_cast<unsigned char*>(ws) + pl.planes + pl.res);
  int rc = oz_column_exponents(J, ld, k, n, pl.npad, e, part, st);
  if (rc) return rc;
  const dim3 g((unsigned)(rup(k, KS) / 64), (unsigned)(pl.npad / 32));
  if (GN_NOTE(cudaFuncSetAttribute(crt_residues, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPrepSmem)) !=
      cudaSuccess)
    return GN_ERR_CUDA;
  crt_residues<<<g, 256, kPrepSmem, st>>>(J, ld, k, n, e, pl.npad, rup(k, KS), static_cast<__nv_bfloat16*>(ws), tables().prep);
  count_launch();
  return GN_NOTE(cudaGetLastError()) == cudaSuccess ? GN_OK : GN_ERR_CUDA;
}

// G's lower tiles [tile0, tile0 + ntiles) (256 x 256; all of them: ntiles < 0) from the planes of k rows, on at
// most max_ctas CTAs (0: the device).
int crt_product(const CrtPlan& pl, int64_t k, int64_t n, void* ws, double* G, int64_t ldg, int add, int64_t tile0,
                int64_t ntiles, int colmajor, int max_ctas, int* flag, cudaStream_t st) {
  static const EncodeTiledFn enc = []() -> EncodeTiledFn {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<EncodeTiledFn>(ptr);
    return nullptr;
  }();
  static const int sms = [] {
    int dev = 0, v = 0;
    const bool ok = cudaGetDevice(&dev) == cudaSuccess &&
                    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 1;
    return ok ? v : 152;
  }();
  if (!enc) {
    set_detail(__FILE__, __LINE__, "cuTensorMapEncodeTiled entry point not found");
    return GN_ERR_UNSUPPORTED;
  }
  const int64_t kpad = rup(k, KS), mt = pl.npad / CT, total = mt * (mt + 1) / 2;
  if (ntiles < 0) ntiles = total - tile0;
  CUtensorMap map;
  memset(&map, 0, sizeof(map));
  cuuint64_t dims[2] = {(cuuint64_t)kpad, (cuuint64_t)(NP * pl.npad)};
  cuuint64_t strides[1] = {(cuuint64_t)(kpad * 2)};
  cuuint32_t box[2] = {KS, 128};
  cuuint32_t estr[2] = {1, 1};
  const CUresult cr = enc(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, ws, dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (cr != CUDA_SUCCESS) {
    char msg[64];
    snprintf(msg, sizeof(msg), "cuTensorMapEncodeTiled returned %d", (int)cr);
    set_detail(__FILE__, __LINE__, msg);
    return GN_ERR_CUDA;
  }
  if (GN_NOTE(cudaFuncSetAttribute(crt_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM)) != cudaSuccess)
    return GN_ERR_CUDA;
  unsigned char* base = static_cast<unsigned char*>(ws);
  CrtArgs a;
  a.npad = pl.npad;
  a.nk = (int)(kpad / KS);
  a.mt = mt;
  a.colmajor = colmajor;
  a.res = reinterpret_cast<uint16_t*>(base + pl.planes);
  a.flag = flag;
  a.wait_ns = g_oz_wait_ns.load(std::memory_order_relaxed);
  a.starve = g_oz_starve.load(std::memory_order_relaxed);
  const int* e = reinterpret_cast<const int*>(base + pl.planes + pl.res);
  int64_t pairs = (max_ctas > 0 && max_ctas < sms ? max_ctas : sms) / 2;
  if (pairs < 1) pairs = 1;
  for (int64_t t = tile0; t < tile0 + ntiles; t += pl.batch) {
    a.tile0 = t;
    a.ntiles = t + pl.batch < tile0 + ntiles ? pl.batch : tile0 + ntiles - t;
    const int64_t used = a.ntiles * NP < pairs ? a.ntiles * NP : pairs;
    crt_gemm<<<(unsigned)(2 * used), THREADS, SMEM, st>>>(map, tables().mod, a);
    count_launch();
    crt_reconstruct<<<dim3((unsigned)a.ntiles, CT / 8), 256, 0, st>>>(a.res, mt, t, colmajor, e, n, G, ldg, add,
                                                                      tables().rec);
    count_launch();
  }
  return GN_NOTE(cudaGetLastError()) == cudaSuccess ? GN_OK : GN_ERR_CUDA;
}

}  // namespace gn
