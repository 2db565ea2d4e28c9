// Layered evaluation of many points: the network's hidden layers as split GEMMs on the tcgen05
// tensor cores, the rest pointwise (Methods, "Solution Modeling", "Training Loss" and
// "Second-order Optimizer": the same rows, Jacobian rows and adjoint as jet.cu).
//
// jet.cu carries one point per warp and spends nearly all its time in the FP64 products of the
// hidden layers (GB300 runs one FP64 warp instruction per 17 clocks and SM).  Here the jets of a
// chunk of points pass through each hidden layer together, as the rows of a (points x components)
// x width product, and only the pointwise work stays FP64:
//
//   lay_inputs    q, beta of the points; the hidden weights cut into slices
//   lay_gemm      forward, per hidden layer j: H_j = tanh jets of Z_j, Z_{j+1} = W_j H_j + b_j
//   lay_last      H_{L-1} and the network outputs NN
//   lay_chain     one thread per point and tangent direction: residuals, the lambda column and the
//                 reverse-pass seeds (chain.cuh, the chain jet.cu evaluates per warp)
//   lay_gemm      reverse, per hidden layer: abar_{j+1} = Hbar_{j+1} through the tanh jets,
//                 Hbar_j = W_j^T abar_{j+1}
//   lay_entries   the Jacobian rows sum_c abar_c[o] h_c[i] (lay_hidden_entries for wide 2D layers); or,
//                 for the gradient, their sums over the points (lay_outer, lay_sums)
//
// Precision of the products: that of an FP64 sum, for every element.  A power of two per contraction index
// (2^c_k, from the weights alone) moves from the weights to the activations, which evens out neurons of
// different scale; then every row of either operand is scaled by a power of two 2^-e and rounded to a 62-bit
// integer, written as 8 balanced base-256 digits, digit q in units of 256^-q (exact in BF16).  The digit pairs of
// the eight leading levels are summed in FP32 accumulators: levels 0 to 5 each in its own, exactly (at most 6 * 64
// products of at most 2^14 units), levels 6 and 7 in one; one more takes S, the sum of the products' magnitudes, from
// BF16 forms of the operands rounded down.  The levels are combined in 64-bit integers and rounded once.
// In units of 2^(e_a + e_w) an element of n terms is off by at most n 7.03 2^-62 for the missing levels (7 pairs of digits
// of at most 2^7 on the first of them, 2^64 * 2^12 below the unit), n 2^-62 for the operands' roundings and 2.8 n 2^-60 for
// the 15 ceil(n / 16) additions of the last accumulator, each off by at most two of its units of 2^-60: less than n 2^-57.7
// together.  The FP64 sum is off by up to n 2^-53 S; so wherever S >= 2^-4.7 2^(e_a + e_w) the element is as good, and
// elsewhere, or with an operand that is not finite, it is summed in FP64 (lay_exact; no element of a Xavier network).
#include <cmath>
#include <cstring>

#include "chain.cuh"
#include "tc.cuh"

namespace gn {
namespace {

constexpr int kLayS = 8;                           // digits per value
constexpr int kLaySl = kLayS + 1;                  // slices of an operand: the digits and the magnitude
constexpr int kLayW = 64;                          // widest hidden layer
constexpr int kLayThreads = 512;
constexpr int kLayASlice = 2 * 128 * 64;           // one slice of the A tile: two 32-wide K stages
constexpr int kLayWSlice = 2 * kLayW * 64;         // one slice of the weights
constexpr int kLayA = kLaySl * kLayASlice;         // 144 KB
constexpr size_t kLaySmem = 1024 + kLayA + kLaySl * kLayWSlice + 1024;
constexpr int kLayBad = 0x3fffffff;                // exponent of a row with a non-finite element
constexpr int kLayZero = -100000;                  // exponent of a row of zeros

struct LayArgs {
  int64_t items;            // points (forward) or points x rows (reverse)
  int nr;                   // rows per point
  int K, N;                 // width of the producing and of the resulting layer
  int nf, cz;               // network fields; components per point in zin
  const double* qb;         // [point][2]: q, beta
  const double* W0;         // first layer (K x d) and its bias, for the analytic Z_1
  const double* b0;
  const double* zin;        // [point][cz][K]: preactivation jets of the producing layer, without its bias
  const double* bias;       // forward: of the producing layer
  double* hout;             // forward: [point][CR][K] activation jets (null: not kept)
  int* hexp;                // forward: [point][CR] exponents of those rows (with hout)
  const double* hin;        // reverse: the same, of the layer the adjoint passes
  const double* seeds;      // reverse from the outputs: [item][nf][CR]
  const double* Wlast;      // [nf][K]
  const double* hbar;       // reverse: [item][CR][K]
  double* abar;             // reverse out: [item][CR][K]
  double* out;              // [item][C][N]
  const unsigned char* wsl; // weight slices, kLaySl x 64 x 64 BF16
  const int* we;            // weight exponents [64]
  const int* wc;            // powers c_k of the contraction's indices [64]
  const double* W;          // the weights themselves: element (output o, index k) at W[o * wso + k * wsk]
  int64_t wso, wsk;
  int* flag;
  unsigned long long wait_ns;
  int starve;               // testing: no product is issued, so the waits run out
};

// tanh jets at one neuron: h[0..C) from the preactivation components z[0..C)
template <int D, int C>
__device__ __forceinline__ void tanh_jet(const double* z, double* h) {
  const double t = tanh(z[0]);
  const double t1 = 1.0 - t * t;
  h[0] = t;
  if constexpr (D == 1) {
    h[1] = t1 * z[1];
    if constexpr (C > 2) {
      const double t2 = -2.0 * t * t1;
      h[2] = t2 * z[1] * z[1] + t1 * z[2];
    }
  } else {
    const double t2 = -2.0 * t * t1;
    const double q = z[1], b = z[2];
    h[1] = t1 * q;
    h[2] = t1 * b;
    const double t2q = t2 * q, t2b = t2 * b;
    h[3] = t2q * q + t1 * z[3];
    h[4] = t2q * b + t1 * z[4];
    h[5] = t2b * b + t1 * z[5];
    if constexpr (C > 6) {
      const double t3 = -2.0 * t1 * t1 - 2.0 * t * t2;
      const double t3qq = t3 * q * q;
      h[6] = t3qq * q + 3.0 * t2q * z[3] + t1 * z[6];
      h[7] = t3qq * b + t2 * (2.0 * q * z[4] + b * z[3]) + t1 * z[7];
      h[8] = t3 * q * b * b + t2 * (2.0 * b * z[4] + q * z[5]) + t1 * z[8];
    }
  }
}

// adjoint of the tanh jets at one neuron: g = Hbar on entry, abar on exit; t = tanh, z[1..CR) the
// preactivation derivatives
template <int D>
__device__ __forceinline__ void tanh_jet_adjoint(double t, const double* z, double* g) {
  const double t1 = 1.0 - t * t, t2 = -2.0 * t * t1;
  if constexpr (D == 1) {
    g[0] = g[0] * t1 + g[1] * t2 * z[1];
    g[1] = g[1] * t1;
  } else {
    const double t3 = -2.0 * t1 * t1 - 2.0 * t * t2;
    const double q = z[1], b = z[2];
    const double g3q = g[3] * q, g4b = g[4] * b, g4q = g[4] * q, g5b = g[5] * b;
    g[0] = g[0] * t1 + t2 * (g[1] * q + g[2] * b + g[3] * z[3] + g[4] * z[4] + g[5] * z[5]) +
           t3 * (g3q * q + g4q * b + g5b * b);
    g[1] = g[1] * t1 + t2 * (2.0 * g3q + g4b);
    g[2] = g[2] * t1 + t2 * (g4q + 2.0 * g5b);
    g[3] *= t1;
    g[4] *= t1;
    g[5] *= t1;
  }
}

// preactivation jets of the first hidden layer: linear in (q, beta)
template <int D, int C>
__device__ __forceinline__ void first_layer(const double* W0, const double* b0, int o, double q, double beta,
                                            double* z) {
#pragma unroll
  for (int c = 1; c < C; c++) z[c] = 0.0;
  if constexpr (D == 1) {
    const double w = W0[o];
    z[0] = fma(w, q, b0[o]);
    z[1] = w;
  } else {
    const double w = W0[2 * o], v = W0[2 * o + 1];
    z[0] = fma(v, beta, fma(w, q, b0[o]));
    z[1] = w;
    z[2] = v;
  }
}

__device__ __forceinline__ unsigned abs_hi(double x) {
  return (unsigned)((unsigned long long)__double_as_longlong(x) >> 32) & 0x7fffffffu;
}
// e with 2^e > |x| 2^c (kLayZero: x = 0, kLayBad: x is not finite); a row's exponent is the largest
__device__ __forceinline__ int exponent_above(double x, int c) {
  const int ex = (int)(abs_hi(x) >> 20);
  int e = ex - 1022 + c;
  if ((unsigned)(ex - 1) >= 0x7feu)   // rare: one branch for the normal numbers
    e = ex ? kLayBad : (unsigned long long)__double_as_longlong(x) << 1 ? 1 - 1022 + c : kLayZero;
  return e;
}
// x 2^(62 - e) to the nearest integer plus the digits' bias (|x| <= 2^e; far above |x|: 0): byte 7 - q is
// then digit q plus 128, |digit 0| <= 64
constexpr unsigned long long kDigitBias = 0x8080808080808080ull;
__device__ __forceinline__ unsigned long long biased_digits(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  if (ex > 0) m |= 1ull << 52;
  const int sh = (ex > 0 ? ex : 1) - 1013 - e;   // <= 9
  unsigned long long v;
  if (sh >= 0) v = sh > 9 ? 0ull : m << sh;
  else v = sh < -54 ? 0ull : (m + (1ull << (-sh - 1))) >> -sh;
  return ((b >> 63) ? 0ull - v : v) + kDigitBias;
}
// digit q of a biased value, times 256^-q, as BF16 bits (at most 8 significant bits: the upper half of its
// FP32 form).  The byte goes to the low end of the significand of 2^(23 - 8 q).
__device__ __forceinline__ unsigned short digit_bf16(unsigned long long u, int q) {
  const int byte = 7 - q;
  const unsigned w = byte < 4 ? (unsigned)u : (unsigned)(u >> 32), base = 0x4B000000u - ((unsigned)q << 26);
  const float f = __uint_as_float(__byte_perm(w, base, 0x7640 + (byte & 3))) - __uint_as_float(base | 128u);
  return (unsigned short)(__float_as_uint(f) >> 16);
}
// |x| 2^-e < 1 as BF16 bits, rounded down (0 below 2^-126)
__device__ __forceinline__ unsigned short magnitude_bf16(double x, int e) {
  const unsigned h = abs_hi(x);
  const int ex = (int)(h >> 20) - 896 - e;
  return ex > 0 && ex < 128 ? (unsigned short)(ex << 7 | (h >> 13 & 0x7f)) : (unsigned short)0;
}
constexpr int kNoDigits = 5000;   // an exponent far above every value: all slices zero
// byte offset of element (row, k) in a K-major operand tile with the 64-byte swizzle, `rows` rows
__device__ __forceinline__ int swz(int row, int k, int rows) {
  return (k >> 5) * rows * 64 + row * 64 + ((((k & 31) >> 3) ^ ((row >> 1) & 3)) << 4) + (k & 7) * 2;
}

__device__ __noinline__ double scaled_int_edge(long long T, int k) { return ldexp((double)T, k); }
// T 2^k rounded to nearest even, by integer operations (an I2F and a multiply would take two slots of the FP64
// pipe per element); FP64 where the result leaves the normal range
__device__ __forceinline__ double scaled_int(long long T, int k) {
  if (T == 0) return 0.0;
  const unsigned long long m = T < 0 ? (unsigned long long)-T : (unsigned long long)T;
  const int lz = __clzll((long long)m);
  const int e = 1023 + 63 - lz + k;
  if (e <= 0 || e >= 2046) return scaled_int_edge(T, k);   // (a call: as a predicated instruction it costs its slot)
  const unsigned long long n = m << lz;                       // leading one at bit 63
  const unsigned long long rem = n & 0x7ff;
  unsigned long long r = ((unsigned long long)(e - 1) << 52) + (n >> 11);   // the leading one carries into e
  if (rem > 0x400 || (rem == 0x400 && (r & 1))) r++;
  return __longlong_as_double((long long)(r | ((unsigned long long)T & 0x8000000000000000ull)));
}

// ---- inputs and weight slices --------------------------------------------------------------------
struct LayPrep {
  const double* y;
  int64_t ystride, pt0, npt;
  double lam;
  const double* lamp;
  double* qb;
  const double* theta;
  NetDesc net;
  unsigned char* wsl;       // [(layer - 1) * 2 + direction][kLaySl][64][64] BF16
  int* we;                  // [...][64]
  int* wc;                  // [...][64]
  int pt_blocks;
};
template <int D>
__global__ void __launch_bounds__(256) lay_inputs(const LayPrep p) {
  if ((int)blockIdx.x < p.pt_blocks) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= p.npt) return;
    const double lam = p.lamp ? *p.lamp : p.lam;
    double u = 1.0, y1 = 0.0;
#pragma unroll
    for (int k = 0; k < D; k++) {
      const double v = p.y[(int64_t)k * p.ystride + p.pt0 + i];
      u = fma(v, v, u);
      if (k == 1) y1 = v;
    }
    const Dl a = {1.0 / (1.0 + lam), 0.0};
    p.qb[2 * i] = pow_cb(u, -0.5 * a).v;
    p.qb[2 * i + 1] = D == 2 ? y1 / sqrt(u) : 0.0;
    return;
  }
  // weights, one warp per operand row, 8 rows per block.  Forward operand of layer l: row o is
  // W_l[o][.]; reverse: row i is W_l[.][i].
  const int t = threadIdx.x, wb = (int)blockIdx.x - p.pt_blocks, lane = t & 31;
  const int op = wb / (kLayW / 8), row = wb % (kLayW / 8) * 8 + (t >> 5), l = 1 + op / 2, rev = op & 1;
  const int in = p.net.w[l], out = p.net.w[l + 1];
  const int nrow = rev ? in : out, nk = rev ? out : in;
  const double* W = p.theta + p.net.offW[l];
  auto weight = [&](int r, int k) {
    const int o = rev ? k : r, i = rev ? r : k;
    return (r < nrow && k < nk) ? W[(int64_t)o * in + i] : 0.0;
  };
  // The contraction index k's power c_k: the mean exponent of its weights.  Weights 2^16 and more below
  // the largest count as 2^-16 of it, so that zeros and outliers hardly move it; a column times a
  // power of two moves by exactly that.
  __shared__ int top[4][kLayW], sum[4][kLayW], cnt[4][kLayW], cs[kLayW];
  {
    const int k = t & 63, g = t >> 6;
    int ex[kLayW / 4], m = kLayZero;
#pragma unroll
    for (int q = 0; q < kLayW / 4; q++) {
      const int r = g + 4 * q;
      const int e = exponent_above(weight(r, k), 0);
      ex[q] = r >= nrow || e == kLayBad ? kLayBad : e;   // (not counted)
      if (ex[q] != kLayBad) m = ex[q] > m ? ex[q] : m;
    }
    top[g][k] = m;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; q++) m = top[q][k] > m ? top[q][k] : m;
    int s = 0, n = 0;
#pragma unroll
    for (int q = 0; q < kLayW / 4; q++)
      if (ex[q] != kLayBad) {
        s += ex[q] > m - 16 ? ex[q] : m - 16;
        n++;
      }
    sum[g][k] = s;
    cnt[g][k] = n;
    __syncthreads();
    if (t < kLayW) {
      s = sum[0][k] + sum[1][k] + sum[2][k] + sum[3][k];
      n = cnt[0][k] + cnt[1][k] + cnt[2][k] + cnt[3][k];
      cs[k] = m == kLayZero ? 0 : (int)floorf((float)s / (float)n + 0.5f);
      if (row == t >> 5) p.wc[op * kLayW + k] = cs[k];   // (the first of the operand's blocks)
    }
    __syncthreads();
  }
  double x[2];
  int e = kLayZero;
#pragma unroll
  for (int q = 0; q < 2; q++) {
    const int k = lane + 32 * q;
    x[q] = weight(row, k);
    const int ek = exponent_above(x[q], -cs[k]);
    e = ek > e ? ek : e;
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if (lane == 0) p.we[op * kLayW + row] = e;
  unsigned short* dst = reinterpret_cast<unsigned short*>(p.wsl) + (size_t)op * kLaySl * kLayW * kLayW + row * kLayW;
#pragma unroll
  for (int q = 0; q < 2; q++) {
    const int k = lane + 32 * q, ek = e == kLayBad || e == kLayZero ? kNoDigits : e + cs[k];
    const unsigned long long u = biased_digits(x[q], ek);
#pragma unroll
    for (int s = 0; s < kLayS; s++) dst[s * kLayW * kLayW + k] = digit_bf16(u, s);
    dst[kLayS * kLayW * kLayW + k] = magnitude_bf16(x[q], ek);
  }
}

// ---- one hidden layer ------------------------------------------------------------------------------
enum LayKind : int { LAY_FWD_FIRST = 0, LAY_FWD = 1, LAY_REV_LAST = 2, LAY_REV = 3 };

// the operand's elements at index k of an item: FP64 jets through tanh, or the adjoint through them
template <int D, int C, int KIND>
__device__ __forceinline__ void lay_operand(const LayArgs& p, int64_t item, int64_t pt, int k, double q, double beta,
                                            double* x) {
  constexpr int CR = JT<D>::CR;
  if constexpr (KIND <= LAY_FWD) {
    double z[C];
    if (KIND == LAY_FWD_FIRST) {
      first_layer<D, C>(p.W0, p.b0, k, q, beta, z);
    } else {
#pragma unroll
      for (int c = 0; c < C; c++) z[c] = p.zin[(pt * C + c) * p.K + k];
      z[0] += p.bias[k];
    }
    tanh_jet<D, C>(z, x);
  } else {
    if (KIND == LAY_REV_LAST) {
      for (int f = 0; f < p.nf; f++) {
        const double w = p.Wlast[f * p.K + k];
#pragma unroll
        for (int c = 0; c < C; c++) x[c] = fma(w, p.seeds[(item * p.nf + f) * CR + c], x[c]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < C; c++) x[c] = p.hbar[(item * C + c) * p.K + k];
    }
    double z[CR];
#pragma unroll
    for (int c = 1; c < CR; c++) z[c] = p.zin[(pt * p.cz + c) * p.K + k];
    tanh_jet_adjoint<D>(p.hin[pt * CR * p.K + k], z, x);
  }
}

// One element (a whole warp: component c of an item, output col) as an FP64 sum.  The operand is computed
// again where it is not kept (forward).
template <int D, int C, int KIND>
__device__ __noinline__ double lay_exact(const LayArgs& p, int col, int64_t item, int c) {
  const int lane = threadIdx.x & 31;
  const int64_t pt = KIND <= LAY_FWD ? item : item / p.nr;
  double sum = 0.0;
#pragma unroll 1
  for (int k = lane; k < p.K; k += 32) {
    double a;
    if constexpr (KIND <= LAY_FWD) {
      double x[C];
      const bool first = KIND == LAY_FWD_FIRST;
      lay_operand<D, C, KIND>(p, item, pt, k, first ? p.qb[2 * pt] : 0.0, first ? p.qb[2 * pt + 1] : 0.0, x);
      a = x[0];
#pragma unroll
      for (int i = 1; i < C; i++) a = i == c ? x[i] : a;
    } else {
      a = p.abar[(item * C + c) * p.K + k];   // (stored by this block before its last barrier)
    }
    sum = fma(a, p.W[col * p.wso + k * p.wsk], sum);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return sum;
}

// One CTA per SM, persistent over tiles of 128 rows (128 / C items of C components).  Its 16 warps
// first produce the tile's A operand, one item per warp: FP64 jets through tanh (or its adjoint),
// the rows' exponents, their slices into shared memory in the layout the MMA reads.  One thread
// then issues the 36 digit-pair products and that of the magnitudes into eight tensor-memory accumulators of
// 64 columns, and all warps combine the levels and store the layer's FP64 result.  The three phases follow one
// another: the tile fills the shared memory (144 KB of A beside 72 KB of weights) and the tensor memory.
template <int D, int C, int KIND>
__global__ void __launch_bounds__(kLayThreads, 1) lay_gemm(const __grid_constant__ LayArgs p) {
  constexpr int CR = JT<D>::CR;
  constexpr int IPT = 128 / C;               // items per tile
  constexpr bool kFwd = KIND <= LAY_FWD;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* As =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* Ws = As + kLayA;
  __shared__ uint64_t done;
  __shared__ uint32_t tmem_slot;
  __shared__ int eA[128], eW[kLayW];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int ks_n = (p.K + 31) >> 5;
  for (int idx = t; idx < kLaySl * kLayW * 8; idx += kLayThreads) {   // 16-byte chunks
    const int s = idx / (kLayW * 8), row = (idx >> 3) % kLayW, c8 = idx & 7;
    *reinterpret_cast<uint4*>(Ws + s * kLayWSlice + swz(row, c8 * 8, kLayW)) =
        *reinterpret_cast<const uint4*>(p.wsl + (size_t)idx * 16);
  }
  if (t < kLayW) eW[t] = p.we[t];
  const int ck[2] = {p.wc[lane], p.wc[lane + 32]};
  if (t == 0) {
    mbar_init(&done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "n"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int64_t tiles = (p.items + IPT - 1) / IPT;
  uint32_t phase = 0;
  bool ok = true;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int64_t i0 = tile * IPT;
    const int ni = (int)(p.items - i0 < IPT ? p.items - i0 : IPT);
    // ---- A operand ---------------------------------------------------------------------------------
    for (int it = warp; it < ni; it += kLayThreads / 32) {
      const int64_t item = i0 + it;
      const int64_t pt = kFwd ? item : item / p.nr;
      double x[2][C];
      int m[C];
#pragma unroll
      for (int c = 0; c < C; c++) m[c] = kLayZero;
      double q = 0.0, beta = 0.0;
      if (KIND == LAY_FWD_FIRST) {
        q = p.qb[2 * pt];
        beta = p.qb[2 * pt + 1];
      }
#pragma unroll
      for (int s = 0; s < 2; s++) {
        const int k = lane + 32 * s;
#pragma unroll
        for (int c = 0; c < C; c++) x[s][c] = 0.0;
        if (k >= p.K) continue;
        lay_operand<D, C, KIND>(p, item, pt, k, q, beta, x[s]);
        if constexpr (kFwd) {
          if (p.hout) {
#pragma unroll
            for (int c = 0; c < CR; c++) p.hout[(pt * CR + c) * p.K + k] = x[s][c];
          }
        } else {
#pragma unroll
          for (int c = 0; c < C; c++) p.abar[(item * C + c) * p.K + k] = x[s][c];
        }
#pragma unroll
        for (int c = 0; c < C; c++) {
          const int e = exponent_above(x[s][c], ck[s]);
          m[c] = e > m[c] ? e : m[c];
        }
      }
#pragma unroll
      for (int c = 0; c < C; c++) {
        const int row = it * C + c;
        const int e = __reduce_max_sync(0xffffffffu, m[c]);
        if (lane == 0) {
          eA[row] = e;
          if (kFwd && c < CR && p.hexp) p.hexp[pt * CR + c] = e == kLayZero ? 0 : e;
        }
#pragma unroll
        for (int s = 0; s < 2; s++) {
          if (s < ks_n) {
            const int ek = e == kLayBad || e == kLayZero ? kNoDigits : e - ck[s];
            const unsigned long long u = biased_digits(x[s][c], ek);
            unsigned char* dst = As + swz(row, lane + 32 * s, 128);
#pragma unroll
            for (int d = 0; d < kLayS; d++)
              *reinterpret_cast<unsigned short*>(dst + d * kLayASlice) = digit_bf16(u, d);
            *reinterpret_cast<unsigned short*>(dst + kLayS * kLayASlice) = magnitude_bf16(x[s][c], ek);
          }
        }
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMA reads what the threads wrote
    tc_fence_before();
    __syncthreads();
    // ---- products ----------------------------------------------------------------------------------
    if (t == 0 && !p.starve) {
      tc_fence_after();
      // (four MMAs take about 128 clocks: one thread must not spend them on descriptors)
      const uint64_t a0 = smem_desc(smem_u32(As)), w0 = smem_desc(smem_u32(Ws));
      auto product = [&](int slot, int sa, int sw, uint32_t acc) {
        const uint64_t a = a0 + (uint32_t)(sa * (kLayASlice >> 4)), w = w0 + (uint32_t)(sw * (kLayWSlice >> 4));
        const uint32_t d = tmem + slot * kLayW;
        mma_bf16<kLayW>(d, a, w, acc);
        mma_bf16<kLayW>(d, a + 2, w + 2, 1);
        if (ks_n > 1) {
          mma_bf16<kLayW>(d, a + (128 * 64 >> 4), w + (kLayW * 64 >> 4), 1);
          mma_bf16<kLayW>(d, a + (128 * 64 >> 4) + 2, w + (kLayW * 64 >> 4) + 2, 1);
        }
      };
      product(7, kLayS, kLayS, 0);
#pragma unroll 1
      for (int level = kLayS - 1; level >= 0; level--)   // level 7 goes below level 6
#pragma unroll 1
        for (int s = 0; s <= level; s++)
          product(level < 6 ? level : 6, s, level - s, (s == 0 && level != 6) ? 0u : 1u);
      mma_commit(&done);
    }
    // (read here: behind the next barrier the producers of the next tile overwrite the exponents)
    const int row = (warp & 3) * 32 + lane, ea = eA[row];
    ok = __syncthreads_and(mbar_wait(&done, phase, p.flag, p.wait_ns));
    phase ^= 1;
    if (!ok) {   // the host sees the status bit; this CTA's remaining rows become NaN
      for (; tile < tiles; tile += gridDim.x)
        for (int64_t i = tile * IPT * C * p.N + t; i < (tile + 1) * IPT * C * p.N && i < p.items * C * p.N;
             i += kLayThreads)
          p.out[i] = nan("");
      mbar_wait(&done, phase ^ 1, p.flag, p.wait_ns);   // products in flight use the tensor memory to be released
      break;
    }
    tc_fence_after();
    // ---- levels to FP64 ------------------------------------------------------------------------------
    {
      const int cg = warp >> 2;   // 16 columns per warp
      const bool valid = row < ni * C;
      const int64_t orow = i0 * C + row;
#pragma unroll
      for (int part = 0; part < 2; part++) {
        const int col0 = cg * 16 + part * 8;
        if (col0 >= p.N) continue;   // the same for the whole warp
        uint32_t r[kLayS][8];
#pragma unroll
        for (int s = 0; s < kLayS; s++)
          tmem_ld8_async(tmem + ((uint32_t)((warp & 3) * 32) << 16) + s * kLayW + col0, r[s]);
        tmem_wait_ld();
#pragma unroll
        for (int s = 0; s < kLayS; s++) tmem_use8(r[s]);
        unsigned weak = 0;   // columns whose products are too small for their digits
#pragma unroll
        for (int j = 0; j < 8; j++) {
          int v[7];   // accumulator s is v_s 256^-s
#pragma unroll
          for (int s = 0; s < 7; s++)
            v[s] = __float2int_rn(__uint_as_float(r[s][j]) * __uint_as_float(0x3f800000u + ((unsigned)s << 26)));
          // sum_s v_s 256^(6 - s) = hi 2^24 + low, 0 <= low < 2^24, |hi| < 2^43; four bits of low go where hi is large
          const long long lo = (long long)v[4] * 65536 + (v[5] * 256 + v[6]);
          const long long hi = (long long)v[0] * 16777216 + (long long)v[1] * 65536 + (v[2] * 256 + v[3]) + (lo >> 24);
          const unsigned low = (unsigned)lo & 0xffffffu;
          const bool large = (unsigned long long)(hi + (1ll << 39)) >> 40;
          const long long T = large ? hi * (1 << 20) + (low >> 4) : hi * (1 << 24) + low;
          const int ew = eW[col0 + j];
          const bool bad = ea == kLayBad || ew == kLayBad, zero = ea == kLayZero || ew == kLayZero;
          const float S = __uint_as_float(r[7][j]);   // never above the true one
          if (valid && col0 + j < p.N) {
            p.out[orow * p.N + col0 + j] = zero ? 0.0 : scaled_int(T, ea + ew - (large ? 56 : 60));
            if (bad || !(zero || S >= 0.04f)) weak |= 1u << j;   // 2^-4.64
          }
        }
        if (__any_sync(0xffffffffu, weak)) {
#pragma unroll 1
          for (int j = 0; j < 8; j++)
            for (unsigned b = __ballot_sync(0xffffffffu, weak >> j & 1); b; b &= b - 1) {
              const int src = __ffs(b) - 1, rs = (warp & 3) * 32 + src;
              const double v = lay_exact<D, C, KIND>(p, col0 + j, i0 + rs / C, rs % C);
              if (lane == src) p.out[orow * p.N + col0 + j] = v;
            }
        }
      }
    }
    tc_fence_before();   // the next tile's MMAs overwrite the accumulators after its barrier
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(512));
  }
}

// ---- last hidden layer and the outputs --------------------------------------------------------------
// One warp per point; the NF * C sums over the width are reduced by halving: after step o every
// lane holds half as many partial sums, so NF * C sums cost about that many additions, not five
// times as many.
template <int D, int C, int NF>
__global__ void __launch_bounds__(256) lay_last(int64_t npt, int K, const double* __restrict__ zin,
                                                const double* __restrict__ bias, double* hout,
                                                const double* __restrict__ W, const double* __restrict__ b,
                                                double* nn) {
  constexpr int CR = JT<D>::CR, V = NF * C;
  constexpr int VP = V <= 2 ? 2 : V <= 4 ? 4 : V <= 8 ? 8 : V <= 16 ? 16 : 32;
  const int lane = threadIdx.x & 31;
  const int64_t pt = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (pt >= npt) return;
  double v[VP];
#pragma unroll
  for (int i = 0; i < VP; i++) v[i] = 0.0;
#pragma unroll
  for (int s = 0; s < 2; s++) {
    const int k = lane + 32 * s;
    if (k >= K) continue;
    double z[C], h[C];
#pragma unroll
    for (int c = 0; c < C; c++) z[c] = zin[(pt * C + c) * K + k];
    z[0] += bias[k];
    tanh_jet<D, C>(z, h);
    if (hout) {
#pragma unroll
      for (int c = 0; c < CR; c++) hout[(pt * CR + c) * K + k] = h[c];
    }
#pragma unroll
    for (int f = 0; f < NF; f++) {
      const double w = W[f * K + k];
#pragma unroll
      for (int c = 0; c < C; c++) v[f * C + c] = fma(w, h[c], v[f * C + c]);
    }
  }
  int o = 16, idx = 0;
#pragma unroll
  for (int n = VP; n > 1; n >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < n / 2; i++) {
      const double send = up ? v[i] : v[i + n / 2], keep = up ? v[i + n / 2] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
    if (up) idx += n / 2;
    o >>= 1;
  }
  for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  constexpr int kDup = 32 / VP;   // lanes that hold the same sum
  if (idx < V && lane % kDup == 0) nn[pt * V + idx] = v[0] + (idx % C == 0 ? b[idx / C] : 0.0);
}

// ---- residual chain ------------------------------------------------------------------------------------
// One thread per (point, tangent direction): 32 points per warp, the directions over the block's
// warps (direction 0: lambda; 1 + f C_R + c: output f, component c).  jet.cu evaluates the same
// chain once per warp and point, its lanes being the directions, 19 of 32 at most.
struct LayChain {
  int64_t npt, p0;          // points of this chunk, the first one's index
  const double* nn;         // [point][NF * CF]
  double* seeds;            // [point][rows][NF * CR]
  double* lamg;             // gradient mode: d / d lambda per point
};
template <int EQ, int MODE>
__global__ void __launch_bounds__(MODE == MODE_RESIDUAL ? 128 : 32 * (1 + Eq<EQ>::NF * JT<Eq<EQ>::D>::CR))
    lay_chain(const JetArgs A, const LayChain L) {
  constexpr int D = Eq<EQ>::D, NF = Eq<EQ>::NF, NE = Eq<EQ>::NE, CR = JT<D>::CR;
  constexpr int CF = (MODE == MODE_RESIDUAL) ? CR : JT<D>::CF;
  const int dir = MODE == MODE_RESIDUAL ? 0 : threadIdx.y;
  const int64_t pl = (MODE == MODE_RESIDUAL ? (int64_t)blockIdx.x * blockDim.y + threadIdx.y : blockIdx.x) * 32 +
                     threadIdx.x;
  if (pl >= L.npt) return;
  const int64_t pt = L.p0 + pl;
  const double lam = A.lamp ? *A.lamp : A.lam;
  double y[D];
  double u = 1.0;
#pragma unroll
  for (int k = 0; k < D; k++) y[k] = A.y[(int64_t)k * A.ystride + pt];
#pragma unroll
  for (int k = 0; k < D; k++) u = fma(y[k], y[k], u);
  const bool tl = dir == 0 && MODE != MODE_RESIDUAL;
  const Dl a = {1.0 / (1.0 + lam), tl ? -1.0 / ((1.0 + lam) * (1.0 + lam)) : 0.0};
  const Dl q = pow_cb(u, -0.5 * a);
  double beta = 0.0;
  if (D == 2) beta = y[1] / sqrt(u);
  const double* NN = L.nn + pl * (NF * CF);
  Dl nn[NF][CR];
#pragma unroll
  for (int f = 0; f < NF; f++)
#pragma unroll
    for (int c = 0; c < CR; c++) {
      double dv = 0.0;
      if (MODE != MODE_RESIDUAL) {
        if (dir == 0) dv = NN[f * CF + q_shift<D>(c)] * q.d;
        else if (dir == 1 + f * CR + c) dv = 1.0;
      }
      nn[f][c] = {NN[f * CF + c], dv};
    }
  const Dl lamd = {lam, tl ? 1.0 : 0.0};
  YJ<D> F[NF];
  field_jets<EQ>(y, u, a, q, lamd, beta, nn, F);
  Dl R[NE];
  double sUv;
  const int kind = A.kind;
  residual_rows<EQ>(A, kind, pt, y, u, a, lamd, nn, F, R, sUv);
  const int nrow = kind == KIND_INTERIOR ? NE : 1;
  double w = A.wscale;
  if (kind == KIND_INTERIOR && A.rho) w *= sqrt(A.rho[pt]);
  const int64_t rbase = A.row0 + pt * nrow;
  const bool su = EQ == GN_CCF && kind == KIND_INTERIOR && A.sU;
  if (dir == 0) {
#pragma unroll
    for (int e = 0; e < NE; e++) {
      if (e >= nrow) break;
      const double rv = w * R[e].v;
      if (A.r) A.r[rbase + e] = rv;
      if (!isfinite(rv)) atomicOr(A.flag, 1);
    }
    if (su && MODE != MODE_GRADIENT) A.sU[pt] = w * sUv;
  }
  if (MODE == MODE_RESIDUAL) return;
  if (MODE == MODE_JACOBIAN) {
#pragma unroll
    for (int e = 0; e < NE; e++) {
      if (e >= nrow) break;
      const double sd = w * R[e].d;
      if (dir > 0) {
        L.seeds[(pl * nrow + e) * (NF * CR) + dir - 1] = sd;
      } else {
        const int64_t row = rbase + e;
        if (row >= A.jrow_lo && row < A.jrow_hi)
          A.J[(row - A.jrow_lo) * A.ldJ + A.net.P] = A.lam_frozen ? 0.0 : sd;
      }
    }
  } else {
    double sd = 0.0;
#pragma unroll
    for (int e = 0; e < NE; e++) {
      if (e >= nrow) break;
      const double comb = A.seed ? A.seed[rbase + e] : w * R[e].v;
      if (e == 0 && dir == 0 && su) A.sU[pt] = comb * w * sUv;
      sd += comb * w * R[e].d;
    }
    if (dir > 0) L.seeds[pl * (NF * CR) + dir - 1] = sd;
    else L.lamg[pl] = A.lam_frozen ? 0.0 : sd;
  }
}

// ---- the first hidden layer's adjoint (no product follows it) -------------------------------------------
template <int D>
__global__ void __launch_bounds__(256) lay_first_adjoint(const LayArgs p) {
  constexpr int CR = JT<D>::CR;
  const int64_t n = p.items * p.K;
  for (int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x; idx < n; idx += (int64_t)gridDim.x * 256) {
    const int64_t item = idx / p.K;
    const int k = (int)(idx - item * p.K);
    double g[CR], z[CR];
#pragma unroll
    for (int c = 0; c < CR; c++) {
      g[c] = p.hbar[(item * CR + c) * p.K + k];
      z[c] = 0.0;
    }
    z[1] = p.W0[k * D];
    if constexpr (D == 2) z[2] = p.W0[k * D + 1];
    tanh_jet_adjoint<D>(p.hin[(item / p.nr) * CR * p.K + k], z, g);
#pragma unroll
    for (int c = 0; c < CR; c++) p.abar[(item * CR + c) * p.K + k] = g[c];
  }
}

// ---- Jacobian rows -------------------------------------------------------------------------------------
struct LayEntries {
  NetDesc net;
  int64_t npt, p0, row0, ldJ, jlo, jhi;
  int nr;
  const double* qb;
  const double* H[GN_MAX_LAYERS + 1];      // [point][CR][w_j], j = 1 .. L - 1
  const double* Ab[GN_MAX_LAYERS + 1];     // [item][CR][w_j]
  const int* He[GN_MAX_LAYERS + 1];        // [point][CR] exponents of H's rows, j = 1 .. L - 2
  const double* seeds;                     // [item][NF][CR]
  double* J;
  int hidden;                              // 0: the hidden-to-hidden weights are lay_hidden_entries'
  int* flag;
  unsigned long long wait_ns;
  int starve;
};
// One warp per (point, layer): the layer's activation jets stay in registers (two neurons per
// lane) for all rows of the point, the adjoints are read at one address per warp, consecutive lanes
// store consecutive columns.  FP64-bound: C_R multiply-adds per entry.
template <int D>
__global__ void __launch_bounds__(256) lay_entries(const LayEntries p) {
  constexpr int CR = JT<D>::CR;
  const int L = p.net.L, lane = threadIdx.x & 31;
  const int64_t w = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int64_t pl = w / L;
  const int l = (int)(w - pl * L);
  if (pl >= p.npt) return;
  const int in = p.net.w[l], out = p.net.w[l + 1];
  double h[2][CR];
#pragma unroll
  for (int s = 0; s < 2; s++)
#pragma unroll
    for (int c = 0; c < CR; c++) {
      const int k = lane + 32 * s;
      h[s][c] = (l > 0 && k < in) ? p.H[l][(pl * CR + c) * in + k] : 0.0;
    }
  for (int e = 0; e < p.nr; e++) {
    const int64_t row = p.row0 + (p.p0 + pl) * p.nr + e;
    if (row < p.jlo || row >= p.jhi) continue;
    double* Jw = p.J + (row - p.jlo) * p.ldJ + p.net.offW[l];
    double* Jb = p.J + (row - p.jlo) * p.ldJ + p.net.offB[l];
    const int64_t item = pl * p.nr + e;
    // adjoint component c of output o: ab[c * cs + o * os]
    const double* ab = l < L - 1 ? p.Ab[l + 1] + item * CR * out : p.seeds + item * out * CR;
    const int cs = l < L - 1 ? out : 1, os = l < L - 1 ? 1 : CR;
    if (l == 0) {
      const double q = p.qb[2 * pl], beta = p.qb[2 * pl + 1];
      for (int o = lane; o < out; o += 32) {
        const double a0 = ab[o];
        Jw[o * D] = fma(a0, q, ab[out + o]);
        if constexpr (D == 2) Jw[o * D + 1] = fma(a0, beta, ab[2 * out + o]);
      }
    } else if (l == L - 1 || p.hidden) {
#pragma unroll 4
      for (int o = 0; o < out; o++) {
        double v0 = 0.0, v1 = 0.0;
#pragma unroll
        for (int c = 0; c < CR; c++) {
          const double a = __ldg(ab + c * cs + o * os);
          v0 = fma(a, h[0][c], v0);
          if (in > 32) v1 = fma(a, h[1][c], v1);
        }
        if (lane < in) Jw[(int64_t)o * in + lane] = v0;
        if (lane + 32 < in) Jw[(int64_t)o * in + lane + 32] = v1;
      }
    }
    for (int o = lane; o < out; o += 32) Jb[o] = ab[o * os];
  }
}

// Hidden-to-hidden weights of 2D rows as products: sum_c abar_c[o] h_c[i] over the six components is a
// (rows x out) x 6 x in contraction per point and layer, whose FP64 form (lay_entries) bounds the 2D
// Jacobian.  One CTA per SM, persistent over (point, layer, pair of rows): 128 x 64 outputs, K = 6 of 16.
// A component's scale moves between the factors by powers of two (h_c is taken relative to its own
// row's exponent 2^eh_c, abar_c times that); then every output row and column has one exponent over
// its six terms.  62-bit integers in eight digits and the 36 digit pairs of the eight leading levels, as in
// lay_gemm; what is dropped is at most 6 * 2^-58.99 2^(e_a + e_b) and the last level's rounding 2^-61 of that unit, which is
// within the 6 * 2^-53 S of the FP64 sum wherever S >= 2^-5.9 2^(e_a + e_b), S the sum of the six products'
// magnitudes.  S comes from FP32 forms of the operands; an entry below that line (Xavier weights, 4 x 64:
// 0.05 to 0.4 % of them), or with a factor that is not finite, is summed in FP64.  (Its operands stay in shared
// memory for that: a warp in sixteen has such an entry, and all wait for the slowest.)
// Bound by the digits and the 64-bit recombination (integer pipes) and by J's stores.
// Jacobian of 8192 IPM points, three hidden layers of 64, FP64 form -> products: 2.67 -> 2.27 ms; 32,768 rows of four
// layers take 5.73 ms.  Digits dealt over all threads and stores of the unit before beside the products were 2 % slower.
constexpr int kEntS = 8;
constexpr int kEntASlice = 128 * 64, kEntBSlice = 64 * 64;   // K padded to 32: the layout of lay_gemm
constexpr int kEntOps = kEntS * (kEntASlice + kEntBSlice);
constexpr int kEntLd = 7;   // doubles per operand row of the FP64 sums
constexpr size_t kEntSmem = 1024 + kEntOps + 128 * 65 * 8 + 192 * kEntLd * 8;
// (a call: predicated, its FP64 instructions would take their slots for every entry, 9.0 ms instead of 5.7 for the Jacobian above)
__device__ __noinline__ double entry_sum(const double* a, const double* h) {
  return fma(a[2], h[2], fma(a[1], h[1], a[0] * h[0])) + fma(a[5], h[5], fma(a[4], h[4], a[3] * h[3]));
}
__global__ void __launch_bounds__(kLayThreads, 1) lay_hidden_entries(const LayEntries p) {
  constexpr int CR = 6;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* As =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* Bs = As + kEntS * kEntASlice;
  double* out_tile = reinterpret_cast<double*>(As + kEntOps);   // [128][65]
  double* xs = out_tile + 128 * 65;                             // [192][kEntLd]: the operand rows themselves
  __shared__ uint64_t done;
  __shared__ uint32_t tmem_slot;
  __shared__ int eA[128], eB[64];
  __shared__ float fA[128][7];                  // |factors| relative to 2^eA, 2^eB (pitch 7: no bank conflicts)
  __shared__ __align__(16) float fB[64][8];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  for (int idx = t; idx < kEntOps / 16; idx += kLayThreads)   // components 6 .. 31 stay zero
    reinterpret_cast<uint4*>(As)[idx] = make_uint4(0, 0, 0, 0);
  if (t == 0) {
    mbar_init(&done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "n"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int nl = p.net.L - 2, ng = (p.nr + 1) / 2;
  const int64_t units = p.npt * nl * ng;
  // this thread's operand row of a unit (threads 0 .. 127: A row = (row of the pair, o); 128 .. 191:
  // B row = i), loaded a unit ahead
  double x[CR];
  int eh[CR];
  auto load = [&](int64_t u) {
#pragma unroll
    for (int c = 0; c < CR; c++) {
      x[c] = 0.0;
      eh[c] = 0;
    }
    if (u >= units || t >= 192) return;
    const int64_t pl = u / (nl * ng);
    const int l = 1 + (int)(u / ng % nl), g = (int)(u % ng);
    const int in = p.net.w[l], out = p.net.w[l + 1];
#pragma unroll
    for (int c = 0; c < CR; c++) eh[c] = p.He[l][pl * CR + c];
    if (t < 128) {
      const int e = 2 * g + (t >> 6), o = t & 63;
      if (e < p.nr && o < out)
#pragma unroll
        for (int c = 0; c < CR; c++) x[c] = p.Ab[l + 1][((pl * p.nr + e) * CR + c) * out + o];
    } else {
      const int i = t - 128;
      if (i < in)
#pragma unroll
        for (int c = 0; c < CR; c++) x[c] = p.H[l][(pl * CR + c) * in + i];
    }
  };
  load(blockIdx.x);
  uint32_t phase = 0;
  for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
    const int64_t pl = u / (nl * ng);
    const int l = 1 + (int)(u / ng % nl), g = (int)(u % ng);
    const int in = p.net.w[l], out = p.net.w[l + 1];
    if (t < 192) {
      int m = kLayZero;
#pragma unroll
      for (int c = 0; c < CR; c++) {
        const int e = eh[c] == kLayBad ? kLayBad : exponent_above(x[c], t < 128 ? eh[c] : -eh[c]);
        m = e > m ? e : m;
      }
      (t < 128 ? eA[t] : eB[t - 128]) = m;
      const bool none = m == kLayBad || m == kLayZero;
      unsigned char* row = t < 128 ? As : Bs;
      const int r = t < 128 ? t : t - 128, stride = t < 128 ? kEntASlice : kEntBSlice;
#pragma unroll
      for (int c = 0; c < CR; c++) {
        const unsigned long long v = biased_digits(x[c], none ? kNoDigits : m - (t < 128 ? eh[c] : -eh[c]));
        unsigned char* dst = row + swz(r, c, 0);
#pragma unroll
        for (int d = 0; d < kEntS; d++) *reinterpret_cast<unsigned short*>(dst + d * stride) = digit_bf16(v, d);
        const float f = (float)abs((int)((long long)(v - kDigitBias) >> 32)) * 0x1p-30f;
        (t < 128 ? fA[t][c] : fB[t - 128][c]) = f;
        xs[t * kEntLd + c] = x[c];
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    if (t == 0 && !p.starve) {
      tc_fence_after();
      const uint64_t a0 = smem_desc(smem_u32(As)), b0 = smem_desc(smem_u32(Bs));
#pragma unroll
      for (int slot = 0; slot < kEntS; slot++)
#pragma unroll
        for (int s = 0; s <= slot; s++)
          mma_bf16<64>(tmem + slot * 64, a0 + (uint32_t)(s * (kEntASlice >> 4)),
                       b0 + (uint32_t)((slot - s) * (kEntBSlice >> 4)), s == 0 ? 0u : 1u);
      mma_commit(&done);
    }
    load(u + gridDim.x);   // arrives beside the products and the stores
    const bool ok = __syncthreads_and(mbar_wait(&done, phase, p.flag, p.wait_ns));
    phase ^= 1;
    if (!ok) {   // the host sees the status bit; this CTA's remaining entries become NaN
      mbar_wait(&done, phase ^ 1, p.flag, p.wait_ns);   // (products in flight, as in lay_gemm)
      for (; u < units; u += gridDim.x)
        for (int r = warp; r < 128; r += kLayThreads / 32) {
          const int ul = 1 + (int)(u / ng % nl), e = 2 * (int)(u % ng) + (r >> 6), o = r & 63, ui = p.net.w[ul];
          const int64_t jr = p.row0 + (p.p0 + u / (nl * ng)) * p.nr + e;
          if (e >= p.nr || o >= p.net.w[ul + 1] || jr < p.jlo || jr >= p.jhi) continue;
          double* dst = p.J + (jr - p.jlo) * p.ldJ + p.net.offW[ul] + (int64_t)o * ui;
          for (int i = lane; i < ui; i += 32) dst[i] = nan("");
        }
      break;
    }
    tc_fence_after();
    const int row = (warp & 3) * 32 + lane, ea = eA[row];
    const int re = 2 * g + (row >> 6), ro = row & 63;   // this row's residual row and output
    float fa[CR];
#pragma unroll
    for (int c = 0; c < CR; c++) fa[c] = fA[row][c];
#pragma unroll 1
    for (int part = 0; part < 2; part++) {
      const int col0 = (warp >> 2) * 16 + part * 8;
      if (col0 >= in) continue;
      uint32_t r[kEntS][8];
#pragma unroll
      for (int s = 0; s < kEntS; s++)
        tmem_ld8_async(tmem + ((uint32_t)((warp & 3) * 32) << 16) + s * 64 + col0, r[s]);
      tmem_wait_ld();
#pragma unroll
      for (int s = 0; s < kEntS; s++) tmem_use8(r[s]);
      unsigned weak = 0;
#pragma unroll
      for (int j = 0; j < 8; j++) {
        int v[kEntS];
#pragma unroll
        for (int s = 0; s < kEntS; s++)   // (accumulator s is v_s 256^-s)
          v[s] = __float2int_rn(__uint_as_float(r[s][j]) * __uint_as_float(0x3f800000u + ((unsigned)s << 26)));
        // sum_s v_s 256^(6 - s), the last level rounded in: below 2^63
        const long long hi = v[0] * 65536 + v[1] * 256 + v[2];
        const long long T = (hi << 32) + (long long)v[3] * 16777216 + (long long)v[4] * 65536 +
                            (v[5] * 256 + v[6] + ((v[7] + 128) >> 8));
        const int i = col0 + j, eb = eB[i];
        const bool bad = ea == kLayBad || eb == kLayBad, zero = ea == kLayZero || eb == kLayZero;
        out_tile[row * 65 + i] = zero ? 0.0 : scaled_int(T, ea + eb - 60);
        const float4 b4 = *reinterpret_cast<const float4*>(&fB[i][0]);
        const float2 b2 = *reinterpret_cast<const float2*>(&fB[i][4]);
        const float S = fmaf(fa[0], b4.x, fmaf(fa[1], b4.y, fmaf(fa[2], b4.z, fmaf(fa[3], b4.w, fmaf(fa[4], b2.x, fa[5] * b2.y)))));
        if (bad || (!zero && S < 0.017f)) weak |= 1u << j;   // 2^-5.88
      }
      if (re >= p.nr || ro >= out) weak = 0;
      for (; weak; weak &= weak - 1) {   // every lane its own entries
        const int i = col0 + __ffs(weak) - 1;
        if (i < in) out_tile[row * 65 + i] = entry_sum(xs + row * kEntLd, xs + (128 + i) * kEntLd);
      }
    }
    tc_fence_before();
    __syncthreads();
    // coalesced: a warp stores one output's row of `in` columns at a time
    for (int r = warp; r < 128; r += kLayThreads / 32) {
      const int e = 2 * g + (r >> 6), o = r & 63;
      const int64_t jr = p.row0 + (p.p0 + pl) * p.nr + e;
      if (e >= p.nr || o >= out || jr < p.jlo || jr >= p.jhi) continue;
      double* dst = p.J + (jr - p.jlo) * p.ldJ + p.net.offW[l] + (int64_t)o * in;
      if (lane < in) dst[lane] = out_tile[r * 65 + lane];
      if (lane + 32 < in) dst[lane + 32] = out_tile[r * 65 + lane + 32];
    }
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(512));
  }
}

// ---- gradient ------------------------------------------------------------------------------------------
// Adjoint mode sums the same products over the points: the weights of layer l get
// sum_(point, c) abar_(l+1)[c][o] h_l[c][i], the rest are sums over the points alone.  The points are
// cut into kLayParts parts, each with its own partial gradient (added in part order at the end).
constexpr int kLayParts = 64;
struct LayGrad {
  LayEntries e;
  const double* lamg;
  double* parts;            // [kLayParts][ldg], accumulated
  int64_t ldg;
};
// Hidden-to-hidden weights: one block per 16 x 16 outputs and part, eight groups of 64 threads
// (2 x 2 outputs each) sharing the rows (point, c).  FP64-bound; 16-wide tiles pad the usual widths
// (48, 64) not at all.
template <int D>
__global__ void __launch_bounds__(512) lay_outer(const LayGrad p) {
  constexpr int CR = JT<D>::CR, KG = 8;
  __shared__ double As[KG][16][17], Bs[KG][16][17];
  int l = 1, tile = blockIdx.x;
  for (; l < p.e.net.L - 1; l++) {
    const int nt = ((p.e.net.w[l] + 15) / 16) * ((p.e.net.w[l + 1] + 15) / 16);
    if (tile < nt) break;
    tile -= nt;
  }
  const int in = p.e.net.w[l], out = p.e.net.w[l + 1], ti = (in + 15) / 16;
  const int o0 = tile / ti * 16, i0 = tile % ti * 16;
  const int64_t R = p.e.npt * CR, per = (R + kLayParts - 1) / kLayParts;
  const int64_t r0 = blockIdx.y * per, r1 = r0 + per < R ? r0 + per : R;
  const double* A = p.e.Ab[l + 1];
  const double* B = p.e.H[l];
  const int t = threadIdx.x & 63, kg = threadIdx.x >> 6, tx = t & 7, ty = t >> 3;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int64_t k0 = r0; k0 < r1; k0 += KG * 16) {
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int kk = (t >> 4) + 4 * q, cc = t & 15;
      const int64_t r = k0 + kg * 16 + kk;
      As[kg][kk][cc] = (r < r1 && o0 + cc < out) ? A[r * out + o0 + cc] : 0.0;
      Bs[kg][kk][cc] = (r < r1 && i0 + cc < in) ? B[r * in + i0 + cc] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; kk++) {
      const double a0 = As[kg][kk][ty], a1 = As[kg][kk][ty + 8], b0 = Bs[kg][kk][tx], b1 = Bs[kg][kk][tx + 8];
      acc[0][0] = fma(a0, b0, acc[0][0]);
      acc[0][1] = fma(a0, b1, acc[0][1]);
      acc[1][0] = fma(a1, b0, acc[1][0]);
      acc[1][1] = fma(a1, b1, acc[1][1]);
    }
    __syncthreads();
  }
  // the groups' sums in group order
  double* sum = &As[0][0][0];
#pragma unroll
  for (int q = 0; q < 4; q++) sum[(q * KG + kg) * 64 + t] = acc[q >> 1][q & 1];
  __syncthreads();
  if (threadIdx.x < 256) {
    const int q = threadIdx.x >> 6;
    double v = 0.0;
#pragma unroll
    for (int g = 0; g < KG; g++) v += sum[(q * KG + g) * 64 + t];
    const int o = o0 + ty + 8 * (q >> 1), i = i0 + tx + 8 * (q & 1);
    if (o < out && i < in) p.parts[blockIdx.y * p.ldg + p.e.net.offW[l] + (int64_t)o * in + i] += v;
  }
}
// First and last layer's weights, the biases and lambda: one thread per entry and part.
template <int D>
__global__ void __launch_bounds__(256) lay_sums(const LayGrad p) {
  constexpr int CR = JT<D>::CR;
  const NetDesc& net = p.e.net;
  const int L = net.L;
  const int64_t per = (p.e.npt + kLayParts - 1) / kLayParts;
  const int64_t p0 = blockIdx.y * per, p1 = p0 + per < p.e.npt ? p0 + per : p.e.npt;
  int idx = blockIdx.x * 256 + threadIdx.x;
  double v = 0.0;
  int64_t at = -1;
  if (idx < net.w[1] * D) {
    const int o = idx / D, i = idx % D;
    const double* a = p.e.Ab[1] + o;
    for (int64_t q = p0; q < p1; q++)
      v += fma(a[q * CR * net.w[1]], p.e.qb[2 * q + i], a[(q * CR + 1 + i) * net.w[1]]);
    at = net.offW[0] + idx;
  } else if ((idx -= net.w[1] * D) < net.w[L] * net.w[L - 1]) {
    const int f = idx / net.w[L - 1], i = idx % net.w[L - 1];
    for (int64_t q = p0; q < p1; q++)
#pragma unroll
      for (int c = 0; c < CR; c++)
        v = fma(p.e.seeds[(q * net.w[L] + f) * CR + c], p.e.H[L - 1][(q * CR + c) * net.w[L - 1] + i], v);
    at = net.offW[L - 1] + idx;
  } else if ((idx -= net.w[L] * net.w[L - 1]) == 0) {
    for (int64_t q = p0; q < p1; q++) v += p.lamg[q];
    at = net.P;
  } else {
    idx -= 1;
    for (int l = 0; l < L; l++) {
      const int out = net.w[l + 1];
      if (idx < out) {
        const double* a = l < L - 1 ? p.e.Ab[l + 1] + idx : p.e.seeds + idx * CR;
        const int64_t step = l < L - 1 ? CR * out : out * CR;
        for (int64_t q = p0; q < p1; q++) v += a[q * step];
        at = net.offB[l] + idx;
        break;
      }
      idx -= out;
    }
  }
  if (at >= 0) p.parts[blockIdx.y * p.ldg + at] += v;
}

// ---- host side -----------------------------------------------------------------------------------------
// Scratch of one point, in doubles.
int64_t lay_point_doubles(const NetDesc& net, int d, int nf, int ne, int mode) {
  const int cr = d == 1 ? 2 : 6, cf = mode == MODE_RESIDUAL ? cr : (d == 1 ? 3 : 9);
  const int nr = mode == MODE_JACOBIAN ? ne : 1;
  int64_t n = 2 + nf * cf;
  for (int j = 1; j < net.L; j++) {
    if (j >= 2) n += (int64_t)cf * net.w[j];
    if (mode != MODE_RESIDUAL) n += (int64_t)cr * net.w[j] * (1 + nr) + (cr + 1) / 2;
  }
  if (mode != MODE_RESIDUAL) n += nr * nf * cr + 1 + 2 * (int64_t)nr * cr * kLayW;
  return n;
}
int64_t lay_ldg(const NetDesc& net) { return (net.P + 1 + 15) / 16 * 16; }
int64_t lay_parts_doubles(const NetDesc& net) { return kLayParts * lay_ldg(net); }
constexpr int64_t kLayFixed = 2 * GN_MAX_LAYERS * (kLaySl * kLayW * kLayW * 2 + 2 * kLayW * 4) + 8192;   // weight slices

int sm_count() {
  static const int n = [] {
    int dev = 0, v = 0;
    const bool ok = cudaGetDevice(&dev) == cudaSuccess &&
                    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0;
    return ok ? v : 152;
  }();
  return n;
}

template <int D, int C, int KIND>
cudaError_t run_gemm(const LayArgs& a, cudaStream_t st) {
  cudaError_t e =
      cudaFuncSetAttribute(lay_gemm<D, C, KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLaySmem);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (a.items + 128 / C - 1) / (128 / C);
  const int64_t grid = tiles < sm_count() ? tiles : sm_count();
  lay_gemm<D, C, KIND><<<(unsigned)grid, kLayThreads, kLaySmem, st>>>(a);
  count_launch();
  return cudaGetLastError();
}

// lay_hidden_entries always computes two rows by 64 outputs by 64 columns (and stops at the narrower
// layer's columns); the FP64 form pays for what there is.  Jacobian, FP64 -> products, three hidden layers, 8192
// points.  Two rows per point: width 40 1.96 -> 1.94 ms, 44 2.09 -> 2.01, 52 2.32 -> 2.10, 64 2.67 -> 2.27.
// Three rows (every second pair half empty): 52 3.13 -> 3.17 ms, 56 3.30 -> 3.30, 60 3.51 -> 3.35, 64 3.65 -> 3.42.
// A single row leaves half of every product empty.
template <int D>
bool hidden_entries(const NetDesc& net, int nr) {
  bool wide = D == 2 && nr > 1;
  for (int l = 1; l < net.L; l++) wide = wide && net.w[l] >= (nr % 2 ? 56 : 44);
  return wide;
}

template <int EQ, int MODE>
cudaError_t layers_eq(const JetArgs& A, void* ws, size_t ws_bytes, cudaStream_t st) {
  constexpr int D = Eq<EQ>::D, NF = Eq<EQ>::NF, NE = Eq<EQ>::NE, CR = JT<D>::CR;
  constexpr int C = (MODE == MODE_RESIDUAL) ? CR : JT<D>::CF;
  const NetDesc& net = A.net;
  const int L = net.L;
  const int ne = A.kind == KIND_INTERIOR ? NE : 1;
  const int nr = MODE == MODE_JACOBIAN ? ne : 1;
  unsigned char* wsl = static_cast<unsigned char*>(ws);
  int* we = reinterpret_cast<int*>(wsl + (size_t)2 * (L - 2) * kLaySl * kLayW * kLayW * 2);
  int* wc = we + 2 * (L - 2) * kLayW;
  double* parts = reinterpret_cast<double*>(wsl + kLayFixed);
  double* buf = parts + lay_parts_doubles(net);
  int64_t chunk = (int64_t)((ws_bytes - kLayFixed) / 8 - lay_parts_doubles(net)) /
                  lay_point_doubles(net, D, NF, NE, MODE);
  const int64_t wave = (int64_t)sm_count() * (128 / C);   // points of one round of forward tiles
  if (chunk > 2 * wave) chunk = chunk / wave * wave;
  const size_t opb = (size_t)kLaySl * kLayW * kLayW * 2;
  for (int64_t p0 = A.pt0; p0 < A.pt1; p0 += chunk) {
    const int64_t n = p0 + chunk < A.pt1 ? chunk : A.pt1 - p0;
    double* at = buf;
    auto take = [&](int64_t per) {
      double* r = at;
      at += per * n;
      return r;
    };
    double *Z[GN_MAX_LAYERS + 1] = {}, *H[GN_MAX_LAYERS + 1] = {}, *Ab[GN_MAX_LAYERS + 1] = {}, *hb[2] = {};
    double* qb = take(2);
    double* nn = take(NF * C);
    for (int j = 2; j < L; j++) Z[j] = take((int64_t)C * net.w[j]);
    double *seeds = nullptr, *lamg = nullptr;
    int* He[GN_MAX_LAYERS + 1] = {};
    if (MODE != MODE_RESIDUAL) {
      for (int j = 1; j < L; j++) {
        He[j] = reinterpret_cast<int*>(take((CR + 1) / 2));
        H[j] = take((int64_t)CR * net.w[j]);
        Ab[j] = take((int64_t)nr * CR * net.w[j]);
      }
      seeds = take(nr * NF * CR);
      lamg = take(1);
      hb[0] = take((int64_t)nr * CR * kLayW);
      hb[1] = take((int64_t)nr * CR * kLayW);
    }
    LayPrep pr;
    pr.y = A.y;
    pr.ystride = A.ystride;
    pr.pt0 = p0;
    pr.npt = n;
    pr.lam = A.lam;
    pr.lamp = A.lamp;
    pr.qb = qb;
    pr.theta = A.theta;
    pr.net = net;
    pr.wsl = wsl;
    pr.we = we;
    pr.wc = wc;
    pr.pt_blocks = (int)((n + 255) / 256);
    const int wblocks = p0 == A.pt0 ? (L - 2) * 2 * kLayW / 8 : 0;   // the weights once per pass
    lay_inputs<D><<<pr.pt_blocks + wblocks, 256, 0, st>>>(pr);
    count_launch();
    LayArgs g;
    memset(&g, 0, sizeof(g));
    g.nf = NF;
    g.cz = C;
    g.nr = nr;
    g.qb = qb;
    g.W0 = A.theta + net.offW[0];
    g.b0 = A.theta + net.offB[0];
    g.Wlast = A.theta + net.offW[L - 1];
    g.flag = A.flag + 2;
    g.wait_ns = g_oz_wait_ns.load(std::memory_order_relaxed);
    g.starve = g_oz_starve.load(std::memory_order_relaxed);
    cudaError_t e = cudaSuccess;
    for (int j = 1; j <= L - 2 && e == cudaSuccess; j++) {
      g.items = n;
      g.K = net.w[j];
      g.N = net.w[j + 1];
      g.zin = Z[j];
      g.bias = A.theta + net.offB[j - 1];
      g.hout = H[j];
      g.hexp = He[j];
      g.out = Z[j + 1];
      g.wsl = wsl + (size_t)(2 * (j - 1)) * opb;
      g.we = we + 2 * (j - 1) * kLayW;
      g.wc = wc + 2 * (j - 1) * kLayW;
      g.W = A.theta + net.offW[j];
      g.wso = net.w[j];
      g.wsk = 1;
      e = j == 1 ? run_gemm<D, C, LAY_FWD_FIRST>(g, st) : run_gemm<D, C, LAY_FWD>(g, st);
    }
    if (e != cudaSuccess) return e;
    lay_last<D, C, NF><<<(unsigned)((n + 7) / 8), 256, 0, st>>>(n, net.w[L - 1], Z[L - 1],
                                                                A.theta + net.offB[L - 2], H[L - 1],
                                                                A.theta + net.offW[L - 1],
                                                                A.theta + net.offB[L - 1], nn);
    count_launch();
    LayChain ch = {n, p0, nn, seeds, lamg};
    const dim3 cb(32, MODE == MODE_RESIDUAL ? 4 : 1 + NF * CR);
    const int64_t cpts = MODE == MODE_RESIDUAL ? 128 : 32;
    lay_chain<EQ, MODE><<<(unsigned)((n + cpts - 1) / cpts), cb, 0, st>>>(A, ch);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (MODE == MODE_RESIDUAL) continue;
    const double* hbar = nullptr;
    for (int j = L - 2; j >= 1; j--) {
      g.items = n * nr;
      g.K = net.w[j + 1];
      g.N = net.w[j];
      g.zin = Z[j + 1];
      g.hin = H[j + 1];
      g.seeds = seeds;
      g.hbar = hbar;
      g.abar = Ab[j + 1];
      g.out = hb[j & 1];
      g.wsl = wsl + (size_t)(2 * (j - 1) + 1) * opb;
      g.we = we + (2 * (j - 1) + 1) * kLayW;
      g.wc = wc + (2 * (j - 1) + 1) * kLayW;
      g.W = A.theta + net.offW[j];
      g.wso = 1;
      g.wsk = net.w[j];
      e = j == L - 2 ? run_gemm<D, CR, LAY_REV_LAST>(g, st) : run_gemm<D, CR, LAY_REV>(g, st);
      if (e != cudaSuccess) return e;
      hbar = hb[j & 1];
    }
    g.K = net.w[1];
    g.hin = H[1];
    g.hbar = hbar;
    g.abar = Ab[1];
    {
      int64_t blocks = (g.items * g.K + 255) / 256;
      if (blocks > 16 * sm_count()) blocks = 16 * sm_count();
      lay_first_adjoint<D><<<(unsigned)blocks, 256, 0, st>>>(g);
      count_launch();
    }
    LayEntries en;
    memset(&en, 0, sizeof(en));
    en.net = net;
    en.npt = n;
    en.p0 = p0;
    en.row0 = A.row0;
    en.ldJ = A.ldJ;
    en.jlo = A.jrow_lo;
    en.jhi = A.jrow_hi;
    en.nr = nr;
    en.qb = qb;
    for (int j = 1; j < L; j++) {
      en.H[j] = H[j];
      en.Ab[j] = Ab[j];
    }
    en.seeds = seeds;
    en.J = A.J;
    en.flag = A.flag + 2;
    en.wait_ns = g.wait_ns;
    en.starve = g.starve;
    en.hidden = !hidden_entries<D>(net, nr);
    for (int j = 1; j < L; j++) en.He[j] = He[j];
    if (MODE == MODE_GRADIENT) {
      LayGrad gr = {en, lamg, parts, lay_ldg(net)};
      int tiles = 0, sums = net.w[1] * D + net.w[L] * net.w[L - 1] + 1;
      for (int l = 0; l < L; l++) {
        if (l >= 1 && l < L - 1) tiles += ((net.w[l] + 15) / 16) * ((net.w[l + 1] + 15) / 16);
        sums += net.w[l + 1];
      }
      lay_outer<D><<<dim3((unsigned)tiles, kLayParts), 512, 0, st>>>(gr);
      count_launch();
      lay_sums<D><<<dim3((unsigned)((sums + 255) / 256), kLayParts), 256, 0, st>>>(gr);
      count_launch();
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      continue;
    }
    lay_entries<D><<<(unsigned)((n * L + 7) / 8), 256, 0, st>>>(en);
    count_launch();
    if (!en.hidden) {
      if ((e = cudaFuncSetAttribute(lay_hidden_entries, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kEntSmem)) != cudaSuccess)
        return e;
      const int64_t units = n * (L - 2) * ((nr + 1) / 2);
      lay_hidden_entries<<<(unsigned)(units < sm_count() ? units : sm_count()), kLayThreads, kEntSmem, st>>>(en);
      count_launch();
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int EQ>
cudaError_t layers_mode(const JetArgs& a, void* ws, size_t bytes, cudaStream_t st) {
  switch (a.mode) {
    case MODE_RESIDUAL: return layers_eq<EQ, MODE_RESIDUAL>(a, ws, bytes, st);
    case MODE_JACOBIAN: return layers_eq<EQ, MODE_JACOBIAN>(a, ws, bytes, st);
    default: return layers_eq<EQ, MODE_GRADIENT>(a, ws, bytes, st);
  }
}

}  // namespace

// The layered path takes tanh networks of at least two hidden layers, none wider than the 64 columns of its
// tiles, and point sets (all of them, not a row block's, so that a block's rows equal the whole's) large enough
// for its chain of 2 L launches and wide enough for what its tiles pad.  Pointwise / layered time in us over 2, 3 and 4
// hidden layers (FP64, Burgers and IPM; Boussinesq gains more than IPM):
//   1D residual   24 wide 4096 points 76/76 92/102 111/129, 6000 104/78 131/102 158/129; 32 wide 4096 82/64 102/92 127/119
//   1D Jacobian   28 wide 16384 points 455/409 653/668 852/909; 32 wide 4096 149/141 217/225 285/303, 6000 217/164
//                 317/254 416/352; 40 wide 4096 244/176 389/278 532/377
//   1D gradient   24 wide 16384 points 502/497 707/720 913/946; 28 wide 4096 221/190 307/262 395/333
//   2D residual   24 wide 1024 points 51/63 61/88 70/113, 2048 98/67 121/92 143/117
//   2D Jacobian   24 wide 8192 points 827/876 1223/1292 1656/1786; 32 wide 2048 309/295 477/436 647/614
//   2D gradient   24 wide 1024 points 201/215 269/284 337/348, 2048 314/247 426/333 541/414
// and at 64 wide, 3 hidden layers, 8192 points: Burgers 391/137 1134/557 1760/661, IPM 1177/297 5123/2273 4389/1722.
static bool layers_net(const NetDesc& net) {
  if (net.fourier || net.exp_out || net.L < 3) return false;
  for (int l = 1; l < net.L; l++)
    if (net.w[l] > kLayW || net.w[l] < 24) return false;
  return true;
}
static int64_t layers_min_points(const NetDesc& net, int mode) {
  const int d = net.w[0];
  int w = kLayW;   // the narrowest hidden layer
  for (int l = 1; l < net.L; l++) w = net.w[l] < w ? net.w[l] : w;
  if (w < (mode == MODE_JACOBIAN ? 32 : mode == MODE_GRADIENT && d == 1 ? 28 : 24)) return INT64_MAX;
  if (d == 2) return 2048;
  return mode != MODE_GRADIENT && w < (mode == MODE_JACOBIAN ? 40 : 32) ? 5000 : 4096;
}

bool layers_eligible(const JetArgs& a) {
  return a.kind != KIND_PROBE && layers_net(a.net) && a.n >= layers_min_points(a.net, a.mode);
}

size_t layers_ws_bytes(const NetDesc& net, int d, int nf, int ne, int64_t npt) {
  bool any = false;
  for (int mode : {MODE_RESIDUAL, MODE_JACOBIAN, MODE_GRADIENT})
    any = any || (layers_net(net) && npt >= layers_min_points(net, mode));
  if (!any) return 0;
  const int64_t per = lay_point_doubles(net, d, nf, ne, MODE_JACOBIAN) * 8;
  const int64_t cap = (int64_t)320 << 20;
  return (size_t)(kLayFixed + lay_parts_doubles(net) * 8 + (per * npt < cap ? per * npt : cap));
}
double* layers_parts(void* ws) { return reinterpret_cast<double*>(static_cast<unsigned char*>(ws) + kLayFixed); }
int layers_part_count() { return kLayParts; }

cudaError_t launch_layers(const JetArgs& a, void* ws, size_t ws_bytes, cudaStream_t st) {
  if (a.pt1 <= a.pt0) return cudaSuccess;
  switch (a.eq) {
    case GN_BURGERS: return layers_mode<GN_BURGERS>(a, ws, ws_bytes, st);
    case GN_CCF: return layers_mode<GN_CCF>(a, ws, ws_bytes, st);
    case GN_IPM: return layers_mode<GN_IPM>(a, ws, ws_bytes, st);
    case GN_BOUSSINESQ: return layers_mode<GN_BOUSSINESQ>(a, ws, ws_bytes, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace gn
