// Products of spectra modulo 31-bit primes: the transforms of the fused estimator for
// lengths N = 2^10 .. 2^22.  Included by sk_estimate.cu only.
//
// A length-N transform of a counter vector is split as N = R x 1024 (element n = 1024 n1 + n2,
// frequency nu = k1 + R k2):
//   k_ntt_cols  reads the int64 counters, reduces them modulo the prime, transforms the columns
//               (over n1, length R), multiplies by w_N^(n2 k1) and stores [k1][n2] residues;
//   k_ntt_rows  gives one warp the rows k1 of all r relations of one output: each row's
//               1024-point transform (32 x 32) stays in the warp's registers with one
//               shared-memory transposition, the r spectra are multiplied as they appear and
//               only their sum over nu leaves the SM.
// A relation whose spectrum is taken at -nu is transformed with the inverse root instead, so
// that all factors of a product sit in the same lane and register.  All primes of an estimate
// run in one launch (grid y).
//
// Bound: the integer multiplier, about five modular products per element and pass (a Montgomery
// product is two 32 x 32 -> 64-bit multiplies and one 32-bit one: 64 % of the pipe in the row pass,
// 50 % issue), and in the column pass the bytes.  m = 2^20 and 2^16 with Montgomery products
// throughout: 3.1 ns per 1024 elements and prime in the column pass, 2.3 ns in the row pass,
// against 1.8 and 0.6 ns for their bytes at the measured copy rate.  The chain of eight at m = 2^20,
// d = 16 (6 primes): 3.77 ms; 4.18 ms with Montgomery products throughout, 3.82 with the primes one
// after another over all tiles, 11.4 ms with residues, spectra and products each in their own pass
// over memory.
//
// Residues are plain (not in Montgomery form).  The fixed twiddles of the DFTs and of the row
// exchange come with their quotients (Factor), the others in Montgomery form with R = 2^32, so
// x (*) w is again a plain residue either way.  The r - 1 products of spectra each bring a
// factor 2^-32, which the host takes out of the final sums.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sk {
namespace ntt {

constexpr int kMaxPrimes = 9;
constexpr int kLogRow = 10;                 // row length 1024
constexpr int kMinLog = 10, kMaxLog = 22;   // transform lengths

// A fixed factor w with its quotient floor(w 2^32 / p) (Shoup's modular product).
struct alignas(8) Factor {
  uint32_t w, s;
};

struct PrimeConst {
  uint32_t p, pinv;     // pinv = -p^-1 mod 2^32
  uint32_t r2;          // 2^64 mod p
  Factor w64[2][32];    // w_64^j, j < 32: [0] forward, [1] inverse root
};
__constant__ PrimeConst c_prime[kMaxPrimes];

__device__ __align__(16) Factor g_row[kMaxPrimes][2][1024];   // w_1024^(c b) at 32 c + b, [prime][direction]

// Powers of the roots of unity, Montgomery form, [prime][direction]:
__device__ uint32_t g_root[kMaxPrimes][2][4096];                           // w_4096^e
__device__ uint32_t g_low[kMaxPrimes][2][kMaxLog - kMinLog + 1][1024];     // w_N^e, e < 1024

struct Mod {
  uint32_t p, pinv;
};

// a + b, a - b mod p for a, b < p < 2^31: the wrapped candidate is the larger one
__device__ __forceinline__ uint32_t add(uint32_t a, uint32_t b, Mod q) {
  const uint32_t s = a + b;
  return min(s, s - q.p);
}
__device__ __forceinline__ uint32_t sub(uint32_t a, uint32_t b, Mod q) {
  const uint32_t s = a - b;
  return min(s, s + q.p);
}
// a b 2^-32 mod p for a b < 2^32 * 2^31 (Montgomery): t + q p < 2^64, its high word < 2p
__device__ __forceinline__ uint32_t mul(uint32_t a, uint32_t b, Mod q) {
  const uint64_t t = (uint64_t)a * b;
  const uint32_t m = (uint32_t)t * q.pinv;
  const uint32_t u = (uint32_t)((t + (uint64_t)m * q.p) >> 32);
  return min(u, u - q.p);
}

// a w mod p for any a: with q = floor(a s / 2^32), a w - q p < 2p.  One 64-bit product and two
// 32-bit ones; a Montgomery product takes two and one (32-point DFTs alone: 0.61 -> 0.48 ns
// per 1024 elements).
__device__ __forceinline__ uint32_t mul(uint32_t a, Factor f, Mod q) {
  const uint32_t u = a * f.w - __umulhi(a, f.s) * q.p;
  return min(u, u - q.p);
}

// c mod p for any int64, |c| = h 2^32 + l: two Montgomery products for l, one for h
__device__ __forceinline__ uint32_t residue(int64_t c, Mod q, uint32_t r2) {
  const uint64_t mag = c < 0 ? 0ull - (uint64_t)c : (uint64_t)c;
  const uint32_t v = add(mul(mul((uint32_t)mag, r2, q), 1u, q), mul((uint32_t)(mag >> 32), r2, q), q);
  return c < 0 && v ? q.p - v : v;
}

// x[i] = src[i stride] mod p for i < K, zero where i stride >= left: the loads of a batch of up
// to 16 are in flight together, and one branch per batch decides between the short reduction
// (every |c| < 2^30) and the general one.  With a branch per element each load waited for the
// one before it (column pass 7.1 ns per 1024 elements).
template <int K>
__device__ __forceinline__ void load_residues(uint32_t (&x)[K], const int64_t* __restrict__ src, int64_t stride,
                                              int64_t left, Mod q, uint32_t r2) {
  constexpr int U = K < 16 ? K : 16;
#pragma unroll
  for (int i0 = 0; i0 < K; i0 += U) {
    int64_t c[U];
#pragma unroll
    for (int i = 0; i < U; i++) c[i] = (i0 + i) * stride < left ? __ldg(src + (i0 + i) * stride) : 0;
    uint64_t far = 0;   // bits 31 and up: some |c| >= 2^30
#pragma unroll
    for (int i = 0; i < U; i++) far |= (uint64_t)(c[i] + (1ll << 30));
    if (far < (1ull << 31)) {
#pragma unroll
      for (int i = 0; i < U; i++) x[i0 + i] = min((uint32_t)c[i], (uint32_t)c[i] + q.p);
    } else {
#pragma unroll
      for (int i = 0; i < U; i++) x[i0 + i] = residue(c[i], q, r2);
    }
  }
}

constexpr int rev_bits(int k, int bits) {
  int r = 0;
  for (int i = 0; i < bits; i++) r |= ((k >> i) & 1) << (bits - 1 - i);
  return r;
}

// 2^LOG-point DFT in registers, natural order in and out; w64[j] = w_64^j.  Radix-2 decimation
// in frequency; the difference of a butterfly with a twiddle is left in (0, 2p) for mul.
template <int LOG>
__device__ __forceinline__ void dft(uint32_t (&x)[1 << LOG], const Factor* w64, Mod q) {
  constexpr int N = 1 << LOG;
#pragma unroll
  for (int st = 0; st < LOG; st++) {
    const int h = N >> (st + 1);
#pragma unroll
    for (int blk = 0; blk < N; blk += 2 * h) {
#pragma unroll
      for (int j = 0; j < h; j++) {
        const uint32_t u = x[blk + j], v = x[blk + j + h];
        x[blk + j] = add(u, v, q);
        x[blk + j + h] = j == 0 ? sub(u, v, q) : mul(u - v + q.p, w64[(j << st) << (6 - LOG)], q);
      }
    }
  }
  uint32_t y[N];
#pragma unroll
  for (int k = 0; k < N; k++) y[k] = x[rev_bits(k, LOG)];
#pragma unroll
  for (int k = 0; k < N; k++) x[k] = y[k];
}

// x[i] = L[i stride] for i < K, zero where i stride >= left; with fold, the circular value
// L[i stride] + L[i stride + fold].
template <int K>
__device__ __forceinline__ void load_words(uint32_t (&x)[K], const uint32_t* L, int64_t stride, int64_t left,
                                           int64_t fold, Mod q) {
#pragma unroll
  for (int i = 0; i < K; i++) x[i] = i * stride < left ? L[i * stride] : 0u;
  if (fold) {
    uint32_t y[K];
#pragma unroll
    for (int i = 0; i < K; i++) y[i] = i * stride < left ? L[i * stride + fold] : 0u;
#pragma unroll
    for (int i = 0; i < K; i++) x[i] = add(x[i], y[i], q);
  }
}

// Vectors of one launch.  Counters: vector v is base[v / per] + (v % per) m, its direction (1:
// inverse root) dirs[v] or bit v / per of negmask.  Words: vector v of the prime is the residues
// at words + (prime stride + v) N, direction bit 0 of negmask.  Either is taken as zero from m on,
// and words with fold != 0 as the circular sum of two of them (see load_words).
struct ColArgs {
  const int64_t* const* base;
  int per;
  int64_t m;
  unsigned long long negmask;
  const uint8_t* dirs;
  int logR;
  uint32_t* V;              // [prime][stride vectors][N]
  int64_t stride;           // vectors per prime in V
  int prime0;               // first prime of the launch
  int nvec[kMaxPrimes];     // vectors of each prime (leading ones)
  int primes = 1;           // of the launch
  const uint32_t* words = nullptr;   // may be V: a CTA reads its columns before it writes them
  int64_t fold = 0;
};

__device__ __forceinline__ int dir_of(const ColArgs& a, int64_t v) {
  return a.dirs ? a.dirs[v] : (int)((a.negmask >> (v / a.per)) & 1ull);
}

// w_N^e for e < N = R 1024
__device__ __forceinline__ uint32_t root_pow(int prime, int dir, int logR, uint32_t e, Mod q) {
  const uint32_t lo = g_low[prime][dir][logR][e & 1023u], hi = e >> kLogRow;
  return hi ? mul(lo, g_root[prime][dir][hi << (12 - logR)], q) : lo;
}

// R = 2^(LA + LB).  A thread of a CTA of 256 holds one A- or B-point DFT (A <= B) of one of cb =
// 256 / A columns: the counters go from global memory into registers, through one shared-memory
// exchange between the two levels and back to global memory.  LA = 0: R = B points per thread,
// no exchange.  64-byte column segments of counters are read and 32-byte ones of residues written
// up to R = 1024, where wider tiles would not save sectors.  R = 2048 has the same eight columns; R =
// 4096 has four: it reads 32 bytes (16 of residues) and writes half sectors, which L2 puts together.
//
// WORDS: residues instead of counters.  BACK: the inverse transform's column pass, on residues
// that k_ntt_corr has multiplied by the inverse twiddle already.
template <int LA, int LB, bool WORDS, bool BACK>
__global__ void __launch_bounds__(256, (LB <= 5 ? 4 : 2)) k_ntt_cols(const __grid_constant__ ColArgs a) {
  constexpr int A = 1 << LA, B = 1 << LB, LR = LA + LB;
  constexpr int LCB = LA ? 8 - LA : 8, CB = 1 << LCB;
  // the primes of one tile run next to each other: its counters come from memory once
  const unsigned pi = blockIdx.x % (unsigned)a.primes, tile = blockIdx.x / (unsigned)a.primes;
  const int prime = a.prime0 + (int)pi;
  const int64_t vec = tile >> (kLogRow - LCB);
  if (vec >= a.nvec[prime]) return;
  const int n2 = (int)(tile & ((1u << (kLogRow - LCB)) - 1u)) * CB + (int)(threadIdx.x & (CB - 1));
  const Mod q = {c_prime[prime].p, c_prime[prime].pinv};
  const uint32_t r2 = c_prime[prime].r2;
  const int dir = WORDS ? (int)(a.negmask & 1ull) : dir_of(a, vec);
  const Factor* w64 = c_prime[prime].w64[dir];
  const int64_t at0 = (((int64_t)pi * a.stride + vec) << (LR + kLogRow)) + n2;
  const int64_t* src = WORDS ? nullptr : a.base[vec / a.per] + (vec % a.per) * a.m + n2;
  uint32_t* dst = a.V + at0;
  const int64_t left = a.m - n2;   // counters of this column: rows n1 with 1024 n1 < left
  extern __shared__ uint32_t s_col[];
  const int c = (int)(threadIdx.x >> LCB);   // this thread's k1 residue at the second level
  uint32_t x[B];
  if constexpr (LA > 0) {
    // [c][b] twiddles w_R^(c b), then the exchange tile: element (c, b) of column v at
    // (c (B + 1) + b) CB + v, which keeps writes (b, v fast) and reads (c, v fast) conflict-free
    uint32_t* tw = s_col;
    uint32_t* ex = s_col + A * B;
    for (int i = threadIdx.x; i < A * B; i += 256)
      tw[i] = g_root[prime][dir][((i >> LB) * (i & (B - 1))) << (12 - LR)];
    __syncthreads();
    const int v = (int)(threadIdx.x & (CB - 1));
#pragma unroll
    for (int s = 0; s < B / A; s++) {
      const int b = (int)(threadIdx.x >> LCB) + A * s;
      uint32_t y[A];
      const int64_t at = (int64_t)b << kLogRow;
      if (WORDS) load_words<A>(y, a.words + at0 + at, (int64_t)B << kLogRow, left - at, a.fold, q);
      else load_residues<A>(y, src + at, (int64_t)B << kLogRow, left - at, q, r2);
      dft<LA>(y, w64, q);
#pragma unroll
      for (int i = 0; i < A; i++) ex[(i * (B + 1) + b) * CB + v] = i ? mul(y[i], tw[i * B + b], q) : y[i];
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < B; b++) x[b] = ex[(c * (B + 1) + b) * CB + v];
  } else {
    if (WORDS) load_words<B>(x, a.words + at0, 1 << kLogRow, left, a.fold, q);
    else load_residues<B>(x, src, 1 << kLogRow, left, q, r2);
  }
  dft<LB>(x, w64, q);
  // x[e] is row k1 = c + A e: times w_N^(n2 k1), advanced in two chains of step w_N^(2 A n2)
  const uint32_t k0 = LA ? (uint32_t)c : 0u;
  if constexpr (BACK) {
#pragma unroll
    for (int e = 0; e < B; e++) dst[(int64_t)(k0 + A * e) << kLogRow] = x[e];
  } else if constexpr (LR > 0) {
    uint32_t w0 = root_pow(prime, dir, LR, (uint32_t)n2 * k0, q);
    const uint32_t st = root_pow(prime, dir, LR, (uint32_t)n2 * A, q);
    uint32_t w1 = mul(w0, st, q);
    const uint32_t st2 = mul(st, st, q);
#pragma unroll
    for (int e = 0; e < B; e += 2) {
      dst[(int64_t)(k0 + A * e) << kLogRow] = mul(x[e], w0, q);
      dst[(int64_t)(k0 + A * (e + 1)) << kLogRow] = mul(x[e + 1], w1, q);
      if (e + 2 < B) {
        w0 = mul(w0, st2, q);
        w1 = mul(w1, st2, q);
      }
    }
  } else {
    dst[0] = x[0];
  }
}

// One output: the product over its r vectors base + k step (k < r).
struct Out {
  int64_t base, step;
  int r;
  unsigned long long negmask;   // bit k: vector k was transformed with the inverse root
};

struct RowArgs {
  const uint32_t* V;
  int64_t stride;
  int logR, prime0;
  const Out* outs;            // nullptr: output o is {o, one.step, one.r, one.negmask}
  Out one;
  int nout[kMaxPrimes];
  unsigned long long* sums;   // [out][kMaxPrimes] += sum over nu of the product (residues < p)
};

// 8 warps, one row k1 each; sums of at most 2^22 residues below 2^31 fit 64 bits.  The running
// products live in shared memory: with them in registers the kernel spilled at 128 registers
// (2.40 against 2.24 ns per 1024 elements), and more warps per SM (80 registers) only spilled
// more (2.6): the multiplier pipe, not the number of warps, sets the rate.
__global__ void __launch_bounds__(256, 2) k_ntt_rows(const __grid_constant__ RowArgs a) {
  __shared__ __align__(16) Factor s_tw[2][1024];
  __shared__ uint32_t s_ex[8][32 * 33];
  __shared__ unsigned long long s_sum[8];
  extern __shared__ uint32_t s_prod[];   // 8 x 1024
  const int prime = a.prime0 + (int)blockIdx.y;
  const int R = 1 << a.logR;
  const int lcta = a.logR > 3 ? a.logR - 3 : 0;   // log2 CTAs per output
  const int64_t o = blockIdx.x >> lcta;
  if (o >= a.nout[prime]) return;
  const int lane = (int)(threadIdx.x & 31u), warp = (int)(threadIdx.x >> 5);
  const int k1 = (int)(blockIdx.x & ((1u << lcta) - 1u)) * 8 + warp;
  const Mod q = {c_prime[prime].p, c_prime[prime].pinv};
  for (int i = threadIdx.x; i < 1024; i += 256) ((uint4*)s_tw)[i] = ((const uint4*)g_row[prime])[i];
  __syncthreads();
  unsigned long long sum = 0;
  if (k1 < R) {
    Out f;
    if (a.outs) {
      f = a.outs[o];
    } else {
      f = a.one;
      f.base = o;
    }
    const uint32_t* row =
        a.V + (((int64_t)blockIdx.y * a.stride + f.base) << (a.logR + kLogRow)) + ((int64_t)k1 << kLogRow) + lane;
    const int64_t rstep = f.step << (a.logR + kLogRow);
    uint32_t* ex = s_ex[warp];
    uint32_t* prod = s_prod + warp * 1024 + lane;   // this lane's 32 running products, stride 32
    uint32_t x[32];
#pragma unroll
    for (int i = 0; i < 32; i++) x[i] = __ldcs(row + 32 * i);
    for (int k = 0; k < f.r; k++) {
      const int dir = (int)((f.negmask >> k) & 1ull);
      const Factor* w64 = c_prime[prime].w64[dir];
      const Factor* tw = s_tw[dir];
      dft<5>(x, w64, q);
#pragma unroll
      for (int i = 0; i < 32; i++) ex[i * 33 + lane] = i ? mul(x[i], tw[i * 32 + lane], q) : x[i];
      __syncwarp();
      uint32_t y[32];
#pragma unroll
      for (int i = 0; i < 32; i++) y[i] = ex[lane * 33 + i];
      __syncwarp();
      row += rstep;
      if (k + 1 < f.r) {   // the next vector's row, in flight during this one's second level
#pragma unroll
        for (int i = 0; i < 32; i++) x[i] = __ldcs(row + 32 * i);
      }
      dft<5>(y, w64, q);
      if (k == 0) {
#pragma unroll
        for (int i = 0; i < 32; i++) prod[32 * i] = y[i];
      } else {
#pragma unroll
        for (int i = 0; i < 32; i++) prod[32 * i] = mul(prod[32 * i], y[i], q);
      }
    }
#pragma unroll
    for (int i = 0; i < 32; i++) sum += prod[32 * i];
  }
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, s);
  if (lane == 0) s_sum[warp] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; w++) sum += s_sum[w];
    atomicAdd(a.sums + o * kMaxPrimes + prime, sum);
  }
}

// One correlation of the step-by-step schedule, between the column passes: rows k1 of A (columns
// transformed with the inverse root, so its entries are A(-nu)) and X, both transformed, multiplied
// and transformed back in one warp's registers -- entry k2 = c + 32 e of a product is where the
// inverse transform's first level wants it -- then times w_N^(-n2 k1) for k_ntt_cols<.., BACK>.
// The result carries 2^-32 from the product and M from the missing 1 / M; the caller keeps track.
struct CorrRowArgs {
  const uint32_t *A, *X;   // [prime][stride][N]
  uint32_t* Z;
  int64_t stride;
  int logR, prime0, nvec;
};

__global__ void __launch_bounds__(256, 2) k_ntt_corr(const __grid_constant__ CorrRowArgs a) {
  __shared__ __align__(16) Factor s_tw[2][1024];
  __shared__ uint32_t s_ex[8][32 * 33];
  extern __shared__ uint32_t s_prod[];   // 8 x 1024
  const int prime = a.prime0 + (int)blockIdx.y;
  const int R = 1 << a.logR;
  const int lcta = a.logR > 3 ? a.logR - 3 : 0;
  const int64_t v = blockIdx.x >> lcta;
  const int lane = (int)(threadIdx.x & 31u), warp = (int)(threadIdx.x >> 5);
  const int k1 = (int)(blockIdx.x & ((1u << lcta) - 1u)) * 8 + warp;
  const Mod q = {c_prime[prime].p, c_prime[prime].pinv};
  for (int i = threadIdx.x; i < 1024; i += 256) ((uint4*)s_tw)[i] = ((const uint4*)g_row[prime])[i];
  __syncthreads();
  if (k1 >= R) return;
  const int64_t at = (((int64_t)blockIdx.y * a.stride + v) << (a.logR + kLogRow)) + ((int64_t)k1 << kLogRow) + lane;
  uint32_t* ex = s_ex[warp];
  uint32_t* prod = s_prod + warp * 1024 + lane;
  uint32_t x[32], y[32];
#pragma unroll
  for (int i = 0; i < 32; i++) x[i] = __ldcs(a.A + at + 32 * i);
  // A with the inverse root, X, then the product with the inverse root
#pragma unroll 1
  for (int step = 0; step < 3; step++) {
    const int dir = step == 1 ? 0 : 1;
    const Factor* w64 = c_prime[prime].w64[dir];
    const Factor* tw = s_tw[dir];
    dft<5>(x, w64, q);
#pragma unroll
    for (int i = 0; i < 32; i++) ex[i * 33 + lane] = i ? mul(x[i], tw[i * 32 + lane], q) : x[i];
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 32; i++) y[i] = ex[lane * 33 + i];
    __syncwarp();
    if (step == 0) {
#pragma unroll
      for (int i = 0; i < 32; i++) x[i] = __ldcs(a.X + at + 32 * i);
    }
    dft<5>(y, w64, q);
    if (step == 0) {
#pragma unroll
      for (int i = 0; i < 32; i++) prod[32 * i] = y[i];
    } else if (step == 1) {
#pragma unroll
      for (int i = 0; i < 32; i++) x[i] = mul(prod[32 * i], y[i], q);
    }
  }
  // y[e] is column n2 = lane + 32 e
  uint32_t w0 = root_pow(prime, 1, a.logR, (uint32_t)k1 * (uint32_t)lane, q);
  const uint32_t st = root_pow(prime, 1, a.logR, (uint32_t)k1 * 32u, q);
  uint32_t w1 = mul(w0, st, q);
  const uint32_t st2 = mul(st, st, q);
#pragma unroll
  for (int e = 0; e < 32; e += 2) {
    a.Z[at + 32 * e] = mul(y[e], w0, q);
    a.Z[at + 32 * (e + 1)] = mul(y[e + 1], w1, q);
    w0 = mul(w0, st2, q);
    w1 = mul(w1, st2, q);
  }
}

// A vector operand of the schedule's elementwise steps: row v's counters c + v m, or its residues
// u + (prime stride + v) N, circular (fold) or not; m entries either way.
struct Operand {
  const int64_t* c;
  const uint32_t* u;
  int64_t fold;
};

struct HadArgs {
  Operand x, y;               // y.c and y.u null: x alone (the plain sum)
  uint32_t* out;              // [prime][stride][N] products x y 2^-32; nullptr: only their sums
  unsigned long long* sums;   // [row][kMaxPrimes]
  int64_t stride, m;
  int logN, prime0;
};

__device__ __forceinline__ uint32_t operand_at(const Operand& o, int64_t at, int64_t row, int64_t m, int64_t j, Mod q,
                                               uint32_t r2) {
  if (o.c) {
    const int64_t c = __ldg(o.c + row * m + j);
    if ((uint64_t)(c + (1ll << 30)) < (1ull << 31)) return min((uint32_t)c, (uint32_t)c + q.p);
    return residue(c, q, r2);
  }
  const uint32_t v = o.u[at + j];
  return o.fold ? add(v, o.u[at + j + o.fold], q) : v;
}

// grid (chunks, rows, primes), 256 threads
__global__ void __launch_bounds__(256) k_ntt_had(const __grid_constant__ HadArgs a) {
  __shared__ unsigned long long s_sum[8];
  const int prime = a.prime0 + (int)blockIdx.z;
  const int64_t row = blockIdx.y;
  const Mod q = {c_prime[prime].p, c_prime[prime].pinv};
  const uint32_t r2 = c_prime[prime].r2;
  const int64_t at = ((int64_t)blockIdx.z * a.stride + row) << a.logN;
  const bool two = a.y.c || a.y.u;
  unsigned long long sum = 0;
  for (int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x; j < a.m; j += (int64_t)gridDim.x * 256) {
    uint32_t v = operand_at(a.x, at, row, a.m, j, q, r2);
    if (two) v = mul(v, operand_at(a.y, at, row, a.m, j, q, r2), q);
    if (a.out) a.out[at + j] = v;
    else sum += v;
  }
  if (a.out) return;
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, s);
  if ((threadIdx.x & 31u) == 0) s_sum[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; w++) sum += s_sum[w];
    atomicAdd(a.sums + row * kMaxPrimes + prime, sum);
  }
}

inline cudaError_t corr_rows(const CorrRowArgs& a, int primes, cudaStream_t st) {
  const int lcta = a.logR > 3 ? a.logR - 3 : 0;
  constexpr size_t smem = 8 * 1024 * sizeof(uint32_t);
  const cudaError_t e = allow_dynamic_smem((const void*)k_ntt_corr);
  if (e != cudaSuccess) return e;
  k_ntt_corr<<<dim3((unsigned)((int64_t)a.nvec << lcta), (unsigned)primes), 256, smem, st>>>(a);
  count_launch();
  return cudaGetLastError();
}

inline cudaError_t had(const HadArgs& a, int rows, int primes, int sms, cudaStream_t st) {
  // about four waves of CTAs of at least 1024 entries
  const int64_t want = (4ll * 8 * sms + (int64_t)rows * primes - 1) / ((int64_t)rows * primes);
  const int64_t most = (a.m + 1023) / 1024;
  k_ntt_had<<<dim3((unsigned)(want < most ? want : most), (unsigned)rows, (unsigned)primes), 256, 0, st>>>(a);
  count_launch();
  return cudaGetLastError();
}

template <int LA, int LB, bool WORDS, bool BACK>
cudaError_t launch_cols(ColArgs a, int64_t nvec, int primes, cudaStream_t st) {
  constexpr int LCB = LA ? 8 - LA : 8;
  const size_t smem = LA ? ((size_t)(1 << (LA + LB)) + ((size_t)(1 << LA) * ((1 << LB) + 1) << LCB)) * 4 : 0;
  const cudaError_t e = fit_dynamic_smem((const void*)k_ntt_cols<LA, LB, WORDS, BACK>, smem);
  if (e != cudaSuccess) return e;
  a.primes = primes;
  k_ntt_cols<LA, LB, WORDS, BACK><<<(unsigned)((nvec << (kLogRow - LCB)) * primes), 256, smem, st>>>(a);
  count_launch();
  return cudaGetLastError();
}

template <bool WORDS, bool BACK>
cudaError_t cols_of(const ColArgs& a, int64_t nvec, int primes, cudaStream_t st) {
  switch (a.logR) {
    case 0: return launch_cols<0, 0, WORDS, BACK>(a, nvec, primes, st);
    case 1: return launch_cols<0, 1, WORDS, BACK>(a, nvec, primes, st);
    case 2: return launch_cols<0, 2, WORDS, BACK>(a, nvec, primes, st);
    case 3: return launch_cols<0, 3, WORDS, BACK>(a, nvec, primes, st);
    case 4: return launch_cols<0, 4, WORDS, BACK>(a, nvec, primes, st);
    case 5: return launch_cols<0, 5, WORDS, BACK>(a, nvec, primes, st);
    case 6: return launch_cols<3, 3, WORDS, BACK>(a, nvec, primes, st);
    case 7: return launch_cols<3, 4, WORDS, BACK>(a, nvec, primes, st);
    case 8: return launch_cols<4, 4, WORDS, BACK>(a, nvec, primes, st);
    case 9: return launch_cols<4, 5, WORDS, BACK>(a, nvec, primes, st);
    case 10: return launch_cols<5, 5, WORDS, BACK>(a, nvec, primes, st);
    case 11: return launch_cols<5, 6, WORDS, BACK>(a, nvec, primes, st);
    default: return launch_cols<6, 6, WORDS, BACK>(a, nvec, primes, st);
  }
}

inline cudaError_t cols(const ColArgs& a, int64_t nvec, int primes, cudaStream_t st) {
  return a.words ? cols_of<true, false>(a, nvec, primes, st) : cols_of<false, false>(a, nvec, primes, st);
}

inline cudaError_t cols_back(const ColArgs& a, int64_t nvec, int primes, cudaStream_t st) {
  return cols_of<true, true>(a, nvec, primes, st);
}

inline cudaError_t rows(const RowArgs& a, int64_t nout, int primes, cudaStream_t st) {
  const int lcta = a.logR > 3 ? a.logR - 3 : 0;
  constexpr size_t smem = 8 * 1024 * sizeof(uint32_t);
  const cudaError_t e = allow_dynamic_smem((const void*)k_ntt_rows);   // 82 KB with its static arrays
  if (e != cudaSuccess) return e;
  k_ntt_rows<<<dim3((unsigned)(nout << lcta), (unsigned)primes), 256, smem, st>>>(a);
  count_launch();
  return cudaGetLastError();
}

}  // namespace ntt
}  // namespace sk
