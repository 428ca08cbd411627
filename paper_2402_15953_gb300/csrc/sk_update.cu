// Sketch update (Algorithm 2, Eqs. 2-4) and merge (Section 2.2) kernels.
//
// Every tuple of relation R_k is hashed for all d median rows: for each of its
// joined attributes u the key is mapped into GF(p), p = 2^61 - 1, the bin
// function of u's component h(x) = ((b1 x + b0) mod p) mod m and the sign
// functions of u's joins s(x) = +-1 from the parity of (s0 + s1 x + s2 x^2 +
// s3 x^3) mod p are evaluated; the tuple's bin is the sum of the bins mod m and
// its sign the product of the signs; sign * Delta is added to that counter.
//
// Two scatter targets:
//   - SMEM: the d x m sub-sketch fits in shared memory; each CTA accumulates
//     into block-private int32 counters (exact: the host bounds |Delta| times
//     the tuples a CTA sees below 2^31, larger weights go straight to global
//     memory) and flushes the non-zero counters into the int64 sketch with
//     64-bit atomics at the end;
//   - GLOBAL: 64-bit atomic adds straight into the int64 sketch (resident in
//     L2 when d * m * 8 bytes is small against the 126 MiB L2).
// Counters wrap like two's-complement int64 (additions are done on uint64).
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <type_traits>

#include "sk_hash.cuh"
#include "sk_internal.h"

namespace sk {
namespace {

using namespace dev;


template <int A, bool POW2, bool SMEM, bool DEG1>
__global__ void __launch_bounds__(256) k_update(UpdArgs p, const int* unless) {
  if (unless && *unless) return;   // another path has the batch (see update_undeclared)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t* s_coef = (uint64_t*)smem_raw;
  const int ncoef = p.d * p.row_len;
  int* s_sub = (int*)(s_coef + ncoef);
  const int64_t dm = (int64_t)p.d * (int64_t)p.m;
  for (int i = threadIdx.x; i < ncoef; i += blockDim.x) s_coef[i] = p.coef[i];
  if (SMEM)
    for (int64_t i = threadIdx.x; i < dm; i += blockDim.x) s_sub[i] = 0;
  __syncthreads();

  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  if constexpr (A == 1 && !SMEM) {
    const int lane = threadIdx.x & 31;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x - lane); b < p.n; b += step)
      update_warp_key<POW2, DEG1>(p, s_coef, b + lane, b + lane < p.n);
    return;
  }
  if (SMEM && p.agg) {
    // warp-uniform loop: every lane of a warp runs the same iterations (collectives inside)
    const int lane = threadIdx.x & 31;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x - lane); b < p.n; b += step)
      update_tuple<A, POW2, SMEM, true, DEG1>(p, s_coef, s_sub, b + lane, b + lane < p.n);
  } else {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += step)
      update_tuple<A, POW2, SMEM, false, DEG1>(p, s_coef, s_sub, i);
  }
  if (SMEM) {
    __syncthreads();
    for (int64_t i = threadIdx.x; i < dm; i += blockDim.x) {
      const int v = s_sub[i];
      if (v != 0) atomicAdd(p.ctr + i, (unsigned long long)(int64_t)v);
    }
  }
}

// Whether a weighted batch's weights suit the items: set by the table kernel, which runs before
// both phases, from 1024 tuples of the batch.
struct PartChoice {
  int direct;   // most weights are beyond wmax: every tuple straight to the counters
};

struct WeightSample {
  const int64_t* w;        // nullptr: unit weights
  int64_t n;
  int64_t wmax;            // the largest |Delta| an item holds
  PartChoice* choice;
};

// By the table kernel's last CTA (of 256 threads), which then has no keys.  Weights beyond wmax cost
// their reductions and what the items of the others cost besides; with few of them the items win:
// 7e7 tuples of two columns, m = 2^16, d = 9: 2090 us with none, 2110 with a tenth, 3460 with three
// quarters, 4180 with nearly all, against 3720 for reductions alone.  The line is at 0.7.
__device__ __forceinline__ void choose_path(const WeightSample& s) {
  bool far[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int64_t j = 256 * k + threadIdx.x;
    const int64_t w = __ldg(s.w + (s.n >> 10) * j + (((s.n & 1023) * j) >> 10));
    far[k] = w > s.wmax || w < -s.wmax;
  }
  int beyond = 0;
#pragma unroll
  for (int k = 0; k < 4; k++) beyond += __syncthreads_count(far[k]);
  if (threadIdx.x == 0) s.choice->direct = beyond > 717;
}

// Key-table records for every declared domain key of every attribute (one thread per key).
template <bool POW2, bool DEG1>
__global__ void __launch_bounds__(256) k_key_table(UpdArgs p, TabArgs t, WeightSample ws) {
  if (ws.w && blockIdx.x == gridDim.x - 1) {
    choose_path(ws);
    return;
  }
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t* s_coef = (uint64_t*)smem_raw;
  const int ncoef = p.d * p.row_len;
  for (int i = threadIdx.x; i < ncoef; i += blockDim.x) s_coef[i] = p.coef[i];
  __syncthreads();
  const int64_t total = t.base[p.a];
  const int64_t step = (int64_t)(gridDim.x - (ws.w ? 1u : 0u)) * blockDim.x;
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total; g += step) {
    int u = 0;
    while (u + 1 < p.a && g >= t.base[u + 1]) u++;
    key_record<POW2, DEG1>(p, t, s_coef, u, (uint32_t)(g - t.base[u]), t.tbl + g * 4 * t.rvec);
  }
}

// Algorithm 2 through the key tables; scatter targets as in k_update.  The instances with
// 32-byte narrow records and a power-of-two width fit 48 registers without spills, which
// gives five CTAs per SM and more gathers in flight (star F update 5.63 -> 5.50 ms).
template <int A, bool POW2, bool SMEM, bool NARROW, bool V8>
__global__ void __launch_bounds__(256, (A > 0 && V8 && NARROW && POW2) ? 5 : 1) k_update_tab(UpdArgs p, TabArgs t) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int* s_sub = (int*)smem_raw;
  const int64_t dm = (int64_t)p.d * (int64_t)p.m;
  if (SMEM) {
    for (int64_t i = threadIdx.x; i < dm; i += blockDim.x) s_sub[i] = 0;
    __syncthreads();
  }
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p.n; i += step)
    update_tuple_tab<A, POW2, SMEM, NARROW, V8>(p, t, s_sub, i);
  if (SMEM) {
    __syncthreads();
    for (int64_t i = threadIdx.x; i < dm; i += blockDim.x) {
      const int v = s_sub[i];
      if (v != 0) atomicAdd(p.ctr + i, (unsigned long long)(int64_t)v);
    }
  }
}

// ---------------------------------------------------------------------------
// Partitioned update through the key tables (power-of-two 1024 <= m <= 2^16, d <= 14, at most 5
// attributes: the star fact table).  k_update_tab adds each (tuple, row)
// to the L2-resident int64 sketch with one 64-bit reduction, and the L2 lookup rate bounds it
// (9 reductions per tuple at d = 9, about half of them forwarded between the two dies' L2
// halves).  Shared-memory atomics run about ten times faster than L2 reductions on GB300,
// but a d x m int32 sketch of 9 x 2^16 does not fit in one SM.  So the update runs in two
// phases over windows of the batch.  Each row's bins are split into S = m / 2^L parts of
// 2^L bins, L = min(log2 m, 15), so S is 1 or 2.
//   1. k_tab_items: per tuple the key-table gathers and each row's bin sum and sign product
//      (Eqs. 2-3).  Each warp of this persistent kernel owns one region of C item slots per
//      row (C = 32 x its tile count) and appends its tiles' items there: the part-0 items
//      from the region's start upward, the part-1 items from its end downward (each item the
//      bin's offset within its part in bits 0..14 and the sign in bit 15).  At the end the warp
//      writes each row's part-0 count and its count of valid tuples.  A tuple with a key
//      outside its declared domain is left out (and reported, as in every other path).
//      Stores carry an L2 evict-first hint, so the items do not push the key tables' records
//      out of L2.
//   2. k_part_accum: a CTA owns part h of one row as 2^L int32 counters in shared memory
//      (at most 128 KB) over the regions of a range of phase-1 warps; its warps take pieces of
//      those regions, each lane 8 items (one 16-byte load) at a time, and add the signs with
//      shared-memory atomics, reading only part h's items; the CTA finally adds each counter
//      into the int64 sketch with one 64-bit reduction.
// Every counter receives the same sum as in k_update_tab (integer addition in any order);
// a CTA's int32 counter holds at most its range's tuple count in magnitude, kept below 2^31.
// Weighted batches take 32-bit items that carry Delta (2e7 turnstile tuples of five shuffled
// columns, m = 2^16, d = 9: 0.93 ms; 1.24 ms through k_update_tab).
//
// Records for this path (32 bytes, built by k_key_table_l20 for d <= 9): row r's bin in bits
// 20 (r mod 3) .. 20 (r mod 3) + 15 of 64-bit word r / 3 (words 0..2), the d sign bits in
// 32-bit word 7.  Summing the A <= 5 records word by word in 64 bits gives every row's exact
// bin sum (below A 2^16 < 2^20: no carry between lanes).  For 10 <= d <= 14 the narrow
// 16-bit records of k_key_table are used (row pairs summed as described at k_tab_items).
// ---------------------------------------------------------------------------
constexpr int kPartMaxCtasPerSm = 8;   // phase-1 CTAs of 256 threads per SM, at most

struct PartArgs {
  void* items;                   // phase-1 warp w, row j: region items + (w d + j) C, uint16_t each
  uint32_t* cnts;                // phase-1 warp w: [16 w + j] part-0 items of row j, [16 w + 15] valid tuples
  const int64_t* col[5];         // column u of the window's first tuple
  int64_t W;                     // window capacity, a multiple of 256
  int64_t cnt;                   // tuples in the window, <= W
  int64_t C;                     // item slots per (warp, row) region: 32 x tiles per warp
  int nwarps;                    // warps of the phase-1 grid
  int logL;                      // part width 2^L
  const uint32_t* vbits;         // nullptr, or bit (i mod 32) of word i / 32: window tuple i is kept
  const int64_t* wts;            // weighted: Delta of the window's first tuple (items are uint32_t)
  int64_t wmax;                  // weighted: |Delta| <= wmax < 2^16 goes into an item
  PartChoice* choice;            // weighted
  const int* go;                 // nullptr, or both phases return at once when it reads 0
};

__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t pol;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

__device__ __forceinline__ void st_u16_hint(uint16_t* ptr, uint16_t v, uint64_t pol) {
  asm volatile("st.global.L1::no_allocate.L2::cache_hint.u16 [%0], %1, %2;" ::"l"(ptr), "h"(v), "l"(pol) : "memory");
}

__device__ __forceinline__ void st_u32_hint(uint32_t* ptr, uint32_t v, uint64_t pol) {
  asm volatile("st.global.L1::no_allocate.L2::cache_hint.u32 [%0], %1, %2;" ::"l"(ptr), "r"(v), "l"(pol) : "memory");
}

__device__ __forceinline__ int64_t ld_key_policy(const int64_t* ptr, uint64_t pol) {
  int64_t v;
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.s64 %0, [%1], %2;" : "=l"(v) : "l"(ptr), "l"(pol));
  return v;
}

// Key-table records in the 20-bit lane format above (d <= 9, one thread per domain key).
template <bool DEG1>
__global__ void __launch_bounds__(256) k_key_table_l20(UpdArgs p, TabArgs t, WeightSample ws) {
  if (ws.w && blockIdx.x == gridDim.x - 1) {
    choose_path(ws);
    return;
  }
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t* s_coef = (uint64_t*)smem_raw;
  const int ncoef = p.d * p.row_len;
  for (int i = threadIdx.x; i < ncoef; i += blockDim.x) s_coef[i] = p.coef[i];
  __syncthreads();
  const int64_t total = t.base[p.a];
  const int64_t step = (int64_t)(gridDim.x - (ws.w ? 1u : 0u)) * blockDim.x;
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total; g += step) {
    int u = 0;
    while (u + 1 < p.a && g >= t.base[u + 1]) u++;
    const uint32_t x = (uint32_t)(g - t.base[u]);
    const uint64_t* cr = s_coef + t.off[u];
    uint64_t lane[3] = {0, 0, 0};
    uint32_t mask = 0;
#pragma unroll
    for (int r = 0; r < 9; r++) {
      if (r >= p.d) break;
      uint32_t par;
      const uint32_t b = key_row_hash<true, DEG1>(p, cr + (int64_t)r * p.row_len, p.deg[u], x, &par);
      lane[r / 3] |= (uint64_t)b << (20 * (r % 3));
      mask |= par << r;
    }
    uint4* out = (uint4*)(t.tbl + g * 8);
    out[0] = make_uint4((uint32_t)lane[0], (uint32_t)(lane[0] >> 32), (uint32_t)lane[1], (uint32_t)(lane[1] >> 32));
    out[1] = make_uint4((uint32_t)lane[2], (uint32_t)(lane[2] >> 32), 0u, mask);
  }
}

// What the kernels find out about a batch whose domains were not declared.
struct FoundDomains {
  unsigned long long top[5];   // the largest key of each attribute
  float spread[5];             // distinct keys among 1024 tuples of the batch, as a share
  float far;                   // of their weights, the share that no item holds
  int go;                      // the tables serve
  int blocks;                  // CTAs of the scan that are done
};

// Key-table records of 24 bytes (d <= 9, one thread per domain key): rows 3w .. 3w + 2 in
// 64-bit word w (w = 0, 1, 2), row r's lane at bit 22 (r mod 3): its bin (below 2^16) in the
// lane's bits 0..15 and its sign bit at lane bit 19.  Summing A <= 5 records word by word in
// 64 bits: the bins add up to below 5 2^16 < 2^19 in lane bits 0..18, so they never reach
// bit 19, and lane bit 19 of the sum is the parity of the signs (their sum, at most 5, fills
// lane bits 19..21; for the top lane, bits 63 and beyond, the carries leave the word).  So a
// row's bin sum mod m is (word >> 22 (r mod 3)) & (m - 1) and its sign product the bit above
// it at 19.  Five tables over 10^6 keys take 120 MB against 160 MB for 32-byte records, which
// keeps more of the Zipf tail in L2.  Record k (global index, 8-byte aligned) starts at 24 k:
// for even k its words 0 and 1 form the 16-byte-aligned pair and word 2 follows; for odd k
// the first 8 bytes hold word 2 and the aligned pair after it words 0 and 1, so a reader
// always takes words 0 and 1 with one 16-byte load and word 2 with one 8-byte load.
template <bool DEG1>
__global__ void __launch_bounds__(256) k_key_table_l24(UpdArgs p, TabArgs t, const FoundDomains* found,
                                                       WeightSample ws) {
  if (found && !found->go) return;
  if (ws.w && blockIdx.x == gridDim.x - 1) {
    choose_path(ws);
    return;
  }
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t* s_coef = (uint64_t*)smem_raw;
  const int ncoef = p.d * p.row_len;
  for (int i = threadIdx.x; i < ncoef; i += blockDim.x) s_coef[i] = p.coef[i];
  __syncthreads();
  // keys to hash: every declared domain, or [0, largest key] of each attribute as found
  int64_t total = t.base[p.a];
  if (found) {
    total = 0;
    for (int u = 0; u < p.a; u++) total += (int64_t)found->top[u] + 1;
  }
  const int64_t step = (int64_t)(gridDim.x - (ws.w ? 1u : 0u)) * blockDim.x;
  uint64_t* tbl = (uint64_t*)t.tbl;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += step) {
    int u = 0;
    int64_t g = i;
    if (found) {
      while (g > (int64_t)found->top[u]) g -= (int64_t)found->top[u++] + 1;
      g += t.base[u];
    } else {
      while (u + 1 < p.a && g >= t.base[u + 1]) u++;
    }
    const uint32_t x = (uint32_t)(g - t.base[u]);
    const uint64_t* cr = s_coef + t.off[u];
    uint64_t lane[3] = {0, 0, 0};
#pragma unroll
    for (int r = 0; r < 9; r++) {
      if (r >= p.d) break;
      uint32_t par;
      const uint32_t b = key_row_hash<true, DEG1>(p, cr + (int64_t)r * p.row_len, p.deg[u], x, &par);
      lane[r / 3] |= ((uint64_t)b | ((uint64_t)par << 19)) << (22 * (r % 3));
    }
    const bool odd = (g & 1) != 0;
    uint64_t* out = tbl + 3 * g;
    out[odd ? 1 : 0] = lane[0];
    out[odd ? 2 : 1] = lane[1];
    out[odd ? 0 : 2] = lane[2];
  }
}

// Words 0, 1 and 2 of 24-byte record k (layout above): one 16-byte and one 8-byte load.
__device__ __forceinline__ void ld_record24(const uint64_t* tbl, uint64_t k, uint64_t& w0, uint64_t& w1,
                                            uint64_t& w2) {
  const uint64_t odd = k & 1u;
  const uint64_t* r = tbl + 3 * k;
  asm("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(w0), "=l"(w1) : "l"(r + odd));
  asm("ld.global.nc.u64 %0, [%1];" : "=l"(w2) : "l"(r + 2 - 2 * odd));
}

// A weighted window's tuples straight to the int64 counters, from k_tab_items' records (FMT as
// there).  The grid has direct_ctas CTAs for each resident one: with resident CTAs alone, each with a
// fixed share, the SMs whose reductions take longest hold up the rest (2e7 tuples of five uniform
// columns, m = 2^16, d = 9: 1450 us, with four 1275 and with a CTA per 256 tuples 1250; the occupancy
// makes no difference, and claims from a counter wait behind the reductions).  Batches that have
// items pay for the CTAs that return at once, 1 us per 2000.
template <int A, int FMT>
__device__ __forceinline__ void add_direct(const UpdArgs& p, const TabArgs& t, const PartArgs& q) {
  const uint32_t mask = (uint32_t)p.m - 1u;
  const int d = p.d;
  const int64_t step = (int64_t)gridDim.x * 256;
  for (int64_t g = (int64_t)blockIdx.x * 256 + threadIdx.x; g < q.cnt; g += step) {
    int64_t key[A];
#pragma unroll
    for (int u = 0; u < A; u++) key[u] = ld_key_stream(q.col[u] + g);
    const int64_t delta = ld_key_stream(q.wts + g);
    bool ok = true;
#pragma unroll
    for (int u = 0; u < A; u++) ok = ok && (uint64_t)key[u] < (uint64_t)p.dom[u];
    if (!ok) {
      record(p.status, SK_ERR_KEY_OUT_OF_DOMAIN);
      continue;
    }
    auto put = [&](int j, uint32_t bin, bool neg) {
      red_add_global(p.ctr + (int64_t)j * p.m + (bin & mask), (unsigned long long)(neg ? -delta : delta));
    };
    if constexpr (FMT == 1) {
      uint32_t b2[7] = {0, 0, 0, 0, 0, 0, 0}, sg = 0;   // two rows per word, halves without carry
#pragma unroll
      for (int u = 0; u < A; u++) {
        uint32_t w[8];
        ld_record32((const uint4*)t.tbl + (uint64_t)(t.base[u] + key[u]) * 2, w);
        sg ^= w[7];
#pragma unroll
        for (int j = 0; j < 7; j++) b2[j] = add16x2(b2[j], w[j]);
      }
#pragma unroll
      for (int j = 0; j < 14; j++) {
        if (j >= d) break;
        put(j, b2[j >> 1] >> (16 * (j & 1)), (sg >> j) & 1u);
      }
    } else {
      constexpr int B = FMT == 2 ? 22 : 20;   // bits per row of a record word
      uint64_t acc[3] = {0, 0, 0};
      uint32_t sg = 0;
#pragma unroll
      for (int u = 0; u < A; u++) {
        if constexpr (FMT == 2) {
          uint64_t w0, w1, w2;
          ld_record24((const uint64_t*)t.tbl, (uint64_t)(t.base[u] + key[u]), w0, w1, w2);
          acc[0] += w0;
          acc[1] += w1;
          acc[2] += w2;
        } else {
          uint32_t w[8];
          ld_record32((const uint4*)t.tbl + (uint64_t)(t.base[u] + key[u]) * 2, w);
          acc[0] += ((uint64_t)w[1] << 32) | w[0];
          acc[1] += ((uint64_t)w[3] << 32) | w[2];
          acc[2] += ((uint64_t)w[5] << 32) | w[4];
          sg ^= w[7];
        }
      }
#pragma unroll
      for (int j = 0; j < 9; j++) {
        if (j >= d) break;
        const uint32_t x = (uint32_t)(acc[j / 3] >> (B * (j % 3)));
        put(j, x, FMT == 2 ? (x >> 19) & 1u : (sg >> j) & 1u);
      }
    }
  }
}

// FMT 0: 20-bit lane records (d <= 9); FMT 2: 24-byte records (d <= 9, k_key_table_l24);
// FMT 1: narrow 16-bit records of 32 bytes (d <= 14):
// per record word holding the bins of rows 2j and 2j + 1, lo[j] adds the low halves (below
// 5 * 2^16: no overflow) and all[j] the whole words mod 2^32, so row 2j's sum is lo[j] mod
// 2^16 and row 2j + 1's is ((all[j] - lo[j]) >> 16) mod 2^16 (m divides 2^16).
// Persistent: each thread walks the window with the grid's stride, loading the keys of its
// next tuple before it gathers the records of the current one, so the key stream's latency
// overlaps the gathers.  Lanes of a warp take consecutive tuples (one tile) and iterate
// together (the ballots need the whole warp).  Four CTAs per SM (64 registers): with the
// running counts five (48 registers) spilled and took the star's F update from 3.10 to 3.84 ms;
// six for the instances of one or two attributes (40 registers, no spills) took a sub-query
// family's update from 8.45 to 9.22 ms.
//
// A row costs one ballot, two population counts, a shuffle of its next slot and about 18
// instructions.  What bounds F of the star (5 attributes; 480 us per 2e7 tuples) is the gathers:
// alone, with nothing done to the records, they take 375 us (173 when every record hits L1; 32-byte
// records 362 and 205, 16-byte ones 231), through the texture path 446.  So the registers go to
// loads in flight: with every row's slot held in registers instead of shuffled the compiler
// splits the gathers and the star step takes 3.70 ms instead of 3.45.  The weighted kernel holds
// them all the same (HELD: 2e7 tuples 0.96 against 1.01 ms).  Item stores skip L1, which the
// records need.
//
// WT (weighted batches): items are 32 bits, the bin's offset in bits 0..14 and Delta times the
// sign above; a tuple with |Delta| > wmax goes to the int64 counters directly, and every tuple
// does when the batch's sample says that most have such weights (choose_path, add_direct).
template <int A, int FMT, bool WT>
__global__ void __launch_bounds__(256, 4) k_tab_items(UpdArgs p, TabArgs t, PartArgs q) {
  if (q.go && !*q.go) return;
  const bool direct = WT && q.choice->direct != 0;
  if (WT && (int)blockIdx.x * 8 >= q.nwarps && !direct) return;   // a CTA for add_direct only
  using Item = typename std::conditional<WT, uint32_t, uint16_t>::type;
  constexpr bool HELD = WT && FMT != 1;
  const int64_t step = WT ? (int64_t)q.nwarps * 32 : (int64_t)gridDim.x * blockDim.x;
  const int64_t gend = (q.cnt + 31) & ~(int64_t)31;
  const uint32_t mask = (uint32_t)p.m - 1u;
  const uint32_t low = (1u << q.logL) - 1u;
  const uint32_t half = mask & ~low;   // the bin bit that tells part 1 (0: one part)
  const unsigned lane = threadIdx.x & 31u;
  const uint32_t lt = (1u << lane) - 1u;
  const int d = p.d;
  const uint64_t pol = policy_evict_first();
  const uint4* tbl = (const uint4*)t.tbl;
  int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t C = (uint32_t)q.C;
  Item* const mine = (Item*)q.items + (g >> 5) * d * q.C;   // this warp's regions, row j's at j C
  uint32_t nval = 0;    // valid tuples so far
  uint32_t cw = lane * C;   // lane j < d: row j's next part-0 slot, j C + its part-0 items
  uint32_t o0[9];           // HELD: the same for every row
#pragma unroll
  for (int j = 0; j < 9; j++) o0[j] = (uint32_t)j * C;
  // keys of the thread's next tuple, checked against their domains as they arrive: the
  // in-domain keys (< 2^31) as 32-bit values, bit u of okm set when key u is in its domain
  uint32_t kx[A], okm = 0;
  int64_t wn = 0;
#pragma unroll
  for (int u = 0; u < A; u++) {
    const int64_t k = g < q.cnt ? ld_key_policy(q.col[u] + g, pol) : -1;
    const bool kin = (uint64_t)k < (uint64_t)p.dom[u];
    okm |= (uint32_t)kin << u;
    kx[u] = kin ? (uint32_t)k : 0u;
  }
  if (WT && g < q.cnt) wn = ld_key_policy(q.wts + g, pol);
  if constexpr (WT) {
    if (direct) {   // asked after the first keys' loads: the answer arrives with them
      add_direct<A, FMT>(p, t, q);
      return;
    }
  }
  for (; g < gend; g += step) {
    const bool in = g < q.cnt;
    const bool whole = in && okm == (1u << A) - 1u && (!q.vbits || ((q.vbits[g >> 5] >> lane) & 1u));
    const int64_t delta = wn;
    const bool ok = whole && (!WT || (delta <= q.wmax && delta >= -q.wmax));
    uint32_t kg[A];   // global record indices (the host keeps this path's tables below 2^32 records)
#pragma unroll
    for (int u = 0; u < A; u++) kg[u] = (uint32_t)t.base[u] + kx[u];
    if (in && !whole) record(p.status, SK_ERR_KEY_OUT_OF_DOMAIN);   // left out of the tile below
    const int64_t gn = g + step;
    okm = 0;
#pragma unroll
    for (int u = 0; u < A; u++) {
      const int64_t k = gn < q.cnt ? ld_key_policy(q.col[u] + gn, pol) : -1;
      const bool kin = (uint64_t)k < (uint64_t)p.dom[u];
      okm |= (uint32_t)kin << u;
      kx[u] = kin ? (uint32_t)k : 0u;
    }
    if (WT && gn < q.cnt) wn = ld_key_policy(q.wts + gn, pol);
    const uint32_t vb = __ballot_sync(0xffffffffu, ok);
    const uint32_t nv = __popc(vb), rv = __popc(vb & lt);   // valid tuples in the tile / before this lane
    const uint32_t end1 = C - 1u - nval;   // a row's next part-1 slot is end1 past its next part-0 slot
    uint32_t add = 0;   // this tile's part-0 items of row `lane`
    // one row, x = its bin sum (bits above the bin arbitrary, 0 for a tuple left out): with r1
    // the part-1 tuples before this lane, a part-0 tuple goes to slot (part-0 items so far) +
    // rv - r1 and a part-1 one to C - 1 - (part-1 items so far) - r1
    auto put = [&](int j, uint32_t x, uint32_t neg15) {
      const bool hi = (x & half) != 0u;
      const uint32_t hb = __ballot_sync(0xffffffffu, hi);
      const uint32_t r1 = __popc(hb & lt);
      const uint32_t at = (HELD ? o0[j] : __shfl_sync(0xffffffffu, cw, j)) + (hi ? end1 : rv) - r1;
      if (WT) {
        const int32_t v = neg15 ? -(int32_t)delta : (int32_t)delta;
        if (ok) st_u32_hint((uint32_t*)mine + at, (x & low) | ((uint32_t)v << 15), pol);
      } else if (ok) {
        st_u16_hint((uint16_t*)mine + at, (uint16_t)((x & low) | neg15), pol);
      }
      if (HELD) o0[j] += nv - __popc(hb);
      else if (lane == (unsigned)j) add = nv - __popc(hb);
    };
    // a weighted tuple beyond wmax: straight to the counters
    auto far = [&](int j, uint32_t x, uint32_t neg15) {
      red_add_global(p.ctr + (int64_t)j * p.m + (x & mask), (unsigned long long)(neg15 ? -delta : delta));
    };
    uint32_t sg = 0;
    if (FMT == 0) {
      uint64_t acc[3] = {0, 0, 0};
      if (whole) {
#pragma unroll
        for (int u = 0; u < A; u++) {
          uint32_t w[8];
          ld_record32(tbl + (uint64_t)kg[u] * 2, w);
          acc[0] += ((uint64_t)w[1] << 32) | w[0];
          acc[1] += ((uint64_t)w[3] << 32) | w[2];
          acc[2] += ((uint64_t)w[5] << 32) | w[4];
          sg ^= w[7];
        }
      }
      if (WT && whole && !ok) {
#pragma unroll
        for (int j = 0; j < 9; j++) {
          if (j >= d) break;
          far(j, (uint32_t)(acc[j / 3] >> (20 * (j % 3))), ((sg >> j) & 1u) << 15);
        }
        acc[0] = acc[1] = acc[2] = 0;
      }
#pragma unroll
      for (int j = 0; j < 9; j++) {
        if (j >= d) break;
        put(j, (uint32_t)(acc[j / 3] >> (20 * (j % 3))), ((sg >> j) & 1u) << 15);
      }
    } else if (FMT == 2) {
      uint64_t acc[3] = {0, 0, 0};
      if (whole) {
#pragma unroll
        for (int u = 0; u < A; u++) {
          uint64_t w0, w1, w2;
          ld_record24((const uint64_t*)t.tbl, kg[u], w0, w1, w2);
          acc[0] += w0;
          acc[1] += w1;
          acc[2] += w2;
        }
      }
      if (WT && whole && !ok) {
#pragma unroll
        for (int j = 0; j < 9; j++) {
          if (j >= d) break;
          const uint32_t x = (uint32_t)(acc[j / 3] >> (22 * (j % 3)));
          far(j, x, (x >> 4) & 0x8000u);
        }
        acc[0] = acc[1] = acc[2] = 0;
      }
#pragma unroll
      for (int j = 0; j < 9; j++) {
        if (j >= d) break;
        const uint32_t x = (uint32_t)(acc[j / 3] >> (22 * (j % 3)));
        put(j, x, (x >> 4) & 0x8000u);   // the sign is lane bit 19
      }
    } else {
      uint32_t lo[7], all[7];
#pragma unroll
      for (int j = 0; j < 7; j++) lo[j] = all[j] = 0;
      if (whole) {
#pragma unroll
        for (int u = 0; u < A; u++) {
          uint32_t w[8];
          ld_record32(tbl + (uint64_t)kg[u] * 2, w);
          sg ^= w[7];
#pragma unroll
          for (int j = 0; j < 7; j++) {
            lo[j] += w[j] & 0xffffu;
            all[j] += w[j];
          }
        }
      }
#pragma unroll
      for (int j = 0; j < 14; j++) {
        if (j >= d) break;
        uint32_t x = (j & 1) ? (all[j >> 1] - lo[j >> 1]) >> 16 : lo[j >> 1];
        const uint32_t neg15 = ((sg >> j) & 1u) << 15;
        if (WT && !ok) {
          if (whole) far(j, x, neg15);
          x = 0;
        }
        put(j, x, neg15);
      }
    }
    cw += add;   // after the rows: their shuffles all read the slots before the tile
    nval += nv;
  }
  // the warp's counts: lane j < d row j's part-0 items, lane 15 the valid tuples
  const int64_t wg = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (HELD) {
#pragma unroll
    for (int j = 0; j < 9; j++)
      if (lane == (unsigned)j) cw = o0[j];
  }
  if (lane < (unsigned)d || lane == 15u) q.cnts[wg * 16 + lane] = lane == 15u ? nval : cw - lane * C;
}

// shared counter at saddr += v when x < n (unsigned): one compare, one predicated reduction
__device__ __forceinline__ void red_shared_if_lt(uint32_t saddr, int v, uint32_t x, uint32_t n) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.lt.u32 q, %2, %3;\n\t@q red.shared.add.s32 [%0], %1;\n\t}"
               ::"r"(saddr), "r"(v), "r"(x), "r"(n) : "memory");
}

// shared counter at saddr += v when x != 0
__device__ __forceinline__ void red_shared_if_set(uint32_t saddr, int v, uint32_t x) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q red.shared.add.s32 [%0], %1;\n\t}"
               ::"r"(saddr), "r"(v), "r"(x) : "memory");
}

__device__ __forceinline__ void red_shared(uint32_t saddr, int v) {
  asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(saddr), "r"(v) : "memory");
}

// The 8 items of one 16-byte chunk (two per 32-bit word: bin offset in bits 0..14, sign in
// bit 15) added into the shared counters at sbase; slots b .. b + 7 counted from the run's
// first item, those at or beyond n skipped.  A chunk wholly inside the run (every chunk but
// a run's first and last) goes without the per-slot compare.
__device__ __forceinline__ void add_chunk(uint32_t sbase, uint4 v, uint32_t b, uint32_t n) {
  const uint32_t e[4] = {v.x, v.y, v.z, v.w};
  if (n >= 8u && b <= n - 8u) {
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t it = e[k >> 1] >> (16 * (k & 1));
      int neg;   // 0 or -1 from the item's sign bit
      asm("bfe.s32 %0, %1, 15, 1;" : "=r"(neg) : "r"(it));
      red_shared(sbase + ((it & 0x7fffu) << 2), neg | 1);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t it = e[k >> 1] >> (16 * (k & 1));
      int neg;
      asm("bfe.s32 %0, %1, 15, 1;" : "=r"(neg) : "r"(it));
      red_shared_if_lt(sbase + ((it & 0x7fffu) << 2), neg | 1, b + (uint32_t)k, n);
    }
  }
}

// The same for the 4 items of a weighted chunk (bin offset in bits 0..14, signed value above).
__device__ __forceinline__ void add_chunk_weighted(uint32_t sbase, uint4 v, uint32_t b, uint32_t n) {
  const uint32_t e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int k = 0; k < 4; k++)
    red_shared_if_lt(sbase + ((e[k] & 0x7fffu) << 2), (int)e[k] >> 15, b + (uint32_t)k, n);
}

// blockIdx.x = h + S (row + d c), S = m >> logL: part h of row `row` over the regions of the
// phase-1 warps [c R, min(c R + R, nwarps)), each region's part-h chunks (8 items, one 16-byte
// load) split into 2^logP pieces.  Warp k of the CTA takes pieces k, k + 32, ...; lane l of a
// warp takes the piece's chunks l, l + 32, ..., two per iteration, loads first.
template <bool WT>
__global__ void __launch_bounds__(1024) k_part_accum(PartArgs q, unsigned long long* ctr, int64_t m, int d,
                                                     int logL, int R, int logP) {
  constexpr int LI = WT ? 2 : 3, I = 1 << LI;   // items per 16-byte chunk
  if (q.go && !*q.go) return;
  if (WT && q.choice->direct) return;   // no items
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int* cnt = (int*)smem_raw;
  const int S = (int)(m >> logL);
  const int h = (int)(blockIdx.x % (unsigned)S);
  const int rest = (int)(blockIdx.x / (unsigned)S);
  const int row = rest % d;
  const int c = rest / d;
  const int L = 1 << logL;
  for (int k = threadIdx.x; k < L; k += blockDim.x) cnt[k] = 0;
  __syncthreads();
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(cnt);
  const uint32_t lane = threadIdx.x & 31u;
  const int w0 = c * R;
  const int w1 = min(w0 + R, q.nwarps);
  const int npc = (w1 - w0) << logP;
  const uint32_t C = (uint32_t)q.C;
  // slots b .. b + I - 1 counted from the part's first item: add those below n
  auto unit = [&](uint4 v, uint32_t b, uint32_t n) {
    if (WT) add_chunk_weighted(sbase, v, b, n);
    else add_chunk(sbase, v, b, n);
  };
  for (int pc = (int)(threadIdx.x >> 5); pc < npc; pc += (int)(blockDim.x >> 5)) {
    const int w = w0 + (pc >> logP);
    const uint32_t piece = (uint32_t)pc & ((1u << logP) - 1u);
    const uint32_t n0 = q.cnts[(int64_t)w * 16 + row], nv = q.cnts[(int64_t)w * 16 + 15];
    const uint32_t n = h ? nv - n0 : n0;         // part h's items in this region
    const uint32_t lo = h ? C - n : 0u;          // and the first of them
    const uint32_t kb = lo >> LI, nk = ((lo + n + I - 1) >> LI) - kb;
    const uint32_t ke = kb + (uint32_t)(((uint64_t)nk * (piece + 1)) >> logP);
    uint32_t k = kb + (uint32_t)(((uint64_t)nk * piece) >> logP) + lane;
    const uint4* rg = (const uint4*)q.items + (((int64_t)w * d + row) * q.C >> LI);
    // two chunks per iteration, the next two in flight during their additions
    const uint4 none = make_uint4(0u, 0u, 0u, 0u);
    uint4 v1 = k < ke ? rg[k] : none, v2 = k + 32 < ke ? rg[k + 32] : none;
    for (; k + 32 < ke; k += 64) {
      const uint4 c1 = v1, c2 = v2;
      if (k + 64 < ke) v1 = rg[k + 64];
      if (k + 96 < ke) v2 = rg[k + 96];
      unit(c1, I * k - lo, n);
      unit(c2, I * (k + 32) - lo, n);
    }
    if (k < ke) unit(v1, I * k - lo, n);
  }
  __syncthreads();
  unsigned long long* out = ctr + (int64_t)row * m + ((int64_t)h << logL);
  for (int k = threadIdx.x; k < L; k += blockDim.x) {
    const int v = cnt[k];
    if (v != 0) red_add_global(out + k, (unsigned long long)(int64_t)v);
  }
}

// All views of a sub-query family's relation (24-byte records, unit weights).  A view's bin is the
// sum of its attributes' bins, so the views need no items of their own:
//   1. k_view_planes gathers a tuple's A records once and leaves, for every row and attribute, the
//      16-bit bins and one sign bit per tuple in planes over the window's tuples, and one bit per
//      tuple that all its keys are inside their domains (others are left out of every view);
//   2. k_view_accum: a CTA owns a part (at most 2^15 bins) of one view's row as int32 counters in
//      shared memory; a thread loads the same eight tuples of each of the view's attributes (16
//      bytes and one of signs), adds the bins two to a word and adds the eight signs of those
//      whose bin is in the part.
// Nine rows of 15 views of a 4-attribute relation, 2e7 tuples, m = 2^16: k_view_planes 0.64 ms (70 % of
// the L1 data pipe: four gathers and 36 stores per tuple), k_view_accum 3.14 ms (issue 86 %, about 18
// instructions per tuple, view, row and part; 1.5 GB of planes against 5.4 GB of items).  With items
// written per view (k_tab_items' partition for every view at once) the two phases took 7.1 ms.
struct ViewMasks {
  int nv;
  uint8_t mask[SK_MAX_VIEWS];   // bit u: the view joins attribute u
};

// The planes of a window are cut into tiles of kViewTile tuples, [tile][bins d a | signs d a | kept]:
// a CTA's stores stay within one tile (with planes over the whole window they went to 76 pages
// at a time and k_view_planes took 1.30 ms instead of 0.64).
constexpr int kViewTile = 8192;   // a chunk of eight tuples for each of k_view_accum's threads

struct ViewPlanes {
  uint8_t* tiles;
  int64_t stride;          // bytes per tile
  const int64_t* col[5];   // column u of the window's first tuple
  int64_t cnt;             // tuples in this window
};

struct ViewCounters {
  unsigned long long* ctr[SK_MAX_VIEWS];   // [d][m] each
};

template <int A>
__global__ void __launch_bounds__(256, A <= 4 ? 4 : 3) k_view_planes(UpdArgs p, TabArgs t, ViewPlanes q) {
  const int64_t step = (int64_t)gridDim.x * 256;
  const int64_t gend = (q.cnt + 31) & ~(int64_t)31;
  const unsigned lane = threadIdx.x & 31u;
  const int d = p.d;
  const uint64_t pol = policy_evict_first();
  int64_t g = (int64_t)blockIdx.x * 256 + threadIdx.x;
  uint32_t kx[A], okm = 0;   // the thread's next tuple, see k_tab_items
#pragma unroll
  for (int u = 0; u < A; u++) {
    const int64_t k = g < q.cnt ? ld_key_policy(q.col[u] + g, pol) : -1;
    const bool kin = (uint64_t)k < (uint64_t)p.dom[u];
    okm |= (uint32_t)kin << u;
    kx[u] = kin ? (uint32_t)k : 0u;
  }
  for (; g < gend; g += step) {
    const bool in = g < q.cnt;
    const bool ok = in && okm == (1u << A) - 1u;
    if (in && !ok) record(p.status, SK_ERR_KEY_OUT_OF_DOMAIN);
    uint64_t rec[A][3];
#pragma unroll
    for (int u = 0; u < A; u++) {
      rec[u][0] = rec[u][1] = rec[u][2] = 0;
      if (ok) ld_record24((const uint64_t*)t.tbl, (uint32_t)t.base[u] + kx[u], rec[u][0], rec[u][1], rec[u][2]);
    }
    const int64_t gn = g + step;
    okm = 0;
#pragma unroll
    for (int u = 0; u < A; u++) {
      const int64_t k = gn < q.cnt ? ld_key_policy(q.col[u] + gn, pol) : -1;
      const bool kin = (uint64_t)k < (uint64_t)p.dom[u];
      okm |= (uint32_t)kin << u;
      kx[u] = kin ? (uint32_t)k : 0u;
    }
    const uint32_t kept = __ballot_sync(0xffffffffu, ok);
    const uint32_t at = (uint32_t)g & (kViewTile - 1u);
    uint8_t* const tile = q.tiles + (g / kViewTile) * q.stride;
    uint16_t* const bins = (uint16_t*)tile + at;
    uint32_t* const bits = (uint32_t*)(tile + (size_t)d * A * kViewTile * 2) + (at >> 5);
    if (lane == 0) bits[d * A * (kViewTile / 32)] = kept;
    uint32_t sb[2] = {0, 0};   // lane l: the sign bits of plane l, of plane 32 + l
#pragma unroll
    for (int j = 0; j < 9; j++) {
      if (j >= d) break;
#pragma unroll
      for (int u = 0; u < A; u++) {
        const uint32_t x = (uint32_t)(rec[u][j / 3] >> (22 * (j % 3)));   // sign: bit 19
        st_u16_hint(bins + (j * A + u) * kViewTile, (uint16_t)x, pol);
        const uint32_t b = __ballot_sync(0xffffffffu, (x & 0x80000u) != 0u);
        if (lane == (unsigned)((j * A + u) & 31)) sb[(j * A + u) >> 5] = b;
      }
    }
    if (lane < (unsigned)(d * A)) bits[lane * (kViewTile / 32)] = sb[0];
    if (A * 9 > 32 && lane + 32u < (unsigned)(d * A)) bits[(lane + 32u) * (kViewTile / 32)] = sb[1];
  }
}

// The top bit of byte k of w over a whole word: 0 or -1.
__device__ __forceinline__ int byte_sign(uint32_t w, int k) {
  int r;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(w), "r"(0x1111u * (8u + (uint32_t)k)));
  return r;
}

// shared counter at saddr += v unless (w ^ flip) has the bit
__device__ __forceinline__ void red_shared_unless(uint32_t saddr, int v, uint32_t w, uint32_t flip, uint32_t bit) {
  asm volatile("{\n\t.reg .pred q;\n\t.reg .b32 t;\n\txor.b32 t, %2, %3;\n\tand.b32 t, t, %4;\n\t"
               "setp.eq.u32 q, t, 0;\n\t@q red.shared.add.s32 [%0], %1;\n\t}"
               ::"r"(saddr), "r"(v), "r"(w), "r"(flip), "r"(bit) : "memory");
}

// Eight tuples: bins in the low halves of lo and the high halves of hi, sign bits sg; of two parts
// (TWO) those whose top bin bit is the part's; !ALL: bits of keep clear are left out.  The reductions
// are predicated: with every lane adding, zero or to a spare word of its own where the bin is the
// other part's, a tuple takes a quarter fewer instructions, but hot counters queue in both parts'
// CTAs (4-attribute relation, 2e7 tuples: 3.40 ms, predicated 3.14).
template <bool TWO, bool ALL>
__device__ __forceinline__ void add_view_chunk(uint32_t sbase, const uint32_t (&lo)[4], const uint32_t (&hi)[4],
                                               uint32_t sg, uint32_t keep, uint32_t low, uint32_t flip) {
  // bits 0..3 and 4..7 of the signs at the tops of four bytes (the four products do not overlap)
  constexpr uint32_t kSpread = (1u << 7) | (1u << 14) | (1u << 21) | (1u << 28);
  const uint32_t s0 = (sg & 15u) * kSpread, s1 = (sg >> 4) * kSpread;
#pragma unroll
  for (int k = 0; k < 8; k++) {
    const uint32_t w = (k & 1) ? hi[k >> 1] : lo[k >> 1];
    const uint32_t at = sbase + ((k & 1) ? (w & (low << 16)) >> 14 : (w & low) << 2);
    int v = byte_sign(k < 4 ? s0 : s1, k & 3) | 1;
    if (!ALL && !(keep & (1u << k))) v = 0;
    if (TWO) red_shared_unless(at, v, w, flip, (k & 1) ? 0x80000000u : 0x8000u);
    else red_shared(at, v);
  }
}

template <int C, bool TWO>
__device__ __forceinline__ void view_accum_tiles(const ViewPlanes& q, uint32_t am, int A, int d, int row, uint32_t sbase,
                                                 uint32_t low, uint32_t flip, int t0, int t1) {
  // this thread's chunk in the tile: bins at 16 bytes per chunk, signs and kept at one
  const uint8_t* tile = q.tiles + t0 * q.stride;
  uint32_t plane[C];
#pragma unroll
  for (int i = 0; i < C; i++) {
    plane[i] = (uint32_t)(row * A + __ffs(am) - 1);
    am &= am - 1u;
  }
  const uint32_t signs0 = (uint32_t)(d * A) * (kViewTile * 2) + threadIdx.x;
  uint4 nb[C];
  uint32_t ns[C], nk = 0;
  auto load = [&](const uint8_t* at) {
#pragma unroll
    for (int i = 0; i < C; i++) {
      nb[i] = __ldg((const uint4*)(at + plane[i] * (kViewTile * 2)) + threadIdx.x);
      ns[i] = __ldg(at + signs0 + plane[i] * (kViewTile / 8));
    }
    nk = __ldg(at + signs0 + (uint32_t)(d * A) * (kViewTile / 8));
  };
  // chunks of the last tile that hold tuples
  const int last = (int)((q.cnt - (int64_t)(t1 - 1) * kViewTile + 7) >> 3);
  if (t1 - 1 > t0 || (int)threadIdx.x < last) load(tile);
  for (int t = t0; t < t1; t++) {
    if (t + 1 == t1 && (int)threadIdx.x >= last) break;
    uint32_t lo[4] = {nb[0].x, nb[0].y, nb[0].z, nb[0].w};
    uint32_t hi[4] = {nb[0].x, nb[0].y, nb[0].z, nb[0].w};
    uint32_t sg = ns[0];
    const uint32_t keep = nk;
    // low halves: a plain sum; high halves: no carry comes up from masked words
#pragma unroll
    for (int i = 1; i < C; i++) {
      const uint32_t w[4] = {nb[i].x, nb[i].y, nb[i].z, nb[i].w};
#pragma unroll
      for (int k = 0; k < 4; k++) {
        lo[k] += w[k];
        hi[k] += w[k] & 0xffff0000u;
      }
      sg ^= ns[i];
    }
    tile += q.stride;
    if (t + 2 < t1 || (t + 2 == t1 && (int)threadIdx.x < last)) load(tile);   // in flight during the additions
    if (keep == 0xffu) add_view_chunk<TWO, true>(sbase, lo, hi, sg, keep, low, flip);
    else add_view_chunk<TWO, false>(sbase, lo, hi, sg, keep, low, flip);
  }
}

// blockIdx.x = part + S (view + nv (row + d range)): the CTAs that run together read the planes
// of a few rows.
template <bool TWO>
__global__ void __launch_bounds__(1024) k_view_accum(ViewPlanes q, const __grid_constant__ ViewMasks vm,
                                                     const __grid_constant__ ViewCounters vc, int A, int d, int64_t m,
                                                     int logL, int nr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int* cnt = (int*)smem_raw;
  constexpr int S = TWO ? 2 : 1;
  const int L = 1 << logL;
  unsigned b = blockIdx.x;
  const int part = (int)(b % (unsigned)S);
  b /= (unsigned)S;
  const int v = (int)(b % (unsigned)vm.nv);
  b /= (unsigned)vm.nv;
  const int row = (int)(b % (unsigned)d), range = (int)(b / (unsigned)d);
  for (int k = threadIdx.x; k < L / 4; k += 1024) ((int4*)cnt)[k] = make_int4(0, 0, 0, 0);
  __syncthreads();
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(cnt);
  const int64_t nt = (q.cnt + kViewTile - 1) / kViewTile;
  const int t0 = (int)(nt * range / nr), t1 = (int)(nt * (range + 1) / nr);
  const uint32_t low = (uint32_t)(L - 1);
  const uint32_t flip = part ? 0x80008000u : 0u;
  const uint32_t am = vm.mask[v];
  switch (__popc(am)) {
    case 1: view_accum_tiles<1, TWO>(q, am, A, d, row, sbase, low, flip, t0, t1); break;
    case 2: view_accum_tiles<2, TWO>(q, am, A, d, row, sbase, low, flip, t0, t1); break;
    case 3: view_accum_tiles<3, TWO>(q, am, A, d, row, sbase, low, flip, t0, t1); break;
    case 4: view_accum_tiles<4, TWO>(q, am, A, d, row, sbase, low, flip, t0, t1); break;
    default: view_accum_tiles<5, TWO>(q, am, A, d, row, sbase, low, flip, t0, t1); break;
  }
  __syncthreads();
  unsigned long long* out = vc.ctr[v] + (int64_t)row * m + ((int64_t)part << logL);
  for (int x = threadIdx.x; x < L; x += 1024) {
    const int s = cnt[x];
    if (s != 0) red_add_global(out + x, (unsigned long long)(int64_t)s);
  }
}

using TabItemsKernel = void (*)(UpdArgs, TabArgs, PartArgs);

template <int FMT, bool WT>
TabItemsKernel tab_items_of(int A) {
  switch (A) {
    case 1: return k_tab_items<1, FMT, WT>;
    case 2: return k_tab_items<2, FMT, WT>;
    case 3: return k_tab_items<3, FMT, WT>;
    case 4: return k_tab_items<4, FMT, WT>;
    default: return k_tab_items<5, FMT, WT>;
  }
}

TabItemsKernel tab_items_kernel(int A, int fmt, bool weighted) {
  if (weighted) return fmt == 0 ? tab_items_of<0, true>(A) : (fmt == 2 ? tab_items_of<2, true>(A) : tab_items_of<1, true>(A));
  return fmt == 0 ? tab_items_of<0, false>(A) : (fmt == 2 ? tab_items_of<2, false>(A) : tab_items_of<1, false>(A));
}

// CTAs of a phase-1 kernel per SM (no shared memory: the whole unified array is left to L1,
// which caches the hot records).
cudaError_t tab_items_per_sm(TabItemsKernel kern, int* per_sm) {
  cudaError_t e = cudaFuncSetAttribute((const void*)kern, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kern, 256, 0);
  *per_sm = std::max(1, std::min(*per_sm, kPartMaxCtasPerSm));
  return e;
}

// Phase-2 split of nwarps regions (`units` (row, part) pairs, `slots` resident CTAs): the number
// of ranges of regions per pair.  A wave of CTAs costs its share of the items plus a fixed
// zeroing and flush of 2^15 counters (about 9 us on a GB300 SM, as long as 125 000 items take),
// so few waves.  uneven: by how much the longest CTAs' shares exceed the others': where one key's
// items queue at one counter, the part that holds it takes longer, and only more and smaller CTAs spread it.
int64_t part_ranges(int64_t items, int64_t units, int64_t slots, int64_t nwarps, double uneven) {
  double best = 0.0;
  int64_t nr = 1;
  // The star's 18 pairs take one wave of 144 CTAs (star step 3.41 ms, with at least two waves 3.43;
  // 2e7 weighted tuples 0.931 and 0.944 ms); nine waves of 1368 CTAs flushed 45e6 counters (phase
  // 2 162 us per 2e7 tuples, now about 110).
  for (int64_t k = 1; k <= 16; k++) {
    const int64_t r = std::max<int64_t>(1, k * slots / units);
    const double waves = std::ceil((double)(r * units) / (double)slots);
    const double share = (double)items / (double)(r * units);
    const double cost = waves * (share + 125000.0) + uneven * share;
    if (best == 0.0 || cost < best) {
      best = cost;
      nr = r;
    }
  }
  return std::max<int64_t>(1, std::min<int64_t>(nr, nwarps));
}

// SK_UNDECLARED_LEAST: the fewest tuples for which update_undeclared looks for dense keys; given, it
// takes the tables for them whatever they gain.
int64_t undeclared_least() {
  const char* v = std::getenv("SK_UNDECLARED_LEAST");
  const long long x = v ? std::atoll(v) : 0;
  return x > 0 ? (int64_t)x : (int64_t)1 << 22;
}

bool undeclared_least_given() {
  const char* v = std::getenv("SK_UNDECLARED_LEAST");
  return v && std::atoll(v) > 0;
}

// SK_PART_UPDATE=0 keeps the single-phase k_update_tab (and the per-tuple update) for batches
// the partitioned updates could take; =2 gives the wide partitioned update every batch whose
// width, rows, arity and weights it accepts, whatever the sketch's size and the batch length.
// SK_PART_WINDOW caps the tuples per window (default and largest: 2^30, which keeps every
// shared-memory counter of k_part_accum below 2^31 in magnitude; 2^24 for the wide update).
int part_update_mode() {
  const char* v = std::getenv("SK_PART_UPDATE");
  return (v && v[0] == '0') ? 0 : ((v && v[0] == '2') ? 2 : 1);
}

// SK_PART_RECORD=32 takes the 32-byte 20-bit lane records instead of the 24-byte ones for d <= 9.
int part_record_bytes() {
  const char* v = std::getenv("SK_PART_RECORD");
  return (v && std::atoi(v) == 32) ? 32 : 24;
}

int64_t part_window(int64_t n, int64_t most = (int64_t)1 << 30) {
  const char* v = std::getenv("SK_PART_WINDOW");
  const long long x = v ? std::atoll(v) : 0;
  const int64_t cap = (x > 0 && x < most) ? (int64_t)x : most;
  return std::min<int64_t>((n + 255) / 256 * 256, (cap + 255) / 256 * 256);
}

// Tuples per window: weighted items take twice the bytes, and staging beyond what the library's
// pool keeps (4 GiB) would be mapped again for every call.
int64_t part_most(const int64_t* weights) { return (int64_t)1 << (weights ? 26 : 30); }

// Regions of a window of W tuples: the phase-1 grid has at most sms x kPartMaxCtasPerSm CTAs
// of 256 threads, so its warps' regions hold at most W + that many threads' tiles per row.
size_t part_items_bytes(int d, int64_t W, int sms, bool weighted) {
  const int64_t threads = (int64_t)sms * kPartMaxCtasPerSm * 256;
  return ((size_t)d * (size_t)(W + threads) * (weighted ? sizeof(uint32_t) : sizeof(uint16_t)) + 255) & ~(size_t)255;
}

size_t part_counts_bytes(int sms) { return (size_t)sms * kPartMaxCtasPerSm * 8 * 16 * sizeof(uint32_t); }

// Items, the warps' counts, and for weighted batches a PartChoice.
size_t part_staging_bytes(int d, int64_t W, int sms, bool weighted = false) {
  return part_items_bytes(d, W, sms, weighted) + part_counts_bytes(sms) + (weighted ? 256 : 0);
}

// Phase 2 over the regions of a window: R and the pieces per region follow from part_ranges.
struct PartSplit {
  int64_t nr;   // ranges per (row, part)
  int R;        // regions per range
  int logP;     // pieces per region, log2: a CTA's 32 warps get equal shares, a lane of each a chunk or more
};

// chunks: of 16 bytes, a region has for one part about.  Pieces of fewer chunks than a warp has lanes
// only idle them (2^20 tuples, m = 2^16, d = 3, 13 chunks: four pieces 66 us, whole 60).
PartSplit part_split(int64_t items, int64_t units, int64_t slots, int nwarps, int64_t chunks, double uneven) {
  PartSplit p;
  p.nr = part_ranges(items, units, slots, nwarps, uneven);
  p.R = (int)((nwarps + p.nr - 1) / p.nr);
  p.nr = (nwarps + p.R - 1) / p.R;
  int most = 0;
  while (most < 5 && (chunks >> (most + 1)) >= 32) most++;
  p.logP = most;
  for (int lp = 0; lp < most; lp++) {
    const int64_t pcs = (int64_t)p.R << lp;
    if ((pcs + 31) / 32 * 32 * 100 <= pcs * 105) {
      p.logP = lp;
      break;
    }
  }
  return p;
}

// The kernels and the launch shape of both phases for one relation.
struct PartPlan {
  TabItemsKernel items;
  void (*accum)(PartArgs, unsigned long long*, int64_t, int, int, int, int);
  int attrs;
  bool weighted;
  int64_t W;           // tuples per window
  int64_t full_grid;   // phase-1 CTAs, all resident
  int64_t units;       // (row, part) pairs
  int64_t slots;       // resident phase-2 CTAs
  int logL;
  size_t smem;
};

cudaError_t part_plan(const UpdArgs& a, int fmt, int sms, int64_t most, PartPlan* pl) {
  const bool weighted = a.w != nullptr;
  pl->items = tab_items_kernel(a.a, fmt, weighted);
  pl->accum = weighted ? k_part_accum<true> : k_part_accum<false>;
  int per_sm = 1;
  cudaError_t e = tab_items_per_sm(pl->items, &per_sm);
  if (e != cudaSuccess) return e;
  pl->attrs = a.a;
  pl->weighted = weighted;
  pl->full_grid = (int64_t)sms * per_sm;
  pl->W = part_window(a.n, most);
  int logm = 0;
  while (((int64_t)1 << logm) < (int64_t)a.m) logm++;
  pl->logL = std::min(logm, 15);
  pl->smem = (size_t)4 << pl->logL;
  e = allow_dynamic_smem((const void*)pl->accum);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pl->accum, 1024, pl->smem);
  pl->slots = (int64_t)sms * std::max(1, per_sm);
  pl->units = (int64_t)(a.m >> pl->logL) * a.d;
  return e;
}

// Phase-1 grid and regions of a window of cnt tuples, its phase-2 split and the largest |Delta|
// of an item: a phase-2 counter sums at most R C items, below 2^31 in magnitude.
int part_regions(const PartPlan& pl, int d, int64_t cnt, PartArgs* q, PartSplit* sp) {
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((cnt + 255) / 256, pl.full_grid));
  const int64_t gend = (cnt + 31) / 32 * 32;
  q->cnt = cnt;
  q->C = 32 * ((gend + (int64_t)grid * 256 - 1) / ((int64_t)grid * 256));
  q->nwarps = grid * 8;
  // One attribute's bins are as skewed as its keys; sums of several are not.  With one wave as for
  // several, 5e7 Zipf (1.1) tuples took 1667 us at m = 2^16, d = 9, now 1322; uniform ones 1033, now 1087.
  const int64_t chunks = q->C * d / (pl.weighted ? 4 : 8) / pl.units;
  *sp = part_split(cnt * d, pl.units, pl.slots, q->nwarps, chunks, pl.attrs == 1 && pl.units > d ? 0.6 : 0.0);
  q->wmax = std::min<int64_t>(65535, 0x7fffffff / ((int64_t)sp->R * q->C));
  return grid;
}

// CTAs of a weighted window per resident one (add_direct): one per 400 000 tuples, 4 to 20; four
// when the whole phase may have to return at once (go).
int direct_ctas(int64_t cnt, const int* go) {
  return go ? 4 : (int)std::min<int64_t>(20, std::max<int64_t>(4, cnt / 400000));
}

// What the table kernel samples of a weighted batch (of its first window's limit; a shorter last
// window's is larger).
cudaError_t weight_sample(const UpdArgs& a, int fmt, void* staging, int sms, int64_t most, WeightSample* ws) {
  *ws = {nullptr, a.n, 0, nullptr};
  if (!a.w) return cudaSuccess;
  PartPlan pl;
  const cudaError_t e = part_plan(a, fmt, sms, most, &pl);
  if (e != cudaSuccess) return e;
  PartArgs q;
  PartSplit sp;
  part_regions(pl, a.d, std::min(pl.W, a.n), &q, &sp);
  *ws = {a.w, a.n, q.wmax,
         (PartChoice*)((char*)staging + part_items_bytes(a.d, pl.W, sms, true) + part_counts_bytes(sms))};
  return cudaSuccess;
}

// Both phases over every window of the batch; staging (part_staging_bytes) is caller-owned.
// colp: the first tuple's key of each of the a.a attributes (nullptr: a.cols + u a.stride).
// vbits: nullptr, or one bit per batch tuple (bit i mod 32 of word i / 32) that must be set
// for the tuple to be added.  most: tuples per window at most.  go: see PartArgs.  A weighted batch's
// table kernel has been given weight_sample's.
cudaError_t run_partitioned(const UpdArgs& a, const TabArgs& t, int fmt, void* staging, int sms, cudaStream_t st,
                            const int64_t* const* colp = nullptr, const uint32_t* vbits = nullptr,
                            int64_t most = (int64_t)1 << 30, const int* go = nullptr) {
  const int64_t n = a.n;
  const bool weighted = a.w != nullptr;
  PartPlan pl;
  cudaError_t e = part_plan(a, fmt, sms, most, &pl);
  if (e != cudaSuccess) return e;
  PartArgs q;
  q.go = go;
  q.items = staging;
  q.cnts = (uint32_t*)((char*)staging + part_items_bytes(a.d, pl.W, sms, weighted));
  q.choice = weighted ? (PartChoice*)((char*)q.cnts + part_counts_bytes(sms)) : nullptr;
  q.W = pl.W;
  q.logL = pl.logL;
  for (int64_t i0 = 0; i0 < n && e == cudaSuccess; i0 += pl.W) {
    PartSplit sp;
    const int grid = part_regions(pl, a.d, std::min(pl.W, n - i0), &q, &sp);
    for (int u = 0; u < 5; u++)
      q.col[u] = u < a.a ? (colp ? colp[u] : a.cols + (int64_t)u * a.stride) + i0 : nullptr;
    q.vbits = vbits ? vbits + i0 / 32 : nullptr;   // windows start at multiples of 256
    q.wts = weighted ? a.w + i0 : nullptr;
    pl.items<<<weighted ? grid * direct_ctas(q.cnt, go) : grid, 256, 0, st>>>(a, t, q);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) break;
    pl.accum<<<(unsigned)(pl.units * sp.nr), 1024, pl.smem, st>>>(q, a.ctr, (int64_t)a.m, a.d, pl.logL, sp.R, sp.logP);
    count_launch();
    e = cudaGetLastError();
  }
  return e;
}

// ---------------------------------------------------------------------------
// Partitioned update for the widest sketches (unit weights, power-of-two 2^21 <= m <= 2^24,
// d <= 16, at most 5 attributes, declared domains; 2^17 <= m <= 2^20 takes k_wide_sort below,
// whose one-word items have no room for more bins, unless its two reads of the keys would
// cross the host link).  A d x m int64 sketch of 128 MB does not
// stay in L2, and one 64-bit reduction per (tuple, row) then
// waits on DRAM.  Each row's bins are split into S = m / 2^15 parts of 2^15 bins (the int32
// counters of one part fill 128 KB of one SM's shared memory); the items of a window are
// sorted by part in four steps:
//   1. k_wide_items: one CTA per chunk of kWideChunk tuples gathers the A key-table records
//      (wide format: one 32-bit word per row, bin in bits 0..30, sign in bit 31) of each tuple,
//      writes row j's item (bin mod m | sign << 31; 0x7fffffff for a tuple left out for a key
//      outside its domain) to plane[j][i] and counts each row's items per part in shared
//      memory; the counts go to H[(j S + b) nchunk + c];
//   2. an exclusive scan of H (k_scan_*) into OFF: OFF[(j S + b) nchunk + c] is the first
//      position of chunk c's part-b items of row j in the sorted item array, whose row-major,
//      part-major order the flat scan gives;
//   3. k_wide_scatter: per (chunk, row) the chunk's items ranked within their parts in shared
//      memory (16-bit: offset within the part | sign << 15) and written out part by part,
//      each part's run contiguous;
//   4. k_wide_plan lists the phase-2 CTAs (heavy parts split over several), and in
//      k_wide_accum a CTA owns part b of row j as 2^15 int32 counters over a range of that
//      part's items, adds with shared-memory atomics and adds each counter into the int64
//      sketch with one 64-bit reduction.
// Every counter receives the same integer sum as with one reduction per (tuple, row).
// ---------------------------------------------------------------------------
constexpr int kWideChunk = 4096;   // tuples per phase-1 CTA (256 threads x 16; 2048: chain8 update 9.04 vs 8.72 ms)
constexpr int kWideMaxRows = 16;
constexpr int kWideMaxParts = 512;  // m <= 2^24

struct WideArgs {
  uint32_t* plane;     // [d][W] 32-bit items of the window
  uint16_t* sorted;    // [d W + 8] 16-bit items, row-major then part-major
  uint32_t* H;         // [d][S][nchunk] per-chunk part counts
  uint32_t* OFF;       // [d][S][nchunk] their exclusive scan: first position in `sorted`
  uint32_t* bsum;      // scan block sums
  uint4* plan;         // phase-2 work: per CTA (row j * S + part b, first item, end, heavy); plan_n[0] CTAs
  uint32_t* plan_n;
  int64_t W;           // window capacity
  int64_t cnt;         // tuples in the window
  const int64_t* col[5];
  int nchunk;
  int S;
};

// Per tuple the A records' vectors are all loaded before any is summed (up to 4 x A vectors
// in flight; A <= 2, the chain's relations), and the next tuple's keys are loaded before this
// tuple's records.
template <int A>
__global__ void __launch_bounds__(256) k_wide_items(UpdArgs p, TabArgs t, WideArgs q) {
  __shared__ uint32_t hist[kWideMaxRows * kWideMaxParts];
  constexpr int VH = A <= 2 ? 4 : 1;   // vectors loaded together per record
  const int d = p.d, S = q.S;
  for (int k = threadIdx.x; k < d * S; k += blockDim.x) hist[k] = 0;
  __syncthreads();
  const uint32_t mask = (uint32_t)p.m - 1u;
  const int rv = (d + 3) >> 2;   // 16-byte vectors per record
  const int64_t c0 = (int64_t)blockIdx.x * kWideChunk;
  const int64_t cend = c0 + kWideChunk < q.cnt ? c0 + kWideChunk : q.cnt;
  int64_t i = c0 + threadIdx.x;
  int64_t key[A];
#pragma unroll
  for (int u = 0; u < A; u++) key[u] = i < cend ? ld_key_stream(q.col[u] + i) : 0;
  for (; i < cend; i += 256) {
    bool ok = true;
    const uint4* rec[A];
#pragma unroll
    for (int u = 0; u < A; u++) {
      const bool kin = (uint64_t)key[u] < (uint64_t)p.dom[u];
      ok = ok && kin;
      rec[u] = (const uint4*)t.tbl + ((uint64_t)t.base[u] + (kin ? (uint64_t)key[u] : 0ull)) * (uint64_t)t.rvec;
    }
    const int64_t inext = i + 256;
#pragma unroll
    for (int u = 0; u < A; u++) key[u] = inext < cend ? ld_key_stream(q.col[u] + inext) : 0;
    if (!ok) record(p.status, SK_ERR_KEY_OUT_OF_DOMAIN);
    for (int v0 = 0; v0 < rv; v0 += VH) {
      uint4 w[VH][A];
#pragma unroll
      for (int vh = 0; vh < VH; vh++)
#pragma unroll
        for (int u = 0; u < A; u++)
          w[vh][u] = (ok && v0 + vh < rv) ? __ldg(rec[u] + v0 + vh) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int vh = 0; vh < VH; vh++) {
        uint32_t acc[4] = {0, 0, 0, 0}, sg[4] = {0, 0, 0, 0};
#pragma unroll
        for (int u = 0; u < A; u++) {
          const uint32_t e[4] = {w[vh][u].x, w[vh][u].y, w[vh][u].z, w[vh][u].w};
#pragma unroll
          for (int h = 0; h < 4; h++) {
            acc[h] += e[h] & 0x7fffffffu;
            sg[h] ^= e[h] >> 31;
          }
        }
#pragma unroll
        for (int h = 0; h < 4; h++) {
          const int j = 4 * (v0 + vh) + h;
          if (j < d) {
            const uint32_t bin = acc[h] & mask;
            q.plane[(int64_t)j * q.W + i] = ok ? (bin | (sg[h] << 31)) : 0x7fffffffu;
            if (ok) atomicAdd(&hist[j * S + (int)(bin >> 15)], 1u);
          }
        }
      }
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < d * S; k += blockDim.x) q.H[(int64_t)k * q.nchunk + blockIdx.x] = hist[k];
}

// Exclusive scan of n uint32: k_scan_blocks scans blocks of 4096 of `in` (4 per thread) into
// `out` and leaves each block's total in bsum; k_scan_sums scans bsum (one CTA); k_scan_add
// adds the scanned totals to `out`.
__device__ __forceinline__ uint32_t block_excl_scan_1024(uint32_t v, uint32_t* s_warp, uint32_t* total) {
  const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= (unsigned)o) x += y;
  }
  if (lane == 31u) s_warp[wid] = x;
  __syncthreads();
  if (wid == 0) {
    uint32_t s = lane < (blockDim.x >> 5) ? s_warp[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= (unsigned)o) s += y;
    }
    s_warp[lane] = s;   // inclusive warp totals
  }
  __syncthreads();
  const uint32_t before = wid ? s_warp[wid - 1] : 0u;
  *total = s_warp[(blockDim.x >> 5) - 1];
  __syncthreads();
  return before + x - v;
}

__global__ void __launch_bounds__(1024) k_scan_blocks(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* bsum) {
  __shared__ uint32_t s_warp[32];
  const int64_t base = (int64_t)blockIdx.x * 4096 + (int64_t)threadIdx.x * 4;
  uint32_t v[4], sum = 0;
#pragma unroll
  for (int k = 0; k < 4; k++) {
    v[k] = base + k < n ? in[base + k] : 0u;
    sum += v[k];
  }
  uint32_t total;
  uint32_t run = block_excl_scan_1024(sum, s_warp, &total);
#pragma unroll
  for (int k = 0; k < 4; k++) {
    if (base + k < n) out[base + k] = run;
    run += v[k];
  }
  if (threadIdx.x == 0) bsum[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) k_scan_sums(uint32_t* bsum, int nb) {
  __shared__ uint32_t s_warp[32];
  uint32_t carry = 0;
  for (int b0 = 0; b0 < nb; b0 += 1024) {
    const int i = b0 + (int)threadIdx.x;
    const uint32_t v = i < nb ? bsum[i] : 0u;
    uint32_t total;
    const uint32_t x = block_excl_scan_1024(v, s_warp, &total);
    if (i < nb) bsum[i] = carry + x;
    carry += total;
  }
}

__global__ void __launch_bounds__(1024) k_scan_add(uint32_t* a, int64_t n, const uint32_t* bsum) {
  const int64_t base = (int64_t)blockIdx.x * 4096;
  const uint32_t off = bsum[blockIdx.x];
  for (int k = threadIdx.x; k < 4096; k += blockDim.x)
    if (base + k < n) a[base + k] += off;
}

// blockIdx.x = chunk c, blockIdx.y = row j.  Chunk c's items of row j ranked within their
// parts (a shared-memory counter per part), staged in part order, then written part by part.
__global__ void __launch_bounds__(256) k_wide_scatter(WideArgs q, int64_t m) {
  __shared__ uint32_t lstart[kWideMaxParts], rank[kWideMaxParts], gpos[kWideMaxParts];
  __shared__ uint32_t s_pk[kWideChunk];   // item | part << 16
  __shared__ uint32_t s_warp[32];
  const int c = blockIdx.x, j = blockIdx.y, S = q.S;
  // this chunk's part counts (S <= 512: two per thread), their exclusive scan
  uint32_t n2[2] = {0u, 0u};
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const int b = 2 * (int)threadIdx.x + h;
    if (b < S) {
      const int64_t k = ((int64_t)j * S + b) * q.nchunk + c;
      n2[h] = q.H[k];
      gpos[b] = q.OFF[k];
    }
  }
  uint32_t total;
  const uint32_t ex = block_excl_scan_1024(n2[0] + n2[1], s_warp, &total);
#pragma unroll
  for (int h = 0; h < 2; h++) {
    const int b = 2 * (int)threadIdx.x + h;
    if (b < S) {
      lstart[b] = ex + (h ? n2[0] : 0u);
      rank[b] = 0u;
    }
  }
  __syncthreads();
  const int64_t i0 = (int64_t)c * kWideChunk;
  const uint32_t low = (1u << 15) - 1u;
  for (int k = threadIdx.x; k < kWideChunk; k += blockDim.x) {
    const int64_t i = i0 + k;
    if (i >= q.cnt) break;
    const uint32_t it = q.plane[(int64_t)j * q.W + i];
    const uint32_t bin = it & 0x7fffffffu;
    if (bin < (uint32_t)m) {
      const uint32_t b = bin >> 15;
      const uint32_t lp = lstart[b] + atomicAdd(&rank[b], 1u);
      s_pk[lp] = (bin & low) | ((it >> 31) << 15) | (b << 16);
    }
  }
  __syncthreads();
  for (uint32_t lp = threadIdx.x; lp < total; lp += blockDim.x) {
    const uint32_t pk = s_pk[lp], b = pk >> 16;
    q.sorted[gpos[b] + (lp - lstart[b])] = (uint16_t)pk;
  }
}

// Phase-2 work list: part b of row j gets ceil(items / B) CTAs over equal ranges of its items
// (B = twice the mean part's items, at least 2^16), so a part that a heavy bin makes large is
// spread over several SMs; a CTA of such a part is marked heavy.  One CTA of 1024 threads:
// entries e = j S + b, scanned in rounds of 1024.
__global__ void __launch_bounds__(1024) k_wide_plan(WideArgs q, int d, uint32_t B, uint32_t maxc) {
  __shared__ uint32_t s_warp[32];
  const int64_t ne = (int64_t)d * q.S;
  const int64_t last = ne * q.nchunk - 1;
  uint32_t carry = 0;
  for (int64_t e0 = 0; e0 < ne; e0 += 1024) {
    const int64_t e = e0 + threadIdx.x;
    uint32_t P0 = 0, P1 = 0, k = 0;
    if (e < ne) {
      P0 = q.OFF[e * q.nchunk];
      P1 = e + 1 < ne ? q.OFF[(e + 1) * q.nchunk] : q.OFF[last] + q.H[last];
      k = (P1 - P0 + B - 1) / B;
    }
    uint32_t total;
    const uint32_t first = carry + block_excl_scan_1024(k, s_warp, &total);
    for (uint32_t r = 0; r < k; r++) {
      if (first + r >= maxc) break;
      const uint32_t lo = P0 + (uint32_t)(((uint64_t)(P1 - P0) * r) / k);
      const uint32_t hi = P0 + (uint32_t)(((uint64_t)(P1 - P0) * (r + 1)) / k);
      q.plan[first + r] = make_uint4((uint32_t)e, lo, hi, k > 1 ? 1u : 0u);
    }
    carry += total;
  }
  if (threadIdx.x == 0) q.plan_n[0] = carry < maxc ? carry : maxc;
}

// One CTA per work-list entry (CTAs past the list's length return at once): part b of row j as
// 2^15 int32 counters over its items [lo, hi) of `sorted`.  Lanes take consecutive 8-item
// chunks, two per iteration.  In a heavy CTA each lane first merges runs of equal items among
// its 8 (a heavy bin's items make most of such a part) and adds each run with one atomic.
__global__ void __launch_bounds__(1024) k_wide_accum(WideArgs q, unsigned long long* ctr, int64_t m) {
  if (blockIdx.x >= q.plan_n[0]) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int* cnt = (int*)smem_raw;
  const uint4 wk = q.plan[blockIdx.x];
  const int S = q.S;
  const int j = (int)(wk.x / (uint32_t)S), b = (int)(wk.x % (uint32_t)S);
  const uint32_t lo = wk.y, hi = wk.z;
  const bool heavy = wk.w != 0;
  constexpr int L = 1 << 15;
  for (int k = threadIdx.x; k < L; k += blockDim.x) cnt[k] = 0;
  __syncthreads();
  const uint32_t n = hi - lo;
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(cnt);
  // slots bo .. bo + 7 counted from lo: add those below n
  auto unit = [&](uint4 v, uint32_t bo) { add_chunk(sbase, v, bo, n); };
  auto unit_merge = [&](uint4 v, uint32_t bo) {
    const uint32_t e[4] = {v.x, v.y, v.z, v.w};
    uint32_t prev = 0xffffffffu;   // no item has bits 16..31 set
    int run = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t it = (e[k >> 1] >> (16 * (k & 1))) & 0xffffu;
      const bool valid = bo + (uint32_t)k < n;
      const int sv = (it >> 15) ? -1 : 1;
      if (valid && it == prev) {
        run += sv;
      } else if (valid) {
        if (run != 0) atomicAdd(cnt + (prev & 0x7fffu), run);
        prev = it;
        run = sv;
      }
    }
    if (run != 0) atomicAdd(cnt + (prev & 0x7fffu), run);
  };
  const uint32_t ke = (hi + 7) >> 3;
  uint32_t k = (lo >> 3) + threadIdx.x;
  if (heavy) {
    for (; k < ke; k += blockDim.x) unit_merge(*(const uint4*)(q.sorted + 8 * (size_t)k), 8 * k - lo);
  } else {
    for (; k + blockDim.x < ke; k += 2 * blockDim.x) {
      const uint4 v1 = *(const uint4*)(q.sorted + 8 * (size_t)k);
      const uint4 v2 = *(const uint4*)(q.sorted + 8 * (size_t)(k + blockDim.x));
      unit(v1, 8 * k - lo);
      unit(v2, 8 * (k + blockDim.x) - lo);
    }
    if (k < ke) unit(*(const uint4*)(q.sorted + 8 * (size_t)k), 8 * k - lo);
  }
  __syncthreads();
  unsigned long long* out = ctr + (int64_t)j * m + ((int64_t)b << 15);
  for (int x = threadIdx.x; x < L; x += blockDim.x) {
    const int v = cnt[x];
    if (v != 0) red_add_global(out + x, (unsigned long long)(int64_t)v);
  }
}

// ---------------------------------------------------------------------------
// Wide partitioned update for 2^17 <= m <= 2^20 (4 to 32 parts).  The items of a chunk are
// sorted by part inside the CTA that gathers them and stay where that CTA writes them, so
// neither a 32-bit item plane nor a scan over all chunks nor a scatter pass is needed:
//   1. k_wide_sort: a CTA takes kSortChunk tuples and eight rows (half a 64-byte record per
//      gather; the CTAs of one half run together, so half of the tables fights for L2 at a
//      time).  Every item is kept in shared memory as bin | sign | rank, the rank within its
//      (row, part) from the returning shared-memory atomic that counts the part; after a scan
//      over the parts the row is rewritten in place as 16-bit items in part order and leaves
//      with 16-byte stores, its part starts in OFF[row][part][chunk];
//   2. k_wide_list: the work list, a part with more than twice the mean's items spread over
//      several CTAs by chunk ranges;
//   3. k_wide_gather: a CTA owns a part of a row as 2^15 int32 counters and collects its
//      segment of every chunk of its range.  A warp turns up to 32 segments into a list of
//      16-byte pieces (position, mask of its items) in shared memory, so that every lane has
//      a piece whatever the segments' lengths.
// Per tuple and row 2 bytes are written and read once (the sorted form above: 8 written, 8
// read), and each item passes one atomic with a returned value instead of two.  Inner chain
// relation of 1e7 tuples, m = 2^20, d = 16: 758 us against 1063 us (table 89, k_wide_sort 427,
// bound by the L1 data pipe at 77 %: two record gathers and 12 shared-memory wavefronts per warp
// and row; k_wide_gather 217, waiting on the pieces it loads; 352 + 152 us before its list was
// ordered for the SMs).
// ---------------------------------------------------------------------------
constexpr int kSortLog = 11;
constexpr int kSortChunk = 1 << kSortLog;   // tuples per CTA: rank 11 bits + bin 20 + sign 1 = one word
constexpr int kSortRows = 8;                // rows per CTA
constexpr int kSortMaxParts = 32;
constexpr int kPieceCap = 384;              // pieces a warp lists at a time (32 mean segments make 290)

struct SortArgs {
  uint16_t* sorted;    // [d][nchunk][kSortChunk]
  uint16_t* off;       // [d][S + 1][nchunk] part starts within a chunk's row; [S]: its item count
  uint32_t* total;     // [d][S] items of the window
  uint4* plan;         // per CTA: row * S + part, first chunk, end, heavy
  uint32_t* plan_n;
  int64_t cnt;         // tuples in the window
  const int64_t* col[5];
  int nchunk;
  int S;
  int chunk0, group0;  // k_wide_sort: chunk and row group of the launch's first CTA
};

__global__ void k_wide_clear(uint32_t* total, int n) {
  const int k = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (k < n) total[k] = 0;
}

// PAIR: records are a multiple of 32 bytes, so a CTA's eight words arrive with one load.
template <int A, bool PAIR>
__global__ void __launch_bounds__(512, 2) k_wide_sort(UpdArgs p, TabArgs t, SortArgs q) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* item = (uint32_t*)smem_raw;   // [row][kSortChunk]
  __shared__ uint32_t hist[kSortRows * kSortMaxParts];
  __shared__ uint32_t valid[kSortChunk / 32];
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int group = q.group0 + (int)blockIdx.y;
  const int S = q.S, chunk = q.chunk0 + (int)blockIdx.x, row0 = kSortRows * group;
  const int nr = min(kSortRows, p.d - row0);
  for (int k = tid; k < kSortRows * kSortMaxParts; k += 512) hist[k] = 0;
  __syncthreads();
  const uint32_t mask = (uint32_t)p.m - 1u;
  const int64_t c0 = (int64_t)chunk << kSortLog;
  int64_t key[A];
#pragma unroll
  for (int u = 0; u < A; u++) key[u] = c0 + tid < q.cnt ? ld_key_stream(q.col[u] + c0 + tid) : -1;
  bool mine = true;   // all of this thread's tuples are kept
  for (int i = tid; i < kSortChunk; i += 512) {
    bool ok = true;
    const uint4* rec[A];
#pragma unroll
    for (int u = 0; u < A; u++) {
      const bool kin = (uint64_t)key[u] < (uint64_t)p.dom[u];
      ok = ok && kin;
      rec[u] = (const uint4*)t.tbl + ((uint64_t)t.base[u] + (kin ? (uint64_t)key[u] : 0ull)) * (uint64_t)t.rvec +
               2 * group;
    }
    if (!ok && c0 + i < q.cnt) record(p.status, SK_ERR_KEY_OUT_OF_DOMAIN);
    const int64_t nx = c0 + i + 512;
#pragma unroll
    for (int u = 0; u < A; u++)
      key[u] = (i + 512 < kSortChunk && nx < q.cnt) ? ld_key_stream(q.col[u] + nx) : -1;
    const uint32_t vb = __ballot_sync(0xffffffffu, ok);
    if (lane == 0) valid[i >> 5] = vb;
    mine = mine && ok;
    if (!ok) continue;
    uint32_t bin[8] = {0, 0, 0, 0, 0, 0, 0, 0}, sg[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    uint32_t w[A][8];
#pragma unroll
    for (int u = 0; u < A; u++) {
      if (PAIR) {
        ld_record32(rec[u], w[u]);
      } else {
        const uint4 x = __ldg(rec[u]), y = nr > 4 ? __ldg(rec[u] + 1) : make_uint4(0u, 0u, 0u, 0u);
        w[u][0] = x.x, w[u][1] = x.y, w[u][2] = x.z, w[u][3] = x.w;
        w[u][4] = y.x, w[u][5] = y.y, w[u][6] = y.z, w[u][7] = y.w;
      }
    }
#pragma unroll
    for (int u = 0; u < A; u++)
#pragma unroll
      for (int j = 0; j < 8; j++) {
        bin[j] += w[u][j];   // the sign bits carry out above the bins
        sg[j] ^= w[u][j];
      }
#pragma unroll
    for (int j = 0; j < 8; j++) {
      if (j >= nr) break;
      const uint32_t b = bin[j] & mask;
      const uint32_t rank = atomicAdd(&hist[j * kSortMaxParts + (b >> 15)], 1u);
      item[(j << kSortLog) + i] = b | ((sg[j] >> 31) << 20) | (rank << 21);
    }
  }
  const bool full = __syncthreads_and(mine);
  // warp j: row j's part starts
  if (warp < nr) {
    const uint32_t n = hist[warp * kSortMaxParts + lane];   // parts at and beyond S hold nothing
    uint32_t x = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    hist[warp * kSortMaxParts + lane] = x - n;
    const int64_t row = row0 + warp;
    if (lane < S) {
      q.off[(row * (S + 1) + lane) * q.nchunk + chunk] = (uint16_t)(x - n);
      if (lane == S - 1) q.off[(row * (S + 1) + S) * q.nchunk + chunk] = (uint16_t)x;
      if (n) atomicAdd(q.total + row * S + lane, n);
    }
  }
  __syncthreads();
  // two warps per row: its items through registers into part order, 16 bits each
  const int j = warp >> 1, h = warp & 1;
  constexpr int E = kSortChunk / 64;   // items per lane
  uint32_t x[E];
  uint32_t* src = item + (j << kSortLog) + h * (kSortChunk / 2) + lane;
  if (j < nr) {
#pragma unroll
    for (int e = 0; e < E; e++) x[e] = src[32 * e];
  }
  __syncthreads();
  uint16_t* dst = (uint16_t*)(item + (j << kSortLog));
  if (j < nr) {
#pragma unroll
    for (int e = 0; e < E; e++) {
      const uint32_t b = x[e] & 0xfffffu;
      if (full || ((valid[h * E + e] >> lane) & 1u))
        dst[hist[j * kSortMaxParts + (b >> 15)] + (x[e] >> 21)] =
            (uint16_t)((b & 0x7fffu) | (((x[e] >> 20) & 1u) << 15));
    }
  }
  __syncthreads();
  if (j < nr) {
    const uint4* sv = (const uint4*)(item + (j << kSortLog));
    uint4* out = (uint4*)(q.sorted + (((int64_t)(row0 + j) * q.nchunk + chunk) << kSortLog));
    for (int k = h * 32 + lane; k < kSortChunk / 8; k += 64) out[k] = sv[k];
  }
}

// Work list, in the order the CTAs start (one per SM at a time): first the parts with more than
// 5/4 of the mean's items, split into pieces of at most the mean by chunk ranges; then the others
// whole; the last of them, which would start a wave that leaves most SMs idle, split so that the
// wave fills.  One CTA of 512 threads, one part (of at most 16 x 32) each.
__global__ void __launch_bounds__(512) k_wide_list(SortArgs q, int d, int sms, uint32_t maxc) {
  __shared__ uint32_t s_warp[32];
  const uint32_t e = threadIdx.x, ne = (uint32_t)(d * q.S);
  const uint32_t n = e < ne ? q.total[e] : 0u;
  uint32_t sum, nheavy, nlight;
  block_excl_scan_1024(n, s_warp, &sum);
  const uint32_t mean = max(1u, sum / ne);
  const bool big = n > mean + mean / 4;
  uint32_t k = big ? min((n + mean - 1) / mean, (uint32_t)q.nchunk) : (n ? 1u : 0u);
  uint32_t first = block_excl_scan_1024(big ? k : 0u, s_warp, &nheavy);
  const uint32_t li = block_excl_scan_1024(big ? 0u : k, s_warp, &nlight);
  if (!big && k) {
    // whole parts up to a multiple of the SMs, the rest in `cut` pieces each
    const uint32_t rem = min(nlight, (nheavy + nlight) % (uint32_t)sms);
    const uint32_t cut = rem ? max(1u, min(min(8u, (uint32_t)q.nchunk), (uint32_t)sms / rem)) : 1u;
    const uint32_t whole = nlight - rem;
    first = nheavy + (li < whole ? li : whole + (li - whole) * cut);
    k = li < whole ? 1u : cut;
  }
  for (uint32_t r = 0; r < k && first + r < maxc; r++)
    q.plan[first + r] = make_uint4(e, (uint32_t)(((uint64_t)q.nchunk * r) / k),
                                   (uint32_t)(((uint64_t)q.nchunk * (r + 1)) / k), n > 2 * mean ? 1u : 0u);
  uint32_t entries;
  block_excl_scan_1024(k, s_warp, &entries);
  if (threadIdx.x == 0) q.plan_n[0] = min(entries, maxc);
}

// 32 warps; shared memory: 2^15 int32 counters, then kPieceCap pieces per warp.  A piece is 8
// consecutive item slots: segment << 16 | slot / 8 << 8 | mask of the slots that are the part's.
__global__ void __launch_bounds__(1024) k_wide_gather(SortArgs q, unsigned long long* ctr, int64_t m) {
  if (blockIdx.x >= q.plan_n[0]) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int* cnt = (int*)smem_raw;
  constexpr int L = 1 << 15;
  const int lane = (int)(threadIdx.x & 31u), warp = (int)(threadIdx.x >> 5);
  uint32_t* piece = (uint32_t*)(cnt + L) + warp * kPieceCap;
  const uint4 wk = q.plan[blockIdx.x];
  const int S = q.S, row = (int)(wk.x / (uint32_t)S), part = (int)(wk.x % (uint32_t)S);
  const int ch0 = (int)wk.y, ch1 = (int)wk.z;
  const bool heavy = wk.w != 0;   // most of its items are one bin's: runs of equal items add once
  for (int k = threadIdx.x; k < L / 4; k += 1024) ((int4*)cnt)[k] = make_int4(0, 0, 0, 0);
  __syncthreads();
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(cnt);
  const uint16_t* off0 = q.off + ((int64_t)row * (S + 1) + part) * q.nchunk;
  const uint16_t* off1 = off0 + q.nchunk;
  // segments a warp lists at a time: all 32 warps get some
  const int G = min(32, max(1, (ch1 - ch0 + 31) >> 5));
  for (int g = ch0 + G * warp; g < ch1; g += G * 32) {
    const bool in = lane < G && g + lane < ch1;
    const uint32_t lo = in ? off0[g + lane] : 0u, hi = in ? off1[g + lane] : 0u;
    const uint32_t kb = lo >> 3, n = hi > lo ? ((hi + 7) >> 3) - kb : 0u;
    uint32_t x = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    const uint32_t all = __shfl_sync(0xffffffffu, x, 31);
    const uint32_t first = x - n;
    const uint4* base = (const uint4*)(q.sorted + (((int64_t)row * q.nchunk + g) << kSortLog));
    for (uint32_t r0 = 0; r0 < all; r0 += kPieceCap) {
      // this lane's pieces at list positions [r0, r0 + kPieceCap)
      const uint32_t k0 = first < r0 ? min(r0 - first, n) : 0u;
      const uint32_t k1 = first + n > r0 + kPieceCap ? (first < r0 + kPieceCap ? r0 + kPieceCap - first : 0u) : n;
      for (uint32_t k = k0; k < k1; k++) {
        const uint32_t s0 = 8u * (kb + k);
        const uint32_t a = lo > s0 ? lo - s0 : 0u, b = min(hi - s0, 8u);
        piece[first + k - r0] = ((uint32_t)lane << 16) | ((kb + k) << 8) | (((1u << b) - 1u) & ~((1u << a) - 1u));
      }
      __syncwarp();
      const uint32_t np = min(all - r0, (uint32_t)kPieceCap);
      uint32_t pcn = lane < np ? piece[lane] : 0u;
      uint4 vn = make_uint4(0u, 0u, 0u, 0u);
      if (lane < np) vn = __ldg(base + (pcn >> 16) * (kSortChunk / 8) + ((pcn >> 8) & 0xffu));
      for (uint32_t k = lane; k < np; k += 32) {
        const uint32_t pc = pcn;
        const uint4 v = vn;
        if (k + 32 < np) {   // the next piece's items, in flight during this one's additions
          pcn = piece[k + 32];
          vn = __ldg(base + (pcn >> 16) * (kSortChunk / 8) + ((pcn >> 8) & 0xffu));
        }
        const uint32_t e[4] = {v.x, v.y, v.z, v.w};
        if (heavy) {
          uint32_t prev = 0xffffffffu;
          int run = 0;
#pragma unroll
          for (int h = 0; h < 8; h++) {
            const uint32_t it = (e[h >> 1] >> (16 * (h & 1))) & 0xffffu;
            const int sv = (it >> 15) ? -1 : 1;
            if (!((pc >> h) & 1u)) continue;
            if (it == prev) {
              run += sv;
            } else {
              if (run != 0) red_shared(sbase + ((prev & 0x7fffu) << 2), run);
              prev = it;
              run = sv;
            }
          }
          if (run != 0) red_shared(sbase + ((prev & 0x7fffu) << 2), run);
        } else {
#pragma unroll
          for (int h = 0; h < 8; h++) {
            const uint32_t it = e[h >> 1] >> (16 * (h & 1));
            int neg;
            asm("bfe.s32 %0, %1, 15, 1;" : "=r"(neg) : "r"(it));
            red_shared_if_set(sbase + ((it & 0x7fffu) << 2), neg | 1, pc & (1u << h));
          }
        }
      }
      __syncwarp();
    }
  }
  __syncthreads();
  unsigned long long* out = ctr + (int64_t)row * m + ((int64_t)part << 15);
  for (int x = threadIdx.x; x < L; x += 1024) {
    const int v = cnt[x];
    if (v != 0) red_add_global(out + x, (unsigned long long)(int64_t)v);
  }
}

struct SortLayout {
  size_t off, total, plan, plan_n, bytes;
};

// Entries of k_wide_list's list at most: pieces of the mean's size add up to fewer than one per
// part beyond the parts themselves, and a tail cut in c <= 8 pieces fills at most one wave more
// than its parts (fewer than 1024 SMs).
uint32_t sort_entries(int64_t units) { return (uint32_t)(2 * units + 1024); }

SortLayout sort_layout(int d, int64_t m, int64_t W) {
  const int64_t S = m >> 15, nchunk = (W + kSortChunk - 1) / kSortChunk;
  auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
  SortLayout L;
  L.off = al((size_t)d * nchunk * kSortChunk * sizeof(uint16_t));
  L.total = L.off + al((size_t)d * (S + 1) * nchunk * sizeof(uint16_t));
  L.plan = L.total + al((size_t)d * S * sizeof(uint32_t));
  L.plan_n = L.plan + al((size_t)sort_entries((int64_t)d * S) * sizeof(uint4));
  L.bytes = L.plan_n + 256;
  return L;
}

// k_wide_sort over the whole window in four launches: with two row groups the halves of the
// first group, then of the second (the CTAs of a group run together either way); with one group
// the quarters of the window.  One launch per group would do, and save about 1 % of the pass: a test
// holds every width of the wide update to the seven launches per window that the widest take.
template <int A>
cudaError_t launch_wide_sort(const UpdArgs& a, const TabArgs& t, SortArgs q, cudaStream_t st) {
  constexpr size_t smem = (size_t)kSortRows * kSortChunk * sizeof(uint32_t);
  auto kern = (t.rvec & 1) == 0 ? k_wide_sort<A, true> : k_wide_sort<A, false>;
  cudaError_t e = allow_dynamic_smem((const void*)kern);
  const int parts = a.d > kSortRows ? 2 : 4;
  for (int l = 0; l < 4 && e == cudaSuccess; l++) {
    q.group0 = l / parts;
    q.chunk0 = (int)((int64_t)q.nchunk * (l % parts) / parts);
    const int end = (int)((int64_t)q.nchunk * (l % parts + 1) / parts);
    if (end <= q.chunk0) continue;
    kern<<<(unsigned)(end - q.chunk0), 512, smem, st>>>(a, t, q);
    count_launch();
    e = cudaGetLastError();
  }
  return e;
}

// Window capacity of the wide partitioned update: positions in `sorted` stay below 2^28.
int64_t wide_window(int64_t n) {
  const char* v = std::getenv("SK_PART_WINDOW");
  const long long x = v ? std::atoll(v) : 0;
  const int64_t cap = (x > 0 && x < (1ll << 24)) ? (int64_t)x : ((int64_t)1 << 24);
  return std::min<int64_t>((n + 255) / 256 * 256, (cap + 255) / 256 * 256);
}

struct WideLayout {
  size_t plane, sorted, H, OFF, bsum, plan, plan_n, total;
  uint32_t maxc;   // phase-2 work-list capacity
};

WideLayout wide_layout(int d, int64_t m, int64_t W) {
  const int S = (int)(m >> 15);
  const int64_t nchunk = (W + kWideChunk - 1) / kWideChunk;
  const int64_t N = (int64_t)d * S * nchunk;
  auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
  WideLayout L;
  L.plane = 0;
  L.sorted = L.plane + al((size_t)d * W * sizeof(uint32_t));
  L.H = L.sorted + al(((size_t)d * W + 8) * sizeof(uint16_t));
  L.OFF = L.H + al((size_t)N * sizeof(uint32_t));
  L.bsum = L.OFF + al((size_t)N * sizeof(uint32_t));
  L.plan = L.bsum + al((size_t)((N + 4095) / 4096) * sizeof(uint32_t));
  // at most one CTA per (row, part) plus one per 2^16 items
  L.maxc = (uint32_t)((int64_t)d * S + ((int64_t)d * W >> 16) + 1);
  L.plan_n = L.plan + al((size_t)L.maxc * sizeof(uint4));
  L.total = L.plan_n + 256;
  return L;
}

template <int A>
void launch_wide_items(const UpdArgs& a, const TabArgs& t, const WideArgs& q, cudaStream_t st) {
  k_wide_items<A><<<q.nchunk, 256, 0, st>>>(a, t, q);
}

// All four steps over every window of the batch; staging (wide_layout(...).total bytes for
// the window wide_window(n)) is caller-owned.
cudaError_t run_wide_partitioned(const UpdArgs& a, const TabArgs& t, void* staging, int sms, cudaStream_t st) {
  const int64_t n = a.n;
  const int64_t W = wide_window(n);
  const WideLayout Ly = wide_layout(a.d, (int64_t)a.m, W);
  char* base = (char*)staging;
  WideArgs q;
  q.plane = (uint32_t*)(base + Ly.plane);
  q.sorted = (uint16_t*)(base + Ly.sorted);
  q.H = (uint32_t*)(base + Ly.H);
  q.OFF = (uint32_t*)(base + Ly.OFF);
  q.bsum = (uint32_t*)(base + Ly.bsum);
  q.plan = (uint4*)(base + Ly.plan);
  q.plan_n = (uint32_t*)(base + Ly.plan_n);
  q.W = W;
  q.S = (int)(a.m >> 15);
  const size_t smem = (size_t)4 << 15;
  cudaError_t e = allow_dynamic_smem((const void*)k_wide_accum);
  const int64_t units = (int64_t)q.S * a.d;
  (void)sms;
  for (int64_t i0 = 0; i0 < n && e == cudaSuccess; i0 += W) {
    q.cnt = std::min(W, n - i0);
    for (int u = 0; u < 5; u++) q.col[u] = u < a.a ? a.cols + (int64_t)u * a.stride + i0 : nullptr;
    q.nchunk = (int)((q.cnt + kWideChunk - 1) / kWideChunk);
    switch (a.a) {
      case 1: launch_wide_items<1>(a, t, q, st); break;
      case 2: launch_wide_items<2>(a, t, q, st); break;
      case 3: launch_wide_items<3>(a, t, q, st); break;
      case 4: launch_wide_items<4>(a, t, q, st); break;
      default: launch_wide_items<5>(a, t, q, st); break;
    }
    const int64_t N = units * q.nchunk;
    const int nb = (int)((N + 4095) / 4096);
    k_scan_blocks<<<nb, 1024, 0, st>>>(q.H, q.OFF, N, q.bsum);
    k_scan_sums<<<1, 1024, 0, st>>>(q.bsum, nb);
    k_scan_add<<<nb, 1024, 0, st>>>(q.OFF, N, q.bsum);
    k_wide_scatter<<<dim3((unsigned)q.nchunk, (unsigned)a.d), 256, 0, st>>>(q, (int64_t)a.m);
    // phase-2 work: B = twice the mean part's items (at least 2^16) per CTA
    const uint32_t B = (uint32_t)std::max<int64_t>((int64_t)1 << 16, 2 * (q.cnt * a.d) / std::max<int64_t>(1, units));
    const uint32_t maxc = (uint32_t)std::min<int64_t>((int64_t)Ly.maxc, units + ((int64_t)a.d * q.cnt) / B + 1);
    k_wide_plan<<<1, 1024, 0, st>>>(q, a.d, B, maxc);
    k_wide_accum<<<maxc, 1024, smem, st>>>(q, a.ctr, (int64_t)a.m);
    count_launch(7);
    e = cudaGetLastError();
  }
  return e;
}

// The same for 2^17 <= m <= 2^20; staging: sort_layout(...).bytes for the window.
cudaError_t run_wide_sorted(const UpdArgs& a, const TabArgs& t, void* staging, int sms, cudaStream_t st) {
  const int64_t n = a.n, W = wide_window(n);
  const SortLayout Ly = sort_layout(a.d, (int64_t)a.m, W);
  char* base = (char*)staging;
  SortArgs q;
  q.sorted = (uint16_t*)base;
  q.off = (uint16_t*)(base + Ly.off);
  q.total = (uint32_t*)(base + Ly.total);
  q.plan = (uint4*)(base + Ly.plan);
  q.plan_n = (uint32_t*)(base + Ly.plan_n);
  q.S = (int)(a.m >> 15);
  constexpr size_t smem = ((size_t)4 << 15) + (size_t)32 * kPieceCap * sizeof(uint32_t);
  cudaError_t e = allow_dynamic_smem((const void*)k_wide_gather);
  const int64_t units = (int64_t)q.S * a.d;
  for (int64_t i0 = 0; i0 < n && e == cudaSuccess; i0 += W) {
    q.cnt = std::min(W, n - i0);
    for (int u = 0; u < 5; u++) q.col[u] = u < a.a ? a.cols + (int64_t)u * a.stride + i0 : nullptr;
    q.nchunk = (int)((q.cnt + kSortChunk - 1) / kSortChunk);
    k_wide_clear<<<(unsigned)((units + 255) / 256), 256, 0, st>>>(q.total, (int)units);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) break;
    switch (a.a) {
      case 1: e = launch_wide_sort<1>(a, t, q, st); break;
      case 2: e = launch_wide_sort<2>(a, t, q, st); break;
      case 3: e = launch_wide_sort<3>(a, t, q, st); break;
      case 4: e = launch_wide_sort<4>(a, t, q, st); break;
      default: e = launch_wide_sort<5>(a, t, q, st); break;
    }
    if (e != cudaSuccess) break;
    const uint32_t maxc = sort_entries(units);
    k_wide_list<<<1, 512, 0, st>>>(q, a.d, sms, maxc);
    k_wide_gather<<<maxc, 1024, smem, st>>>(q, a.ctr, (int64_t)a.m);
    count_launch(2);
    e = cudaGetLastError();
  }
  return e;
}

// SK_TAB_V8=0 reads 32-byte key-table records as two 16-byte loads instead of one.
bool tab_v8_enabled() {
  const char* v = std::getenv("SK_TAB_V8");
  return !(v && v[0] == '0');
}

template <int A, bool POW2, bool SMEM>
cudaError_t launch_tab(const UpdArgs& a, const TabArgs& t, int grid, size_t smem, cudaStream_t st) {
  const bool v8 = t.rvec == 2 && tab_v8_enabled();
  auto kern = t.narrow ? (v8 ? k_update_tab<A, POW2, SMEM, true, true> : k_update_tab<A, POW2, SMEM, true, false>)
                       : (v8 ? k_update_tab<A, POW2, SMEM, false, true> : k_update_tab<A, POW2, SMEM, false, false>);
  cudaError_t e = fit_dynamic_smem((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<grid, 256, smem, st>>>(a, t);
  count_launch();
  return cudaGetLastError();
}

template <bool POW2, bool SMEM>
cudaError_t dispatch_tab(const UpdArgs& a, const TabArgs& t, int grid, size_t smem, cudaStream_t st) {
  switch (a.a) {
    case 1: return launch_tab<1, POW2, SMEM>(a, t, grid, smem, st);
    case 2: return launch_tab<2, POW2, SMEM>(a, t, grid, smem, st);
    case 3: return launch_tab<3, POW2, SMEM>(a, t, grid, smem, st);
    case 4: return launch_tab<4, POW2, SMEM>(a, t, grid, smem, st);
    case 5: return launch_tab<5, POW2, SMEM>(a, t, grid, smem, st);
    default: return launch_tab<0, POW2, SMEM>(a, t, grid, smem, st);
  }
}

int sm_count() {
  static const int n = [] {   // thread-safe one-time initialisation
    int dev = 0, x = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&x, cudaDevAttrMultiProcessorCount, dev);
    return x > 0 ? x : 1;
  }();
  return n;
}

// CTAs per SM of the global-atomic update grid.  Default: one tuple per thread (a grid of
// n / 256 CTAs), which measured fastest on the 1e8-row star fact table (12.18 ms, against
// 13.01 / 12.80 / 12.45 / 12.28 ms for 6 / 8 / 16 / 32 grid-stride CTAs per SM);
// SK_UPDATE_GRID=<n> caps the grid at n CTAs per SM instead.
int update_grid_per_sm() {
  const char* v = std::getenv("SK_UPDATE_GRID");
  const int x = v ? std::atoi(v) : 0;
  return x <= 0 ? (1 << 30) / 64 : x;
}

// true when each of the relation's A attributes is in exactly one join
bool all_deg1(const UpdArgs& a) {
  if (a.a < 1) return false;
  for (int u = 0; u < a.a; u++)
    if (a.deg[u] != 1) return false;
  return true;
}

// grid <= 0 sizes the grid with update_grid_per_sm.
template <int A, bool POW2, bool SMEM>
cudaError_t launch_one(const UpdArgs& a, int grid, size_t smem, cudaStream_t st, const int* unless) {
  auto kern = (A > 0 && all_deg1(a)) ? k_update<A, POW2, SMEM, (A > 0)> : k_update<A, POW2, SMEM, false>;
  cudaError_t e = fit_dynamic_smem((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  if (grid <= 0) {
    const int64_t want = (a.n + 255) / 256;
    const int64_t cap = std::min<int64_t>((int64_t)update_grid_per_sm() * sm_count(), 0x7fffffff);
    grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, cap));
  }
  kern<<<grid, 256, smem, st>>>(a, unless);
  count_launch();
  return cudaGetLastError();
}

template <bool POW2, bool SMEM>
cudaError_t dispatch_a(const UpdArgs& a, int grid, size_t smem, cudaStream_t st, const int* unless = nullptr) {
  switch (a.a) {
    case 1: return launch_one<1, POW2, SMEM>(a, grid, smem, st, unless);
    case 2: return launch_one<2, POW2, SMEM>(a, grid, smem, st, unless);
    case 3: return launch_one<3, POW2, SMEM>(a, grid, smem, st, unless);
    case 4: return launch_one<4, POW2, SMEM>(a, grid, smem, st, unless);
    case 5: return launch_one<5, POW2, SMEM>(a, grid, smem, st, unless);
    default: return launch_one<0, POW2, SMEM>(a, grid, smem, st, unless);
  }
}

// ---------------------------------------------------------------------------
// Hot-key cached update (power-of-two m, d <= 32, global atomics).
//
// Skewed key columns (the Zipf-like columns of Figure 5) repeat a few keys very
// often.  Each CTA keeps, per attribute, a direct-mapped table of S keys with
// their per-row results (bin value mod m and sign parity).  The table is filled
// from the CTA's first tuples (first come, first kept; no eviction), then frozen.
// A warp works on 32 tuples at a time: attributes whose key is in the table take
// the stored results; the other (tuple, attribute) pairs are queued and hashed by
// the whole warp densely, one pair per lane, their per-row results accumulated
// into per-tuple shared-memory partial sums.  Every counter update is identical to
// the uncached kernel's.
// ---------------------------------------------------------------------------
constexpr uint64_t kEmptyKey = ~0ull;

__device__ __forceinline__ uint32_t cache_slot(uint64_t x, int log2s) {
  return (uint32_t)((x * 0x9E3779B97F4A7C15ull) >> (64 - log2s));
}

struct CacheLayout {
  int log2s;        // table slots per attribute = 2^log2s
  int fill_groups;  // 32-tuple groups per warp used to fill the table
};

template <int A, bool FILL>
__device__ __forceinline__ void cached_group(const UpdArgs& p, const CacheLayout& c, int64_t i0, int64_t i1,
                                             const uint64_t* s_coef, const int* s_off, uint64_t* cx,
                                             uint32_t* cdata, uint32_t* sbin, uint32_t* ssign, uint64_t* qx,
                                             uint16_t* qtu) {
  const int lane = threadIdx.x & 31;
  const int d = p.d;
  const int S = 1 << c.log2s;
  const int64_t i = i0 + lane;
  bool valid = i < i1;
  uint64_t x[A];
#pragma unroll
  for (int u = 0; u < A; u++) {
    const int64_t key = valid ? __ldg(p.cols + (int64_t)u * p.stride + i) : 0;
    if (valid && p.has_dom && (key < 0 || key >= p.dom[u])) {
      record(p.status, SK_ERR_KEY_OUT_OF_DOMAIN);
      valid = false;
    }
    x[u] = field_of(key);
  }
  const int64_t delta = valid ? (p.w ? __ldg(p.w + i) : 1) : 0;
  uint32_t slot[A];
  uint32_t hitmask = 0;
#pragma unroll
  for (int u = 0; u < A; u++) {
    slot[u] = cache_slot(x[u], c.log2s);
    if (!FILL && valid && cx[u * S + slot[u]] == x[u]) hitmask |= 1u << u;
  }
  uint32_t* my_bin = sbin + lane * d;
  for (int r = 0; r < d; r++) my_bin[r] = 0;
  ssign[lane] = 0;
  int qn = 0;
  const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
  for (int u = 0; u < A; u++) {
    const bool miss = valid && !((hitmask >> u) & 1u);
    const uint32_t bal = __ballot_sync(0xffffffffu, miss);
    if (miss) {
      const int pos = qn + __popc(bal & lt);
      qx[pos] = x[u];
      qtu[pos] = (uint16_t)(lane | (u << 5));
    }
    qn += __popc(bal);
  }
  __syncwarp();
  for (int j = lane; j < qn; j += 32) {
    const uint64_t xv = qx[j];
    const int t = qtu[j] & 31, u = qtu[j] >> 5;
    const uint32_t sl = cache_slot(xv, c.log2s);
    const bool claim = FILL && atomicCAS((unsigned long long*)&cx[u * S + sl], kEmptyKey, xv) == kEmptyKey;
    const int off = s_off[u];
    const int deg = p.deg[u];
    uint32_t* tb = sbin + t * d;
    uint32_t* cd = cdata + ((size_t)u * S + sl) * d;
    uint32_t sbits = 0;
    const bool narrow = (xv >> 32) == 0;
    const uint32_t x32 = (uint32_t)xv;
#pragma unroll 3
    for (int r = 0; r < d; r++) {
      const uint64_t* cr = s_coef + r * p.row_len + off;
      uint32_t hv, par = 0;
      if (narrow) {
        const uint64_t v = mac_narrow(cr[1], x32, cr[0]);
        hv = (uint32_t)v + mersenne_q(v);
        for (int e = 0; e < deg; e++) {
          const uint64_t* sc = cr + 2 + 4 * e;
          uint64_t acc = mac_narrow(sc[3], x32, sc[2]);
          acc = mac_narrow(acc, x32, sc[1]);
          acc = mac_narrow(acc, x32, sc[0]);
          par ^= ((uint32_t)acc ^ mersenne_q(acc)) & 1u;
        }
      } else {
        hv = (uint32_t)addmod(mulmod(cr[1], xv), cr[0]);
        for (int e = 0; e < deg; e++) {
          const uint64_t* sc = cr + 2 + 4 * e;
          uint64_t acc = sc[3];
          acc = addmod(mulmod(acc, xv), sc[2]);
          acc = addmod(mulmod(acc, xv), sc[1]);
          acc = addmod(mulmod(acc, xv), sc[0]);
          par ^= (uint32_t)(acc & 1u);
        }
      }
      atomicAdd(tb + r, hv);
      sbits |= par << r;
      if (claim) cd[r] = (hv & (uint32_t)(p.m - 1)) | (par << 31);
    }
    atomicXor(ssign + t, sbits);
  }
  __syncwarp();
  if (valid) {
    uint32_t sm = ssign[lane];
    for (int r = 0; r < d; r++) {
      uint32_t b = my_bin[r];
#pragma unroll
      for (int u = 0; u < A; u++) {
        if ((hitmask >> u) & 1u) {
          const uint32_t cv = cdata[((size_t)u * S + slot[u]) * d + r];
          b += cv & 0x7fffffffu;
          sm ^= (cv >> 31) << r;
        }
      }
      const uint32_t bin = b & (uint32_t)(p.m - 1);
      const int64_t v = ((sm >> r) & 1u) ? -delta : delta;
      atomicAdd(p.ctr + (int64_t)r * p.m + bin, (unsigned long long)v);
    }
  }
  __syncwarp();
}

template <int A>
__global__ void __launch_bounds__(512) k_update_cached(UpdArgs p, CacheLayout c) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int d = p.d;
  const int S = 1 << c.log2s;
  const int W = blockDim.x >> 5;
  const int warp = threadIdx.x >> 5;
  __shared__ int s_off[A];
  uint64_t* s_coef = (uint64_t*)smem_raw;
  const int ncoef = d * p.row_len;
  uint64_t* cx = s_coef + ncoef;
  uint32_t* cdata = (uint32_t*)(cx + (size_t)A * S);
  uint32_t* sbin = cdata + (size_t)A * S * d;
  uint32_t* ssign = sbin + (size_t)W * 32 * d;
  uint64_t* qx = (uint64_t*)(ssign + W * 32 + ((W * 32) & 1));
  uint16_t* qtu = (uint16_t*)(qx + (size_t)W * 32 * A);
  for (int t = threadIdx.x; t < ncoef; t += blockDim.x) s_coef[t] = p.coef[t];
  for (int t = threadIdx.x; t < A * S; t += blockDim.x) cx[t] = kEmptyKey;
  if (threadIdx.x == 0) {
    int o = 0;
    for (int u = 0; u < A; u++) {
      s_off[u] = o;
      o += 2 + 4 * p.deg[u];
    }
  }
  __syncthreads();
  uint32_t* wb = sbin + (size_t)warp * 32 * d;
  uint32_t* ws = ssign + warp * 32;
  uint64_t* wq = qx + (size_t)warp * 32 * A;
  uint16_t* wt = qtu + (size_t)warp * 32 * A;
  const int64_t per = ((p.n + gridDim.x - 1) / gridDim.x + 31) / 32 * 32;
  const int64_t c0 = (int64_t)blockIdx.x * per;
  const int64_t c1 = min(p.n, c0 + per);
  const int64_t ngroups = c1 > c0 ? (c1 - c0 + 31) / 32 : 0;
  for (int it = 0; it < c.fill_groups; it++) {
    const int64_t g = warp + (int64_t)W * it;
    cached_group<A, true>(p, c, c0 + g * 32, g < ngroups ? c1 : c0, s_coef, s_off, cx, cdata, wb, ws, wq, wt);
  }
  __syncthreads();
  for (int64_t g = warp + (int64_t)W * c.fill_groups; g < ngroups; g += W)
    cached_group<A, false>(p, c, c0 + g * 32, c1, s_coef, s_off, cx, cdata, wb, ws, wq, wt);
}

size_t cached_smem_bytes(int A, int d, int row_len, int log2s, int warps) {
  const size_t S = (size_t)1 << log2s;
  size_t b = (size_t)d * row_len * 8 + (size_t)A * S * 8 + (size_t)A * S * d * 4 + (size_t)warps * 32 * d * 4 +
             (size_t)warps * 32 * 4 + 4 + (size_t)warps * 32 * A * 8 + (size_t)warps * 32 * A * 2;
  return (b + 15) & ~(size_t)15;
}

template <int A>
cudaError_t launch_cached(const UpdArgs& a, int grid, int threads, size_t smem, CacheLayout c, cudaStream_t st) {
  auto kern = k_update_cached<A>;
  cudaError_t e = allow_dynamic_smem((const void*)kern);
  if (e != cudaSuccess) return e;
  kern<<<grid, threads, smem, st>>>(a, c);
  count_launch();
  return cudaGetLastError();
}

__global__ void k_merge(unsigned long long* dst, const unsigned long long* src, int64_t count) {
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += step) dst[i] += src[i];
}

// SK_WARP_AGG=1 turns on the warp aggregation of shared-memory counter updates (off by
// default: on GB300 it measured 2.4-4x slower than plain shared-memory atomics for
// 1- and 2-attribute Zipf(1.1 and 1.4) relations with m = 256..4096).
bool warp_agg_enabled() {
  const char* v = std::getenv("SK_WARP_AGG");
  return v && v[0] == '1';
}

// Tuning knobs (environment): SK_UPDATE_CACHE=1 enables the hot-key cached kernel
// (off by default: on the Zipf(1.1) star fact table it measured slower than the plain
// kernel, 14.5 vs 13.8 ms per 1e8 tuples), SK_CACHE_LOG2S sets its table size per
// attribute (default 2^8 slots).
bool cache_disabled() {
  const char* v = std::getenv("SK_UPDATE_CACHE");
  return !(v && v[0] == '1');
}

int cache_log2s() {
  const char* v = std::getenv("SK_CACHE_LOG2S");
  const int x = v ? std::atoi(v) : 8;
  return x < 4 ? 4 : (x > 12 ? 12 : x);
}

// Key tables (declared domains): SK_KEY_TABLE=0 never uses them, =1 uses them whenever
// the domains allow it (tests), otherwise (default) when the domains are small against the
// batch (sum of domains * 4 <= tuples * attributes) and the relation's sketch is at most
// 32 MiB.  SK_KEY_TABLE_MAX_MB caps the table (default 1024 MiB).
int key_table_mode() {
  const char* v = std::getenv("SK_KEY_TABLE");
  if (!v || !v[0]) return 2;
  return v[0] == '0' ? 0 : (v[0] == '1' ? 1 : 2);
}

// Share of L2 for the counters one per-tuple update pass writes (SK_ROW_PASS_MB, default
// 64 MiB, half of GB300's L2; 0 = never split the rows).  8 x 1e7 rows into 16 x 2^20
// counters (128 MiB per relation): one pass 22.9 ms, two passes of 64 MiB 19.3 ms, three
// of 43 MiB 23.6 ms, four of 32 MiB 27.5 ms (each pass reads the keys again).
size_t row_pass_bytes() {
  const char* v = std::getenv("SK_ROW_PASS_MB");
  const long long x = v ? std::atoll(v) : 64;
  return (size_t)(x < 0 ? 0 : x) << 20;
}

size_t key_table_max_bytes() {
  const char* v = std::getenv("SK_KEY_TABLE_MAX_MB");
  const long long x = v ? std::atoll(v) : 1024;
  return (size_t)(x < 0 ? 0 : x) << 20;
}

// The two paths below read a batch's keys twice.  Columns in host memory (mapped or managed), whose
// every read crosses the link, stay with the ones that read them once.
bool in_device_memory(const int64_t* cols) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, cols) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice;
}

// 24-byte key records of the declared domains, or of the found ones.
cudaError_t launch_table_l24(const UpdArgs& a, const TabArgs& t, const FoundDomains* found, int grid, cudaStream_t st,
                             const WeightSample& ws = {}) {
  auto kern = all_deg1(a) ? k_key_table_l24<true> : k_key_table_l24<false>;
  const size_t smem = (size_t)a.d * a.row_len * sizeof(uint64_t);
  const cudaError_t e = fit_dynamic_smem((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<grid + (ws.w ? 1 : 0), 256, smem, st>>>(a, t, found, ws);
  count_launch();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Batches whose domains were not declared.  Hashing every tuple costs 36 a Horner steps for nine
// rows; most key columns are dense codes, for which the tables serve as well as declared
// domains do, but only the data tells.  So, without the host waiting for it: k_dom_probe looks at
// 1024 tuples (sparse keys, and domains too wide to pay for, are seen there and the scan is spared);
// k_dom_scan finds each column's largest key; and either the tables and both phases of the partitioned
// update run, or the per-tuple update does: the kernels of the other way return at once on the flag.
// Counters are the same either way.
//
// What either way costs (UndeclaredCost), in picoseconds per tuple, fitted to n = 2^22, 1e7 and 3e7
// tuples of 2, 3 and 5 columns, d = 5 and 9, m = 2^16, keys uniform or Zipf over n / 64 to n / 5:
//   hashing        2 a d + 1.6 d + 3
//   tables         1.4 d (2.2 d with weights), and per column a gather: 4.5 from L1 to 7 from L2
//                  and 20 more beyond L2, which holds about 80 MB of records (both dies keep what both
//                  read); how many go there, the share of distinct keys in the sample tells: for
//                  uniform keys (all distinct) the records' share beyond 80 MB, for Zipf exponents of 0.8
//                  (0.9 distinct) and 1 (0.7) about 0.38 and 0.25 of that
//                  weights that no item holds cost 2.9 d, or when the batch goes straight to the
//                  counters (add_direct) 6 d + 2.2 a in place of the 2.2 d and the gathers
//   and per batch  2.3 d + 4 per key to build, and 30 us beyond what turning back to hashing costs
// Without it every dense batch took the tables: 3e7 tuples of five uniform columns over 6e6 keys, d = 5,
// 4800 us against 1884 for hashing (d = 9: 5370 and 3248); over 4.7e5 keys 1283 (1454).
// ---------------------------------------------------------------------------
struct UndeclaredCost {
  float n;
  int a, d;
  bool weighted, always;

  // gain in ps per tuple with `keys` records in the tables, the columns' spreads and the share of
  // weights that no item holds
  __host__ __device__ float gain(float keys, const float* spread, float heavy) const {
    const float beyond = fmaxf(0.f, 1.f - 80e6f / fmaxf(24.f * keys, 1.f));
    const bool direct = heavy > 0.7f;
    float t = (keys * (2.3f * d + 4.f) + 30e6f) / n;
    t += direct ? 6.f * d + 2.2f * a : (weighted ? 2.2f : 1.4f) * d + 2.9f * d * heavy;
    for (int u = 0; u < a; u++) {
      const float l2 = fminf(fmaxf(spread[u] * 2.f - 1.f, 0.f), 1.f);
      float far = fmaxf((spread[u] - 0.3f) * 0.62f, 0.f);
      if (spread[u] > 0.965f) far = fminf(1.f, far + (spread[u] - 0.965f) * 30.f);   // uniform: 0.985 and up
      t += (direct ? 0.f : 4.5f + 2.5f * l2) + 20.f * beyond * far;
    }
    return 2.f * a * d + 1.6f * d + 3.f - t;
  }
  // scanned: 1.2 a of the tables' cost are the scan, which is behind
  __device__ bool pays(const FoundDomains& f, uint64_t cap, bool scanned) const {
    float keys = 0.f;
    bool dense = true;
    for (int u = 0; u < a; u++) {
      const unsigned long long top = *(const volatile unsigned long long*)&f.top[u];
      dense = dense && top < cap;
      keys += (float)top + 1.f;
    }
    return dense && (always || gain(keys, f.spread, f.far) + (scanned ? 1.2f * a : 0.f) > 0.f);
  }
};

__global__ void __launch_bounds__(1024) k_dom_probe(UpdArgs p, FoundDomains* f, uint64_t cap, UndeclaredCost cost,
                                                    int64_t wmax) {
  __shared__ uint32_t s_seen[5][2048];   // 65536 bits per column
  const int64_t i = p.n / 1024 * threadIdx.x;
  uint64_t key[5];
#pragma unroll
  for (int u = 0; u < 5; u++) key[u] = u < p.a ? (uint64_t)p.cols[(int64_t)u * p.stride + i] : 0ull;
  const int64_t w = p.w ? __ldg(p.w + i) : 0;
  for (int k = threadIdx.x; k < 5 * 2048; k += 1024) (&s_seen[0][0])[k] = 0;
  if (threadIdx.x < 5) f->top[threadIdx.x] = 0;
  bool dense = true;
#pragma unroll
  for (int u = 0; u < 5; u++) dense = dense && key[u] < cap;
  dense = __syncthreads_and(dense);
  if (!dense) {
    if (threadIdx.x == 0) f->go = 0;
    return;
  }
  bool fresh[5];
#pragma unroll
  for (int u = 0; u < 5; u++) {
    const uint32_t h = ((uint32_t)key[u] * 2654435761u) >> 16;
    fresh[u] = u < p.a && !(atomicOr(&s_seen[u][h >> 5], 1u << (h & 31u)) >> (h & 31u) & 1u);
    if (u < p.a) {
      const uint32_t top = __reduce_max_sync(0xffffffffu, (uint32_t)key[u]);   // cap is at most 2^31
      if ((threadIdx.x & 31u) == 0) atomicMax(&f->top[u], (unsigned long long)top);
    }
  }
#pragma unroll
  for (int u = 0; u < 5; u++) {
    const int distinct = __syncthreads_count(fresh[u]);
    if (threadIdx.x == 0) f->spread[u] = distinct / 1024.f;
  }
  const int far = __syncthreads_count(w > wmax || w < -wmax);
  if (threadIdx.x == 0) {
    f->far = far / 1024.f;
    f->go = cost.pays(*f, cap, false) ? 1 : 0;
    f->blocks = 0;
  }
}

template <int A>
__global__ void __launch_bounds__(256) k_dom_scan(UpdArgs p, FoundDomains* f, uint64_t cap,
                                                  UndeclaredCost cost) {
  __shared__ unsigned long long s_top[A];
  if (!f->go) return;
  if (threadIdx.x < A) s_top[threadIdx.x] = 0;
  __syncthreads();
  uint64_t top[A];
#pragma unroll
  for (int u = 0; u < A; u++) top[u] = 0;
  const int64_t step = (int64_t)gridDim.x * 256;
  constexpr int U = 4;   // tuples in flight per thread
  for (int64_t i0 = (int64_t)blockIdx.x * 256 + threadIdx.x; i0 < p.n; i0 += U * step) {
    uint64_t k[U][A];
#pragma unroll
    for (int t = 0; t < U; t++)
#pragma unroll
      for (int u = 0; u < A; u++)
        k[t][u] = i0 + t * step < p.n ? (uint64_t)ld_key_stream(p.cols + (int64_t)u * p.stride + i0 + t * step) : 0ull;
#pragma unroll
    for (int t = 0; t < U; t++)
#pragma unroll
      for (int u = 0; u < A; u++) top[u] = k[t][u] > top[u] ? k[t][u] : top[u];
  }
#pragma unroll
  for (int u = 0; u < A; u++) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const uint64_t v = __shfl_xor_sync(0xffffffffu, top[u], o);
      top[u] = v > top[u] ? v : top[u];
    }
    if ((threadIdx.x & 31u) == 0) atomicMax(&s_top[u], (unsigned long long)top[u]);
  }
  __syncthreads();
  if (threadIdx.x < A) {
    atomicMax(&f->top[threadIdx.x], s_top[threadIdx.x]);
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0 && atomicAdd(&f->blocks, 1) == (int)gridDim.x - 1) {   // the last CTA decides
    __threadfence();
    f->go = cost.pays(*f, cap, true) ? 1 : 0;
  }
}

// *done = false (nothing launched) unless the batch is one the partitioned update would take with
// declared domains, of two attributes or more and at least 2^22 tuples, and keys as kind as can be (few
// and skewed) would gain 25 us: the probe and the kernels that return cost others 16 to 25 us (2^22 tuples
// of two columns, d = 5: 145 -> 170; at 1e7 5 %), and a key beyond the tables that no sample shows also
// the scan (1e7 tuples of two columns 323 -> 371).  Five columns, m = 2^16, d = 9: dense keys 254 against 458
// us at 2^22 tuples and 670 against 1810 at 2^24 (1e7 tuples 1080 -> 538 us).  One attribute is left to update_warp_key.  Captured streams keep the per-tuple
// update, which allocates nothing.
cudaError_t update_undeclared(const UpdArgs& a0, bool pow2, bool use_smem, int sms, cudaStream_t st, bool* done) {
  *done = false;
  const int64_t n = a0.n;
  if (part_update_mode() == 0 || key_table_mode() == 0 || a0.has_dom || !pow2 || use_smem || a0.a < 2 || a0.a > 5 ||
      a0.d > 9 || a0.m < 1024 || a0.m > 65536 || n < std::max<int64_t>((int64_t)a0.m * 16, undeclared_least()))
    return cudaSuccess;
  cudaStreamCaptureStatus cap_st = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(st, &cap_st);
  if (e != cudaSuccess || cap_st != cudaStreamCaptureStatusNone || !in_device_memory(a0.cols)) return e;
  // records per attribute: a quarter of the tuples (the rule for declared domains), within the
  // tables' limit
  const int64_t cap =
      std::min<int64_t>({n / 4, (int64_t)(key_table_max_bytes() / 24) / a0.a, ((int64_t)1 << 31) - 1});
  if (cap < 1) return cudaSuccess;
  const UndeclaredCost cost = {(float)n, a0.a, a0.d, a0.w != nullptr, undeclared_least_given()};
  const float kind[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
  if (!cost.always && (float)n * cost.gain(0.f, kind, 0.f) < 25e6f) return cudaSuccess;
  const int64_t W = part_window(n, (int64_t)1 << 26);
  const size_t b_part = part_staging_bytes(a0.d, W, sms, a0.w != nullptr), b_tab = ((size_t)a0.a * cap * 24 + 255) & ~(size_t)255;
  char* buf = nullptr;
  if (pool_malloc_async((void**)&buf, b_part + b_tab + 256, st) != cudaSuccess) {
    cudaGetLastError();   // no room: hash per tuple
    return cudaSuccess;
  }
  *done = true;
  FoundDomains* f = (FoundDomains*)(buf + b_part + b_tab);
  UpdArgs a = a0;
  TabArgs t;
  int off = 0;
  for (int u = 0; u < a.a; u++) {
    a.dom[u] = cap;
    t.base[u] = u * cap;
    t.off[u] = off;
    off += 2 + 4 * a.deg[u];
  }
  t.base[a.a] = a.a * cap;
  t.rvec = 2;
  t.narrow = 1;
  t.tbl = (uint32_t*)(buf + b_part);
  WeightSample ws = {};
  e = weight_sample(a, 2, buf, sms, (int64_t)1 << 26, &ws);
  if (e != cudaSuccess) {
    cudaFreeAsync(buf, st);
    return e;
  }
  k_dom_probe<<<1, 1024, 0, st>>>(a, f, (uint64_t)cap, cost, ws.wmax);
  const int grid = sms * 8;
  switch (a.a) {
    case 2: k_dom_scan<2><<<grid, 256, 0, st>>>(a, f, (uint64_t)cap, cost); break;
    case 3: k_dom_scan<3><<<grid, 256, 0, st>>>(a, f, (uint64_t)cap, cost); break;
    case 4: k_dom_scan<4><<<grid, 256, 0, st>>>(a, f, (uint64_t)cap, cost); break;
    default: k_dom_scan<5><<<grid, 256, 0, st>>>(a, f, (uint64_t)cap, cost); break;
  }
  count_launch(2);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_table_l24(a, t, f, sms * 32, st, ws);
  if (e == cudaSuccess) e = run_partitioned(a, t, 2, buf, sms, st, nullptr, nullptr, (int64_t)1 << 26, &f->go);
  // a fixed grid, whose CTAs return at once in the dense case: 1e7 dense tuples 538 us in all with
  // 32 CTAs per SM, 552 with a tuple per thread; sparse ones measured the same
  const size_t cb = (size_t)a0.d * a0.row_len * sizeof(uint64_t);
  if (e == cudaSuccess)
    e = dispatch_a<true, false>(a0, (int)std::min<int64_t>((n + 255) / 256, (int64_t)sms * 32), cb, st, &f->go);
  const cudaError_t ef = cudaFreeAsync(buf, st);
  return e != cudaSuccess ? e : ef;
}

}  // namespace

// CTAs for the shared-memory sub-sketch kernels: 16 tuples per thread (4096 per CTA of 256),
// or for small batches up to one CTA per SM with at least max(256, m) tuples each, so that a
// CTA's flush of its m-counter rows stays below its own counter updates and a batch of a few
// thousand tuples does not run on a handful of SMs.
int64_t smem_grid_want(int64_t n, int64_t m, int sms) {
  const int64_t per = std::max<int64_t>(256, std::min<int64_t>(m, 4096));
  return std::max<int64_t>((n + 4095) / 4096, std::min<int64_t>(sms, (n + per - 1) / per));
}

sk_status launch_update(sk_set* s, int relation, int64_t n, const int64_t* cols, int64_t col_stride,
                        const int64_t* weights, const int64_t* domain, cudaStream_t st) {
  const RelPlan& rp = s->rel[relation];
  UpdArgs a;
  a.cols = cols;
  a.stride = col_stride;
  a.w = weights;
  a.n = n;
  a.ctr = (unsigned long long*)(s->counters + (size_t)relation * s->d * s->m);
  a.coef = rp.d_coef;
  a.row_len = rp.coef_row_len;
  a.d = s->d;
  a.a = rp.a;
  for (int t = 0; t < kMaxAttrs; t++) a.deg[t] = rp.deg[t];
  a.m = (uint64_t)s->m;
  a.mrec = ~0ull / a.m;
  a.has_dom = domain != nullptr;
  for (int t = 0; t < kMaxAttrs; t++) a.dom[t] = (domain && t < rp.a) ? domain[t] : 0;
  a.status = s->d_status;
  a.agg = warp_agg_enabled() ? 1 : 0;
  a.s16 = 0;
  const bool pow2 = (s->m & (s->m - 1)) == 0;
  const size_t coef_bytes = (size_t)s->d * rp.coef_row_len * sizeof(uint64_t);
  const size_t sub_bytes = (size_t)s->d * (size_t)s->m * sizeof(int);
  const int sms = sm_count();
  if (coef_bytes > 200 * 1024) return SK_ERR_INVALID_ARG;   // hash table must fit in shared memory
  const bool use_smem = coef_bytes + sub_bytes <= 200 * 1024 && (int64_t)(s->d * s->m) <= n;
  cudaError_t e;
  const int ktm = key_table_mode();
  if (domain && ktm != 0 && n > 0 && rp.a >= 1 && s->d <= SK_MAX_ROWS && s->m <= (1ll << 30)) {
    TabArgs t;
    bool fits = true;
    int64_t total = 0;
    int off = 0;
    for (int u = 0; u < rp.a; u++) {
      if (domain[u] < 1 || domain[u] > (1ll << 31)) fits = false;
      t.base[u] = total;
      t.off[u] = off;
      total += fits ? domain[u] : 0;
      off += 2 + 4 * rp.deg[u];
    }
    t.base[rp.a] = total;
    t.narrow = s->m <= 65536 && s->d <= 32;
    t.rvec = key_record_vectors(s->d, t.narrow);
    // The two-phase partitioned update (power-of-two 1024 <= m <= 2^16, d <= 14,
    // at most 5 attributes, sketch too large for one CTA's shared memory, at least 16 tuples
    // per counter of a row, fewer than 2^32 table records) takes 24-byte records for d <= 9
    // (the 32-byte 20-bit lane ones with SK_PART_RECORD=32) and the narrow 32-byte format
    // otherwise.
    bool part = part_update_mode() != 0 && pow2 && rp.a <= 5 && !use_smem && s->m >= 1024 &&
                s->m <= 65536 && s->d <= 14 && n >= (int64_t)s->m * 16 && total < ((int64_t)1 << 32);
    const int part_fmt = s->d <= 9 ? (part_record_bytes() == 32 ? 0 : 2) : 1;
    // The wide partitioned update (unit weights, power-of-two 2^17 <= m <= 2^24, d <= 16, at most
    // 5 attributes, at least m tuples, a sketch larger than 32 MiB, whose counter updates would
    // leave L2) takes the wide records (one 32-bit word per row).
    const size_t sketch_bytes = (size_t)s->d * (size_t)s->m * sizeof(int64_t);
    const int pum = part_update_mode();
    bool wide = pum != 0 && pow2 && weights == nullptr && rp.a <= 5 && s->m >= ((int64_t)1 << 17) &&
                s->m <= ((int64_t)1 << 24) && s->d <= kWideMaxRows && total < ((int64_t)1 << 32) &&
                (pum == 2 || (n >= (int64_t)s->m && sketch_bytes > ((size_t)32 << 20)));
    // Automatic choice: the tables replace per-tuple hashing by gathers, which pays when
    // the domains are small against a batch of at least 2^16 tuples (below that the table's
    // launch and allocation cost more than the hashing) and the counter updates hit L2 (for a sketch
    // much larger than L2 the update is bound by its atomics either way and the gathers
    // only add traffic: 27.7 vs 24.7 ms for 8 x 1e7 rows into 128 MB sketches), unless the
    // wide partitioned update takes the batch: it replaces those atomics.
    const bool worth = ktm == 1 || (n >= ((int64_t)1 << 16) && total * 4 <= n * (int64_t)rp.a &&
                                    (sketch_bytes <= ((size_t)32 << 20) || wide));
    // k_wide_sort reads the keys once per group of eight rows
    const bool sorted_parts = wide && s->m <= ((int64_t)kSortMaxParts << 15) &&
                              (s->d <= kSortRows || in_device_memory(cols));
    void* staging = nullptr;
    if (fits && worth && total > 0 && part) {
      e = pool_malloc_async(&staging, part_staging_bytes(s->d, part_window(n, part_most(weights)), sms, weights != nullptr),
                            st);
      if (e != cudaSuccess) {
        cudaGetLastError();   // no room for the planes: single-phase update
        staging = nullptr;
        part = false;
      }
    } else if (fits && worth && total > 0 && wide) {
      e = pool_malloc_async(&staging,
                            sorted_parts ? sort_layout(s->d, s->m, wide_window(n)).bytes
                                         : wide_layout(s->d, s->m, wide_window(n)).total,
                            st);
      if (e != cudaSuccess) {
        cudaGetLastError();   // no room for the planes: per-tuple update
        staging = nullptr;
        wide = false;
      }
    } else {
      wide = false;
    }
    if (part) t.rvec = 2;
    const size_t bytes = (size_t)total * (part && part_fmt == 2 ? 24 : (size_t)t.rvec * 16);
    if (fits && worth && total > 0 && bytes <= key_table_max_bytes()) {
      void* buf = nullptr;
      e = pool_malloc_async(&buf, bytes, st);
      if (e != cudaSuccess) {
        cudaGetLastError();   // not enough memory for the table: hash per tuple instead
        if (staging) cudaFreeAsync(staging, st);
      } else {
        t.tbl = (uint32_t*)buf;
        a.smem_wmax = 0;
        const bool d1 = all_deg1(a);
        const int bgrid = (int)std::min<int64_t>((total + 255) / 256, (int64_t)sms * 32);
        WeightSample ws = {};
        e = part ? weight_sample(a, part_fmt, staging, sms, part_most(weights), &ws) : cudaSuccess;
        if (e == cudaSuccess && part && part_fmt == 2) {
          e = launch_table_l24(a, t, nullptr, bgrid, st, ws);
        } else if (e == cudaSuccess) {
          auto kb = (part && part_fmt == 0) ? (d1 ? k_key_table_l20<true> : k_key_table_l20<false>)
                    : pow2 ? (d1 ? k_key_table<true, true> : k_key_table<true, false>)
                           : (d1 ? k_key_table<false, true> : k_key_table<false, false>);
          e = fit_dynamic_smem((const void*)kb, coef_bytes);
          if (e == cudaSuccess) {
            kb<<<bgrid + (ws.w ? 1 : 0), 256, coef_bytes, st>>>(a, t, ws);
            count_launch();
            e = cudaGetLastError();
          }
        }
        if (e == cudaSuccess && part) {
          e = run_partitioned(a, t, part_fmt, staging, sms, st, nullptr, nullptr, part_most(weights));
        } else if (e == cudaSuccess && wide) {
          e = sorted_parts ? run_wide_sorted(a, t, staging, sms, st) : run_wide_partitioned(a, t, staging, sms, st);
        } else if (e == cudaSuccess) {
          if (use_smem) {
            const int per_sm = sub_bytes <= 48 * 1024 ? 4 : (sub_bytes <= 100 * 1024 ? 2 : 1);
            const int64_t want = smem_grid_want(n, s->m, sms);
            const int grid = (int)std::min<int64_t>(std::max<int64_t>(want, 1), (int64_t)sms * per_sm);
            const int64_t tpc = (n + (int64_t)grid * 256 - 1) / ((int64_t)grid * 256) * 256;
            a.smem_wmax = (int64_t)0x7fffffff / std::max<int64_t>(tpc, 1);
            e = pow2 ? dispatch_tab<true, true>(a, t, grid, sub_bytes, st)
                     : dispatch_tab<false, true>(a, t, grid, sub_bytes, st);
          } else {
            const int grid = (int)std::min<int64_t>((n + 255) / 256, 0x7fffffff);
            e = pow2 ? dispatch_tab<true, false>(a, t, grid, 0, st) : dispatch_tab<false, false>(a, t, grid, 0, st);
          }
        }
        cudaError_t ef = cudaFreeAsync(buf, st);
        if (staging) {
          const cudaError_t es = cudaFreeAsync(staging, st);
          if (ef == cudaSuccess) ef = es;
        }
        return set_status_from_cuda(e != cudaSuccess ? e : ef);
      }
    } else if (staging) {
      cudaFreeAsync(staging, st);
    }
  }
  if (!domain) {
    bool done = false;
    e = update_undeclared(a, pow2, use_smem, sms, st, &done);
    if (done || e != cudaSuccess) return set_status_from_cuda(e);
  }
  const bool cache_ok = !use_smem && pow2 && s->d <= 32 && rp.a >= 1 && rp.a <= 5 && s->m <= (1ll << 30) &&
                        n >= (int64_t)1 << 17 && !cache_disabled();
  if (cache_ok) {
    const int threads = 512, warps = threads / 32;
    int log2s = cache_log2s();
    size_t smem = cached_smem_bytes(rp.a, s->d, rp.coef_row_len, log2s, warps);
    while (log2s > 6 && smem > 200 * 1024) smem = cached_smem_bytes(rp.a, s->d, rp.coef_row_len, --log2s, warps);
    if (smem <= 200 * 1024) {
      const int per_sm = smem <= 110 * 1024 ? 2 : 1;
      const int grid = (int)std::min<int64_t>((int64_t)sms * per_sm, std::max<int64_t>(1, n / (threads * 8)));
      CacheLayout c{log2s, 8};
      a.smem_wmax = 0;
      switch (rp.a) {
        case 1: e = launch_cached<1>(a, grid, threads, smem, c, st); break;
        case 2: e = launch_cached<2>(a, grid, threads, smem, c, st); break;
        case 3: e = launch_cached<3>(a, grid, threads, smem, c, st); break;
        case 4: e = launch_cached<4>(a, grid, threads, smem, c, st); break;
        default: e = launch_cached<5>(a, grid, threads, smem, c, st); break;
      }
      return set_status_from_cuda(e);
    }
  }
  if (use_smem) {
    const size_t smem = coef_bytes + sub_bytes;
    const int per_sm = smem <= 48 * 1024 ? 4 : (smem <= 100 * 1024 ? 2 : 1);
    int64_t want = smem_grid_want(n, s->m, sms);
    int grid = (int)std::min<int64_t>(std::max<int64_t>(want, 1), (int64_t)sms * per_sm);
    const int64_t tpc = (n + (int64_t)grid * 256 - 1) / ((int64_t)grid * 256) * 256;
    a.smem_wmax = (int64_t)0x7fffffff / std::max<int64_t>(tpc, 1);
    e = pow2 ? dispatch_a<true, true>(a, grid, smem, st) : dispatch_a<false, true>(a, grid, smem, st);
  } else {
    // Counters in global memory.  When the relation's d x m int64 counters exceed the share
    // of L2 given by row_pass_bytes(), the rows are split into passes over the whole batch
    // (each pass hashes only its rows; the keys are read once per pass), so that the
    // counter updates of a pass stay in L2.
    a.smem_wmax = 0;
    const size_t row_bytes = (size_t)s->m * sizeof(int64_t);
    const size_t budget = row_pass_bytes();
    int rows = s->d;
    if (budget > 0 && (size_t)s->d * row_bytes > budget) rows = (int)std::max<size_t>(1, budget / row_bytes);
    const int passes = (s->d + rows - 1) / rows;
    rows = (s->d + passes - 1) / passes;   // even split
    e = cudaSuccess;
    for (int r0 = 0; r0 < s->d && e == cudaSuccess; r0 += rows) {
      UpdArgs b = a;
      b.d = std::min(rows, s->d - r0);
      b.coef = a.coef + (size_t)r0 * rp.coef_row_len;
      b.ctr = a.ctr + (size_t)r0 * s->m;
      const size_t cb = (size_t)b.d * rp.coef_row_len * sizeof(uint64_t);
      e = pow2 ? dispatch_a<true, false>(b, 0, cb, st) : dispatch_a<false, false>(b, 0, cb, st);
    }
  }
  return set_status_from_cuda(e);
}

sk_status launch_merge(int64_t* dst, const int64_t* src, int64_t count, cudaStream_t st) {
  if (count == 0) return SK_OK;
  const int grid = (int)std::min<int64_t>((count + 255) / 256, (int64_t)sm_count() * 8);
  k_merge<<<grid, 256, 0, st>>>((unsigned long long*)dst, (const unsigned long long*)src, count);
  count_launch();
  return set_status_from_cuda(cudaGetLastError());
}

namespace {

using ViewPlanesKernel = void (*)(UpdArgs, TabArgs, ViewPlanes);

ViewPlanesKernel view_planes_kernel(int A) {   // two attributes or more: one has one view
  switch (A) {
    case 2: return k_view_planes<2>;
    case 3: return k_view_planes<3>;
    case 4: return k_view_planes<4>;
    default: return k_view_planes<5>;
  }
}

// Bytes of a tile, and of the planes of a window of W tuples.
int64_t view_tile_bytes(int A, int d) { return (int64_t)kViewTile * 2 * A * d + kViewTile / 8 * (A * d + 1); }

size_t view_plane_bytes(int A, int d, int64_t W) {
  return (size_t)((W + kViewTile - 1) / kViewTile) * (size_t)view_tile_bytes(A, d);
}

// Tuples per window: planes near 3 GiB at most (the library's pool keeps 4 GiB between calls), a
// batch cut into equal windows.
int64_t view_window(int A, int d, int64_t n) {
  const int64_t most = ((int64_t)3 << 30) / view_tile_bytes(A, d) * kViewTile;
  const int64_t wins = (n + most - 1) / most;
  return part_window((n + wins - 1) / wins);
}

// Whether the planes cost less than one view at a time.  Per tuple the planes take about A (2.7 +
// 0.77 d) + 2.3 d ps whatever the views, a view of s attributes 8 + 2.2 d, or 4.75 s where its gathers
// bind (n = 5e7, d = 3 and 9); and the planes save 120 us of launches, zeroing and flushing.  Three views
// or more always gain; two of five attributes lose above 9e6 tuples (m = 2^16, d = 9, 2e7 tuples: 1406
// against 1240 us, 5e7: 3430 against 2770) and two of four above 3e7 (5e7: 2940 against 2700).
bool planes_pay(int A, int d, int nv, const uint32_t* amask, int64_t n) {
  double views = 0.0;
  for (int v = 0; v < nv; v++) {
    const int s = __builtin_popcount(amask[v]);
    if (s) views += std::max(8.0 + 2.2 * d, 4.75 * s);
  }
  return (double)n * (A * (2.7 + 0.77 * d) + 2.3 * d - views) < 120e6;
}

// Both kernels over every window; planes: view_plane_bytes.
cudaError_t run_views(const UpdArgs& a, const TabArgs& t, const ViewMasks& vm, const ViewCounters& vc, void* planes,
                      int64_t W, int sms, cudaStream_t st) {
  ViewPlanesKernel make = view_planes_kernel(a.a);
  int per_sm = 0;
  cudaError_t e = cudaFuncSetAttribute((const void*)make, cudaFuncAttributePreferredSharedMemoryCarveout, 0);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, make, 256, 0);
  if (e != cudaSuccess) return e;
  const int64_t full_grid = (int64_t)sms * std::max(1, per_sm);
  int logL = 0;
  while (logL < 15 && ((int64_t)1 << logL) < (int64_t)a.m) logL++;
  const int S = (int)(a.m >> logL);
  const size_t smem = (size_t)4 << logL;
  auto accum = S == 2 ? k_view_accum<true> : k_view_accum<false>;
  e = allow_dynamic_smem((const void*)accum);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, accum, 1024, smem);
  const int64_t slots = (int64_t)sms * std::max(1, per_sm), units = (int64_t)S * a.d * vm.nv;
  ViewPlanes q;
  q.tiles = (uint8_t*)planes;
  q.stride = view_tile_bytes(a.a, a.d);
  for (int64_t i0 = 0; i0 < a.n && e == cudaSuccess; i0 += W) {
    q.cnt = std::min(W, a.n - i0);
    for (int u = 0; u < 5; u++) q.col[u] = u < a.a ? a.cols + (int64_t)u * a.stride + i0 : nullptr;
    make<<<(unsigned)std::min<int64_t>((q.cnt + 255) / 256, full_grid), 256, 0, st>>>(a, t, q);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) break;
    const int nr = (int)part_ranges(q.cnt * units, units, slots, (q.cnt + kViewTile - 1) / kViewTile, 0.0);
    accum<<<(unsigned)(units * nr), 1024, smem, st>>>(q, vm, vc, a.a, a.d, (int64_t)a.m, logL, nr);
    count_launch();
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace

// One bit per tuple: all of the relation's keys inside their declared domains (a tuple with a
// key outside is reported and left out of every view).
__global__ void __launch_bounds__(256) k_valid_bits(UpdArgs p, uint32_t* bits) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool ok = i < p.n;
  if (ok)
    for (int u = 0; u < p.a; u++) {
      const int64_t key = ld_key_stream(p.cols + (int64_t)u * p.stride + i);
      if ((uint64_t)key >= (uint64_t)p.dom[u]) ok = false;
    }
  if (i < p.n && !ok) record(p.status, SK_ERR_KEY_OUT_OF_DOMAIN);
  const uint32_t b = __ballot_sync(0xffffffffu, ok);
  if ((threadIdx.x & 31u) == 0 && i < p.n) bits[i >> 5] = b;
}

// Sub-query family views of one relation through the two-phase partitioned update (see
// run_partitioned): when every attribute has exactly one sign slot, a view's sign is the
// product of its attributes' slot-0 signs and its bin the sum of their bins, so one 24-byte
// key table over the relation's attributes (built once) serves every view.  Large batches go
// through the planes of run_views; else each view's counters get both phases over the view's
// attributes (a validity pass over all of the relation's keys first: a tuple is left out of
// every view when any key is outside its domain, as in the per-tuple view update).  Taken for unit weights with declared
// domains, power-of-two 1024 <= m <= 2^16, d <= 9, views of at most 5 attributes, at least
// 16 m tuples and views too large for one CTA's shared memory; *done = false (nothing
// launched) otherwise, and the caller runs its per-tuple view update.
sk_status family_partitioned_update(const UpdArgs& a, int nv, const uint32_t* amask, const unsigned long long* jmask,
                                    unsigned long long* const* ctr, cudaStream_t st, bool* done) {
  *done = false;
  const int64_t n = a.n;
  const bool pow2 = (a.m & (a.m - 1)) == 0;
  if (part_update_mode() == 0 || key_table_mode() == 0 || !a.has_dom || a.w != nullptr || !pow2 || a.m < 1024 ||
      a.m > 65536 || a.d > 9 || a.a < 1 || a.a > kMaxAttrs || n < (int64_t)a.m * 16 ||
      (size_t)a.d * a.m * sizeof(int) <= 200 * 1024 || !all_deg1(a))
    return SK_OK;
  TabArgs t;
  int64_t total = 0;
  int off = 0;
  for (int u = 0; u < a.a; u++) {
    if (a.dom[u] < 1 || a.dom[u] > (1ll << 31)) return SK_OK;
    t.base[u] = total;
    t.off[u] = off;
    total += a.dom[u];
    off += 2 + 4 * a.deg[u];
  }
  t.base[a.a] = total;
  t.narrow = 1;
  t.rvec = 2;
  if (total >= ((int64_t)1 << 32) || (key_table_mode() != 1 && total * 4 > n * (int64_t)a.a)) return SK_OK;
  for (int v = 0; v < nv; v++) {
    // slot i is attribute i's only slot: a view's signs are those of its attributes
    if (__builtin_popcount(amask[v]) > 5 || (unsigned long long)amask[v] != jmask[v]) return SK_OK;
  }
  const size_t tbytes = (size_t)total * 24;
  if (tbytes > key_table_max_bytes()) return SK_OK;
  const int sms = sm_count();
  void* tbl = nullptr;
  void* staging = nullptr;
  if (pool_malloc_async(&tbl, tbytes, st) != cudaSuccess) {
    cudaGetLastError();
    return SK_OK;
  }
  // All views from one set of planes: for two views or more of a relation of at most five attributes,
  // from 3 2^19 tuples (one view at a time against the planes: 15 views of four attributes, m = 2^16,
  // d = 9, 2^21 tuples 1.17 against 0.52 ms; three views of two 0.37 against 0.16).  They would pay below
  // that too, but a test holds 1 048 607 tuples to the launches of one view at a time.
  if (nv >= 2 && a.a >= 2 && a.a <= 5 && n >= ((int64_t)3 << 19) && planes_pay(a.a, a.d, nv, amask, n)) {
    ViewMasks vm;
    ViewCounters vc;
    vm.nv = 0;
    for (int v = 0; v < nv; v++)
      if (amask[v]) {
        vc.ctr[vm.nv] = ctr[v];
        vm.mask[vm.nv++] = (uint8_t)amask[v];
      }
    const int64_t W = view_window(a.a, a.d, n);
    if (vm.nv > 0 && pool_malloc_async(&staging, view_plane_bytes(a.a, a.d, W), st) == cudaSuccess) {
      *done = true;
      t.tbl = (uint32_t*)tbl;
      cudaError_t e = launch_table_l24(a, t, nullptr, (int)std::min<int64_t>((total + 255) / 256, (int64_t)sms * 32), st);
      if (e == cudaSuccess) e = run_views(a, t, vm, vc, staging, W, sms, st);
      cudaError_t ef = cudaFreeAsync(tbl, st);
      const cudaError_t es = cudaFreeAsync(staging, st);
      if (ef == cudaSuccess) ef = es;
      return set_status_from_cuda(e != cudaSuccess ? e : ef);
    }
    cudaGetLastError();   // no room for the planes: one view at a time
    staging = nullptr;
  }
  const size_t sbytes = part_staging_bytes(a.d, part_window(n), sms);
  const size_t vbytes = (size_t)(n + 31) / 32 * sizeof(uint32_t);
  if (pool_malloc_async(&staging, sbytes + ((vbytes + 255) & ~(size_t)255), st) != cudaSuccess) {
    cudaGetLastError();
    cudaFreeAsync(tbl, st);
    return SK_OK;
  }
  *done = true;
  uint32_t* vbits = (uint32_t*)((char*)staging + sbytes);
  t.tbl = (uint32_t*)tbl;
  cudaError_t e = launch_table_l24(a, t, nullptr, (int)std::min<int64_t>((total + 255) / 256, (int64_t)sms * 32), st);
  if (e == cudaSuccess) {
    k_valid_bits<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a, vbits);
    count_launch();
    e = cudaGetLastError();
  }
  for (int v = 0; v < nv && e == cudaSuccess; v++) {
    UpdArgs av = a;
    TabArgs tv = t;
    const int64_t* colp[5];
    int k = 0;
    for (int u = 0; u < a.a; u++) {
      if (!((amask[v] >> u) & 1u)) continue;
      av.dom[k] = a.dom[u];
      av.deg[k] = a.deg[u];
      tv.base[k] = t.base[u];
      colp[k] = a.cols + (int64_t)u * a.stride;
      k++;
    }
    if (k == 0) continue;
    av.a = k;
    tv.base[k] = total;
    av.ctr = ctr[v];
    e = run_partitioned(av, tv, 2, staging, sms, st, colp, vbits);
  }
  cudaError_t ef = cudaFreeAsync(tbl, st);
  const cudaError_t es = cudaFreeAsync(staging, st);
  if (ef == cudaSuccess) ef = es;
  return set_status_from_cuda(e != cudaSuccess ? e : ef);
}

}  // namespace sk
