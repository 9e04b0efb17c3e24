// Split-precision tensor-core contraction engine (tcgen05, sm_103a).
//
// Each FP64 operand is carried as s integer-valued BF16 slices with one
// power-of-two scale per tensor: x = 2^(e-7) sum_p d_p 2^(-8p), |d_p| <= 128,
// slice p stored as the exact BF16 value d_p 2^(-8p).  A contraction
// sum_k A[m][k] B[n][k] becomes the triangle of slice products p + q <= s-1
// (the products with p + q >= s are below the representation error).  Every
// slice product is exact in FP32, but the tensor core's FP32 accumulation
// does not round to nearest when addends of very different size meet, so
// each level L = p + q <= 3 gets its own tensor-memory accumulator, whose
// values stay exactly representable (multiples of 2^-8L below 2^(24-8L))
// because it is drained into 64-bit fixed-point registers every 256 to 900 K;
// the levels >= 4 share a fifth, rounded accumulator that a tile keeps to its
// end.  What that rounds off grows with the tile's K steps n: at most
// 22 2^-23 5 2^-32 16 n (n + 1) / 2 of the largest digit product at 6 slices; on
// random operands 6e-14 of it at n = 100, 4.8e-13 at 400 and 1.4e-12 at 800, next to
// 1.1e-13, 2.1e-13 and 3.0e-13 that the products left out cost.
//
// Warp roles (608 threads): warp 18 decodes tiles and their terms ahead of the
// others; warp 0 issues one bulk copy per operand tile (all
// s slices of a 128 x 16 A tile, resp. an Ntile x 16 B tile, pre-tiled in
// global memory in the canonical no-swizzle order with the slices interleaved
// per row group; one copy per slab when the A rows are flattened over slabs)
// into a ring of stages; warp 1 issues tcgen05.mma (M = 128, N = Ntile <= 96,
// K = 16, FP32 accumulate, A kept in the collector buffer across the products
// of one A slice) and owns the tensor-memory allocation (5 x 96 columns);
// warps 2-17 drain and finish the accumulators (each quadrant of 32 TMEM lanes
// is read by four warps, one per column quarter, 4 columns per load) and write
// the outputs (double-float stores, FP64 atomics or 128-bit fixed-point
// atomics) through up to four output descriptors.  At a drain point the issuer
// queues the next steps' products into the other accumulators before it waits
// for the drain; at a tile's end it issues levels 0..3 first, so that they are
// read while the shared accumulator's products run, and the next tile starts
// with levels 0..3 while that one is read.
//
// What bounds it: a 128 x 96 x 16 product takes 53 clocks here (48 at the
// nominal rate), the 21 of a K step 1118 next to 43 KB of operands arriving, so
// the issuer must add little to that.  It takes 1271 on 96 triples of the no=22
// nv=250 residual (1902 with one divergent thread issuing, double-float sums and
// the tile's ends one after the other): its operands are known to be uniform (4
// instructions per product, not 11), one level is drained at a time, the last
// column tile is trimmed, steps run in sequence (pairs with interleaved A runs
// hold a stage 1000 clocks longer: 158.8 ms for those triples, so 166.9) and the
// next pair's signs are read ahead.  The kernel's code is kept at 88 KB: at 178 KB
// it had outgrown the instruction cache.  Every wait is
// bounded: on timeout the CTA sets an error word that the host turns into
// CC3_ERR_TIMEOUT; before it exits, the CTA waits (bounded again) for its own
// bulk copies and tensor-core products in flight, then frees its tensor
// memory.
#include <cuda.h>
#include <cuda_runtime.h>

#include <mutex>

#include <algorithm>
#include <cstring>
#include <vector>

#include <cuda_bf16.h>

#include "dd.cuh"
#include "sm100_prims.cuh"
#include "fx128.cuh"
#include "split_engine.h"

namespace cc3 {
using namespace sm100;

size_t s_smem_bytes(int slices, int ntile) {
  return (size_t)s_stages(slices) * slices * (S_BM + ntile) * 32 + 1024;
}

__device__ __forceinline__ long long s_rowoff(int m, int m_in, long long s1, long long s0) {
  return (long long)(m / m_in) * s1 + (long long)(m % m_in) * s0;
}

// A value that all lanes of the warp hold, as one the compiler knows to be
// uniform: tcgen05.mma takes its operands from uniform registers.
__device__ __forceinline__ int uniform(int x) { return __shfl_sync(0xffffffffu, x, 0); }
__device__ __forceinline__ uint32_t uniform(uint32_t x) { return __shfl_sync(0xffffffffu, x, 0); }

// The next group of (one or two) K steps: whether its stages have landed, and
// then the signs of their terms.  The issuer looks while it still has products
// to queue, so that a landed stage costs no round trip between two groups.
struct Ahead {
  uint64_t *b0, *b1;  // full barriers of the next two stages
  uint32_t p0, p1;    // their parities
  const int *neg;     // sign marks of the stages
  int s0, s1;         // the stages
  bool r0, r1;
  int n0, n1;  // their signs, valid where r0 / r1 holds
  __device__ __forceinline__ void look() {
    r0 = __all_sync(0xffffffffu, mbar_test(b0, p0));
    r1 = __all_sync(0xffffffffu, mbar_test(b1, p1));
    n0 = uniform(neg[s0]);
    n1 = uniform(neg[s1]);
  }
};

// All slice products of one K step, A slice by A slice.  Product p x q goes
// into accumulator min(p + q, 4), each at a fixed column so that tiles of
// different N keep out of each other's.  Each run keeps its A slice in the
// collector buffer: A is read from shared memory S times per step instead of
// once per product (53 clocks per 128 x 96 x 16 product, 57 without).  Slices
// are 256 bytes (16 descriptor units) apart.  LOOK: looks for the next group
// 6 products before the end.
template <int S, bool LOOK>
__device__ __forceinline__ void issue_all(uint32_t lead, uint32_t tmem, uint64_t dA, uint64_t dB,
                                          uint32_t id, Ahead &next) {
#pragma unroll
  for (int p = 0; p < S; ++p) {
    if (LOOK && p == S - 3) next.look();
    const uint64_t a = dA + (uint64_t)(p * 16);
#pragma unroll
    for (int q = 0; q < S - p; ++q) {
      const uint32_t d = tmem + (uint32_t)((p + q < 4 ? p + q : 4) * S_NT_MAX);
      const uint64_t b = dB + (uint64_t)(q * 16);
      if (S - p == 1)
        umma_f16_a<0>(lead, d, a, b, id, 1u);
      else if (q == 0)
        umma_f16_a<1>(lead, d, a, b, id, 1u);
      else if (q == S - p - 1)
        umma_f16_a<3>(lead, d, a, b, id, 1u);
      else
        umma_f16_a<2>(lead, d, a, b, id, 1u);
    }
  }
}

// The slice products of one or two K steps that go into the accumulators of
// MASK (bit L: accumulator L), A slice by A slice; with FRESH they start anew.
template <int S, uint32_t MASK, bool FRESH>
__device__ __forceinline__ void issue_some(uint32_t lead, uint32_t tmem, uint64_t dA0,
                                           uint64_t dB0, uint32_t id0, uint64_t dA1, uint64_t dB1,
                                           uint32_t id1, bool two) {
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    if (j == 1 && !two) break;
    const uint64_t dA = j ? dA1 : dA0, dB = j ? dB1 : dB0;
    const uint32_t id = j ? id1 : id0;
#pragma unroll
    for (int p = 0; p < S; ++p) {
      int n = 0, i = 0;
#pragma unroll
      for (int q = 0; q < S - p; ++q) n += (MASK >> (p + q < 4 ? p + q : 4)) & 1u;
#pragma unroll
      for (int q = 0; q < S - p; ++q) {
        const int L = p + q < 4 ? p + q : 4;
        if (!((MASK >> L) & 1u)) continue;
        const uint32_t d = tmem + (uint32_t)(L * S_NT_MAX);
        const uint64_t a = dA + (uint64_t)(p * 16), b = dB + (uint64_t)(q * 16);
        // an accumulator's first product is its one with A slice 0
        const uint32_t en = FRESH && j == 0 && p == 0 && q <= 4 ? 0u : 1u;
        if (n == 1)
          umma_f16_a<0>(lead, d, a, b, id, en);
        else if (i == 0)
          umma_f16_a<1>(lead, d, a, b, id, en);
        else if (i == n - 1)
          umma_f16_a<3>(lead, d, a, b, id, en);
        else
          umma_f16_a<2>(lead, d, a, b, id, en);
        ++i;
      }
    }
  }
}

// Drains keep the exact accumulators exact: per K at most 1, 2, 3, 4 products
// of |d d'| <= 2^14 reach level 0, 1, 2, 3, so level 3 is emptied after at most
// 16 K steps of 16, level 2 after 20, level 1 after 28 and level 0 after 56
// (sums within 2^24, 0.94 2^24, 0.88 2^24 and 0.88 2^24 of their unit 2^-8L).
// One level is emptied at a time, between two K steps, so that the products
// into the other four accumulators (17 to 20 of the 21 of each step) cover the
// read-back: drained four levels at a time, a drain took 2900 clocks, 1800 of
// them stalls.  A level is due once it holds drain_at(L) steps, unless the
// tile ends within its limit; level 3 goes first.  Since a drain is followed
// by two K steps before the next, the limits hold: 12 + 2, 16 + 2 + 2,
// 24 + 3 and 48 + 6.
__device__ __forceinline__ constexpr int drain_at(int L) {
  return L == 3 ? 12 : (L == 2 ? 16 : (L == 1 ? 24 : 48));
}
__device__ __forceinline__ constexpr int drain_limit(int L) {
  return L == 3 ? 16 : (L == 2 ? 20 : (L == 1 ? 28 : 56));
}
constexpr int EV_END = 4;  // epilogue event: 0..3 = drain that level, 4 = the tile's end

// Conversions to int run at a quarter of the FP32 rate, so at a tile's end two
// of the four levels take none: adding FX_R0 = 1.5 2^25 to an integer |v0| <
// 2^24 leaves v0 in units of 4 in the low bits of the sum's pattern (above
// those of FX_R0 itself), and adding FX_R2 = 1.5 2^9 to |v2| <= 240 leaves v2
// in units of 2^-14; what the two round off, at most 2 and 2^-15, joins levels
// 1 and 3 exactly.  FX_BIAS: what the patterns of the constants add.
constexpr float FX_R0 = 50331648.f, FX_R2 = 768.f;
constexpr unsigned long long FX_W2 = 1ull << (S_ACC_FRAC - 14);
constexpr unsigned long long FX_BIAS = (0x4C400000ull << (S_ACC_FRAC + 2)) + 0x44400000ull * FX_W2;
__device__ __forceinline__ long long fx_levels(long long a, float v0, float v1, float v2,
                                               float v3) {
  const float t0 = __fadd_rn(v0, FX_R0), t2 = __fadd_rn(v2, FX_R2);
  const float r0 = __fsub_rn(v0, __fsub_rn(t0, FX_R0)), r2 = __fsub_rn(v2, __fsub_rn(t2, FX_R2));
  const int i1 = __float2int_rn(__fadd_rn(r0, v1) * 0x1p8f),
            i3 = __float2int_rn(__fadd_rn(r2, v3) * 0x1p24f);
  unsigned long long u = (unsigned long long)a + ((unsigned long long)__float_as_uint(t0) << (S_ACC_FRAC + 2));
  u += (unsigned long long)__float_as_uint(t2) * FX_W2 - FX_BIAS;
  return (long long)u + (long long)i1 * (1ll << (S_ACC_FRAC - 8)) +
         (long long)i3 * (1ll << (S_ACC_FRAC - 24));
}
// Reads one level of this warp's columns (nch chunks of 4 from TMEM address tb,
// which is that level's) into the sums: v 2^(8L) as an integer, times 2^(S_ACC_FRAC - 8L).
__device__ __forceinline__ void drain_level(uint32_t tb, int L, int nch, long long (&acc)[6][4]) {
  const float up = __int_as_float((127 + 8 * L) << 23);
  const long long w = 1ll << (S_ACC_FRAC - 8 * L);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    if (c >= nch) break;
    float v[4];
    tmem_ld4(tb + c * 4, v);
    tmem_wait_ld();
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[c][k] += (long long)__float2int_rn(v[k] * up) * w;
  }
}

// The shared accumulator's sum v joins a, of unit 2^-S_ACC_FRAC.  With 7 slices
// (levels 5 and 6: products down to 2^-48) an element small enough to show it
// takes FX_MORE bits more, and bit `at` of its thread's flags says so; for the
// others the unit is below 2^-49 of them.  (At 6 slices this gains 1 % of the
// error at K = 80 and costs 1.4 to 4 % of the time.)
constexpr int FX_MORE = 14;
template <int S>
__device__ __forceinline__ long long fx_shared(long long a, float v, int at, unsigned int &fine) {
  const float t = v * (float)(1ll << S_ACC_FRAC);
  const int i = __float2int_rn(t);
  a += (long long)i;
  if constexpr (S >= 7) {
    constexpr long long LIMIT = 1ll << (62 - FX_MORE);
    if (a + LIMIT >= 0 && a < LIMIT) {
      a = a * (1ll << FX_MORE) + (long long)__float2int_rn((t - (float)i) * (float)(1 << FX_MORE));
      fine |= 1u << at;
    }
  }
  return a;
}
__device__ __forceinline__ int fine_bits(unsigned int fine, int at) {
  return (fine >> at) & 1u ? FX_MORE : 0;
}

// Moves chunk 1 to 0, 2 to 1, ...: the output loops take chunk 0 of a rolled
// loop, which costs 40 moves per chunk but keeps their code a sixth of the
// unrolled size (it was 98 KB, more than half of the kernel).
__device__ __forceinline__ void next_chunk(long long (&acc)[6][4]) {
#pragma unroll
  for (int c = 0; c < 5; ++c)
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[c][k] = acc[c + 1][k];
}

// a 2^e2 as a double, rounded once, from integer operations: the FP64 pipe of
// this part takes ~16 clocks per warp instruction and SM, and the conversions
// through it were most of the output time.
__device__ __forceinline__ double fixed_to_double(long long a, int e2) {
  const unsigned long long sign = (unsigned long long)a & 0x8000000000000000ull;
  const unsigned long long u = sign ? 0ull - (unsigned long long)a : (unsigned long long)a;
  const int lz = __clzll((long long)u);
  const int e = 63 - lz + e2 + 1022;  // biased exponent less one: the mantissa carries it
  if (u == 0ull || e < 0) return 0.0;
  const unsigned long long m = u << lz;
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);
  // (beyond the largest double: infinite)
  const unsigned long long b = e > 2045 ? 0x7FF0000000000000ull : ((unsigned long long)e << 52) + r;
  return __longlong_as_double((long long)(b | sign));
}
// a 2^e2 as a double-float pair: the leading 24 bits, rounded, and 24 more
// (infinite from 2^127 on).
__device__ __forceinline__ float2 fixed_to_dd(long long a, int e2) {
  const unsigned int sign = a < 0 ? 0x80000000u : 0u;
  const unsigned long long u = a < 0 ? 0ull - (unsigned long long)a : (unsigned long long)a;
  const int lz = __clzll((long long)u);
  const int e = 64 - lz + e2 + 127;  // u << lz is 2^64 times a value in [1/2, 1)
  if (u == 0ull || e < 1) return make_float2(0.f, 0.f);
  const unsigned long long m = u << lz;
  const unsigned int h = (unsigned int)(m >> 40) + ((unsigned int)(m >> 39) & 1u);
  const int rest = (int)((long long)(m - ((unsigned long long)h << 40)) >> 9);  // |.| <= 2^30
  const float f = __int_as_float((int)(((unsigned int)min(e, 255) << 23) | sign));
  return make_float2(__uint2float_rn(h) * 0x1p-24f * f, __int2float_rn(rest) * 0x1p-55f * f);
}

// Kept out of line: inlined into the unrolled output loop it would make the
// kernel large enough for instruction-cache misses to stall the MMA warp.
__device__ __noinline__ void fx_add_call(unsigned long long *slot, double v) { fx_add(slot, v); }

// Position of one tile within its job: batch index, K-split part, M/N tile
// and its K-step range [g0, g1) over the concatenated terms.
struct TileInfo {
  int bi, m0, n0, Nt, g0, g1;
};
__device__ __forceinline__ TileInfo decode_tile(const SJob &J, long long tile) {
  TileInfo t;
  const int local = (int)(tile - J.tile_base);
  const int per_batch = J.tiles_m * J.tiles_n * J.ksplit;
  t.bi = local / per_batch;
  int r = local % per_batch;
  const int ks = r % J.ksplit;
  r /= J.ksplit;
  t.m0 = r / J.tiles_n * S_BM;
  t.n0 = r % J.tiles_n * J.Ntile;
  t.Nt = min(J.Ntile, (J.N - t.n0 + 15) / 16 * 16);  // the last column tile is trimmed
  const int per = (J.ksteps + J.ksplit - 1) / J.ksplit;
  t.g0 = min(J.ksteps, ks * per);
  t.g1 = min(J.ksteps, t.g0 + per);
  return t;
}

// A term of a tile as bulk copies, from its first K step in the tile: copy c
// takes bytes[c] from src[c] (kbs[c] elements further each K step) to dst[c]
// in the stage; total bytes per K step; steps = 0: no more terms.
struct TermSlot {
  static constexpr int LANES = 28;
  const __nv_bfloat16 *src[LANES];
  long long kbs[LANES];
  uint32_t bytes[LANES], dst[LANES];
  uint32_t total;
  int steps, neg;
};

// One entry of the tile hand-off ring (tile < 0: no more tiles).
struct TileSlot {
  long long tile;
  TileInfo ti;
  SJob job;
};

// Persistent: one CTA per SM takes tiles from a launch-wide counter (the plan
// lists long tiles first) and keeps the stage ring, the TMEM allocation and
// the barriers across tiles.  The decoder fetches each tile index and hands
// it, decoded, to the MMA warp and the epilogue warps through a small ring in
// shared memory; the epilogue releases the accumulators as soon as it has read them,
// so the next tile's products start while it finishes the previous outputs.
// 96 registers: the 19 warps sit 5 to a sub-partition of 16,384 registers.
template <int S>
__global__ void __maxnreg__(96)
split_engine_kernel(const SJob *__restrict__ jobs, int njobs, const STerm *__restrict__ terms,
                    const __grid_constant__ SArrTable arrs, VPtrTable P,
                    int *status, unsigned int *tile_ctr,
                    long long ntiles) {
  constexpr int s = S;
  constexpr int S_STAGES = s_stages(S);
  constexpr int TQ = 4, KQ = 4;  // depths of the tile and the term hand-off rings
  // accumulators that receive products: level L <= 3 exists iff L <= S-1
  // (S >= 3), the shared one (levels >= 4) iff S >= 5
  constexpr int NLOW = S < 4 ? S : 4;
  constexpr bool HAS_HIGH = S >= 5;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full[S_STAGES], empty[S_STAGES];
  // evfull: an event for the epilogue (drain a level, or the tile's end), which
  // answers on drainempty or lowempty; accfull / accempty: the shared accumulator
  // at the tile's end.  One event is outstanding at a time.
  __shared__ __align__(8) uint64_t evfull, drainempty, lowempty, accfull, accempty, mmafin;
  __shared__ volatile int event;
  __shared__ __align__(8) uint64_t tfull[TQ], tempty[TQ];
  // the decoder decodes each tile once for everyone, with a copy of its job
  // (the output loop reads its fields for every element), and marks each stage
  // with the sign of its term, so that no other warp reads the tables
  __shared__ TileSlot tslot[TQ];
  __shared__ STerm sterm[S_TERM_CHUNK];  // the decoder's terms of the current tile
  __shared__ TermSlot termslot[KQ];
  __shared__ __align__(8) uint64_t termfull[KQ], termempty[KQ];
  __shared__ int sneg[S_STAGES];
  __shared__ uint32_t tmem_base_sh;
  __shared__ volatile int err;

  // broadcast, so that the compiler knows the roles' branches to be uniform
  const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < S_STAGES; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < TQ; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 1 + S_EPI_WARPS);
    }
    for (int i = 0; i < KQ; ++i) {
      mbar_init(&termfull[i], 1);
      mbar_init(&termempty[i], 1);
    }
    mbar_init(&evfull, 2);  // the event's word and the products before it
    mbar_init(&lowempty, S_EPI_WARPS);
    mbar_init(&accfull, 1);
    mbar_init(&accempty, S_EPI_WARPS);
    mbar_init(&drainempty, S_EPI_WARPS);
    mbar_init(&mmafin, 1);
    err = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base_sh, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = uniform(tmem_base_sh);
  const uint32_t a_bytes = S_BM * 32;

  if (warp == 0) {
    // producer: the bulk copies of every K step, one lane each (see the decoder)
    int issued = 0;
    bool ok = true;
    for (int k = 0; ok; ++k) {
      TermSlot &ts = termslot[k % KQ];
      if (!__all_sync(0xffffffffu, mbar_wait(&termfull[k % KQ], (k / KQ) & 1, &err))) break;
      const int steps = ts.steps, neg = ts.neg;
      if (steps == 0) break;
      const uint32_t total = ts.total;
      const int own = min(lane, TermSlot::LANES - 1);
      const __nv_bfloat16 *src = ts.src[own];
      const long long kbs = ts.kbs[own];
      const uint32_t bytes = lane < TermSlot::LANES ? ts.bytes[own] : 0u, dst = ts.dst[own];
      __syncwarp();
      if (lane == 0) mbar_arrive(&termempty[k % KQ]);
      for (int g = 0; g < steps; ++g) {
        const int st = issued % S_STAGES, ph = (issued / S_STAGES) & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(&empty[st], ph ^ 1, &err))) {
          ok = false;
          break;
        }
        if (lane == 0) {
          sneg[st] = neg;
          mbar_arrive_expect_tx(&full[st], total);
        }
        __syncwarp();
        // stage layout: s A slices (128 rows) then s B slices (S_NT_MAX rows)
        if (bytes)
          bulk_load(smem + (size_t)st * ((size_t)s * (a_bytes + S_NT_MAX * 32)) + dst, src, bytes,
                    &full[st]);
        __syncwarp();
        src += kbs;
        ++issued;
      }
    }
    // let every issued copy land before the CTA may exit, also after a
    // give-up (bounded; the wait ignores the error word)
    for (int i = (issued > S_STAGES ? issued - S_STAGES : 0); i < issued; ++i)
      mbar_wait_quiet(&full[i % S_STAGES], (i / S_STAGES) & 1, 500000000ull);
  } else if (warp == 18) {
    // decoder: takes tiles, hands each with its job to the issuer and the
    // epilogue, and resolves its terms into bulk copies a few terms ahead of
    // the producer (resolving one takes ~2000 clocks, a W build tile has two
    // terms of two K steps each).  Each lane owns one of a K step's copies
    // (source, stride, destination and size are fixed for a term): lanes 0..23
    // the A segments (one per slab the tile's rows touch), lane 24 A2, 25 B,
    // 26 Bt, 27 Bt2.
    // The counter returns to 0 by itself: a launch takes each tile once and one
    // index past the end per CTA, after which the increment wraps.
    const unsigned int wrap = (unsigned int)ntiles + gridDim.x - 1u;
    int j = 0, k = 0;
    bool fail = false;
    long long next = 0;
    if (lane == 0) next = (long long)atomicInc(tile_ctr, wrap);
    for (int i = 0; !fail; ++i) {
      const int q = i % TQ;
      if (!__all_sync(0xffffffffu, mbar_wait_sleep(&tempty[q], ((i / TQ) & 1) ^ 1, &err))) break;
      const long long tile = __shfl_sync(0xffffffffu, next, 0);
      TileSlot &slot = tslot[q];
      if (tile >= ntiles) {
        if (lane == 0) {
          slot.tile = -1;
          mbar_arrive(&tfull[q]);
        }
        if (!__all_sync(0xffffffffu,
                        mbar_wait_sleep(&termempty[k % KQ], ((k / KQ) & 1) ^ 1, &err)))
          break;
        if (lane == 0) {
          termslot[k % KQ].steps = 0;  // no more copies
          mbar_arrive(&termfull[k % KQ]);
        }
        break;
      }
      if (lane == 0) next = (long long)atomicInc(tile_ctr, wrap);  // back by the next tile
      // its job: the last one with tile_base <= tile (tiles come in increasing
      // order, so the search moves forward only), 32 jobs at a time
      for (;;) {
        const int c = j + 1 + lane;
        const bool before = c < njobs && jobs[c].tile_base <= tile;
        const int n = __popc(__ballot_sync(0xffffffffu, before));
        j += n;
        if (n < 32) break;
      }
      {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(jobs + j);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&slot.job);
        for (int w = lane; w < (int)(sizeof(SJob) / 4); w += 32) dst[w] = src[w];
      }
      __syncwarp();
      const TileInfo ti = decode_tile(slot.job, tile);
      const int term0 = slot.job.term0, nterm = slot.job.nterm;
      if (lane == 0) {
        slot.tile = tile;
        slot.ti = ti;
        mbar_arrive(&tfull[q]);
      }
      const int Nt = ti.Nt, bi = ti.bi, m0 = ti.m0, n0 = ti.n0;
      int kend = 0;
      for (int t = 0; t < nterm && kend < ti.g1; ++t) {
        if (t % S_TERM_CHUNK == 0) {
          __syncwarp();
          const int n = min((int)S_TERM_CHUNK, nterm - t) * (int)(sizeof(STerm) / 4);
          const uint32_t *from = reinterpret_cast<const uint32_t *>(terms + term0 + t);
          uint32_t *to = reinterpret_cast<uint32_t *>(sterm);
          for (int w = lane; w < n; w += 32) to[w] = from[w];
          __syncwarp();
        }
        const STerm &T = sterm[t % S_TERM_CHUNK];
        const int kbase = kend;
        kend += T.ksteps;
        if (kend <= ti.g0) continue;
        const SArr &XA = arrs.a[T.A.map], &XB = arrs.a[T.B.map], &XT = arrs.a[T.Bt.map];
        const int ar = T.A.row0 + bi * T.A.row_b + m0, as = T.A.slab0 + bi * T.A.slab_b;
        const int bs = T.B.slab0 + bi * T.B.slab_b, ts = T.Bt.slab0 + bi * T.Bt.slab_b;
        // B tile rows [n0, n0 + Nt): main rows from B, rows in [nbm, nbm2) from
        // the tail Bt, rows >= nbm2 from the second tail Bt2
        const int nbm = T.nbm > 0 ? T.nbm : (1 << 30);
        const int nbm2 = T.nbm2 > 0 ? T.nbm2 : (1 << 30);
        const int br = T.B.row0 + bi * T.B.row_b + n0;
        const int nmain = max(0, min(min(Nt, nbm - n0), XB.rows - br));
        const int tfirst = max(n0, nbm);           // first tail row of the tile
        const int tr = T.Bt.row0 + tfirst - nbm;   // its row in Bt
        const int ntail = T.nbm > 0 ? max(0, min(min(n0 + Nt, nbm2) - tfirst, XT.rows - tr)) : 0;
        int kmax = XA.kblocks;
        if (nmain > 0) kmax = min(kmax, XB.kblocks);
        if (ntail > 0) kmax = min(kmax, XT.kblocks);
        // A rows: [ar, ar + ra) of slab as, or flattened over slabs as, as + 1, ...
        int ra = 0, fs = as, fr = ar;
        bool abad = as < 0 || ar < 0;
        if (!abad && T.aflat > 0) {
          ra = min(S_BM, T.aflat - ar);
          fs = as + ar / XA.rows;
          fr = ar % XA.rows;
          abad = ra <= 0 || as + (ar + ra - 1) / XA.rows >= XA.slabs || T.asplit > 0;
        } else if (!abad) {
          abad = as >= XA.slabs || ar >= XA.rows;
          ra = min(S_BM, XA.rows - ar);
          if (T.asplit > 0) ra = min(ra, T.asplit);
        }
        bool bad = abad || (nmain > 0 && (bs < 0 || bs >= XB.slabs || br < 0)) ||
              (ntail > 0 && (ts < 0 || ts >= XT.slabs || tr < 0 || ((tfirst - n0) & 7) != 0));
        // second A segment
        const SArr &XA2 = arrs.a[T.A2.map];
        const int ar2 = T.A2.row0 + bi * T.A2.row_b, as2 = T.A2.slab0 + bi * T.A2.slab_b;
        int ra2 = 0;
        if (!bad && T.asplit > 0) {
          ra2 = min(S_BM - T.asplit, XA2.rows - ar2);
          bad = as2 < 0 || as2 >= XA2.slabs || ar2 < 0 || ra2 <= 0 || (T.asplit & 7) != 0;
          kmax = min(kmax, XA2.kblocks);
        }
        // second tail
        const SArr &XT2 = arrs.a[T.Bt2.map];
        const int t2first = max(n0, nbm2), ts2 = T.Bt2.slab0 + bi * T.Bt2.slab_b;
        const int tr2 = T.Bt2.row0 + t2first - nbm2;
        int ntail2 = 0;
        if (!bad && T.nbm2 > 0) {
          ntail2 = max(0, min(n0 + Nt - t2first, XT2.rows - tr2));
          if (ntail2 > 0) {
            bad = ts2 < 0 || ts2 >= XT2.slabs || tr2 < 0 || ((t2first - n0) & 7) != 0;
            kmax = min(kmax, XT2.kblocks);
          }
        }
        if (bad || kend - kbase > kmax) {
          fail = true;  // a plan addressed outside its slice array
          break;
        }
        // this lane's copy: rows [row, row + n) of a slab to rows at d of A or B
        const SArr *X = &XA;
        int slab = fs, row = fr, n = 0, d = 0;
        uint32_t side = 0;
        if (lane < 24) {
          // segment `lane` of the A rows: the first slab's rest, then whole slabs
          const int first = T.aflat > 0 ? min(ra, XA.rows - fr) : ra;
          d = lane == 0 ? 0 : first + (lane - 1) * XA.rows;
          n = lane == 0 ? first : min(ra - d, XA.rows);
          slab = fs + lane;
          row = lane == 0 ? fr : 0;
        } else if (lane == 24) {
          X = &XA2, slab = as2, row = ar2, n = ra2, d = T.asplit;
        } else {
          side = (uint32_t)s * a_bytes;
          if (lane == 25) X = &XB, slab = bs, row = br, n = nmain;
          if (lane == 26) X = &XT, slab = ts, row = tr, n = ntail, d = tfirst - n0;
          if (lane == 27) X = &XT2, slab = ts2, row = tr2, n = ntail2, d = t2first - n0;
        }
        const uint32_t bytes = n > 0 ? (uint32_t)n * 32u * s : 0u;
        const uint32_t dst = side + (uint32_t)d * 32u * s;
        const __nv_bfloat16 *src = reinterpret_cast<const __nv_bfloat16 *>(X->base) +
              (long long)slab * X->slab_stride + (long long)row * 16 * s;
        const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
        const int ks = max(ti.g0, kbase), ke = min(ti.g1, kend);
        TermSlot &out = termslot[k % KQ];
        if (!__all_sync(0xffffffffu,
                        mbar_wait_sleep(&termempty[k % KQ], ((k / KQ) & 1) ^ 1, &err))) {
          fail = true;
          break;
        }
        if (lane < TermSlot::LANES) {
          out.src[lane] = src + (long long)(ks - kbase) * X->kb_stride;
          out.kbs[lane] = X->kb_stride;
          out.bytes[lane] = bytes;
          out.dst[lane] = dst;
        }
        __syncwarp();
        if (lane == 0) {
          out.steps = ke - ks;
          out.neg = T.negA;
          out.total = total;
          mbar_arrive(&termfull[k % KQ]);
        }
        ++k;
      }
      if (fail && lane == 0 && !err) err = 2;
    }
  } else if (warp == 1) {
    {
      // MMA issuer: the warp stays converged (every lane waits and steps, the
      // elected one issues), see umma_f16_a
      const uint32_t lead = elect_one();
      int nd = 0, st0 = 0;  // drains so far, the next stage and its parity
      uint32_t ph0 = 0;
      Ahead next = {&full[0], &full[0], 0u, 0u, sneg, 0, 0, false, false, 0, 0};
      bool ok = true;
      for (int i = 0; ok; ++i) {
        const int q = i % TQ;
        if (!__all_sync(0xffffffffu, mbar_wait(&tfull[q], (i / TQ) & 1, &err))) break;
        const int more = uniform(tslot[q].tile >= 0);
        const int Nt = uniform(tslot[q].ti.Nt), g0 = uniform(tslot[q].ti.g0),
                  g1 = uniform(tslot[q].ti.g1);
        __syncwarp();  // every lane has read the slot before it is handed back
        if (lead) mbar_arrive(&tempty[q]);
        if (!more) break;
        const uint32_t id_pos = idesc_bf16(S_BM, Nt, 0), id_neg = idesc_bf16(S_BM, Nt, 1);
        // the epilogue has read the previous tile's accumulators: levels 0..3
        // and, later, the shared one
        auto low_free = [&]() {
          if (i > 0 && !__all_sync(0xffffffffu, mbar_wait(&lowempty, (i - 1) & 1, &err)))
            return false;
          tc_fence_after();
          return true;
        };
        // an event for the epilogue, due when the products issued so far are done
        auto signal = [&](int ev) {
          if (lead) {
            event = ev;
            mbar_arrive(&evfull);
            umma_commit(&evfull);
          }
          __syncwarp();
        };
        auto high_free = [&]() {
          if (i > 0 && !__all_sync(0xffffffffu, mbar_wait(&accempty, (i - 1) & 1, &err)))
            return false;
          tc_fence_after();
          return true;
        };
        int held[4] = {0, 0, 0, 0};  // K steps that each level holds
        int pending = -1;            // the level being drained
        // K steps two at a time; a lone last step of a tile goes alone
        for (int g = g0; g < g1;) {
          const bool first = g == g0, last = g + 2 >= g1;
          const bool two = g + 1 < g1;
          const int n = two ? 2 : 1;
          const int st1 = st0 + 1 == S_STAGES ? 0 : st0 + 1;
          const uint32_t ph1 = st1 == 0 ? ph0 ^ 1 : ph0;
          int neg0 = next.n0, neg1 = next.n1;
          if (!next.r0 || (two && !next.r1)) {
            bool here = next.r0 || mbar_wait(&full[st0], ph0, &err);
            if (two) here = here && (next.r1 || mbar_wait(&full[st1], ph1, &err));
            if (!__all_sync(0xffffffffu, here)) { ok = false; break; }
            neg0 = uniform(sneg[st0]);
            neg1 = uniform(sneg[st1]);
          }
          tc_fence_after();
          // the stages after this group's
          const int sn = two ? (st1 + 1 == S_STAGES ? 0 : st1 + 1) : st1;
          const uint32_t pn = two ? (sn == 0 ? ph1 ^ 1 : ph1) : ph1;
          const int sm = sn + 1 == S_STAGES ? 0 : sn + 1;
          next = Ahead{&full[sn], &full[sm], pn,    sm == 0 ? pn ^ 1 : pn, sneg, sn, sm,
                       false,     false,     neg0,  neg1};
          const uint32_t id0 = neg0 ? id_neg : id_pos, id1 = neg1 ? id_neg : id_pos;
          const size_t stage_bytes = (size_t)s * (a_bytes + S_NT_MAX * 32);
          const uint32_t sa0 = smem_u32(smem + (size_t)st0 * stage_bytes),
                         sa1 = smem_u32(smem + (size_t)st1 * stage_bytes);
          // slice p of a tile starts 256 p bytes in; row groups are 256 s bytes apart
          const uint64_t dA0 = smem_desc_kmajor(sa0, 256u * s),
                         dB0 = smem_desc_kmajor(sa0 + (uint32_t)s * a_bytes, 256u * s),
                         dA1 = smem_desc_kmajor(sa1, 256u * s),
                         dB1 = smem_desc_kmajor(sa1 + (uint32_t)s * a_bytes, 256u * s);
          const bool both = pending < 0 && !first && !last;
          if (!both) {
            // in two parts.  After a drain point: the products into the
            // accumulators that are not being emptied, then, once the epilogue
            // has read it, the one that is, which starts anew.  At a tile's
            // ends: levels 0..3, then the shared accumulator, so that the
            // epilogue reads the ones while products go to the other.
#define CC3_SOME(MASK, FRESH) \
  issue_some<S, MASK, FRESH>(lead, tmem, dA0, dB0, id0, dA1, dB1, id1, two)
            if (pending >= 0) {
              switch (pending) {
                case 0: CC3_SOME(0x1Eu, false); break;
                case 1: CC3_SOME(0x1Du, false); break;
                case 2: CC3_SOME(0x1Bu, false); break;
                default: CC3_SOME(0x17u, false); break;
              }
              next.look();
              ok = __all_sync(0xffffffffu, mbar_wait(&drainempty, nd & 1, &err));
              if (!ok) break;
              tc_fence_after();
              ++nd;
              switch (pending) {
                case 0: CC3_SOME(0x1u, true); break;
                case 1: CC3_SOME(0x2u, true); break;
                case 2: CC3_SOME(0x4u, true); break;
                default: CC3_SOME(0x8u, true); break;
              }
              pending = -1;
            } else if (first) {
              ok = low_free();
              if (!ok) break;
              CC3_SOME(0xFu, true);
              if (last) signal(EV_END);
              next.look();
              ok = high_free();
              if (!ok) break;
              CC3_SOME(0x10u, true);
            } else {
              CC3_SOME(0xFu, false);
              signal(EV_END);
              next.look();
              CC3_SOME(0x10u, false);
            }
#undef CC3_SOME
          } else {
            // (neither end of the tile: there are two steps)
            issue_all<S, false>(lead, tmem, dA0, dB0, id0, next);
            umma_commit_a(lead, &empty[st0]);
            issue_all<S, true>(lead, tmem, dA1, dB1, id1, next);
          }
          g += n;
          if (!both) umma_commit_a(lead, &empty[st0]);
          if (two) umma_commit_a(lead, &empty[st1]);
          st0 = sn;
          ph0 = pn;
          const int left = g1 - g;
#pragma unroll
          for (int L = 0; L < 4; ++L) held[L] += n;
          if (left > 2) {  // never right before the tile's last steps
#pragma unroll
            for (int L = NLOW - 1; L >= 0; --L)
              if (pending < 0 && held[L] >= drain_at(L) && held[L] + left > drain_limit(L)) {
                pending = L;
                held[L] = 0;
              }
            if (pending >= 0) signal(pending);
          }
        }
        if (!ok) break;
        if (g0 == g1) {  // no K steps: nothing to wait for but the protocol
          if (!low_free() || !high_free()) break;
          signal(EV_END);
        }
        if (lead) umma_commit(&accfull);
        __syncwarp();
      }
      // every product this thread issued has landed in tensor memory before
      // the CTA frees it, also after a give-up (bounded)
      __syncwarp();
      if (lead) umma_commit(&mmafin);
      mbar_wait_quiet(&mmafin, 0, 500000000ull);
    }
  } else {
    // epilogue: warps 2..17
    const int ew = warp - 2, quad = warp & 3, part = ew >> 2;
    const int row = quad * 32 + lane;
    int nev = 0;
    for (int i = 0;; ++i) {
      const int q = i % TQ;
      if (i > 0) {  // done with the previous tile's slot
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[(i - 1) % TQ]);
      }
      if (!__all_sync(0xffffffffu, mbar_wait_sleep(&tfull[q], (i / TQ) & 1, &err))) break;
      if (tslot[q].tile < 0) break;
      const SJob &J = tslot[q].job;
      const TileInfo &ti = tslot[q].ti;
      const int Nt = ti.Nt;
      const int nsteps = ti.g1 - ti.g0;
      const int qc = Nt >> 2;   // columns per quarter (multiple of 4, <= 24)
      const int nch = qc >> 2;  // 4-column chunks (<= 6)
      const uint32_t tb = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(part * qc);
      long long acc[6][4];
#pragma unroll
      for (int c = 0; c < 6; ++c)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[c][k] = 0ll;
      // the drains, then levels 0..3 at the tile's end
      bool ok = true;
      for (;;) {
        ok = __all_sync(0xffffffffu, mbar_wait(&evfull, nev & 1, &err));
        if (!ok) break;
        ++nev;
        const int ev = event;
        tc_fence_after();
        if (ev == EV_END) break;
        drain_level(tb + (uint32_t)(ev * S_NT_MAX), ev, nch, acc);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&drainempty);
      }
      if (!ok) break;
      if (nsteps > 0) {
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          if (c >= nch) break;
          float v[4][4];
#pragma unroll
          for (int k = 0; k < 4; ++k) v[3][k] = 0.f;
#pragma unroll
          for (int L = 0; L < NLOW; ++L) tmem_ld4(tb + L * S_NT_MAX + c * 4, v[L]);
          tmem_wait_ld();
#pragma unroll
          for (int k = 0; k < 4; ++k)
            acc[c][k] = fx_levels(acc[c][k], v[0][k], v[1][k], v[2][k], v[3][k]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&lowempty);
      // the shared accumulator
      unsigned int fine = 0u;
      if (!__all_sync(0xffffffffu, mbar_wait(&accfull, i & 1, &err))) break;
      if (HAS_HIGH && nsteps > 0) {
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          if (c >= nch) break;
          float v[4];
          tmem_ld4(tb + 4 * S_NT_MAX + c * 4, v);
          tmem_wait_ld();
#pragma unroll
          for (int k = 0; k < 4; ++k) acc[c][k] = fx_shared<S>(acc[c][k], v[k], c * 4 + k, fine);
        }
        tc_fence_before();
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&accempty);
      const int bi = ti.bi, n0 = ti.n0 + part * qc, m = ti.m0 + row;
      const int *slot_ex = reinterpret_cast<const int *>(P.p[B_SLOTEXP]);
      const bool seg2 = J.msplit > 0 && m >= J.msplit;  // second row segment
      // the per-triple exponent table is read only by jobs that name a slot
      const int es = seg2 ? J.expo_slot2 : J.expo_slot;
      const int e2 = J.expo + (es >= 0 ? slot_ex[es] : 0) - S_ACC_FRAC;
      const int mo = seg2 ? m - J.msplit : m;  // row within its output
      const bool row_ok = m < J.M && !(J.m_pad > 0 && (m + J.m_off) % J.m_pad >= J.m_valid);
      // the thread's row is fixed for the tile: its output row offsets once.
      // Main columns n < Nm go to C (C2 for second-segment rows), tail
      // column tcol (tcol2) to Ct (Ct2); columns map linearly (n_in >= N,
      // checked when the plan is uploaded)
      const OutD &Cm = seg2 ? J.C2 : J.C;
      const long long rowM =
          row_ok ? Cm.off + (long long)bi * Cm.sb + s_rowoff(mo, Cm.m_in, Cm.sm1, Cm.sm0) : 0;
      if (J.mode == SEPI_DD_STORE) {  // main columns only (checked at upload)
        float2 *out = reinterpret_cast<float2 *>(P.p[Cm.buf]) + rowM + (long long)n0 * Cm.sn0;
        const long long sn = Cm.sn0;
        const int ncol = row_ok ? J.n_valid - n0 : 0;
#pragma unroll 1
        for (int c = 0; c < nch; ++c) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (c * 4 + k < ncol) *out = fixed_to_dd(acc[0][k], e2 - fine_bits(fine, c * 4 + k));
            out += sn;
          }
          next_chunk(acc);
        }
        continue;
      }
      if (!row_ok) continue;
      const int mq = mo / Cm.m_in, mr = mo % Cm.m_in;  // route 1: shared by its outputs
#pragma unroll 1
      for (int c = 0; c < nch; ++c, next_chunk(acc)) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int n = n0 + c * 4 + k;
          long long off;
          int buf;
          if (J.route == 1) {  // two column segments (see SJob)
            const bool sg = n >= J.Nm2;
            const int jc = sg ? n - J.Nm2 : n;
            if (n >= J.N || jc >= J.Nm + J.tw) continue;
            const OutD &O = jc < J.Nm ? (sg ? J.C2 : J.C) : (sg ? J.Ct2 : J.Ct);
            off = O.off + (long long)bi * O.sb + (long long)mq * O.sm1 + (long long)mr * O.sm0 +
                  (long long)(jc < J.Nm ? jc : jc - J.Nm) * O.sn0;
            buf = O.buf;
          } else if (n < J.Nm) {
            if (n >= J.n_valid) continue;
            off = rowM + (long long)n * Cm.sn0;
            buf = Cm.buf;
          } else {  // tail columns are few: their offsets on the fly
            const OutD &Ctl = seg2 ? J.Ct2 : J.Ct;
            if (n != (seg2 ? J.tcol2 : J.tcol)) continue;
            off = Ctl.off + (long long)bi * Ctl.sb + s_rowoff(mo, Ctl.m_in, Ctl.sm1, Ctl.sm0);
            buf = Ctl.buf;
          }
          const double x = fixed_to_double(acc[0][k], e2 - fine_bits(fine, c * 4 + k));
          if (P.fx[buf])
            fx_add_call(P.fx[buf] + 2 * off, x);
          else
            atomicAdd(reinterpret_cast<double *>(P.p[buf]) + off, x);
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
  if (threadIdx.x == 0 && err) atomicExch(status, err);
}

int s_upload_plan(const SPlan &p, SDevPlan *d, cudaStream_t s) {
  s_free_plan(d);
  // the epilogue maps output columns linearly (n * sn0): no output may split
  // its columns (n_in >= N)
  for (const SJob &j : p.jobs) {
    const bool two = j.msplit > 0;
    const bool r1 = j.route == 1;
    const OutD *outs[4] = {&j.C, &j.Ct, two || r1 ? &j.C2 : nullptr, two || r1 ? &j.Ct2 : nullptr};
    for (const OutD *o : outs)
      if (o && (o->n_in < j.N || (r1 && o->m_in != j.C.m_in))) return CC3_ERR_ARG;
    if (r1 && (two || j.Nm2 <= 0 || j.Nm + j.tw > j.Nm2)) return CC3_ERR_ARG;
    // stores take the main columns of one row segment
    if (j.mode == SEPI_DD_STORE && (two || r1 || j.Nm < j.N || j.ksplit != 1)) return CC3_ERR_ARG;
  }
  // tiles of more than S_MAX_TILE_STEPS K steps are split over K (their
  // partial sums add in the output)
  std::vector<SJob> jobs = p.jobs;
  long long tiles = 0;
  for (SJob &j : jobs) {
    long long steps = 0;
    for (int t = 0; t < j.nterm; ++t) steps += p.terms[j.term0 + t].ksteps;
    if (steps > 0x7fffffffLL || (long long)j.batch * j.tiles_m * j.tiles_n * j.ksplit > 0x7fffffffLL)
      return CC3_ERR_ARG;
    j.ksteps = (int)steps;
    const long long need = (steps + S_MAX_TILE_STEPS - 1) / S_MAX_TILE_STEPS;
    if (need > j.ksplit) {
      if (j.mode == SEPI_DD_STORE) return CC3_ERR_ARG;
      j.ksplit = (int)need;
    }
    j.tile_base = tiles;
    tiles += (long long)j.batch * j.tiles_m * j.tiles_n * j.ksplit;
  }
  d->njobs = (int)jobs.size();
  d->tiles = tiles;
  d->flop = p.flop;
  d->slice_flop = p.slice_flop;
  // one allocation: the tile counter, the jobs, the terms
  const size_t jb = (sizeof(SJob) * jobs.size() + 15) / 16 * 16,
               tb = sizeof(STerm) * p.terms.size();
  std::vector<char> host(16 + jb + tb, 0);
  if (!jobs.empty()) std::memcpy(host.data() + 16, jobs.data(), sizeof(SJob) * jobs.size());
  if (tb) std::memcpy(host.data() + 16 + jb, p.terms.data(), tb);
  char *base = nullptr;
  if (dev_malloc(&base, host.size() + sizeof(STerm)) != cudaSuccess) {
    cudaGetLastError();
    return CC3_ERR_OOM;
  }
  d->counter = reinterpret_cast<unsigned int *>(base);
  d->jobs = reinterpret_cast<SJob *>(base + 16);
  d->terms = reinterpret_cast<STerm *>(base + 16 + jb);
  return dev_upload(base, host.data(), host.size(), s);
}

void s_free_plan(SDevPlan *d) {
  if (d->counter) dev_free(d->counter);
  d->counter = nullptr;
  d->jobs = nullptr;
  d->terms = nullptr;
  d->njobs = 0;
  d->tiles = 0;
}

int s_launch_plan(const SDevPlan &d, const SArrTable &arrs, const VPtrTable &ptrs,
                  int slices, int *status, cudaStream_t s,
                  long long *launches) {
  if (d.njobs == 0 || d.tiles == 0) return CC3_OK;
  if (d.tiles > 0x7fffffffLL) return CC3_ERR_ARG;
  if (slices < 3 || slices > S_MAX_SLICES) return CC3_ERR_ARG;
  // at least 120 KB so that one CTA (and one 512-column TMEM allocation) per SM
  const size_t smem = std::max<size_t>(s_smem_bytes(slices, S_NT_MAX), 120 * 1024);
  // per device, once; several host threads (serving slots) may get here at once
  static std::mutex attr_mu;
  static bool attr_set[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return CC3_FAIL(CC3_ERR_CUDA, "device index");
  std::lock_guard<std::mutex> attr_lk(attr_mu);
  if (!attr_set[dev]) {
    const void *fns[] = {(const void *)split_engine_kernel<3>, (const void *)split_engine_kernel<4>,
                         (const void *)split_engine_kernel<5>, (const void *)split_engine_kernel<6>,
                         (const void *)split_engine_kernel<7>};
    for (int S = 3; S <= 7; ++S) {
      const void *f = fns[S - 3];
      const int mx = (int)std::max<size_t>(s_smem_bytes(S, S_NT_MAX), 120 * 1024);
      cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
      if (e != cudaSuccess) return CC3_FAIL(CC3_ERR_CUDA, cudaGetErrorString(e));
      int nb = 0;
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, S_THREADS, (size_t)mx);
      if (e != cudaSuccess || nb < 1)
        return CC3_FAIL(CC3_ERR_CUDA, "split engine kernel does not fit on an SM");
    }
    attr_set[dev] = true;
  }
  static int sms[64] = {0};
  if (!sms[dev]) cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev);
  const unsigned grid = (unsigned)std::min<long long>(d.tiles, std::max(1, sms[dev]));
  switch (slices) {
#define CC3_SPLIT_LAUNCH(S_)                                                              \
  case S_:                                                                                \
    split_engine_kernel<S_><<<grid, S_THREADS, smem, s>>>(                                \
        d.jobs, d.njobs, d.terms, arrs, ptrs, status, d.counter, d.tiles);                \
    break;
    CC3_SPLIT_LAUNCH(3)
    CC3_SPLIT_LAUNCH(4)
    CC3_SPLIT_LAUNCH(5)
    CC3_SPLIT_LAUNCH(6)
    CC3_SPLIT_LAUNCH(7)
#undef CC3_SPLIT_LAUNCH
    default:
      return CC3_FAIL(CC3_ERR_ARG, "slices");
  }
  if (launches) ++*launches;
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? CC3_OK : CC3_FAIL(CC3_ERR_CUDA, cudaGetErrorString(e));
}

}  // namespace cc3
