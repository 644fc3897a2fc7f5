// Exact products of fixed-point rows on the tcgen05 tensor cores: what the FP64
// contraction (syrk_sl.cu) and the Cholesky's trailing update (chol_fx.cu) share.
//
// A row entry is an integer X (its value X 2^-55, |X| < 2^55.5) cut into the seven
// balanced base-256 digits x = sum_t d_t 2^(-7-8t), each exact in BF16, stored per
// (128-row block, K block of 32) as one contiguous 56 KB block [digit][row][k].
// d_t(i) d_u(j) and their sums over a K block at equal t + u = g, g = 0..6, stay
// below 2^22: exact in the FP32 accumulators.  The 28 pairs t + u <= 6 are formed by
// 7 MMAs per K step instead of 28: the J digits u = 0..6 of a group of 32 columns are
// stacked in shared memory, the accumulators of the seven levels lie side by side in
// TMEM, and one MMA of digit t against the first 32 (7 - t) stacked rows lands on the
// levels t..6 (N = 224, 192, ..., 32).  Small-N MMAs would read the 4 KB of the I digit
// from shared memory for 8 cycles of work each.  The level sums of a K block combine exactly
// to one 64-bit integer per element, in units of 2^-62, modulo 2^64: the Cholesky's rows
// share one scale and it adds them as they are; the contraction's K blocks have exponents of
// their own, and it aligns them first.
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"

#define SL_S 7
#define SL_BM 128                                   // tile rows, and tile columns
#define SL_BK 32                                    // K block
#define SL_BN 32                                    // columns per accumulator group
#define SL_DIGIT (SL_BM * SL_BK * 2)                // 8 KB: one digit of 128 rows x 32 K
#define SL_BLOCK (SL_S * SL_DIGIT)                  // 56 KB: one (row block, K block)
#define SL_GROUP (SL_S * SL_BN * SL_BK * 2)         // 14 KB: the digits of 32 rows
#define SL_STAGES 2
#define SL_EPI 8                                    // epilogue warps: two per TMEM lane quarter, 16 columns each
#define SL_THREADS (64 + 32 * SL_EPI)
#define SL_SPIN (1u << 22)
#define SL_MAGIC 0x4B400000u                        // bits of 1.5 2^23: f + 1.5 2^23 holds the integer f in its low bits

template <int NG>
struct SlShape {  // NG groups of 32 columns
  static constexpr int kStage = SL_BLOCK + NG * SL_GROUP;  // 112 KB for 128 columns
  static constexpr int kSmem = SL_STAGES * kStage + 1024;
};

// X = RN(x 2^(55 - e)) (ties to even) for |x| < 2^(e + 2), by integer operations on the bits
// of x; 0 for an infinity or NaN, which no digit holds (its K block is marked, see k_sl_rows)
__device__ __forceinline__ long long sl_int(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7FFu);
  if (E == 0x7FF) return 0;
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);  // (subnormals round to 0 either way)
  const int sh = 1020 - E + e;  // X = RN(m / 2^sh); sh >= -3
  unsigned long long q;
  if (sh <= 0) {
    q = m << -sh;
  } else if (sh >= 64) {
    q = 0;
  } else {
    q = m >> sh;
    const unsigned long long rem = m & ((1ull << sh) - 1), half = 1ull << (sh - 1);
    q += (rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull;
  }
  return (b >> 63) ? -(long long)q : (long long)q;
}

// The digits of eight integers (consecutive k of one row) as BF16: out[t] holds digit
// t's 16 bytes.  d_t = byte_t(X + 128 sum_t 256^t) - 128; the top digit keeps its sign
// and ninth bit.  |d| <= 256 has at most 8 significant bits, so the upper half of its
// FP32 value is its BF16 form.
__device__ __forceinline__ void sl_digits8(const long long* X, uint4* out) {
  uint32_t d[SL_S][4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    unsigned long long y[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) y[h] = (unsigned long long)X[2 * p + h] + 0x0080808080808080ull;
#pragma unroll
    for (int t = 0; t < SL_S; ++t) {
      float f[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int by = t == 0 ? (int)((long long)y[h] >> 48) : (int)((y[h] >> (8 * (SL_S - 1 - t))) & 255u);
        f[h] = __int_as_float(SL_MAGIC + by) - (12582912.0f + 128.0f);
      }
      d[t][p] = __byte_perm(__float_as_uint(f[0]), __float_as_uint(f[1]), 0x7632);
    }
  }
#pragma unroll
  for (int t = 0; t < SL_S; ++t) out[t] = make_uint4(d[t][0], d[t][1], d[t][2], d[t][3]);
}

// ---------------------------------------------------------------- barriers, copies, descriptors
__device__ __forceinline__ uint32_t sl_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void sl_init(uint64_t* bar, uint32_t n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sl_u32(bar)), "r"(n) : "memory");
}
__device__ __forceinline__ void sl_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(sl_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void sl_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sl_u32(bar)) : "memory");
}
__device__ __forceinline__ void sl_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(sl_u32(bar))
               : "memory");
}
__device__ __forceinline__ uint32_t sl_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(sl_u32(bar)), "r"(parity)
      : "memory");
  return ok;
}
// bounded wait that also gives up once any CTA has raised the status word
__device__ __forceinline__ bool sl_wait(uint64_t* bar, uint32_t parity, int* status) {
  for (uint32_t i = 0; i < SL_SPIN; ++i) {
    if (sl_try(bar, parity)) return true;
    if ((i & 1023u) == 1023u && *(volatile int*)status) return false;
  }
  atomicExch(status, 1);
  return false;
}
__device__ __forceinline__ void sl_tma(const CUtensorMap* map, uint64_t* bar, void* dst, int row, int blk) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
      "[%2];" ::"r"(sl_u32(dst)),
      "l"((uint64_t)map), "r"(sl_u32(bar)), "r"(0), "r"(row), "r"(0), "r"(blk)
      : "memory");
}
__device__ __forceinline__ void sl_prefetch(const CUtensorMap* map, int row, int blk) {
  asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global.tile [%0, {%1, %2, %3, %4}];" ::"l"((uint64_t)map), "r"(0),
               "r"(row), "r"(0), "r"(blk)
               : "memory");
}
__device__ __forceinline__ uint64_t sl_desc(uint32_t saddr) {  // K-major, 64-byte rows, SWIZZLE_64B
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;  // 8 rows x 64 B
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}
// Four TMEM words per thread and instruction, in one of two shapes.  Rows (FRAG false):
// 32 lanes x 4 columns, thread t holds lane t.  Fragments: 16 lanes x 8 columns, thread t
// holds lanes t / 4 (r[0], r[1]) and t / 4 + 8 (r[2], r[3]), columns 2 (t % 4) and the
// next; four threads then hold 64 bytes of a row of 64-bit sums, so that entries move to
// and from memory in whole sectors, but the reads are slower (M = 6375, K = 12416: 11.7 ms
// against 10.0).  The caller issues tcgen05.wait::ld / ::st.
template <bool FRAG>
__device__ __forceinline__ void sl_tmem_ld4(uint32_t taddr, uint32_t* r) {
  if (FRAG)
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
  else
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}
template <bool FRAG>
__device__ __forceinline__ void sl_tmem_st4(uint32_t taddr, uint32_t v) {
  if (FRAG)
    asm volatile("tcgen05.st.sync.aligned.16x256b.x1.b32 [%0], {%1,%1,%1,%1};" ::"r"(taddr), "r"(v) : "memory");
  else
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%1,%1,%1};" ::"r"(taddr), "r"(v) : "memory");
}
// TMEM address of part h (0..3) of a warp's 32 lanes x 16 columns
template <bool FRAG>
__device__ __forceinline__ uint32_t sl_part(int h) {
  return FRAG ? ((uint32_t)(h >> 1) << 20) + (uint32_t)(8 * (h & 1)) : (uint32_t)(4 * h);
}

// ---------------------------------------------------------------- roles of one tile
// Barriers of a CTA; initialised by one thread (sl_bars_init),
// then a block barrier.
struct SlBars {
  uint64_t full[SL_STAGES], empty[SL_STAGES], tfull[2], tempty[2], mma_done;
};
__device__ __forceinline__ void sl_bars_init(SlBars* b) {
  for (int s = 0; s < SL_STAGES; ++s) {
    sl_init(&b->full[s], 1);
    sl_init(&b->empty[s], 1);
  }
  for (int i = 0; i < 2; ++i) {
    sl_init(&b->tfull[i], 1);
    sl_init(&b->tempty[i], SL_EPI);
  }
  sl_init(&b->mma_done, 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// The roles below run over the K blocks of one tile; it counts the K blocks of all tiles
// of the CTA so far (the barriers' phases), and false means that a wait expired.
//
// One thread: K blocks of the I row block (digit blocks bi, bi + 1, ...; one box each)
// and of NG column groups (rows jrow, jrow + 32, ... of the digit blocks bj, ...).
template <int NG>
__device__ __forceinline__ bool sl_produce(const CUtensorMap* map_i, const CUtensorMap* map_j, uint8_t* smem, SlBars* B,
                                           int bi, int bj, int jrow, int nkb, int& it, int* status) {
  constexpr int STAGE = SlShape<NG>::kStage;
  for (int w = 0; w < nkb; ++w, ++it) {
    const int s = it % SL_STAGES;
    if (!sl_wait(&B->empty[s], (uint32_t)((it / SL_STAGES) & 1) ^ 1u, status)) return false;
    uint8_t* st = smem + (size_t)s * STAGE;
    sl_expect(&B->full[s], STAGE);
    sl_tma(map_i, &B->full[s], st, 0, bi + w);
    for (int j = 0; j < NG; ++j) sl_tma(map_j, &B->full[s], st + SL_BLOCK + j * SL_GROUP, jrow + j * SL_BN, bj + w);
    if (w + 2 < nkb) {
      sl_prefetch(map_i, 0, bi + w + 2);
      if (bi != bj) sl_prefetch(map_i, 0, bj + w + 2);
    }
  }
  return true;
}

// One warp: the MMAs, issued by one elected lane.  The loop is warp-uniform, so that
// descriptors and addresses live in uniform registers (inside a one-lane branch every
// operand goes through a register move, ~100 cycles per MMA: more than the MMA itself);
// the 512 allocated columns start at TMEM address 0.  NEG: the I operand is negated (the
// sums come out as -A B^T).  LV 8 forms the level t + u = 7 as well (six pairs of digits).
template <int NG, bool NEG, int LV = SL_S>
__device__ __forceinline__ bool sl_issue(uint8_t* smem, SlBars* B, int nkb, int& it, int* status) {
  constexpr int STAGE = SlShape<NG>::kStage;
  uint32_t leader;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(leader));
  for (int w = 0; w < nkb; ++w, ++it) {
    const int s = it % SL_STAGES;
    if (!__all_sync(0xffffffffu, sl_wait(&B->full[s], (uint32_t)((it / SL_STAGES) & 1), status))) return false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t base_i = sl_u32(smem + (size_t)s * STAGE);
#pragma unroll 1
    for (int j = 0; j < NG; ++j) {
      const int b = j & 1, use = (NG / 2) * it + (j >> 1);  // use-th filling of accumulator set b
      if (!__all_sync(0xffffffffu, sl_wait(&B->tempty[b], (uint32_t)(use & 1), status))) return false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t base_j = base_i + SL_BLOCK + j * SL_GROUP, dt = (uint32_t)(b * 256);
#pragma unroll
      for (int k = 0; k < SL_BK / 16; ++k)
#pragma unroll
        for (int t = 0; t < SL_S; ++t) {
          // BF16 x BF16 -> FP32, K-major, M = 128, N = 32 per digit: digit t against the digits 0 .. LV - 1 - t
          const int nu = LV - t < SL_S ? LV - t : SL_S;
          const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (NEG ? 1u << 13 : 0u) |
                                 ((uint32_t)((SL_BN * nu) >> 3) << 17) | ((uint32_t)(SL_BM >> 4) << 24);
          asm volatile(
              "{\n .reg .pred p, q;\n setp.ne.b32 p, 1, 0;\n setp.ne.b32 q, %4, 0;\n @q "
              "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dt + (uint32_t)(t * SL_BN)),
              "l"(sl_desc(base_i + t * SL_DIGIT + k * 32)), "l"(sl_desc(base_j + k * 32)), "r"(idesc), "r"(leader)
              : "memory");
        }
      if (leader) sl_commit(&B->tfull[b]);
      __syncwarp();
    }
    if (leader) sl_commit(&B->empty[s]);
    __syncwarp();
  }
  return true;
}
// after the last tile: every MMA of this CTA has completed before its TMEM is released
__device__ __forceinline__ void sl_issue_end(SlBars* B, int lane) {
  if (lane == 0) {
    sl_commit(&B->mma_done);
    for (uint32_t i = 0; i < SL_SPIN && !sl_try(&B->mma_done, 0u); ++i) {
    }
  }
  __syncwarp();
}

// What the offset of the accumulators leaves in a 64-bit sum per K block (sl_drain)
#define SL_BIAS                                                                                                   \
  (((unsigned long long)SL_MAGIC << 48) + ((257ull * SL_MAGIC) << 32) + ((257ull * SL_MAGIC & 0xFFFFFFFFull) << 16) + \
   (257ull * SL_MAGIC & 0xFFFFFFFFull))

// Epilogue warps, once per CTA: the starting value into both accumulator sets
template <bool FRAG, int LV = SL_S>
__device__ __forceinline__ void sl_drain_init(SlBars* B, uint32_t tmem, int q, int half, int lane) {
  const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * 16);
#pragma unroll
  for (int b = 0; b < 2; ++b) {
#pragma unroll
    for (int g = 0; g < LV; ++g) {
#pragma unroll
      for (int h = 0; h < 4; ++h) sl_tmem_st4<FRAG>(tbase + sl_part<FRAG>(h) + (uint32_t)(b * 256 + g * SL_BN), SL_MAGIC);
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    if (lane == 0) sl_arrive(&B->tempty[b]);
  }
}

// Place in the tile of a thread's sum acc[j][c]: warp q + 4 half owns rows 32 q .. and
// columns 16 half .. of each group of 32
template <bool FRAG>
__device__ __forceinline__ int sl_row(int q, int lane, int c) {
  return q * 32 + (FRAG ? 16 * (c >> 3) + 8 * ((c >> 1) & 1) + (lane >> 2) : lane);
}
template <bool FRAG>
__device__ __forceinline__ int sl_col(int half, int lane, int j, int c) {
  return j * SL_BN + half * 16 + (FRAG ? 8 * ((c >> 2) & 1) + 2 * (lane & 3) + (c & 1) : c);
}

// Epilogue warps (8): acc[j][c] += the level sums of its element, plus SL_BIAS per K block.  The accumulators start at 1.5 2^23 instead of 0:
// a sum below 2^22 then leaves its integer value in the low bits of the FP32 word, and
// no conversion is needed.  Each warp puts the constant back after reading.
// False when a wait expired (warp-uniform).
template <int NG, bool FRAG>
__device__ __forceinline__ bool sl_drain(unsigned long long (&acc)[NG][16], SlBars* B, uint32_t tmem, int q, int half,
                                         int lane, int nkb, int& it, int* status) {
  int ok = 1;
  const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * 16);
  for (int w = 0; w < nkb && ok; ++w, ++it) {
#pragma unroll
    for (int j = 0; j < NG; ++j) {
      if (ok) {  // (warp-uniform: the TMEM accesses are warp-collective)
        if (lane == 0) ok = sl_wait(&B->tfull[j & 1], (uint32_t)(((NG / 2) * it + (j >> 1)) & 1), status);
        ok = __shfl_sync(0xffffffffu, ok, 0);
        __syncwarp();
      }
      if (ok) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          uint32_t r[SL_S][4];
          const uint32_t ta = tbase + (uint32_t)((j & 1) * 256) + sl_part<FRAG>(h);
#pragma unroll
          for (int g = 0; g < SL_S; ++g) sl_tmem_ld4<FRAG>(ta + g * SL_BN, r[g]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int g = 0; g < SL_S; ++g)
#pragma unroll
            for (int c = 0; c < 4; ++c) asm volatile("" : "+r"(r[g][c]));
#pragma unroll
          for (int g = 0; g < SL_S; ++g) sl_tmem_st4<FRAG>(ta + g * SL_BN, SL_MAGIC);
          if (h == 3) {  // the set's values are in registers, the constants in place
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) sl_arrive(&B->tempty[j & 1]);
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            // a_0 2^48 + (a_1 2^8 + a_2) 2^32 + (a_3 2^8 + a_4) 2^16 + (a_5 2^8 + a_6), biased
            unsigned long long x = acc[j][h * 4 + c];
            x += (unsigned long long)(r[3][c] * 256u + r[4][c]) * 65536ull;
            x += (unsigned long long)(r[5][c] * 256u + r[6][c]);
            x += (unsigned long long)(r[0][c] * 65536u + r[1][c] * 256u + r[2][c]) << 32;
            acc[j][h * 4 + c] = x;
          }
        }
      }
    }
  }
  return ok != 0;
}

__device__ __forceinline__ void sl_tmem_alloc(uint32_t* sh) {  // one warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sl_u32(sh)), "r"(512));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void sl_tmem_free(uint32_t tmem) {  // the same warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}
// after an expired wait some copies may still be in flight: a bounded pause (~1 ms)
// lets them land before the CTA's shared memory is released (one thread)
__device__ __forceinline__ void sl_pause(const int* status) {
  if (*(const volatile int*)status != 0)
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);
}

// tensor map of a buffer of digit blocks, boxes of box_rows rows of all digits (syrk_sl.cu)
int wl_sl_map(cov_handle* h, CUtensorMap* map, void* base, int64_t blocks, int box_rows);
