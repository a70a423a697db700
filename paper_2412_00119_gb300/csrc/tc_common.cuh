// tc_common.cuh -- device helpers shared by the tcgen05 kernels: mbarrier
// waits (bounded), asynchronous copies, shared-memory matrix descriptors, the
// tcgen05.mma issue (kind::mxf4; kind::f8f6f4 for the peak kernel) and commit,
// the expansion of bit-packed +-1 vectors into e2m1, and the tensor-memory
// loads and stores around them.
#pragma once

#include "bmlp_internal.cuh"

namespace bk {
namespace tc {

constexpr unsigned kFull = 0xffffffffu;
constexpr int KB = 128;  // K elements (bytes of e4m3) per stage row
constexpr unsigned long long kWaitCycles = 4000000000ull;  // ~2 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Bounded wait for the phase with the given parity; false on expiry (after
// `limit` SM clock cycles) or when another thread already recorded a failure.
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, uint32_t parity,
                                          volatile int* failed,
                                          unsigned long long limit = kWaitCycles) {
  const uint32_t a = smem_u32(bar);
  uint32_t ok;
  auto try_wait = [&]() {
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok) : "r"(a), "r"(parity) : "memory");
  };
  try_wait();                       // most waits end here, without reading the clock
  if (ok) return true;
  const unsigned long long t0 = clock64();
  while (true) {
    try_wait();
    if (ok) return true;
    if (*failed) return false;
    if (clock64() - t0 > limit) {
      *failed = 1;
      return false;
    }
  }
}

// One lane of the calling (converged) warp.  MMAs are issued by a whole warp with
// this lane elected around the instruction alone: the operands are then computed
// in uniform registers, where the instruction takes them from (under `lane == 0`
// every operand is moved there one by one, 90 clocks per MMA).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(p));
  return p != 0u;
}
// A value that is the same in every lane, into a uniform register.
__device__ __forceinline__ uint32_t uniform(uint32_t v) { return __reduce_max_sync(kFull, v); }

// Shared-memory matrix descriptor: K-major, SWIZZLE_128B, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);           // start address
  d |= (uint64_t)1 << 16;                              // leading byte offset (unused for SW128 K-major)
  d |= (uint64_t)(1024 >> 4) << 32;                    // stride byte offset
  d |= (uint64_t)1 << 46;                              // descriptor version (sm_100 family)
  d |= (uint64_t)2 << 61;                              // swizzle: 128B
  return d;
}

// Instruction descriptor, kind::f8f6f4: D fp32, A = B = e4m3, both K-major,
// M x N per instruction (K = 32).
constexpr uint32_t idesc_f8(int M, int N) {
  return (1u << 4)                        // D format: f32
         | (0u << 7) | (0u << 10)         // A, B format: e4m3
         | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

template <uint32_t kIdesc>
__device__ __forceinline__ void mma_f8(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(kIdesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(unsigned long long* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_tx(unsigned long long* bar, uint32_t bytes) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}"
               ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// 1-D bulk copy global -> this CTA's shared memory, completing on `bar`
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// ---------------------------------------------------------------------------
// +-1 as e2m1 (4 bits), tcgen05.mma kind::mxf4 with unit scales.
//
// +-1 (0x2 / 0xA) is exact in e2m1, a zero nibble is 0, and with every block
// scale 1 (UE8M0 0x7F) each product is +-1 or 0 and every partial sum an
// integer of magnitude <= K < 2^24, exact in fp32 in any order.  One MMA
// (M128 N256 K64) takes the time of an e4m3 one with half the K, and a stage
// row of 128 bytes holds 256 elements: 4,474 T MAC/s (operands in shared
// memory) and 4,846 T (A in tensor memory) against 1,935 T for e4m3, random
// +-1 on all 152 SMs.
//
// A 32-bit word x of bits becomes four words of eight nibbles: word j holds
// the sign bits of x's bits 4 n + 3 - j (n = 0..7), so each output word is one
// shift and one logical operation.  The order of the K-elements inside a
// group of 32 differs from the bit order, alike in both operands, and so does
// the sign (a set bit, +1, becomes -1): neither changes a product sum.
// ---------------------------------------------------------------------------
constexpr int KF = 256;  // K elements (two e2m1 per byte) per 128-byte stage row
constexpr uint32_t kUnitScales = 0x7F7F7F7Fu;  // four UE8M0 scales of 1

__device__ __forceinline__ void e2m1_words(uint32_t x, uint32_t (&w)[4]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) w[j] = ((x << j) & 0x88888888u) ^ 0x22222222u;
}

// Instruction descriptor, kind::mxf4: A = B = e2m1, UE8M0 scales, both
// K-major, M x N per instruction (K = 64).
__host__ __device__ constexpr uint32_t idesc_f4(int M, int N) {
  return (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | (1u << 23) | ((uint32_t)(M >> 4) << 24);
}

// A in tensor memory (lane = row, eight e2m1 per 32-bit column), B in shared
// memory, the block scales of both at tensor-memory columns sf (all 1).
__device__ __forceinline__ void mma_f4_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc,
                                          uint32_t idesc, uint32_t sfa, uint32_t sfb,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %6, 0;\n"
      " tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], [%1], %2, %3, [%4], [%5], p;\n}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(sfa), "r"(sfb), "r"(accumulate));
}

// 16: every row of a matrix of nw-word rows allows 16-byte copies; else 8.
__host__ __device__ __forceinline__ int row_align(const void* base, int nw) {
  return ((reinterpret_cast<uintptr_t>(base) | (uintptr_t)(8 * (uint32_t)nw)) & 15) == 0 ? 16 : 8;
}

// Asynchronous copy of kBytes (16 past L1, or 8 or 4) to shared memory; zeros
// instead when !live (src is then not read, but must be a valid address).
template <int kBytes>
__device__ __forceinline__ void cp_async_or_zero(uint32_t dst, const void* src, bool live) {
  const int n = live ? kBytes : 0;
  if constexpr (kBytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %3, %2;" ::"r"(dst), "l"(src), "r"(n), "n"(kBytes) : "memory");
}
// Arrive on the barrier when this thread's copies so far have completed.
__device__ __forceinline__ void cp_async_arrive(unsigned long long* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts128(uint32_t a, const uint32_t (&v)[4]) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// 16 TMEM columns of this warp's 32 lanes.
__device__ __forceinline__ void tmem_store16(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}

// 32 TMEM columns of this warp's 32 lanes from each lane's 256 bits.
__device__ __forceinline__ void tmem_store_row256(uint32_t taddr, const uint32_t (&x)[8]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {   // 16 columns at a time (registers)
    uint32_t v[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t w[4];
      e2m1_words(x[4 * h + q], w);
#pragma unroll
      for (int j = 0; j < 4; ++j) v[4 * q + j] = w[j];
    }
    tmem_store16(taddr + 16u * (uint32_t)h, v);
  }
}

// 16 TMEM columns of this warp's 32 lanes; tmem_wait_ld before they are used.
__device__ __forceinline__ void tmem_load16(uint32_t (&v)[16], uint32_t taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}
// v: loaded values that may be used after it.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                 "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
               :: "memory");
}

// Sign words of 32 kWords accumulator columns from taddr on, for this lane's row:
// bit j of word w is 1 where column 32 w + j minus npad is >= 0.  Each 16 columns
// are in flight while the 16 before are shifted into their word.
template <int kWords>
__device__ __forceinline__ void sign_words(uint32_t (&word)[kWords], uint32_t taddr, int words, float npad) {
  uint32_t v[2][16];
  tmem_load16(v[0], taddr);
  tmem_wait_ld(v[0]);
#pragma unroll
  for (int h = 0; h < 2 * kWords; ++h) {
    if (h >= 2 * words) break;
    if (h + 1 < 2 * words) tmem_load16(v[(h + 1) & 1], taddr + 16u * (uint32_t)(h + 1));
    uint32_t acc = (h & 1) ? word[h >> 1] : 0u;   // column 0 first; its sign ends in bit 31
    if (npad == 0.0f) {
#pragma unroll
      for (int j = 0; j < 16; ++j) acc = __funnelshift_l(v[h & 1][j], acc, 1);
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j)
        acc = __funnelshift_l(__float_as_uint(__uint_as_float(v[h & 1][j]) - npad), acc, 1);
    }
    word[h >> 1] = (h & 1) ? ~__brev(acc) : acc;
    if (h + 1 < 2 * words) tmem_wait_ld(v[(h + 1) & 1]);
  }
}

}  // namespace tc
}  // namespace bk
