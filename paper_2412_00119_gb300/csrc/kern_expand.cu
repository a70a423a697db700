// kern_expand.cu -- fixed random expansion layer for integer-valued inputs
// (Sec. 3.2, footnote to the binarisation step: a fixed random input layer
// with weights in {+-1} and sign activation lets the BMLP take non-binary
// inputs directly).
//
//   a_mu,k = +1  iff  z = sum_i x[mu][i] e_k,i >= 0    (sign(0) = +1)
//
// x: unsigned 8-bit inputs (pixel intensities); e_k,i: bit i of row k of the
// packed expansion matrix E (1 <-> +1).  z is summed exactly in int32
// (|z| <= 255 D < 2^31).  The output is packed like every activation (bit
// k % 64 of word k / 64, pad bits 0), i.e. bmlp_train / bmlp_predict input
// for K_0 = K.
//
// k_expand_tc (D <= kTcMaxD, x aligned to 4 bytes): the product on the tensor
// cores, exact in 4-bit operands.  A byte is four base-4 digits, x = d0 + 4 d1 + 16 d2 + 64 d3, and 0,
// 1, 2, 3 and +-1 are e2m1 values, so z is the sum of four e2m1 x e2m1 products
// with block scales 1, 4, 16 and 64 (UE8M0 holds powers of two); every product
// is an integer and |z| <= 255 D < 2^24, so the fp32 sums are exact in any
// order.  A CTA keeps one tile of up to 256 neurons, expanded into shared memory
// once (K-major, 128B swizzle), and walks over tiles of 128 patterns:
//   - 4 loader warps copy pieces of 256 bytes per row into a ring of two;
//   - 16 producer warps in four groups take chunks of 64 inputs in turn: a lane
//     per pattern row turns 64 bytes into 4 x 8 tensor-memory columns (digit
//     planes; 3 operations per byte);
//   - one thread issues the four MMAs (K = 64) of a chunk, one per plane, each
//     with its plane's scales, all against the same weight columns: the weights
//     are read from shared memory and never written again;
//   - 8 epilogue warps read the sums (a lane per pattern), shift the sign bits
//     into words and store them.
// Bound: the producers, 560 to 590 clocks per chunk at any width; at 256 neurons
// its MMAs take 512.  A tile takes 2,200 more for its epilogue.  60,000 x 784 ->
// 1024: 70 us repeated, 76 with x from memory (the dp4a kernel 804), of which the MMAs
// are 43.
// Every mbarrier wait is bounded like all others of the library.  This entry
// point has no handle that could report an expiry, so a CTA whose waits gave up
// writes its tiles again by a plain loop (expand_plain): the output is whole.
//
// k_expand_sign (the rest): a 128-pattern x 128-neuron tile per CTA of 256 threads, the
// inputs in chunks of 64 (one word of E per neuron): the chunk's bytes of x
// and the chunk's E bits, expanded to +-1 bytes, are staged in shared memory
// (rows padded to 17 words: conflict-free reads; the next chunk's raw words
// are already in flight in registers), then thread (tx, ty) runs
// dp4a.u32.s32 for patterns ty + 16 i and neurons tx + 16 j, i, j < 8 (64
// int32 sums).  Each warp ballots the signs of 2 patterns x 16 neurons and
// writes 16-bit pieces of the packed rows.  Neuron tiles vary fastest in the
// grid, so the CTAs of one pattern tile run together and read x from L2.
//
// k_expand_weights: E from the Philox stream of the expansion weights,
// e_k,i = +1 iff bit 31 of word i%4 of Philox (i/4, k, 33*2^16, 0) (the
// library's stream layout is listed in bmlp_internal.cuh); pad bits 0.
#include <algorithm>

#include "tc_common.cuh"

namespace bk {
namespace {

constexpr int kXThreads = 256;
constexpr int kXM = 128;         // patterns per CTA
constexpr int kXN = 128;         // neurons per CTA
constexpr int kXLd = 64 / 4 + 1; // 32-bit words per staged row (64 inputs + pad)
constexpr int kXMaxRowTiles = 65535;

__device__ __forceinline__ int dp4a_us(uint32_t a, uint32_t b, int c) {
  int d;
  asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

__global__ void __launch_bounds__(kXThreads, 2)
    k_expand_sign(const uint8_t* __restrict__ x, int64_t n, int D, bool vec,
                  const uint64_t* __restrict__ E, int K, int nwD, uint64_t* __restrict__ out,
                  int nwK) {
  __shared__ uint32_t xs[kXM][kXLd];
  __shared__ uint32_t es[kXN][kXLd];
  const int n0 = blockIdx.x * kXN;
  const int64_t m0 = (int64_t)blockIdx.y * kXM;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  int acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0;

  // thread t stages words q = t + 256 v (v < 8) of the x tile -- staged row
  // q / 16, word q % 16 = inputs 4 (q % 16) .. + 3 of the chunk, byte b = input
  // 4 (q % 16) + b, 0 past D and past n -- and half t & 1 of the E word of
  // neuron n0 + t / 2.  The raw words of chunk kc + 1 are loaded into
  // registers before chunk kc is computed, so the loads overlap the dp4a work.
  uint32_t xr[8], er;
  auto load_chunk = [&](int kc) {
    const int i0 = 64 * kc;
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const int q = threadIdx.x + kXThreads * v;
      const int r = q >> 4, c4 = q & 15;
      const int64_t m = m0 + r;
      const int i = i0 + 4 * c4;
      uint32_t w = 0;
      if (m < n) {
        const uint8_t* row = x + m * (int64_t)D;
        if (vec && i + 4 <= D) {
          w = __ldg(reinterpret_cast<const uint32_t*>(row + i));
        } else {
#pragma unroll
          for (int b = 0; b < 4; ++b)
            if (i + b < D) w |= (uint32_t)__ldg(row + i + b) << (8 * b);
        }
      }
      xr[v] = w;
    }
    const int k = n0 + (threadIdx.x >> 1);
    er = k < K ? (uint32_t)(E[(int64_t)k * nwD + kc] >> (32 * (threadIdx.x & 1))) : 0u;
  };
  load_chunk(0);

#pragma unroll 1
  for (int kc = 0; kc < nwD; ++kc) {
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const int q = threadIdx.x + kXThreads * v;
      xs[q >> 4][q & 15] = xr[v];
    }
    {
      // E half -> eight words of +-1 bytes (0x01 / 0xFF); neurons past K
      // stage zeros
      const int r = threadIdx.x >> 1, h = threadIdx.x & 1;
      const bool live = n0 + r < K;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        // nibble -> one bit per byte (the shifted copies do not overlap)
        const uint32_t p = (((er >> (4 * q)) & 0xFu) * 0x00204081u) & 0x01010101u;
        es[r][8 * h + q] = live ? ~(p * 0xFEu) : 0u;
      }
    }
    __syncthreads();
    if (kc + 1 < nwD) load_chunk(kc + 1);
#pragma unroll 4
    for (int c4 = 0; c4 < 16; ++c4) {
      uint32_t a[8], b[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) a[i] = xs[ty + 16 * i][c4];
#pragma unroll
      for (int j = 0; j < 8; ++j) b[j] = es[tx + 16 * j][c4];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = dp4a_us(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }

  // lanes 0..15 hold pattern ty = 2 warp, lanes 16..31 pattern ty = 2 warp + 1,
  // lane tx neuron n0 + tx + 16 j: each half of the ballot is 16 consecutive
  // neurons of one pattern
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int64_t m = m0 + ty + 16 * i;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int nn = n0 + tx + 16 * j;
      const unsigned bits = __ballot_sync(0xffffffffu, nn < K && acc[i][j] >= 0);
      const int piece = (n0 + 16 * j) >> 4;   // 16-bit piece of the packed row
      if ((lane & 15) == 0 && m < n && piece < 4 * nwK)
        reinterpret_cast<uint16_t*>(out + m * (int64_t)nwK)[piece] = (uint16_t)(bits >> (lane & 16));
    }
  }
}

// ---------------------------------------------------------------------------
// The tensor-core kernel.
// ---------------------------------------------------------------------------
using namespace tc;

constexpr int XM = 128;                   // patterns per tile (MMA M)
constexpr int kXMaxN = 256;               // neurons per CTA at most (MMA N)
constexpr int kChunk = 64;                // inputs per MMA
constexpr int kXPiece = 256;              // bytes per row and piece (4 chunks)
constexpr int kXPieces = 2;
constexpr int kXRow = kXPiece + 16;       // staged row (16 of padding: banks)
constexpr int kXPieceBytes = XM * kXRow;
constexpr int kXStages = 5;
constexpr int kXGroups = 4;
constexpr int kXProdWarps = 4 * kXGroups, kXLoadWarps = 4, kXEpiWarps = 8;
constexpr int kXMma = kXProdWarps, kXLoad0 = kXMma + 1, kXEpi0 = kXLoad0 + kXLoadWarps;
constexpr int kXTcThreads = 32 * (kXEpi0 + kXEpiWarps);
constexpr int kXSfA = kXMaxN, kXSfB = kXSfA + 4 * 16, kXStageCol = kXSfB + 16;
static_assert(kXStageCol + 32 * kXStages <= 512, "TMEM budget");
constexpr uint32_t kNoTile = 0xFFFFFFFFu;
constexpr int kXWeightBytes = 4 * kXMaxN * 128;   // 4 blocks of 256 inputs x 256 neurons, and the like
constexpr int kTcMaxD = 4608;                     // 18 blocks of 256 inputs x 64 neurons

struct __align__(8) XShared {
  unsigned long long piece_full[kXPieces], piece_empty[kXPieces];
  unsigned long long full[kXStages], empty[kXStages];
  unsigned long long done, drained;
  unsigned long long left;   // the MMAs of an issuer that gave up completed
  uint32_t tmem_base;
  int failed, left_failed;
};
constexpr size_t kXSmem = 1024 + 18 * 64 * 128 + kXPieces * kXPieceBytes + sizeof(XShared);
static_assert(18 * 64 * 128 >= kXWeightBytes, "the weight buffer holds every choice of tile");
static_assert(kXSmem <= 232448, "shared memory of one CTA");

// 64 bytes (16 words) -> digit plane 2 h of columns v[0..7], plane 2 h + 1 of
// v[8..15].  Column g holds the digits of words 2 g and 2 g + 1: nibble i is
// byte i / 2 of word 2 g + i % 2.  Digit d becomes the e2m1 value d: 2 d, and 5
// for d = 3.
__device__ __forceinline__ void digit_planes(const uint32_t (&w)[16], int h, uint32_t (&v)[16]) {
#pragma unroll
  for (int g = 0; g < 8; ++g) {
    const uint32_t a = w[2 * g], b = w[2 * g + 1];
    const uint32_t u = h == 0 ? ((a & 0x0F0F0F0Fu) | ((b << 4) & 0xF0F0F0F0u))
                              : (((a >> 4) & 0x0F0F0F0Fu) | (b & 0xF0F0F0F0u));
    v[g] = ((u << 1) & 0x66666666u) - (u & (u >> 1) & 0x11111111u);
    v[8 + g] = ((u >> 1) & 0x66666666u) - ((u >> 2) & (u >> 3) & 0x11111111u);
  }
}

// A weight byte (8 inputs) as e2m1 in the same order: nibble i is input
// i / 2 + 4 (i % 2); bit 1 -> 0x2 (+1), bit 0 -> 0xA (-1).
__device__ __forceinline__ uint32_t weight_nibbles(uint32_t byte) {
  const uint32_t neg = ~byte;
  const uint32_t even = ((neg & 0xFu) * 0x01020408u) & 0x08080808u;
  const uint32_t odd = (((neg >> 4) & 0xFu) * 0x01020408u) & 0x08080808u;
  return 0x22222222u | even | (odd << 4);
}

// The tiles of this CTA without the tensor cores, barriers or shared memory, by one
// warp (only that one looks for a failure: a check by every warp at the end of the
// kernel cost small calls 0.2 to 0.4 us): a 32-bit word of the output per lane
// and turn.
__device__ __noinline__ void expand_plain(const uint8_t* x, int64_t n, int D, const uint64_t* E, int K, int nwD,
                                          uint64_t* out, int nwK, int nb) {
  const int words = nb / 32;
#pragma unroll 1
  for (int64_t t = blockIdx.y; t * XM < n; t += gridDim.y) {
#pragma unroll 1
    for (int i = threadIdx.x & 31; i < XM * words; i += 32) {
      const int64_t m = t * XM + i / words;
      const int nn = (int)blockIdx.x * nb + 32 * (i % words);
      if (m >= n || (nn >> 5) >= 2 * nwK) continue;
      uint32_t word = 0u;
#pragma unroll 1
      for (int j = 0; j < 32 && nn + j < K; ++j) {
        const uint64_t* e = E + (int64_t)(nn + j) * nwD;
        int z = 0;
#pragma unroll 1
        for (int c = 0; c < D; ++c) {
          const int v = x[m * D + c];
          z += (e[c >> 6] >> (c & 63) & 1u) != 0u ? v : -v;
        }
        word |= z >= 0 ? 1u << j : 0u;
      }
      reinterpret_cast<uint32_t*>(out + m * nwK)[nn >> 5] = word;
    }
  }
}

// kBytes: 16 or 4, the copies that every row of x allows, or 1: rows that start at
// any byte of an x aligned to words.  Those are copied as the words that hold
// them, zeros past the row's end, and shifted by the producers: 600 x 70 -> 1024
// 7.3 us, 20,000 x 785 -> 1024 53 (byte loads in the loaders 16.5 and 100, the dp4a
// kernel 12.4 and 357).
// fail_tile: the wait for the sums of each CTA's tile of this number is taken as
// expired (tests; kNoTile: none).
template <int kBytes>
__global__ void __launch_bounds__(kXTcThreads, 1)
    k_expand_tc(const uint8_t* __restrict__ x, int64_t n, int D, const uint64_t* __restrict__ E, int K, int nwD,
                uint64_t* __restrict__ out, int nwK, int nb, uint32_t fail_tile) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* pieces = base + 18 * 64 * 128;
  XShared* sh = reinterpret_cast<XShared*>(pieces + kXPieces * kXPieceBytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* failed = &sh->failed;
  const int n0 = blockIdx.x * nb;
  const int nchunks = (D + kChunk - 1) / kChunk, npc = (D + kXPiece - 1) / kXPiece;
  const int64_t tiles = (n + XM - 1) / XM;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kXPieces; ++s) {
      mbar_init(&sh->piece_full[s], 32 * kXLoadWarps);
      mbar_init(&sh->piece_empty[s], kXProdWarps);
    }
    for (int s = 0; s < kXStages; ++s) {
      mbar_init(&sh->full[s], 4);
      mbar_init(&sh->empty[s], 1);
    }
    mbar_init(&sh->done, 1);
    mbar_init(&sh->drained, kXEpiWarps);
    mbar_init(&sh->left, 1);
    sh->failed = sh->left_failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kXMma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(&sh->tmem_base)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // the tile's weights: block b of 256 inputs is nb rows of 128 bytes; 32 inputs
  // of one neuron are one 16-byte chunk c of its row, at chunk c ^ (row % 8)
  for (int i = threadIdx.x; i < nb * 8 * npc; i += kXTcThreads) {
    const int c = i % (8 * npc), r = i / (8 * npc);
    const uint32_t bitsw = (n0 + r < K && c < 2 * nwD)
                               ? reinterpret_cast<const uint32_t*>(E + (int64_t)(n0 + r) * nwD)[c] : 0u;
    uint32_t v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = weight_nibbles(bitsw >> (8 * q));
    sts128(smem_u32(base) + (uint32_t)((c >> 3) * nb * 128 + r * 128 + 16 * ((c & 7) ^ (r & 7))), v);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sh->tmem_base;
  if (warp < 4) {
    const uint32_t at = tmem + ((uint32_t)(32 * warp) << 16);
#pragma unroll
    for (int p = 0; p < 5; ++p) {
      // scales of plane p (4^p: UE8M0 127 + 2 p), then the weights' (1)
      const uint32_t v = (p < 4 ? 127u + 2u * p : 127u) * 0x01010101u;
      asm volatile(
          "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, "
          "%1, %1, %1, %1};" ::"r"(at + (uint32_t)(kXSfA + 16 * p)), "r"(v) : "memory");
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  if (warp < kXProdWarps) {
    // ---------------- producers ----------------
    const int grp = warp >> 2, q = warp & 3;
    const uint32_t row0 = smem_u32(pieces) + (uint32_t)((32 * q + lane) * kXRow);
    const uint32_t lanes = (uint32_t)(32 * q) << 16;
    uint32_t slot = 0, pph = 0;                        // ring slot of the piece, its parity
    uint32_t s = (uint32_t)grp, eph = 1;               // stage of the group's next chunk, parity of "empty"
    int ch = grp;                                      // that chunk, counted in the current tile
    bool ok = true;
#pragma unroll 1
    for (int64_t t = blockIdx.y; t < tiles && ok; t += gridDim.y, ch -= nchunks) {
      // bits before the row's first byte in its words
      const uint32_t skew =
          kBytes == 1 ? 8u * (uint32_t)((reinterpret_cast<uintptr_t>(x) + (t * XM + 32 * q + lane) * D) & 3) : 0u;
#pragma unroll 1
      for (int p = 0; p < npc && ok; ++p) {
        ok = __all_sync(0xffffffffu, mbar_wait(&sh->piece_full[slot], pph, failed));
        const int cend = min(nchunks, 4 * (p + 1));
#pragma unroll 1
        for (; ch < cend && ok; ch += kXGroups) {
          uint32_t w[16];
          const uint32_t src = row0 + slot * (uint32_t)kXPieceBytes + (uint32_t)(kChunk * (ch - 4 * p));
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint4 v = lds128(src + 16u * i);
            w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
          }
          if constexpr (kBytes == 1) {
            uint32_t next;
            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(next) : "r"(src + 64u) : "memory");
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = __funnelshift_r(w[i], i < 15 ? w[i + 1] : next, skew);
          }
          ok = __all_sync(0xffffffffu, mbar_wait(&sh->empty[s], eph, failed));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t v[16];
            digit_planes(w, h, v);
            tmem_store16(tmem + lanes + (uint32_t)kXStageCol + 32u * s + 16u * h, v);
          }
          asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh->full[s]);
          s += kXGroups;
          if (s >= kXStages) {
            s -= kXStages;
            eph ^= 1u;
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh->piece_empty[slot]);
        if (++slot == kXPieces) {
          slot = 0;
          pph ^= 1u;
        }
      }
    }
  } else if (warp >= kXLoad0 && warp < kXEpi0) {
    // ---------------- loaders ----------------
    constexpr int kStep = kBytes == 1 ? 4 : kBytes;   // bytes per store to shared memory
    constexpr int kPer = kXPiece / kStep;
    const int tid = threadIdx.x - 32 * kXLoad0;
    constexpr int kRows = 32 * kXLoadWarps / kPer > 0 ? 32 * kXLoadWarps / kPer : 1;   // rows per round of copies
    constexpr int kCols = kPer / (32 * kXLoadWarps) > 0 ? kPer / (32 * kXLoadWarps) : 1;   // columns of a thread
    const int r0 = tid / kPer, c0 = kStep * (tid % kPer);
    uint32_t slot = 0, ph = 1;
    bool ok = true;
#pragma unroll 1
    for (int64_t t = blockIdx.y; t < tiles && ok; t += gridDim.y) {
      const uint8_t* rows = x + (t * XM + r0) * D + (kBytes == 1 ? 0 : c0);
      // rows past n keep what is there: their outputs are dropped (e2m1 has no NaN)
      const int live = (int)min((int64_t)XM, n - t * XM) - r0;
#pragma unroll 1
      for (int p = 0; p < npc && ok; ++p) {
        ok = mbar_wait(&sh->piece_empty[slot], ph, failed);
        if (!ok) break;
        if constexpr (kBytes == 1) {
          // the aligned word that is c past the first of a row, its bytes of the row
          auto copy = [&](const uint8_t* row, uint32_t to, int c) {
            const int skew = (int)(reinterpret_cast<uintptr_t>(row) & 3);
            const int size = min(4, max(0, D + skew - c));
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;"
                         ::"r"(to), "l"(size > 0 ? row + (c - skew) : x), "r"(size) : "memory");
          };
          const uint32_t to0 = smem_u32(pieces) + slot * (uint32_t)kXPieceBytes;
          const uint8_t* row = rows;
          uint32_t to = to0 + (uint32_t)(r0 * kXRow + c0);
#pragma unroll 8
          for (int i = 0; i < live; i += kRows, row += kRows * D, to += (uint32_t)(kRows * kXRow))
            copy(row, to, kXPiece * p + c0);
          static_assert(32 * kXLoadWarps == XM, "a row's last word by a thread each");
          if (t * XM + tid < n)
            copy(x + (t * XM + tid) * D, to0 + (uint32_t)(tid * kXRow + kXPiece), kXPiece * (p + 1));
        } else {
#pragma unroll 1
          for (int e = 0; e < kCols; ++e) {
            const int c = kXPiece * p + c0 + e * 32 * kXLoadWarps * kStep;   // the copy's first input
            const uint8_t* src = rows + kXPiece * p + e * 32 * kXLoadWarps * kStep;
            uint32_t to = smem_u32(pieces) + slot * (uint32_t)kXPieceBytes +
                          (uint32_t)(r0 * kXRow + c0 + e * 32 * kXLoadWarps * kStep);
#pragma unroll 4
            for (int i = 0; i < live; i += kRows, src += kRows * D, to += (uint32_t)(kRows * kXRow)) {
              const bool on = c < D;   // D is a multiple of kBytes
              cp_async_or_zero<kBytes>(to, on ? src : x, on);
            }
          }
        }
        cp_async_arrive(&sh->piece_full[slot]);
        if (++slot == kXPieces) {
          slot = 0;
          ph ^= 1u;
        }
      }
    }
    cp_async_wait_all();   // no copy outlives its thread
  } else if (warp == kXMma) {
    // ---------------- MMA issuer ----------------
    const bool lead = elect_one();
    const uint32_t d = uniform(tmem);
    const uint64_t bd0 = smem_desc(uniform(smem_u32(base)));
    const uint32_t idesc = idesc_f4(XM, nb);
    uint32_t s = 0, ph = 0, dph = 1;
    bool ok = true;
#pragma unroll 1
    for (int64_t t = blockIdx.y; t < tiles && ok; t += gridDim.y) {
      ok = __all_sync(0xffffffffu, mbar_wait(&sh->drained, dph, failed));
      dph ^= 1u;
#pragma unroll 1
      for (int ch = 0; ch < nchunks && ok; ++ch) {
        ok = __all_sync(0xffffffffu, mbar_wait(&sh->full[s], ph, failed));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t bd = bd0 + (uint64_t)((uint32_t)(ch >> 2) * (uint32_t)(8 * nb) + 2u * (uint32_t)(ch & 3));
        const uint32_t ta = d + (uint32_t)kXStageCol + 32u * s;
        if (lead) {
#pragma unroll
          for (int p = 0; p < 4; ++p)
            mma_f4_ts(d, ta + 8 * p, bd, idesc, d + kXSfA + 16 * p, d + kXSfB, (ch > 0 || p > 0) ? 1u : 0u);
          mma_commit(&sh->empty[s]);
        }
        if (++s == kXStages) {
          s = 0;
          ph ^= 1u;
        }
      }
      if (ok && lead) mma_commit(&sh->done);
      __syncwarp();
    }
    if (!ok && lead) {
      // no MMA outlives its operands and its tensor memory
      mma_commit(&sh->left);
      mbar_wait(&sh->left, 0, &sh->left_failed);
    }
    __syncwarp();
  } else if (warp >= kXEpi0) {
    // ---------------- epilogue ----------------
    const int sub = warp & 3, half = (warp - kXEpi0) >> 2;
    // this warp's words of 32 neurons
    const int first = half * ((nb / 32 + 1) / 2), words = (nb / 32 + 1 - half) / 2;
    uint32_t tile = 0;
#pragma unroll 1
    for (int64_t t = blockIdx.y; t < tiles; t += gridDim.y, ++tile) {
      if (!__all_sync(0xffffffffu, mbar_wait(&sh->done, tile & 1u, failed))) break;
      if (tile == fail_tile) {
        *failed = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      uint32_t word[4] = {0u, 0u, 0u, 0u};
      sign_words<4>(word, tmem + ((uint32_t)(32 * sub) << 16) + (uint32_t)(32 * first), words, 0.0f);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->drained);
      const int64_t m = t * XM + 32 * sub + lane;
      if (m < n) {
        uint32_t* row = reinterpret_cast<uint32_t*>(out + m * nwK);
#pragma unroll
        for (int cb = 0; cb < 4; ++cb) {
          const int nn = n0 + 32 * (first + cb), valid = K - nn;
          const uint32_t keep = valid >= 32 ? 0xffffffffu : (valid <= 0 ? 0u : (1u << valid) - 1u);
          // words wholly past K (inside the row's last 64-bit word) are written 0
          if (cb < words && (nn >> 5) < 2 * nwK) row[nn >> 5] = word[cb] & keep;
        }
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == kXMma) {
    const bool redo = *failed != 0;
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    if (redo) expand_plain(x, n, D, E, K, nwD, out, nwK, nb);
  }
}

template <int kBytes>
cudaError_t launch_expand_tc(const uint8_t* x, int64_t n, int D, const uint64_t* E, int K, uint64_t* out,
                             cudaStream_t st, uint32_t fail_tile) {
  const int blocks = (D + kXPiece - 1) / kXPiece;   // of 256 inputs
  const int64_t tiles = (n + XM - 1) / XM;
  const int sms = sm_count();
  // Neurons per CTA: a chunk takes 560 to 590 clocks at any width, so the fewest
  // rounds of pattern tiles over the widths whose weights fit, of equal ones the
  // narrowest (halvings of 256 in place of steps of 32: 60,000 x 3072 -> 1024
  // 770 us, now 507; 600 x 784 -> 2048 14.5, now 10.4).
  const int words = (K + 63) / 64;   // of 64 neurons in a packed row
  int nb = 64;
  int64_t gy = 1, rounds = INT64_MAX;
  for (int w = 64; w <= kXMaxN && w * blocks <= 18 * 64; w += 32) {
    const int64_t nt = (64ll * words + w - 1) / w, g = std::min(tiles, std::max<int64_t>(1, sms / nt));
    const int64_t r = (tiles + g - 1) / g * ((nt * g + sms - 1) / sms);
    if (r < rounds) {
      rounds = r;
      nb = w;
      gy = g;
    }
  }
  const unsigned nt = (unsigned)((64ll * words + nb - 1) / nb);
  const cudaError_t e = cudaFuncSetAttribute(k_expand_tc<kBytes>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kXSmem);
  if (e != cudaSuccess) return e;
  k_expand_tc<kBytes><<<dim3(nt, (unsigned)gy), kXTcThreads, kXSmem, st>>>(x, n, D, E, K, (D + 63) / 64, out,
                                                                          (K + 63) / 64, nb, fail_tile);
  return cudaGetLastError();
}

__global__ void k_expand_weights(uint32_t key0, uint32_t key1, int K, int D, int nwD,
                                 uint64_t* __restrict__ E) {
  const int64_t total = (int64_t)K * nwD;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int k = (int)(idx / nwD), w = (int)(idx % nwD);
    uint64_t word = 0;
#pragma unroll 1
    for (int g = 0; g < 16; ++g) {  // inputs 64 w + 4 g .. + 3: one Philox call
      const int i = 64 * w + 4 * g;
      if (i >= D) break;
      const uint4 u = philox4x32_10(make_uint4((uint32_t)(i / 4), (uint32_t)k, 33u << 16, 0u), key0, key1);
      const uint64_t s = (u.x >> 31) | ((u.y >> 31) << 1) | ((u.z >> 31) << 2) | ((u.w >> 31) << 3);
      word |= s << (4 * g);
    }
    const int valid = D - 64 * w;
    if (valid < 64) word &= (1ull << valid) - 1ull;
    E[idx] = word;
  }
}

}  // namespace

void launch_expand_weights(uint64_t seed, int K, int D, uint64_t* E, cudaStream_t st) {
  const int nwD = (D + 63) / 64;
  const int64_t total = (int64_t)K * nwD;
  const int64_t blocks = (total + 255) / 256;
  k_expand_weights<<<(unsigned)(blocks < 4096 ? blocks : 4096), 256, 0, st>>>(
      (uint32_t)(seed & 0xFFFFFFFFu), (uint32_t)(seed >> 32), K, D, nwD, E);
}

cudaError_t launch_expand_sign(const uint8_t* x, int64_t n, int D, const uint64_t* E, int K, uint64_t* out,
                               cudaStream_t st, int64_t fail_tile) {
  const int nwD = (D + 63) / 64, nwK = (K + 63) / 64;
  const uint32_t ft = fail_tile < 0 ? kNoTile : (uint32_t)fail_tile;
  if (D <= kTcMaxD && reinterpret_cast<uintptr_t>(x) % 4 == 0) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(x) | (uintptr_t)(uint32_t)D;
    return (a & 15) == 0 ? launch_expand_tc<16>(x, n, D, E, K, out, st, ft)
                         : ((a & 3) == 0 ? launch_expand_tc<4>(x, n, D, E, K, out, st, ft)
                                         : launch_expand_tc<1>(x, n, D, E, K, out, st, ft));
  }
  const unsigned ntiles = (unsigned)((K + kXN - 1) / kXN);
  // patterns in launches of at most 65,535 tiles of 128 (the grid's y limit)
  const int64_t per = (int64_t)kXMaxRowTiles * kXM;
  for (int64_t off = 0; off < n; off += per) {
    const int64_t cnt = (n - off < per) ? n - off : per;
    const uint8_t* xo = x + off * (int64_t)D;
    const bool vec = (D % 4 == 0) && (reinterpret_cast<uintptr_t>(xo) % 4 == 0);
    const dim3 grid(ntiles, (unsigned)((cnt + kXM - 1) / kXM));
    k_expand_sign<<<grid, kXThreads, 0, st>>>(xo, cnt, D, vec, E, K, nwD, out + off * (int64_t)nwK, nwK);
  }
  return cudaGetLastError();
}

}  // namespace bk
