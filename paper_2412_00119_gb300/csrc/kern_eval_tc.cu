// kern_eval_tc.cu -- tensor-core forward for forward-only evaluation
// (Sec. 3.1; Alg. 1 l.8-9 without the training side outputs), large batches.
//
// The same exact e2m1 formulation as the mini-batch kernel (+-1 with unit
// block scales, elements past K_in +1 in both operands and subtracted from the
// sums).
//
// A cluster of two CTAs computes 256 patterns x 256 neurons with
// tcgen05.mma.cta_group::2 (M = 256, N = 256, K = 64): CTA r of the pair holds
// pattern rows m0 + 128 r .. + 127 in its tensor memory (A operand) and stages
// weight rows n0 + 128 r .. + 127 in its shared memory (half of B; the MMA reads
// both halves); its tensor memory receives D rows 128 r .. + 127 for all 256
// neurons.  A pair moves 16 KB of operand per SM and k-step through shared
// memory, written and read once, in 512 clocks of MMA: half its bandwidth (with
// both operands in shared memory it would be all of it).
// The grid is persistent, one pair per two SMs; a pair takes tiles p, p + pairs,
// ..., neuron tiles varying fastest, so that the pairs in flight share pattern
// tiles and the layer's packed W (8 MB at 8192 x 8192) stays in L2.  All roles
// run on across tiles; only the MMAs of the next tile wait for the epilogue to
// have read the accumulators.  Warps of a CTA:
//   - 4 loader warps copy pieces of 1,024 K-elements (whole 128-byte lines of
//     128 pattern and 128 weight rows) into a ring of kPieces, with asynchronous
//     copies that complete on the piece's mbarrier;
//   - 16 producer warps in two groups take alternate k-steps of 256 elements: in
//     a group four warps expand the pattern rows into 32 tensor-memory columns
//     and four the weight rows into a 16 KB stage (128B swizzle);
//   - one thread of the even CTA issues the MMAs and commits to the "empty"
//     barriers of both; kRelays threads of the odd CTA, each in a warp of its own,
//     take its k-steps in turn and forward their "full" barriers (a remote
//     arrival with cluster-scope release takes 720 clocks; one thread doing them
//     all set the pace, 1,000 clocks per k-step);
//   - 8 epilogue warps read D (a lane per pattern), shift the sign bits into
//     words and store 128 neurons of a row at once.
// Measured, 65,536 patterns through 8192 -> 8192x4: 4.60 ms = 7.67 PFLOP/s (the
// e4m3 kernel before it 11.2 ms; this one with one relay and the MMAs issued
// under `lane == 0` 7.43 ms).  A k-step takes 566 clocks where its MMAs take 512,
// and a tile 3,100 more until both CTAs' accumulators are read (with the MMAs as
// two N = 128 halves, so that a half is read beside the other's, 5.02 ms).
// Every mbarrier wait is bounded; the first expiry stops every other wait of
// the CTA and the kernel counts it in *timeouts, releases its tensor memory
// and returns.
#include "tc_common.cuh"

namespace bk {
namespace {

using namespace tc;

constexpr int TM = 128;                  // pattern rows per CTA (MMA M = 256 per pair)
constexpr int TB = 128;                  // weight rows per CTA
constexpr int TN = 2 * TB;               // neurons per pair (MMA N)
constexpr int kSteps = 4;                // k-steps of KF = 256 elements per piece
constexpr int kPieceWords = 16;
constexpr int kPieces = 3;               // ring of bit pieces
constexpr int kBitRow = 144;             // bytes per staged bit row (16 of padding: banks)
constexpr int kBitBytes = (TM + TB) * kBitRow;
constexpr int kStages = 6;               // k-step stages
constexpr int B_BYTES = TB * 128;        // one weight stage
constexpr int kGroups = 2;
constexpr int kProdWarps = 8 * kGroups;
constexpr int kLoadWarps = 4, kEpiWarps = 8;
constexpr int kRelays = 4;               // the MMA warp (of the odd CTA) and three more
constexpr int kMmaWarp = kProdWarps;
constexpr int kLoad0 = kMmaWarp + kRelays, kEpi0 = kLoad0 + kLoadWarps;
constexpr int THREADS = 32 * (kEpi0 + kEpiWarps);
constexpr int TMEM_COLS = 512;
constexpr int kSfCol = TN;               // 16 + 16 columns of unit scales (A, B)
constexpr int kStageCol = kSfCol + 32;   // pattern stages of 32 columns
static_assert(kStageCol + 32 * kStages <= TMEM_COLS, "TMEM budget");
static_assert(THREADS <= 1024, "threads of a CTA");
constexpr uint32_t kIdesc = idesc_f4(2 * TM, TN);

struct __align__(8) EvShared {
  unsigned long long bits_full[kPieces];   // a piece's copies arrived
  unsigned long long bits_empty[kPieces];  // every producer warp has read it
  unsigned long long full[kStages];        // a k-step is expanded
  unsigned long long empty[kStages];       // its MMAs completed
  unsigned long long done;                 // a tile's MMAs completed
  unsigned long long drained;              // both CTAs' epilogues have read D (even CTA)
  uint32_t tmem_base;
  int failed;
};

constexpr size_t kSmemBytes = 1024 + kStages * B_BYTES + kPieces * kBitBytes + sizeof(EvShared);

__device__ __forceinline__ uint32_t pair_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ void pair_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;"
               ::: "memory");
}

// Bounded wait with cluster-scope acquire (the barrier collects an arrival
// from the peer CTA).
__device__ __forceinline__ bool mbar_wait_cluster(unsigned long long* bar, uint32_t parity,
                                                  volatile int* failed) {
  const uint32_t a = smem_u32(bar);
  uint32_t ok;
  auto try_wait = [&]() {
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok) : "r"(a), "r"(parity) : "memory");
  };
  try_wait();
  if (ok) return true;
  const unsigned long long t0 = clock64();
  while (true) {
    try_wait();
    if (ok) return true;
    if (*failed) return false;
    if (clock64() - t0 > kWaitCycles) {
      *failed = 1;
      return false;
    }
  }
}

// Arrive on the barrier at the same offset in CTA 0 of the cluster.
__device__ __forceinline__ void mbar_arrive_rank0(unsigned long long* bar) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(remote) : "r"(smem_u32(bar)));
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
}

__device__ __forceinline__ void mma_f4_pair(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t sfa,
                                            uint32_t sfb, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %6, 0;\n"
      " tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], [%1], %2, %3, [%4], [%5], p;\n}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(kIdesc), "r"(sfa), "r"(sfb), "r"(accumulate));
}

// Arrive once on the barrier at this offset in both CTAs of the pair when the
// MMAs issued so far complete.
__device__ __forceinline__ void mma_commit_pair(unsigned long long* bar) {
  const uint16_t mask = 0x3;
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
      ::"r"(smem_u32(bar)), "h"(mask) : "memory");
}

// kAlign: 16 where every row of both operands allows 16-byte copies, else 8.
template <int kAlign>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
    k_forward_eval_tc(const uint64_t* __restrict__ A, int64_t M, int nw, const uint64_t* __restrict__ W, int N,
                      int Kin, uint64_t* __restrict__ Aout, int nw_out, int ntiles, int64_t tiles,
                      unsigned int* __restrict__ timeouts) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* bits = base + kStages * B_BYTES;
  EvShared* sh = reinterpret_cast<EvShared*>(bits + kPieces * kBitBytes);
  const uint32_t rank = pair_rank();
  const int64_t pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  const int npc = (nw + kPieceWords - 1) / kPieceWords;   // pieces of a tile
  const int nks = (Kin + KF - 1) / KF;                    // k-steps of a tile
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* failed = &sh->failed;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kPieces; ++s) {
      mbar_init(&sh->bits_full[s], 32 * kLoadWarps);
      mbar_init(&sh->bits_empty[s], kProdWarps);
    }
    for (int s = 0; s < kStages; ++s) {
      // the warps of a producer group and, on the even CTA, the odd CTA's relayed arrival
      mbar_init(&sh->full[s], 8 + (rank == 0 ? 1 : 0));
      mbar_init(&sh->empty[s], 1);
    }
    mbar_init(&sh->done, 1);
    mbar_init(&sh->drained, 2 * kEpiWarps);
    sh->failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(&sh->tmem_base)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sh->tmem_base;
  if (warp < 4) {
    // unit scales, before any MMA of the pair
    const uint32_t at = tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)kSfCol;
#pragma unroll
    for (int h = 0; h < 2; ++h)
      asm volatile(
          "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, "
          "%1, %1, %1, %1};" ::"r"(at + 16u * h), "r"(kUnitScales) : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  pair_sync();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // set up beside the tail of the layer before this one
  pdl_wait();
  pdl_trigger();

  if (warp < kProdWarps) {
    // ---------------- producers ----------------
    const int grp = warp >> 3, q = warp & 3;
    const bool awarp = (warp & 4) == 0;
    const int r = 32 * q + lane;
    const uint32_t brow0 = smem_u32(bits) + (uint32_t)((awarp ? r : TM + r) * kBitRow);
    const uint32_t srow = smem_u32(base) + 128u * (uint32_t)r;
    const uint32_t lanes = (uint32_t)(32 * q) << 16;
    const uint32_t sw = 16u * (uint32_t)(r & 7);
    uint32_t slot = 0, bph = 0;                        // ring slot of the piece, its parity
    uint32_t s = (uint32_t)grp, eph = 1;               // stage of the group's next k-step, parity of "empty"
    int ks = grp;                                      // that k-step, counted in the current tile
    bool ok = true;
#pragma unroll 1
    for (int64_t t = pair; t < tiles && ok; t += pairs, ks -= nks) {
#pragma unroll 1
      for (int p = 0; p < npc && ok; ++p) {
        ok = __all_sync(kFull, mbar_wait(&sh->bits_full[slot], bph, failed));
        const uint32_t brow = brow0 + slot * (uint32_t)kBitBytes;
        const int kend = min(nks, kSteps * (p + 1));
#pragma unroll 1
        for (; ks < kend && ok; ks += kGroups) {
          const uint32_t src = brow + 32u * (uint32_t)(ks - kSteps * p);
          const uint4 lo = lds128(src), hi = lds128(src + 16);
          uint32_t x[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
          ok = __all_sync(kFull, mbar_wait(&sh->empty[s], eph, failed));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (awarp) {
            if (Kin - KF * ks < KF) {
              // pad bits, whatever the caller left in the rows' last word, count as +1
              const int valid = Kin - KF * ks;
#pragma unroll
              for (int c = 0; c < 8; ++c)
                x[c] &= valid >= 32 * c + 32 ? kFull : (valid <= 32 * c ? 0u : (1u << (valid - 32 * c)) - 1u);
            }
            tmem_store_row256(tmem + lanes + (uint32_t)kStageCol + 32u * s, x);
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          } else {
            const uint32_t row = (srow + s * (uint32_t)B_BYTES) | sw;   // chunk c at row ^ 16 c
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              uint32_t v[4];
              e2m1_words(x[c], v);
              sts128(row ^ (16u * c), v);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh->full[s]);
          s += kGroups;
          if (s >= kStages) {
            s -= kStages;
            eph ^= 1u;
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh->bits_empty[slot]);
        if (++slot == kPieces) {
          slot = 0;
          bph ^= 1u;
        }
      }
    }
  } else if (warp >= kLoad0 && warp < kEpi0) {
    // ---------------- loaders ----------------
    constexpr int kPer = 128 / kAlign;      // copies per row
    const int tid = threadIdx.x - 32 * kLoad0;
    const int c = tid % kPer, r0 = tid / kPer;
    constexpr int kStep = 32 * kLoadWarps / kPer;   // rows between a thread's copies
    uint32_t slot = 0, ph = 1;
    bool ok = true;
    const uint32_t dst0 = smem_u32(bits) + (uint32_t)(r0 * kBitRow + kAlign * c);
#pragma unroll 1
    for (int64_t t = pair; t < tiles && ok; t += pairs) {
      const int64_t m0 = (t / ntiles) * (2 * TM) + (int64_t)rank * TM;
      const int nb = (int)(t % ntiles) * TN + (int)rank * TB;
      // copies of this thread that are inside the operands' rows
      const int la = (int)max((int64_t)0, min((int64_t)(TM / kStep), (M - m0 - r0 + kStep - 1) / kStep));
      const int lw = max(0, min(TB / kStep, (N - nb - r0 + kStep - 1) / kStep));
      const uint64_t* arow = A + (m0 + r0) * nw + (kAlign / 8) * c;
      const uint64_t* wrow = W + (int64_t)(nb + r0) * nw + (kAlign / 8) * c;
#pragma unroll 1
      for (int p = 0; p < npc && ok; ++p) {
        ok = mbar_wait(&sh->bits_empty[slot], ph, failed);
        if (!ok) break;
        const uint32_t dst = dst0 + slot * (uint32_t)kBitBytes;
        const bool won = kPieceWords * p + (kAlign / 8) * c < nw;
        const uint64_t* pa = arow + kPieceWords * p;
        const uint64_t* pw = wrow + kPieceWords * p;
#pragma unroll 4
        for (int i = 0; i < TM / kStep; ++i, pa += kStep * nw) {
          const bool on = won && i < la;
          cp_async_or_zero<kAlign>(dst + (uint32_t)(i * kStep * kBitRow), on ? pa : A, on);
        }
#pragma unroll 4
        for (int i = 0; i < TB / kStep; ++i, pw += kStep * nw) {
          const bool on = won && i < lw;
          cp_async_or_zero<kAlign>(dst + (uint32_t)((TM + i * kStep) * kBitRow), on ? pw : W, on);
        }
        cp_async_arrive(&sh->bits_full[slot]);
        if (++slot == kPieces) {
          slot = 0;
          ph ^= 1u;
        }
      }
    }
    cp_async_wait_all();   // no copy outlives its thread
  } else if (warp >= kMmaWarp && warp < kLoad0) {
    bool ok = true;
    if (rank == 0 && warp == kMmaWarp) {
      // ---------------- MMA issuer of the pair ----------------
      const bool lead = elect_one();
      const uint32_t d = uniform(tmem);
      const uint64_t bd0 = smem_desc(uniform(smem_u32(base)));
      uint32_t s = 0, ph = 0, dph = 1;
#pragma unroll 1
      for (int64_t t = pair; t < tiles && ok; t += pairs) {
        ok = __all_sync(kFull, mbar_wait_cluster(&sh->drained, dph, failed));
        dph ^= 1u;
#pragma unroll 1
        for (int ks = 0; ks < nks && ok; ++ks) {
          ok = __all_sync(kFull, mbar_wait_cluster(&sh->full[s], ph, failed));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t bd = bd0 + (uint64_t)(s * (uint32_t)(B_BYTES >> 4));
          const uint32_t ta = d + (uint32_t)kStageCol + 32u * s;
          if (lead) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              mma_f4_pair(d, ta + 8 * e, bd + 2 * e, d + kSfCol, d + kSfCol + 16, (ks > 0 || e > 0) ? 1u : 0u);
            mma_commit_pair(&sh->empty[s]);
          }
          if (++s == kStages) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (ok && lead) mma_commit_pair(&sh->done);
        __syncwarp();
      }
    } else if (rank != 0 && lane == 0) {
      // relays of the odd CTA: its stage is full -> one arrival on the even CTA's
      const int64_t mine = (tiles - pair + pairs - 1) / pairs;   // tiles of this pair
      const uint64_t last = pair < tiles ? (uint64_t)mine * (uint64_t)nks : 0ull;
#pragma unroll 1
      for (uint64_t k = (uint64_t)(warp - kMmaWarp); k < last && ok; k += kRelays) {
        const uint32_t s = (uint32_t)(k % kStages);
        ok = mbar_wait(&sh->full[s], (uint32_t)(k / kStages) & 1u, failed);
        if (ok) mbar_arrive_rank0(&sh->full[s]);
      }
    }
  } else if (warp >= kEpi0) {
    // ---------------- epilogue ----------------
    const int sub = warp & 3, half = (warp - kEpi0) >> 2;   // lane quarter; neurons 128 half .. + 127
    const int r = 32 * sub + lane;
    const float npad = (float)(KF * nks - Kin);
    const bool vec = (nw_out % 2 == 0) && (reinterpret_cast<uintptr_t>(Aout) % 16 == 0);
    uint32_t tile = 0;
#pragma unroll 1
    for (int64_t t = pair; t < tiles; t += pairs, ++tile) {
      if (!__all_sync(kFull, mbar_wait(&sh->done, tile & 1u, failed))) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      uint32_t word[4];
      sign_words<4>(word, tmem + ((uint32_t)(32 * sub) << 16) + (uint32_t)(128 * half), 4, npad);
      // D is read: the pair's next tile may overwrite it
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_rank0(&sh->drained);
      const int64_t m = (t / ntiles) * (2 * TM) + (int64_t)rank * TM + r;
      const int n0 = (int)(t % ntiles) * TN + 128 * half;
      if (m < M) {
        uint32_t* row = reinterpret_cast<uint32_t*>(Aout + m * nw_out);
        const int w0 = n0 >> 5;
        if (vec && n0 + 128 <= N) {
          *reinterpret_cast<uint4*>(row + w0) = make_uint4(word[0], word[1], word[2], word[3]);
        } else {
#pragma unroll
          for (int cb = 0; cb < 4; ++cb) {
            // words wholly past N (inside the row's last 64-bit word) are written 0
            const int valid = N - n0 - 32 * cb;
            const uint32_t keep = valid >= 32 ? kFull : (valid <= 0 ? 0u : (1u << valid) - 1u);
            if (w0 + cb < 2 * nw_out) row[w0 + cb] = word[cb] & keep;
          }
        }
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  pair_sync();   // no CTA releases TMEM or leaves while its peer may still use the pair
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (threadIdx.x == 0 && *failed) atomicAdd(timeouts, 1u);
  if (warp == kMmaWarp)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

// Failure-path probe: the bounded mbarrier wait of the kernels above on a
// barrier whose phase completes only if `arrive` (one arrival before the wait).
__global__ void k_wait_probe(unsigned int* __restrict__ timeouts, int arrive,
                             unsigned long long limit) {
  __shared__ unsigned long long bar;
  __shared__ int failed;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (arrive) mbar_arrive(&bar);
    if (!mbar_wait(&bar, 0, &failed, limit)) atomicAdd(timeouts, 1u);
  }
}

}  // namespace

void launch_wait_probe(unsigned int* timeouts, int arrive, unsigned long long limit_cycles,
                       cudaStream_t st) {
  k_wait_probe<<<1, 32, 0, st>>>(timeouts, arrive, limit_cycles);
}

cudaError_t prepare_forward_eval_tc() {
  cudaError_t e = cudaFuncSetAttribute(k_forward_eval_tc<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kSmemBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_forward_eval_tc<8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kSmemBytes);
}

cudaError_t launch_forward_eval_tc(const uint64_t* A, int64_t M, int nw_in, const uint64_t* W, int N, int Kin,
                                   uint64_t* Aout, int nw_out, unsigned int* timeouts, cudaStream_t st, bool pdl) {
  const int ntiles = (N + TN - 1) / TN;
  const int64_t tiles = (M + 2 * TM - 1) / (2 * TM) * ntiles;
  const int64_t pairs = sm_count() / 2 < tiles ? sm_count() / 2 : tiles;
  const bool wide = row_align(A, nw_in) == 16 && row_align(W, nw_in) == 16;
  return launch_kernel(wide ? k_forward_eval_tc<16> : k_forward_eval_tc<8>, dim3((unsigned)(2 * pairs)),
                       dim3(THREADS), kSmemBytes, st, pdl, A, M, nw_in, W, N, Kin, Aout, nw_out, ntiles, tiles,
                       timeouts);
}

}  // namespace bk
