// kern_forward_tc.cu -- tensor-core forward contraction of the BMLP
// (Alg. 1 l.8-9) on sm_103a with tcgen05, for mini-batches and small batches.
//
//   z^mu_k = sum_i a^mu_i w_ik,  a, w in {-1, +1}
//
// is computed exactly as an e2m1 x e2m1 -> fp32 matrix product with unit block
// scales (tcgen05.mma kind::mxf4; tc_common.cuh has the element format).
// Elements past K_in are +1 in both operands (their bits are 0 in the weights,
// and cleared in the activations), so the epilogue subtracts their number.
//
// Tiling.  The weights are the M operand: a tile is 128 neurons (tensor-memory
// lanes) x up to kMaxPat patterns (accumulator columns), so a mini-batch of
// 100 costs 112 columns and not 128 rows, the weights, which are the larger
// operand, are expanded into tensor memory (which shared-memory bandwidth does
// not limit), and a warp's 32 lanes are 32 consecutive neurons of one
// pattern: one ballot per pattern packs the sign bits and the pre-activations
// are stored as contiguous runs.  The K range is split over a cluster of S
// CTAs where the tiles alone leave SMs idle.
//
// A CTA is 288 threads.  K goes in pieces of 1,024 elements (a 128-byte line of
// every packed row), four k-steps of 256:
//   - the 256 producer threads copy a piece of the tile's 128 weight rows and of
//     its pattern rows into shared memory with asynchronous copies of whole
//     lines;
//   - two k-steps at a time (their latencies overlap), weight warp q (of four) expands neuron rows 32 q .. + 31, a
//     lane per row, into 32 tensor-memory columns, and activation warp q expands
//     pattern rows 32 q .. + 31 into a shared-memory stage, rows of 128 bytes
//     with the 128B swizzle (16-byte chunk c of row r at chunk c ^ (r % 8));
//   - one MMA thread waits on a stage's "full" mbarrier (one arrival per
//     producer warp), issues the four MMAs (K = 64) and commits to "empty";
//   - epilogue, S = 1: each producer warp reads 16 columns at a time and writes
//     z (int16) and the sign bits.  S > 1: CTA r finalises the blocks of 16
//     patterns b with b % S = r; the others' partials of a block (at most
//     16,384 in magnitude for S >= 2, so they fit 16 bits) go into the owner's
//     shared memory with remote stores, one cluster barrier, and the owner adds
//     them to its own.
// The loops are kept rolled: a CTA runs through its code once or twice, and
// with the k-steps of a piece unrolled the warps waited longer for instructions
// (2.5 clocks per instruction issued) than for anything but memory.
// Shared memory (103 KB) and tensor memory (256 columns) are sized for two CTAs
// per SM: one expands while the other's MMAs run, and the CTAs of the next layer,
// launched as programmatic dependents, set up beside the running ones.  Registers
// are held to 72, so that CTAs of the event draws and of the selection fit
// beside two of these (a step of 8192-8192x4 154 us at 72, 156 at 96).
//
// What bounds it: latency, and L2 bandwidth for the widest layers.  At 100
// patterns, launches back to back as programmatic dependents: 8192 -> 8192
// 11.0 us (14.7 MB through L2 1.5 us, MMAs 1.7 us; the e4m3 kernel before it,
// 128 x 256 tiles with the activations in tensor memory, 18-19 us), 4096 -> 4096
// 6.0 us (10), 1024 -> 1024 3.6 us (6).  Of the last, 0.5 us are the set-up before
// the wait, 0.4 the copies, 1.8 the four k-steps (a warp alone on its scheduler
// takes 3 clocks an instruction) and 0.6 the epilogue.
//
// Every mbarrier wait is bounded; the first expiry sets a shared flag that
// stops every other wait, the kernel counts the failure (host: BMLP_ETIMEOUT),
// still passes the barriers, releases its tensor memory and returns.
#include "tc_common.cuh"

namespace bk {

int sm_count() {
  static const int n = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1)
      v = 152;
    return v;
  }();
  return n;
}

namespace {

using namespace tc;

constexpr int TN = 128;             // neurons per tile (MMA M)
constexpr int kMaxPat = 112;        // patterns per tile at most (MMA N, a multiple of 16)
constexpr int kSteps = 4;           // k-steps (of KF = 256 elements) per piece
constexpr int kPieceWords = 16;     // 64-bit words per row and piece
constexpr int kStages = 3;          // stages of one k-step: activations in shared memory, weights in TMEM
constexpr int kProdWarps = 8;       // four for the weights, four for the activations
constexpr int kProducers = 32 * kProdWarps;
constexpr int THREADS = kProducers + 32;
constexpr int B_BYTES = kMaxPat * 128;            // one activation stage
constexpr int TMEM_COLS = 256;
constexpr int kSfCol = kMaxPat;                   // 16 columns of unit scales
constexpr int kStageCol = kSfCol + 16;            // weight stages of 32 columns
static_assert(kStageCol + 32 * kStages <= TMEM_COLS, "TMEM budget");
static_assert(B_BYTES % 1024 == 0, "swizzle atoms");
constexpr int kMaxSplit = 4;
constexpr int kBlocks = kMaxPat / 16;             // blocks of 16 patterns
// partial buffers: from S - 1 peers, ceil(kBlocks / S) blocks of 8 column
// pairs x 128 lanes x 4 bytes (S = 2: 4 blocks, S = 3: 2 x 3, S = 4: 3 x 2)
constexpr int kBlockWords = 8 * TN;
constexpr int kPartBytes = 6 * kBlockWords * 4;
// bits of a piece: 128 weight rows, then kMaxPat pattern rows, 144 bytes apart
// (eight lanes reading 16 bytes of eight rows each: no bank conflict)
constexpr int kBitRow = 144;
constexpr int kBitBytes = (TN + kMaxPat) * kBitRow;

struct __align__(8) TcShared {
  unsigned long long full[kStages];   // the producers filled stage s
  unsigned long long empty[kStages];  // the MMAs that read stage s completed
  unsigned long long done;            // all MMAs completed
  uint32_t tmem_base;
  int failed;
};

constexpr size_t kSmemBytes = 1024 /*alignment slack*/ + kStages * B_BYTES + kPartBytes + kBitBytes +
                              sizeof(TcShared);

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t peer_addr(uint32_t local_addr, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local_addr), "r"(rank));
  return a;
}

// 16 accumulator columns of this warp's 32 lanes, as integers (exact).
__device__ __forceinline__ void load_cols16(int (&z)[16], uint32_t taddr) {
  uint32_t v[16];
  tmem_load16(v, taddr);
  tmem_wait_ld(v);
#pragma unroll
  for (int j = 0; j < 16; ++j) z[j] = __float2int_rn(__uint_as_float(v[j]));
}

// A piece (words w0 .. w0 + 15) of nrows rows of nw words -> the bit rows from
// `dst` on; rows >= live and words >= nw become 0.
template <int kAlign>
__device__ __forceinline__ void copy_piece(uint32_t dst, const uint64_t* rows, int nrows, int live, int w0,
                                           int nw) {
  constexpr int kPer = 128 / kAlign;            // copies per row
  constexpr int kW = kAlign / 8;                // words per copy
  const int c = threadIdx.x % kPer;
  const int w = w0 + kW * c;
#pragma unroll 2
  for (int r = threadIdx.x / kPer; r < nrows; r += kProducers / kPer) {
    const bool on = r < live && w < nw;
    cp_async_or_zero<kAlign>(dst + (uint32_t)(r * kBitRow + kAlign * c),
                             on ? rows + (int64_t)r * nw + w : rows, on);
  }
}

__device__ __forceinline__ void producers_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kProducers) : "memory");
}

struct Place {
  uint8_t* stages;
  uint32_t* part;
  uint8_t* bits;
  TcShared* sh;
};
__device__ __forceinline__ Place place(uint8_t* raw) {
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* bits = base + kStages * B_BYTES + kPartBytes;
  return Place{base, reinterpret_cast<uint32_t*>(base + kStages * B_BYTES), bits,
               reinterpret_cast<TcShared*>(bits + kBitBytes)};
}

struct TileIn {
  const uint64_t* A;   // packed rows of the patterns, row 0
  const uint64_t* W;
  int nw, N, Kin;
  int16_t* Z;          // [pattern][N], or null
  uint64_t* Aout;      // [pattern][nw_out]
  int nw_out;
  int32_t* labels;     // kLabels: the row's argmax of W A (lowest index on ties)
};

// Barriers and tensor memory, set up before the inputs are waited for.
__device__ __forceinline__ void tile_setup(TcShared* sh, int warp, int lane) {
  if (warp == kProdWarps) {
    if (lane == 0) {
      for (int s = 0; s < kStages; ++s) {
        mbar_init(&sh->full[s], kProdWarps);   // one arrival per producer warp
        mbar_init(&sh->empty[s], 1);
      }
      mbar_init(&sh->done, 1);
      sh->failed = 0;
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(&sh->tmem_base)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// One tile.  ready(): waits for the inputs and returns the rows of pattern 0
// and the number of patterns; w_early: the weights may be read before that.
// kLabels: W's rows are the classes (one tile, S = 1) and the output is the
// argmax over them instead of z and the signs.
template <int kAlign, bool kLabels = false, typename Ready>
__device__ __forceinline__ void run_tile(TileIn T, const Place& pl, int pat, bool w_early, Ready ready,
                                         unsigned int* timeouts) {
  TcShared* sh = pl.sh;
  uint8_t* stages = pl.stages;
  uint32_t* part = pl.part;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* failed = &sh->failed;
  const uint32_t rank = cluster_rank(), S = cluster_size();
  const int n0 = (int)(blockIdx.x / S) * TN;
  const int npc = (T.nw + kPieceWords - 1) / kPieceWords;
  const int pc0 = (int)((npc * rank) / S);
  int np = (int)((npc * (rank + 1)) / S) - pc0;   // pieces of this CTA
  const bool producer = warp < kProdWarps, wwarp = warp < kProdWarps / 2;
  const int q = warp & 3;
  const uint32_t bits0 = smem_u32(pl.bits);
  auto copy_w = [&](int i) {
    copy_piece<kAlign>(bits0, T.W + (int64_t)n0 * T.nw, TN, T.N - n0, kPieceWords * (pc0 + i), T.nw);
  };
  if (producer && w_early) copy_w(0);
  tile_setup(sh, warp, lane);
  const uint32_t tmem = sh->tmem_base;
  int64_t M;
  ready(T.A, M);
  const int64_t m0 = (int64_t)blockIdx.y * pat;
  const int mt = (int)max((int64_t)0, min((int64_t)pat, M - m0));
  if (mt == 0) np = 0;               // a short last mini-batch leaves this tile empty
  const int nblk = (mt + 15) >> 4;   // blocks of 16 patterns
  const uint32_t lanes = (uint32_t)(32 * q) << 16;
  const int nks = (T.Kin + KF - 1) / KF;
  const int ks0 = kSteps * pc0, ks1 = min(nks, kSteps * (pc0 + np));   // k-steps of this CTA
  if (S > 1) cluster_arrive();   // this CTA runs: its shared memory may be written by its peers

  if (producer) {
    const uint64_t* arows = T.A + m0 * (int64_t)T.nw;
    auto copy_a = [&](int i) {
      copy_piece<kAlign>(bits0 + TN * kBitRow, arows, mt, mt, kPieceWords * (pc0 + i), T.nw);
    };
    if (np > 0) {
      copy_a(0);
      if (!w_early) copy_w(0);
    }
    if (wwarp)
      // unit scales (ordered before the first MMA by this warp's first arrival)
      asm volatile(
          "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, "
          "%1, %1, %1, %1};" ::"r"(tmem + lanes + (uint32_t)kSfCol), "r"(kUnitScales) : "memory");
    const int r = 32 * q + lane;                 // this lane's row of its operand
    const bool live = wwarp || r < mt;
    const uint32_t brow = bits0 + (uint32_t)((wwarp ? r : (live ? TN + r : 0)) * kBitRow);
    const uint32_t srow = smem_u32(stages) + 128u * (uint32_t)r;
    bool ok = true;                              // (a failed wait leaves the loop's barriers matched)
#pragma unroll 1
    for (int ks = ks0; ks < ks1; ks += 2) {
      const int k = ks - ks0;
      if (k % kSteps == 0) {
        if (k > 0) {
          producers_sync();                      // every warp has read the last piece
          copy_a(k / kSteps);
          copy_w(k / kSteps);
        }
        cp_async_wait_all();
        producers_sync();
      }
      const int s[2] = {k % kStages, (k + 1) % kStages};
      const bool two = ks + 1 < ks1;
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (ok && k + i >= kStages && (i == 0 || two))
          ok = __all_sync(kFull, mbar_wait(&sh->empty[s[i]], (uint32_t)(((k + i) / kStages - 1) & 1), failed));
      if (!ok) continue;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t src = brow + 32u * (uint32_t)(ks % kSteps);
      uint32_t x[2][8];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint4 lo = lds128(src + 32 * i), hi = lds128(src + 32 * i + 16);
        x[i][0] = lo.x; x[i][1] = lo.y; x[i][2] = lo.z; x[i][3] = lo.w;
        x[i][4] = hi.x; x[i][5] = hi.y; x[i][6] = hi.z; x[i][7] = hi.w;
      }
      if (wwarp) {
        // rows past N hold whatever: their outputs are dropped (e2m1 has no NaN)
#pragma unroll
        for (int i = 0; i < 2; ++i)
          if (i == 0 || two) tmem_store_row256(tmem + lanes + (uint32_t)(kStageCol + 32 * s[i]), x[i]);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      } else if (live) {
        const int valid = T.Kin - KF * ks;       // inputs from here on
        if (valid < 2 * KF) {
          // pad bits, whatever the caller left in the rows' last word, count as +1
#pragma unroll
          for (int c = 0; c < 16; ++c)
            x[c >> 3][c & 7] &= valid >= 32 * c + 32 ? kFull : (valid <= 32 * c ? 0u : (1u << (valid - 32 * c)) - 1u);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const uint32_t row = (srow + (uint32_t)(s[i] * B_BYTES)) | (16u * (uint32_t)(r & 7));   // chunk c at row ^ 16 c
          if (i == 0 || two) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              uint32_t v[4];
              e2m1_words(x[i][c], v);
              sts128(row ^ (16u * c), v);
            }
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&sh->full[s[0]]);
        if (two) mbar_arrive(&sh->full[s[1]]);
      }
    }
    // no copy outlives its thread: the early weights of a tile without patterns
    // are read by nobody
    cp_async_wait_all();
  } else {
    // ---------------- MMA issuer ----------------
    const bool lead = elect_one();
    const uint32_t idesc = uniform(idesc_f4(TN, 16 * nblk));
    const uint32_t d = uniform(tmem);
    const uint64_t bd0 = smem_desc(uniform(smem_u32(stages)));
    uint32_t s = 0, par = 0;
    bool ok = true;
#pragma unroll 1
    for (int ks = ks0; ks < ks1 && ok; ++ks) {
      ok = __all_sync(kFull, mbar_wait(&sh->full[s], par, failed));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint64_t bd = bd0 + (uint64_t)(s * (uint32_t)(B_BYTES >> 4));
      const uint32_t ta = d + (uint32_t)kStageCol + 32u * s;
      if (lead) {
#pragma unroll
        for (int e = 0; e < 4; ++e)   // K = 64 per MMA: 8 TMEM columns, 32 bytes of the stage rows
          mma_f4_ts(d, ta + 8 * e, bd + 2 * e, idesc, d + kSfCol, d + kSfCol + 8, (ks > ks0 || e > 0) ? 1u : 0u);
        mma_commit(&sh->empty[s]);
      }
      if (++s == kStages) {
        s = 0;
        par ^= 1u;
      }
    }
    if (np > 0 && ok && lead) mma_commit(&sh->done);
  }
  __syncwarp();

  // ---------------- epilogue ----------------
  const int cq = warp >> 2;   // this warp's share of the blocks
  bool go = false;
  if (producer) {
    go = np > 0 && !*failed && mbar_wait(&sh->done, 0, failed);
    go = __all_sync(kFull, go);   // tcgen05.ld is warp-collective
    if (go) asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
  const int slane = 32 * q + lane;   // lane of the tile
  const uint32_t per = ((uint32_t)kBlocks + S - 1) / S;
  if (S > 1) {
    cluster_wait();   // every peer runs
    if (producer) {
      const uint32_t base = smem_u32(part);
#pragma unroll 1
      for (int b = cq; b < nblk; b += kProdWarps / 4) {
        const uint32_t own = (uint32_t)b % S;
        if (own == rank) continue;
        int z[16];
        if (go) load_cols16(z, tmem + lanes + (uint32_t)(16 * b));
        else {
#pragma unroll
          for (int j = 0; j < 16; ++j) z[j] = 0;
        }
        // my slot in the owner's buffer, the block's place in the slot
        const uint32_t slot = rank < own ? rank : rank - 1;
        const uint32_t dst = peer_addr(base + 4u * (kBlockWords * (slot * per + (uint32_t)b / S) + slane), own);
#pragma unroll
        for (int p = 0; p < 8; ++p) {
          const uint32_t v = ((uint32_t)z[2 * p] & 0xFFFFu) | ((uint32_t)z[2 * p + 1] << 16);
          asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(dst + 4u * TN * (uint32_t)p), "r"(v) : "memory");
        }
      }
    }
    cluster_arrive();
    cluster_wait();
  }
  if (go && !*failed) {
    const int n = n0 + slane;
    const int word = (n0 >> 5) + q;   // 32-bit word of the packed rows
    const int npad = KF * nks - T.Kin;
    // blocks of this CTA, dealt to the producer warps of each lane quarter
#pragma unroll 1
    for (int b = (int)(rank + S * (uint32_t)cq); b < nblk; b += (int)(kProdWarps / 4 * S)) {
      int z[16];
      load_cols16(z, tmem + lanes + (uint32_t)(16 * b));
#pragma unroll
      for (int j = 0; j < 16; ++j) z[j] -= npad;
#pragma unroll 1
      for (uint32_t p = 0; p + 1 < S; ++p) {
        const uint32_t* src = part + kBlockWords * (p * per + (uint32_t)b / S) + slane;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t v = src[TN * j];
          z[2 * j] += (int)(int16_t)(v & 0xFFFFu);
          z[2 * j + 1] += (int)(int16_t)(v >> 16);
        }
      }
      const int64_t mb = m0 + 16 * b;
      const int rows = min(16, mt - 16 * b);
      uint32_t mine = 0;
      if constexpr (kLabels) {
        // largest score, then lowest class, of this warp's 32 classes: scores
        // are within +-32767, a class never needs more than 7 bits
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const uint32_t k = n < T.N ? ((uint32_t)(z[j] + 32768) << 7) | (uint32_t)(TN - 1 - n) : 0u;
          const uint32_t best = __reduce_max_sync(kFull, k);
          if (lane == j) mine = best;
        }
        if (lane < 16) part[TN * q + 16 * b + lane] = mine;
        continue;
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const uint32_t bits = __ballot_sync(kFull, n < T.N && z[j] >= 0);
        if (lane == j) mine = bits;
      }
      // words wholly past N (inside the row's last 64-bit word) are written 0
      if (lane < rows && word < 2 * T.nw_out)
        reinterpret_cast<uint32_t*>(T.Aout + (mb + lane) * T.nw_out)[word] = mine;
      if (T.Z != nullptr && n < T.N) {
        int16_t* zp = T.Z + mb * T.N + n;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (j < rows) *zp = (int16_t)z[j];
          zp += T.N;
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if constexpr (kLabels) {
    if ((int)threadIdx.x < mt && !*failed) {
      uint32_t best = 0u;
#pragma unroll
      for (int e = 0; e < 4; ++e) best = max(best, part[TN * e + threadIdx.x]);
      T.labels[m0 + threadIdx.x] = TN - 1 - (int)(best & 127u);
    }
  }
  if (threadIdx.x == 0 && *failed) atomicAdd(timeouts, 1u);
  if (warp == kProdWarps)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

// One layer of the current training mini-batch.  Grid (S x neuron tiles,
// pattern tiles of pat), clusters of S.
__global__ void __launch_bounds__(THREADS, 3) k_train_forward_tc(const StepParams* __restrict__ P, int l,
                                                                 int pat, const OneBatch one) {
  extern __shared__ uint8_t smem_raw[];
  const DevLayer& Ly = P->layer[l - 1];
  const uint64_t* x = l > 1 ? P->layer[l - 2].A : (one.x ? one.x : P->x);
  const TileIn T{x, Ly.W, Ly.nw_in, Ly.Kout, Ly.Kin, Ly.Z, Ly.A, Ly.nw_out, nullptr};
  const int64_t ncall = one.x ? one.n : P->n;
  const int bs = P->bs;
  // Layers >= 2: the weights (the previous step's update), the batch index
  // and every pointer were written two or more launches back, so the weights
  // are read before waiting for the previous layer, whose activations are read
  // after.  Layer 1 waits first: its weights and batch index come from the
  // update launched just before it.
  auto ready = [&](const uint64_t*& A, int64_t& M) {
    pdl_wait();
    pdl_trigger();
    const int64_t start = one.x ? 0 : (int64_t)batch_index(P) * bs;
    M = min((int64_t)bs, ncall - start);
    if (l == 1) {
      A = x + start * T.nw;
      if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) begin_step(P);
    }
  };
  if (row_align(T.A, T.nw) == 16 && row_align(T.W, T.nw) == 16)
    run_tile<16>(T, place(smem_raw), pat, l > 1, ready, &P->ctrl->timeouts);
  else
    run_tile<8>(T, place(smem_raw), pat, l > 1, ready, &P->ctrl->timeouts);
}

// One layer of forward-only evaluation on a small batch.  w_early: no kernel that
// may still run beside this one writes the weights.
template <int kAlign>
__global__ void __launch_bounds__(THREADS, 2)
    k_forward_tile(const uint64_t* __restrict__ A, int64_t M, int nw, const uint64_t* __restrict__ W, int N,
                   int Kin, uint64_t* __restrict__ Aout, int nw_out, unsigned int* __restrict__ timeouts,
                   int pat, bool w_early) {
  extern __shared__ uint8_t smem_raw[];
  const TileIn T{A, W, nw, N, Kin, nullptr, Aout, nw_out, nullptr};
  auto ready = [&](const uint64_t*&, int64_t& m) {
    pdl_wait();
    pdl_trigger();
    m = M;
  };
  run_tile<kAlign>(T, place(smem_raw), pat, w_early, ready, timeouts);
}

// Evaluation output on at most 128 classes: labels = argmax_j (A PT^T)_j, lowest j
// on ties (PT: the packed classifier columns, c rows of nw words; K = its bits).
template <int kAlign>
__global__ void __launch_bounds__(THREADS, 2)
    k_predict_tile(const uint64_t* __restrict__ A, int64_t M, int nw, const uint64_t* __restrict__ PT, int c,
                   int K, int32_t* __restrict__ labels, unsigned int* __restrict__ timeouts, int pat) {
  extern __shared__ uint8_t smem_raw[];
  const TileIn T{A, PT, nw, c, K, nullptr, nullptr, 0, labels};
  auto ready = [&](const uint64_t*&, int64_t& m) {
    pdl_wait();
    pdl_trigger();
    m = M;
  };
  run_tile<kAlign, true>(T, place(smem_raw), pat, true, ready, timeouts);
}

// Patterns per tile, pattern tiles and K split of M patterns on an N x Kin
// layer.  The K range is split over up to kMaxSplit CTAs while every CTA keeps
// a piece, all CTAs fit two per SM and the tiles alone fill at most half of the
// SMs (3072-2048x3 at 512 patterns, 80 tiles: 717 us a call unsplit, 733 split);
// then the patterns are dealt to more tiles (of equal size, a multiple of 16)
// while all fit one per SM.  Measured at 100 patterns, back to back:
// 8192 -> 8192 split 1 / 2 / 4 21.8 / 14.2 / 11.4 us; 4096 -> 4096 split 2 / 4
// 7.7 / 6.1 us; 1024 -> 1024 (no split) pattern tiles of 64 / 32 / 16
// 4.3 / 3.9 / 3.8 us.
struct Shape {
  int pat, mtiles, ntiles, split;
};
Shape shape_of(int64_t M, int N, int Kin, int sms) {
  Shape s;
  s.ntiles = (N + TN - 1) / TN;
  int64_t mt = (M + kMaxPat - 1) / kMaxPat;
  const int npc = (Kin + KF * kSteps - 1) / (KF * kSteps);
  s.split = 1;
  for (int c = 2; c <= kMaxSplit; ++c)
    if (npc >= c && s.ntiles * mt * c <= 2 * sms && s.ntiles * mt * 2 <= sms) s.split = c;
  while (mt * s.ntiles * s.split * 2 <= sms && M > 16 * mt) mt *= 2;
  s.pat = (int)(((M + mt - 1) / mt + 15) / 16 * 16);
  s.mtiles = (int)((M + s.pat - 1) / s.pat);
  return s;
}

template <typename... KArgs, typename... Args>
cudaError_t launch_tiles(void (*k)(KArgs...), const Shape& s, cudaStream_t st, bool pdl, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(s.ntiles * s.split), (unsigned)s.mtiles);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)s.split;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

template <typename K>
cudaError_t allow_smem(K k) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
}

}  // namespace

cudaError_t prepare_train_forward_tc() {
  cudaError_t e = allow_smem(k_train_forward_tc);
  if (e == cudaSuccess) e = allow_smem(k_forward_tile<8>);
  if (e == cudaSuccess) e = allow_smem(k_forward_tile<16>);
  if (e == cudaSuccess) e = allow_smem(k_predict_tile<8>);
  if (e == cudaSuccess) e = allow_smem(k_predict_tile<16>);
  return e;
}

cudaError_t launch_train_forward_tc(int bs, int Kout, int Kin, cudaStream_t st, bool pdl,
                                    const StepParams* P, int l, const OneBatch& one) {
  const Shape s = shape_of(bs, Kout, Kin, sm_count());
  return launch_tiles(k_train_forward_tc, s, st, pdl, P, l, s.pat, one);
}

cudaError_t launch_forward_tile(const uint64_t* A, int64_t M, int nw_in, const uint64_t* W, int N, int Kin,
                                uint64_t* Aout, int nw_out, unsigned int* timeouts, cudaStream_t st,
                                bool pdl, bool w_early) {
  const Shape s = shape_of(M, N, Kin, sm_count());
  const bool wide = row_align(A, nw_in) == 16 && row_align(W, nw_in) == 16;
  return launch_tiles(wide ? k_forward_tile<16> : k_forward_tile<8>, s, st, pdl, A, M, nw_in, W, N, Kin, Aout,
                      nw_out, timeouts, s.pat, w_early);
}

bool forward_tiles_win(int64_t M, int N, int Kin) {
  if (M <= kMaxPat) return true;
  const int64_t tiles = (M + kMaxPat - 1) / kMaxPat * ((N + TN - 1) / TN);
  const int64_t npc = (Kin + KF * kSteps - 1) / (KF * kSteps);
  return tiles <= sm_count() && 5 * tiles * npc <= 8 * sm_count();
}

cudaError_t launch_predict_tile(const uint64_t* A, int64_t M, int nw, const uint64_t* PT, int c, int K,
                                int32_t* labels, unsigned int* timeouts, cudaStream_t st, bool pdl) {
  Shape s = shape_of(M, TN, TN, sm_count());   // one tile of classes, never split
  const bool wide = row_align(A, nw) == 16 && row_align(PT, nw) == 16;
  return launch_tiles(wide ? k_predict_tile<16> : k_predict_tile<8>, s, st, pdl, A, M, nw, PT, c, K, labels,
                      timeouts, s.pat);
}

}  // namespace bk
