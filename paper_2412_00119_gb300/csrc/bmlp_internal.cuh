// bmlp_internal.cuh -- device-side data layout and shared device helpers of the
// BMLP library (fully binary training rule of arXiv 2412.00119, Alg. 1-3).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/bmlp.h"

namespace bk {

// ---------------------------------------------------------------------------
// HBM layout of one layer l (K_in = K_{l-1}, K_out = K_l):
//   H    uint32 [K_out][ldh]     hidden weights, neuron-major, bit-sliced: a weight h
//                                 (odd, |h| <= h_max) is stored as its lattice index
//                                 u = (h + h_max)/2 in [0, h_max], a CP or R event
//                                 moves u by +-1 with clamping, and h > 0 iff
//                                 u >= (h_max + 1)/2.  Inputs are grouped by 32:
//                                 group g of row k (inputs 32 g .. 32 g + 31) is
//                                 nplanes words, word p holding bit p of u of the 32
//                                 weights (bit j <-> input 32 g + j); nbits planes are
//                                 used (the bits of h_max), nplanes = nbits rounded
//                                 up to a power of two (unused planes 0); ldh =
//                                 ngrp * nplanes rounded up to a multiple of 4 words
//                                 (16-byte rows).  Inputs i >= K_in hold u = 0 and
//                                 are never stepped
//   W    uint64 [K_out][nw_in]    packed sign(H), bit (i%64) of word i/64 = (h_ik > 0)
//   PT   uint64 [c][nw_out]       packed P_l^T, bit (k%64) of word k/64 = (rho_kj > 0)
//   rho  int8  [K_out][c]         P_l itself, for the stability rho_{k,y}
//   rhoT int8  [c][K_out]         the same, class-major
//   Z    int16 [bs][K_out]        pre-activations of the current mini-batch
//   A    uint64 [bs][nw_out]      packed activations a_l of the current mini-batch
//   mark uint8 [bs]               1 iff the pattern is in M_l
//   sel  int16 [G][bs]            selected neuron per (group, pattern), -1 = none
// ---------------------------------------------------------------------------
struct DevLayer {
  uint32_t* H;
  uint64_t* W;
  uint64_t* PT;
  int8_t* rho;
  int8_t* rhoT;       // [c][K_out]: rho transposed (class-major), for the selection
  int16_t* Z;
  uint64_t* A;
  uint8_t* mark;
  uint16_t* sel;      // [G][bs] selected neuron per group and pattern (group-major), bit 15
                      // set where its rho_{k,y} is -1; kNoSel: none
  int16_t* member;    // [K_out] group order (neuron at position j), or null: contiguous groups
  int16_t* group_of;  // [K_out] group of neuron k (with member)
  int32_t Kin, Kout, nw_in, nw_out, ldh, gamma, G;
  int32_t ngrp;          // groups of 32 inputs per neuron row (ceil(K_in / 32))
  int32_t ev_cta_base;   // first CTA of this layer in the event-draw grid
  int32_t row_base;      // first row of this layer in the numbering of the large models' update
  int32_t nblk;          // blocks of 64 inputs per neuron row (ceil(K_in / 64))
  uint64_t* EV;          // [K_out][ev_stride] reinforcement events of the current step (large
                         // models), bit i % 64 of word i / 64 = input i reinforced
  int32_t ev_stride;     // words per EV row: nblk rounded up to even (16-byte rows)
};

// Statistics of the update kernel, accumulated until read with reset: neuron
// rows visited (layers with M_l non-empty), rows streamed (at least one CP
// tuple) and algorithmic bytes (H read + write and W write of the streamed rows,
// the planes of a group read + written per group with an event of a row without
// tuple).  Spread over slots, so that CTAs do not queue for one address.
struct UpdStat {
  unsigned long long rows, streamed, bytes;
};
constexpr int kStatSlots = 64;

// Device-resident step control, so that one captured graph replays step after
// step without host involvement.  The first layer's forward pass copies s and t
// to s_cur and t_cur and clears the marks; the update kernel, which reads only
// the copies, advances s and t when it ends.
struct Ctrl {
  unsigned long long t;         // global mini-batch counter since creation
  unsigned long long err;       // last-layer 01-loss count since the last epoch end
  unsigned long long bad_labels;// labels outside 0..c-1 seen by the kernels
  uint32_t s_cur;               // the mini-batch in progress
  unsigned long long t_cur;
  uint32_t timeouts;            // bounded device waits that expired (BMLP_ETIMEOUT)
  uint32_t upd_next;            // next row for the warps of the large models' update
  uint32_t any_mark[BMLP_MAX_LAYERS];
  UpdStat stat[kStatSlots];
  unsigned long long layer_err[BMLP_MAX_LAYERS];  // local 01-loss count of each layer
};

// Thresholds of the reinforcement sampler of one layer (Alg. 3 l.5-12): the
// events of a neuron row are drawn per block of 64 inputs (the last block
// holds K_in mod 64 when that is not 0).  For a block of n inputs:
//   any      = thr(1 - (1-q)^n)        at least one event iff the block draw < any
//   first[j] = thr((1 - (1-q)^(j+1)) / (1 - (1-q)^n))   first event: least j with V < first[j]
//   gap[g]   = thr(1 - (1-q)^(g+1))    next event p + 1 + g: least g <= n-2-p with V < gap[g]
// thr(x) = ceil(x 2^32) (0 for x <= 0, 2^32 for x >= 1); (1-q)^m a left-to-right
// IEEE product.  Index [0]: n = 64, [1]: the last, shorter block.
struct RTables {
  unsigned long long any[2];
  unsigned long long first[2][64];
  unsigned long long gap[64];       // entries g < 63 (independent of n)
};

struct StepParams {
  DevLayer layer[BMLP_MAX_LAYERS];
  const uint64_t* x;            // packed inputs of the current train call
  const int32_t* y;             // labels of the current train call
  int64_t n;                    // patterns in the current train call
  uint32_t s;                   // mini-batch index within the current train call (the update kernel
                                // advances it; one copy to the device sets it with x, y and n)
  const RTables* rt;            // [L] reinforcement sampler thresholds
  int32_t nblk_max;             // max over layers of ceil(K_in / 64)
  Ctrl* ctrl;
  int32_t L, c, bs, h_max, r_num, r_den, nw0;
  int32_t rows_total;           // sum of K_l over the layers
  int32_t nbits, nplanes;       // bit-planes of H used / stored per group (see H above)
  uint32_t key0, key1;          // Philox key = (seed mod 2^32, seed div 2^32)
};


constexpr uint16_t kNoSel = 0xFFFFu;   // K_l <= 32767, so no neuron has index 0x7FFF


// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11), device version.
// Counter layout of the library's random streams (purpose tag in c2):
//   initial h_ik of layer l : (i/4, k, 1*2^16 + l, 0)   word i%4, +1 iff bit 31
//   rho_kj of P_l           : (j/4, k, 2*2^16 + l, 0)   word j%4, +1 iff bit 31
//   block draw U of block b (inputs 64b .. 64b+63) of neuron k at step t:
//                             (b/4, k, 3*2^16 + l, t)   word b%4
//   event draws V_0, V_1, .. of that block: words 0..3 of (b, k, (4+r)*2^16 + l, t),
//                             r = 0, 1, ..
//   group-order key u_k of neuron k: (k/4, 0, 32*2^16 + l, t')   word k%4
//   expansion weight e_ki   : (i/4, k, 33*2^16, 0)      word i%4, +1 iff bit 31
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 ctr, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)0xD2511F53u * ctr.x;  // one wide multiply each
    const uint64_t p1 = (uint64_t)0xCD9E8D57u * ctr.z;
    ctr = make_uint4((uint32_t)(p1 >> 32) ^ ctr.y ^ (k0 + (uint32_t)r * 0x9E3779B9u), (uint32_t)p1,
                     (uint32_t)(p0 >> 32) ^ ctr.w ^ (k1 + (uint32_t)r * 0xBB67AE85u), (uint32_t)p0);
  }
  return ctr;
}

// Programmatic dependent launch: a kernel launched with the
// programmatic-stream-serialization attribute may start while the kernel
// before it in the stream is still running.  pdl_wait() returns once that
// kernel has completed and its memory is visible (at once without the
// attribute); pdl_trigger() lets the next kernel start launching.  Every
// kernel that triggers does so only after its own wait, so when a kernel
// starts, every kernel two or more launches before it has completed.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The inputs of a call of one mini-batch, passed to its kernels by value (no copy
// to StepParams and no graph); x null: they are in StepParams.
struct OneBatch {
  const uint64_t* x;
  const int32_t* y;
  int64_t n;
};

// The mini-batch index (past the L1 cache: kernels that overlap this one write it).
__device__ __forceinline__ uint32_t batch_index(const StepParams* P) { return __ldcg(&P->s); }

// One thread of the first layer's forward pass, after its wait.
__device__ __forceinline__ void begin_step(const StepParams* P) {
  Ctrl* c = P->ctrl;
  c->s_cur = batch_index(P);
  c->t_cur = c->t;
  c->upd_next = 0u;
  for (int i = 0; i < P->L; ++i) c->any_mark[i] = 0u;
}

// Launch with or without the programmatic-stream-serialization attribute.
template <typename... KArgs, typename... Args>
cudaError_t launch_kernel(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                          bool pdl, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------
// Forward of layer l (1-based) for the current training mini-batch.
__global__ void k_train_forward(const StepParams* P, int l);
// Local classifier, 01-loss, margin, marks, and the group selection, all layers.
// ClsArgs: what the kernel needs of the model, passed by value.
struct ClsLayer {
  const uint64_t* A;
  const uint64_t* PT;
  const int16_t* Z;
  const int8_t* rhoT;
  uint16_t* sel;
  uint8_t* mark;
  const int16_t* member;
  int32_t Kout, nw_out, gamma, G;
};
struct ClsArgs {
  ClsLayer layer[BMLP_MAX_LAYERS];
  const StepParams* P;
  Ctrl* ctrl;
  int32_t L, c, bs, r_num, r_den;
  int32_t early;   // the CTAs of the layers below the last work before they wait
  OneBatch one;
};
cudaError_t launch_cls_select(const ClsArgs& C, int max_K, cudaStream_t st, bool pdl);
// Group order of every layer with a random partition (DevLayer::member /
// group_of); redraw: keyed by the current step (else by step 0).
constexpr int kMaxOrderK = 16384;   // widest layer that may have a random partition
cudaError_t prepare_group_order();  // shared-memory attribute
cudaError_t launch_group_order(int L, int max_K, bool redraw, cudaStream_t st, bool pdl, const StepParams* P);
// Reinforcement events of every neuron row of every layer for the current
// step into DevLayer::EV (Alg. 3 l.5-12).
void launch_r_events(unsigned grid, cudaStream_t st, const StepParams* P, uint32_t key0, uint32_t key1);
constexpr int kEvThreads = 128, kEvRowsPerWarp = 4;
constexpr int kEvRowsPerCta = kEvThreads / 32 * kEvRowsPerWarp;
// Generic forward for evaluation: A (M x nw_in) against W -> Aout (M x nw_out).
__global__ void k_forward_eval(const uint64_t* __restrict__ A, int64_t M, int nw_in,
                               const uint64_t* __restrict__ W, int N, int Kin,
                               uint64_t* __restrict__ Aout, int nw_out);
// Final classifier argmax for evaluation.
__global__ void k_predict_out(const uint64_t* __restrict__ A, int64_t M, int nw,
                              const uint64_t* __restrict__ PT, int c, int K,
                              int32_t* __restrict__ out);
// Initialisation of H, W of one layer and rho, PT.
__global__ void k_init_hw(uint32_t* H, uint64_t* W, int Kin, int Kout, int ldh, int ngrp, int nplanes,
                          int l, uint32_t key0, uint32_t key1, int h_max);
__global__ void k_init_rho(int8_t* rho, int Kout, int c, int l, uint32_t key0, uint32_t key1);
__global__ void k_pack_pt(const int8_t* rho, uint64_t* PT, int Kout, int c, int nw_out);
__global__ void k_transpose_rho(const int8_t* rho, int8_t* rhoT, int Kout, int c);
// Re-derive W from H for one layer (after set_state).
__global__ void k_repack_w(const uint32_t* H, uint64_t* W, int Kin, int Kout, int ldh, int ngrp,
                           int nplanes, int h_max);
// Tensor-core forward (tcgen05, +-1 as e2m1, exact fp32 sums), training layer
// l.  The activations of layer l - 1 (the inputs for l = 1) are read as packed
// bits.  pdl: launched with the programmatic-stream-serialization attribute.
cudaError_t prepare_train_forward_tc();
cudaError_t launch_train_forward_tc(int bs, int Kout, int Kin, cudaStream_t st, bool pdl,
                                    const StepParams* P, int l, const OneBatch& one);
// The same tiles for one layer of forward-only evaluation on a small batch: A
// (M x nw_in) against W -> Aout (M x nw_out); an expired bounded wait adds one
// to *timeouts.  w_early: with pdl, the launch before it does not write W.
cudaError_t launch_forward_tile(const uint64_t* A, int64_t M, int nw_in, const uint64_t* W, int N, int Kin,
                                uint64_t* Aout, int nw_out, unsigned int* timeouts, cudaStream_t st,
                                bool pdl, bool w_early);
// Whether these tiles or the pairs of launch_forward_eval_tc run an evaluation
// layer faster.  One pattern tile always; else while the tiles fit the SMs once
// and their 1,024-element pieces 1.6 times (tile against pair, us: 1000 -> 525 at
// 2,000 / 4,096 patterns 5.9 / 7.2 and 7.7 / 7.3; 1024 -> 1024 at 2,000 / 4,096 5.8 /
// 6.9 and 7.7 / 7.0; 3072 -> 2048 at 512 / 1,024 9.4 / 9.5 and 11.5 / 9.5; 4096 -> 4096
// at 64 / 256 6.1 / 10.3 and 11.0 / 10.7).
bool forward_tiles_win(int64_t M, int N, int Kin);
// The evaluation output on the same tiles, for at most kPredictTileClasses
// classes: labels[mu] = argmax_j of row mu of A against the c rows of PT (lowest
// j on ties), K the width of the layer.
constexpr int kPredictTileClasses = 128;
cudaError_t launch_predict_tile(const uint64_t* A, int64_t M, int nw, const uint64_t* PT, int c, int K,
                                int32_t* labels, unsigned int* timeouts, cudaStream_t st, bool pdl);
// Median binarisation of n x K fp32 patterns into n x nw packed words.
void launch_binarize_median(const float* x, int64_t n, int K, int nw, uint64_t* out,
                            cudaStream_t st);
// Expansion layer for uint8 inputs: E (K x ceil(D/64) words) from the
// expansion-weight stream, and out = packed sign(x E^T) (n x ceil(K/64)).
void launch_expand_weights(uint64_t seed, int K, int D, uint64_t* E, cudaStream_t st);
// fail_tile >= 0: the tensor-core kernel's CTAs take their wait for the tile of
// this number as expired.
cudaError_t launch_expand_sign(const uint8_t* x, int64_t n, int D, const uint64_t* E, int K,
                               uint64_t* out, cudaStream_t st, int64_t fail_tile = -1);
// SMs of the current device (looked up once).
int sm_count();
// Tensor-core forward for evaluation on large batches: A (M x nw_in) against W
// -> Aout (M x nw_out), 256-pattern x 256-neuron tiles per CTA pair; an expired
// bounded wait adds one to *timeouts.
cudaError_t prepare_forward_eval_tc();
// One CTA waiting (bounded by limit_cycles) on an mbarrier that completes only
// with arrive != 0; an expired wait adds one to *timeouts.
void launch_wait_probe(unsigned int* timeouts, int arrive, unsigned long long limit_cycles,
                       cudaStream_t st);
cudaError_t launch_forward_eval_tc(const uint64_t* A, int64_t M, int nw_in, const uint64_t* W, int N,
                            int Kin, uint64_t* Aout, int nw_out, unsigned int* timeouts,
                            cudaStream_t st, bool pdl);

// One layer on the b1 mma.sync path (kern_forward_b1.cu): Aout (M x nw_out)
// = packed sign(A W^T), sign(0) = +1, pad bits 0.
cudaError_t launch_forward_b1(const uint64_t* A, int64_t M, int nw_in, const uint64_t* W, int N,
                              int Kin, uint64_t* Aout, int nw_out, cudaStream_t st);
// CP + R + repack of every layer with a non-empty M_l, its reinforcement events
// drawn by the kernel, then advance the step (kern_update_rows.cu).  UpdArgs: what the kernel needs of the model, passed by
// value.
struct UpdLayer {
  uint32_t* H;
  uint64_t* W;
  const uint16_t* sel;
  const int16_t* group_of;
  const uint64_t* aprev;   // the layer's input activations of this mini-batch (null: layer 1)
  int32_t Kin, Kout, gamma, ldh, nw_in;
  int32_t lanes;           // lanes of a warp per row
  int32_t upr;             // warps per row
  int32_t cta_base;        // first CTA of the layer
};
struct UpdArgs {
  UpdLayer layer[BMLP_MAX_LAYERS];
  StepParams* P;
  Ctrl* ctrl;
  const RTables* rt;
  int32_t L, bs, nw0, h_max;
  uint32_t key0, key1;
  OneBatch one;
};
// Sets lanes, upr and cta_base of a layer (Kin and Kout given); returns the first
// CTA of the next one.
int update_rows_layout(UpdLayer& Ly, int cta_base);
// pdl: launched with the programmatic-stream-serialization attribute.
cudaError_t launch_update_rows(int nplanes, unsigned grid, cudaStream_t st, bool pdl, const UpdArgs& U);
// The same for large models (kern_update_ws.cu): bulk copies into a ring of
// shared-memory slots, one CTA per SM (grid = the SM count); reads the events
// from DevLayer::EV.
cudaError_t prepare_update_ws();
cudaError_t launch_update_ws(int nplanes, int h_max, int bs, unsigned grid, cudaStream_t st, bool pdl,
                             StepParams* P, const OneBatch& one);
// Attributes of the update kernel: fails when the library holds no sm_103a image.
cudaError_t update_kernel_image(cudaFuncAttributes* fa);
// Peak-rate kernel of one contraction engine (BMLP_FWD_*): launches it on
// `sms` SMs' worth of CTAs and returns the bit-pairs (MACs) it performs.
cudaError_t launch_engine_peak(int engine, int64_t iters, int sms, int* sink, unsigned int* timeouts,
                               cudaStream_t st, double* bitpairs);

// Launch helpers implemented in the kernel files (grid shapes live next to the
// kernels they describe).
dim3 train_forward_grid(int bs, int Kout);
dim3 train_forward_block();
dim3 eval_forward_grid(int64_t M, int Kout);
dim3 eval_forward_block();

}  // namespace bk
