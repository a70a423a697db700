// kern_update_rows.cu -- the hidden-weight update of one training step (Alg. 3:
// clipped perceptron, then reinforcement; Sec. 3.1: W = sign(H) re-packed in
// the same pass) for small and medium models (bmlp_api.cu has the line; above
// it kern_update_ws.cu and k_r_events take its place).
//
// The hidden weights are bit-sliced (DevLayer::H, update_common.cuh): a group
// of 32 inputs of a neuron row is kP words, word p holding bit p of the
// lattice index u = (h + h_max)/2 of the 32 weights.  A clipped step of +-1 is
// a ripple of word operations through the planes, on 32 weights at once.  The
// perceptron step of a tuple (mu, rho) moves weight i up where
// a^mu_i rho_{k,y^mu} = +1 and down elsewhere, so its direction word is the
// group's activation word, complemented when rho = -1 (the selection kernel
// stores rho's sign with the selected neuron); reinforcement moves the weights
// of its events away from 0, so its direction word is the group's h > 0 lanes,
// which is also the group's W word (a step away from 0 never flips a sign).
//
// A lane owns one block of 64 inputs of one row (two groups: 8 kP bytes of
// planes, one 64-bit word of activations per tuple and of W, and one block of
// the reinforcement sampler), a warp 32 consecutive blocks of a row, or the
// blocks of several rows where rows are shorter; nothing is shared between
// warps.  Before it waits for the selection kernel a warp draws its blocks'
// reinforcement events (they depend on the step counter only), loads its planes
// and finds its mini-batch; then it reads its rows' selections (DevLayer::sel of the row's
// group: the patterns whose entry is the row are its tuples), applies the
// tuples in ascending mu, then the events, and writes planes and W.  A row
// without tuple is written only where it has an event.  Layers with an empty
// M_l are skipped (no CP, no R).
// What bounds it: latency (two dependent rounds of L2 loads after the wait) up to
// a few million weights, then instructions (about 700 per warp of 2,048
// weights).  Per step, between CUDA events (5 us of which is their own cost):
// 784 -> 1024 x3 12.3 us against 18.2 for the ring kernel and 10.4 for the event
// draws it replaces, 3072 -> 2048 x3 at 512 patterns 27 against 34 + 12.
#include "update_common.cuh"

namespace bk {
namespace {

using namespace upd;

constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;
constexpr int kEager = 4;   // tuples whose activation words are loaded together

template <int kP, bool kOnes>
__global__ void __launch_bounds__(kThreads) k_update_rows(const __grid_constant__ UpdArgs U) {
  __shared__ Tables tab;
  __shared__ unsigned long long stat[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  Ctrl* ctrl = U.ctrl;
  int li = 0;
  while (li + 1 < U.L && (int)blockIdx.x >= U.layer[li + 1].cta_base) ++li;
  const UpdLayer& Ly = U.layer[li];
  // this lane's row and block
  const int unit = ((int)blockIdx.x - Ly.cta_base) * kWarps + warp;
  const int sub = lane / Ly.lanes;                       // row of the warp (rows shorter than a warp)
  const int k = (unit / Ly.upr) * (32 / Ly.lanes) + sub;
  const int b = (unit % Ly.upr) * 32 + lane % Ly.lanes;
  const int n_in = Ly.Kin - 64 * b;                      // inputs of the block, 64 at most
  const bool live = k < Ly.Kout && n_in > 0;
  if (threadIdx.x == 0) stat[0] = stat[1] = 0ull;
  load_tables<kThreads>(tab, U.rt[li]);
  __syncthreads();
  // ---- before the wait: the block's events and planes ----
  uint64_t ev = 0ull;
  if (live) {
    const uint32_t t = (uint32_t)ctrl->t_cur;
    const int x = n_in >= 64 ? 0 : 1;
    const uint4 u = philox4x32_10(make_uint4((uint32_t)b >> 2, (uint32_t)k, (3u << 16) + (uint32_t)(li + 1), t),
                                  U.key0, U.key1);
    if ((unsigned long long)word_of(u, b & 3) < tab.any[x])
      ev = block_events(tab, x, min(64, n_in), (uint32_t)b, (uint32_t)k, (uint32_t)(li + 1), t, U.key0, U.key1);
  }
  uint32_t u[2][kP];
  uint32_t* hrow = Ly.H + (int64_t)k * Ly.ldh + (int64_t)(2 * b) * kP;
  const bool two = n_in > 32;   // the block's second group exists
  const uint32_t en[2] = {live ? group_mask(0, n_in) : 0u, live ? group_mask(1, n_in) : 0u};
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int p = 0; p < kP; ++p) u[i][p] = 0u;
  if (live) {
    load_planes<kP>(u[0], hrow);
    if (two) load_planes<kP>(u[1], hrow + kP);
  }
  const uint32_t sidx = ctrl->s_cur;
  const int bs = U.bs;
  const int64_t start = U.one.x ? 0 : (int64_t)sidx * bs;
  const int64_t rem = (U.one.x ? U.one.n : U.P->n) - start;
  const int bsz = (int)(rem < bs ? rem : bs);
  const uint64_t* a0 = li == 0 ? (U.one.x ? U.one.x : U.P->x + start * U.nw0) : Ly.aprev;
  pdl_wait();
  pdl_trigger();
  const int gk = live ? (Ly.group_of ? (int)Ly.group_of[k] : k / Ly.gamma) : 0;
  // an expired bounded wait in this step's forward pass: no CP, no R (the
  // selection kernel marked nothing either); the counters still advance
  const bool skip = ctrl->timeouts != 0u || ctrl->any_mark[li] == 0u;
  const Sliced<kP, kOnes> S(U.h_max);
  bool hit_any = false;
  if (!skip) {
    const uint64_t* acol = a0 + b;
    const int nwa = Ly.nw_in;
#pragma unroll 1
    for (int m0 = 0; m0 < bsz; m0 += 128) {
      // tuples of this lane's row among patterns m0 .. m0 + 127: bit i of word q
      uint32_t hit[4] = {0u, 0u, 0u, 0u}, neg[4] = {0u, 0u, 0u, 0u};
      const int rows = 32 / Ly.lanes;
#pragma unroll 1
      for (int r = 0; r < rows; ++r) {
        const int kr = __shfl_sync(kFull, k, r * Ly.lanes), gr = __shfl_sync(kFull, gk, r * Ly.lanes);
        if (kr >= Ly.Kout) break;
        const uint16_t* selg = Ly.sel + (int64_t)gr * bs + m0;
        uint32_t v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = m0 + 32 * q + lane < bsz ? (uint32_t)selg[32 * q + lane] : 0xFFFFu;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t h = __ballot_sync(kFull, (v[q] & 0x7FFFu) == (uint32_t)kr);
          const uint32_t ng = __ballot_sync(kFull, v[q] >> 15);
          if (sub == r) {
            hit[q] = h;
            neg[q] = ng;
          }
        }
      }
      // ---- CP tuples, ascending mu ----
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t h = live ? hit[q] : 0u;
        hit_any |= h != 0u;
        while (h != 0u) {
          // the next tuples of this word, their activation words loaded together
          uint64_t a[kEager];
          uint32_t dir[kEager];
          int cnt = 0;
#pragma unroll
          for (int e = 0; e < kEager; ++e) {
            if (h != 0u) {
              const int i = __ffs(h) - 1;
              h &= h - 1u;
              a[e] = acol[(int64_t)(m0 + 32 * q + i) * nwa];
              dir[e] = ((neg[q] >> i) & 1u) ? kFull : 0u;   // rho = -1: complement
              cnt = e + 1;
            }
          }
#pragma unroll
          for (int e = 0; e < kEager; ++e) {
            if (e < cnt) {
              S.step(u[0], (uint32_t)a[e] ^ dir[e], en[0]);
              S.step(u[1], (uint32_t)(a[e] >> 32) ^ dir[e], en[1]);
            }
          }
        }
      }
    }
    // ---- R: the events step away from 0; W = the lanes with h > 0 ----
    const uint32_t r0 = (uint32_t)ev, r1 = (uint32_t)(ev >> 32);
    const uint32_t pos0 = S.positive(u[0]) & en[0], pos1 = S.positive(u[1]) & en[1];
    if (ev != 0ull) {
      S.step(u[0], pos0, r0);
      S.step(u[1], pos1, r1);
    }
    if (hit_any) Ly.W[(int64_t)k * nwa + b] = (uint64_t)pos0 | ((uint64_t)pos1 << 32);
    if (live && (hit_any || r0 != 0u)) store_planes<kP>(hrow, u[0]);
    if (live && two && (hit_any || r1 != 0u)) store_planes<kP>(hrow + kP, u[1]);
    // ---- statistics: rows, rows streamed (packed), bytes ----
    const bool head = live && b == 0;
    const unsigned hb = __ballot_sync(kFull, head), sb = __ballot_sync(kFull, head && hit_any);
    const unsigned sp = __popc(__ballot_sync(kFull, live && !hit_any && r0 != 0u)) +
                        __popc(__ballot_sync(kFull, live && !hit_any && r1 != 0u));
    if (lane == 0) {
      const unsigned long long bytes =
          (unsigned long long)__popc(sb) * (8ull * Ly.ldh + 8ull * nwa) + 8ull * kP * sp;
      if (hb) atomicAdd(&stat[0], ((unsigned long long)__popc(hb) << 32) | (unsigned)__popc(sb));
      if (bytes) atomicAdd(&stat[1], bytes);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    UpdStat& o = ctrl->stat[blockIdx.x % kStatSlots];
    if (stat[0]) atomicAdd(&o.rows, stat[0] >> 32);
    if (stat[0] & 0xFFFFFFFFull) atomicAdd(&o.streamed, stat[0] & 0xFFFFFFFFull);
    if (stat[1]) atomicAdd(&o.bytes, stat[1]);
    if (blockIdx.x == 0) {
      // the next step's counters (this kernel reads only the copies)
      U.P->s = sidx + 1;
      ctrl->t = ctrl->t_cur + 1;
    }
  }
}

template <int kP, bool kOnes>
cudaError_t launch_one(unsigned grid, cudaStream_t st, bool pdl, const UpdArgs& U) {
  return launch_kernel(k_update_rows<kP, kOnes>, dim3(grid), dim3(kThreads), 0, st, pdl, U);
}

}  // namespace

int update_rows_layout(UpdLayer& Ly, int cta_base) {
  const int nblk = (Ly.Kin + 63) / 64;
  int lanes = 1;
  while (lanes < nblk && lanes < 32) lanes <<= 1;
  Ly.lanes = lanes;
  Ly.upr = (nblk + 31) / 32;
  Ly.cta_base = cta_base;
  const int rows = 32 / lanes;
  const int units = (Ly.Kout + rows - 1) / rows * Ly.upr;
  return cta_base + (units + kWarps - 1) / kWarps;
}

cudaError_t launch_update_rows(int nplanes, unsigned grid, cudaStream_t st, bool pdl, const UpdArgs& U) {
  const bool ones = U.h_max == (1 << nplanes) - 1;
  switch (nplanes) {
    case 1: return launch_one<1, true>(grid, st, pdl, U);
    case 2: return launch_one<2, true>(grid, st, pdl, U);
    case 4: return ones ? launch_one<4, true>(grid, st, pdl, U) : launch_one<4, false>(grid, st, pdl, U);
    case 8: return ones ? launch_one<8, true>(grid, st, pdl, U) : launch_one<8, false>(grid, st, pdl, U);
    case 16: return launch_one<16, false>(grid, st, pdl, U);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t update_kernel_image(cudaFuncAttributes* fa) {
  return cudaFuncGetAttributes(fa, k_update_rows<8, true>);
}

}  // namespace bk
