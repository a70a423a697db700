// kern_update.cu -- local classifiers, selection and the hidden-weight update of
// the BMLP training rule (arXiv 2412.00119, Alg. 1 l.10-18, Alg. 2, Alg. 3), plus
// initialisation and the evaluation output.
#include <climits>

#include "update_common.cuh"

namespace bk {
namespace {

__device__ __forceinline__ int warp_sum(int v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

}  // namespace

// ---------------------------------------------------------------------------
// Local classifier, 01-loss, robustness margin and group selection.
// Grid (bs, L): CTA (mu, l) handles pattern mu of layer l.
//   yhat_j = K_l - 2 popc(A_l[mu] XOR P_l^T[j])                      (Alg. 1 l.10)
//   pred = argmax (lowest j), loss = [pred != y], tau = top1 - top2   (Eq. 1, l.12-13)
//   mark = loss or tau * r_den < r_num * K_l                         (l.14-15)
//   for marked mu, group g: sel = argmax_{k in g} {delta_k < 0},
//   delta_k = z_k rho_{k,y}, ties to the lowest k; none if there is none
//                                                                    (Alg. 2 l.4-8)
// Launched as a programmatic dependent of the last layer's forward pass: the
// CTAs of layers l < L read only what kernels two or more launches back wrote
// (their layer's Z and A, the batch index), so they do all their work before
// waiting, overlapping that forward pass; the CTAs of layer L wait first (all
// CTAs where the kernel before this one writes the group order).  Every CTA
// waits before it lets the next kernel start, so a kernel two launches back
// has always completed.
// Bound: a chain of dependent L2 loads (batch index, label, rho) and two
// barriers, so the model comes as a kernel parameter, label, rho and classifier are
// read before the wait and z beside the activations, and one warp finds the two largest scores
// (with one thread walking over 100 classes the launch of 3072-4096x4 took 16.3 us,
// now 12.3, 5 of them the two events around it).
// ---------------------------------------------------------------------------
namespace {

// A candidate: larger is better.  delta < 0 first, then the lowest neuron; the
// low half is the complement of 2 k + [rho = -1] (delta = z rho < 0, so rho is -1
// exactly where z > 0).  0: no candidate.
__device__ __forceinline__ uint32_t candidate(int k, int z, int rho) {
  const int d = z * rho;
  return d < 0 ? ((uint32_t)(d + 32768) << 16) | (0xFFFFu - (uint32_t)(2 * k + (z > 0 ? 1 : 0))) : 0u;
}
__device__ __forceinline__ uint16_t selection(uint32_t cand) {
  const uint32_t key = 0xFFFFu - (cand & 0xFFFFu);
  return cand == 0u ? kNoSel : (uint16_t)((key >> 1) | ((key & 1u) << 15));
}

__device__ __forceinline__ void cls_select_body(const ClsArgs& C, int li, int mu, bool early) {
  const ClsLayer& Ly = C.layer[li];
  Ctrl* ctrl = C.ctrl;
  __shared__ int yh[BMLP_MAX_CLASSES];
  __shared__ int s_mark, s_timeout;
  const int64_t start = C.one.x ? 0 : (int64_t)batch_index(C.P) * C.bs;
  const bool in = mu < (C.one.x ? C.one.n : C.P->n) - start;
  const int c = C.c;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  const int label = in ? (C.one.x ? C.one.y : C.P->y)[start + mu] : 0;
  const int y = (label < 0 || label >= c) ? 0 : label;  // memory-safe stand-in; the host reports BMLP_EINVAL
  const int K = Ly.Kout, gamma = Ly.gamma, nw = Ly.nw_out;
  const int16_t* z = Ly.Z + (int64_t)mu * K;
  const int8_t* rt = Ly.rhoT + (int64_t)y * K;
  // contiguous groups of 8, 16, .. 256 neurons: one thread per 8 neurons
  const int per = gamma >> 3;  // 8-neuron chunks per group
  const bool chunks = Ly.member == nullptr && (gamma & 7) == 0 && per <= 32 && (per & (per - 1)) == 0;
  const int nchunk = K >> 3;
  const bool mine = chunks && (int)threadIdx.x < nchunk;
  // what no forward pass writes, before the wait: rho, and the classifier's
  // words of this warp's first classes (rows of at most 32 words)
  uint2 rv = make_uint2(0, 0);
  if (mine) rv = *reinterpret_cast<const uint2*>(rt + 8 * threadIdx.x);
  constexpr int kPre = 3;
  uint64_t pre[kPre];
#pragma unroll
  for (int i = 0; i < kPre; ++i)
    pre[i] = (warp + i * nwarps < c && lane < nw) ? Ly.PT[(int64_t)(warp + i * nwarps) * nw + lane] : 0ull;
  if (!early) {
    pdl_wait();
    pdl_trigger();
  }
  if (!in) return;
  // one read of the counter for the whole CTA (the last forward pass may be
  // running beside an early CTA and could raise it meanwhile)
  if (threadIdx.x == 0) s_timeout = ctrl->timeouts != 0u;
  uint4 zv = make_uint4(0, 0, 0, 0);
  if (mine) zv = *reinterpret_cast<const uint4*>(z + 8 * threadIdx.x);
  const uint64_t* a = Ly.A + (int64_t)mu * nw;
  const uint64_t a0 = lane < nw ? a[lane] : 0ull;
#pragma unroll
  for (int i = 0; i < kPre; ++i) {
    const int j = warp + i * nwarps;
    if (j >= c) break;
    int cnt = __popcll(a0 ^ pre[i]);
    for (int w = lane + 32; w < nw; w += 32) cnt += __popcll(a[w] ^ Ly.PT[(int64_t)j * nw + w]);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) yh[j] = K - 2 * cnt;
  }
  for (int j = warp + kPre * nwarps; j < c; j += nwarps) {
    const uint64_t* pt = Ly.PT + (int64_t)j * nw;
    int cnt = 0;
    for (int w = lane; w < nw; w += 32) cnt += __popcll(a[w] ^ pt[w]);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) yh[j] = K - 2 * cnt;
  }
  __syncthreads();
  if (s_timeout) {
    // a bounded wait of this step's forward pass expired (or an earlier one
    // is not yet reported): Z and A are not valid, so the pattern is marked
    // for nothing; with every mark 0 the update leaves H and W as they are
    // and only advances the step counters (the update kernel also skips the
    // step on its own reading of the counter)
    if (threadIdx.x == 0) Ly.mark[mu] = 0;
    return;
  }
  if (warp == 0) {
    // the two largest scores; equal ones differ in the class (lowest first)
    uint32_t b1 = 0u, b2 = 0u;
    for (int j = lane; j < c; j += 32) {
      const uint32_t v = ((uint32_t)(yh[j] + 32768) << 10) | (uint32_t)(BMLP_MAX_CLASSES - 1 - j);
      b2 = max(b2, min(b1, v));
      b1 = max(b1, v);
    }
    const uint32_t m1 = __reduce_max_sync(0xffffffffu, b1);
    const uint32_t m2 = __reduce_max_sync(0xffffffffu, b1 == m1 ? b2 : b1);
    if (lane == 0) {
      if (label != y && li == 0) atomicAdd(&ctrl->bad_labels, 1ull);
      const int tau = (int)(m1 >> 10) - (int)(m2 >> 10);
      const int loss = (BMLP_MAX_CLASSES - 1 - (int)(m1 & 1023u)) != y ? 1 : 0;
      const int mark = loss || ((long long)tau * C.r_den < (long long)C.r_num * K);
      Ly.mark[mu] = (uint8_t)mark;
      if (mark) atomicOr(&ctrl->any_mark[li], 1u);
      if (loss) atomicAdd(&ctrl->layer_err[li], 1ull);
      if (li == C.L - 1 && loss) atomicAdd(&ctrl->err, 1ull);
      s_mark = mark;
    }
  }
  __syncthreads();

  // selections are stored group-major (sel[g][mu]): the update kernel reads a
  // group's bs selections as one contiguous run
  uint16_t* sel = Ly.sel + mu;
  const int64_t sstride = C.bs;
  if (!s_mark) {
    for (int g = threadIdx.x; g < Ly.G; g += blockDim.x) sel[g * sstride] = kNoSel;
    return;
  }
  if (chunks) {
    // the group's per lanes (consecutive, aligned) reduce with shuffles
    for (int base = 0; base < nchunk; base += blockDim.x) {
      const int ci = base + threadIdx.x;
      if (base > 0 && ci < nchunk) {
        zv = *reinterpret_cast<const uint4*>(z + 8 * ci);
        rv = *reinterpret_cast<const uint2*>(rt + 8 * ci);
      }
      uint32_t best = 0u;
      if (ci < nchunk) {
        const uint32_t zw[4] = {zv.x, zv.y, zv.z, zv.w};
        const uint32_t rw[2] = {rv.x, rv.y};
#pragma unroll
        for (int j = 0; j < 8; ++j)
          best = max(best, candidate(8 * ci + j, (int)(int16_t)(zw[j >> 1] >> (16 * (j & 1))),
                                     (int)(int8_t)(rw[j >> 2] >> (8 * (j & 3)))));
      }
      for (int off = per >> 1; off > 0; off >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, off));
      if (ci < nchunk && (ci & (per - 1)) == 0) sel[(ci / per) * sstride] = selection(best);
    }
    return;
  }
  // warp per group; the group's neurons are contiguous or listed by the group
  // order (random partition)
  const int16_t* member = Ly.member;
  for (int g = warp; g < Ly.G; g += nwarps) {
    uint32_t best = 0u;
    for (int kk = lane; kk < gamma; kk += 32) {
      const int k = member ? (int)member[g * gamma + kk] : g * gamma + kk;
      best = max(best, candidate(k, (int)z[k], (int)rt[k]));
    }
    best = __reduce_max_sync(0xffffffffu, best);
    if (lane == 0) sel[g * sstride] = selection(best);
  }
}

__global__ void __launch_bounds__(512, 3) k_cls_select(const __grid_constant__ ClsArgs C) {
  const int li = blockIdx.y;
  const int mu = blockIdx.x;
  const bool early = C.early && li < C.L - 1;
  cls_select_body(C, li, mu, early);
  if (early) {
    pdl_wait();
    pdl_trigger();
  }
}

}  // namespace

cudaError_t launch_cls_select(const ClsArgs& C, int max_K, cudaStream_t st, bool pdl) {
  // a thread per 8 neurons of the widest layer, 4 to 16 warps
  const int threads = max_K <= 1024 ? 128 : (max_K <= 2048 ? 256 : 512);
  return launch_kernel(k_cls_select, dim3((unsigned)C.bs, (unsigned)C.L), dim3(threads), 0, st, pdl, C);
}

namespace {

using namespace upd;

}  // namespace

// Reinforcement events of the current step (Alg. 3 l.5-12): a warp takes
// kEvRowsPerWarp neuron rows; lane j draws the block draws of blocks 4j .. 4j+3 of
// each (one Philox call), the blocks that hold an event are listed per warp, and
// the lanes share that list for the event draws; the rows' bitmaps go to
// DevLayer::EV, zeros first.  It depends only on (seed, layer, neuron, step, p_r),
// so it runs beside the forward passes.  Bound: instruction issue.  A list of
// several rows leaves fewer lanes idle in its last round than one of a row (32
// candidates of 128 blocks at 8192 inputs): 24.3 us for the four
// layers of 8192 alone, 28.6 with a list per row, 31 with a CTA of eight rows.  Registers are
// held to twelve CTAs per SM, so that they fit beside the CTAs of a forward pass.
__global__ void __launch_bounds__(kEvThreads, 12) k_r_events(const StepParams* __restrict__ P,
                                                             uint32_t key0, uint32_t key1) {
  constexpr int kW = kEvThreads / 32;
  __shared__ Tables s_rt;
  __shared__ uint16_t s_cand[kW][128 * kEvRowsPerWarp];   // row * 128 + block
  const int bid = blockIdx.x;
  int li = 0;
  while (li + 1 < P->L && bid >= P->layer[li + 1].ev_cta_base) ++li;
  const DevLayer& Ly = P->layer[li];
  load_tables<kEvThreads>(s_rt, P->rt[li]);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t l = (uint32_t)li + 1u;
  const uint32_t tt = (uint32_t)P->ctrl->t;   // the first pass may not have copied it yet
  const int Kin = Ly.Kin, nblk = Ly.nblk, stride = Ly.ev_stride;
  uint16_t* cand = s_cand[warp];
  const int k0 = (bid - Ly.ev_cta_base) * kEvRowsPerCta + warp * kEvRowsPerWarp;
  const int rows = min(kEvRowsPerWarp, Ly.Kout - k0);
  uint64_t* ev0 = Ly.EV + (int64_t)k0 * stride;
  const uint32_t below = (1u << lane) - 1u;
  __syncthreads();
  // rounds of 128 blocks
#pragma unroll 1
  for (int g0 = 0; 4 * g0 < nblk && rows > 0; g0 += 32) {
    const int gq = g0 + lane;
    int total = 0;
#pragma unroll 1
    for (int r = 0; r < rows; ++r) {
      uint4 u = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
      if (4 * gq < nblk) {
        u = philox4x32_10(make_uint4((uint32_t)gq, (uint32_t)(k0 + r), (3u << 16) + l, tt), key0, key1);
        // rows are 16-byte aligned and stride is even
        uint4* z = reinterpret_cast<uint4*>(ev0 + (int64_t)r * stride + 4 * gq);
        z[0] = make_uint4(0, 0, 0, 0);
        if (4 * gq + 2 < stride) z[1] = make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int wq = 0; wq < 4; ++wq) {
        const int b = 4 * gq + wq;
        const bool in = b < nblk && (unsigned long long)word_of(u, wq) < s_rt.any[(Kin - 64 * b >= 64) ? 0 : 1];
        const uint32_t bal = __ballot_sync(kFull, in);
        if (in) cand[total + __popc(bal & below)] = (uint16_t)(128 * r + 4 * lane + wq);
        total += __popc(bal);
      }
    }
    __syncwarp();   // the list and the zeros
#pragma unroll 1
    for (int i = lane; i < total; i += 32) {
      const int c = cand[i], b = 4 * g0 + (c & 127), r = c >> 7;
      const int n = min(64, Kin - 64 * b);
      ev0[(int64_t)r * stride + b] = block_events(s_rt, (n == 64) ? 0 : 1, n, (uint32_t)b, (uint32_t)(k0 + r), l,
                                                  tt, key0, key1);
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// Group order of a layer with a random partition (Sec. 4.3): the neurons in
// ascending order of the keys u_k = word k%4 of Philox (k/4, 0, 32*2^16 + l, t'),
// ties to the smaller k; member[j] = the j-th neuron and group_of[k] = j / gamma.
// t' = the step counter when redrawn every step, else 0.
// A neuron's place is the number of keys before its own: every CTA draws all of
// the layer's keys into shared memory (a Philox call for four) and ranks
// kOrderPer neurons, kOrderSplit threads sharing the comparisons of each.  K^2
// comparisons over the whole GPU take less time than a sort of K keys in one
// CTA (2048 neurons, three layers: 23.4 us sorted; a step of
// 3072-2048x3 at 512 patterns 88.4 -> 78.0 us).  As a programmatic dependent (redraw) it ranks before it
// waits: t and what it overwrites were settled two launches back.
// ---------------------------------------------------------------------------
constexpr int kOrderThreads = 256, kOrderSplit = 8, kOrderPer = kOrderThreads / kOrderSplit;

__global__ void __launch_bounds__(kOrderThreads) k_group_order(const StepParams* __restrict__ P, int redraw) {
  extern __shared__ uint4 keys4[];
  const DevLayer& Ly = P->layer[blockIdx.y];
  const int K = Ly.Kout, k0 = (int)blockIdx.x * kOrderPer;
  if (Ly.member != nullptr && k0 < K) {
    const uint32_t t = redraw ? (uint32_t)P->ctrl->t : 0u;
    const int n4 = (K + 3) / 4;
    for (int i = threadIdx.x; i < n4; i += kOrderThreads)
      keys4[i] = philox4x32_10(make_uint4((uint32_t)i, 0u, (32u << 16) + (uint32_t)(blockIdx.y + 1), t), P->key0,
                               P->key1);
    __syncthreads();
    const uint32_t* keys = reinterpret_cast<const uint32_t*>(keys4);
    const int k = k0 + (int)threadIdx.x / kOrderSplit, part = (int)threadIdx.x % kOrderSplit;
    const uint32_t mine = k < K ? keys[k] : 0u;
    uint32_t before = 0u;
    // the four keys of i: all before k, all after it, or (one i) around it
    for (int i = part; i < n4; i += kOrderSplit) {
      const uint4 v = keys4[i];
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = 4 * i + e;
        before += (j < K && (w[e] < mine || (w[e] == mine && j < k))) ? 1u : 0u;
      }
    }
#pragma unroll
    for (int off = kOrderSplit / 2; off > 0; off >>= 1) before += __shfl_xor_sync(0xffffffffu, before, off);
    if (part == 0 && k < K) {
      Ly.member[before] = (int16_t)k;
      Ly.group_of[k] = (int16_t)((int)before / Ly.gamma);
    }
  }
  pdl_wait();
  pdl_trigger();
}

static size_t group_order_smem(int max_K) { return sizeof(uint4) * (size_t)((max_K + 3) / 4); }

// The widest layer's for every handle: the attribute belongs to the kernel, not to a handle.
cudaError_t prepare_group_order() {
  return cudaFuncSetAttribute(k_group_order, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)group_order_smem(kMaxOrderK));
}

cudaError_t launch_group_order(int L, int max_K, bool redraw, cudaStream_t st, bool pdl, const StepParams* P) {
  return launch_kernel(k_group_order, dim3((unsigned)((max_K + kOrderPer - 1) / kOrderPer), (unsigned)L),
                       dim3(kOrderThreads), group_order_smem(max_K), st, pdl, P, redraw ? 1 : 0);
}

void launch_r_events(unsigned grid, cudaStream_t st, const StepParams* P, uint32_t key0, uint32_t key1) {
  k_r_events<<<grid, kEvThreads, 0, st>>>(P, key0, key1);
}

// ---------------------------------------------------------------------------
// Evaluation output: pred = argmax_j (K_L - 2 popc(A_L[mu] XOR P_L^T[j])),
// lowest j on ties.  One warp per pattern.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_predict_out(const uint64_t* __restrict__ A, int64_t M,
                                                     int nw, const uint64_t* __restrict__ PT,
                                                     int c, int K, int32_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t mu = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (mu >= M) return;
  const uint64_t* a = A + mu * nw;
  int best = INT_MIN, bestj = 0;
  for (int j = 0; j < c; ++j) {
    const uint64_t* pt = PT + (int64_t)j * nw;
    int cnt = 0;
    for (int w = lane; w < nw; w += 32) cnt += __popcll(a[w] ^ pt[w]);
    cnt = warp_sum(cnt);
    const int v = K - 2 * cnt;
    if (v > best) {
      best = v;
      bestj = j;
    }
  }
  if (lane == 0) out[mu] = bestj;
}

// ---------------------------------------------------------------------------
// Initialisation (Alg. 1 l.2): h_ik = +-1 from Philox purpose 1, stored
// bit-sliced (DevLayer::H) as the lattice index u = (h + h_max)/2, i.e.
// (h_max + 1)/2 for +1 and (h_max - 1)/2 for -1; inputs i >= K_in keep u = 0
// and W bit 0; W = packed sign(H).  One thread per group of 32 inputs of one
// neuron row; H and W are zeroed beforehand (row padding).
// ---------------------------------------------------------------------------
__global__ void k_init_hw(uint32_t* H, uint64_t* W, int Kin, int Kout, int ldh, int ngrp, int nplanes,
                          int l, uint32_t key0, uint32_t key1, int h_max) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)Kout * ngrp) return;
  const int k = (int)(idx / ngrp);
  const int g = (int)(idx % ngrp);
  uint32_t pos = 0u;   // bit j: h of input 32 g + j is +1
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const uint4 r = philox4x32_10(make_uint4(8u * g + q, (uint32_t)k, (1u << 16) + (uint32_t)l, 0u), key0, key1);
    pos |= ((r.x >> 31) << (4 * q)) | ((r.y >> 31) << (4 * q + 1)) | ((r.z >> 31) << (4 * q + 2)) |
           ((r.w >> 31) << (4 * q + 3));
  }
  const uint32_t valid = upd::group_mask(g, Kin);
  pos &= valid;
  const int up = (h_max + 1) / 2, dn = up - 1;   // u of h = +1, h = -1
  uint32_t* hg = H + (int64_t)k * ldh + (int64_t)g * nplanes;
  for (int p = 0; p < nplanes; ++p) {
    const uint32_t m1 = ((up >> p) & 1) ? upd::kFull : 0u, m0 = ((dn >> p) & 1) ? upd::kFull : 0u;
    hg[p] = ((pos & m1) | (~pos & m0)) & valid;
  }
  reinterpret_cast<uint32_t*>(W + (int64_t)k * ((ngrp + 1) / 2))[g] = pos;
}

// rho_kj = +-1 from Philox purpose 2 (Sec. 3.1).
__global__ void k_init_rho(int8_t* rho, int Kout, int c, int l, uint32_t key0, uint32_t key1) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)Kout * c) return;
  const int k = (int)(idx / c);
  const int j = (int)(idx % c);
  const uint4 r = philox4x32_10(make_uint4((uint32_t)(j >> 2), (uint32_t)k, (2u << 16) + (uint32_t)l, 0u), key0, key1);
  const uint32_t w = (j & 3) == 0 ? r.x : (j & 3) == 1 ? r.y : (j & 3) == 2 ? r.z : r.w;
  rho[idx] = (w >> 31) ? (int8_t)1 : (int8_t)-1;
}

// PT[j] = packed column j of P_l (bit k%64 of word k/64 = rho_kj > 0).
__global__ void k_pack_pt(const int8_t* rho, uint64_t* PT, int Kout, int c, int nw_out) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)c * nw_out) return;
  const int j = (int)(idx / nw_out);
  const int w = (int)(idx % nw_out);
  uint64_t bits = 0;
  for (int b = 0; b < 64; ++b) {
    const int k = 64 * w + b;
    if (k < Kout && rho[(int64_t)k * c + j] > 0) bits |= 1ull << b;
  }
  PT[idx] = bits;
}

// rhoT[j][k] = rho[k][j].
__global__ void k_transpose_rho(const int8_t* rho, int8_t* rhoT, int Kout, int c) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)Kout * c) return;
  const int j = (int)(idx / Kout);
  const int k = (int)(idx % Kout);
  rhoT[idx] = rho[(int64_t)k * c + j];
}

// W = packed sign(H) for one layer (H bit-sliced), pad bits 0: per group of
// 32 inputs, the lanes with u >= (h_max + 1)/2.  One thread per group.
__global__ void k_repack_w(const uint32_t* H, uint64_t* W, int Kin, int Kout, int ldh, int ngrp,
                           int nplanes, int h_max) {
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (int64_t)Kout * ngrp) return;
  const int k = (int)(idx / ngrp);
  const int g = (int)(idx % ngrp);
  const int m = (h_max + 1) / 2;
  const uint32_t* hg = H + (int64_t)k * ldh + (int64_t)g * nplanes;
  uint32_t gt = 0u, eq = upd::kFull;
  for (int p = nplanes - 1; p >= 0; --p) {
    const uint32_t mp = ((m >> p) & 1) ? upd::kFull : 0u;
    gt |= eq & hg[p] & ~mp;
    eq &= ~(hg[p] ^ mp);
  }
  reinterpret_cast<uint32_t*>(W + (int64_t)k * ((ngrp + 1) / 2))[g] = (gt | eq) & upd::group_mask(g, Kin);
}

}  // namespace bk
