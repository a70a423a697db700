// kern_binarize.cu -- MedianBinarization of real-valued input patterns
// (Alg. 1 l.5; Sec. 3.2: the median value is the threshold).
//
//   a_i = +1  iff  x_i > m,   m = the ceil(K/2)-th smallest of the pattern's K
//                              values (lower median), compared in fp32
//
// packed as bits (bit i % 64 of word i / 64 = 1 <-> +1, pad bits 0), the input
// format of bmlp_train / bmlp_predict.
//
// k_binarize_regs (K <= kRegMax): a warp, or four warps, per pattern, with the
// pattern's values in registers as order-preserving 32-bit keys (bits ^
// 0x80000000 for a clear sign bit, ~bits for a set one), so that memory is read
// once.  The median is the key p with #{key < p} <= rank < #{key <= p}.  It is
// bracketed: the median lies in [lo, hi], with #{key < lo} and #{key <= hi}
// known.  The smallest value is tried first (the median of image-like data, which
// is mostly zeros), then keys inside the bracket, interpolated linearly between
// its ends by the counts (from the sixth round on in turn with the middle of the
// key range, which alone ends after 32 rounds).  A round is one comparison per
// value and a warp sum.  Once at most 32 candidates are left a warp lists them,
// one per lane, and ranks each against the others; with many equal values the
// bracket's ends move onto values instead.  Then the values are compared with
// the median as floats, so -0 and +0 are equal as they are in fp32, and one
// ballot packs 32 of them.
// Bound: memory, then instructions (about 8 per value).  60,000 x 784 of
// grey levels: 52.4 us = 3.7 TB/s (the radix select 299 us).
//
// k_binarize_median (larger K): one CTA per pattern.  The median is found
// exactly by a radix select over the same keys: four passes of 8-bit digits,
// most significant first, each a shared-memory histogram of the keys that share
// the digits chosen so far, then one warp scans the 256 counts and picks the
// bucket holding the target rank.  The pattern's row is read five times (four
// passes and the packing); it stays in L1 between them.
#include "bmlp_internal.cuh"

namespace bk {
namespace {

constexpr int kBinThreads = 256;

__device__ __forceinline__ uint32_t float_key(float v) {
  const uint32_t u = __float_as_uint(v);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float key_float(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

constexpr int kRegWarps = 4;        // warps of a CTA
constexpr int kRegMax = 32 * kRegWarps * 32;

// kWarps warps per pattern (1 or kRegWarps), kR values per lane: K <= 32 kWarps kR.
// Value j of lane l of the pattern's warp w is x[32 (w + kWarps j) + l].
template <int kWarps, int kR>
__global__ void __launch_bounds__(32 * kRegWarps)
    k_binarize_regs(const float* __restrict__ x, int64_t n, int K, int nw, uint64_t* __restrict__ out) {
  __shared__ uint32_t red[2][kRegWarps];
  __shared__ uint32_t cand[kWarps == 1 ? kRegWarps : 1][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int w = kWarps == 1 ? 0 : warp;
  constexpr int kPats = kRegWarps / kWarps;     // patterns per CTA
  const uint32_t rank = (uint32_t)((K + 1) / 2 - 1);   // 0-based rank of the lower median
  int flip = 0;
  // a sum (or minimum / maximum) over the pattern's warps
  auto all_warps = [&](uint32_t v, int op) -> uint32_t {
    const uint32_t r = op == 0 ? __reduce_add_sync(0xffffffffu, v)
                               : (op == 1 ? __reduce_min_sync(0xffffffffu, v) : __reduce_max_sync(0xffffffffu, v));
    if constexpr (kWarps == 1) return r;
    if (lane == 0) red[flip][warp] = r;
    __syncthreads();
    uint32_t t = red[flip][0];
#pragma unroll
    for (int i = 1; i < kRegWarps; ++i)
      t = op == 0 ? t + red[flip][i] : (op == 1 ? min(t, red[flip][i]) : max(t, red[flip][i]));
    flip ^= 1;   // the next round writes the other buffer: no second barrier
    return t;
  };
  for (int64_t mu = (int64_t)blockIdx.x * kPats + (kWarps == 1 ? warp : 0); mu < n;
       mu += (int64_t)gridDim.x * kPats) {
    const float* row = x + mu * (int64_t)K;
    uint32_t key[kR];   // values past K: the largest key, never below a pivot
#pragma unroll
    for (int j = 0; j < kR; ++j) {
      const int i = 32 * (w + kWarps * j) + lane;
      key[j] = i < K ? __float_as_uint(__ldcs(row + i)) : 0x7FFFFFFFu;
    }
    uint32_t kmin = 0xFFFFFFFFu, kmax = 0u;
#pragma unroll
    for (int j = 0; j < kR; ++j) {
      key[j] ^= (uint32_t)((int32_t)key[j] >> 31) | 0x80000000u;
      kmin = min(kmin, key[j]);
      if (32 * (w + kWarps * j) + lane < K) kmax = max(kmax, key[j]);
    }
    uint32_t lo = all_warps(kmin, 1), hi = all_warps(kmax, 2);
    uint32_t clo = 0u, chi = (uint32_t)K;   // #{key < lo}, #{key <= hi}
    uint32_t p = lo;
#pragma unroll 1
    for (int it = 0;; ++it) {
      uint32_t c = 0u;   // #{key <= p} (p < hi, or every value is p: padding never counts)
#pragma unroll
      for (int j = 0; j < kR; ++j) c += key[j] <= p ? 1u : 0u;
      c = all_warps(c, 0);
      if (c > rank) {
        hi = p;
        chi = c;
      } else {
        lo = p + 1u;
        clo = c;
      }
      if (lo >= hi) break;
      if (kWarps == 1 && chi - clo <= 32u && hi != 0xFFFFFFFFu) {
        // at most a warp of candidates: one per lane, ranked against the others
        uint32_t* list = cand[warp];
        uint32_t cnt = 0u;
#pragma unroll
        for (int j = 0; j < kR; ++j) {
          const bool in = key[j] >= lo && key[j] <= hi;
          const unsigned b = __ballot_sync(0xffffffffu, in);
          if (in) list[cnt + __popc(b & ((1u << lane) - 1u))] = key[j];
          cnt += __popc(b);
        }
        __syncwarp();
        const uint32_t mine = (uint32_t)lane < cnt ? list[lane] : 0xFFFFFFFFu;
        uint32_t below = 0u;
        for (uint32_t i = 0; i < cnt; ++i) {
          const uint32_t o = list[i];
          below += (o < mine || (o == mine && i < (uint32_t)lane)) ? 1u : 0u;
        }
        const unsigned at = __ballot_sync(0xffffffffu, (uint32_t)lane < cnt && below == rank - clo);
        hi = __shfl_sync(0xffffffffu, mine, __ffs(at) - 1);
        __syncwarp();
        break;
      }
      if (it >= 3 || chi - clo == 1u) {
        // the bracket's ends onto values (many equal ones, or one candidate)
        uint32_t a = 0xFFFFFFFFu, z = 0u;
#pragma unroll
        for (int j = 0; j < kR; ++j) {
          if (key[j] >= lo) a = min(a, key[j]);
          if (key[j] <= hi) z = max(z, key[j]);
        }
        lo = all_warps(a, 1);
        hi = all_warps(z, 2);
        if (lo >= hi) break;
      }
      p = lo + ((hi - lo) >> 1);
      if (it < 6 || (it & 1) == 0) {
        const float flo = key_float(lo), fhi = key_float(hi);
        const float f = flo + (fhi - flo) * (((float)(rank - clo) + 0.5f) / (float)(chi - clo));
        const uint32_t kf = float_key(f);
        if (kf >= lo && kf < hi) p = kf;   // (a NaN's or an infinity's key: the middle)
      }
    }
    const float m = key_float(hi);
    uint32_t mine = 0u;
#pragma unroll
    for (int j = 0; j < kR; ++j) {
      const int i = 32 * (w + kWarps * j) + lane;
      const unsigned bits = __ballot_sync(0xffffffffu, i < K && key_float(key[j]) > m);
      if (lane == j) mine = bits;
    }
    // lane j holds word w + kWarps j of the row
    const int word = w + kWarps * lane;
    if (word < 2 * nw) reinterpret_cast<uint32_t*>(out + mu * (int64_t)nw)[word] = mine;
  }
}

__global__ void __launch_bounds__(kBinThreads)
    k_binarize_median(const float* __restrict__ x, int64_t n, int K, int nw, uint64_t* __restrict__ out) {
  __shared__ uint32_t hist[256];
  __shared__ uint32_t s_prefix, s_rank;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int64_t mu = blockIdx.x; mu < n; mu += gridDim.x) {
    const float* row = x + mu * (int64_t)K;
    uint32_t prefix = 0, mask = 0;
    uint32_t rank = (uint32_t)((K + 1) / 2 - 1);  // 0-based rank of the lower median
    for (int shift = 24; shift >= 0; shift -= 8) {
      for (int i = threadIdx.x; i < 256; i += kBinThreads) hist[i] = 0;
      __syncthreads();
      for (int i = threadIdx.x; i < K; i += kBinThreads) {
        const uint32_t key = float_key(row[i]);
        if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 0xFFu], 1u);
      }
      __syncthreads();
      if (warp == 0) {
        // lane j owns buckets 8j .. 8j + 7; an inclusive scan of the lane sums
        // finds the lane whose buckets hold the rank, then that lane walks them
        uint32_t c[8], sum = 0;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          c[b] = hist[8 * lane + b];
          sum += c[b];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t v = __shfl_up_sync(0xffffffffu, incl, d);
          if (lane >= d) incl += v;
        }
        const uint32_t excl = incl - sum;
        if (excl <= rank && rank < incl) {
          uint32_t below = excl;
          int b = 0;
          while (below + c[b] <= rank) below += c[b++];
          s_prefix = prefix | ((uint32_t)(8 * lane + b) << shift);
          s_rank = rank - below;
        }
      }
      __syncthreads();
      prefix = s_prefix;
      rank = s_rank;
      mask |= 0xFFu << shift;
    }
    const float m = key_float(prefix);
    uint32_t* o = reinterpret_cast<uint32_t*>(out + mu * (int64_t)nw);
    for (int w = warp; w < 2 * nw; w += kBinThreads / 32) {
      const int i = 32 * w + lane;
      const unsigned bits = __ballot_sync(0xffffffffu, i < K && row[i] > m);
      if (lane == 0) o[w] = bits;
    }
    __syncthreads();  // hist, s_prefix and s_rank are reused by the next pattern
  }
}

}  // namespace

void launch_binarize_median(const float* x, int64_t n, int K, int nw, uint64_t* out,
                            cudaStream_t st) {
  const int64_t grid = n < (int64_t)1 << 20 ? n : (int64_t)1 << 20;
  auto regs = [&](auto kern, int pats) {
    const int64_t ctas = (n + pats - 1) / pats;
    kern<<<(unsigned)(ctas < grid ? ctas : grid), 32 * kRegWarps, 0, st>>>(x, n, K, nw, out);
  };
  if (K <= 32 * 8) regs(k_binarize_regs<1, 8>, kRegWarps);
  else if (K <= 32 * 16) regs(k_binarize_regs<1, 16>, kRegWarps);
  else if (K <= 32 * 25) regs(k_binarize_regs<1, 25>, kRegWarps);
  else if (K <= 32 * 32) regs(k_binarize_regs<1, 32>, kRegWarps);
  else if (K <= kRegMax / 2) regs(k_binarize_regs<kRegWarps, 16>, 1);
  else if (K <= kRegMax) regs(k_binarize_regs<kRegWarps, 32>, 1);
  else k_binarize_median<<<(unsigned)grid, kBinThreads, 0, st>>>(x, n, K, nw, out);
}

}  // namespace bk
